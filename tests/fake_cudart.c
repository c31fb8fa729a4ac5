/* Stand-ins for the CUDA runtime's memory calls on a machine without a GPU, loaded with LD_PRELOAD in
 * front of libcudart: device memory is host memory, kernels do nothing, and a test can make an
 * allocation fail, change the context and ask what was allocated, freed and waited for. */
#include <stdlib.h>
#include <string.h>

#define MAX_BLOCKS 4096
enum { OK = 0, INVALID = 1, OOM = 2, NO_CALL = 900 };
enum { MALLOC = 1, POOL = 2 };

static struct {
    void* p;
    size_t bytes;
    int kind;
} blocks[MAX_BLOCKS];
static size_t fail_bytes = (size_t)-1;
static int fail_in = -1;
static unsigned long long context = 1;
static unsigned word;
static int has_word, unwaited, bad_frees, dead_pool, trims, device_syncs;
struct pool {
    unsigned long long context;
};

/* for the tests */
void fake_fail_from(size_t bytes) { fail_bytes = bytes; }             /* allocations of that size or more */
void fake_fail_nth(int n) { fail_in = n; }                              /* the n-th allocation from here */
void fake_new_context(void) {                                           /* as cudaDeviceReset does */
    ++context;
    for (int i = 0; i < MAX_BLOCKS; ++i)
        if (blocks[i].p) {
            free(blocks[i].p);
            blocks[i].p = NULL;
        }
}
int fake_bad_frees(void) { return bad_frees; }       /* of addresses that are not allocated */
void fake_copy_word(int on, unsigned v) { has_word = on, word = v; }    /* what a 4-byte copy to the host brings */
int fake_live(int kind) {
    int n = 0;
    for (int i = 0; i < MAX_BLOCKS; ++i) n += blocks[i].p && (blocks[i].kind & kind);
    return n;
}
int fake_dead_pool(void) { return dead_pool; }       /* allocations from a pool of an earlier context */
int fake_trims(void) { return trims; }
int fake_device_syncs(void) { return device_syncs; } /* an error while any stream of the process is captured */
int fake_unwaited(void) { return unwaited; }         /* pool memory released by cudaFree with nothing waited for */

static int waited;
static int take(void** p, size_t bytes, int kind) {
    *p = NULL;
    if (bytes >= fail_bytes || (fail_in > 0 && --fail_in == 0)) return OOM;
    for (int i = 0; i < MAX_BLOCKS; ++i)
        if (!blocks[i].p) {
            *p = blocks[i].p = aligned_alloc(256, (bytes + 511) / 256 * 256);
            memset(*p, 0, (bytes + 511) / 256 * 256);
            blocks[i].bytes = bytes, blocks[i].kind = kind;
            return OK;
        }
    return OOM;
}
static int drop(void* p, int plain) {
    if (!p) return OK;
    for (int i = 0; i < MAX_BLOCKS; ++i)
        if (blocks[i].p == p) {
            if (plain && blocks[i].kind == MALLOC) waited = 1; /* cudaFree waits for the device */
            if (plain && blocks[i].kind == POOL && !waited) ++unwaited;
            free(p);
            blocks[i].p = NULL;
            return OK;
        }
    ++bad_frees;
    return INVALID;
}
int cudaMalloc(void** p, size_t n) { return take(p, n, MALLOC); }
int cudaFree(void* p) { return drop(p, 1); }
int cudaMallocAsync(void** p, size_t n, void* s) { return take(p, n, POOL); }
int cudaFreeAsync(void* p, void* s) { return drop(p, 0); }
int cudaMemPoolCreate(void** out, const void* props) {
    struct pool* q = malloc(sizeof(*q));
    q->context = context;
    *out = q;
    return OK;
}
int cudaMemPoolSetAttribute(void* q, int attr, void* v) { return OK; }
int cudaMemPoolTrimTo(void* q, size_t keep) {
    if (((struct pool*)q)->context != context) ++dead_pool;
    ++trims;
    return OK;
}
int cudaMallocFromPoolAsync(void** p, size_t n, void* q, void* s) {
    waited = 0; /* work on the new block may follow */
    if (((struct pool*)q)->context != context) {
        ++dead_pool;
        return INVALID;
    }
    return take(p, n, POOL);
}
int cudaMemcpyAsync(void* d, const void* s, size_t n, int kind, void* stream) {
    memcpy(d, s, n);
    if (kind == 2 && n == 4 && has_word) memcpy(d, &word, 4);
    return OK;
}
int cudaMemcpy(void* d, const void* s, size_t n, int kind) { return cudaMemcpyAsync(d, s, n, kind, NULL); }
int cudaMemsetAsync(void* d, int v, size_t n, void* s) {
    memset(d, v, n);
    return OK;
}
int cudaMemset(void* d, int v, size_t n) { return cudaMemsetAsync(d, v, n, NULL); }
int cudaGetDevice(int* d) { return *d = 0, OK; }
int cudaSetDevice(int d) { return OK; }
int cudaGetLastError(void) { return OK; }
int cudaStreamSynchronize(void* s) { return OK; }
int cudaDeviceSynchronize(void) { return ++device_syncs, waited = 1, OK; }
int cudaDeviceGetAttribute(int* v, int attr, int d) { return *v = 4, OK; }
int cudaOccupancyMaxActiveBlocksPerMultiprocessor(int* n, const void* f, int b, size_t s) { return *n = 1, OK; }
int cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void* f, int b, size_t s, unsigned x) { return *n = 1, OK; }
int cudaFuncSetAttribute(const void* f, int attr, int v) { return OK; }
int __cudaGetKernel(void** k, const void* f) { return *k = (void*)f, OK; }
struct dim {
    unsigned x, y, z;
};
/* the batch kernels are the ones launched by this call; their second argument is */
struct batch_args {
    struct {
        int kernel;
        const double *x, *y, *z;
        long long n;
        float* u;
        int* host;
        long long tile0;
    } g[16];
    int ng;
    long long ntiles;
    int pts;
};
static struct batch_args batch[8];
static int n_batch;
int cudaLaunchKernel(const void* f, struct dim g, struct dim b, void** a, size_t m, void* s) {
    if (n_batch < 8) batch[n_batch++] = *(struct batch_args*)a[1];
    return OK;
}
/* bytes from p to the end of the allocation that holds it, as it was asked for; -1: in none */
static long long room(const void* p) {
    for (int i = 0; i < MAX_BLOCKS; ++i) {
        const char* b = blocks[i].p;
        if (b && (const char*)p >= b && (const char*)p < b + blocks[i].bytes) return b + blocks[i].bytes - (const char*)p;
    }
    return -1;
}
/* whether group g's arrays of launch i (positions and results) lie within their allocations, apart from one another */
int fake_batch_fits(int i, int g) {
    const long long n = batch[i].g[g].n;
    const char* a[5] = {(const char*)batch[i].g[g].x, (const char*)batch[i].g[g].y, (const char*)batch[i].g[g].z,
                        (const char*)batch[i].g[g].u, (const char*)batch[i].g[g].host};
    const long long bytes[5] = {8 * n, 8 * n, 8 * n, 12 * n, 4 * n};
    for (int k = 0; k < 5; ++k) {
        if (!a[k]) continue;
        if (room(a[k]) < bytes[k]) return 0;
        for (int j = 0; j < k; ++j)
            if (a[j] && a[k] < a[j] + bytes[j] && a[j] < a[k] + bytes[k]) return 0;
    }
    return 1;
}
int fake_batch_launches(void) { return n_batch; }
int fake_batch_kernel(int i) { return batch[i].g[0].kernel; }
int fake_batch_pts(int i) { return batch[i].pts; }
int fake_batch_tiles(int i) { return (int)batch[i].ntiles; }
void fake_forget_batches(void) { n_batch = 0; }
int cudaStreamCreateWithFlags(void** s, unsigned f) { return *s = NULL, OK; }
int cudaStreamDestroy(void* s) { return OK; }
int cudaStreamBeginCapture(void* s, int mode) { return OK; }
int cudaStreamEndCapture(void* s, void** g) { return *g = malloc(1), OK; }
int cudaGraphInstantiate(void** e, void* g, unsigned long long f) { return *e = malloc(1), OK; }
int cudaGraphDestroy(void* g) { return free(g), OK; }
int cudaGraphExecDestroy(void* e) { return free(e), OK; }
int __cudaLaunchKernel(void* f, struct dim g, struct dim b, void** a, size_t m, void* s) { return OK; }
static int get_current(void** c) { return *c = &context, OK; }
static int get_id(void* c, unsigned long long* id) { return *id = context, OK; }
int cudaGetDriverEntryPointByVersion(const char* name, void** f, unsigned v, unsigned long long fl, int* found) {
    *f = !strcmp(name, "cuCtxGetCurrent") ? (void*)get_current : !strcmp(name, "cuCtxGetId") ? (void*)get_id : NULL;
    if (found) *found = *f ? 0 : 1;
    return OK;
}
