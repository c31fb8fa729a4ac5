"""Octrees destroyed, re-mapped and given tables on one thread while another captures a CUDA graph in its
own mode: the capture ends well, and its replay gives what it should; and an octree's memory is
not released before the work on other streams that reads it is done."""
import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

BALL = np.array([[0.5, 0.5, 0.5, 0.2, 0.05]])


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_2605_20565_gb300 as ot
    return torch, ot


@pytest.mark.parametrize("what", ["destroy", "map_level", "mates"])
def test_another_threads_capture(env, what):
    torch, ot = env
    keep, other = (ot.ot_octree_build(BALL, 3, 6) for _ in range(2))
    ot.ot_octree_build_mates(other)
    rng = np.random.default_rng(0)
    x = [torch.as_tensor(rng.random(1000), device="cuda") for _ in range(3)]
    want = ot.ot_locate(keep, *x)
    host = torch.empty_like(want)
    torch.cuda.synchronize()
    state = {}
    started, go_on = threading.Event(), threading.Event()

    def capture():
        try:
            s = torch.cuda.Stream()
            g = torch.cuda.CUDAGraph()
            with torch.cuda.stream(s):
                g.capture_begin(capture_error_mode="thread_local")
                ot.ot_locate(keep, *x, host=host, stream=s)
                started.set()
                go_on.wait(60)
                ot.ot_locate(keep, *x, host=host, stream=s)
                g.capture_end()
            state["graph"] = g
        except Exception as e:  # noqa: BLE001
            state["error"] = e
            started.set()

    th = threading.Thread(target=capture)
    th.start()
    started.wait(60)
    try:
        if what == "destroy":
            ot.ot_octree_destroy(other)
        elif what == "map_level":
            ot.ot_octree_set_map_level(other, 4, stream=torch.cuda.Stream())
        else:
            ot.ot_octree_build_mates(other, stream=torch.cuda.Stream())
    finally:
        go_on.set()
        th.join(60)
    assert "error" not in state, state["error"]
    host.fill_(-7)
    state["graph"].replay()
    torch.cuda.synchronize()
    assert torch.equal(host, want)


def test_destroy_waits_for_other_streams(env):
    torch, ot = env
    tree = ot.ot_octree_build(BALL, 3, 6)
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        torch.cuda._sleep(200_000_000)  # about 0.1 s
        e = torch.cuda.Event()
        e.record()
    assert not e.query()
    ot.ot_octree_destroy(tree)
    assert e.query()
