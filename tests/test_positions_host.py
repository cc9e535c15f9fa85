"""As many positions as sequences: a list that is longer or shorter is an error before anything is enqueued (the
kernel writes one entry of pos0 and n_cand per position), a list of one goes for every sequence.  They are set where
the state lives: in host memory, or by a launch on its own device."""
import ctypes as C

import pytest

from paper_2502_13542_b200 import build as lib_build
from paper_2502_13542_b200 import workloads as wl


@pytest.fixture(scope="module")
def B():
    lib_build.build()
    from paper_2502_13542_b200 import binding
    return binding


@pytest.mark.parametrize("n", [0, 1, 2, 4, 400])
def test_a_list_of_another_length_is_refused(B, n):
    import torch
    cfg = B.make_config(wl.tiny_pr1())
    pos0, n_cand = torch.zeros(3, dtype=torch.int64), torch.zeros(3, dtype=torch.int32)
    with pytest.raises(B.ActQKVError, match="positions for 3 sequences"):
        B.set_positions(cfg, [7] * n, pos0, n_cand)
    with pytest.raises(B.ActQKVError, match="positions for 3 sequences"):
        B.set_positions(cfg, [7] * n, torch.zeros(n, dtype=torch.int64), n_cand)


@pytest.mark.parametrize("n_seq,n_next", [(1, 2), (2, 1), (2, 3), (3, 0)])
def test_step_refuses_positions_of_another_number_of_sequences(B, n_seq, n_next):
    lib = C.CDLL(B.LIB_PATH)
    lib.actqkv_step.argtypes, lib.actqkv_step.restype = B._SIGS["actqkv_step"]
    cfg, batch, buffers = B.make_config(wl.tiny_pr1()), B.Batch(n_seq, 1, 0), B.StepBuffers()
    after = (C.c_int64 * 8)()

    def call(n):
        return lib.actqkv_step(C.byref(cfg), C.byref(batch), C.byref(buffers), 16, 1, after, n, None)

    assert call(n_next) == -3          # ahead of the first stage, which would refuse the NULL buffers
    assert call(n_seq) == -1


def test_positions_of_a_state_on_the_host(B):
    cfg = B.make_config(wl.tiny_pr1())
    st = B.RetrievalState(cfg, n_seq=3, device="cpu")
    st.set_positions([10, 700, 3000])
    assert st.pos0.tolist() == st.host_pos0 == [10, 700, 3000]
    assert st.n_cand.tolist() == [B.n_candidates(cfg, p) for p in (10, 700, 3000)]
    st.set_positions([640])
    assert st.pos0.tolist() == st.host_pos0 == [640] * 3
    for bad in ([], [1, 2], [1, 2, 3, 4]):
        with pytest.raises(B.ActQKVError):
            st.set_positions(bad)
    assert st.pos0.tolist() == st.host_pos0 == [640] * 3


def test_positions_are_set_on_the_device_of_the_state(B, monkeypatch):
    """Another device is current: the launch goes to the state's own device and its stream."""
    import contextlib
    import torch
    current, seen = [0], []

    @contextlib.contextmanager
    def device(d):
        before, current[0] = current[0], torch.device(d).index
        yield
        current[0] = before

    class Pos0:
        is_cuda, device = True, torch.device("cuda:1")

        def get_device(self):
            return 1

    monkeypatch.setattr(torch.cuda, "device", device)
    monkeypatch.setattr(torch.cuda, "current_device", lambda: current[0])
    monkeypatch.setattr(B, "set_positions", lambda *args: seen.append((current[0], args[1])))
    st = B.RetrievalState(B.make_config(wl.tiny_pr1()), n_seq=2, device="cpu")
    st.pos0 = Pos0()
    st.set_positions([3, 4])
    current[0] = 1
    st.set_positions([5, 6])
    assert seen == [(1, [3, 4]), (1, [5, 6])] and current[0] == 1


@pytest.mark.gpu
def test_positions_of_a_state():
    import torch
    from paper_2502_13542_b200 import binding as B
    cfg = B.make_config(wl.tiny_pr1())
    st = B.RetrievalState(cfg, n_seq=3)
    pool, counts = torch.full((8,), -5, dtype=torch.int64, device="cuda"), torch.full((8,), -5, dtype=torch.int32, device="cuda")
    st.pos0, st.n_cand = pool[:3], counts[:3]
    st.set_positions([400])
    assert st.host_pos0 == [400] * 3
    for bad in ([1, 2], [1, 2, 3, 4], [9] * 300, []):
        with pytest.raises(B.ActQKVError):
            st.set_positions(bad)
    torch.cuda.synchronize()
    n = B.n_candidates(cfg, 400)
    assert pool.tolist() == [400] * 3 + [-5] * 5 and counts.tolist() == [n] * 3 + [-5] * 5
    assert st.host_pos0 == [400] * 3
    st.host_pos0 = [1, 2, 3, 4]
    x = torch.zeros(3, 16, 4, 64, device="cuda")
    with pytest.raises(B.ActQKVError):
        st.step(x, x[:, :, :2].contiguous(), x[:, :, :2].contiguous(), torch.zeros_like(x))
    torch.cuda.synchronize()
    assert pool.tolist() == [400] * 3 + [-5] * 5 and int(st.stats_count.sum()) == 0


@pytest.mark.gpu
@pytest.mark.parametrize("kw", [{}, {"fused": False}, {"overlap_append": True}])
def test_a_capture_takes_no_positions(kw):
    """Their values would be frozen into the graph: refused, with nothing of the step enqueued and the capture and
    the state as they were."""
    import torch
    from paper_2502_13542_b200 import binding as B
    spec = wl.tiny_pr1()
    st = B.RetrievalState(B.make_config(spec))
    gen = torch.Generator(device="cuda").manual_seed(3)
    q, k, v = (torch.randn(1, spec.window, h, 64, device="cuda", generator=gen) for h in (4, 2, 2))
    out = torch.zeros_like(q)
    st.set_positions([640])
    st.step(q, k, v, out, advance=False, **kw)
    torch.cuda.synchronize()
    seen = st.stats_count.clone()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        with pytest.raises(B.ActQKVError):
            st.set_positions([0])
        with pytest.raises(B.ActQKVError):
            st.step(q, k, v, out, **kw)
        st.step(q, k, v, out, advance=False, **kw)
    assert st.host_pos0 == [640]
    graph.replay()
    torch.cuda.synchronize()
    assert st.pos0.tolist() == [640] and torch.equal(st.stats_count, seen + spec.window)
    assert int(st.status.item()) == 0
