"""Selection of the c highest scores at the edges of its counting: one candidate, one per thread and one more, what the
registers hold (1,024) and one more, counts of 1, half and all but one, ties across the cut (lowest index first), NaN
scores (last), negative zeros; for a single layer (fused chain) and for batched layers.  Exact."""
import pytest

from paper_2502_13542_b200 import workloads as wl

pytestmark = pytest.mark.gpu


def pick(row, c):
    """Indices of the c highest scores, equal ones by lower index, NaN last, ascending."""
    key = [(-(float("-inf") if x != x else x + 0.0), i) for i, x in enumerate(row)]
    return sorted(i for _, i in sorted(key)[:c])


@pytest.mark.parametrize("layers", [1, 2])
@pytest.mark.parametrize("n", [1, 2, 31, 255, 256, 257, 1023, 1024, 1025, 3000])
@pytest.mark.parametrize("kind", ["random", "ties", "nan"])
def test_selection_edges(layers, n, kind):
    import torch
    from paper_2502_13542_b200 import binding as B
    L = 3
    for c in sorted({1, max(1, n // 2), max(1, n - 1)}):
        spec = wl.llama3_8b_layer().replace(n_layers=L, k_blocks=c, cap_blocks=c, n_kv_heads=8)
        cfg = B.make_config(spec, n_cap=n, beta=1.0)
        gen = torch.Generator(device="cuda").manual_seed(n + c)
        U = 2 * layers
        scores = torch.rand(U, 8, n, device="cuda", generator=gen) * 2 - 1
        if kind == "ties":
            scores = (scores * 3).round() / 3                    # few values, negative zeros among them
        if kind == "nan":
            scores[torch.rand(U, 8, n, device="cuda", generator=gen) < 0.3] = float("nan")
        theta = torch.ones(U, 8, device="cuda")
        n_cand = torch.full((2,), n, dtype=torch.int32, device="cuda")
        state = torch.zeros(2, 1 + 2 * L, dtype=torch.float64, device="cuda")
        sel = torch.full((U, 8, c), -7, dtype=torch.int32, device="cuda")
        cnt = torch.zeros(U, dtype=torch.int32, device="cuda")
        B.select_cutoff(cfg, B.Batch(2, layers, 0), scores, theta, n_cand, state, sel, cnt)
        torch.cuda.synchronize()
        counts = cnt.tolist()
        host = scores.cpu().tolist()
        got = sel.cpu().tolist()
        for u in range(U):
            k = counts[u]
            assert 1 <= k <= c
            for g in range(0, 8, 3):
                assert got[u][g] == pick(host[u][g], k) + [-1] * (c - k), (u, g, k)


@pytest.mark.parametrize("seqs", [1, 12])            # up to 9 sequences of 8 KV heads take a thread per candidate up to 512
@pytest.mark.parametrize("n", [5, 32, 33, 129, 256, 257, 384, 385, 511, 513, 1500])
def test_density_and_selection_of_one_layer(seqs, n):
    """Density, count and set of one layer from its own scores: lengths at the edges of a warp, of the ranked range and of
    the key threads.  The density is a sum of n fp32 terms about 1: n * 2^-24 of it, and a few roundings of exp and ln."""
    import torch
    from paper_2502_13542_b200 import binding as B
    L, c, beta = 3, min(n, 40), 8.0
    spec = wl.llama3_8b_layer().replace(n_layers=L, k_blocks=c, cap_blocks=c, n_kv_heads=8)
    cfg = B.make_config(spec, n_cap=n, beta=beta)
    gen = torch.Generator(device="cuda").manual_seed(n)
    table = torch.randn(seqs, 8, n, 4, 128, device="cuda", generator=gen).bfloat16()
    norms = 1.0 / table.float().norm(dim=-1)
    probe = torch.randn(seqs, 8, 128, device="cuda", generator=gen)
    n_cand = torch.full((seqs,), n, dtype=torch.int32, device="cuda")
    n_cand[-1] = max(1, n - 3)
    state = torch.zeros(seqs, 1 + 2 * L, dtype=torch.float64, device="cuda")
    scores, theta = torch.zeros(seqs, 8, n, device="cuda"), torch.zeros(seqs, 8, device="cuda")
    sel = torch.full((seqs, 8, c), -7, dtype=torch.int32, device="cuda")
    cnt = torch.zeros(seqs, dtype=torch.int32, device="cuda")
    for layer in range(L):
        B.score_select(cfg, B.Batch(seqs, 1, layer), probe, table, norms, n_cand, state, scores, theta, sel, cnt)
        torch.cuda.synchronize()
        for u in range(seqs):
            m = int(n_cand[u])
            x = beta * scores[u, :, :m].double()
            w = torch.softmax(x, dim=-1)
            want = torch.special.entr(w).sum(-1)
            assert torch.allclose(theta[u].double(), want, rtol=(n + 16) * 2.0 ** -24, atol=1e-6)
            k = int(cnt[u])
            assert 1 <= k <= min(c, m)
            for g in range(8):
                assert sel[u, g].tolist() == pick(scores[u, g, :m].tolist(), k) + [-1] * (c - k)


@pytest.mark.parametrize("n", [256, 257, 300, 511, 512, 513, 769, 1023, 1500])
def test_density_does_not_depend_on_the_batch(n):
    """A sequence's density, count, set and budget are the same bits alone, beside 8 others and beside 11 others (up to 9
    sequences of 8 heads have 512 key threads where there are more than 256 candidates, more of them have 256)."""
    import torch
    from paper_2502_13542_b200 import binding as B
    L, c = 2, 24
    spec = wl.llama3_8b_layer().replace(n_layers=L, k_blocks=c, cap_blocks=2 * c, n_kv_heads=8)
    cfg = B.make_config(spec, n_cap=n, beta=6.0)
    gen = torch.Generator(device="cuda").manual_seed(n)
    table = torch.randn(12, 8, n, 4, 128, device="cuda", generator=gen).bfloat16()
    norms = 1.0 / table.float().norm(dim=-1)
    probe = torch.randn(12, 8, 128, device="cuda", generator=gen)
    n_cand = torch.full((12,), n, dtype=torch.int32, device="cuda")
    n_cand[1] = n - 7

    def run(seqs):
        scores, theta = torch.zeros(seqs, 8, n, device="cuda"), torch.zeros(seqs, 8, device="cuda")
        sel, cnt = torch.zeros(seqs, 8, 2 * c, dtype=torch.int32, device="cuda"), torch.zeros(seqs, dtype=torch.int32, device="cuda")
        state = torch.zeros(seqs, 1 + 2 * L, dtype=torch.float64, device="cuda")
        for layer in range(L):
            B.score_select(cfg, B.Batch(seqs, 1, layer), probe[:seqs].contiguous(), table[:seqs].contiguous(),
                           norms[:seqs].contiguous(), n_cand[:seqs].contiguous(), state, scores, theta, sel, cnt)
        torch.cuda.synchronize()
        return scores, theta, sel, cnt, state

    many = run(12)
    for seqs in (1, 9):
        for i, (x, y) in enumerate(zip(run(seqs), many)):
            assert torch.equal(x, y[:seqs]), (seqs, i)


@pytest.mark.parametrize("dtype,D,r", [("bf16", 128, 4), ("bf16", 64, 8), ("f32", 128, 2), ("f32", 64, 4)])
@pytest.mark.parametrize("n", [0, 1, 3, 31, 32, 33, 65, 127, 128, 129])
def test_scores_taken_by_the_selection(dtype, D, r, n):
    """Small tables of 1 KiB blocks: a step that takes its probe from its own window (up to 128 candidates and 16 heads) has
    the scores taken by the selection; the bits are those of score_select, which takes two kernels.  (At 129 rows both do.)"""
    import torch
    from paper_2502_13542_b200 import binding as B
    L, c, nt, seqs = 2, 7, 3, 2
    spec = wl.llama3_8b_layer().replace(n_layers=L, k_blocks=c, cap_blocks=c, n_q_heads=8, n_kv_heads=8, head_dim=D, dtype=dtype,
                                        n_repr=r, window=16)
    cap = max(n, 1)
    kw = dict(n_cap=cap, beta=4.0, max_pages=2, n_phys_pages=2)
    cfg = B.make_config(spec, **kw)
    gen = torch.Generator(device="cuda").manual_seed(n + D)
    rnd = lambda *shape: torch.randn(*shape, device="cuda", generator=gen)      # noqa: E731
    table = rnd(seqs, 8, cap, r, D).to(cfg.torch_dtype)
    norms = 1.0 / table.float().norm(dim=-1)
    q = rnd(seqs, nt, 8, D).to(cfg.torch_dtype)
    kv = torch.zeros_like(q)
    out = torch.empty_like(q)

    def run(counts, q=q, cfg=cfg):
        """The step of two layers, and score_select on the probes it left; results and status bits of both."""
        got, want, bits = [], [], [0, 0]
        state = torch.zeros(seqs, 1 + 2 * L, dtype=torch.float64, device="cuda")
        other = state.clone()
        for layer in range(L):
            st = B.RetrievalState(cfg, n_seq=seqs, n_layers=1, layer0=layer)
            st.repr_k.copy_(table), st.repr_inv_norm.copy_(norms)
            st.budget_state, st.n_cand = state, torch.tensor(counts, dtype=torch.int32, device="cuda")
            st.step(q, kv, kv, out, advance=False)        # (position 0: the attention and the append see none of this)
            torch.cuda.synchronize()
            bits[0] |= int(st.status.item()) & ~B.DEV_BAD_SELECTION        # (the attention knows of no candidates)
            got += [st.scores.clone(), st.theta.clone(), st.sel_idx.clone(), st.sel_count.clone(), state.clone()]
            st.status.zero_(), st.scores.zero_(), st.theta.zero_(), st.sel_idx.fill_(-7), st.sel_count.zero_()
            B.score_select(cfg, st.batch, st.probe_kv, st.repr_k, st.repr_inv_norm, st.n_cand, other, st.scores, st.theta,
                           st.sel_idx, st.sel_count, None, st.status)
            torch.cuda.synchronize()
            bits[1] |= int(st.status.item())
            want += [st.scores, st.theta, st.sel_idx, st.sel_count, other.clone()]
        for i, (a, b) in enumerate(zip(got, want)):
            assert torch.equal(a, b), i
        return bits

    assert run([n, n // 2]) == [0, 0]
    assert run([n, cap + 1]) == [B.DEV_NCAND_CLAMPED] * 2
    zero = q.clone()
    zero[1, :, 2] = 0
    assert run([n, n], q=zero) == [B.DEV_BAD_PROBE if n else 0] * 2
    if 0 < n <= 128:                                      # the step takes the form in question: only there rows can be late
        for late, bit in ((99, 0), (8, B.DEV_TIMEOUT), (99, 0)):
            hooked = B.make_config(spec, **kw)
            hooked.test_wait_limit, hooked.test_drop_k_tile = 20000, late
            st = B.RetrievalState(hooked, n_seq=seqs)
            st.repr_k.copy_(table), st.repr_inv_norm.copy_(norms), st.n_cand.fill_(n)
            st.step(q, kv, kv, out, advance=False)
            torch.cuda.synchronize()
            assert int(st.status.item()) & B.DEV_TIMEOUT == bit


@pytest.mark.parametrize("layers", [1, 2])
def test_two_threads_with_tables_of_different_size(layers):
    """Two host threads select from tables of 5,200 and 25,600 rows (the largest): each launch asks for its own amount of
    shared memory, and neither thread's call may refuse the other's."""
    import threading
    import torch
    from paper_2502_13542_b200 import binding as B
    spec = wl.llama3_8b_layer().replace(n_layers=layers, k_blocks=16, cap_blocks=16, n_kv_heads=8)
    done, errors = [], []
    ready = threading.Barrier(2)

    def work(n):
        try:
            cfg, stream = B.make_config(spec, n_cap=n), torch.cuda.Stream()
            with torch.cuda.stream(stream):
                scores = torch.rand(layers, 8, n, device="cuda")
                theta = torch.full((layers, 8), 3.0, device="cuda")
                n_cand = torch.full((1,), n, dtype=torch.int32, device="cuda")
                state = torch.zeros(1, 1 + 2 * layers, dtype=torch.float64, device="cuda")
                sel = torch.full((layers, 8, 16), -7, dtype=torch.int32, device="cuda")
                cnt = torch.zeros(layers, dtype=torch.int32, device="cuda")
                stream.synchronize()
                ready.wait()
                for _ in range(1000):
                    B.select_cutoff(cfg, B.Batch(1, layers, 0), scores, theta, n_cand, state, sel, cnt, stream=stream)
                stream.synchronize()
            k = int(cnt[0])
            assert sel[0, 0, :k].tolist() == pick(scores[0, 0].tolist(), k)
            done.append(n)
        except Exception as e:                            # noqa: BLE001  (handed to the test's thread)
            errors.append((n, e))

    threads = [threading.Thread(target=work, args=(n,)) for n in (5200, 25600)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors and sorted(done) == [5200, 25600]
