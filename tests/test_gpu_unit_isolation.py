"""A step's result depends on its own sequence only.  Non-finite keys and values in the next unit's new tokens, and in
the cache rows behind p0 (nobody's), leave every other unit's output bit for bit as it is with finite ones there: a
tile of new tokens that is no multiple of the copies' 8 or 128 rows ends inside the next unit's tokens, and the last
granule of the past in rows that were never written; both get weight 0, and 0 x NaN is NaN.

Every kernel that serves ragged steps: the transposed decode kernel (at most 32 rows per KV head), the padded one (33
to 128 rows of batches that fill the SMs; rows behind p0 are a stated precondition of it), the prefill kernel, the
general one."""
import pytest

from paper_2502_13542_b200 import workloads as wl

pytestmark = pytest.mark.gpu

CASES = [  # dtype, q heads, kv heads, units, new tokens, past, page tokens, rows behind p0 are poisoned as well
    ("bf16", 32, 8, 3, 1, 1003, 16, True), ("bf16", 32, 8, 3, 1, 1008, 16, True), ("bf16", 32, 8, 3, 5, 641, 16, True),
    ("bf16", 32, 8, 18, 8, 777, 16, True), ("bf16", 8, 8, 3, 17, 901, 32, True), ("bf16", 64, 8, 2, 2, 1151, 128, True),
    ("bf16", 24, 8, 3, 3, 127, 64, True), ("bf16", 32, 8, 20, 3, 15, 16, True), ("bf16", 32, 8, 40, 1, 529, 16, True),
    ("bf16", 32, 8, 12, 9, 700, 16, False), ("bf16", 32, 8, 12, 31, 700, 16, False), ("bf16", 8, 8, 11, 40, 1024, 16, False),
    ("bf16", 32, 8, 3, 33, 1003, 16, True), ("bf16", 7, 1, 2, 51, 999, 32, True), ("f32", 8, 2, 3, 5, 801, 16, True),
]


@pytest.mark.parametrize("dtype,hq,hkv,units,nt,past,page,tail", CASES)
def test_a_neighbour_that_is_not_finite_changes_nothing(dtype, hq, hkv, units, nt, past, page, tail):
    import torch
    from paper_2502_13542_b200 import binding as B
    spec = wl.llama3_8b_layer().replace(n_q_heads=hq, n_kv_heads=hkv, page_tokens=page, k_blocks=3, cap_blocks=3, dtype=dtype,
                                        context=past + nt, n_local_prev=256)
    per_seq = -(-(past + nt) // page) + 1
    table = torch.randperm(units * per_seq, dtype=torch.int32).reshape(units, per_seq)
    kw = dict(n_phys_pages=units * per_seq, max_pages=per_seq)
    cfg = B.make_config(spec, **kw)
    st = B.RetrievalState(cfg, n_seq=units, page_table=table)
    gen = torch.Generator(device="cuda").manual_seed(nt + past)

    def rnd(n, h):
        return torch.randn(units, n, h, 128, device="cuda", generator=gen).to(cfg.torch_dtype)

    big = B.make_config(spec.replace(window=max(past, 512)), **kw)
    st.set_positions([0] * units)
    B.append_window(big, st.batch, rnd(past, hkv), rnd(past, hkv), past, st.pos0, st.k_pages, st.v_pages, st.page_table, st.repr_k,
                    st.repr_inv_norm, st.status)
    st.set_positions([past] * units)
    n = B.n_candidates(cfg, past)
    c = min(3, n)
    if c:
        st.sel_idx[:, :, :c] = torch.arange(c, dtype=torch.int32, device="cuda")
    st.sel_count.fill_(c)
    q, k, v = rnd(nt, hq), rnd(nt, hkv), rnd(nt, hkv)

    def run(k, v):
        out = torch.full((units, nt, hq, 128), float("nan"), device="cuda", dtype=cfg.torch_dtype)
        lse = torch.full((units, hq, nt), float("nan"), device="cuda")
        B.retrieval_attention(cfg, st.batch, q, k, v, nt, st.k_pages, st.v_pages, st.page_table, st.pos0, st.sel_idx,
                              st.sel_count, out, lse, st.status)
        torch.cuda.synchronize()
        assert int(st.status.item()) == 0
        return out, lse

    want, want_lse = run(k, v)
    assert torch.isfinite(want).all() and torch.isfinite(want_lse).all()
    if tail and past % page:
        for u in range(units):
            rows = (0, int(table[u, past // page]), slice(None), slice(past % page, None))
            st.k_pages[rows] = float("nan")
            st.v_pages[rows] = float("inf") if u % 2 else float("nan")
    bad = torch.arange(units, device="cuda") % 2 == 1      # every second unit
    k[bad, 0] = float("nan")
    v[bad] = float("nan")
    v[bad, :1] = float("inf")
    got, lse = run(k, v)
    assert torch.equal(got[~bad], want[~bad]) and torch.equal(lse[~bad], want_lse[~bad])
