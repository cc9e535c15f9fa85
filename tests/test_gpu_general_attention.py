"""The general fp32 attention kernel against the same sums in fp64, at the edges of its tiling: 32 rows of (token,
head) pairs per CTA and chunks of 64 keys (one row, a row more than a tile, a key more than a chunk), key streams
cut over 1 to 8 CTAs, group sizes that do not divide 32, both head sizes and cache types, a page size and a local
segment that only this kernel takes.

Bound: a score is an fp32 dot product of D terms: D u sum |q k| at worst (u = 2^-24), sqrt(D) u sum |q k| when the
roundings are independent; twice that is allowed.  The weights, and with them the output as a share of |v|, are off
by as much, on average far less."""
import pytest

from paper_2502_13542_b200 import workloads as wl

pytestmark = pytest.mark.gpu

CASES = [  # dtype, D, q heads, kv heads, units, step tokens, past, page tokens, local
    ("f32", 64, 4, 2, 1, 256, 1500, 16, 0), ("f32", 64, 4, 2, 3, 17, 129, 16, 0), ("f32", 64, 2, 2, 1, 1, 63, 16, 0),
    ("f32", 128, 8, 1, 1, 5, 2000, 16, 40), ("f32", 128, 3, 1, 2, 65, 700, 16, 0), ("f32", 64, 7, 1, 1, 33, 0, 16, 0),
    ("bf16", 64, 10, 2, 2, 129, 1000, 8, 0), ("bf16", 128, 4, 4, 9, 64, 300, 16, 24), ("f32", 64, 32, 8, 2, 128, 640, 64, 0),
]


@pytest.mark.parametrize("dtype,D,hq,hkv,units,nt,past,page,local", CASES)
def test_general_attention_against_fp64(dtype, D, hq, hkv, units, nt, past, page, local):
    import torch
    from paper_2502_13542_b200 import binding as B
    spec = wl.tiny_pr1().replace(n_q_heads=hq, n_kv_heads=hkv, head_dim=D, dtype=dtype, page_tokens=page, k_blocks=4,
                                 cap_blocks=4, context=past + nt, n_local_prev=local)
    per_seq = -(-(past + nt) // page) + 1
    table = torch.randperm(units * per_seq, dtype=torch.int32).reshape(units, per_seq)
    kw = dict(out_dtype=B.F32, n_phys_pages=units * per_seq, max_pages=per_seq, attention_kernel=B.ATTN_GENERAL)
    cfg = B.make_config(spec, **kw)
    st = B.RetrievalState(cfg, n_seq=units, page_table=table)
    gen = torch.Generator(device="cuda").manual_seed(7 * nt + past)

    def rnd(n, h):
        x = torch.randn(units, n, h, D, device="cuda", generator=gen)
        x[..., :2] *= 8.0
        return x.to(cfg.torch_dtype)

    pk, pv = rnd(max(past, 1), hkv), rnd(max(past, 1), hkv)
    if past:
        big = B.make_config(spec.replace(window=max(past, 256)), **kw)
        st.set_positions([0] * units)
        B.append_window(big, st.batch, pk, pv, past, st.pos0, st.k_pages, st.v_pages, st.page_table, st.repr_k,
                        st.repr_inv_norm, st.status)
    st.set_positions([past] * units)
    n = B.n_candidates(cfg, past) if past > spec.n_init else 0
    c = min(4, n)
    chosen = [[torch.randperm(n)[:c].sort().values for _ in range(hkv)] for _ in range(units)]
    for u in range(units):
        for g in range(hkv):
            st.sel_idx[u, g, :c] = chosen[u][g].to(torch.int32).cuda()
    st.sel_count.fill_(c)
    q, k, v = rnd(nt, hq), rnd(nt, hkv), rnd(nt, hkv)
    out = torch.full((units, nt, hq, D), float("nan"), device="cuda")
    lse = torch.full((units, hq, nt), float("nan"), device="cuda")
    B.retrieval_attention(cfg, st.batch, q, k, v, nt, st.k_pages, st.v_pages, st.page_table, st.pos0, st.sel_idx,
                          st.sel_count, out, lse, st.status)
    torch.cuda.synchronize()
    assert int(st.status.item()) == 0
    G = hq // hkv
    for u in range(units):
        for g in range(hkv):
            if past <= spec.n_init:
                tok = torch.arange(past)
            else:
                tok = torch.cat([torch.arange(spec.n_init),
                                 (spec.n_init + chosen[u][g][:, None] * spec.block + torch.arange(spec.block)).reshape(-1),
                                 torch.arange(spec.n_init + n * spec.block, past)])
            tok = tok.cuda()
            K = torch.cat([pk[u, tok, g], k[u, :, g]]).double()
            V = torch.cat([pv[u, tok, g], v[u, :, g]]).double()
            s = torch.einsum("jhd,kd->hjk", q[u, :, g * G:(g + 1) * G].double(), K) / D ** 0.5
            mask = torch.ones(nt, len(tok) + nt, dtype=torch.bool, device="cuda")
            mask[:, len(tok):] = torch.tril(mask[:, len(tok):])
            s = s.masked_fill(~mask, -float("inf"))
            want = torch.einsum("hjk,kd->jhd", torch.softmax(s, -1), V)
            size = torch.einsum("jhd,kd->hjk", q[u, :, g * G:(g + 1) * G].double().abs(), K.abs()).max().item() / D ** 0.5
            score = 2 * D ** 0.5 * 2.0 ** -24 * max(1.0, size)
            err = (out[u, :, g * G:(g + 1) * G].double() - want).abs()
            assert err.max().item() < score * V.abs().max().item()
            assert err.mean().item() < 0.01 * score * V.abs().max().item()
            assert (lse[u, g * G:(g + 1) * G].double() - torch.logsumexp(s, -1)).abs().max().item() < score + 1e-6


# The keys ahead of the selection (64 initial ones, the local past, the step's own) end on a chunk, one before and one
# behind it; fewer of them than ranks; several rows per lane group and rows past the last token.
EARLY_EDGES = [("f32", 64, 4, 2, 1, nt, past, 16, 0) for nt in (63, 64, 65) for past in (704, 705)] + [
    ("f32", 64, 4, 2, 40, 16, 832, 16, 0), ("f32", 128, 4, 1, 1, 31, 897, 16, 0), ("f32", 128, 4, 1, 1, 32, 768, 16, 0),
    ("bf16", 64, 8, 2, 1, 127, 761, 16, 8), ("bf16", 128, 2, 1, 2, 33, 831, 16, 0), ("bf16", 64, 2, 2, 1, 1, 704, 16, 0)] + [
    ("bf16", 128, hq, 2, 2, nt, past, 16, 0) for hq, nt, past in ((4, 63, 704), (4, 64, 704), (6, 65, 705), (2, 1, 769), (16, 31, 737))]


@pytest.mark.parametrize("dtype,D,hq,hkv,units,nt,past,page,local", EARLY_EDGES)
def test_keys_ahead_of_the_selection(dtype, D, hq, hkv, units, nt, past, page, local):
    test_general_attention_against_fp64(dtype, D, hq, hkv, units, nt, past, page, local)
