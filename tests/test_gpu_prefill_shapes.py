"""The two-set prefill kernel against the general fp32 kernel at the sizes where it can go wrong: steps that
fill no whole query tile (one token more or less than a tile, than two), steps whose last key tile runs into
the next unit's tokens, group sizes that do not divide 128, a second query tile without tokens, key streams cut
over 1, 2, 4 and 8 CTAs, every page size, pasts off the page grid with NaN in the cache rows behind them.

Bounds: P carries 16 significant bits (|v| <= 45 here: 45 * 2^-17 = 4e-4) or, for whole tiles and an even group
size, 11 (45 * 2^-12 = 1.1e-2); the scores differ by the order of their fp32 sums."""
import pytest

from paper_2502_13542_b200 import workloads as wl

pytestmark = pytest.mark.gpu

CASES = [  # q heads, kv heads, units, step tokens, past, page tokens
    (32, 8, 1, 33, 700, 16), (32, 8, 2, 63, 1024, 16), (32, 8, 3, 65, 2048 + 21, 16), (32, 8, 1, 129, 0, 16),
    (32, 8, 2, 127, 130, 32), (32, 8, 1, 511, 3000, 128), (32, 8, 5, 97, 1500, 64), (32, 8, 1, 256, 2048, 16),
    (24, 8, 2, 200, 999, 16), (10, 2, 1, 90, 1777, 16), (7, 1, 2, 51, 640, 16), (8, 8, 1, 300, 1234, 16),
    (8, 8, 2, 128, 1024, 16), (16, 2, 1, 128, 2048, 16), (16, 2, 1, 17, 2048, 16), (64, 8, 2, 384, 1111, 16),
    (2, 1, 1, 65, 4000, 16),
]


# A local past of several key tiles whose last one is ragged, in streams that are not cut and that are; with 16-token
# pages also steps of 33 to 128 rows per KV head (a cut stream takes the prefill kernel).
LOCAL_CASES = [  # ..., local past
    (32, 8, 5, 97, 1501, 16, 512), (32, 8, 10, 40, 2003, 16, 1024), (8, 8, 6, 200, 1777, 32, 896), (7, 1, 2, 51, 1640, 16, 640),
    (64, 8, 20, 33, 1333, 64, 768), (32, 8, 1, 9, 3001, 16, 512), (32, 8, 5, 16, 1500, 16, 512), (64, 8, 3, 16, 1777, 16, 256),
]


# More streams than SMs: behind the first 148 (or 296) at most 74 are left, whose query tiles take a CTA each from 1,024 keys on
# (not one tile of 40 tokens, nor 300 and 430 keys; 300 tokens at G = 1 are three tiles, a last pair of one); both forms of P.
ROUND_CASES = [(8, 8, 20, 129, 1501, 16, 512), (16, 8, 20, 128, 1408, 16, 512), (8, 8, 27, 40, 2003, 32, 1024), (8, 8, 28, 40, 2003, 32, 1024),
               (1, 1, 149, 200, 999, 16, 256), (16, 8, 37, 256, 1152, 16, 256), (24, 8, 46, 41, 801, 16, 0), (8, 8, 20, 300, 0, 16, 512), (8, 8, 10, 300, 130, 16, 512),
               (8, 8, 10, 300, 1500, 16, 512), (24, 8, 46, 83, 1701, 32, 256), (16, 8, 28, 200, 1777, 16, 0)]


@pytest.mark.parametrize("hq,hkv,units,nt,past,page,local", ROUND_CASES)
def test_thin_last_round(hq, hkv, units, nt, past, page, local):
    check(hq, hkv, units, nt, past, page, local, bf16=True)      # (fp32 results of ragged steps are the general kernel's)


def test_thin_last_round_of_whole_tiles_fp32_results():
    check(16, 8, 20, 256, 1408, 16, 512)


@pytest.mark.parametrize("hq,hkv,units,layers,nt,past,f32", [
    (8, 8, 20, 1, 129, 1501, False), (16, 8, 20, 2, 256, 1408, False), (16, 8, 20, 1, 256, 1408, True), (32, 8, 20, 2, 60, 2200, False),
    (8, 8, 20, 2, 300, 1200, False), (32, 8, 8, 1, 500, 900, False), (32, 8, 8, 4, 512, 900, False), (24, 8, 44, 2, 83, 0, False), (24, 8, 44, 2, 83, 1700, False)])
def test_results_do_not_depend_on_the_place(hq, hkv, units, layers, nt, past, f32):
    """Equal sequences (and layers) in one call of more streams than SMs: the bits of every one are those of the first, and of a
    call of half of them, whose streams are fewer but not cut either (75 and more)."""
    import torch
    from paper_2502_13542_b200 import binding as B
    spec = wl.llama3_8b_layer().replace(n_layers=layers, n_q_heads=hq, n_kv_heads=hkv, k_blocks=9, cap_blocks=9, context=past + nt)
    per = -(-(past + nt) // 16) + 1
    cfg = B.make_config(spec, out_dtype=B.F32 if f32 else B.BF16, n_phys_pages=per, max_pages=per)
    gen = torch.Generator(device="cuda").manual_seed(nt)

    def rnd(*shape):
        x = torch.randn(*shape, 128, device="cuda", generator=gen)
        x[..., :3] *= 10.0
        return x.to(torch.bfloat16)

    table = torch.randperm(per, dtype=torch.int32)
    pages = [rnd(1, per, hkv, 16).expand(layers, -1, -1, -1, -1).contiguous() for _ in range(2)]
    step = [rnd(1, nt, h) for h in (hq, hkv, hkv)]
    n = B.n_candidates(cfg, past) if past > spec.n_init else 0
    c = min(9, n)
    sel = torch.stack([torch.randperm(n)[:c].sort().values for _ in range(hkv)]).to(torch.int32)

    def run(units):
        st = B.RetrievalState(cfg, n_seq=units // layers, n_layers=layers, page_table=table.repeat(units // layers, 1), shared_pages=pages)
        st.set_positions([past])
        st.sel_idx[:, :, :c] = sel.cuda()
        st.sel_count.fill_(c)
        q, k, v = (x.expand(units, -1, -1, -1).contiguous() for x in step)
        out = torch.full(q.shape, float("nan"), dtype=cfg.torch_out_dtype, device="cuda")
        lse = torch.full((units, hq, nt), float("nan"), device="cuda")
        B.retrieval_attention(cfg, st.batch, q, k, v, nt, st.k_pages, st.v_pages, st.page_table, st.pos0, st.sel_idx, st.sel_count,
                              out, lse, st.status)
        torch.cuda.synchronize()
        assert int(st.status.item()) == 0 and torch.isfinite(out).all()
        return out, lse

    small, small_lse = run(units // 2)
    out, lse = run(units)
    for u in range(units):
        assert torch.equal(out[u], small[0]) and torch.equal(lse[u], small_lse[0]), u


@pytest.mark.parametrize("hq,hkv,units,nt,past,page,local", LOCAL_CASES)
def test_long_ragged_local_past(hq, hkv, units, nt, past, page, local):
    check(hq, hkv, units, nt, past, page, local)


@pytest.mark.parametrize("hq,hkv,units,nt,past,page", CASES)
def test_prefill_shapes_match_general_kernel(hq, hkv, units, nt, past, page):
    check(hq, hkv, units, nt, past, page, None)


def check(hq, hkv, units, nt, past, page, local, bf16=False):
    import torch
    assert torch.cuda.is_available()
    from paper_2502_13542_b200 import binding as B
    spec = wl.llama3_8b_layer().replace(n_q_heads=hq, n_kv_heads=hkv, page_tokens=page, k_blocks=5, cap_blocks=5,
                                        context=past + nt)
    if local is not None:
        spec = spec.replace(n_local_prev=local)
    per_seq = -(-(past + nt) // page) + 1
    table = torch.randperm(units * per_seq, dtype=torch.int32).reshape(units, per_seq)
    kw = dict(out_dtype=B.BF16 if bf16 else B.F32, n_phys_pages=units * per_seq, max_pages=per_seq)
    cfg = B.make_config(spec, **kw)
    st = B.RetrievalState(cfg, n_seq=units, page_table=table)
    gen = torch.Generator(device="cuda").manual_seed(nt + past)

    def rnd(n, h):
        x = torch.randn(units, n, h, 128, device="cuda", generator=gen)
        x[..., :3] *= 10.0
        return x.to(torch.bfloat16)

    st.set_positions([0] * units)
    big = B.make_config(spec.replace(window=max(past, 512)), **kw)
    if past:
        B.append_window(big, st.batch, rnd(past, hkv), rnd(past, hkv), past, st.pos0, st.k_pages, st.v_pages, st.page_table,
                        st.repr_k, st.repr_inv_norm, st.status)
        lp, t0 = past // page, past % page
        for s in range(units):                     # what lies behind the past is nobody's: it must not matter
            if t0:
                st.k_pages[0, int(table[s, lp]), :, t0:] = float("nan")
                st.v_pages[0, int(table[s, lp]), :, t0:] = float("nan")
    st.set_positions([past] * units)
    n = B.n_candidates(cfg, past) if past > spec.n_init else 0
    c = min(5, n)
    for u in range(units):
        for g in range(hkv):
            st.sel_idx[u, g, :c] = torch.randperm(n)[:c].sort().values.to(torch.int32).cuda() if c else 0
    st.sel_count.fill_(c)
    q, k, v = rnd(nt, hq), rnd(nt, hkv), rnd(nt, hkv)

    def run(kernel):
        out = torch.full((units, nt, hq, 128), float("nan"), dtype=torch.bfloat16 if bf16 else torch.float32, device="cuda")
        lse = torch.full((units, hq, nt), float("nan"), device="cuda")
        B.retrieval_attention(B.make_config(spec, attention_kernel=kernel, **kw), st.batch, q, k, v, nt, st.k_pages, st.v_pages,
                              st.page_table, st.pos0, st.sel_idx, st.sel_count, out, lse, st.status)
        torch.cuda.synchronize()
        assert int(st.status.item()) == 0
        return out, lse

    want, want_lse = run(B.ATTN_GENERAL)
    got, lse = run(B.ATTN_AUTO)
    again, _ = run(B.ATTN_AUTO)
    assert torch.equal(got, again)
    fp16 = nt % 128 == 0 and (hq // hkv) % 2 == 0
    err = (got.float() - want.float()).abs()
    if bf16:                                       # either result is rounded by half a spacing, 2^-8 of its size at most
        err = (err - 2.0 ** -7 * want.float().abs()).clamp(min=0)
    assert err.max().item() < (2e-2 if fp16 else 2e-3)
    assert err.mean().item() < (2e-3 if fp16 else 1e-4)
    assert (lse - want_lse).abs().max().item() < 2e-3
