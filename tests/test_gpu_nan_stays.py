"""A NaN that a row attends to comes out as NaN, in that row and in no other: in one key of the past, in one query, in
one value.  Decode steps with and without a cut key stream, the padded decode kernel, the prefill kernels."""
import pytest

from paper_2502_13542_b200 import workloads as wl

pytestmark = pytest.mark.gpu

CASES = [  # q heads, kv heads, units, new tokens, page tokens
    (32, 8, 2, 1, 16), (32, 8, 40, 1, 16), (32, 8, 2, 5, 16), (32, 8, 24, 2, 16), (64, 8, 2, 2, 32), (8, 8, 3, 17, 64),
    (32, 8, 12, 9, 16), (32, 8, 2, 65, 16), (32, 8, 2, 128, 16), (32, 8, 6, 256, 16),
]


@pytest.mark.parametrize("hq,hkv,units,nt,page", CASES)
def test_nan_stays_nan(hq, hkv, units, nt, page):
    import torch
    from paper_2502_13542_b200 import binding as B
    past, G = 1024, hq // hkv
    spec = wl.llama3_8b_layer().replace(n_q_heads=hq, n_kv_heads=hkv, page_tokens=page, k_blocks=2, cap_blocks=2,
                                        context=past + nt, n_local_prev=256)
    per_seq = -(-(past + nt) // page) + 1
    kw = dict(n_phys_pages=units * per_seq, max_pages=per_seq)
    cfg = B.make_config(spec, **kw)
    st = B.RetrievalState(cfg, n_seq=units, page_table=torch.arange(units * per_seq, dtype=torch.int32).reshape(units, per_seq))
    gen = torch.Generator(device="cuda").manual_seed(nt)

    def rnd(n, h):
        return torch.randn(units, n, h, 128, device="cuda", generator=gen).to(torch.bfloat16)

    big = B.make_config(spec.replace(window=past), **kw)
    B.append_window(big, st.batch, rnd(past, hkv), rnd(past, hkv), past, st.pos0, st.k_pages, st.v_pages, st.page_table, st.repr_k,
                    st.repr_inv_norm, st.status)
    st.set_positions([past] * units)
    st.sel_idx[:] = torch.arange(2, dtype=torch.int32, device="cuda")
    st.sel_count.fill_(2)
    q, k, v = rnd(nt, hq), rnd(nt, hkv), rnd(nt, hkv)

    def rows_with_nan():
        out = torch.zeros(units, nt, hq, 128, device="cuda", dtype=torch.bfloat16)
        lse = torch.zeros(units, hq, nt, device="cuda")
        B.retrieval_attention(cfg, st.batch, q, k, v, nt, st.k_pages, st.v_pages, st.page_table, st.pos0, st.sel_idx,
                              st.sel_count, out, lse, st.status)
        torch.cuda.synchronize()
        assert int(st.status.item()) == 0
        return out.isnan().any(-1), out.isnan().all(-1)

    none = torch.zeros(units, nt, hq, dtype=torch.bool, device="cuda")
    any_, _ = rows_with_nan()
    assert torch.equal(any_, none)
    u, g = units - 1, hkv - 1
    heads = slice(g * G, (g + 1) * G)
    for tok in (3, past - 1):                              # an initial and a local token
        at = (0, u * per_seq + tok // page, g, tok % page, 7)
        keep = st.k_pages[at].clone()
        st.k_pages[at] = float("nan")
        any_, all_ = rows_with_nan()
        st.k_pages[at] = keep
        want = none.clone()
        want[u, :, heads] = True
        assert torch.equal(any_, want) and torch.equal(all_, want), f"key {tok}"
    q[0, nt - 1, 1, 5] = float("nan")
    any_, all_ = rows_with_nan()
    want = none.clone()
    want[0, nt - 1, 1] = True
    assert torch.equal(any_, want) and torch.equal(all_, want), "query"
    q[0, nt - 1, 1, 5] = 0.0
    st.v_pages[0, 0, 0, 9, 11] = float("nan")
    any_, all_ = rows_with_nan()
    want = none.clone()
    want[0, :, :G] = True
    assert torch.equal(any_, want) and not all_.any(), "value"
