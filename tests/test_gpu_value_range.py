"""Values up to 2^80 with two-term weights: a row's scores grow by 2^50 (in powers of two) after its first tile, so
weights taken against the first tile's maximum would bring the products to 2^130, beyond fp32.  With weights of at
most 2^32 and 2^11 keys the sums stay below 2^123.  Against the general fp32 kernel, bf16 results: half an ulp each (2^-8),
relative to the row's largest value."""
import pytest

from paper_2502_13542_b200 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("hq,hkv,units,nt", [(32, 8, 1, 1), (32, 8, 40, 1), (32, 8, 1, 5), (32, 8, 20, 3), (32, 8, 12, 9),
                                             (32, 8, 2, 65), (8, 8, 1, 128), (24, 8, 6, 300)])
@pytest.mark.parametrize("growth", [31.0, 50.0, 70.0])
def test_large_values(hq, hkv, units, nt, growth):
    import torch
    from paper_2502_13542_b200 import binding as B
    past = 1500
    spec = wl.llama3_8b_layer().replace(n_q_heads=hq, n_kv_heads=hkv, k_blocks=4, cap_blocks=4, context=past + nt, n_local_prev=512)
    per_seq = -(-(past + nt) // 16) + 1
    kw = dict(n_phys_pages=units * per_seq, max_pages=per_seq)
    st = B.RetrievalState(B.make_config(spec, **kw), n_seq=units,
                          page_table=torch.arange(units * per_seq, dtype=torch.int32).reshape(units, per_seq))
    gen = torch.Generator(device="cuda").manual_seed(nt)

    def rnd(n, h):
        return torch.randn(units, n, h, 128, device="cuda", generator=gen)

    def keys(n, first):                       # channel 0 carries the growth: nothing for tokens below 128
        x = 0.1 * rnd(n, hkv)
        x[..., 0] = torch.where(torch.arange(first, first + n, device="cuda") < 128, 0.0, growth / 16 / 0.127517)[None, :, None]
        return x.to(torch.bfloat16)

    def values(n):
        return (rnd(n, hkv) * 2.0 ** 80).to(torch.bfloat16)

    big = B.make_config(spec.replace(window=past), **kw)
    B.append_window(big, st.batch, keys(past, 0), values(past), past, st.pos0, st.k_pages, st.v_pages, st.page_table, st.repr_k,
                    st.repr_inv_norm, st.status)
    st.set_positions([past] * units)
    n = B.n_candidates(st.cfg, past)
    st.sel_idx[:] = torch.arange(n - 4, n, dtype=torch.int32, device="cuda")
    st.sel_count.fill_(4)
    q = rnd(nt, hq)
    q[..., 0] = 16.0
    q, k, v = q.to(torch.bfloat16), keys(nt, past), values(nt)
    res = []
    for kernel in (B.ATTN_GENERAL, B.ATTN_AUTO):
        cfg = B.make_config(spec, attention_kernel=kernel, **kw)
        out = torch.zeros(q.shape, device="cuda", dtype=torch.bfloat16)
        B.retrieval_attention(cfg, st.batch, q, k, v, nt, st.k_pages, st.v_pages, st.page_table, st.pos0, st.sel_idx,
                              st.sel_count, out, None, st.status)
        torch.cuda.synchronize()
        assert int(st.status.item()) == 0
        res.append(out.float() * 2.0 ** -80)
    want, got = res
    assert torch.isfinite(got).all()
    assert ((got - want).abs() / want.abs().amax(-1, keepdim=True)).max().item() <= 2 * 2.0 ** -8
