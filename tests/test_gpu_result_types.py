"""The same attention with bf16 and with fp32 results.

bf16: the tensor-core kernels against the general fp32 kernel, at the shapes of the decode and prefill tests.  Bound:
half a bf16 ulp of the result (8 significant bits: 2^-8 relative at most, on average below 2^-9) on top of what the weights' 16 bits (11 for whole tiles and an even
group) and the scores' other summation order give, as in those tests.

fp32: steps whose weights were always fp32 ones have them still: the chosen kernel is no further from fp64 than the
general one, also where the scores lie close together and nothing but the weights' rounding is left."""
import pytest

from paper_2502_13542_b200 import workloads as wl
from tests.test_gpu_decode_shapes import CASES as DECODE
from tests.test_gpu_prefill_shapes import CASES as PREFILL, LOCAL_CASES

pytestmark = pytest.mark.gpu

SHAPES = ([(hq, hkv, u, nt, past, page, 256, late) for hq, hkv, u, nt, past, page, _, late in DECODE]
          + [(*c, 0, False) for c in PREFILL] + [(*c, False) for c in LOCAL_CASES])


class Step:
    def __init__(self, hq, hkv, units, nt, past, page, local, late=False, scale=1.0):
        import torch
        from paper_2502_13542_b200 import binding as B
        self.torch, self.B = torch, B
        self.spec = spec = wl.llama3_8b_layer().replace(n_q_heads=hq, n_kv_heads=hkv, page_tokens=page, k_blocks=5, cap_blocks=5,
                                                        context=past + nt, n_local_prev=local)
        per_seq = -(-(past + nt) // page) + 1
        self.kw = dict(n_phys_pages=units * per_seq, max_pages=per_seq)
        table = torch.randperm(units * per_seq, dtype=torch.int32).reshape(units, per_seq)
        self.st = st = B.RetrievalState(B.make_config(spec, **self.kw), n_seq=units, page_table=table)
        gen = torch.Generator(device="cuda").manual_seed(nt + past)

        def rnd(n, h, s=1.0):
            x = torch.randn(units, n, h, 128, device="cuda", generator=gen) * s
            x[..., :3] *= 10.0
            return x.to(torch.bfloat16)

        self.nt, self.past, self.units, self.hq, self.hkv = nt, past, units, hq, hkv
        self.pk, self.pv = rnd(max(past, 1), hkv), rnd(max(past, 1), hkv)
        if past:
            if late:
                self.pk = (self.pk.float() * torch.linspace(0.2, 6.0, past, device="cuda")[None, :, None, None]).to(torch.bfloat16)
            big = B.make_config(spec.replace(window=max(past, 512)), **self.kw)
            st.set_positions([0] * units)
            B.append_window(big, st.batch, self.pk, self.pv, past, st.pos0, st.k_pages, st.v_pages, st.page_table, st.repr_k,
                            st.repr_inv_norm, st.status)
        st.set_positions([past] * units)
        self.n = B.n_candidates(st.cfg, past) if past > spec.n_init else 0
        c = min(5, self.n)
        self.chosen = [[torch.randperm(self.n)[:c].sort().values for _ in range(hkv)] for _ in range(units)]
        for u in range(units):
            for g in range(hkv):
                st.sel_idx[u, g, :c] = self.chosen[u][g].to(torch.int32).cuda()
        st.sel_count.fill_(c)
        self.q, self.k, self.v = rnd(nt, hq, scale), rnd(nt, hkv), rnd(nt, hkv)

    def run(self, kernel, out_dtype):
        torch, B, st = self.torch, self.B, self.st
        cfg = B.make_config(self.spec, attention_kernel=kernel, out_dtype=out_dtype, **self.kw)
        out = torch.full(self.q.shape, float("nan"), device="cuda", dtype=torch.float32 if out_dtype == B.F32 else torch.bfloat16)
        lse = torch.full((self.units, self.hq, self.nt), float("nan"), device="cuda")
        B.retrieval_attention(cfg, st.batch, self.q, self.k, self.v, self.nt, st.k_pages, st.v_pages, st.page_table, st.pos0,
                              st.sel_idx, st.sel_count, out, lse, st.status)
        torch.cuda.synchronize()
        assert int(st.status.item()) == 0
        return out, lse

    def fp64(self):
        torch, spec, G = self.torch, self.spec, self.hq // self.hkv
        want = torch.zeros(self.q.shape, dtype=torch.float64, device="cuda")
        for u in range(self.units):
            for g in range(self.hkv):
                tok = torch.arange(self.past)
                if self.past > spec.n_init:
                    blocks = spec.n_init + self.chosen[u][g][:, None] * spec.block + torch.arange(spec.block)
                    tok = torch.cat([torch.arange(spec.n_init), blocks.reshape(-1),
                                     torch.arange(spec.n_init + self.n * spec.block, self.past)])
                K = torch.cat([self.pk[u, tok.cuda(), g], self.k[u, :, g]]).double()
                V = torch.cat([self.pv[u, tok.cuda(), g], self.v[u, :, g]]).double()
                s = torch.einsum("jhd,kd->hjk", self.q[u, :, g * G:(g + 1) * G].double(), K) / 128 ** 0.5
                mask = torch.ones(self.nt, K.shape[0], dtype=torch.bool, device="cuda")
                mask[:, len(tok):] = torch.tril(mask[:, len(tok):])
                p = torch.softmax(s.masked_fill(~mask, -float("inf")), -1)
                want[u, :, g * G:(g + 1) * G] = torch.einsum("hjk,kd->jhd", p, V)
        return want


@pytest.mark.parametrize("hq,hkv,units,nt,past,page,local,late", SHAPES)
def test_bf16_results_match_the_general_kernel(hq, hkv, units, nt, past, page, local, late):
    step = Step(hq, hkv, units, nt, past, page, local, late)
    want, want_lse = step.run(step.B.ATTN_GENERAL, step.B.F32)
    got, lse = step.run(step.B.ATTN_AUTO, step.B.BF16)
    again, _ = step.run(step.B.ATTN_AUTO, step.B.BF16)
    assert step.torch.equal(got, again)
    fp16 = nt % 128 == 0 and (hq // hkv) % 2 == 0
    err = (got.float() - want).abs()
    assert (err - want.abs() * 2.0 ** -8).max().item() < (2e-2 if fp16 else 2e-3)
    assert err.mean().item() < (2e-3 if fp16 else 1e-4) + want.abs().mean().item() * 2.0 ** -9
    assert (lse - want_lse).abs().max().item() < 2e-3


@pytest.mark.parametrize("scale", [1.0, 0.03])
@pytest.mark.parametrize("hq,hkv,units,nt,past,page", [(32, 8, 1, 511, 3000, 16), (32, 8, 2, 97, 1500, 64), (7, 1, 2, 51, 640, 16),
                                                       (64, 8, 2, 1, 1024, 32), (24, 8, 1, 1, 900, 16), (10, 2, 3, 3, 1333, 16),
                                                       (7, 1, 2, 130, 2640, 32)])
def test_fp32_results_keep_fp32_weights(hq, hkv, units, nt, past, page, scale):
    step = Step(hq, hkv, units, nt, past, page, 256, scale=scale)
    want = step.fp64()

    def off(kernel):
        return ((step.run(kernel, step.B.F32)[0].double() - want).norm() / want.norm()).item()

    assert off(step.B.ATTN_AUTO) <= off(step.B.ATTN_GENERAL)
