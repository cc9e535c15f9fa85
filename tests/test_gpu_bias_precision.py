"""Activation Bias against fp64 where it is ill conditioned: channels whose mean is many standard deviations (R of
them) from zero, channels without variance.  Both kernels of the stage (few and many (unit, head) items), the fused
call and the stages one by one, with and without the full phi, a second window merged into the statistics.

Bound: z = (q - mean) / sigma is off by R u for the rounding of the mean to fp32 (u = 2^-24) and by about as much
again for its sum; a token's ||phi||_1 = sum z^2 then by 2 R u each, relative: 8 R u leaves a factor of two.  The
variance and the sum over the channels are fp32 sums: 1e-5."""
import pytest

from paper_2502_13542_b200 import workloads as wl

pytestmark = pytest.mark.gpu

CASES = [  # dtype, q heads, kv heads, D, units, tokens, R
    ("bf16", 32, 8, 128, 1, 300, 0), ("bf16", 32, 8, 128, 2, 512, 30), ("bf16", 32, 8, 128, 3, 512, 30), ("bf16", 32, 8, 128, 12, 300, 30),
    ("f32", 32, 8, 128, 1, 200, 300), ("f32", 32, 8, 128, 3, 200, 300), ("f32", 32, 8, 128, 10, 511, 1000), ("f32", 4, 2, 64, 1, 256, 1000),
    ("f32", 4, 2, 64, 20, 256, 1000), ("f32", 4, 2, 64, 80, 100, 300), ("bf16", 8, 1, 64, 40, 130, 30),
]


@pytest.mark.parametrize("dtype,hq,hkv,D,units,nt,R", CASES)
def test_phi_and_probe_against_fp64(dtype, hq, hkv, D, units, nt, R):
    import torch
    from paper_2502_13542_b200 import binding as B
    spec = wl.llama3_8b_layer().replace(n_q_heads=hq, n_kv_heads=hkv, head_dim=D, dtype=dtype)
    cfg = B.make_config(spec, max_context=1024)
    gen = torch.Generator(device="cuda").manual_seed(units + nt)
    mean = R * torch.randn(units, 1, hq, D, device="cuda", generator=gen).sign()
    mean[..., ::5] = 0.0

    def window():
        q = torch.randn(units, nt, hq, D, device="cuda", generator=gen) + mean
        q[..., 7], q[..., 11], q[..., 13] = 3.0, 0.0, -45.25       # no variance
        return q.to(cfg.torch_dtype)

    windows = [window(), window()]
    f32 = dict(dtype=torch.float32, device="cuda")
    for fused, full in ((True, False), (True, True), (False, False), (False, True)):
        count = torch.zeros(units, hq, dtype=torch.int64, device="cuda")
        m, m2 = torch.zeros(units, hq, D, **f32), torch.zeros(units, hq, D, **f32)
        phi_l1, phi = torch.zeros(units, hq, nt, **f32), torch.zeros(units, nt, hq, D, **f32) if full else None
        qh, kv = torch.zeros(units, hq, D, **f32), torch.zeros(units, hkv, D, **f32)
        status = torch.zeros(1, dtype=torch.int32, device="cuda")
        batch = B.Batch(units, 1, 0)
        for i, q in enumerate(windows):
            if fused:
                B.bias_probe(cfg, batch, q, nt, count, m, m2, phi_l1, phi, qh, kv, status)
            else:
                B.activation_bias(cfg, batch, q, nt, count, m, m2, phi_l1, phi, status)
                B.probe_query(cfg, batch, q, nt, phi_l1, qh, kv, status)
            seen = torch.cat(windows[:i + 1], 1).double()
            mu, var = seen.mean(1), seen.var(1)
            want_phi = (q.double() - mu[:, None]) ** 2 / var.clamp_min(1e-12)[:, None]
            want = want_phi.sum(-1).transpose(1, 2)
            bound = 1e-5 + 8 * R * 2.0 ** -24
            what = f"fused {fused}, full {full}, window {i}"
            err = ((phi_l1.double() - want).abs() / want.mean()).max().item()
            assert err < bound, f"{what}: ||phi|| off by {err:.2e}, bound {bound:.2e}"
            if full:
                assert ((phi.double() - want_phi).abs() / want_phi.clamp_min(1.0)).max().item() < 8 * bound, what
            weight = want / want.sum(-1, keepdim=True)
            probe = torch.einsum("uhj,ujhc->uhc", weight, q.double())
            off = (qh.double() - probe).abs().max().item()
            assert off < 4 * bound * max(1.0, q.abs().max().item()), f"{what}: probe off by {off:.2e}"
            assert ((kv.double() - qh.double().reshape(units, hkv, -1, D).mean(2)).abs().max().item()
                    <= 4e-7 * max(1.0, qh.abs().max().item())), what
        assert int(status.item()) == 0 and (count == 2 * nt).all()
