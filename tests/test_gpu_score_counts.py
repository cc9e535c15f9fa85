"""Candidate counts that are not counts: a negative one is a sequence without candidates, one beyond the table is
clamped with a status bit, and the sequences around them get their scores all the same; both score kernels."""
import pytest

from paper_2502_13542_b200 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("counts,n_cap", [([-3, 20, -1000, 33, -1], 40), ([-7, 4000, -2 ** 31, 4799, 9999, -4, 13], 4799)])
def test_negative_and_large_counts(counts, n_cap):
    import torch
    from paper_2502_13542_b200 import binding as B
    cfg = B.make_config(wl.llama3_8b_layer(), n_cap=n_cap)
    U = len(counts)
    gen = torch.Generator(device="cuda").manual_seed(1)
    table = torch.randn(U, 8, n_cap, 4, 128, device="cuda", generator=gen).to(cfg.torch_dtype)
    inv = 1.0 / table.float().norm(dim=-1)
    probe = torch.randn(U, 8, 128, device="cuda", generator=gen)
    scores, theta = torch.full((U, 8, n_cap), 7.0, device="cuda"), torch.full((U, 8), 7.0, device="cuda")
    n_cand = torch.tensor(counts, dtype=torch.int32, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    B.score_blocks(cfg, B.Batch(U, 1, 0), probe, table, inv, n_cand, scores, theta, status)
    torch.cuda.synchronize()
    assert int(status.item()) == (B.DEV_NCAND_CLAMPED if max(counts) > n_cap else 0)
    want = (torch.einsum("uhd,uhbrd->uhbr", probe.double(), table.double()) * inv.double()).mean(-1) / probe.double().norm(dim=-1)[..., None]
    for u, c in enumerate(counts):
        n = max(0, min(c, n_cap))
        assert (scores[u, :, n:] == 7.0).all()
        if n:
            assert (scores[u, :, :n].double() - want[u, :, :n]).abs().max().item() < 32 * 2.0 ** -24
        else:
            assert (theta[u] == 0).all()
