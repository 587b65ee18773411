"""The projection's launch variants (lanes per column, groups per column, few and many columns)
against the oracle's sort, at the longest column of each variant and one entry beyond, with
guesses on both sides of the multiplier and columns on which the sampled start is misled."""
import numpy as np
import pytest

from oracle import pdmcf as O

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n,m", [(1, 16390), (32, 16400), (33, 16385), (64, 16384), (65, 16391), (112, 16384),
                                 (113, 16389), (256, 16384), (257, 16385), (416, 16384), (417, 4099), (512, 4096),
                                 (513, 4097), (1024, 4096), (1025, 4096), (2048, 4097), (2049, 4096), (3072, 4096),
                                 (3073, 1025), (4096, 1024), (4097, 1024), (6144, 1025), (6145, 1024), (10240, 1030),
                                 (10241, 1024), (16384, 1024), (16385, 520), (32768, 512), (103, 1024)])
def test_variant_matches_oracle(lib, n, m):
    ld = (n + 3) // 4 * 4
    gen = torch.Generator(device="cuda").manual_seed(n)
    Q = torch.randn((m, ld), device="cuda", generator=gen)
    Q[1::5] = Q[1::5].sort(dim=1, descending=True).values   # the first chunks hold the largest entries
    Q[2::5] = Q[2::5].sort(dim=1).values                    # ... or the smallest
    cap = torch.rand(m, device="cuda", generator=gen) * 4.0 + 0.05
    cap[3::5] = 1e6                                         # below capacity: mu = 0
    guess = torch.rand(m, device="cuda", generator=gen) * 0.5
    guess[4::5] = 50.0                                      # right of the multiplier
    mu = guess.clone()
    F = torch.full_like(Q, -3.0)
    stream = torch.cuda.current_stream().cuda_stream
    d2 = lib.mcf_project_capped_simplex(n, m, ld, Q.data_ptr(), cap.data_ptr(), F.data_ptr(), mu.data_ptr(), stream)
    mu2, F2 = guess.clone(), Q.clone()                      # in place, without the distance
    lib.mcf_project_capped_simplex_noalloc(n, m, ld, F2.data_ptr(), cap.data_ptr(), F2.data_ptr(), mu2.data_ptr(),
                                           stream, want_dist2=False)
    torch.cuda.synchronize()
    assert torch.equal(F, F2) and torch.equal(mu, mu2)
    assert (F[:, n:] == 0).all()
    rows = np.unique(np.concatenate([np.arange(min(m, 15)), np.arange(m - 5, m)]))
    q = Q[rows, :n].cpu().numpy().astype(np.float64)
    Fr, mur = O.project_capped_simplex(q.T, cap[rows].cpu().numpy().astype(np.float64))
    assert np.abs(F[rows, :n].cpu().numpy() - Fr.T).max() <= 2e-5 * 6.0
    assert np.abs(mu[rows].cpu().numpy() - mur).max() <= 2e-5 * 6.0
    ref = (F[:, :n].double() - Q[:, :n].double()).square().sum().item()
    assert d2 == pytest.approx(ref, rel=1e-5)
