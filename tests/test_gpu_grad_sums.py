"""The gradient's last kernels: the sums over the ranges of samples by a kernel of their
own (few tiles, or many ranges) or inside grad_controls_kernel, and that kernel's fetch
ahead.  The same ranges give the same bits in every form: a call of few particles against
the same particles at the head of a call whose tiles fill the chip."""
import numpy as np
import pytest

import scenarios as S

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

FILL = 304           # tiles from which the chip is filled


def _problem(N, M, H, L):
    rng = np.random.default_rng(N + H)
    base = S.config5(n_scen=1)[0]
    p = base.copy(N=N, M=M, H=H, L=L, grid=(5, 4, 3), sep_mode=1, aircraft=None, S=min(4, H))
    p.aircraft = S._traffic(rng, (N + 1) // 2, N // 2, ring=25000.0, z_top=4000.0, sep_h=p.sep_h / 4, sep_v=p.sep_v / 4)
    a = p.aircraft[0]                                        # lands within some horizons, at steps that the wind decides
    a["x"], a["y"], a["z"], a["v"], a["chi"] = 16000.0, 0.0, 250.0, 80.0, np.pi
    u = S.mild_controls(p, L, rng, frac=0.1)
    u[1::4] = S.random_controls(p, L, rng)[1::4]             # infeasible particles among the others
    return p, u


# samples capped so that few and many tiles split them alike: one a range
@pytest.mark.parametrize("N,M,H", [(1, 9, 21), (1, 2, 5), (2, 1, 4), (3, 6, 21), (3, 2, 9), (8, 1, 33), (9, 2, 21), (9, 1, 7),
                                   (17, 2, 22), (32, 2, 17), (32, 1, 1), (8, 3, 50), (12, 2, 63)])
def test_every_form_of_the_sums_returns_the_same_bits(N, M, H):
    import paper_1506_02869_gb300 as pkg
    tp = 32 if N <= 8 else (16 if N <= 16 else 8)
    p, u = _problem(N, M, H, FILL * tp + 5)
    ud = torch.from_numpy(u).cuda()
    sol = pkg.Solver(p)
    whole = [x.clone() for x in sol.rollout_grad(ud, 3, cbar=True)]
    feasible = torch.isfinite(whole[0])
    assert bool(feasible.any()) and bool((whole[1][feasible] != 0).any())
    for n in (1, tp + 1, 3 * tp - 5, 40 * tp):
        cost, grad, cbar = sol.rollout_grad(ud[:n].contiguous(), 3, cbar=True)
        assert torch.equal(cost, whole[0][:n]) and torch.equal(grad, whole[1][:n]) and torch.equal(cbar, whole[2][:, :n]), n
    sol.close()
