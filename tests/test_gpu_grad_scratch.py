"""The gradient's scratch: never above its bound, taken with care on a nearly full
device, and calls that get less of it (more slabs, fewer ranges of samples) return
the gradient all the same."""
import numpy as np
import pytest

import scenarios as S
from gpu_helpers import cuda

pytestmark = pytest.mark.gpu

BOUND = 6 << 30
GRAD_TOL = 1e-3      # relative L2 norm per particle, the gradient's bar (the sums over samples may be regrouped)


@pytest.fixture(scope="module")
def torch():
    return cuda()


@pytest.fixture(scope="module")
def pkg(torch):
    import paper_1506_02869_gb300 as pkg
    return pkg


def _problem(N, H, M, L, grid=(4, 4, 3)):
    rng = np.random.default_rng(N + H)
    base = S.config5(n_scen=1)[0]
    p = base.copy(N=N, H=H, M=M, L=L, grid=grid, sep_mode=1, aircraft=None)
    p.aircraft = S._traffic(rng, (N + 1) // 2, N // 2, ring=45000.0, z_top=9000.0, sep_h=p.sep_h, sep_v=p.sep_v,
                            dep_r=(2000.0, 30000.0))
    u = S.mild_controls(p, L, rng) * np.float32(min(1.0, 20.0 / H))     # long horizons: nearly straight
    return p, u


def _free(torch):
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return torch.cuda.mem_get_info()[0]


def _gradient(torch, sol, u, n):
    cost, grad, cbar = sol.rollout_grad(torch.from_numpy(u[:n]).cuda(), 1, cbar=True)
    torch.cuda.synchronize()
    return cost.cpu().numpy(), grad.cpu().numpy(), cbar.cpu().numpy()


def _same(got, ref, exact):
    """The costs are the same bits whatever the slabs and ranges; so is the gradient with the ranges equal."""
    assert np.isfinite(ref[0]).any()
    assert np.array_equal(got[0], ref[0]) and np.array_equal(got[2], ref[2])
    if exact:
        assert np.array_equal(got[1], ref[1])
        return
    for a, b in zip(got[1], ref[1]):
        assert np.linalg.norm(a - b) <= GRAD_TOL * np.linalg.norm(b)


def test_few_particles_of_many_samples_stay_within_the_bound(torch, pkg):
    p, u = _problem(32, 320, 512, 32)
    sol = pkg.Solver(p)
    before = _free(torch)
    whole = _gradient(torch, sol, u, 32)
    few = _gradient(torch, sol, u, 8)                    # a tile: the most ranges
    costs = 4 * p.M * p.N * p.L
    assert before - _free(torch) <= BOUND + costs + (32 << 20)
    _same(few, tuple(x[:8] if x.ndim != 2 else x[:, :8] for x in whole), False)
    sol.close()


@pytest.mark.parametrize("N,H,M,L,few", [(12, 60, 1, 4100, 17), (9, 61, 3, 3001, 16), (32, 320, 256, 72, 8)])
def test_a_nearly_full_device(torch, pkg, N, H, M, L, few):
    """With 1.5 GB left the scratch takes a sixteenth of it: slabs with a ragged last one (and, with
    several samples, fewer ranges), the same gradients; the rest of the memory stays the program's."""
    p, u = _problem(N, H, M, L)
    sol = pkg.Solver(p)
    ref = _gradient(torch, sol, u, L), _gradient(torch, sol, u, few)
    sol.close()
    sol = pkg.Solver(p)
    hold = torch.empty(_free(torch) - (3 << 29), dtype=torch.uint8, device="cuda")
    before = _free(torch)
    got = _gradient(torch, sol, u, L), _gradient(torch, sol, u, few)      # then more ranges in the same scratch
    taken = before - _free(torch)
    del hold
    sol.close()
    torch.cuda.empty_cache()
    assert taken <= before // 16 + 4 * M * N * L + (64 << 20)
    for g, r in zip(got, ref):
        _same(g, r, M == 1)
