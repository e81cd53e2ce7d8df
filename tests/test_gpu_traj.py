"""The two-kernel rollout (variants 18-19) against the one-sample kernel: the same
bits, at the edges of its tiles (32, 16 and 8 particles per block), chunks (four
steps) and slabs."""
import numpy as np
import pytest

import scenarios as S

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import paper_1506_02869_gb300 as pkg
    return pkg


def _problem(n, rng, **kw):
    base = S.config5(n_scen=1)[0]
    p = base.copy(N=n, aircraft=None, **kw)
    # close enough traffic for many pairs within reach
    p.aircraft = S._traffic(rng, (n + 1) // 2, n // 2, ring=25000.0, z_top=4000.0, sep_h=base.sep_h / 4,
                            sep_v=base.sep_v / 4)
    return p


CASES = {
    # name: (aircraft, particles, samples, steps, further fields)
    "n1": (1, 33, 2, 9, {}),
    "n2_h1": (2, 31, 3, 1, dict(S=1)),
    "n8_h5": (8, 65, 2, 5, dict(S=3)),
    "n9_h6": (9, 17, 3, 6, {}),
    "n16_h7": (16, 50, 2, 7, {}),
    "n17_h30": (17, 257, 3, 30, {}),
    "n32_h60": (32, 130, 5, 60, {}),
    "own_wind": (10, 75, 3, 11, dict(wind_mode=1, grid=(2, 2, 2))),
    "own_wind_n2": (2, 40, 2, 6, dict(wind_mode=1, grid=(2, 2, 2))),
    "rolling": (13, 70, 3, 23, dict(rolling=1, mpc_step=3)),
    "own_wind_rolling": (7, 33, 2, 10, dict(rolling=1, mpc_step=3, wind_mode=1, grid=(2, 2, 2))),
    "noise": (11, 90, 2, 21, dict(w_noise=0.2)),
    # beyond one slab of the workspace (512 MB: about 2200 particles)
    "slabs": (32, 2300, 2, 270, dict(grid=(4, 3, 2))),
}


@pytest.mark.parametrize("sep", [0, 2])
@pytest.mark.parametrize("case", sorted(CASES))
def test_two_kernel_rollout_returns_the_one_sample_bits(pkg, case, sep):
    n, L, M, H, kw = CASES[case]
    rng = np.random.default_rng(7 + n + H)
    p = _problem(n, rng, L=L, M=M, H=H, sep_mode=sep, **{"S": min(4, H), "grid": (9, 12, 5), **kw})
    if p.rolling:
        p.aircraft["t_enter"] = 3 + np.arange(n) % 6       # odd and even entry steps, some at once
    if p.w_noise:
        p.popdense, p.pop_lo, p.pop_hi = S.popdense_grid(rng)
        p.pop_n = p.popdense.shape
    u = S.mild_controls(p, L, rng)
    u[: L // 4] = S.random_controls(p, L // 4, rng)        # many stopped by a limit
    u = torch.from_numpy(u).cuda()
    sol = pkg.Solver(p)
    outs = []
    for v in (4, 18, 19):
        pkg.tma_set_tuning(sol.h, v)
        for soft in ([False, True] if sep else [False]):
            c, cs = sol.rollout_cost(u, 3, soft=soft)
            outs.append((v, soft, c.clone(), None if cs is None else cs.clone(), sol.sample_costs(L).clone(),
                         sol.sample_costs(L, soft=True).clone() if soft else None, sol.live_steps()))
    sol.close()
    assert torch.isfinite(outs[0][2]).any()
    per = len(outs) // 3
    for k, got in enumerate(outs):
        ref = outs[k % per]
        for a, b in zip(got[2:], ref[2:]):
            assert torch.equal(a, b) if torch.is_tensor(a) else a == b, (case, got[:2])


def test_two_kernel_rollout_needs_two_samples(pkg):
    p = _problem(4, np.random.default_rng(5), L=64, M=1, H=8, sep_mode=0, grid=(4, 4, 3))
    sol = pkg.Solver(p)
    with pytest.raises(pkg.TmaError):
        pkg.tma_set_tuning(sol.h, 18)
    sol.close()
