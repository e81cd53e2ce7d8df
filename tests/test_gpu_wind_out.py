"""The wind field at every level count (lanes of a column, partly used and partly filled
tiles of the product), single and batched, and its plain values in a caller's buffer at
any float-aligned address."""
import ctypes as C

import numpy as np
import pytest

import oracle as O
import scenarios as S
from gpu_helpers import compare_costs, oracle_wind

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import paper_1506_02869_gb300 as pkg
    return pkg


def _problem(grid, M=2, H=5):
    return S.shrink(S.config1(), L=64, M=M, H=H).copy(grid=grid)


@pytest.mark.parametrize("grid", [(9, 8, 5), (17, 12, 4), (2, 2, 2)])
def test_field_into_a_view_at_an_odd_offset(pkg, grid):
    """The buffer's first float is 4- but not 8-byte aligned; what lies beside it stays."""
    p = _problem(grid)
    sol = pkg.Solver(p)
    ref = sol.wind_field()
    for off in (1, 2, 3):
        buf = torch.full((ref.numel() + 8,), -7.0, device="cuda")
        pkg.tma_wind_field(sol.h, buf[off:off + ref.numel()])
        assert torch.equal(buf[off:off + ref.numel()], ref.reshape(-1)), off
        assert bool((buf[:off] == -7.0).all()) and bool((buf[off + ref.numel():] == -7.0).all()), off
    sol.close()


def test_an_address_that_holds_no_float_is_refused(pkg):
    """Refused on the host, before any launch."""
    sol = pkg.Solver(_problem((4, 4, 3)))
    torch.cuda.synchronize()
    out = torch.empty(2 * 5 * 48 * 2 + 2, device="cuda")
    before = pkg.lib().tma_launch_count()
    for off in (1, 2, 3):
        assert pkg.lib().tma_wind_field(sol.h, C.c_void_p(out.data_ptr() + off), None) == 1
    assert pkg.lib().tma_launch_count() == before
    sol.close()


@pytest.mark.parametrize("nz", range(2, 17))
def test_field_matches_oracle_at_every_level_count(pkg, nz):
    """65 rows (one beyond a tile of the product), nine fields (the last column tile ends within)."""
    p = _problem((5, 13, nz), M=3, H=3).copy(S=2)
    sol = pkg.Solver(p)
    got = sol.wind_field().double().cpu().numpy()
    sol.close()
    assert np.abs(got - O.wind_field(p)).max() / p.wind_sigma < 2e-5


@pytest.mark.parametrize("nz", [3, 9, 13, 16])
def test_records_of_many_levels_in_the_rollout(pkg, nz):
    """The packed records (differences to the level above) through the costs, against the oracle; and a
    batch's field, bit for bit the single solver's."""
    ps = [p for p in sorted(S.config5(n_scen=24), key=lambda p: p.N)[2:24:10]]
    ps = [S.shrink(p, L=96, M=2, H=16, J_max=2, grid=(6, 11, nz)) for p in ps]
    p = ps[1]
    rng = np.random.default_rng(nz)
    u = S.mild_controls(p, p.L, rng)
    sol = pkg.Solver(p)
    got = sol.rollout_cost(torch.from_numpy(u).cuda(), 1)[0].cpu().numpy().astype(np.float64)
    sol.close()
    ref = O.rollout(p, u, 1, W=oracle_wind(p))
    assert compare_costs(got, ref["cbar"], ref["margin"], ref["smargin"], f"nz={nz}")[1] > 50
    b = pkg.tma_batch_create(ps)
    for form in (0, 1):
        pkg.tma_batch_set_dispatch(b, form)
        pkg.tma_batch_solve(b)
        res = pkg.tma_batch_results(b, [q.N for q in ps], ps[0].S)
        for k, q in enumerate(ps):
            sol = pkg.Solver(q)
            best_u = sol.solve()[0]
            assert np.array_equal(res["best_u"][k], best_u.cpu().numpy()) and res["best"][k] == sol.best_index(), (form, k)
            sol.close()
    pkg.tma_batch_destroy(b)
