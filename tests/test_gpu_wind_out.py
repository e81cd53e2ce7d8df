"""The plain field in a caller's buffer: any float-aligned address."""
import ctypes as C

import pytest

import scenarios as S

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
