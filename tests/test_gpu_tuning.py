"""The tuner: what it times, and which solvers share a choice through its cache."""
import numpy as np
import pytest

import scenarios as S

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _solver(pkg, N, L, M):
    rng = np.random.default_rng(N)
    base = S.config5(n_scen=1)[0]
    p = base.copy(N=N, L=L, M=M, H=12, grid=(5, 4, 3), sep_mode=2, aircraft=None)
    p.aircraft = S._traffic(rng, (N + 1) // 2, N // 2, ring=45000.0, z_top=9000.0, sep_h=p.sep_h, sep_v=p.sep_v,
                            dep_r=(2000.0, 30000.0))
    return pkg.Solver(p)


@pytest.mark.parametrize("N,order", [(26, (1, 2)), (22, (2, 1))])
def test_one_sample_and_two_samples_of_one_size_class(N, order):
    """One sample has no two-kernel variants; the same size class (tiles times samples) with two has.
    (Kinds of problem that no other test tunes.)"""
    import paper_1506_02869_gb300 as pkg
    for M in order:
        sol = _solver(pkg, N, 4096 // M, M)
        variant, timed = pkg.tma_get_tuning(sol.h)
        assert timed, M                                   # its own variants were timed, not another's choice taken
        assert (18 in timed) == (M == 2), (M, timed)
        pkg.tma_set_tuning(sol.h, variant)                # what was chosen can be chosen
        sol.close()
    again = _solver(pkg, N, 4096 // order[1], order[1])
    assert not pkg.tma_get_tuning(again.h)[1]             # from the cache
    again.close()


def test_small_work_times_the_smaller_tiles_too():
    """Beside the two-kernel form the smaller tiles are the fastest for some small work; for large work
    only the variants that can be are timed."""
    import paper_1506_02869_gb300 as pkg
    for L, M, small in ((223, 12, True), (8192, 64, False)):
        sol = _solver(pkg, 28, L, M)
        timed = pkg.tma_get_tuning(sol.h)[1]
        assert {18, 19, 4, 13} <= set(timed), timed
        assert ({15, 16, 17} <= set(timed)) == small, timed
        sol.close()


def test_few_samples_of_many_particles_are_a_class_of_their_own():
    """With two samples 32768 particles are tuned as such, not by the choice for 8192."""
    import paper_1506_02869_gb300 as pkg
    for L in (8192, 32768):
        sol = _solver(pkg, 30, L, 2)
        assert pkg.tma_get_tuning(sol.h)[1], L
        sol.close()


def test_older_variant_names_without_a_workspace():
    """8-12 are accepted for the problems they always were; where the two-kernel form has no workspace
    (a long horizon beyond 1024 particles) they run the one-sample kernel: the same bits."""
    import paper_1506_02869_gb300 as pkg
    rng = np.random.default_rng(3)
    base = S.config5(n_scen=1)[0]
    p = base.copy(N=24, L=1056, M=2, H=900, grid=(4, 3, 2), sep_mode=0, aircraft=None)
    p.aircraft = S._traffic(rng, 12, 12, ring=45000.0, z_top=9000.0, sep_h=p.sep_h, sep_v=p.sep_v, dep_r=(2000.0, 30000.0))
    sol = pkg.Solver(p)
    with pytest.raises(pkg.TmaError):
        pkg.tma_set_tuning(sol.h, 18)
    u = torch.from_numpy(S.mild_controls(p, p.L, rng) * np.float32(0.02)).cuda()
    pkg.tma_set_tuning(sol.h, 4)
    ref = sol.rollout_cost(u, 1)[0].clone()
    assert bool(torch.isfinite(ref).any())
    for v in (8, 11):
        with pytest.raises(pkg.TmaError):                 # block caps of 256 and 512 threads
            pkg.tma_set_tuning(sol.h, v)
    pkg.tma_set_tuning(sol.h, 12)
    assert torch.equal(sol.rollout_cost(u, 1)[0], ref)
    sol.close()


def test_a_solver_without_room_for_the_workspace():
    """On a nearly full device the two-kernel form's workspace is left out: the one-sample kernels run,
    with the same bits, and a later solver of the same class has all its variants again."""
    import paper_1506_02869_gb300 as pkg
    ref = _solver(pkg, 14, 65536, 2)
    assert 18 in pkg.tma_get_tuning(ref.h)[1]
    g = torch.Generator(device="cuda").manual_seed(4)
    u = 1e-3 * torch.randn((65536, 14, ref.S, 3), generator=g, device="cuda")
    want = ref.rollout_cost(u, 1)[0].clone()
    ref.close()
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    hold = torch.empty(torch.cuda.mem_get_info()[0] - (3 << 29), dtype=torch.uint8, device="cuda")
    sol = _solver(pkg, 14, 65536, 2)
    timed = pkg.tma_get_tuning(sol.h)[1]
    with pytest.raises(pkg.TmaError):
        pkg.tma_set_tuning(sol.h, 18)
    got = sol.rollout_cost(u, 1)[0].clone()
    sol.close()
    del hold
    torch.cuda.empty_cache()
    assert timed and not {18, 19} & set(timed)
    assert bool(torch.isfinite(want).any()) and torch.equal(got, want)
    again = _solver(pkg, 14, 65536, 2)
    pkg.tma_set_tuning(again.h, 18)
    assert torch.equal(again.rollout_cost(u, 1)[0], want)
    again.close()
