"""The final selection sums in FP64 only the particles that FP32 bounds leave in
question: the chosen particle, its sum and its count are those of summing all."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _select(pkg, c):
    N, L = c.shape
    d = torch.from_numpy(np.ascontiguousarray(c)).cuda()
    best = torch.empty(1, dtype=torch.int64, device="cuda")
    bsum = torch.empty(1, dtype=torch.float64, device="cuda")
    ninf = torch.empty(1, dtype=torch.int32, device="cuda")
    work = torch.empty(max(16, pkg.lib().tma_select_workspace(L)), dtype=torch.uint8, device="cuda")
    pkg.tma_select(d, best, bsum, ninf, work)
    return int(best), float(bsum), int(ninf)


def _reference(c):
    bad = ~np.isfinite(c)
    n = bad.sum(0)
    s = np.zeros(c.shape[1])
    for row, b in zip(c, bad):                     # aircraft in order, FP64
        s = s + np.where(b, 0.0, row.astype(np.float64))
    l = int(np.lexsort((np.arange(c.shape[1]), s, n))[0])
    return l, float(s[l]) if n[l] == 0 else math.inf, int(n[l])


@pytest.mark.parametrize("N,L", [(1, 1), (3, 255), (24, 257), (32, 4096), (8, 151553), (2, 700001)])
@pytest.mark.parametrize("kind", ["near", "spread", "inf", "huge", "signed", "tiny"])
def test_selection_equals_summing_every_particle(N, L, kind):
    import paper_1506_02869_gb300 as pkg
    rng = np.random.default_rng(N * 1000 + L)
    c = rng.exponential(0.5, (N, L)).astype(np.float32)
    if kind == "near":                             # sums that differ in the last bits of FP32 and below
        c = (1.0 + rng.integers(0, 3, (N, L)) * 2.0 ** -23).astype(np.float32)
    if kind == "inf":
        c[rng.random((N, L)) < 0.4] = math.inf
        c[rng.random((N, L)) < 0.1] = math.nan
        c[rng.random((N, L)) < 0.01] = -math.inf
    if kind == "huge":                             # FP32 sums overflow, FP64 ones do not
        c = (3e38 * (1 - rng.random((N, L)) * 1e-3)).astype(np.float32)
    if kind == "signed":
        c = (rng.standard_normal((N, L)) * 10.0 ** rng.integers(-6, 6, (N, L))).astype(np.float32)
    if kind == "tiny":                             # normal numbers close to the smallest
        c = (2e-38 * (1 + rng.random((N, L)))).astype(np.float32)
    assert _select(pkg, c) == _reference(c)
