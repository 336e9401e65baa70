"""The FP64 sweeps' integer lines at the edges of their range, through the inverse mass operator: lines of one
magnitude and of widely mixed ones, the ends of the range and values beyond it (the FP64 path), zeros, infinities
and NaN, at line lengths 2 to 7 and a ragged number of cells."""
import math

import numpy as np
import pytest
import torch

from oracle.basis import gauss_legendre_01, lagrange_1d, lgl_nodes_01
from paper_1806_03095_gb300 import api

pytestmark = pytest.mark.gpu


def _one(k):
    """S^-1, S^-T and the weights of the k+1 mass points."""
    x, w = gauss_legendre_01(k + 1)
    S, _ = lagrange_1d(lgl_nodes_01(k), x)
    return np.linalg.inv(S), w


@pytest.mark.parametrize("k", [1, 2, 3, 4, 5, 6])
@pytest.mark.parametrize("values", ["unit", "mixed", "tiny", "huge", "denormal", "zeros"])
def test_inverse_mass_over_the_range_of_magnitudes(k, values):
    n, cells = k + 1, (3, 2, 5)
    nq = {1: (2, 2), 2: (4, 3), 3: (5, 4), 4: (7, 5), 5: (8, 6), 6: (10, 7)}[k]
    g = api.DGCNS(cells, (-math.pi,) * 3, (math.pi,) * 3, (1, 1, 1), k, *nq)
    gen = torch.Generator().manual_seed(11 + k)
    r = torch.rand(g.shape, generator=gen, dtype=torch.float64) * 2 - 1
    scale = {"unit": 1.0, "tiny": 1e-200, "huge": 1e200, "denormal": 1e-306, "mixed": 1.0, "zeros": 1.0}[values]
    if values == "mixed":
        r = r * torch.exp2(torch.randint(-70, 71, g.shape, generator=gen).double())
    if values == "zeros":
        r = r * (torch.rand(g.shape, generator=gen) < 0.15)
        r[0] = 0.0
    out = (g.inverse_mass((r * scale).cuda()) / scale).cpu()
    Si, w = _one(k)
    detJ = np.prod([2 * math.pi / c for c in cells])
    a = r.numpy().reshape(-1, 5, n, n, n)
    W = 1.0 / (np.einsum("z,y,x->zyx", w, w, w) * detJ)
    b = a
    for ax in (2, 3, 4):
        b = np.moveaxis(np.tensordot(Si.T, b, (1, ax)), 0, ax)
    b = b * W
    for ax in (2, 3, 4):
        b = np.moveaxis(np.tensordot(Si, b, (1, ax)), 0, ax)
    # each of the six sweeps and the scaling errs by at most 4 2^-53 of its largest input times its row sum
    amp = np.abs(Si.T).sum(1).max() ** 3 * W.max() * np.abs(Si).sum(1).max() ** 3
    tol = 7 * 4 * 2.0 ** -53 * amp * np.abs(a).reshape(a.shape[0], 5, -1).max(-1)
    err = np.abs(out.numpy().reshape(b.shape) - b).reshape(a.shape[0], 5, -1).max(-1)
    assert (err <= tol).all(), float((err / np.maximum(tol, 1e-300)).max())


@pytest.mark.parametrize("bad", [float("nan"), float("inf"), -float("inf")])
def test_non_finite_values_stay_in_their_block(bad):
    g = api.DGCNS((3, 2, 5), (-math.pi,) * 3, (math.pi,) * 3, (1, 1, 1), 3, 5, 4)
    r = torch.rand(g.shape, generator=torch.Generator().manual_seed(3), dtype=torch.float64)
    clean = g.inverse_mass(r.cuda()).cpu()
    r[7, 2, 13] = bad
    out = g.inverse_mass(r.cuda()).cpu()
    assert not torch.isfinite(out[7, 2]).any()
    keep = torch.ones(g.shape[:2], dtype=torch.bool)
    keep[7, 2] = False
    assert torch.equal(out[keep], clean[keep])


@pytest.mark.parametrize("in_place", [False, True])
@pytest.mark.parametrize("cells", [(2, 2, 2), (3, 2, 5), (23, 23, 23)])
def test_inverse_mass_of_fp32_residuals(cells, in_place):
    """Fewer blocks than a tile of 32 per warp, a ragged last tile, and more tiles than resident warps."""
    n, k = 4, 3
    g = api.DGCNS(cells, (-math.pi,) * 3, (math.pi,) * 3, (1, 1, 1), k, 5, 4, precision=api.MIXED)
    r = (torch.rand(g.shape, generator=torch.Generator().manual_seed(5)) * 2 - 1).float()
    rg = r.cuda()
    out = g.inverse_mass(rg, rg) if in_place else g.inverse_mass(rg)
    if not in_place:
        assert torch.equal(rg.cpu(), r)
    Si, w = _one(k)
    W = 1.0 / (np.einsum("z,y,x->zyx", w, w, w) * np.prod([2 * math.pi / c for c in cells]))
    b = a = r.double().numpy().reshape(-1, 5, n, n, n)
    for ax in (2, 3, 4):
        b = np.moveaxis(np.tensordot(Si.T, b, (1, ax)), 0, ax)
    b = b * W
    for ax in (2, 3, 4):
        b = np.moveaxis(np.tensordot(Si, b, (1, ax)), 0, ax)
    # six sweeps and the scaling, each with its rounded table at most 8 2^-24 of its largest input times its row sum
    amp = np.abs(Si.T).sum(1).max() ** 3 * W.max() * np.abs(Si).sum(1).max() ** 3
    tol = 7 * 8 * 2.0 ** -24 * amp * np.abs(a).reshape(a.shape[0], 5, -1).max(-1)
    err = np.abs(out.cpu().double().numpy().reshape(b.shape) - b).reshape(a.shape[0], 5, -1).max(-1)
    assert (err <= tol).all(), float((err / tol).max())
