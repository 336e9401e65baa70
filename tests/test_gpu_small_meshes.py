"""Meshes around the sizes where the collocation kernels change their batches (as long as the smaller ones are resident
at once: 608 thread blocks and more, by the kernel's occupancy), against the element-centric kernels and, for the mixed
form, against FP64."""
import math

import pytest
import torch

from paper_1806_03095_gb300 import api, inputs

pytestmark = pytest.mark.gpu
NQ = {1: (2, 2), 2: (4, 3), 3: (5, 4), 4: (7, 5), 5: (8, 6)}
CELLS = [(3, 3, 11), (5, 6, 7), (8, 4, 19), (7, 3, 29), (8, 8, 12), (9, 9, 13), (8, 8, 19), (7, 11, 16), (11, 13, 15)]


def _context(cells, k, kernel, precision=0, **kw):
    return api.DGCNS(cells, (-math.pi,) * 3, (math.pi,) * 3, kw.pop("periodic", (1, 1, 1)), k, *NQ[k], kernel=kernel,
                     precision=precision, **kw)


def _err(a, b):
    a, b = a.double(), b.double()
    return float((a - b).norm() / b.norm()), float((a - b).abs().max() / b.abs().max())


@pytest.mark.parametrize("cells", CELLS)
@pytest.mark.parametrize("k,kw", [(1, {}), (2, {}), (3, {}), (3, dict(periodic=(0, 1, 0))), (2, dict(mapping=api.MAP_SINE, map_param=0.05))])
def test_fp64(cells, k, kw):
    f, e = _context(cells, k, api.KERNEL_FACES, **kw), _context(cells, k, api.KERNEL_FUSED, **kw)
    U = inputs.random_state(f.n_cells, f.n ** 3, 31).cuda()
    two, mx = _err(f.apply(U), e.apply(U))
    assert two < 2e-12 and mx < 2e-12  # (both sides within 1e-12 of the oracle on these states)


@pytest.mark.parametrize("cells", CELLS)
@pytest.mark.parametrize("k,kw", [(3, {}), (4, {}), (5, {}), (3, dict(periodic=(0, 1, 0))), (3, dict(mapping=api.MAP_SINE, map_param=0.05))])
def test_mixed(cells, k, kw):
    f, m = _context(cells, k, api.KERNEL_FACES, **kw), _context(cells, k, api.KERNEL_FACES, api.MIXED, **kw)
    U = inputs.random_state(f.n_cells, f.n ** 3, 31).cuda()
    two, mx = _err(m.apply(U), f.apply(U))
    assert two < 1e-5 and mx < 1e-4
