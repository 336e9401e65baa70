"""FP64 accuracy cell by cell: what an evaluation gives in a cell depends on that cell and its face neighbours only, to
the last bit, and is as accurate where the flow is quiet as where it is strong, whatever cells or faces a thread block
carries together."""
import math

import pytest
import torch

from paper_1806_03095_gb300 import api, inputs

pytestmark = pytest.mark.gpu
NQ = {1: (2, 2), 2: (4, 3), 3: (5, 4), 4: (7, 5), 5: (8, 6), 6: (10, 7)}
MESH = {"affine": {}, "walls": dict(periodic=(0, 0, 0)), "force": dict(body_force=(1.0, 0.3, -0.2)),
        "sine": dict(mapping=api.MAP_SINE, map_param=0.05),
        "channel": dict(periodic=(1, 0, 1), mapping=api.MAP_CHANNEL, map_param=1.8, body_force=(1.0, 0.3, -0.2)),
        "rotated": dict(mapping=api.MAP_ROTATED, map_param=7, deform=0.05)}
CASES = [(k, m) for k in NQ for m in ("affine", "walls", "force")] + [(k, m) for k in (2, 3, 5) for m in ("sine", "channel", "rotated")]
OPS = (api.OP_L, api.OP_F, api.OP_FC, api.OP_FV)


def _context(cells, k, kernel, periodic=(1, 1, 1), **kw):
    return api.DGCNS(cells, (-math.pi,) * 3, (math.pi,) * 3, periodic, k, *NQ[k], kernel=kernel, **kw)


def _cells(k):
    # beyond 1216 cells a thread block carries several of them (k <= 3); faces always come several to a block
    return (11, 11, 11) if k <= 3 else (5, 3, 7)


def _states(cells, k, scale, seed=17):
    """The random state with every deviation from the uniform state scaled, and the same with one cell at full size: the
    last of the first row, whose successor in index order starts the next row and is not its neighbour."""
    n = cells[0] * cells[1] * cells[2]
    ref = torch.tensor([1.0, 0.0, 0.0, 0.0, 178.57142857142858], dtype=torch.float64)[None, :, None]
    U = inputs.random_state(n, (k + 1) ** 3, seed)
    quiet = ref + (U - ref) * scale
    strong = quiet.clone()
    strong[cells[0] - 1] = U[cells[0] - 1]
    idx = torch.arange(n)
    far = torch.zeros(n, dtype=torch.long)
    at = cells[0] - 1
    for d, (a, b) in enumerate(((1, cells[0]), (cells[0], cells[1]), (cells[0] * cells[1], cells[2]))):
        r = (idx // a % b - at // a % b).abs()
        far += torch.minimum(r, b - r)
    return quiet.cuda(), strong.cuda(), (far > 1).cuda()


@pytest.mark.parametrize("k,mesh", CASES)
def test_a_strong_cell_does_not_change_a_bit_beyond_its_neighbours(k, mesh):
    cells = _cells(k)
    g = _context(cells, k, api.KERNEL_FACES, **MESH[mesh])
    quiet, strong, far = _states(cells, k, 2.0 ** -30)
    for op in OPS:
        a, b = g.apply(quiet, op=op), g.apply(strong, op=op)
        assert not torch.equal(a[~far], b[~far])
        assert torch.equal(a[far], b[far]), op
    out = []
    for U in (quiet, strong):
        dU, V = torch.zeros_like(U), torch.empty_like(U)
        g.rk_stage(2, 1e-3, 0.0, U, dU, V)
        out.append((dU[far], V[far]))
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])


@pytest.mark.parametrize("scale", [2.0 ** -12, 2.0 ** -30])
@pytest.mark.parametrize("k,mesh", CASES)
def test_quiet_cells_are_as_accurate_as_strong_ones(k, mesh, scale):
    cells = _cells(k)
    f, e = (_context(cells, k, o, **MESH[mesh]) for o in (api.KERNEL_FACES, api.KERNEL_FUSED))
    _, U, _ = _states(cells, k, scale)
    for op in OPS:
        a, b = f.apply(U, op=op), e.apply(U, op=op)
        # per cell and row, against the general path, whose lines round on their own: some 20 sweeps and point operations,
        # each within 8 2^-53 of its largest input times a row sum, which the 1D derivatives amplify by at most 30 over
        # the result (k = 6), and another 10 for cells whose result happens to be small
        tol = 20 * 8 * 2.0 ** -53 * 30 * 10
        top = b.abs().amax(2)
        err = (a - b).abs().amax(2)
        assert (err <= tol * top).all(), (op, float((err / top).max()))
