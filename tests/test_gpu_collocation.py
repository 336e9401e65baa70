"""The collocation kernels of the face-centric organisation against the general path (the element-centric fused
kernels, which test with the nodal basis) over the forms they accept: degrees, ragged meshes whose last batch is
short, meshes around the size where the batches change, walls, stored geometry, rotated frames, every operator, both
precisions; and what they do with non-finite and extreme states."""
import math

import pytest
import torch

from paper_1806_03095_gb300 import api, inputs

pytestmark = pytest.mark.gpu
NQ = {1: (2, 2), 2: (4, 3), 3: (5, 4), 4: (7, 5), 5: (8, 6), 6: (10, 7)}


def _pair(cells, k, nq=None, periodic=(1, 1, 1), **kw):
    return [api.DGCNS(cells, (-math.pi,) * 3, (math.pi,) * 3, periodic, k, *(nq or NQ[k]), kernel=o, **kw)
            for o in (api.KERNEL_FACES, api.KERNEL_FUSED)]


def _err(a, b):
    a, b = a.double(), b.double()
    return float((a - b).norm() / b.norm()), float((a - b).abs().max() / b.abs().max())


CASES = [(k, m, None) for k in NQ for m in ("affine", "walls")] + [(3, "affine", (4, 4)), (5, "affine", (6, 6))] + [
    (k, m, None) for k in (2, 3, 5) for m in ("sine", "channel", "rotated")]


@pytest.mark.parametrize("k,mesh,nq", CASES)
def test_against_the_general_path_fp64(k, mesh, nq):
    kw = {"affine": {}, "walls": dict(periodic=(0, 0, 0)), "sine": dict(mapping=api.MAP_SINE, map_param=0.05),
          "channel": dict(periodic=(1, 0, 1), mapping=api.MAP_CHANNEL, map_param=1.8, body_force=(1.0, 0.3, -0.2)),
          "rotated": dict(mapping=api.MAP_ROTATED, map_param=7, deform=0.05)}[mesh]
    f, e = _pair((3, 5, 3), k, nq, **kw)
    U = inputs.random_state(f.n_cells, f.n ** 3, 5).cuda()
    for op in (api.OP_L, api.OP_F, api.OP_FC, api.OP_FV):
        two, mx = _err(f.apply(U, op=op), e.apply(U, op=op))
        # both sides round 1e-12 from the oracle at most on these states (test_gpu_parity)
        assert two < 2e-12 and mx < 2e-12, (op, two, mx)


@pytest.mark.parametrize("cells", [(1, 1, 1), (7, 11, 13), (8, 8, 19), (10, 11, 11), (11, 11, 11), (9, 9, 15)])
@pytest.mark.parametrize("k", [2, 3])
def test_batches_and_sizes(cells, k):
    f, e = _pair(cells, k)
    U = inputs.random_state(f.n_cells, f.n ** 3, 9).cuda()
    outs = []
    for g in (f, e):
        dU = (0.01 * U).clone()
        V = g.empty_state()
        g.rk_stage(2, 1e-3, 0.0, U, dU, V)
        outs.append((dU, V))
    for a, b in zip(*outs):
        two, mx = _err(a, b)
        assert two < 2e-12 and mx < 2e-12


@pytest.mark.parametrize("k,mesh", [(3, "affine"), (4, "affine"), (5, "affine"), (3, "sine"), (5, "channel"), (3, "walls"),
                                    (3, "rotated")])
@pytest.mark.parametrize("cells", [(3, 5, 3), (11, 11, 13)])
def test_mixed_against_fp64(k, mesh, cells):
    kw = {"affine": {}, "walls": dict(periodic=(0, 0, 0)), "sine": dict(mapping=api.MAP_SINE, map_param=0.05),
          "channel": dict(periodic=(1, 0, 1), mapping=api.MAP_CHANNEL, map_param=1.8, body_force=(1.0, 0.3, -0.2)),
          "rotated": dict(mapping=api.MAP_ROTATED, map_param=7, deform=0.05)}[mesh]
    f, _ = _pair(cells, k, **kw)
    m, _ = _pair(cells, k, precision=api.MIXED, **kw)
    U = inputs.random_state(f.n_cells, f.n ** 3, 5).cuda()
    for op in (api.OP_L, api.OP_F, api.OP_FC, api.OP_FV):
        two, mx = _err(m.apply(U, op=op), f.apply(U, op=op))
        assert two < 1e-5 and mx < 1e-4, (op, two, mx)


@pytest.mark.parametrize("scale", [1e-80, 1e-3, 1e60])
def test_scaled_units(scale):
    # momenta scaled by s and energies by s^2 (the reference state with them): L scales alike, far from one (s^3, the
    # size of the energy flux, has to be representable)
    k, cells = 3, (3, 3, 5)
    U = inputs.random_state(45, 64, 21).cuda()
    s = torch.tensor([1.0, scale, scale, scale, scale * scale], dtype=torch.float64, device="cuda")[None, :, None]
    kw = dict(R=287.0, Ma=0.1)
    a = api.DGCNS(cells, (-math.pi,) * 3, (math.pi,) * 3, (1, 1, 1), k, *NQ[k], U0=1.0, Re=1600.0, **kw)
    b = api.DGCNS(cells, (-math.pi,) * 3, (math.pi,) * 3, (1, 1, 1), k, *NQ[k], U0=scale, Re=1600.0, **kw)
    La, Lb = a.apply(U), b.apply((U * s).contiguous()) / (s * scale)
    two, mx = _err(Lb, La)
    assert two < 1e-12 and mx < 1e-12


@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
def test_non_finite_states(bad):
    f, e = _pair((5, 5, 5), 3)
    U = inputs.random_state(125, 64, 2).cuda()
    clean = f.apply(U).clone()
    U[62, 1, 5] = bad
    a, b = f.apply(U), e.apply(U)
    fa, fb = torch.isfinite(a).all(2), torch.isfinite(b).all(2)
    assert not fa[62].all()
    # every cell the general path spoils is spoilt here (not every row of it: at a NaN the LLF speed is the other
    # side's, and the two organisations take different sides as their own)
    assert not (fa.all(1) & ~fb.all(1)).any()
    far = torch.tensor([i for i in range(125) if abs(i % 5 - 2) + abs(i // 5 % 5 - 2) + abs(i // 25 - 2) > 2])
    assert torch.isfinite(a[far.cuda()]).all()
    two, _ = _err(a[far.cuda()], clean[far.cuda()])
    assert two < 1e-13
