"""Kernels that are launched while their predecessor on the stream still runs (programmatic dependent launch): the
arrays the predecessor writes may not be read before the wait.  On the host: no such array is declared constant for the
whole kernel.  On the GPU: stages launched back to back give the bits of stages synchronised one by one."""
import math
import os
import re

import pytest
import torch

from paper_1806_03095_gb300 import build

DEPENDENT = ("dg_coll_cell_kernel", "dg_coll_face_kernel", "dg_face_task_kernel", "dg_dev_kernel")
# the functions those kernels hand the state, the deviation state or the face shares to
HELPERS = ("coll_face_terms", "lift_body", "lift_fp64", "chain_lift_dir", "chain_lift", "face_task_body", "face_traces",
           "stage_update")
STATE = r"(?:double|float|T)\s*\*\s*__restrict__\s*(?:U|Ud|F|FB|FBuf|D|src|dU|Uout|Rout)\b"


def _sources():
    return "\n".join(open(os.path.join(build.CSRC, n)).read() for n in sorted(os.listdir(build.CSRC))
                     if n.endswith((".cuh", ".cu", ".h")))


def _definition(text, name):
    """Parameter list and body of the function `name`."""
    m = re.search(r"\b%s\(([^;{]*?)\)\s*\{" % name, text)
    depth, i = 1, m.end()
    while depth:
        depth += {"{": 1, "}": -1}.get(text[i], 0)
        i += 1
    return m.group(1), text[m.end():i]


def test_every_dependent_kernel_is_known():
    text = _sources()
    found = set()
    for m in re.finditer(r"\b(dg_\w+_kernel)\(const KParams kp", text):
        if "wait_for_predecessor()" in _definition(text, m.group(1))[1]:
            found.add(m.group(1))
    assert found == set(DEPENDENT)


@pytest.mark.parametrize("name", DEPENDENT + HELPERS)
def test_state_arrays_are_not_declared_constant(name):
    params, body = _definition(_sources(), name)
    assert not re.search(STATE, params), params
    assert not re.search(STATE, body)


@pytest.mark.gpu
@pytest.mark.parametrize("cells", [(1, 1, 1), (3, 2, 3), (8, 8, 8), (13, 7, 11)])
@pytest.mark.parametrize("k,precision", [(1, 0), (2, 0), (3, 0), (5, 0), (3, 1), (4, 1), (5, 1)])
def test_stages_back_to_back_equal_synchronised_stages(cells, k, precision):
    from paper_1806_03095_gb300 import api, inputs
    g = api.DGCNS(cells, (-math.pi,) * 3, (math.pi,) * 3, (1, 1, 1), k, (3 * k) // 2 + 1, k + 1, precision=precision)
    U = inputs.random_state(g.n_cells, g.n ** 3, 3).cuda()
    out = []
    for wait in (False, True):
        for in_place in (False, True):
            a, b, dU = U.clone(), torch.empty_like(U), g.empty_residual().zero_()
            for i in range(30):
                g.rk_stage(i % 5, 1e-5, 0.0, a, dU, a if in_place else b)
                if not in_place:
                    a, b = b, a
                if wait:
                    torch.cuda.synchronize()
            out.append((a, dU))
    torch.cuda.synchronize()
    assert torch.isfinite(out[0][0]).all()
    for a, dU in out[1:]:
        assert torch.equal(a, out[0][0]) and torch.equal(dU, out[0][1])
