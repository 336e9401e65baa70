"""FP64 reciprocal and square root of the point fluxes against CUDA's own division and square root."""
import ctypes
import os
import subprocess

import numpy as np
import pytest
import torch

from paper_1806_03095_gb300 import build

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("device_functions") / "device_functions.so")
    subprocess.check_call([build.nvcc(), *build.ARCH, *build.FLAGS, "-shared", "--cudart", "static",
                           os.path.join(HERE, "device_functions.cu"), "-o", so])
    return ctypes.CDLL(so)


def _apply(lib, kind, x):
    x = torch.as_tensor(np.asarray(x, dtype=np.float64)).cuda()
    mine, ref = torch.empty_like(x), torch.empty_like(x)
    torch.cuda.synchronize()
    ptr = [ctypes.c_void_p(t.data_ptr()) for t in (x, mine, ref)]
    assert lib.point_function(kind, x.numel(), *ptr) == 0
    return mine.cpu().numpy(), ref.cpu().numpy()


def _random(kind, n=1 << 20):
    rng = np.random.default_rng(23 + kind)
    x = (1.0 + rng.random(n)) * np.exp2(rng.integers(-1000, 980, n).astype(np.float64))
    x[: n // 2] = 1.0 + 3.0 * rng.random(n // 2)  # every mantissa and both parities of the exponent, often
    return x if kind == 1 else x * rng.choice([-1.0, 1.0], n)


@pytest.mark.parametrize("kind,share", [(0, 2 * 2.0 ** -7), (1, 2 * 2.0 ** -5.5)])
def test_error_bound(lib, kind, share):
    # an error below 1/2 + d ulp: at most one unit from the correctly rounded value, and another value than that only
    # where the exact one lies within d ulp of a midpoint, 2 d of the random arguments
    mine, ref = _apply(lib, kind, _random(kind))
    off = np.abs(mine.view(np.int64) - ref.view(np.int64))
    assert off.max() <= 1
    assert (off != 0).mean() <= share


def test_exact_values(lib):
    n = np.arange(1, 200001, dtype=np.float64) * 12345.0
    for s in (1.0, 2.0 ** -400, 2.0 ** 400):
        mine, _ = _apply(lib, 1, (n * s) ** 2)
        assert np.array_equal(mine, n * s)
    p = np.exp2(np.arange(-990, 991).astype(np.float64))
    mine, _ = _apply(lib, 0, p)
    assert np.array_equal(mine, 1.0 / p)


@pytest.mark.parametrize("kind", [0, 1])
def test_edges_of_the_range(lib, kind):
    # around the first and last high word that takes the seed, and everything beyond it: CUDA's result
    words = [0x00000000, 0x00000001, 0x000FFFFF, 0x00100000, 0x00FFFFFF, 0x01000000, 0x01000001, 0x7DFFFFFF, 0x7E000000,
             0x7E000001, 0x7FE00000, 0x7FEFFFFF]
    lows = np.array([0, 1, 0x80000000, 0xFFFFFFFF], dtype=np.uint64)
    x = np.concatenate([(np.uint64(w) << np.uint64(32) | lows) for w in words]).view(np.float64)
    mine, ref = _apply(lib, kind, x)
    inside = (x.view(np.uint64) >> np.uint64(32) >= 0x01000000) & (x.view(np.uint64) >> np.uint64(32) <= 0x7E000000)
    assert np.array_equal(mine[~inside].view(np.int64), ref[~inside].view(np.int64))
    assert np.abs(mine[inside].view(np.int64) - ref[inside].view(np.int64)).max() <= 1
    special = np.array([0.0, -0.0, np.inf, -np.inf, np.nan, -1.0, -1e-320])
    mine, ref = _apply(lib, kind, special)
    same = (mine.view(np.int64) == ref.view(np.int64)) | (np.isnan(mine) & np.isnan(ref))
    if kind == 0:
        same[5] = mine[5] == ref[5]
    assert same.all(), (special, mine, ref)
