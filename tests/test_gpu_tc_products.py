"""What the bounds of the prompt pass on tcgen05 rest on: accumulators hold sums of whole numbers exactly as
far as the pieces take them (2^23), and round other sums by at most 17 times 2^-23 of what they hold per step of 16 terms."""
import ctypes
import os
import subprocess

import numpy as np
import pytest
import torch

from paper_2404_15949_b200.build import NVCC_FLAGS

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("tc") / "tc_products.so")
    subprocess.check_call([os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")] + NVCC_FLAGS + ["-o", so, os.path.join(HERE, "tc_products.cu")])
    lib = ctypes.CDLL(so)
    lib.tc_products.argtypes = [ctypes.c_int] + [ctypes.c_void_p] * 4
    return lib


def bf16(x):
    return torch.from_numpy(np.asarray(x, np.float64)).to(torch.bfloat16).double().numpy()


def to_grid(x, step):
    return np.rint(x / step) * step                     # ties to even, as an addition of 1.5 2^n steps rounds


def pieces(q, k):
    """corm_mma.cuh's: rows on a grid of their own, keys by eights."""
    gq = 2.0 ** (np.floor(np.log2(np.abs(q).max(1, keepdims=True))) - 7)
    q1 = to_grid(q, gq)
    q2 = to_grid(q - q1, gq / 512)
    top = np.abs(k).reshape(8, 8, -1).max((1, 2)).repeat(8)[:, None]
    g = 2.0 ** (np.floor(np.log2(top)) - 5)
    k1 = to_grid(k, g)
    k2 = to_grid(k - k1, g / 128)
    return (q1, q2, q - q1 - q2), (k1, k2, k - k1 - k2), gq, g, top


def operands(what, d, rng):
    q, k = rng.standard_normal((128, d)), rng.standard_normal((64, d))
    if what == "one sign":
        q, k = np.abs(q) + 0.01, np.abs(k) + 0.01
    elif what == "near 2^23":                           # k2.q1: d times half a step of the keys' grid and the rows' largest numbers
        q, k = rng.integers(250, 256, (128, d)) / 128.0, (2 * rng.integers(16, 31, (64, d)) + 0.5) / 32.0
    elif what == "near 2^23, signs":
        q, k = rng.integers(250, 256, (128, d)) / 128.0, (2 * rng.integers(16, 31, (64, d)) + 0.5) / 32.0
        s = rng.choice([-1.0, 1.0], d)
        q, k = q * s, k * np.where(np.arange(d) < d - 8, s, -s)
    elif what == "wide":                                # elements over 2^20: all three pieces of rows and keys
        q, k = (x * 2.0 ** rng.integers(-20, 1, x.shape) for x in (q, k))
    return bf16(q), bf16(k)


@pytest.mark.parametrize("d", [128, 64])
@pytest.mark.parametrize("what", ["random", "one sign", "near 2^23", "near 2^23, signs", "wide"])
def test_accumulators(lib, what, d):
    rng = np.random.default_rng(d + len(what))
    for _ in range(10):
        q, k = operands(what, d, rng)
        (q1, q2, q3), (k1, k2, r2), gq, g, top = pieces(q, k)
        for x in (q1, q2, q3, k1, k2, r2):
            assert np.array_equal(bf16(x), x)
        rows, keys = (torch.from_numpy(np.stack(x)).to(torch.bfloat16).cuda() for x in ((q1, q2, q3, q), (k1, k2, r2, k)))
        out = torch.full((5, 128, 64), float("nan"), device="cuda")
        status = torch.zeros(1, dtype=torch.int32, device="cuda")
        assert lib.tc_products(d, rows.data_ptr(), keys.data_ptr(), out.data_ptr(), status.data_ptr()) == 0
        torch.cuda.synchronize()
        assert int(status) == 0
        acc = out.cpu().numpy().astype(np.float64)
        mid = q2 @ k1.T + q1 @ k2.T                     # fp64 holds these sums exactly as well
        units = np.abs(mid / (gq * g.T / 512)).max()
        assert units < 2.0 ** 24 and (not what.startswith("near") or units > 2.0 ** 22.5 * d / 128 * (0.8 if "signs" in what else 1))
        assert np.array_equal(acc[0], q1 @ k1.T) and np.array_equal(acc[1], mid) and np.array_equal(acc[2], q2 @ k2.T)
        n1, n2, n3 = (np.abs(x).sum(1, keepdims=True) for x in (q, q2, q3))
        a, step, n = top.T, 17.0 * 2.0 ** -23, d // 16
        # what has been added up so far is at most the sum of magnitudes: r2.q1's steps, r2.q2's before them, k1.q3's first
        bound = n * step * (n1 * a / 8192 + 2 * n2 * a / 8192 + 3 * n3 * a * 1.05)
        small = q3 @ k1.T + q2 @ r2.T + q1 @ r2.T
        assert (np.abs(acc[3] - small) <= bound).all(), (np.abs(acc[3] - small) / np.maximum(bound, 1e-300)).max()
        raw = n * step * n1 * a
        assert (np.abs(acc[4] - q @ k.T) <= raw).all(), (np.abs(acc[4] - q @ k.T) / raw).max()
