"""The two-link build from FP32 slices gives the bits of the FP64 product rounded to nearest.

tls_export_twolink of an FP64 build returns the FP64 products; rounding them to FP32 on the host must
reproduce the FP32 build exactly: for random and near-unit SU(3) links, the free field (exact zeros
and ones), links scaled up or down (entries above the range of the slices, tiny entries), products on
and next to a rounding tie, signed zeros, and lattices with odd half extents.
"""

import numpy as np
import pytest
import torch

from paper_2301_05518_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def T():
    from paper_2301_05518_gb300 import tls as t
    return t


def _fields():
    rng = np.random.default_rng(9)
    haar = synth.gauge_haar((16, 12, 10, 3), 81, nd=3)
    yield "haar", haar
    yield "near", synth.gauge_near_unit((6, 10, 14, 2), 0.2, 82, nd=3)
    yield "unit", synth.gauge_unit((4, 6, 2, 2), nd=3)
    small = haar.clone()
    small *= torch.from_numpy(2.0 ** rng.integers(-70, 3, small.shape[:5] + (1, 1)).astype(np.float64))
    yield "scaled", small
    ties = torch.zeros((1, 4, 4, 8, 3, 3, 3), dtype=torch.complex128)
    base = rng.integers(2 ** 23, 2 ** 24, ties.shape) * 2.0 ** -24 + 2.0 ** -25  # halfway between two floats
    off = rng.choice([0.0, 2.0 ** -52, -2.0 ** -52, 2.0 ** -40, -2.0 ** -37, 2.0 ** -36], ties.shape)
    ties += torch.from_numpy((base + off) * rng.choice([-1.0, 1.0], ties.shape))
    for t in (ties,):  # odd sites along each direction: the identity (with signed zeros), so that W = U
        idx = torch.stack(torch.meshgrid(torch.arange(4), torch.arange(4), torch.arange(8), indexing="ij"))
        for d, ax in enumerate((2, 1, 0)):
            odd = (idx[ax] % 2 == 1)
            eye = torch.eye(3, dtype=torch.complex128)
            t[0, odd, d] = torch.complex(eye.real, torch.full((3, 3), -0.0, dtype=torch.float64))
    yield "ties", ties
    odd = haar.clone()
    odd[0, 0, 0, 0, 0, 0, 0] = complex(float("inf"), 1.0)
    odd[0, 1, 1, 1, 1, 2, 2] = complex(float("nan"), 0.0)
    odd[0, 2, 1, 1, 2, 1, 0] = 1.2
    odd[1, 2, 1, 1, 2, 1, 0] = 1.125
    yield "special", odd


@pytest.mark.parametrize("recon", [18, 12])
def test_build_bits_equal_rounded_fp64_product(T, recon):
    with T.Context(0) as ctx:
        for name, U in _fields():
            Lt, Lz, Ly, Lx = U.shape[:4]
            gid = ctx.load_gauge(U.contiguous().cuda(), 3, (Lx, Ly, Lz, Lt))
            ctx.build_twolink(gid, T.TLS_F64, 18)
            full = np.zeros((Lt, Lz, Ly, Lx, 3, 3, 3), dtype=np.complex128)
            ctx.export_twolink(gid, full)
            ctx.build_twolink(gid, T.TLS_F32, recon)
            got = np.zeros_like(full)
            ctx.export_twolink(gid, got)
            ctx.free_gauge(gid)
            rows = 3 if recon == 18 else 2  # the stored rows
            want = full[..., :rows, :].copy().view(np.float64).astype(np.float32)
            have = got[..., :rows, :].copy().view(np.float64).astype(np.float32)
            same = (want.view(np.uint32) == have.view(np.uint32)) | (np.isnan(want) & np.isnan(have))
            assert same.all(), (name, int((~same).sum()))
