"""Two-link build of links with exact zeros: the bits of the rounded FP64 product.

Elements whose products all have a zero factor are written as +0 without the FP64 chain.  Diagonal and
SU(2) links, single zeros and signed zeros in random links, entries too small for the FP32 slices next to
zeros, and infinities and NaN that meet a zero (0 * inf is not 0).
"""

import numpy as np
import pytest
import torch

from paper_2301_05518_gb300 import synth

pytestmark = pytest.mark.gpu


def _fields():
    rng = np.random.default_rng(11)
    shape = (2, 6, 10, 14, 3, 3, 3)
    haar = synth.gauge_haar((14, 10, 6, 2), 83, nd=3)
    diag = torch.zeros(shape, dtype=torch.complex128)
    ph = torch.from_numpy(rng.uniform(0, 2 * np.pi, shape[:5] + (3,)))
    for k in range(3):
        diag[..., k, k] = torch.polar(torch.ones_like(ph[..., k]), ph[..., k])
    yield "diagonal", diag
    su2 = haar.clone()
    su2[..., 2, :2] = 0
    su2[..., :2, 2] = 0
    yield "block", su2
    perm = torch.zeros_like(diag)  # rows permuted, with phases 1, -1, i, -i
    p = torch.from_numpy(rng.permuted(np.tile(np.arange(3), (int(np.prod(shape[:5])), 1)), axis=1)).reshape(shape[:5] + (3,))
    perm.scatter_(-1, p[..., None], torch.from_numpy(rng.choice([1, -1, 1j, -1j], shape[:5] + (3, 1))).to(torch.complex128))
    yield "permutations", perm
    holes = haar.clone()
    v = torch.view_as_real(holes)
    v[torch.from_numpy(rng.random(v.shape) < 0.5)] = 0.0
    v[torch.from_numpy(rng.random(v.shape) < 0.2)] = -0.0
    yield "holes", holes
    tiny = holes.clone()
    t = torch.view_as_real(tiny)
    t[torch.from_numpy(rng.random(t.shape) < 0.3)] *= 2.0 ** -70
    t[torch.from_numpy(rng.random(t.shape) < 0.1)] = 5e-324
    yield "tiny", tiny
    bad = diag.clone()
    b = torch.view_as_real(bad)
    b[torch.from_numpy(rng.random(b.shape) < 0.02)] = float("inf")
    b[torch.from_numpy(rng.random(b.shape) < 0.02)] = float("nan")
    yield "infinite", bad


@pytest.mark.parametrize("recon", [18, 12])
def test_zeros(recon):
    from paper_2301_05518_gb300 import tls as T
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
            with np.errstate(over="ignore", under="ignore"):
                want = full[..., :rows, :].copy().view(np.float64).astype(np.float32)
            have = got[..., :rows, :].copy().view(np.float64).astype(np.float32)
            same = (want.view(np.uint32) == have.view(np.uint32)) | (np.isnan(want) & np.isnan(have))
            assert same.all(), (name, int((~same).sum()))
