"""Pack and unpack of the interleaved records: what goes in comes out, whatever the split of the work."""

import pytest
import torch

from paper_2301_05518_gb300 import synth

pytestmark = pytest.mark.gpu


# rows that do and do not divide a slice, more and fewer pairs than a chunk, odd counts (half pairs)
@pytest.mark.parametrize("dims,nvec", [((2, 2, 2, 1), 1), ((4, 6, 10, 3), 9), ((12, 10, 6, 2), 72), ((6, 6, 14, 2), 33),
                                       ((66, 4, 6, 1), 7), ((10, 2, 2, 2), 255), ((34, 6, 2, 1), 24), ((4, 4, 4, 2), 300)])
@pytest.mark.parametrize("io", ["F32", "F64"])
def test_round_trip(dims, nvec, io):
    """No smearing step (N = 0): FP32 vectors come back bit for bit; 16-bit storage gives the values of
    one vector per launch, whose pack and unpack are other kernels; other slices stay as they are."""
    from paper_2301_05518_gb300 import tls as T
    dt = torch.complex64 if io == "F32" else torch.complex128
    prec = getattr(T, "TLS_" + io)
    vecs = synth.gaussian_vectors(dims, nvec, 71, dtype=torch.complex64).to(dt).cuda()
    with T.Context(0) as c:
        gid = c.load_gauge(synth.gauge_haar(dims, 70, nd=3).cuda(), 3, dims)
        c.build_twolink(gid, T.TLS_F32, 18)
        for storage in (T.TLS_F32, T.TLS_F16, T.TLS_BF16):
            for t0 in (-1, dims[3] - 1):
                want = vecs.clone()
                c.smear(gid, want, prec, nvec, 0, 0.0, timeslice=t0, storage=storage, kernel=T.TLS_KERNEL_SINGLE)
                if storage == T.TLS_F32:
                    assert torch.equal(want, vecs)
                for tile in ((0, 6, 0), (8, 9, 1 | 1 << 8), (24, 9, 1 | 1 << 8), (2, 9, 1 | 1 << 8)):
                    c.tune_set(gid, nvec, storage, t0, T.TLS_KERNEL_MRHS, 2, 0, tile)
                    got = vecs.clone()
                    c.smear(gid, got, prec, nvec, 0, 0.0, timeslice=t0, storage=storage)
                    assert torch.equal(got, want), (storage, t0, tile)
