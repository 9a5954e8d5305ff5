"""One-link smearing of FP32 and 16-bit vectors on whole slices (the two-link step kernels with
+-1 hops in canonical order): the column kernel, the row kernel and, on rows longer than a CTA, the
plain interleaved kernel, against the FP64 oracle.  Tolerances as for every other smear."""

import numpy as np
import pytest
import torch

import oracle
from helpers import per_vector_rel_l2
from paper_2301_05518_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,nvec,storage,t0", [((32, 24, 16, 3), 12, "F32", -1), ((260, 2, 2, 1), 3, "F32", -1),
                                                  ((64, 16, 8, 2), 24, "F16", 1), ((16, 16, 16, 8), 41, "BF16", -1),
                                                  ((14, 10, 6, 2), 1, "F32", 0), ((2, 2, 2, 2), 5, "F32", -1),
                                                  ((48, 32, 32, 2), 7, "F32", -1)])
def test_onelink_on_slices_matches_oracle(dims, nvec, storage, t0):
    from paper_2301_05518_gb300 import tls as T
    U = synth.gauge_haar(dims, 61, nd=3)
    vecs = synth.gaussian_vectors(dims, nvec, 62, dtype=torch.complex64)
    N, alpha = 5, 0.06
    want = oracle.smear_onelink(U.numpy(), vecs.numpy().astype(np.complex128), N, alpha, t0=t0)
    st = getattr(T, "TLS_" + storage)
    with T.Context(0) as ctx:
        gid = ctx.load_gauge(U, 3, dims)
        ctx.build_links(gid, T.TLS_F32)
        x = vecs.clone().cuda()
        norms = ctx.smear_onelink(gid, x, T.TLS_F32, nvec, N, alpha, timeslice=t0, storage=st, norms=True)
        host = vecs.clone()
        ctx.smear_onelink(gid, host, T.TLS_F32, nvec, N, alpha, timeslice=t0, storage=st)
        assert torch.equal(host, x.cpu())
        ctx.free_gauge(gid)
    got = x.cpu().numpy().astype(np.complex128)
    assert max(per_vector_rel_l2(got, want)) <= (2e-6 * N if storage == "F32" else 5e-3)
    sl = slice(None) if t0 < 0 else slice(t0, t0 + 1)
    assert np.allclose(norms, (np.abs(got[:, sl]) ** 2).reshape(nvec, -1).sum(1), rtol=1e-12, atol=0)


def test_onelink_batch_past_32_bit_offsets():
    """Rows too long for a CTA of the column or row kernel, and a batch whose records of one slice
    pass 4 GiB: every vector as in a batch of two."""
    from paper_2301_05518_gb300 import tls as T
    dims, nvec = (520, 64, 64, 1), 132
    with T.Context(0) as ctx:
        gid = ctx.load_gauge(synth.gauge_haar(dims, 63, nd=3), 3, dims)
        ctx.build_links(gid, T.TLS_F32)
        torch.manual_seed(64)
        x = torch.randn((nvec, 1, 64, 64, 520, 3), dtype=torch.complex64, device="cuda")
        pairs = [x[v:v + 2].clone() for v in (0, 124, 126, 130)]
        ctx.smear_onelink(gid, x, T.TLS_F32, nvec, 2, 0.05, storage=T.TLS_F16)
        for v, y in zip((0, 124, 126, 130), pairs):
            ctx.smear_onelink(gid, y, T.TLS_F32, 2, 2, 0.05, storage=T.TLS_F16)
            assert torch.equal(x[v:v + 2], y), v
        ctx.free_gauge(gid)
