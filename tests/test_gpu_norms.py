"""Norms: a vector's norm has the same bits alone and in a batch, from device and from host vectors."""

import pytest
import torch

from paper_2301_05518_gb300 import synth

pytestmark = pytest.mark.gpu


# one subset of the slice per part (small slices, fewer reals than threads among them), four spread over
# a cluster (few vectors) and four in one CTA (many), slices on both sides of the line between them
@pytest.mark.parametrize("dims,nvec", [((2, 2, 2, 3), 30), ((10, 6, 4, 2), 5), ((28, 28, 26, 1), 80), ((28, 28, 28, 1), 80),
                                       ((34, 30, 26, 2), 40), ((48, 32, 32, 2), 40)])
@pytest.mark.parametrize("io", ["F32", "F64"])
def test_norms_of_a_batch_are_those_of_its_vectors(dims, nvec, io):
    from paper_2301_05518_gb300 import tls as T
    prec = getattr(T, "TLS_" + io)
    dt = torch.complex64 if io == "F32" else torch.complex128
    vecs = synth.gaussian_vectors(dims, nvec, 81, dtype=torch.complex64).to(dt)
    # partial sums of at most n / 4096 + 16 roundings of 2^-53 each, all terms positive
    n = 6 * dims[0] * dims[1] * dims[2]
    tol = (n / 4096 + 16 + 16 * dims[3]) * 2.0 ** -53
    with T.Context(0) as c:
        gid = c.load_gauge(synth.gauge_near_unit(dims, 0.2, 80, nd=3).cuda(), 3, dims)
        c.build_twolink(gid, T.TLS_F32, 18)
        for t0 in (-1, dims[3] - 1):
            x = vecs.clone().cuda()
            got = c.smear(gid, x, prec, nvec, 0, 0.0, timeslice=t0, norms=True)
            part = vecs if t0 < 0 else vecs[:, t0:t0 + 1]
            want = (torch.view_as_real(part).double() ** 2).reshape(nvec, -1).sum(1).numpy()
            assert (abs(got - want) <= 2 * tol * want).all()
            for v in (0, nvec - 1):
                one = vecs[v:v + 1].clone().cuda()
                assert c.smear(gid, one, prec, 1, 0, 0.0, timeslice=t0, norms=True)[0] == got[v]
            host = vecs.clone()
            assert (c.smear(gid, host, prec, nvec, 0, 0.0, timeslice=t0, norms=True) == got).all()
