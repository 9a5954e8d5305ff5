"""The column kernel (tiles of rows marching along z') against one vector per launch, bitwise.

Every kernel performs the same FMA sequence per vector, so results are equal bit for bit for each
storage and W format.  The shapes sit at the edges: rows that are not a multiple of 16 bytes, rows
per tile that do not divide the block, one row, one plane, L = 2, odd vector counts (padded groups),
z' segments, one slice, and more than 256 vectors.
"""

import pytest
import torch

from paper_2301_05518_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def T():
    from paper_2301_05518_gb300 import tls as t
    return t


@pytest.fixture(scope="module")
def ctx(T):
    c = T.Context(0)
    yield c
    c.close()


# dims, nvec, storage, W precision, reals, tile shapes (vectors per group, rows, z' segments, units)
CASES = [
    ((8, 8, 8, 2), 8, "F32", "F32", 18, [(8, 2, 1, 0), (4, 4, 2, 3), (2, 1, 1, 0), (6, 4, 1, 0)]),
    ((10, 6, 4, 2), 5, "F32", "F32", 18, [(6, 3, 1, 0), (2, 2, 2, 0), (4, 1, 1, 4)]),
    ((2, 2, 2, 1), 3, "F32", "F32", 12, [(4, 1, 1, 0)]),
    ((14, 2, 6, 1), 2, "F32", "F32", 18, [(2, 1, 3, 0)]),
    ((12, 10, 2, 2), 6, "F16", "F16", 18, [(6, 5, 1, 0), (2, 3, 1, 0)]),
    ((6, 14, 6, 2), 6, "F16", "F16", 12, [(6, 3, 1, 0), (4, 7, 3, 0)]),
    ((14, 6, 10, 2), 4, "BF16", "BF16", 18, [(4, 3, 1, 0)]),
    ((10, 10, 10, 2), 7, "F32", "F32", 8, [(8, 5, 1, 0), (4, 2, 5, 0)]),
    ((8, 8, 6, 3), 9, "BF16", "F32", 12, [(10, 4, 1, 0)]),
    ((64, 12, 8, 1), 24, "F32", "F32", 18, [(24, 1, 1, 0), (12, 2, 2, 0), (8, 3, 1, 3)]),
    ((34, 12, 8, 1), 24, "F16", "F32", 18, [(8, 5, 1, 0)]),
]


@pytest.mark.parametrize("dims,nvec,storage,wprec,recon,shapes", CASES)
def test_column_kernel_bitwise_equals_single(ctx, T, dims, nvec, storage, wprec, recon, shapes):
    U = synth.gauge_haar(dims, 51, nd=3)
    vecs = synth.gaussian_vectors(dims, nvec, 52, dtype=torch.complex64)
    st = getattr(T, "TLS_" + storage)
    gid = ctx.load_gauge(U, 3, dims)
    ctx.build_twolink(gid, getattr(T, "TLS_" + wprec), recon)
    for t0 in (-1, dims[3] - 1):
        want = vecs.clone().cuda()
        ctx.smear(gid, want, T.TLS_F32, nvec, 5, 1.1, timeslice=t0, storage=st, kernel=T.TLS_KERNEL_SINGLE)
        for nvg, ny, nseg, units in shapes:
            ctx.tune_set(gid, nvec, st, t0, T.TLS_KERNEL_MRHS, 2, 0, (nvg, 9, ny | nseg << 8 | units << 16))
            got = vecs.clone().cuda()
            ctx.smear(gid, got, T.TLS_F32, nvec, 5, 1.1, timeslice=t0, storage=st)
            assert torch.equal(got, want), (t0, nvg, ny, nseg, units)
    ctx.free_gauge(gid)


@pytest.mark.parametrize("dims,nvec,storage", [((16, 16, 16, 8), 3, "F32"), ((30, 18, 22, 4), 7, "F32"),
                                               ((32, 32, 32, 4), 12, "F16"), ((24, 24, 24, 8), 72, "F32"),
                                               ((50, 10, 10, 2), 24, "BF16"), ((8, 8, 4, 2), 301, "F32"),
                                               ((4, 4, 4, 2), 1, "F32"), ((16, 16, 16, 32), 4, "F32"),
                                               ((10, 6, 8, 3), 2, "F16"), ((6, 6, 10, 2), 3, "F64"),
                                               ((16, 8, 8, 2), 4, "F64")])
def test_planner_choice_bitwise_equals_single(ctx, T, dims, nvec, storage):
    """Without a tune entry the planner picks the kernel and the tile shape: same results, host
    buffers included."""
    U = synth.gauge_haar(dims, 53, nd=3)
    f64 = storage == "F64"
    vecs = synth.gaussian_vectors(dims, nvec, 54, dtype=torch.complex128 if f64 else torch.complex64)
    st = getattr(T, "TLS_" + storage)
    io = T.TLS_F64 if f64 else T.TLS_F32
    gid = ctx.load_gauge(U, 3, dims)
    ctx.build_twolink(gid, io, 18)
    for t0 in (-1, 1):
        want = vecs.clone().cuda()
        nw = ctx.smear(gid, want, io, nvec, 4, 0.9, timeslice=t0, storage=st, kernel=T.TLS_KERNEL_SINGLE,
                       norms=True)
        for kern in (T.TLS_KERNEL_AUTO, T.TLS_KERNEL_MRHS):
            got = vecs.clone().cuda()
            ng = ctx.smear(gid, got, io, nvec, 4, 0.9, timeslice=t0, storage=st, kernel=kern, norms=True)
            assert torch.equal(got, want) and (ng == nw).all()
        host = vecs.clone()
        ctx.smear(gid, host, io, nvec, 4, 0.9, timeslice=t0, storage=st)
        assert torch.equal(host, want.cpu())
    ctx.free_gauge(gid)


@pytest.mark.parametrize("records,slack", [(50, 1 << 17), (60, 1 << 13)])
def test_padded_groups_do_not_cost_admission(T, records, slack):
    """A smear whose buffers fit under the HBM cap runs although the padded vector groups of the
    column kernel (60 records), or what is allocated after them, would not fit."""
    dims, nvec = (16, 16, 16, 8), 49
    bufs = 2 * records * 24 * 16 ** 3 * 8      # two packed buffers
    fixed = 3 * 144 * 16 ** 3 * 8 + 216 * 16 ** 3 * 8
    with T.Context(0, hbm_cap_bytes=bufs + fixed + slack) as c:
        gid = c.load_gauge(synth.gauge_haar(dims, 55, nd=3).cuda(), 3, dims)
        c.build_twolink(gid, T.TLS_F32, 18)
        c.tune_set(gid, nvec, T.TLS_F32, T.TLS_ALL_T, T.TLS_KERNEL_MRHS, 2, 0, (12, 9, 4 | 1 << 8))
        x = synth.gaussian_vectors(dims, nvec, 56, dtype=torch.complex64).cuda()
        want = x.clone()
        c.smear(gid, want[:7].contiguous(), T.TLS_F32, 7, 3, 0.6, kernel=T.TLS_KERNEL_SINGLE)
        one = want[7:8].contiguous()
        c.smear(gid, one, T.TLS_F32, 1, 3, 0.6, kernel=T.TLS_KERNEL_SINGLE)
        c.smear(gid, x, T.TLS_F32, nvec, 3, 0.6, norms=True)
        assert torch.equal(x[7:8], one)


def test_serving_batch_follows_a_rebuilt_field(T):
    """An idle batch made for one two-link field is not reused after tls_build_twolink replaced it."""
    dims = (16, 16, 16, 4)
    with T.Context(0) as c:
        gid = c.load_gauge(synth.gauge_haar(dims, 57, nd=3).cuda(), 3, dims)
        vecs = synth.gaussian_vectors(dims, 5, 58, dtype=torch.complex64)
        c.build_twolink(gid, T.TLS_F32, 18)
        c.serve_start(max_slots=12, steps_per_launch=2, use_graphs=1)
        for recon in (18, 12, 18):
            c.build_twolink(gid, T.TLS_F32, recon)
            got, want = vecs.clone().cuda(), vecs.clone().cuda()
            torch.cuda.synchronize()
            c.serve_wait(c.serve_submit(gid, got, T.TLS_F32, 5, 7, 1.4), 60)
            c.smear(gid, want, T.TLS_F32, 5, 7, 1.4, kernel=T.TLS_KERNEL_MRHS)
            assert torch.equal(got, want)
        c.serve_stop()
