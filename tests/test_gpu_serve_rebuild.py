"""A two-link field that serving jobs use is not rebuilt under them."""

import pytest
import torch

from paper_2301_05518_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("recon", [12, 18])
def test_rebuild_is_refused_while_jobs_use_the_field(recon):
    """In another format (the field is freed) and in the same one (it is overwritten): the call returns
    TLS_ERR_STATE, the job gets the bits of the field it was submitted with, and the rebuild runs
    once the job has been waited for."""
    from paper_2301_05518_gb300 import tls as T
    dims, N = (16, 16, 16, 8), 8000  # some tenths of a second of rounds
    with T.Context(0) as c:
        gid = c.load_gauge(synth.gauge_haar(dims, 61, nd=3).cuda(), 3, dims)
        c.build_twolink(gid, T.TLS_F32, 18)
        vecs = synth.gaussian_vectors(dims, 6, 62, dtype=torch.complex64)
        got, want = vecs.clone().cuda(), vecs.clone().cuda()
        c.smear(gid, want, T.TLS_F32, 6, N, 0.2 * N, kernel=T.TLS_KERNEL_MRHS)
        torch.cuda.synchronize()
        c.serve_start(max_slots=12, steps_per_launch=4, use_graphs=1)
        job = c.serve_submit(gid, got, T.TLS_F32, 6, N, 0.2 * N)
        for _ in range(3):  # queued, on its way to a batch, in one
            with pytest.raises(T.TLSError) as e:
                c.build_twolink(gid, T.TLS_F32, recon)
            assert e.value.status == T.TLS_ERR_STATE
        c.serve_wait(job, 60)
        assert torch.equal(got, want)
        c.build_twolink(gid, T.TLS_F32, recon)
        again, ref = vecs.clone().cuda(), vecs.clone().cuda()
        torch.cuda.synchronize()
        c.serve_wait(c.serve_submit(gid, again, T.TLS_F32, 6, 5, 1.0), 60)
        c.smear(gid, ref, T.TLS_F32, 6, 5, 1.0, kernel=T.TLS_KERNEL_MRHS)
        assert torch.equal(again, ref)
        c.serve_stop()
