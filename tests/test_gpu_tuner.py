"""What the autotuner offers: every kernel that won at some measured shape, the fastest one kept."""

import pytest
import torch

from paper_2301_05518_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("recon,nvec", [(18, 8), (12, 8), (8, 16), (12, 5), (18, 2)])
def test_candidates(recon, nvec):
    from paper_2301_05518_gb300 import tls as T
    dims = (16, 12, 12, 4)
    vecs = synth.gaussian_vectors(dims, nvec, 92, dtype=torch.complex64).cuda()
    with T.Context(0) as c:
        gid = c.load_gauge(synth.gauge_haar(dims, 91, nd=3).cuda(), 3, dims)
        c.build_twolink(gid, T.TLS_F32, recon)
        best, every = c.autotune(gid, nvec, T.TLS_F32, steps=2)
        tiles = {(e["vecs_per_thread"], tuple(e["tile"])) for e in every if e["kernel"] == T.TLS_KERNEL_MRHS}
        for tile in ((0, 0, 0), (0, 2, 0), (0, 6, 0), (0, 6, -1), (0, 7, 0), (0, 8, 0)):
            assert any(t == tile for _, t in tiles), tile
        eight = {t for vb, t in tiles if vb == 8 and t[1] != 10}
        assert eight == ({(0, 6, 0), (0, 7, 0), (0, 7, -1)} if recon != 18 and nvec % 8 == 0 else set())
        assert best["ms_per_step"] == min(e["ms_per_step"] for e in every)
        want, got = vecs.clone(), vecs.clone()
        c.smear(gid, want, T.TLS_F32, nvec, 4, 0.8, kernel=T.TLS_KERNEL_SINGLE)
        c.smear(gid, got, T.TLS_F32, nvec, 4, 0.8)
        assert torch.equal(got, want)
