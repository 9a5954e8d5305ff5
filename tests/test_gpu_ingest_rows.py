"""Links of lattices with short rows: tls_load_gauge and tls_export_gauge give the links back bit for bit."""

import pytest
import torch

pytestmark = pytest.mark.gpu


# rows together (the last CTA full or not, planes that its rows do and do not divide), and by themselves
@pytest.mark.parametrize("dims", [(2, 96, 96, 4), (2, 34, 34, 10), (4, 50, 38, 6), (6, 62, 50, 3), (6, 10, 6, 90), (2, 4, 4, 3),
                                  (8, 10, 10, 40), (66, 6, 6, 4)])
@pytest.mark.parametrize("nd", [3, 4])
def test_round_trip(dims, nd):
    from paper_2301_05518_gb300 import tls as T
    Lx, Ly, Lz, Lt = dims
    g = torch.Generator().manual_seed(5)
    U = torch.view_as_complex(torch.randn((Lt, Lz, Ly, Lx, nd, 3, 3, 2), generator=g, dtype=torch.float64))
    with T.Context(0) as c:
        for u in (U.cuda(), U):
            gid = c.load_gauge(u, nd, dims)
            out = torch.zeros((Lt, Lz, Ly, Lx, 3, 3, 3), dtype=torch.complex128, device="cuda")
            c.export_gauge(gid, out)
            assert torch.equal(out.cpu(), U[..., :3, :, :])
            c.free_gauge(gid)
