"""Density and velocity of half-storage D3Q19 lattices large enough that gathered layouts too take two
cells per thread, against the moments of the exported populations in float64."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
CHANNEL = ("periodic", "periodic", "wall", "wall", "periodic", "periodic")
TUNNEL = ("inflow", "outflow", "freeslip", "freeslip", "freeslip", "freeslip")


@pytest.mark.parametrize("nx,ny,nz,precision,streaming,faces", [
    (66, 128, 161, "f16", "pull", CHANNEL), (67, 128, 160, "bf16", "aa", CHANNEL), (98, 127, 130, "f16", "aa", TUNNEL),
    (127, 126, 129, "bf16", "pull", TUNNEL)])
def test_moments_of_large_lattices(nx, ny, nz, precision, streaming, faces):
    import torch

    from paper_2305_09910_gb300 import lbm

    q, n = 19, nx * ny * nz
    g = torch.Generator(device="cuda").manual_seed(nx)
    flags = (torch.rand((nz, ny, nx), generator=g, device="cuda") < 0.01).to(torch.uint8)
    lat = lbm.Lattice(nx, ny, nz, stencil=q, tau=0.6, faces=faces, u_inflow=(0.05, 0, 0), streaming=streaming,
                      precision=precision)
    lat.set_flags(flags.cpu().numpy())
    lat.set_force(1e-5, 2e-5, -1e-5)
    lat.init_equilibrium((0.98 + 0.04 * torch.rand((nz, ny, nx), generator=g, device="cuda")),
                         0.1 * torch.rand((3, nz, ny, nx), generator=g, device="cuda") - 0.05)
    c = torch.from_numpy(lbm.lbm_stencil(q)[0]).double().cuda()
    force = torch.tensor([1e-5, 2e-5, -1e-5], dtype=torch.float64, device="cuda")
    pops, store = torch.zeros((q, nz, ny, nx), device="cuda"), torch.full((4 * n + 2,), 7.0, device="cuda")
    fluid = flags == 0
    lat.step(1)
    for _ in range(2):
        lbm.lbm_get_populations(lat.h, pops)
        df = pops.double()
        rho = 1.0 + df.sum(0)
        u = (torch.einsum("qa,qzyx->azyx", c, df) + 0.5 * force[:, None, None, None]) / rho
        for off in (0, 1):  # 1: arrays at odd multiples of 4 bytes
            r, v = store[off:off + n].view(nz, ny, nx), store[off + n:off + 4 * n].view(3, nz, ny, nx)
            r.fill_(7.0)
            v.fill_(7.0)
            lbm.lbm_moments(lat.h, r, v)
            # q additions of values below 0.4 in float32 (sum of magnitudes below 1), then a division
            assert (r - rho)[fluid].abs().max().item() <= (q + 2) * 2.0 ** -24
            assert (v - u)[:, fluid].abs().max().item() <= 2 * (q + 4) * 2.0 ** -24
            assert r[~fluid].eq(0).all() and v[:, ~fluid].eq(0).all()
        lat.step(1)
    lat.close()
