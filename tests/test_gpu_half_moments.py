"""Density and velocity of half-storage lattices (two cells per thread) against the moments of the
exported populations, for rows that end inside a pair or a warp, all boundary types, the layouts
of AA after even and odd steps and of pull, and output arrays that are not 8-byte aligned."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
CHANNEL = ("periodic", "periodic", "wall", "wall", "periodic", "periodic")
TUNNEL = ("inflow", "outflow", "freeslip", "freeslip", "freeslip", "freeslip")


@pytest.mark.parametrize("q,precision,streaming", [(19, "f16", "aa"), (19, "bf16", "pull"), (27, "f16", "pull"), (27, "bf16", "aa")])
@pytest.mark.parametrize("nx,faces", [(2, CHANNEL), (31, CHANNEL), (64, CHANNEL), (98, TUNNEL), (127, TUNNEL), (130, CHANNEL)])
def test_moments_match_populations(nx, faces, q, precision, streaming):
    import torch

    from paper_2305_09910_gb300 import lbm

    ny, nz = 7, 5
    rng = np.random.default_rng(nx * q)
    lat = lbm.Lattice(nx, ny, nz, stencil=q, tau=0.6, faces=faces, u_inflow=(0.05, 0, 0), streaming=streaming,
                      precision=precision)
    flags = (rng.random((nz, ny, nx)) < 0.03).astype(np.uint8)
    lat.set_flags(flags)
    lat.set_force(1e-5, 2e-5, -1e-5)
    lat.init_equilibrium(rng.uniform(0.98, 1.02, (nz, ny, nx)).astype(np.float32),
                         rng.uniform(-0.05, 0.05, (3, nz, ny, nx)).astype(np.float32))
    c, _ = lbm.lbm_stencil(q)
    force = np.array([1e-5, 2e-5, -1e-5])
    n = nx * ny * nz
    store = torch.full((4 * n + 2,), 7.0, device="cuda")
    for _ in range(3):
        df = lat.get_populations().astype(np.float64)
        rho = 1.0 + df.sum(0)
        u = (np.einsum("qa,qzyx->azyx", c, df) + 0.5 * force[:, None, None, None]) / rho
        for off in (0, 1):  # 1: arrays at odd multiples of 4 bytes
            r, v = store[off:off + n].view(nz, ny, nx), store[off + n:off + 4 * n].view(3, nz, ny, nx)
            r.fill_(7.0)
            v.fill_(7.0)
            lbm.lbm_moments(lat.h, r, v)
            got_r, got_u = r.cpu().numpy(), v.cpu().numpy()
            fluid = flags == 0
            # q additions of values below 0.4 in float32 (sum of magnitudes below 1), then a division
            assert np.abs(got_r - rho)[fluid].max() <= (q + 2) * 2.0 ** -24
            assert np.abs(got_u - u)[:, fluid].max() <= 2 * (q + 4) * 2.0 ** -24
            assert np.all(got_r[~fluid] == 0) and np.all(got_u[:, ~fluid] == 0)
        lat.step(1)
    lat.close()
