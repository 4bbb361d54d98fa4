"""lbm_reduce and lbm_stats_sample over row counts and row lengths around the work split of the sum
kernel (several rows per block with a remainder, more or fewer row segments than a block's 4 warps,
ragged rows, solid cells, an outflow column), against float64 sums of the exported fields."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
CHANNEL = ("periodic", "periodic", "wall", "wall", "periodic", "periodic")
TUNNEL = ("inflow", "outflow", "freeslip", "freeslip", "freeslip", "freeslip")


@pytest.mark.parametrize("nx,ny,nz,q,streaming,precision,faces", [
    (7, 3, 2, 19, "aa", "f32", CHANNEL), (33, 83, 61, 19, "pull", "f32", CHANNEL), (96, 71, 73, 19, "aa", "f32", CHANNEL),
    (160, 50, 101, 27, "pull", "f16", CHANNEL), (290, 20, 9, 19, "pull", "bf16", TUNNEL), (62, 90, 113, 27, "aa", "f32", TUNNEL)])
def test_sums_match_the_exported_fields(nx, ny, nz, q, streaming, precision, faces):
    from paper_2305_09910_gb300 import lbm

    rng = np.random.default_rng(nx)
    with lbm.Lattice(nx, ny, nz, stencil=q, tau=0.6, faces=faces, u_inflow=(0.05, 0, 0), streaming=streaming,
                     precision=precision) as lat:
        flags = (rng.random((nz, ny, nx)) < 0.03).astype(np.uint8)
        lat.set_flags(flags)
        lat.set_force(1e-5, 2e-5, 0.0)
        lat.init_equilibrium(rng.uniform(0.99, 1.01, (nz, ny, nx)).astype(np.float32),
                             rng.uniform(-0.05, 0.05, (3, nz, ny, nx)).astype(np.float32))
        for steps in (0, 1, 2):
            lat.step(min(steps, 1))
            rho, u = lat.moments()
            fluid = flags == 0
            got = lat.reduce()
            n = int(fluid.sum())
            # every density is the rounding of 1 + drho (half an ulp of values below 2); j = rho u
            # within three float32 roundings of products below 0.06
            assert abs(got[0] - rho[fluid].astype(np.float64).sum()) <= n * 2.0 ** -24 + 1e-9
            for a in range(3):
                j = (rho.astype(np.float64) * u[a])[fluid].sum()
                assert abs(got[1 + a] - j) <= n * 0.06 * 3 * 2.0 ** -24 + 1e-9
            lbm.lbm_stats_reset(lat.h)
            lbm.lbm_stats_sample(lat.h)
            st, _ = lbm.lbm_stats_get(lat.h, ny)
            prod = [u[0] * u[0], u[1] * u[1], u[2] * u[2], u[0] * u[1], u[0] * u[2], u[1] * u[2]]
            want = np.stack([fluid.sum((0, 2))] + [v.astype(np.float64).sum((0, 2)) for v in (*u, *prod)], 1)
            # the summed values are the exported float32 ones: only float64 rounding remains
            mag = np.stack([fluid.sum((0, 2))] + [np.abs(v).astype(np.float64).sum((0, 2)) for v in (*u, *prod)], 1)
            assert np.all(np.abs(st - want) <= 1e-12 * mag + 1e-15)
