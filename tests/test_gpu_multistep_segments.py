"""lbm_step(n) on lattices around the limits of the multi-step launch: fewer row segments than a
block has warps, one segment per resident warp, and several per warp with a remainder (pull); the
bits are those of n single steps, with walls, solid cells and the inflow/outflow faces."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
CHANNEL = ("periodic", "periodic", "wall", "wall", "periodic", "periodic")
TUNNEL = ("inflow", "outflow", "freeslip", "freeslip", "freeslip", "freeslip")


@pytest.mark.parametrize("nx,ny,nz,q,streaming,precision,faces", [
    (5, 3, 2, 19, "aa", "f32", CHANNEL), (35, 7, 5, 27, "pull", "f32", TUNNEL), (64, 48, 50, 19, "aa", "f32", TUNNEL),
    (64, 49, 50, 19, "aa", "bf16", CHANNEL), (96, 53, 47, 19, "pull", "f32", TUNNEL), (62, 70, 68, 19, "pull", "f32", CHANNEL),
    (40, 35, 33, 27, "aa", "f32", TUNNEL), (64, 31, 70, 27, "pull", "f32", CHANNEL), (64, 20, 30, 19, "pull", "f16", CHANNEL)])
def test_steps_match_single_launches(nx, ny, nz, q, streaming, precision, faces):
    from paper_2305_09910_gb300 import lbm

    rng = np.random.default_rng(nx * ny)
    flags = (rng.random((nz, ny, nx)) < 0.01).astype(np.uint8)
    u = rng.uniform(-0.04, 0.04, (3, nz, ny, nx)).astype(np.float32)
    lats = []
    for _ in range(2):
        lat = lbm.Lattice(nx, ny, nz, stencil=q, tau=0.6, closure="smag", faces=faces, u_inflow=(0.05, 0, 0),
                          streaming=streaming, precision=precision)
        lat.set_flags(flags)
        lat.set_force(1e-5)
        lat.init_equilibrium(None, u)
        lats.append(lat)
    a, b = lats
    for n in (5, 4):
        a.step(n)
        for _ in range(n):
            b.step(1)
        assert np.array_equal(a.get_populations(), b.get_populations()), n
    a.sync()
    a.close()
    b.close()
