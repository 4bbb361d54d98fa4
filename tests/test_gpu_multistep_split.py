"""How a multi-step launch deals its row segments out to blocks: sizes whose share per SM is no
multiple of a block's warps, one segment more than is resident at once, and two passes with a
remainder; and the lattices on either side of the lines between such launches and graph replays,
without and with solid cells in turn.  The bits are those of n single steps."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
CHANNEL = ("periodic", "periodic", "wall", "wall", "periodic", "periodic")
BOX = ("periodic",) * 6


@pytest.mark.parametrize("nx,ny,nz,q,streaming,precision,faces", [
    (64, 40, 38, 19, "pull", "f32", CHANNEL), (60, 40, 38, 19, "aa", "f32", BOX), (64, 64, 64, 19, "pull", "f32", CHANNEL),
    (33, 57, 43, 19, "pull", "bf16", BOX), (64, 40, 38, 27, "aa", "f16", CHANNEL), (64, 40, 38, 27, "pull", "f32", BOX),
    (31, 61, 60, 27, "pull", "f32", CHANNEL), (96, 43, 37, 27, "pull", "f32", CHANNEL), (64, 40, 38, 27, "pull", "f16", BOX)])
def test_steps_match_single_launches(nx, ny, nz, q, streaming, precision, faces):
    from paper_2305_09910_gb300 import lbm

    rng = np.random.default_rng(nx * ny)
    flags = (rng.random((nz, ny, nx)) < 0.01).astype(np.uint8)
    u = rng.uniform(-0.04, 0.04, (3, nz, ny, nx)).astype(np.float32)
    lats = []
    for _ in range(2):
        lat = lbm.Lattice(nx, ny, nz, stencil=q, tau=0.6, closure="smag", faces=faces, streaming=streaming,
                          precision=precision)
        if faces is not BOX:
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


@pytest.mark.parametrize("nx,ny,nz,q,streaming,precision", [
    (64, 38, 32, 19, "aa", "f32"), (64, 39, 32, 19, "aa", "f32"), (61, 38, 32, 19, "pull", "bf16"), (64, 39, 32, 27, "pull", "f32"),
    (64, 49, 50, 19, "aa", "f16"), (63, 19, 17, 19, "pull", "f16"), (64, 57, 32, 27, "pull", "bf16"), (33, 58, 32, 27, "pull", "f16")])
def test_both_sides_of_the_lines(nx, ny, nz, q, streaming, precision):
    from paper_2305_09910_gb300 import lbm

    rng = np.random.default_rng(nx * ny + nz)
    u = rng.uniform(-0.04, 0.04, (3, nz, ny, nx)).astype(np.float32)
    solid = (rng.random((nz, ny, nx)) < 0.01).astype(np.uint8)
    a, b = (lbm.Lattice(nx, ny, nz, stencil=q, tau=0.6, closure="smag", faces=BOX, streaming=streaming, precision=precision)
            for _ in range(2))
    for flags in (None, solid, 0 * solid):
        for lat in (a, b):
            if flags is not None:
                lat.set_flags(flags)
            lat.set_force(1e-5)
            lat.init_equilibrium(None, u)
        a.step(19)
        for _ in range(19):
            b.step(1)
        assert np.array_equal(a.get_populations(), b.get_populations())
    a.sync()
    a.close()
    b.close()
