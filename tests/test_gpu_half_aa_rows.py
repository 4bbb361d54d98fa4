"""The x-pair AA steps of half storage where the dispatch takes them: D3Q19 odd steps of rows long
enough for their odd end, inflow, outflow or wall faces, against the one-cell code of a multi-step
launch; D3Q27 even steps of lattices of more than a wave of blocks, against the two-grid pull lattice.
The same bits."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
CHANNEL = ("periodic", "periodic", "wall", "wall", "periodic", "periodic")
TUNNEL = ("inflow", "outflow", "freeslip", "freeslip", "freeslip", "freeslip")
WALLS = ("wall",) * 6
BOX = ("periodic",) * 6


def _lattice(nx, ny, nz, q, precision, faces, streaming="aa"):
    from paper_2305_09910_gb300 import lbm

    rng = np.random.default_rng(nx + q)
    lat = lbm.Lattice(nx, ny, nz, stencil=q, tau=0.6, closure="smag", faces=faces, u_inflow=(0.05, 0, 0),
                      streaming=streaming, precision=precision)
    lat.set_flags((rng.random((nz, ny, nx)) < 0.01).astype(np.uint8))
    lat.set_force(1e-5)
    lat.init_equilibrium(None, rng.uniform(-0.04, 0.04, (3, nz, ny, nx)).astype(np.float32))
    return lat


@pytest.mark.parametrize("precision", ["f16", "bf16"])
@pytest.mark.parametrize("nx,faces", [(641, BOX), (705, CHANNEL), (767, BOX), (1474, ("wall", "wall") + BOX[2:]), (2946, TUNNEL),
                                      (2944, WALLS), (3651, TUNNEL), (3647, WALLS)])
def test_odd_steps_of_long_rows(nx, faces, precision):
    a, b = _lattice(nx, 6, 5, 19, precision, faces), _lattice(nx, 6, 5, 19, precision, faces)
    for n in (3, 4):
        for _ in range(n):
            a.step(1)
        b.step(n)
        assert np.array_equal(a.get_populations(), b.get_populations()), n
    a.sync()
    a.close()
    b.close()


@pytest.mark.parametrize("precision", ["f16", "bf16"])
@pytest.mark.parametrize("nx,faces", [(33, BOX), (64, CHANNEL), (67, CHANNEL), (95, BOX), (98, TUNNEL), (130, WALLS)])
def test_even_steps_of_large_lattices(nx, faces, precision):
    a, b = _lattice(nx, 50, 49, 27, precision, faces), _lattice(nx, 50, 49, 27, precision, faces, "pull")
    for n in (3, 4):
        for _ in range(n):
            a.step(1)
            b.step(1)
        assert np.array_equal(a.get_populations(), b.get_populations()), n
    a.sync()
    a.close()
    b.close()
