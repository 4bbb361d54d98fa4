"""The x-pair AA step of half storage (single launches) against the one-cell code (multi-step
launches): the same bits for rows that end inside a pair, a warp or a tile, with walls, periodic
seams, free-slip, inflow and outflow faces and solid cells; and the plane statistics a sampling
step takes against those of the exported state."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
CHANNEL = ("periodic", "periodic", "wall", "wall", "periodic", "periodic")
TUNNEL = ("inflow", "outflow", "freeslip", "freeslip", "freeslip", "freeslip")
MIXED = ("inflow", "outflow", "wall", "freeslip", "periodic", "periodic")
BOX = ("periodic",) * 6


def _lattice(nx, q, precision, faces, ny=9, nz=7):
    from paper_2305_09910_gb300 import lbm

    rng = np.random.default_rng(nx + q)
    lat = lbm.Lattice(nx, ny, nz, stencil=q, tau=0.6, closure="smag" if nx % 4 else "none", faces=faces,
                      u_inflow=(0.05, 0, 0), streaming="aa", precision=precision)
    lat.set_flags((rng.random((nz, ny, nx)) < 0.02).astype(np.uint8))
    lat.set_force(1e-5)
    lat.init_equilibrium(None, rng.uniform(-0.04, 0.04, (3, nz, ny, nx)).astype(np.float32))
    return lat


@pytest.mark.parametrize("q,precision", [(19, "f16"), (27, "bf16"), (19, "bf16"), (27, "f16")])
@pytest.mark.parametrize("faces", [CHANNEL, TUNNEL, MIXED, BOX])
@pytest.mark.parametrize("nx", [3, 31, 34, 63, 64, 65, 96, 99, 127, 130, 193])
def test_pairs_match_one_cell_code(nx, faces, q, precision):
    if faces[1] == "outflow" and nx % 32 == 1:
        nx += 1  # the outflow face does not take such rows
    a, b = _lattice(nx, q, precision, faces), _lattice(nx, q, precision, faces)
    for n in (3, 4):
        for _ in range(n):
            a.step(1)
        b.step(n)
        assert np.array_equal(a.get_populations(), b.get_populations()), n
    a.sync()
    a.close()
    b.close()


@pytest.mark.parametrize("nx,q,faces", [(99, 19, CHANNEL), (130, 27, TUNNEL), (64, 27, CHANNEL)])
def test_statistics_of_a_sampling_step(nx, q, faces):
    from paper_2305_09910_gb300 import lbm

    a, b = _lattice(nx, q, "f16", faces), _lattice(nx, q, "f16", faces)
    a.step(1)
    b.step(1)
    for lat in (a, b):
        lbm.lbm_stats_reset(lat.h)
    lbm.lbm_step_stats(a.h, 3, 1)
    for _ in range(3):
        lbm.lbm_stats_sample(b.h)
        b.step(1)
    sa, na = lbm.lbm_stats_get(a.h, a.ny)
    sb, nb = lbm.lbm_stats_get(b.h, b.ny)
    assert na == nb == 3
    # sums of 64 float32 values each in float32 against float64 sums of the same values: 2^-24 of
    # the magnitude per addition, six levels of additions
    assert np.all(np.abs(sa - sb) <= 7 * 2.0 ** -24 * 3 * a.nx * a.nz * 0.1 + 1e-12)
    assert np.array_equal(a.get_populations(), b.get_populations())
    a.close()
    b.close()
