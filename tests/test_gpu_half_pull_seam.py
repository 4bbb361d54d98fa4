"""The x-pair pull step of half storage where a row's last cell is the first of its pair (odd nx) and
streams across the periodic x seam: the bits of the in-place (AA) lattice, whose cells of such rows
take the one-cell code, and of the multi-step launch; on lattices below the size limit of the
multi-step launch and above it, as single launches and as graph replays."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
CHANNEL = ("periodic", "periodic", "wall", "wall", "periodic", "periodic")
BOX = ("periodic",) * 6


def _lattice(nx, ny, nz, q, precision, faces, streaming):
    from paper_2305_09910_gb300 import lbm

    rng = np.random.default_rng(nx + q)
    lat = lbm.Lattice(nx, ny, nz, stencil=q, tau=0.6, closure="smag", faces=faces, streaming=streaming,
                      precision=precision)
    lat.set_flags((rng.random((nz, ny, nx)) < 0.02).astype(np.uint8))
    lat.set_force(1e-5)
    lat.init_equilibrium(None, rng.uniform(-0.04, 0.04, (3, nz, ny, nx)).astype(np.float32))
    return lat


@pytest.mark.parametrize("q,precision", [(19, "f16"), (27, "f16"), (19, "bf16"), (27, "bf16")])
@pytest.mark.parametrize("faces", [CHANNEL, BOX])
@pytest.mark.parametrize("nx,ny,nz", [(1, 9, 7), (3, 9, 7), (31, 9, 7), (33, 9, 7), (63, 9, 7), (64, 9, 7), (65, 9, 7),
                                      (99, 9, 7), (63, 40, 36), (97, 31, 30)])
def test_seam_of_odd_rows(nx, ny, nz, faces, q, precision):
    single, many, aa = (_lattice(nx, ny, nz, q, precision, faces, s) for s in ("pull", "pull", "aa"))
    for n in (3, 18):
        for _ in range(n):
            single.step(1)
        many.step(n)
        aa.step(n)
        want = aa.get_populations()
        assert np.array_equal(single.get_populations(), want), n
        assert np.array_equal(many.get_populations(), want), n
    for lat in (single, many, aa):
        lat.sync()
        lat.close()
