"""The sums of tests/test_gpu_row_sums.py for the ways rows are dealt out to blocks: one, two and three
planes (the face planes come first), more planes than blocks wanted, more rows per plane than a block
takes, and several rows per block with all rows of a z plane boundary cells."""
import pytest

from tests import test_gpu_row_sums as base

pytestmark = pytest.mark.gpu
BOX = ("periodic",) * 6


@pytest.mark.parametrize("nx,ny,nz,q,streaming,precision,faces", [
    (40, 1, 9, 19, "aa", "f32", BOX), (33, 2, 17, 19, "pull", "f16", base.CHANNEL), (20, 3, 700, 27, "pull", "f32", base.CHANNEL),
    (18, 5200, 2, 19, "pull", "f32", base.CHANNEL), (70, 64, 80, 27, "pull", "f16", base.TUNNEL),
    (130, 48, 60, 19, "aa", "bf16", base.TUNNEL)])
def test_sums_of_planes(nx, ny, nz, q, streaming, precision, faces):
    base.test_sums_match_the_exported_fields(nx, ny, nz, q, streaming, precision, faces)
