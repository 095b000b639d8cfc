"""Assembly against the oracle on both sides of the line between tiles and one
cell per thread: planes that fill five eighths of their 32 x 8 tiles (15/16 with
the harmonic mean) and a little less, ragged in x, y and z, masked."""
import pytest

torch = pytest.importorskip("torch")

from paper_1809_10895_gb300 import rf
from tests.test_gpu_assemble_tiles import test_tiled_assembly_matches_oracle as matches_oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1809_10895_gb300 import build as B
    B.build()
    rf.load()
    torch.cuda.set_device(0)


# 40 x 40 fills 0.625 of its tiles, 41 x 39 0.6246; the others 0.64 to 0.97
@pytest.mark.parametrize("shape", [(40, 40, 21), (41, 39, 21), (45, 29, 33), (31, 8, 140), (60, 13, 48)])
@pytest.mark.parametrize("form", ["chord", "modified", "tilted"])
def test_arithmetic_mean(shape, form):
    matches_oracle(shape, form)


# 120 x 16 fills 15/16 (one cell per thread), 121 x 16 more, 95 x 24 0.99
@pytest.mark.parametrize("shape", [(120, 16, 18), (121, 16, 18), (95, 24, 16), (64, 32, 17)])
def test_harmonic_mean(shape):
    matches_oracle(shape, "harmonic")
