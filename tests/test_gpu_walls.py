"""The tile kernels' wall rules at the sizes where a warp holds wall nodes, nodes away from the
walls and lanes beyond the lattice in every mix: against the FP64 oracle, with one and two nodes per
thread and one and two thermal sets. Small lattices go to the cluster kernel by default, so the tile
kernels are asked for by name. The bar is the parity tests' 1e-5 per field (FP32 against FP64)."""
import pytest

from tests import _parity as P

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    P.ensure_built()


@pytest.mark.parametrize("nx,ny", [(2, 2), (3, 3), (31, 9), (32, 8), (33, 7), (34, 17), (65, 3),
                                   (2, 70), (67, 2), (128, 33)])
@pytest.mark.parametrize("sets,variant,vec", [(1, "tma", 1), (1, "tma", 2), (1, "tile", 1),
                                              (1, "two", 1), (2, "tile", 1)])
def test_tile_kernels_at_walls_match_oracle(nx, ny, sets, variant, vec, monkeypatch):
    monkeypatch.setenv("MCLBM_STEP_VARIANT", variant)
    if sets == 1:
        monkeypatch.setenv("MCLBM_STEP_VEC", str(vec))
    gpu, ref = P.make_pair(nx, ny, 1e4, 6.2, 0.02, 30e-9, seed=6, thermal_sets=sets)
    gpu.step(150)
    ref.step(150)
    errs, bad = P.compare_fields(gpu, ref)
    assert not bad, errs
