"""Which kernels mclbm_step launches (mclbm_step_launches): that the cases that compare the resident kernels
with the tile kernel run them, and where the lines of the default choice lie."""
import pytest

from tests import _parity as P
from tests import test_gpu_cluster as cluster
from tests import test_gpu_resident as resident

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    P.ensure_built()


def _cases(test):
    mark = next(m for m in test.pytestmark if m.name == "parametrize")
    return mark.args[1]


def _step_by_step(n):
    """Steps in graphs of 2^k (2 .. 1024), each with a kernel for the epoch; an odd last one alone."""
    k = bin((n % 1024) & ~1).count("1") + n // 1024
    return n + k


def _cavity(nx, ny, **kw):
    import paper_1511_04552_gb300 as m
    return m.Cavity(nx, ny, 1e4, 6.2, 0.02, 30e-9, **kw)


@pytest.mark.parametrize("nx,ny,storage,rounding,sets,mask,calls",
                         _cases(resident.test_resident_kernel_equals_tile_kernel))
def test_resident_cases_run_the_resident_kernel(nx, ny, storage, rounding, sets, mask, calls, monkeypatch):
    kw = dict(storage=storage, rounding=rounding, thermal_sets=sets, force_mask=mask)
    monkeypatch.setenv("MCLBM_STEP_VARIANT", "resident")
    c = _cavity(nx, ny, **kw)
    assert [c.step_launches(n) for n in calls] == [1 + n % 2 for n in calls]
    monkeypatch.setenv("MCLBM_STEP_VARIANT", "tile")
    c = _cavity(nx, ny, **kw)
    assert [c.step_launches(n) for n in calls] == [_step_by_step(n) for n in calls]
    assert c.step_kernel()["variant"] == 0


@pytest.mark.parametrize("nx,ny,storage,rounding,sets,mask,calls",
                         _cases(cluster.test_cluster_kernel_equals_tile_kernel))
def test_cluster_cases_run_the_cluster_kernel(nx, ny, storage, rounding, sets, mask, calls, monkeypatch):
    kw = dict(storage=storage, rounding=rounding, thermal_sets=sets, force_mask=mask)
    monkeypatch.setenv("MCLBM_STEP_VARIANT", "cluster")
    c = _cavity(nx, ny, **kw)
    assert [c.step_launches(n) for n in calls] == [1] * len(calls)


def test_default_choice(monkeypatch):
    for k in ("MCLBM_STEP_VARIANT", "MCLBM_STEP_VEC", "MCLBM_STEP_TILE_H"):
        monkeypatch.delenv(k, raising=False)
    long_call = 16384 + 1024 + 6
    c = _cavity(24, 24, storage=1)  # the cluster kernel, any number of steps
    assert [c.step_launches(n) for n in (3, 4, 5, 16384, long_call)] == [_step_by_step(3), 1, 1, 1, 2]
    c = _cavity(120, 120, storage=1)  # the grid: even numbers
    assert [c.step_launches(n) for n in (15, 16, 64, 16384, 16384 + 17, long_call)] == [
        _step_by_step(15), 1, 1, 1, 3, 2]
    for kw in (dict(nx=256, ny=256), dict(nx=128, ny=128, thermal_sets=2), dict(nx=130, ny=67)):
        assert _cavity(**kw).step_launches(1000) == 1
    c = _cavity(1024, 1024)  # beyond shared memory
    assert c.step_launches(1000) == _step_by_step(1000)
    assert c.step_launches(0) == 0
    assert c.step_launches(-1) == -1
