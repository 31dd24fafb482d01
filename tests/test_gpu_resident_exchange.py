"""The words that neighbouring CTAs of the grid-resident step kernel exchange: run after run the states of
the plain tile kernel, so that a word taken before all of it has arrived, however rarely, shows."""
import pytest

import workloads
from tests import _parity as P

pytestmark = pytest.mark.gpu

RUNS = 25


@pytest.fixture(scope="module", autouse=True)
def _built():
    P.ensure_built()


@pytest.mark.parametrize("nx,ny,storage,sets", [
    (100, 100, 0, 2), (128, 128, 0, 2),  # words of values of several nodes and directions
    (24, 24, 0, 2), (128, 128, 1, 2), (128, 128, 0, 1), (256, 256, 2, 1),
])
def test_every_run_gives_the_same_states(nx, ny, storage, sets, monkeypatch):
    import torch
    import paper_1511_04552_gb300 as m
    warm = torch.from_numpy(workloads.perturbed_rest_fields(nx, ny, 0.02, seed=4)).cuda()

    def cavity(variant):
        monkeypatch.setenv("MCLBM_STEP_VARIANT", variant)
        return m.Cavity(nx, ny, 1e4, 6.2, 0.02, 30e-9, storage=storage, thermal_sets=sets)

    def run(c):
        c.init(warm=warm)
        for n in (16, 50, 50):
            c.step(n)
        return c.state_get()

    want = run(cavity("tile")).view(torch.int32)
    if storage == 0:
        c = cavity("resident")
        assert c.step_launches(50) == 1
        for _ in range(RUNS):
            assert torch.equal(run(c).view(torch.int32), want)
    else:  # stochastic rounding goes on with the handle's epochs: a handle per run
        for _ in range(RUNS):
            c = cavity("resident")
            assert c.step_launches(50) == 1
            assert torch.equal(run(c).view(torch.int32), want)
