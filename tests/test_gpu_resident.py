"""The grid-resident step kernel (middling lattices, several steps per launch, edges exchanged
between the CTAs) against the plain tile kernel, one launch per step: the same states and step counts,
bit for bit."""
import numpy as np
import pytest

import workloads
from tests import _parity as P

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    P.ensure_built()


@pytest.mark.parametrize("nx,ny,storage,rounding,sets,mask,calls", [
    (8, 8, 0, 1, 1, 127, (32,)),             # the smallest tiles
    (5, 200, 0, 1, 1, 127, (33, 40)),        # one CTA wide
    (300, 7, 1, 0, 1, 127, (35, 64)),        # one CTA high, FP16 stochastic
    (37, 29, 2, 1, 1, 103, (101,)),          # BF16 to nearest, some forces off
    (110, 97, 2, 0, 1, 127, (1060, 32)),     # blocks of 1024, 32 and 4; BF16
    (128, 128, 0, 1, 2, 127, (50, 51)),      # two thermal sets: four values per node and direction
    (130, 131, 1, 0, 2, 127, (47,)),         # two sets, FP16
    (256, 256, 0, 1, 1, 127, (64,)),         # tiles of 22 x 22, most threads
    (283, 241, 1, 0, 1, 127, (39,)),         # tiles of differing sizes
    (700, 64, 0, 1, 1, 126, (36,)),          # long and narrow
])
def test_resident_kernel_equals_tile_kernel(nx, ny, storage, rounding, sets, mask, calls,
                                            monkeypatch):
    import torch
    import paper_1511_04552_gb300 as m
    warm = torch.from_numpy(workloads.perturbed_rest_fields(nx, ny, 0.02, seed=4)).cuda()
    states, steps = [], []
    for variant in ("resident", "tile"):
        monkeypatch.setenv("MCLBM_STEP_VARIANT", variant)
        c = m.Cavity(nx, ny, 1e4, 6.2, 0.02, 30e-9, storage=storage, rounding=rounding,
                     thermal_sets=sets, force_mask=mask).init(warm=warm)
        for n in calls:
            c.step(n)
        states.append(c.state_get())
        steps.append(c.steps_done())
    a, b = (x.cpu().numpy() for x in states)
    np.testing.assert_array_equal(a, b)  # NaN equals NaN
    assert steps[0] == steps[1] == sum(calls)


def test_resident_kernel_long_call_streams_and_capture():
    """A call longer than one launch takes (2^14 steps); two cavities on streams of their own at once;
    calls recorded into a CUDA graph whose replays continue the run."""
    import torch
    import paper_1511_04552_gb300 as m

    def cavity(**kw):
        return m.Cavity(120, 120, 1e5, 6.2, 0.02, 30e-9, **kw).init()

    a = cavity(storage=1)
    a.step(16384 + 1024 + 6)
    b = cavity(storage=1)
    for n in (16384, 1024, 6):  # the last call: too few steps for the kernel
        b.step(n)
    assert torch.equal(a.state_get(), b.state_get())
    ref = cavity()
    ref.step(192)
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in range(2)]
    pair = [cavity(stream=s) for s in streams]
    for _ in range(3):
        for c in pair:
            c.step(64)
    torch.cuda.synchronize()
    for c in pair:
        assert torch.equal(c.state_get(), ref.state_get())
    c = cavity(stream=streams[0])
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=streams[0]):
        c.step(64)
    for _ in range(3):
        g.replay()
    torch.cuda.synchronize()
    assert torch.equal(c.state_get(), ref.state_get())
