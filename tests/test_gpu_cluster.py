"""The cluster-resident step kernel (small lattices, several steps per launch) against the plain
tile kernel, one launch per step: the same states, step counts and checkpoint files, bit for bit."""
import numpy as np
import pytest

import workloads
from tests import _parity as P

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    P.ensure_built()


@pytest.mark.parametrize("nx,ny,storage,rounding,sets,mask,calls", [
    (2, 2, 0, 1, 1, 127, (8,)),              # one CTA
    (2, 41, 0, 1, 1, 127, (9,)),             # lines of two nodes
    (41, 2, 1, 0, 1, 127, (9,)),             # numbered by column, FP16 stochastic
    (16, 16, 0, 1, 1, 127, (4, 5, 6)),       # runs of two lines
    (37, 29, 2, 0, 1, 127, (1027, 1, 8)),    # blocks of 1024 and 2, an odd last step; BF16
    (37, 29, 2, 1, 1, 103, (300, 301)),      # BF16 to nearest, some forces off
    (37, 29, 2, 1, 1, 115, (300, 301)),      # without drag the run diverges: NaN like NaN
    (29, 37, 0, 1, 2, 127, (33, 8)),         # two thermal sets
    (90, 96, 1, 0, 2, 127, (17, 20)),        # two sets, FP16, most threads
    (31, 300, 0, 1, 1, 127, (12,)),          # long and narrow
    (330, 31, 1, 0, 1, 127, (21, 11)),       # the largest runs, numbered by column
    (130, 67, 0, 1, 1, 126, (40,)),          # ring nodes without a thread of their own
    (101, 101, 0, 1, 1, 127, (15, 15)),      # near the most nodes a cluster takes
])
def test_cluster_kernel_equals_tile_kernel(nx, ny, storage, rounding, sets, mask, calls, tmp_path,
                                           monkeypatch):
    import torch
    import paper_1511_04552_gb300 as m
    warm = torch.from_numpy(workloads.perturbed_rest_fields(nx, ny, 0.02, seed=4)).cuda()
    states, files, steps = [], [], []
    for variant in ("cluster", "tile"):
        monkeypatch.setenv("MCLBM_STEP_VARIANT", variant)
        c = m.Cavity(nx, ny, 1e4, 6.2, 0.02, 30e-9, storage=storage, rounding=rounding,
                     thermal_sets=sets, force_mask=mask).init(warm=warm)
        for n in calls:
            c.step(n)
        path = tmp_path / variant
        c.save(str(path))
        states.append(c.state_get())
        files.append(np.fromfile(path, dtype=np.uint8))
        steps.append(c.steps_done())
    a, b = (x.cpu().numpy() for x in states)
    np.testing.assert_array_equal(a, b)  # NaN equals NaN
    assert steps[0] == steps[1] == sum(calls)
    # the rows' padding beyond nx is never written by either kernel, nor is it compared here
    head = 104
    np.testing.assert_array_equal(files[0][:head], files[1][:head])


def test_cluster_kernel_long_call_and_capture():
    """A call longer than one launch takes (2^14 steps), and calls recorded into a CUDA graph whose
    replays continue the run."""
    import torch
    import paper_1511_04552_gb300 as m
    a = m.Cavity(24, 24, 1e3, 6.2, 0.01, 20e-9, storage=1).init()
    b = m.Cavity(24, 24, 1e3, 6.2, 0.01, 20e-9, storage=1).init()
    a.step(16384 + 1024 + 6)
    b.step(16384)
    b.step(1024)
    b.step(6)
    assert torch.equal(a.state_get(), b.state_get())
    s = torch.cuda.Stream()
    c = m.Cavity(24, 24, 1e3, 6.2, 0.01, 20e-9, stream=s).init()
    d = m.Cavity(24, 24, 1e3, 6.2, 0.01, 20e-9).init()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        c.step(64)
    for _ in range(3):
        g.replay()
    d.step(192)
    torch.cuda.synchronize()
    assert torch.equal(c.state_get(), d.state_get())
