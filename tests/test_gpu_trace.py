"""rs_trace of few rays through many lenses sums the lens groups of a ray side by side; of many rays, one thread
sums all lenses of its rays.  Both must give the same bits: positions, deflections and error bands."""
import numpy as np
import pytest
import torch

import rs_inputs as ri
from gpu_helpers import rs

pytestmark = pytest.mark.gpu

RAYS = 135000  # three blocks of the split path


@pytest.mark.parametrize("mass", ["equal", "salpeter", "wide"])
@pytest.mark.parametrize("n", [511, 512, 513, 575, 640, 1023, 1280, 5001])
def test_split_trace_equals_direct_trace(n, mass):
    """Lens counts about group, renormalisation and tile boundaries; ray counts about a ray block, a workspace that
    takes the field in two chunks (65536 rays, 5001 lenses) and blocks of rays one after the other.  The direct
    kernel runs where the workspace is refused."""
    m = rs()
    spec = ri.disc_field("tr", n, 0.5, 0.1, 0.3, 512, 64, seed=5, mass="equal" if mass == "equal" else "salpeter")
    masses = spec.masses if mass != "wide" else (spec.masses.astype(np.float64) * 2.0 ** 65).astype(np.float32)
    ij = torch.from_numpy(ri.sample_rays(spec.grid, RAYS, seed=n))
    f = m.Field(spec.lens_xy, masses, spec.kappa_c, spec.gamma)
    v = f.view(256, n - 256)  # the lens arrays of a view start inside its parent's
    try:
        for g in (f, v):
            m.rs_set_alloc_failure(0)
            want = [t.cpu().numpy() for t in g.trace(spec.grid, ij, with_alpha=True, with_err=True)]
            m.rs_set_alloc_failure(-1)
            for k in (1, 127, 128, 129, 511, 512, 4000, 65536, 65537, RAYS) if g is f else (300, 700):
                got = [t.cpu().numpy() for t in g.trace(spec.grid, ij[:k], with_alpha=True, with_err=True)]
                for a, b in zip(got, want):
                    assert np.array_equal(a, b[:k], equal_nan=True), k
            y = g.trace(spec.grid, ij[:200]).cpu().numpy()
            assert np.array_equal(y, want[0][:200], equal_nan=True)
    finally:
        m.rs_set_alloc_failure(-1)
        v.close()
        f.close()


def test_split_trace_without_workspace_and_under_capture():
    """A failed workspace allocation and a captured stream take the direct kernel: same bits, no error."""
    m = rs()
    spec = ri.disc_field("trc", 3000, 0.5, 0.0, 0.3, 512, 64, seed=8, mass="salpeter")
    ij = torch.from_numpy(ri.sample_rays(spec.grid, 700, seed=2)).cuda()
    f = m.Field.from_spec(spec)
    try:
        want = f.trace(spec.grid, ij)
        m.rs_set_alloc_failure(0)
        got = f.trace(spec.grid, ij)
        m.rs_set_alloc_failure(-1)
        assert torch.equal(got, want)
        y = torch.zeros_like(want)
        st = torch.cuda.Stream()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=st):
            m.rs_trace(f.handle, spec.grid, ij, y, stream=st)
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(y, want)
    finally:
        m.rs_set_alloc_failure(-1)
        f.close()
