"""Light curves bit for bit against the oracle where the kernel's divisions and lane pairs
change: point counts around a CTA, pixel widths inside and outside the range of its integer
division, tracks along pixel edges, off the map and of zero length."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

import workloads as W  # noqa: E402
from oracle import lightcurve as LC  # noqa: E402
from paper_1703_09707_gb300 import mlens as M  # noqa: E402


@pytest.mark.parametrize("n", [1, 2, 3, 31, 32, 33, 65, 4097])
@pytest.mark.parametrize("box", [(-2.0, 2.0, -1.0, 3.0), (0.1, 0.7, -5.3, 1.9), (-1e-70, 1e-70, 0.0, 3e-71),
                                 (-1e66, 1e66, 1.0, 2e65)])
def test_curves_equal_the_oracle(n, box):
    rng = np.random.default_rng(n)
    src = W.Grid(*box, 37, 23)
    m = rng.normal(0.0, 10.0, (23, 37)).astype(np.float32)
    md = torch.from_numpy(m.reshape(-1)).cuda()
    wx, wy = box[1] - box[0], box[3] - box[2]
    at = lambda fx, fy: (box[0] + fx * wx, box[2] + fy * wy)  # noqa: E731
    for p, q in ((at(0.02, 0.1), at(0.9, 0.97)), (at(-0.5, 0.5), at(1.5, 0.4)), (at(0.25, 0.25), at(0.25, 0.25)),
                 (at(0.0, 0.0), at(1.0, 1.0)), (at(5.0 / 37, 0.5), at(5.0 / 37, 7.0 / 23))):
        out = torch.empty(n, dtype=torch.float32, device="cuda")
        M.mlens_light_curve(md, src, p, q, n, out)
        ref = LC.light_curve(m, src, p, q, n).astype(np.float32)
        assert np.array_equal(out.cpu().numpy().view(np.uint32), ref.view(np.uint32)), (p, q)
