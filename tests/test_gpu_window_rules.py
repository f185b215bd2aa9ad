"""The built-in choice of up and down kernels for few columns: a flat strip
(no children that share a phi step) whose coarsest level has 4,232 samples, a
cube whose levels have pairs, and column counts on both sides of every line of
the rule, against FP64 products of single columns.  FP32 rounding magnified by
the growth of the Hankel terms stays within 1e-4 for three digits."""
import numpy as np
import pytest

import workloads

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1412_1756_gb300 import mlfma as M  # noqa: E402


@pytest.mark.parametrize("mesh,levels", [
    (lambda: workloads.plate(12.0, 0.6, 120, 6), 6),
    (lambda: workloads.cube(4.0, 40), 5),
])
def test_builtin_up_and_down_for_few_columns(mesh, levels):
    v, t = mesh()
    P = M.MlfmaPlan(v, t, 2 * np.pi, levels, 3.0, max_batch=24)
    g = torch.Generator(device="cuda").manual_seed(7)
    x = torch.randn((P.n, 24), generator=g, device="cuda", dtype=torch.float32)
    one = torch.cat([P.matvec(x[:, c:c + 1].double()) for c in range(24)], 1)
    for B in (1, 2, 3, 4, 5, 8, 9, 12, 13, 16, 17, 20, 21, 24):
        y = P.matvec(x[:, :B].contiguous()).to(torch.complex128)
        assert float((y - one[:, :B]).norm() / one[:, :B].norm()) < 1e-4, B
    P.close()
