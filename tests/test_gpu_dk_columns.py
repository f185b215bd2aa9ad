"""dZ/dk products of odd column counts on a plan with up and down passes: the
tangent half of every field row then starts 8 bytes off a 16-byte boundary,
which the windowed kernels, the translation and the leaf tiles must respect.
FP32 against FP64 products of single columns; FP32 rounding magnified by the
growth of the Hankel terms stays within 1e-4."""
import pytest

import workloads

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1412_1756_gb300 import mlfma as M  # noqa: E402


def test_dk_odd_columns_on_five_levels():
    W = workloads.get("sphere-r2m-ico5")
    v, t = W.mesh()
    P = M.MlfmaPlan(v, t, W.k, W.levels, W.digits, max_batch=34)
    g = torch.Generator(device="cuda").manual_seed(6)
    x = torch.randn((P.n, 17), generator=g, device="cuda", dtype=torch.float32)
    one = torch.cat([P.matvec_dk(x[:, c:c + 1].double()) for c in range(17)], 1)
    for B in (1, 2, 3, 5, 7, 8, 9, 17):
        y = P.matvec_dk(x[:, :B].contiguous()).to(torch.complex128)
        assert float((y - one[:, :B]).norm() / one[:, :B].norm()) < 1e-4, B
    P.close()
