"""FP32 rounding of reception.  With five digits on quarter-wavelength boxes
the far field cancels several hundred-fold, so the roundings of the running
sum over samples show in the product.  Sixteen columns take the kernel with
one rounding per sample; every other width below 32 must be as close to the
FP64 product, whichever kernel and split of the samples it takes.  Tolerance:
the same number of roundings of the running sum's size gives the same error
but for the order of the terms, for which a fifth is allowed (four roundings
per sample instead of one double it).  The sin-kernel product, whose incoming
field does not cancel, shows the sum's own rounding.  (From 32 columns up the
sum is chained, and results keep their bits.)"""
import numpy as np
import pytest

import workloads

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1412_1756_gb300 import mlfma as M  # noqa: E402


def test_narrow_five_digit_products_round_as_sixteen_columns_do():
    v, t = workloads.icosphere(5, 2.0)
    P = M.MlfmaPlan(v, t, 2 * np.pi, 5, 5.0, max_batch=31)
    g = torch.Generator(device="cuda").manual_seed(1)
    x = torch.randn((P.n, 31), generator=g, device="cuda", dtype=torch.float32)
    for product in (P.matvec, P.matvec_r):
        ref = torch.cat([product(x[:, c:c + 1].double()) for c in range(31)], 1)

        def err(B):
            e = product(x[:, :B].contiguous()).to(torch.complex128) - ref[:, :B]
            return float((e.norm(dim=0) / ref[:, :B].norm(dim=0)).mean())
        e16 = err(16)
        for B in (1, 2, 3, 4, 5, 7, 8, 9, 12, 15, 17, 18, 24, 31):
            assert err(B) < 1.2 * e16, (product.__name__, B, err(B), e16)
    P.close()
