"""Products of many columns on long thin bodies: the samples of a coarse level
times the columns exceed what one further grid dimension can count (65,535
CTAs of 128 items), in the built-in translations of FP32 and of FP64 fields.
Checked against products of 16 of the same columns.  Tolerances (relative
2-norm, fixed from the arithmetic): FP32 rounding magnified by the growth of
the Hankel terms, |h_L(kr)| up to ~70 for three digits, 1e-4; FP64 sums in
another order 1e-10."""
import numpy as np
import pytest

import workloads

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1412_1756_gb300 import mlfma as M  # noqa: E402

K = 2 * np.pi


@pytest.mark.parametrize("length,levels,per_item,dt,tol", [
    (19.2, 7, 4, torch.float32, 1e-4),     # 9,248 samples at level 2, four columns per item
    (12.8, 6, 2, torch.float64, 1e-10),    # 4,802 samples, two columns per thread
])
def test_translation_grid_of_long_bodies(length, levels, per_item, dt, tol):
    v, t = workloads.plate(length, 0.2, int(round(10 * length)), 2)
    prec = M.FP64 if dt == torch.float64 else M.FP32
    P = M.MlfmaPlan(v, t, K, levels, 3.0, max_batch=4096, precisions=(prec,))
    assert P.info()["samples_K"][2] * (4096 // per_item) > 128 * 65535
    g = torch.Generator(device="cuda").manual_seed(5)
    x = torch.randn((P.n, 4096), generator=g, device="cuda", dtype=dt)
    y = P.matvec(x)
    for c in (0, 2040, 4080):
        ref = P.matvec(x[:, c:c + 16].contiguous())
        assert float((y[:, c:c + 16] - ref).norm() / ref.norm()) < tol, c
    P.close()
