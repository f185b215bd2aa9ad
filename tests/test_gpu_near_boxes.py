"""The near-field tiles where their staging or columns are cut to fit: boxes
of up to ~230 rows at every width whose chunk of strip columns has to shrink,
remainders of columns that are shared out, and two and three columns on trees
of more than 608 leaf boxes.  With two levels the product is the near field.
Tolerances (relative 2-norms): sums of ~1,000 FP32 products 1e-5, magnified by
the growth of the Hankel terms (~70 for three digits) where the product has a
far field, 1e-4; FP64 sums in another order 1e-10."""
import numpy as np
import pytest

import workloads

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1412_1756_gb300 import mlfma as M  # noqa: E402

K = 2 * np.pi


def rel(a, b):
    return float((a.to(torch.complex128) - b).norm() / b.norm())


def singles(P, x):
    return torch.cat([P.matvec(x[:, c:c + 1].double()) for c in range(x.shape[1])], 1)


def test_large_boxes_and_shared_remainders():
    v, t = workloads.plate(2.0, 1.6, 20, 16)   # 4 boxes of ~230 rows
    P = M.MlfmaPlan(v, t, K, 2, 3.0, max_batch=70)
    g = torch.Generator(device="cuda").manual_seed(2)
    x = torch.randn((P.n, 70), generator=g, device="cuda", dtype=torch.float32)
    one = singles(P, x)
    for B in (4, 5, 7, 8, 9, 16, 65, 66, 70):
        assert rel(P.matvec(x[:, :B].contiguous()), one[:, :B]) < 1e-5, B
    for B in (4, 5, 8, 16, 17, 18, 23):
        assert rel(P.matvec(x[:, :B].double()), one[:, :B]) < 1e-10, B
    P.close()


def test_few_columns_on_many_boxes():
    W = workloads.get("sphere-r2m-ico5")
    v, t = W.mesh()
    P = M.MlfmaPlan(v, t, W.k, W.levels, W.digits, max_batch=4)
    leaf = P.info()["leaf_level"]
    assert 608 <= P.info()["box_count"][leaf] < 2432
    g = torch.Generator(device="cuda").manual_seed(4)
    x = torch.randn((P.n, 4), generator=g, device="cuda", dtype=torch.float32)
    one, S = [], []
    for c in range(4):
        one.append(P.matvec(x[:, c:c + 1].double()))
        S.append(P.export_field(M.FP64, 0, leaf, 1)[..., 0])
    one = torch.cat(one, 1)
    for B in (2, 3):
        assert rel(P.matvec(x[:, :B].contiguous()), one[:, :B]) < 1e-4, B
        f = P.export_field(M.FP32, 0, leaf, B)
        for c in range(B):
            assert np.linalg.norm(f[..., c] - S[c]) < 1e-5 * np.linalg.norm(S[c]), (B, c)
    z = torch.complex(x[:, 0], x[:, 1])   # one complex column is two internal ones
    assert rel(P.matvec(z.reshape(-1, 1)), one[:, :1] + 1j * one[:, 1:2]) < 1e-4
    P.close()
