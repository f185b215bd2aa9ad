"""Built-in kernels that follow the number of columns: register-tiled near
field, radiation and reception, the flattened translation, and the windowed
passes' choice of shape.  Column counts at the edges of their tiles (1, 2, 4,
16, 32, 64 columns, one less and one more), boxes from one unknown to several
row passes, trees with few leaf boxes (row and sample splits) and many.

Tolerances (relative 2-norms, fixed from the arithmetic): FP32 sums of at most
~1,000 rounded products stay within 1e-5; a far field's FP32 rounding is
magnified by the growth of the Hankel terms, |h_L(kr)| up to ~70 for three
digits on boxes of a quarter wavelength or more, so 1e-4 on the product; FP64
sums in another order within 1e-10."""
import numpy as np
import pytest

import workloads
from oracle import efie

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1412_1756_gb300 import mlfma as M  # noqa: E402

K = 2 * np.pi


def rel(a, b):
    return float(np.linalg.norm(np.asarray(a, complex) - b) / np.linalg.norm(b))


def gpu(x, dt):
    return torch.from_numpy(np.ascontiguousarray(x)).to("cuda", dt)


@pytest.mark.parametrize("mesh", [lambda: workloads.icosphere(2, 0.5),             # 8 boxes of ~60 rows
                                  lambda: workloads.plate(2.0, 1.6, 20, 16)])      # 4 boxes of ~230 rows
def test_near_only_matches_oracle(mesh):
    """With two levels all leaf boxes touch: the product is the near field.
    FP32 against the dense oracle; FP64 against single columns, which the
    kernel without tiles computes (triangle pairs exactly at the extraction
    distance, as a regular grid has them, may fall on either side of it in the
    oracle and in the library, 2e-7 of the product)."""
    v, t = mesh()
    Z = efie.Problem(v, t, K).dense()
    P = M.MlfmaPlan(v, t, K, 2, 3.0, max_batch=80)
    for B in (1, 2, 3, 4, 5, 8, 15, 16, 17, 33, 64, 65, 80):
        x = workloads.rhs(P.n, B, B)
        ref = Z @ x
        assert rel(P.matvec(gpu(x, torch.float32)).cpu().numpy(), ref) < 1e-5, B
        if 1 < B <= 20:
            one = np.concatenate([P.matvec(gpu(x[:, c:c + 1], torch.float64)).cpu().numpy() for c in range(B)], 1)
            assert rel(P.matvec(gpu(x, torch.float64)).cpu().numpy(), one) < 1e-10, B
    P.close()


@pytest.mark.parametrize("mesh,levels", [
    (lambda: workloads.icosphere(2, 0.5), 3),                # 56 boxes of up to 12 unknowns
    (lambda: workloads.plate(3.1, 2.3, 31, 23), 3),          # few boxes of up to ~180 unknowns: several row passes
    (lambda: workloads.plate_with_strips(), 5),              # 256 boxes, three far levels, thin strips
])
def test_columns_agree_with_single_fp64_columns(mesh, levels):
    """Every column count against FP64 products of one column at a time (the
    kernels without tiles), product and leaf fields."""
    v, t = mesh()
    P = M.MlfmaPlan(v, t, K, levels, 3.0, max_batch=66)
    leaf = P.info()["leaf_level"]
    x = workloads.rhs(P.n, 66, 11)
    cols = list(range(8)) + [65]
    one, S = {}, {}
    for c in cols:
        one[c] = P.matvec(gpu(x[:, c:c + 1], torch.float64)).cpu().numpy()[:, 0]
        S[c] = P.export_field(M.FP64, 0, leaf, 1)[..., 0]
    for B in (2, 3, 4, 5, 7, 8, 9, 15, 16, 17, 31, 32, 33, 34, 40, 63, 64, 65, 66):
        y = P.matvec(gpu(x[:, :B], torch.float32)).cpu().numpy()
        f = P.export_field(M.FP32, 0, leaf, B)
        for c in cols:
            if c < B:
                assert rel(y[:, c], one[c]) < 1e-4, (B, c)
                assert rel(f[..., c], S[c]) < 1e-5, (B, c)
        if B in (3, 4, 5, 8, 9, 16, 17):
            y = P.matvec(gpu(x[:, :B], torch.float64)).cpu().numpy()
            for c in cols:
                if c < B:
                    assert rel(y[:, c], one[c]) < 1e-10, (B, c)
    P.close()


def test_builtin_window_shapes_agree_with_pinned_ones():
    """The built-in up and down shapes against pinned windowed shapes and the
    new ones (754, 758, 854), for column counts on both sides of the rule:
    FP32 rounding only."""
    W = workloads.get("sphere-r2m-ico5")
    v, t = W.mesh()
    P = M.MlfmaPlan(v, t, W.k, W.levels, W.digits, max_batch=40, precisions=(M.FP32,))
    L = M.MAX_LEVELS
    for B in (1, 2, 3, 9, 12, 13, 16, 36, 40):
        x = gpu(workloads.rhs(P.n, B, B), torch.float32)
        P.tune_set(B, np.zeros(M.TUNE_FIELDS, np.int32))
        y0 = P.matvec(x).cpu().numpy()
        for u, d in ((304, 304), (754, 854), (758, 804)):
            c = np.zeros(M.TUNE_FIELDS, np.int32)
            c[3 + 2], c[3 + 3], c[3 + L + 2], c[3 + L + 3] = u, u, d, d
            P.tune_set(B, c)
            assert rel(P.matvec(x).cpu().numpy(), y0) < 1e-5, (B, u, d)
    P.close()
