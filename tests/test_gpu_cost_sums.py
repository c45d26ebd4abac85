"""The sums behind the selection and d_KL in the float32 forms, against what float64 sums give.
An infinite term (z = 0 where v > 0) leaves +infinity, not a value that no comparison holds
for; the call reports DNA_ERR_NONFINITE all the same.  Terms that are exact in float32 and
whose sum is exact in float64 are added exactly, and sums past float32's range stay finite."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _lib():
    import paper_1301_3389_gb300._lib as L
    return L


class Bound:
    """V, W, H bound to a context of the dense or sparse form, or to a group of one problem."""

    def __init__(self, form, V, W, H):
        import torch
        L = self.L = _lib()
        self.form = form
        self.N, self.T = V.shape
        R = W.shape[1]
        V, self.W, self.H = (torch.from_numpy(np.ascontiguousarray(x, dtype=np.float32)).cuda()
                             for x in (V, W, H))
        self.keep = [V]
        bf16 = form in ("bf16", "group_bf16")
        opts = L.make_opts(dtype=L.DNA_BF16 if bf16 else L.DNA_F32)
        if form.startswith("group"):
            self.h = L.dna_group_create([self.N], [self.T], [R], opts)
            L.dna_group_set_stream(self.h)
            L.dna_group_bind(self.h, [V], [self.W], [self.H])
        elif form == "sparse":
            nz = V.nonzero()
            rows = torch.bincount(nz[:, 0], minlength=self.N).cumsum(0)
            self.keep = [torch.cat([rows.new_zeros(1), rows]), nz[:, 1].to(torch.int32),
                         V[nz[:, 0], nz[:, 1]].contiguous()]
            self.h = L.dna_create_sparse(self.N, self.T, R, nz.shape[0], opts)
            L.dna_set_stream(self.h)
            L.dna_bind_csr(self.h, *self.keep, self.W, self.H)
        else:
            self.h = L.dna_create(self.N, self.T, R, opts)
            L.dna_set_stream(self.h)
            L.dna_bind(self.h, V, self.W, self.H)

    def __enter__(self):
        return self

    def __exit__(self, *exc):
        (self.L.dna_group_destroy if self.form.startswith("group") else self.L.dna_destroy)(self.h)

    def step(self, which):
        g = "group_" if self.form.startswith("group") else ""
        getattr(self.L, f"dna_{g}step_{'HW'[which]}")(self.h)

    def kl(self):
        """(return code, value)"""
        if self.form.startswith("group"):
            out = np.zeros(1)
            return self.L.LIB.dna_group_kl(self.h, out.ctypes.data), float(out[0])
        out = ctypes.c_double()
        return self.L.LIB.dna_kl(self.h, ctypes.byref(out)), out.value

    def choice(self, which):
        out = np.zeros((self.T, self.N)[which], dtype=np.uint8)
        if self.form.startswith("group"):
            code = self.L.LIB.dna_group_get_choice(self.h, 0, which, out.ctypes.data, len(out))
        else:
            code = self.L.LIB.dna_get_choice(self.h, which, out.ctypes.data, len(out))
        return code, out

    def costs(self, which):
        dm, dd = np.zeros((self.T, self.N)[which]), np.zeros((self.T, self.N)[which])
        code = self.L.LIB.dna_get_costs(self.h, which, dm.ctypes.data, dd.ctypes.data, len(dm))
        return code, dm, dd


@pytest.mark.parametrize("which", [0, 1])
@pytest.mark.parametrize("form,R", [("f32", 2), ("f32", 70), ("f32", 120), ("group_f32", 2),
                                    ("group_f32", 50), ("sparse", 2), ("sparse", 40),
                                    ("sparse", 120)])
def test_infinite_mu_cost_keeps_newton(form, R, which):
    """Column 0 (row 0 for the W step): the MU gain of component a is v y / z = 2e-38, so the
    MU z of row 0, 1e-8 * 2e-38, underflows to 0 where v = 2e-38 > 0: infinite cost.  The
    Newton gain is floored at eps = 0.01 and its cost is finite.  Component b is R - 1 equal
    components, each an equal share."""
    V = np.array([[2e-38, 0.0, 1.0], [0.0, 1.0, 2.0], [1.0, 1.0, 3.0]])
    Y = np.array([[1e-8, 0.0], [1.0, 0.0], [0.0, 1.0]])[:, [0] + (R - 1) * [1]]
    X = np.ones((R, 3))
    X[1:] /= R - 1
    # the third column needs z > 0 everywhere; its selection does not matter
    with Bound(form, *((V, Y, X) if which == 0 else (V.T, X.T, Y.T))) as b:
        b.step(which)
        code, choice = b.choice(which)
        assert code == b.L.DNA_ERR_NONFINITE and choice[0] == 1
        if not form.startswith("group"):
            code, dm, dd = b.costs(which)
            assert code == b.L.DNA_ERR_NONFINITE
            assert dm[0] == np.inf and np.isfinite(dd[0]) and np.isfinite(dm[1:]).all()


@pytest.mark.parametrize("form,R", [(f, R) for f in ("f32", "bf16", "group_f32", "group_bf16",
                                                    "sparse") for R in (4, 40)] +
                         [("f32", 90), ("f32", 128), ("bf16", 100), ("sparse", 128)])
def test_infinite_kl(form, R):
    rng = np.random.default_rng(R)
    V, W, H = rng.random((150, 70)) + 0.1, rng.random((150, R)), rng.random((R, 70))
    W[5] = 0.0
    with Bound(form, V, W, H) as b:
        assert b.kl() == (b.L.DNA_ERR_NONFINITE, np.inf)


# 1 + 2^-27 + 2^-52: exact in float64, and neither in float32 nor in a pair of float32 values
PARTS = (1.0, 2.0 ** -27, 2.0 ** -52)
# columns of the dense problems: two o-blocks of 64 per SM, so that one CTA runs over all rows
COLS = 2 * 64 * 152


def _spread(rows, values, N, T):
    """V = 0 (N x T), W (N x 1) with `values` in `rows`, H (1 x T) with 1 in column 0."""
    W = np.zeros((N, 1))
    W[list(rows), 0] = values
    H = np.zeros((1, T))
    H[0, 0] = 1.0
    return np.zeros((N, T), dtype=np.float32), W, H


@pytest.mark.parametrize("form,rows,N", [("f32", (0, 64, 128), 192), ("bf16", (0, 64, 128), 192),
                                         ("group_f32", (0, 64, 128), 192),
                                         ("group_bf16", (0, 64, 128), 192),
                                         ("f32", (0, 64 * 300, 64 * 301), 64 * 310)])
def test_kl_exact(form, rows, N):
    """d_KL of V = 0 is the sum of z: the rows' values, each in another chunk of one thread."""
    V, W, H = _spread(rows, PARTS, N, 1 if form.startswith("group") else COLS)
    with Bound(form, V, W, H) as b:
        assert b.kl() == (b.L.DNA_OK, sum(PARTS))


def test_kl_exact_sparse():
    """v = z at three non-zeros: each term v log(v / z) - v is -v, and their sum and that of z
    cancel exactly (rows of different 32-row blocks, so that the sum of z is exact too)."""
    W = np.zeros((70, 1))
    W[[0, 32, 64], 0] = PARTS
    with Bound("sparse", W, W, np.ones((1, 1))) as b:
        assert b.kl() == (b.L.DNA_OK, 0.0)


@pytest.mark.parametrize("form,rows,N", [("f32", (0, 64, 128), 192), ("sparse", (0, 32, 64), 70)])
def test_costs_exact(form, rows, N):
    """v = z = 1 at one entry (a = 0, so both candidates are the starting x = 1, and log z = 0)
    and v = 0 elsewhere: both costs are the sum of z."""
    V, W, H = _spread(rows, PARTS, N, COLS if form == "f32" else 1)
    V[0, 0] = 1.0
    with Bound(form, V, W, H) as b:
        b.step(0)
        code, dm, dd = b.costs(0)
        assert code == b.L.DNA_OK and dm[0] == sum(PARTS) and dd[0] == sum(PARTS)


@pytest.mark.parametrize("form,N", [("f32", 256), ("sparse", 256)])
def test_costs_past_float32_range(form, N):
    """v = z = 2e36 in four rows: -v log z is -1.7e38 in each, -6.7e38 in all.  Both candidates
    are the starting column up to rounding: 1e-5 of the sum (float32 terms, |z' / z - 1| and
    |log z' - log z| / 84 a few float32 roundings)."""
    rows, v = (0, 64, 128, 192), float(np.float32(2e36))
    V, W, H = _spread(rows, 1.0, N, COLS if form == "f32" else 1)
    V[list(rows), 0] = v
    H[0, 0] = v
    ref = 4.0 * (v - v * np.log(v))
    with Bound(form, V, W, H) as b:
        b.step(0)
        code, dm, dd = b.costs(0)
        assert code == b.L.DNA_OK
        assert abs(dm[0] - ref) <= 1e-5 * abs(ref) and abs(dd[0] - ref) <= 1e-5 * abs(ref)


def test_kl_past_float32_range():
    """V = 0, z = 2e38 in two rows of different chunks: their sum."""
    z = np.float32(2e38)
    for form, T in (("f32", COLS), ("group_f32", 1)):
        with Bound(form, *_spread((0, 64), z, 128, T)) as b:
            assert b.kl() == (b.L.DNA_OK, 2.0 * float(z))
