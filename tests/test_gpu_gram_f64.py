"""The FP64 Gram on tensor cores (csrc/gram_f64.cu) at the edges of its tiles,
K blocks, accumulator chunks and integer segments, against the same Gram in
extended precision, and its route to the CUDA cores for data whose columns
the digits do not resolve.

Tolerance, relative to sqrt(s_ii s_jj): the preparation rounds every z twice
and takes its scale from an FP64 sum of n squares in chunks (n / 32 + 32
additions, half of their relative error in the scale, twice in S), the
products and the sum round as an FP64 sum of n products in the worst case:
(n / 32 + 32 + 8) 2^-53 + n 2^-53 on the CUDA cores and less with digits."""
import numpy as np
import pytest

from paper_2106_09382_gb300 import concord as C

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def data(n, p, seed):
    rng = np.random.default_rng(seed)
    X = rng.standard_normal((n, p))
    X[:, 1:] += 0.5 * X[:, :-1]
    return X * rng.uniform(0.5, 3.0, p) + rng.uniform(-2, 2, p)


def rows_of(X, prep, pick):
    """Rows `pick` of S and the norms sqrt(s_ii), in extended precision."""
    Z = X.astype(np.longdouble)
    if prep >= 1:
        Z = Z - Z.mean(0)
    ss = (Z * Z).sum(0)
    if prep == 2:
        Z = Z / np.sqrt(ss / len(X))
        ss = (Z * Z).sum(0)
    return (Z[:, pick].T @ Z) / len(X), np.sqrt(ss / len(X))


def check(X, prep, S):
    n, p = X.shape
    pick = np.unique(np.r_[0, p - 1, p // 2, np.arange(min(p, 7)) * (p // 7 or 1) % p, min(p - 1, 127),
                           min(p - 1, 128)])
    want, norm = rows_of(X, prep, pick)
    tol = (n / 32 + 40 + n) * 2.0 ** -53
    assert np.array_equal(S, S.T)
    err = np.abs(S[pick].astype(np.longdouble) - want) / (norm[pick][:, None] * norm[None, :])
    assert err.max() <= tol, (float(err.max()), tol)
    return float(err.max())


SIZES = [(31, 5), (32, 2), (33, 127), (64, 128), (65, 129), (127, 257), (128, 64), (129, 40),
         (200, 300), (257, 384), (1000, 131), (14336, 40), (14339, 33), (29000, 17)]


@pytest.mark.parametrize("n,p", SIZES)
def test_edges_against_extended_precision(n, p):
    X = data(n, p, n + p)
    for prep in (C.PREP_NONE, C.PREP_CENTER, C.PREP_STANDARDIZE):
        for dt in (torch.float64, torch.float32):
            Xt = torch.as_tensor(X, dtype=dt, device="cuda")
            S = C.concord_gram(Xt, prep, C.GRAM_FP64)
            check(Xt.double().cpu().numpy(), prep, S.cpu().numpy())


def test_row_stride_and_out_of_place_stride():
    X = torch.as_tensor(data(300, 200, 1), device="cuda")
    wide = torch.full((300, 211), float("nan"), dtype=torch.float64, device="cuda")
    wide[:, 3:203] = X
    S = C.concord_gram(wide[:, 3:203], C.PREP_STANDARDIZE, C.GRAM_FP64)
    assert torch.equal(S, C.concord_gram(X, C.PREP_STANDARDIZE, C.GRAM_FP64))


@pytest.mark.parametrize("scale", [1e-140, 1.0, 1e140])
def test_columns_the_digits_do_not_resolve(scale):
    """One entry 1e12 times its column's others: against the columns that are
    zero in its row, S rests on the small entries alone.  Their sum is held
    to the FP64 bound relative to those entries, which digits relative to
    the column's largest would miss by 2^17."""
    X = data(400, 150, 3) * scale
    X[0, :] = 0.0
    X[0, 5] = 1e12 * scale
    S = C.concord_gram(torch.as_tensor(X, device="cuda"), C.PREP_NONE, C.GRAM_FP64).cpu().numpy()
    Y = X[1:].astype(np.longdouble)
    want = Y[:, 5] @ Y / len(X)
    bound = np.abs(Y[:, 5]) @ np.abs(Y) / len(X) * (400 + 2) * 2.0 ** -53
    others = np.arange(150) != 5
    assert (np.abs(S[5].astype(np.longdouble) - want) <= bound)[others].all()
    assert np.array_equal(S, S.T)


def test_zero_columns_and_one_value_columns():
    X = data(100, 140, 4)
    X[:, 9] = 0.0
    X[:, 77] = 3.0
    S = C.concord_gram(torch.as_tensor(X, device="cuda"), C.PREP_NONE, C.GRAM_FP64).cpu().numpy()
    assert not S[9].any() and not S[:, 9].any()
    assert S[77, 77] == 9.0
    S = C.concord_gram(torch.as_tensor(X, device="cuda"), C.PREP_CENTER, C.GRAM_FP64).cpu().numpy()
    assert not S[9].any() and not S[77].any()


def test_solve_state_follows_the_route():
    """A state's Gram (its kept workspace) equals the free-standing one, on
    both routes and for fewer rows than the state holds."""
    X = torch.as_tensor(data(300, 120, 5), device="cuda")
    Y = X.clone()
    Y[0, 3] += 1e7
    with C.State(120, C.FP64, n_cap=300) as st:
        for A in (X, Y, X[:40].contiguous(), X[:31].contiguous(), X):
            st.solve_device(A, 0.9, tol=1e-6)
            S = C.concord_gram(A, C.PREP_STANDARDIZE, C.GRAM_FP64)
            st2 = C.State(120, C.FP64)
            st2.set_S(S)
            st2.run(0.9, tol=1e-6)
            assert torch.equal(st.get_omega(), st2.get_omega())
            st2.close()
