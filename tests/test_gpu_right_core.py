"""The angular core of a rounded two-core state has orthonormal rows, as tt_internal_ranks asks for it, whatever
the singular values are: close to each other, graded below the round-off of the largest, or zero.

Bar: the root mean square of the entries of V V^T - I below two units of 2^-52.  An element of the core is off by
at most two units of itself (a product and a sum of a polar step, or a subtraction and a division), so an
entry of V V^T by at most four."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ROWS = 1100
ORDINATES = [1, 2, 8, 16, 31, 32, 33, 40, 64]


@pytest.fixture(scope="module")
def tt():
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    import __graft_entry__
    __graft_entry__.build()
    import paper_2602_00290_gb300 as mod
    return mod


def rounded(tt, a, b):
    ctx = tt.Context(0)
    r = a.shape[1]
    x = tt.TT.from_cores([a[None], b[:, :, None]], rcap=[r])
    tt.tt_round(ctx, x, 0.0, r, "fp64")
    ctx.sync()
    z, v = x.to_cores()
    z, v = z[0], v[:, :, 0]
    want = a @ b
    assert np.linalg.norm(z @ v - want) <= 1e-13 * np.linalg.norm(want)
    return np.sqrt(np.mean((v @ v.T - np.eye(v.shape[0])) ** 2))


@pytest.mark.parametrize("grade", [1.0, 0.8, 0.4])
@pytest.mark.parametrize("n", ORDINATES)
def test_graded_singular_values(tt, n, grade):
    rng = np.random.default_rng(n)
    a = np.linalg.qr(rng.standard_normal((ROWS, n)))[0] * grade ** np.arange(n)
    b = np.linalg.qr(rng.standard_normal((n, n)))[0]
    assert rounded(tt, a, b) <= 2.0 * 2.0 ** -52


@pytest.mark.parametrize("n", [8, 32, 40])
def test_dependent_columns(tt, n):
    rng = np.random.default_rng(n)
    a = rng.standard_normal((ROWS, 3)) @ rng.standard_normal((3, n))
    b = np.linalg.qr(rng.standard_normal((n, n)))[0]
    assert rounded(tt, a, b) <= 2.0 * 2.0 ** -52


@pytest.mark.parametrize("n", [8, 40])
def test_zero_state(tt, n):
    assert rounded(tt, np.zeros((ROWS, n)), np.linalg.qr(np.random.default_rng(n).standard_normal((n, n)))[0]) <= 2.0 * 2.0 ** -52
