"""Submatrices whose rows are of very different size: A = D S0 D with a well-conditioned S0.

Floating point keeps such rows' relative precision; a fixed point per submatrix does not, so those submatrices are
computed in FP64.  The reference is the same iteration in extended precision (numpy longdouble: 64 or 113 bits).

Tolerance, relative to the largest entry of the result: the iterations take up to about 45 steps of three products
here; an FP64 product of graded factors has an error of a few 2^-53 per entry relative to the entry's own scale
d_i d_j, which enters the next step with a factor of about one.  45 * 3 * 2^-53 = 1.5e-14; 2e-14 is asserted.
"""

import numpy as np
import pytest

from synth import make_mixed_block_system

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 2e-14
N = 24
SCALES = [1.0, 0.3, 0.1, 1e-2, 1e-3, 1e-4, 1e-6]


@pytest.fixture(scope="module", autouse=True)
def _need_cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _graded(kind, d, seed, n=N):
    """A symmetric matrix with rows scaled by 1 .. d: positive definite, or indefinite with a gap."""
    rng = np.random.default_rng(seed)
    g = rng.standard_normal((n, n))
    if kind == "positive":
        a = np.eye(n) + 0.2 / np.sqrt(n) * (g + g.T)
    else:
        q = np.linalg.qr(g)[0]
        a = (q * (np.where(np.arange(n) % 2, 0.5, -0.5) * rng.uniform(0.8, 1.2, n))) @ q.T
    dd = np.where(rng.permutation(n) < n // 2, 1.0, d)
    a = a * dd[:, None] * dd[None, :]
    return 0.5 * (a + a.T)


def _matmul(a, b):
    return np.stack([(a[i][:, None] * b).sum(0) for i in range(a.shape[0])])


def _roots(a):
    """(A^1/2, A^-1/2) by the coupled iteration in extended precision."""
    n = a.shape[0]
    b = np.longdouble(np.abs(a).sum(1).max())
    y, z, eye = a.astype(np.longdouble) / b, np.eye(n, dtype=np.longdouble), np.eye(n, dtype=np.longdouble)
    for _ in range(100):
        zy = _matmul(z, y)
        t = (3 * eye - zy) / 2
        y, z = _matmul(y, t), _matmul(t, z)
        if float(np.abs(zy - eye).max()) < 1e-11:
            break
    return y * np.sqrt(b), z / np.sqrt(b)


def _sign(a):
    n = a.shape[0]
    x, eye = a.astype(np.longdouble) / np.longdouble(np.abs(a).sum(1).max()), np.eye(n, dtype=np.longdouble)
    for _ in range(200):
        x2 = _matmul(x, x)
        x = _matmul(x, (3 * eye - x2) / 2)
        if float(np.abs(x2 - eye).max()) < 1e-11:
            break
    return x


def _reference(f, a):
    if f == "density":
        return (np.eye(a.shape[0]) - _sign(a)) / 2
    root, inv = _roots(a)
    return {"sqrt": root, "inv_sqrt": inv, "inv": _matmul(inv, inv)}[f]


def _full(h, block):
    """The values of h on a complete pattern of equal blocks (column-major blocks, columns in order)."""
    m = h.shape[0] // block
    return h.reshape(m, block, m, block).transpose(2, 0, 3, 1).ravel()


def _dense(v, n, block):
    m = n // block
    return v.reshape(m, m, block, block).transpose(1, 3, 0, 2).reshape(n, n)


def _context(h, block):
    from paper_2205_14741_gb300 import SubmatrixDensity

    s = make_mixed_block_system([block] * (h.shape[0] // block), r_c=np.inf, ell=1.5, seed=1)
    c = SubmatrixDensity.from_system(s)
    c.set_values(_full(h, block))
    return c


def _error(got, ref):
    return float(np.max(np.abs(got - ref)) / np.max(np.abs(ref)))


@pytest.mark.parametrize("d", SCALES)
@pytest.mark.parametrize("f", ["inv_sqrt", "sqrt", "inv", "density"])
def test_functions_of_graded_matrices(f, d):
    for seed in range(3):
        h = _graded("indefinite" if f == "density" else "positive", d, seed)
        for block in (N, 2):  # one submatrix, and twelve (a cluster to each)
            with _context(h, block) as c:
                c.set_function(f)
                c.build_density()
                c.get_trace()
                got = _dense(c.get_density(), N, block)
            assert _error(got, _reference(f, h)) <= TOL, (seed, block)


@pytest.mark.parametrize("d", SCALES)
def test_dense_entry_point_on_graded_matrices(d):
    from paper_2205_14741_gb300 import dense_density_noalloc

    for n in (N, 100):
        h = _graded("indefinite", d, 5, n)
        hd = torch.from_numpy(h).cuda()
        out = torch.empty_like(hd)
        dense_density_noalloc(hd, n, 0.0, out)
        assert _error(out.cpu().numpy(), _reference("density", h)) <= TOL


@pytest.mark.parametrize("mode", ["rho", "gap"])
def test_learned_bound_on_graded_matrices(mode):
    h = _graded("indefinite", 1e-3, 4)
    with _context(h, 2) as c:
        c.bound_model_init(3)
        c.bound_model_collect(24)
        c.bound_model_train(epochs=50, batch=12, lr=2e-3)
        c.set_bound_model(mode)
        c.build_density()
        c.get_trace()
        got = _dense(c.get_density(), N, 2)
    assert _error(got, _reference("density", h)) <= TOL


@pytest.mark.parametrize("d", SCALES)
def test_fermi_keeps_the_small_rows_digits(d):
    # two uncoupled parts, one d times the other: off the diagonal F is -tanh / 2, of the part's own size
    h = np.zeros((N, N))
    h[:12, :12] = _graded("indefinite", 1.0, 1, 12)
    h[12:, 12:] = d * _graded("indefinite", 1.0, 2, 12)
    with _context(h, N) as c:
        c.set_function("fermi")
        c.set_fermi_beta(2.0)
        c.build_density()
        c.get_trace()
        got = _dense(c.get_density(), N, N)
    lam, v = np.linalg.eigh(h[12:, 12:] / d)
    ref = -0.5 * (v * np.tanh(d * lam)) @ v.T
    off = ~np.eye(12, dtype=bool)
    # (numpy's own eigendecomposition, and the entries' rounding when F is formed beside 1/2 on the diagonal)
    assert float(np.max(np.abs(got[12:, 12:] - ref)[off])) <= 1e-13 * float(np.max(np.abs(ref)))


@pytest.mark.parametrize("d", SCALES[:5])
@pytest.mark.parametrize("which", ["overlap", "both", "hamiltonian"])
def test_nonorthogonal_form_of_graded_matrices(which, d):
    # P = 1/2 (I - sign(S^-1 H)) S^-1.  With a graded H, M = L H L is not: its eigenvalues of the order of 0.3 d^2
    # lie beside ones of order 1 in full rows, so the rounding of the two products that form M, 3 * 2^-53 in all,
    # turns its sign by up to 1e-15 / d^2 in any arithmetic of 53 bits
    h = _graded("indefinite", d if which != "overlap" else 1.0, 6)
    s = _graded("positive", d if which != "hamiltonian" else 1.0, 6)
    with _context(h, 2) as c:
        c.set_overlap(_full(s, 2))
        c.build_density()
        c.get_trace()
        got = _dense(c.get_density(), N, 2)
    _, root = _roots(s)
    sign = _sign(_matmul(_matmul(root, h.astype(np.longdouble)), root))
    ref = _matmul(_matmul(root, (np.eye(N) - sign) / 2), root)
    assert _error(got, ref) <= TOL + (0.0 if which == "overlap" else 1e-15 / d ** 2)


@pytest.mark.parametrize("f", ["density", "inv", "fermi", "sqrt", "overlap"])
def test_clusters_on_graded_matrices(f):
    # 100 submatrices take one SM each; column ranges of 60, 30 and 9 take clusters of two, four and eight
    h = _graded("indefinite" if f in ("density", "fermi", "overlap") else "positive", 0.01, 7, 200)
    with _context(h, 2) as c:
        if f == "overlap":
            c.set_overlap(_full(_graded("positive", 0.01, 7, 200), 2))
        else:
            c.set_function(f)
            c.set_fermi_beta(12.0)
        c.build_density()
        c.get_trace()
        full = c.get_density().reshape(100, -1)
        for j0, j1 in ((3, 63), (40, 70), (91, 100)):
            c.set_column_range(j0, j1)
            c.build_density()
            c.get_trace()
            got = c.get_density().reshape(100, -1)[j0:j1]
            # (the same products; the residual, which decides the last step, is summed in another order)
            assert float(np.max(np.abs(got - full[j0:j1]))) <= TOL * float(np.max(np.abs(full))), (j0, j1)


def test_graded_and_other_submatrices_in_one_build():
    # 200 block columns, the rows of every fifth block a thousandth: some submatrices hold such rows, others not.  In one
    # and in several staging chunks, with the bisection decided on the host and on the device: the same bits
    from paper_2205_14741_gb300 import SubmatrixDensity
    from oracle import block_value_offsets, density_submatrix

    s = make_mixed_block_system([4] * 200, r_c=4.0, ell=1.0, seed=12)
    off = block_value_offsets(s.block_size, s.col_ptr, s.row_idx)
    scale = np.where(np.arange(200) % 5 == 0, 1e-3, 1.0)
    for j in range(200):
        for k in range(s.col_ptr[j], s.col_ptr[j + 1]):
            s.values[off[k]:off[k + 1]] *= scale[j] * scale[s.row_idx[k]]
    small = [bool(np.any(scale[s.row_idx[s.col_ptr[j]:s.col_ptr[j + 1]]] < 1.0)) for j in range(200)]
    assert 40 < sum(small) < 200
    with SubmatrixDensity.from_system(s) as c:
        c.build_density()
        whole, trace = c.get_density(), c.get_trace()[0]
        ref = density_submatrix(s.block_size, s.col_ptr, s.row_idx, s.values, 0.0)
        # the oracle's eigendecomposition sees the small rows to 2^-53 of the large ones: to 1e-10 of their own size
        assert float(np.max(np.abs(whole - ref.values))) <= 1e-8
        assert abs(trace - ref.trace) <= 1e-8 * s.n
        c.set_staging_limit(1 << 20)
        c.build_density()
        assert np.array_equal(c.get_density(), whole) and c.get_trace()[0] == trace
        c.set_electron_count(trace - 3.0, max_steps=6, tol=1e-12)
        c.solve_mu()
        host = c.get_density(), c.get_trace()
        c.solve_mu_device()
        assert np.array_equal(c.get_density(), host[0]) and c.get_trace() == host[1]


@pytest.mark.parametrize("f", ["inv_sqrt", "density", "overlap"])
def test_rows_at_the_line_between_the_forms(f):
    # a ratio of the rows at 1/8 and within a few roundings of it, and roots of such an overlap: whichever form takes them
    for step in range(-4, 5):
        d = np.full(N, 1.0)
        d[5::3] = 0.125 * (1.0 + step * 2.0 ** -23)
        s = np.diag(d)
        h = np.diag(np.where(np.arange(N) % 2, d, -d))
        with _context(h if f in ("density", "overlap") else s, 2) as c:
            if f == "overlap":
                c.set_overlap(_full(s, 2))
            elif f != "density":
                c.set_function(f)
            c.build_density()
            c.get_trace()
            got = _dense(c.get_density(), N, 2)
        below = np.diag(np.where(np.arange(N) % 2, 0.0, 1.0))
        ref = {"inv_sqrt": np.diag(d ** -0.5), "density": below, "overlap": below / d}[f]
        assert _error(got, ref) <= TOL, step
