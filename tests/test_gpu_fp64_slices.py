"""The 64-bit forms at the edges of their tensor-core products (digit slices with exact FP32 sums):
dimensions around the 32-row padding, the 64-column tiles, the 128-row blocks and the 192-long exact
sums; operands of extreme magnitude; owner blocks of every width class in the non-orthogonal form.

Tolerance.  A product drops the digit pairs of weight 9 and above: at most 6 K 2^14 2^-72 per entry in the
worst case, about 3.4e-17 sqrt(K / 158) when the digits are uncorrelated; a solve takes up to about 30
products whose errors enter the next ones with factors of at most 2.5.  30 * 2.5 * 3.4e-17 * sqrt(400 / 158) is
4e-15; the oracle's eigendecomposition adds a few 1e-15.  2e-14 max-abs leaves a factor of two or more.
"""

import numpy as np
import pytest

import oracle as O
from synth import make_mixed_block_system, make_nonorth_pair, make_overlap_system, spectrum_matrix

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 2e-14


@pytest.fixture(scope="module", autouse=True)
def _need_cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _gapped(n, seed):
    rng = np.random.default_rng(seed)
    return spectrum_matrix(n, np.where(np.arange(n) < n // 2, -1.0, 1.0) * rng.uniform(0.3, 0.7, n), seed)


def _dense(h, mu=0.0):
    from paper_2205_14741_gb300 import dense_density_noalloc

    hd = torch.from_numpy(np.ascontiguousarray(h)).cuda()
    d = torch.full_like(hd, float("nan"))
    dense_density_noalloc(hd, h.shape[0], mu, d)
    return d.cpu().numpy()


@pytest.mark.parametrize("n", [1, 2, 31, 32, 33, 63, 64, 65, 96, 97, 127, 128, 129, 160, 161, 191, 192, 193, 224, 255, 256])
def test_dense_at_tile_edges(n):
    h = _gapped(n, 100 + n)
    assert float(np.max(np.abs(_dense(h) - O.dense_density(h, 0.0)))) <= TOL


@pytest.mark.parametrize("power", [-300, -40, 40, 300])
def test_power_of_two_scaling_changes_no_bit(power):
    h = _gapped(72, 5)
    assert np.array_equal(_dense(np.ldexp(h, power)), _dense(h))


def test_entries_of_very_different_size():
    # exact zeros, subnormal products and a coherent (rank-one plus diagonal) matrix, whose digits all agree
    n = 160
    v = np.ones(n) / np.sqrt(n)
    h = 0.5 * np.eye(n) - 0.95 * np.outer(v, v)
    assert float(np.max(np.abs(_dense(h) - O.dense_density(h, 0.0)))) <= TOL
    h = np.zeros((64, 64))
    h[np.arange(64), np.arange(64)] = np.where(np.arange(64) % 2, 1.0, -1.0) * np.linspace(0.3, 1.0, 64)
    h[0, 1] = h[1, 0] = 1e-200
    assert float(np.max(np.abs(_dense(h) - O.dense_density(h, 0.0)))) <= TOL


@pytest.mark.parametrize("sizes", [[33, 32], [64, 64, 64, 1], [64] * 5 + [7]])
@pytest.mark.parametrize("f", ["inv_sqrt", "sqrt", "inv", "fermi", "density"])
def test_functions_on_full_patterns(sizes, f):
    # every submatrix is the whole matrix: n = 65, 193 and 327 (contractions in one and two exact parts)
    from paper_2205_14741_gb300 import SubmatrixDensity

    s = make_mixed_block_system(sizes, r_c=np.inf, ell=1.5, seed=3)
    h = O.to_dense(s.block_size, s.col_ptr, s.row_idx, s.values)
    if f in ("inv_sqrt", "sqrt", "inv"):  # positive definite: eigenvalues in about [0.5, 3]
        shift = 2.0 - 0.5 * float(np.linalg.eigvalsh(h)[0] + np.linalg.eigvalsh(h)[-1])
    else:
        shift = 0.0
    with SubmatrixDensity.from_system(s) as c:
        c.set_function(f)
        c.set_fermi_beta(12.0)
        c.set_mu(-shift)
        c.build_density()
        got = O.to_dense(s.block_size, s.col_ptr, s.row_idx, c.get_density())
    lam, v = np.linalg.eigh(h + shift * np.eye(h.shape[0]))
    fn = {"inv_sqrt": lambda x: x ** -0.5, "sqrt": np.sqrt, "inv": lambda x: 1.0 / x,
          "fermi": lambda x: 0.5 * (1.0 - np.tanh(6.0 * x)), "density": lambda x: 0.5 * (1.0 - np.sign(x))}[f]
    ref = (v * fn(lam)) @ v.T
    assert float(np.max(np.abs(got - ref))) <= TOL * max(1.0, float(np.max(np.abs(ref))))


@pytest.mark.parametrize("b", [1, 16, 17, 33])
def test_nonorthogonal_owner_widths(b):
    # the thin products of the owner columns: widths padded to 16, 32 and 64
    from paper_2205_14741_gb300 import SubmatrixDensity

    h, s = make_nonorth_pair(8, b, np.inf, 1.5, 9, sigma_s=0.01 if b > 16 else 0.05)
    with SubmatrixDensity.from_system(h) as c:
        c.set_overlap(s.values)
        c.set_mu(0.02)
        c.build_density()
        got = O.to_dense(h.block_size, h.col_ptr, h.row_idx, c.get_density())
    a = O.to_dense(h.block_size, h.col_ptr, h.row_idx, h.values)
    lam, v = np.linalg.eigh(O.to_dense(h.block_size, h.col_ptr, h.row_idx, s.values))
    root = (v * lam ** -0.5) @ v.T
    mu, w = np.linalg.eigh(root @ a @ root)
    ref = root @ (w * (0.5 * (1.0 - np.sign(mu - 0.02)))) @ w.T @ root
    assert float(np.max(np.abs(got - ref))) <= TOL * max(1.0, float(np.max(np.abs(ref))))


def test_not_positive_definite_is_reported():
    from paper_2205_14741_gb300 import SmxError, SubmatrixDensity, _lib

    s = make_overlap_system(16, 6, np.inf, 1.5, 7)
    with SubmatrixDensity.from_system(s) as c:
        c.set_function("inv_sqrt")
        c.set_mu(1.0)  # eigenvalues on both sides of zero
        with pytest.raises(SmxError) as e:
            c.build_density()
            c.get_trace()
        assert e.value.status in (_lib.ERR_NOCONV, _lib.ERR_NONFINITE)
        c.set_mu(0.0)
        c.build_density()
        c.get_trace()


@pytest.mark.parametrize("f", ["density", "inv", "fermi", "overlap"])
@pytest.mark.parametrize("m,b", [(100, 2), (100, 1)])
def test_clusters_change_no_bit(m, b, f):
    # 100 submatrices take one SM each; column ranges of 60, 30 and 9 take clusters of two, four and eight SMs
    # (n = 200; at n = 100 up to four).  Sums are of integers, and every SM decides from the same ones.
    from paper_2205_14741_gb300 import SubmatrixDensity

    if f == "overlap":
        h, s = make_nonorth_pair(m, b, np.inf, 1.5, 9, sigma_s=0.02)
    else:
        h, s = make_mixed_block_system([b] * m, r_c=np.inf, ell=1.5, seed=4), None
    with SubmatrixDensity.from_system(h) as c:
        if s is not None:
            c.set_overlap(s.values)
        else:
            c.set_function(f)
            c.set_fermi_beta(12.0)
        lam = np.linalg.eigvalsh(O.to_dense(h.block_size, h.col_ptr, h.row_idx, h.values))
        c.set_mu(float(lam[0]) - 0.5 if f == "inv" else 0.02)
        c.build_density()
        full = c.get_density().reshape(m, -1)
        for j0, j1 in ((3, 63), (40, 70), (91, 100)):
            c.set_column_range(j0, j1)
            c.build_density()
            assert np.array_equal(c.get_density().reshape(m, -1)[j0:j1], full[j0:j1]), (j0, j1)


@pytest.mark.parametrize("precision", ["fp64", "fp16x3"])
def test_staged_gather_around_48_kb(precision):
    # row stages just below and above 48 KB of dynamic shared memory, beside the kernel's static arrays
    from paper_2205_14741_gb300 import SubmatrixDensity

    for blocks in list(range(15, 24)) + [30, 34, 38, 42]:
        s = make_mixed_block_system([6] * blocks, r_c=np.inf, ell=1.5, seed=blocks)
        h = O.to_dense(s.block_size, s.col_ptr, s.row_idx, s.values)
        lam, v = np.linalg.eigh(h)
        k = int(np.argmax(np.diff(lam)))  # mu in the middle of the widest gap
        with SubmatrixDensity.from_system(s) as c:
            c.set_precision(precision)
            c.set_mu(0.5 * float(lam[k] + lam[k + 1]))
            c.build_density()
            got = O.to_dense(s.block_size, s.col_ptr, s.row_idx, c.get_density())
        tol = 1e-10 if precision == "fp64" else 1e-5  # the parity bounds of the two forms
        assert float(np.max(np.abs(got - v[:, :k + 1] @ v[:, :k + 1].T))) <= tol, blocks


@pytest.mark.parametrize("n", [64, 160, 192])
def test_finishing_steps_start_from_a_symmetric_iterate(n):
    # every submatrix of a full pattern has the same iterate, so D's asymmetry is that iterate's; the bulk phase's
    # is about 1e-7, and what the mean with the transpose leaves is the rounding of the last product
    from paper_2205_14741_gb300 import SubmatrixDensity

    s = make_mixed_block_system([1] * n, r_c=np.inf, ell=1.5, seed=6)
    with SubmatrixDensity.from_system(s) as c:
        c.set_precision("fp16x3", 1)
        c.set_mu(0.02)
        c.build_density()
        d = O.to_dense(s.block_size, s.col_ptr, s.row_idx, c.get_density())
    assert float(np.max(np.abs(d - d.T))) <= 1e-14
