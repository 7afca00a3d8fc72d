"""The 64-bit forms where their fixed-point arithmetic, their memory or their claims end: sizes, magnitudes and
submatrices that fail."""

import numpy as np
import pytest

import oracle as O
from synth import make_mixed_block_system

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _need_cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


@pytest.mark.parametrize("columns", [3, 131])
def test_fp64_past_the_rows_whose_bound_fits_shared_memory(columns):
    # n = 2081: the vectors of the first bound lie in global memory; a submatrix to a cluster, and one to a CTA.
    # D is known: a reflection I - 2 V V^T with 5 columns V, scaled by 1/2.
    from paper_2205_14741_gb300 import SubmatrixDensity

    s = make_mixed_block_system([16] * 130 + [1], r_c=np.inf, ell=1.5, seed=1)
    v = np.linalg.qr(np.random.default_rng(2).standard_normal((s.n, 5)))[0]
    h = 0.5 * np.eye(s.n) - v @ v.T
    first = np.concatenate([[0], np.cumsum(s.block_size)])
    vals = np.empty_like(s.values)
    off = O.block_value_offsets(s.block_size, s.col_ptr, s.row_idx)
    for j in range(131):
        for k in range(s.col_ptr[j], s.col_ptr[j + 1]):
            r = s.row_idx[k]
            vals[off[k]:off[k + 1]] = h[first[r]:first[r + 1], first[j]:first[j + 1]].T.ravel()
    with SubmatrixDensity.from_system(s) as c:
        c.set_values(vals)
        c.set_column_range(0, columns)
        c.build_density()
        got = O.to_dense(s.block_size, s.col_ptr, s.row_idx, c.get_density())[:, : first[columns]]
    # a product's error is below 3.4e-17 sqrt(2081 / 158) per entry; 30 of them with factors of up to 2.5
    assert float(np.max(np.abs(got - (v @ v.T)[:, : first[columns]]))) <= 30 * 2.5 * 3.4e-17 * np.sqrt(2081 / 158) + 2e-14


@pytest.mark.parametrize("first", ["density", "fermi", "inv_sqrt"])
@pytest.mark.parametrize("m", [9, 200])
def test_fermi_at_infinite_temperature_after_another_build(m, first):
    # F = I/2 whatever the work memory held before: an iterate of another function, or T at another temperature
    from paper_2205_14741_gb300 import SubmatrixDensity

    s = make_mixed_block_system([3] * m, r_c=6.0, ell=1.5, seed=8)
    lam = np.linalg.eigvalsh(O.to_dense(s.block_size, s.col_ptr, s.row_idx, s.values))
    with SubmatrixDensity.from_system(s) as c:
        c.set_function(first)
        c.set_fermi_beta(12.0)
        c.set_mu(float(lam[0]) - 0.5 if first == "inv_sqrt" else 0.02)
        c.build_density()
        c.get_trace()
        c.set_function("fermi")
        c.set_fermi_beta(0.0)
        c.build_density()
        got = O.to_dense(s.block_size, s.col_ptr, s.row_idx, c.get_density())
    assert np.array_equal(got, 0.5 * np.eye(s.n))


def _full(h, block=None):
    """The matrix h on a complete pattern of blocks of at most 64 rows."""
    n = h.shape[0]
    block = block or min(n, 50)
    s = make_mixed_block_system([block] * (n // block) + ([n % block] if n % block else []), r_c=np.inf, ell=1.5, seed=1)
    first = np.concatenate([[0], np.cumsum(s.block_size)])
    off = O.block_value_offsets(s.block_size, s.col_ptr, s.row_idx)
    vals = np.empty_like(s.values)
    for j in range(s.n_blocks):
        for k in range(s.col_ptr[j], s.col_ptr[j + 1]):
            r = s.row_idx[k]
            vals[off[k]:off[k + 1]] = h[first[r]:first[r + 1], first[j]:first[j + 1]].T.ravel()
    s.values[:] = vals
    return s


@pytest.mark.parametrize("coupling", [0.0, 0.005, 0.05, "rotated"])
@pytest.mark.parametrize("n", [2, 6, 48, 200])
@pytest.mark.parametrize("f", ["inv_sqrt", "sqrt", "inv", "overlap"])
def test_one_negative_eigenvalue_is_not_positive_definite(f, n, coupling):
    # a negative eigenvalue of any size, on one row, weakly coupled or spread over all: no root, so no result
    from paper_2205_14741_gb300 import SmxError, SubmatrixDensity, _lib

    rng = np.random.default_rng(n)
    accepted = []
    for x in list(np.linspace(0.1, 1.0, 10)) + [0.137, 0.333, 0.777, 0.9999, 1e-3]:
        if coupling == "rotated":
            v = rng.standard_normal(n)
            h = np.eye(n) - (1.0 + x) * np.outer(v, v) / (v @ v)
        else:
            h = np.eye(n) + coupling * np.triu(rng.standard_normal((n, n)), 1) / np.sqrt(n)
            h = np.triu(h) + np.triu(h, 1).T
            p = int(rng.integers(n))
            h[p, p] = -x
        s = _full(h)
        with SubmatrixDensity.from_system(s) as c:
            if f == "overlap":
                c.set_values(_full(np.diag(np.where(np.arange(n) % 2, 0.5, -0.5))).values)
                c.set_overlap(s.values)
            else:
                c.set_function(f)
            try:
                c.build_density()
                c.get_trace()
                accepted.append(float(x))
            except SmxError as e:
                assert e.status in (_lib.ERR_NOCONV, _lib.ERR_NONFINITE)
    assert accepted == []


@pytest.mark.parametrize("entry", [-0.8, -1e-3])  # rows of one size, and a small one (FP64 multiply-adds)
def test_a_failed_submatrix_leaves_no_numbers(entry):
    # D of a submatrix that failed is NaN, not what the work memory held; the others' columns stand
    from paper_2205_14741_gb300 import SmxError, SubmatrixDensity, _lib, dense_density_noalloc

    s = make_mixed_block_system([4] * 90, r_c=5.0, ell=1.5, seed=3)
    off = O.block_value_offsets(s.block_size, s.col_ptr, s.row_idx)
    diag = [int(k) for j in range(90) for k in range(s.col_ptr[j], s.col_ptr[j + 1]) if s.row_idx[k] == j]
    vals = s.values * 0.05
    for k in diag:
        vals[off[k]:off[k + 1]] = np.eye(4).ravel()
    bad = vals.copy()
    k = diag[7]
    bad[off[k]:off[k] + 4] *= 0.0
    bad[off[k]] = entry  # the submatrices that hold block 7 are not positive definite
    hit = {j for j in range(90) if 7 in s.row_idx[s.col_ptr[j]:s.col_ptr[j + 1]]}
    assert 0 < len(hit) < 90
    out = torch.empty(vals.size, dtype=torch.float64, device="cuda")
    with SubmatrixDensity.from_system(s) as c:
        c.set_function("inv_sqrt")
        c.set_values(vals)
        c.build_density()
        good = c.get_density()
        c.set_values(bad)
        with pytest.raises(SmxError) as e:
            c.build_density()
            c.get_trace()
        assert e.value.status == _lib.ERR_NONFINITE
        got = c.get_density(out).cpu().numpy()  # (a device copy reports no status)
    for j in range(90):
        part = slice(int(off[s.col_ptr[j]]), int(off[s.col_ptr[j + 1]]))
        assert np.all(np.isnan(got[part])) if j in hit else np.array_equal(got[part], good[part])

    h = torch.eye(40, dtype=torch.float64, device="cuda")
    d = torch.zeros_like(h)
    dense_density_noalloc(h, 40, 0.0, d)
    h[3, 5] = h[5, 3] = float("inf")
    with pytest.raises(SmxError) as e:
        dense_density_noalloc(h, 40, 0.0, d)
    assert e.value.status == _lib.ERR_NONFINITE
    assert bool(torch.isnan(d).all())


def test_a_nonfinite_snapshot_leaves_no_numbers():
    from paper_2205_14741_gb300 import SmxError, SubmatrixDensity, _lib

    s = make_mixed_block_system([4] * 90, r_c=5.0, ell=1.5, seed=3)
    off = O.block_value_offsets(s.block_size, s.col_ptr, s.row_idx)
    with SubmatrixDensity.from_system(s) as c:
        c.set_electron_count(180.0, max_steps=3, tol=1e-9)
        c.solve_mu()
        bad = s.values.copy()
        k = next(k for k in range(s.col_ptr[11], s.col_ptr[12]) if s.row_idx[k] == 11)
        bad[off[k]] = np.nan
        c.set_values(torch.from_numpy(bad).cuda(), on_device=True)
        with pytest.raises(SmxError) as e:
            c.solve_mu()
        assert e.value.status == _lib.ERR_NONFINITE
        got = c.get_density(torch.empty(bad.size, dtype=torch.float64, device="cuda")).cpu().numpy()
    for j in range(90):
        if 11 in s.row_idx[s.col_ptr[j]:s.col_ptr[j + 1]]:
            assert np.all(np.isnan(got[off[s.col_ptr[j]]:off[s.col_ptr[j + 1]]])), j
