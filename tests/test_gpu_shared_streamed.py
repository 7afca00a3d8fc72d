"""Clusters that share a submatrix in the streamed form of the sign kernel.

A launch whose submatrices all find room as clusters (a column range of 20 here) takes the shared form, the
whole matrix at these sizes one CTA per submatrix.  The tiles of a product and their accumulation are the
same, only who forms them differs, and the residual's parts are added in another order; so with equal
step counts the owner columns agree bit for bit.
"""

import numpy as np
import pytest

import oracle as O
from synth import make_mixed_block_system

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp16x3", "fp16", "bf16"])
@pytest.mark.parametrize("n", [193, 224, 256, 257, 321, 415])
def test_shared_form_changes_no_bit(n, precision):
    # one row tile and a bit more; widths at and past the 256-column tile; more and fewer tiles than CTAs
    from paper_2205_14741_gb300 import SubmatrixDensity

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    s = make_mixed_block_system([1] * n, r_c=np.inf, ell=1.5, seed=6)
    with SubmatrixDensity.from_system(s) as c:
        c.set_precision(precision)
        c.set_mu(0.02)
        c.build_density()
        full, steps = c.get_density().reshape(n, n), c.get_stats()["iters_max"]
        for j0 in (0, n - 20):
            c.set_column_range(j0, j0 + 20)
            c.build_density()
            assert c.get_stats()["iters_max"] == steps
            assert np.array_equal(c.get_density().reshape(n, n)[j0:j0 + 20], full[j0:j0 + 20])


@pytest.mark.parametrize("model", [False, True])
def test_shared_form_by_size(model):
    # 60 submatrices of n = 780: shared for their size; with and without the learned bound
    from paper_2205_14741_gb300 import SubmatrixDensity

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    s = make_mixed_block_system([13] * 60, r_c=np.inf, ell=1.5, seed=7)
    h = O.to_dense(s.block_size, s.col_ptr, s.row_idx, s.values)
    lam, v = np.linalg.eigh(h)
    k = int(np.argmax(np.diff(lam)))  # mu in the middle of the widest gap
    mu = 0.5 * float(lam[k] + lam[k + 1])
    ref = (v[:, :k + 1]) @ v[:, :k + 1].T
    with SubmatrixDensity.from_system(s) as c:
        c.set_precision("fp16x3")
        c.set_mu(mu)
        if model:
            c.bound_model_init(3)
            c.set_bound_model(True)
        c.build_density()
        got = O.to_dense(s.block_size, s.col_ptr, s.row_idx, c.get_density())
        assert c.get_stats()["iters_max"] < 100
    # split FP16 holds 22 bits of X's entries (at most 1); the errors of the last steps' two products of up to
    # 780 terms, 2^-22 sqrt(780) each, are not amplified: 2e-5 is the bound stated for large submatrices
    assert float(np.max(np.abs(got - ref))) <= 2e-5
