"""The measured work of this framework: what its users have it do, through its public entry points.

A case is one call sequence of a user's program: new matrix values on a known block pattern, a
build or a chemical-potential solve, and the density matrix read back (or the dense entry point,
or one round of training the learned bound).  The inputs follow the repository's synthetic
water-like systems: molecules on a jittered cubic lattice (or in a film with vacuum on both
sides), one block per molecule, two bands of on-site energies around a gap at mu = 0, and
off-diagonal blocks that decay with the distance.  They are written here with numpy alone, so that
the measured inputs do not depend on other files.
"""

from __future__ import annotations

import math
from concurrent.futures import ThreadPoolExecutor

import numpy as np
import torch

import paper_2205_14741_gb300 as smx

SPACING = 3.1  # Angstrom between molecules on the lattice

# Every field a case may leave out: uniform 6 x 6 blocks on the lattice, no filter, fixed mu.
DEFAULTS = dict(kind="build", n_mol=32, block_min=6, block_max=6, cutoff=6.0, decay=1.5, eps=0.0, precision="fp64",
                function="density", mu=0.0, beta=0.0, film=False, host=False, learned=False, symmetrize=False, n=0,
                steps=0)


def listed():
    return [
        # A single small system (32 molecules, N = 192) at fixed mu in plain FP64: the reference
        # run a user checks everything else against, bound by latency.
        dict(name="water32_fp64", n_mol=32, cutoff=5.0),
        # The 1024-molecule system (N = 6144) in plain FP64, mu by bisection: production accuracy.
        dict(name="water1024_fp64_solve", kind="solve", n_mol=1024, eps=1e-5),
        # The same system in split FP16, values and density resident on the device: the headline.
        dict(name="water1024_fp16x3_solve", kind="solve", n_mol=1024, eps=1e-5, precision="fp16x3"),
        # A molecular-dynamics step: the next snapshot from host memory, mu solved with the learned
        # bound, the density back to the host, as a simulation code calls the library.
        dict(name="md1024_learned_host", kind="solve", n_mol=1024, eps=1e-5, precision="fp16x3", host=True, learned=True),
        # Larger basis (23 x 23 blocks, submatrices of about 1100): the size class of the
        # 4096-molecule system, on as many molecules as one shard of it holds.
        dict(name="water343x23_fp16x3", n_mol=343, block_min=23, block_max=23, cutoff=7.0, decay=2.0, eps=1e-6,
             precision="fp16x3"),
        # A film fading into vapour on both sides, wide cutoff: ragged submatrices, small and large.
        dict(name="film400_fp16x3", n_mol=400, cutoff=12.0, decay=2.0, eps=1e-5, precision="fp16x3", film=True),
        # Molecules of different sizes (blocks 1 .. 13) in single-pass FP16, symmetrised result:
        # the quick low-precision estimate.
        dict(name="mixed256_fp16", n_mol=256, block_min=1, block_max=13, eps=1e-5, precision="fp16", symmetrize=True),
        # S^-1/2 of the 1024-molecule overlap matrix: the orthogonalisation before a run.
        dict(name="overlap1024_inv_sqrt", n_mol=1024, function="inv_sqrt"),
        # The non-orthogonal form (H and S given), mu by bisection.
        dict(name="nonorth256_solve", kind="nonorth", n_mol=256, eps=1e-5),
        # The finite-temperature density matrix.
        dict(name="fermi128", n_mol=128, function="fermi", beta=50.0),
        # One dense matrix through the allocation-free entry point, as a plug-in calls it.
        dict(name="dense192_noalloc", kind="noalloc", n=192),
        # Training the learned bound on the current snapshot: features and Lanczos labels of every
        # submatrix, then forward, backward and Adam steps.
        dict(name="bound_training1024", kind="train", n_mol=1024, eps=1e-5, precision="fp16x3", steps=50),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["fp64", "fp64", "fp16x3", "fp16x3", "streamed", "film", "single", "function", "function",
                       "nonorth", "fermi", "noalloc", "train"])
    if kind == "noalloc":
        return dict(kind="noalloc", n=_log_int(rng, 4, 256))
    if kind == "streamed":
        return dict(n_mol=rng.randint(100, 343), block_min=23, block_max=23, cutoff=rng.uniform(6.0, 7.0), decay=2.0,
                    eps=1e-6, precision="fp16x3")
    if kind == "film":
        return dict(n_mol=rng.randint(60, 400), cutoff=rng.uniform(7.0, 12.0), decay=2.0, eps=1e-5, precision="fp16x3",
                    film=True)
    small, large = sorted((rng.randint(1, 13), rng.randint(5, 13)))
    mixed = rng.random() < 0.5
    blocks = dict(block_min=small, block_max=large) if mixed else {}
    cutoff = rng.uniform(4.5, 6.0)
    n_mol = _log_int(rng, 8, 512 if mixed else 1024)
    if kind == "single":
        return dict(n_mol=n_mol, cutoff=cutoff, eps=1e-5, precision=rng.choice(["fp16", "bf16"]),
                    symmetrize=rng.random() < 0.5, **blocks)
    if kind == "function":
        return dict(n_mol=n_mol, cutoff=cutoff, function=rng.choice(["inv_sqrt", "sqrt", "inv"]), **blocks)
    if kind == "nonorth":
        return dict(kind="nonorth", n_mol=_log_int(rng, 8, 256), cutoff=cutoff, eps=1e-5)
    if kind == "fermi":
        return dict(n_mol=_log_int(rng, 8, 128), cutoff=cutoff, function="fermi", beta=math.exp(rng.uniform(0.0, 5.0)))
    if kind == "train":
        return dict(kind="train", n_mol=n_mol, cutoff=cutoff, eps=1e-5, precision="fp16x3", steps=rng.randint(1, 50))
    # uniform blocks for the bisection (its electron count fits the two bands)
    call = dict(kind="solve", eps=1e-5) if not mixed else dict(kind="build", mu=rng.uniform(-0.05, 0.05))
    return dict(n_mol=n_mol, cutoff=cutoff, precision=kind, host=rng.random() < 0.3, **blocks, **call)


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------


def _positions(c, rng):
    n = c["n_mol"]
    if c["film"]:  # 31 x 31 Angstrom in the plane, bulk density inside, edges fading into vapour
        side = 31.0
        thick = n * SPACING ** 3 / side ** 2
        box = np.array([side, side, thick + 140.0])
        per = 10
        layers = int(math.ceil(thick / SPACING)) + 24
        grid = np.stack(np.meshgrid(np.arange(per), np.arange(per), np.arange(layers), indexing="ij"), -1).reshape(-1, 3)
        pos = (grid + 0.5) * SPACING
        pos[:, 2] += 0.5 * (box[2] - layers * SPACING)
        depth = np.abs(pos[:, 2] - 0.5 * box[2]) - 0.5 * thick
        score = depth / 8.0 + rng.logistic(size=pos.shape[0])
        pos = pos[np.argsort(score, kind="stable")[:n]]
    else:
        length = SPACING * n ** (1.0 / 3.0)
        per = int(math.ceil(n ** (1.0 / 3.0) - 1e-9))
        box = np.full(3, length)
        grid = np.stack(np.meshgrid(*(np.arange(per),) * 3, indexing="ij"), -1).reshape(-1, 3)
        pos = (grid[rng.permutation(per ** 3)[:n]] + 0.5) * (length / per)
    return pos + rng.uniform(-0.3, 0.3, size=pos.shape), box


def _distances(pos, box):
    d = pos[:, None, :] - pos[None, :, :]
    d -= box * np.round(d / box)
    return np.sqrt(np.einsum("ijk,ijk->ij", d, d))


def _bands(b, rng, count):
    """count symmetric b x b blocks with half their eigenvalues around -0.5 and the rest around +0.5."""
    q = np.linalg.qr(rng.standard_normal((count, b, b)))[0]
    e = rng.normal(0.5, 0.05, (count, b))
    e[:, : b // 2] -= 1.0
    m = (q * e[:, None, :]) @ q.transpose(0, 2, 1)
    return 0.5 * (m + m.transpose(0, 2, 1))


def _near_identity(b, rng, count):
    g = rng.standard_normal((count, b, b))
    return np.eye(b) + 0.025 * (g + g.transpose(0, 2, 1))


class _System:
    """The block pattern of a case's geometry, and matrices with random blocks on it."""

    def __init__(self, c, rng):
        # the geometry, and with it the pattern and the sizes of a case, is the same for every seed:
        # a user's program sets it up once, and new values arrive on it
        geometry = np.random.default_rng(1001)
        self.c, self.rng = c, rng
        self.pos, self.box = _positions(c, geometry)
        n = c["n_mol"]
        self.bs = (geometry.integers(c["block_min"], c["block_max"] + 1, n) if c["block_max"] > c["block_min"]
                   else np.full(n, c["block_max"])).astype(np.int32)
        near = _distances(self.pos, self.box) < c["cutoff"]
        np.fill_diagonal(near, True)
        cols, rows = np.nonzero(near)  # sorted by column, then row; the pattern is symmetric
        self.rows, self.cols = rows, cols
        self.col_ptr = np.concatenate([[0], np.cumsum(np.bincount(cols, minlength=n))]).astype(np.int64)
        size = self.bs[rows].astype(np.int64) * self.bs[cols]
        self.off = np.concatenate([[0], np.cumsum(size)])
        self.first = np.concatenate([[0], np.cumsum(self.bs)])

    def normals(self):
        b = int(self.bs.max())
        return self.rng.standard_normal((int(np.count_nonzero(self.rows < self.cols)), b, b))

    def values(self, diagonal, normals, sigma, pos=None):
        """Blocks in pattern order, each column-major: diagonal(b, rng, count) on the diagonal, and
        normals * sigma * exp(-distance / decay) off it."""
        pos = self.pos if pos is None else pos
        d = pos[self.rows] - pos[self.cols]
        d -= self.box * np.round(d / self.box)
        amp = sigma * np.exp(-np.sqrt((d * d).sum(1)) / self.c["decay"])
        n = self.bs.size
        upper = np.nonzero(self.rows < self.cols)[0]
        slot = np.zeros((n, n), dtype=np.int64)
        slot[self.rows, self.cols] = np.arange(self.rows.size)
        lower = slot[self.cols[upper], self.rows[upper]]
        diag = slot[np.arange(n), np.arange(n)]
        out = np.empty(int(self.off[-1]))
        if self.bs.min() == self.bs.max():  # uniform blocks: one array of blocks
            b = int(self.bs[0])
            blocks = out.reshape(-1, b, b)  # [block, column, row]
            m = normals * amp[upper, None, None]
            blocks[upper] = m.transpose(0, 2, 1)
            blocks[lower] = m
            blocks[diag] = diagonal(b, self.rng, n)  # symmetric
            return out
        for i in range(n):
            out[self.off[diag[i]]:self.off[diag[i] + 1]] = diagonal(int(self.bs[i]), self.rng, 1)[0].ravel()
        for k, (u, lo) in enumerate(zip(upper, lower)):
            m = normals[k, : self.bs[self.rows[u]], : self.bs[self.cols[u]]] * amp[u]
            out[self.off[u]:self.off[u + 1]] = m.T.ravel()
            out[self.off[lo]:self.off[lo + 1]] = m.ravel()
        return out


def _inputs(case, seed):
    """(full case, system, H values, S values or None, H values of the snapshot before or None)"""
    c = dict(DEFAULTS, **case)
    rng = np.random.default_rng(seed)
    s = _System(c, rng)
    if c["function"] in ("inv_sqrt", "sqrt", "inv"):
        return c, s, s.values(_near_identity, s.normals(), 0.05), None, None
    normals = s.normals()
    state = rng.bit_generator.state
    h = s.values(_bands, normals, 0.1)
    overlap = s.values(_near_identity, s.normals(), 0.05) if c["kind"] == "nonorth" else None
    before = None
    if c["learned"]:  # the same molecules one time step earlier
        moved = s.pos + rng.normal(0.0, 0.05, s.pos.shape)
        rng.bit_generator.state = state
        before = s.values(_bands, normals, 0.1, moved)
    return c, s, h, overlap, before


def _dense_input(case, seed):
    c = dict(DEFAULTS, **case)
    return c, _bands(c["n"], np.random.default_rng(seed), 1)[0]


def prepare(case, seed):
    if case.get("kind") == "noalloc":
        c, h = _dense_input(case, seed)
        h = torch.from_numpy(h).cuda()
        return dict(c=c, h=h, out=torch.empty_like(h), stream=torch.cuda.current_stream().cuda_stream)
    c, s, h, overlap, before = _inputs(case, seed)
    ctx = smx.SubmatrixDensity(s.bs, s.col_ptr, s.rows.astype(np.int32), h if before is None else before,
                               torch.cuda.current_stream().cuda_stream)
    ctx.set_filter_threshold(c["eps"])
    ctx.set_precision(c["precision"])
    ctx.set_mu(c["mu"])
    if c["function"] != "density":
        ctx.set_function(c["function"])
        ctx.set_fermi_beta(c["beta"])
    if c["symmetrize"]:
        ctx.set_symmetrize(True)
    if c["kind"] in ("solve", "nonorth"):
        ctx.set_electron_count(_electrons(s), max_steps=40, tol=1e-2)
    if c["learned"]:  # trained on the snapshot before, as a running simulation has it
        ctx.bound_model_init(7)
        ctx.bound_model_collect(48)
        ctx.bound_model_train(epochs=100, batch=256, lr=2e-3)
        ctx.set_bound_model("gap")
    if c["kind"] == "train":
        ctx.bound_model_init(7)
        return dict(c=c, ctx=ctx, params=ctx.bound_model_get_params(), values=torch.from_numpy(h).cuda())
    if c["host"]:
        values = torch.from_numpy(h).pin_memory().numpy()
        return dict(c=c, ctx=ctx, values=values, out=torch.empty(h.size, dtype=torch.float64).pin_memory().numpy())
    return dict(c=c, ctx=ctx, values=torch.from_numpy(h).cuda(), out=torch.empty(h.size, dtype=torch.float64, device="cuda"),
                overlap=None if overlap is None else torch.from_numpy(overlap).cuda())


def _electrons(s):
    return float(sum(int(b) // 2 for b in s.bs))


def run(state):
    c = state["c"]
    if c["kind"] == "noalloc":
        smx.dense_density_noalloc(state["h"], c["n"], c["mu"], state["out"], state["stream"])
        return [state["out"]]
    ctx = state["ctx"]
    ctx.set_values(state["values"], on_device=not c["host"])
    if c["kind"] == "train":
        ctx.bound_model_set_params(state["params"])
        x, _, t = ctx.bound_model_predict(predict=False, labels=True, lanczos_steps=48)
        loss, grad = ctx.bound_model_fit(x, t, steps=c["steps"], lr=2e-3)
        return [x, t, loss, grad, ctx.bound_model_get_params()]
    if c["kind"] == "nonorth":
        ctx.set_overlap(state["overlap"], on_device=True)
    if c["kind"] == "build":
        ctx.build_density()
    else:
        ctx.solve_mu()
    trace, energy, mu = ctx.get_trace()
    return [ctx.get_density(state["out"]), trace, energy, mu]


# ---------------------------------------------------------------------------
# what one pass cannot do without
# ---------------------------------------------------------------------------

# Products of n x n matrices per submatrix.  The sign iteration takes two products a step and
# the coupled iteration of the roots three; five steps stand for a well-conditioned submatrix.
# The Fermi function takes the order of a hundred products at beta = 50.
_PRODUCTS = {"density": 10, "inv_sqrt": 15, "sqrt": 15, "inv": 15, "fermi": 100}


def work(case):
    c = dict(DEFAULTS, **case)
    if c["kind"] == "noalloc":
        return {"bytes": 16.0 * c["n"] ** 2, "flops": 2.0 * _PRODUCTS["density"] * c["n"] ** 3}
    s = _System(c, np.random.default_rng(0))
    dims = np.add.reduceat(s.bs[s.rows], s.col_ptr[:-1]).astype(np.float64)
    arrays = 2.0 + (c["kind"] == "nonorth")
    nbytes = 8.0 * float(s.off[-1]) * arrays
    if c["kind"] == "train":
        # 48 Lanczos steps on A and on A^2 per submatrix, three passes of the network per step
        flops = float((2.0 * dims ** 2).sum()) * 48 * 3 + (c["steps"] + 1) * 3 * 2.0 * 4930 * c["n_mol"]
        return {"bytes": 0.5 * nbytes, "flops": flops}
    products = _PRODUCTS[c["function"]] + (17 if c["kind"] == "nonorth" else 0)
    return {"bytes": nbytes, "flops": 2.0 * products * float((dims ** 3).sum())}


# ---------------------------------------------------------------------------
# the same results in plain 64-bit numpy and torch
# ---------------------------------------------------------------------------


def _newton_sign(a):
    """sign of each symmetric matrix of a batch by the scaled Newton iteration with inverses."""
    x = a / torch.linalg.matrix_norm(a)[:, None, None]
    for it in range(30):
        y = torch.linalg.inv(x)
        g = (torch.linalg.matrix_norm(y) / torch.linalg.matrix_norm(x)).sqrt()[:, None, None]
        if it > 12 or bool(((g - 1.0).abs() < 1e-2).all()):
            g = torch.ones_like(g)
        new = 0.5 * (g * x + y / g)
        step = float((new - x).abs().max())
        x = new
        if step < 1e-14:
            break
    return 0.5 * (x + x.transpose(1, 2))


def _spectral(a, f):
    lam, v = np.linalg.eigh(a)
    return (v * f(lam)) @ v.T


def exact(case, seed):
    if case.get("kind") == "noalloc":
        c, h = _dense_input(case, seed)
        return [torch.from_numpy(_spectral(h, lambda lam: 0.5 * (1.0 - np.sign(lam - c["mu"]))))]
    if case.get("kind") == "train":
        return None  # Lanczos labels and the network trained on them are single-precision estimates
    c, s, h, overlap, _ = _inputs(case, seed)
    n_mol = s.bs.size
    sq = np.add.reduceat(h * h, s.off[:-1])
    kept = (np.sqrt(sq) >= c["eps"]) | (s.rows == s.cols)
    index = [np.arange(s.first[i], s.first[i + 1]) for i in range(n_mol)]
    lists = [s.rows[s.col_ptr[j]:s.col_ptr[j + 1]][kept[s.col_ptr[j]:s.col_ptr[j + 1]]] for j in range(n_mol)]
    sets = [np.concatenate([index[r] for r in rows]) for rows in lists]
    owns = [slice(int(s.bs[rows[rows < j]].sum()), int(s.bs[rows[rows <= j]].sum())) for j, rows in enumerate(lists)]

    def dense(values):
        m = np.zeros((int(s.first[-1]),) * 2)
        for k in np.nonzero(kept)[0]:
            r, j = s.rows[k], s.cols[k]
            m[s.first[r]:s.first[r + 1], s.first[j]:s.first[j + 1]] = values[s.off[k]:s.off[k + 1]].reshape(s.bs[j], s.bs[r]).T
        return m

    full, full_s = dense(h), dense(overlap) if overlap is not None else None
    largest = max(idx.size for idx in sets)
    eye = np.eye(largest)

    def columns(mu):
        """the kept columns of every submatrix's function"""
        if largest > 400:  # large submatrices: batches of the scaled Newton iteration on the device
            out = []
            for j0 in range(0, n_mol, 48):
                part = range(j0, min(n_mol, j0 + 48))
                n = max(sets[j].size for j in part)
                a = np.tile(np.eye(n), (len(part), 1, 1))  # padded by the identity, whose sign is itself
                for i, j in enumerate(part):
                    m = sets[j].size
                    a[i, :m, :m] = full[np.ix_(sets[j], sets[j])] - mu * eye[:m, :m]
                x = _newton_sign(torch.from_numpy(a).to("cuda" if torch.cuda.is_available() else "cpu"))
                for i, j in enumerate(part):
                    m = sets[j].size
                    out.append(0.5 * (eye[:m, owns[j]] - x[i, :m, owns[j]].cpu().numpy()))
            return out

        def one(j):
            a = full[np.ix_(sets[j], sets[j])]
            m = a.shape[0]
            f = c["function"]
            if c["kind"] == "nonorth":
                root = _root(j)
                x = _spectral(root @ a @ root, lambda lam: 0.5 * (1.0 - np.sign(lam - mu)))
                return (root @ x @ root)[:, owns[j]]
            a = a - mu * eye[:m, :m]
            if f == "density":
                return _spectral(a, lambda lam: 0.5 * (1.0 - np.sign(lam)))[:, owns[j]]
            if f == "fermi":
                return _spectral(a, lambda lam: 0.5 * (1.0 - np.tanh(0.5 * c["beta"] * lam)))[:, owns[j]]
            power = {"inv_sqrt": -0.5, "sqrt": 0.5, "inv": -1.0}[f]
            return _spectral(a, lambda lam: lam ** power)[:, owns[j]]

        with ThreadPoolExecutor(8) as pool:
            return list(pool.map(one, range(n_mol)))

    def _root(j):
        return _spectral(full_s[np.ix_(sets[j], sets[j])], lambda lam: 1.0 / np.sqrt(lam))

    def totals(cols):
        trace = energy = 0.0
        for j, d in enumerate(cols):
            hj = full[np.ix_(sets[j], index[j])]
            energy += float((d * hj).sum())
            trace += float((d * full_s[np.ix_(sets[j], index[j])]).sum()) if full_s is not None else \
                float(np.trace(d[owns[j]]))
        return trace, energy

    mu = c["mu"]
    if c["kind"] in ("solve", "nonorth"):
        if full_s is None:
            radius = np.abs(full).sum(0) - np.abs(np.diag(full))
            lo, hi = float((np.diag(full) - radius).min()), float((np.diag(full) + radius).max())
        else:
            lo, hi = math.inf, -math.inf
            for j in range(n_mol):
                root = _root(j)
                m = root @ full[np.ix_(sets[j], sets[j])] @ root
                radius = np.abs(m).sum(0) - np.abs(np.diag(m))
                lo, hi = min(lo, float((np.diag(m) - radius).min())), max(hi, float((np.diag(m) + radius).max()))
        for _ in range(40):
            mu = 0.5 * (lo + hi)
            cols = columns(mu)
            trace, energy = totals(cols)
            if abs(trace - _electrons(s)) <= 1e-2:
                break
            lo, hi = (mu, hi) if trace < _electrons(s) else (lo, mu)
    else:
        cols = columns(mu)
        trace, energy = totals(cols)
    out = np.zeros(int(s.off[-1]))
    for j, d in enumerate(cols):
        start = 0
        for k in np.nonzero(kept[s.col_ptr[j]:s.col_ptr[j + 1]])[0] + s.col_ptr[j]:
            b = int(s.bs[s.rows[k]])
            out[s.off[k]:s.off[k + 1]] = d[start:start + b].T.ravel()
            start += b
    if c["symmetrize"]:
        where = {(int(r), int(j)): k for k, (r, j) in enumerate(zip(s.rows, s.cols))}
        old = out.copy()
        for k in np.nonzero(kept)[0]:
            r, j = int(s.rows[k]), int(s.cols[k])
            t = where[(j, r)]
            mine = old[s.off[k]:s.off[k + 1]].reshape(s.bs[j], s.bs[r])
            theirs = old[s.off[t]:s.off[t + 1]].reshape(s.bs[r], s.bs[j])
            out[s.off[k]:s.off[k + 1]] = (0.5 * (mine + theirs.T)).ravel()
    return [torch.from_numpy(out), trace, energy, mu]
