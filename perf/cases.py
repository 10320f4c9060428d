"""What this library is asked to do in use, as cases that can be timed and checked.

Every case goes through the public entry points of ``paper_1711_09487_gb300``.  The pencils are Q1
finite-element Laplacians on boxes: the tensor-product pencil of the benchmark with one seeded
diffusion coefficient per axis, so that another seed is another problem with a simple spectrum, and
eigenvalues, eigenvectors and resolvents are known in closed form.

* ``solve``      the whole interval problem on a resident pencil (set-up kept, factors released after
                 each solve, as the serving loop does): eigenvalues and eigenvectors.
* ``factor``     new quadrature nodes on a resident pencil: ``rfdd_factor``, then one refined solve.
* ``resolvent``  many right-hand sides against factors that are kept: ``rfdd_shifted_solve``.
* ``polish``     interior polish of given pairs: ``rfdd_polish``.
* ``inertia``    eigenvalue count below a shift: ``rfdd_inertia``.
* ``gram``       the Gram matrix of a tall basis: ``rfdd_dgemm`` in double-FP32.
* ``cgemm``      a complex-FP32 update on device pointers: ``rfdd_cgemm_noalloc``.
* ``eigh``       the dense symmetric eigensolver: ``rfdd_sym_eig``.
"""
import math

import numpy as np
import torch

import paper_1711_09487_gb300 as R


# --------------------------------------------------------------------------------------
# the cases
# --------------------------------------------------------------------------------------
def _solve(name, N, splits, first, nev, nodes, rule="midpoint", precision="mixed", groups=""):
    return dict(name=name, kind="solve", N=N, splits=splits, first=first, nev=nev, nodes=nodes, rule=rule,
                precision=precision, groups=groups)


def listed():
    return [
        # the benchmark's workload: 3-D, eight subdomains of up to 8000 unknowns, 202 eigenpairs
        _solve("solve_3d_40", 40, "2x2x2", 300, 202, 8),
        # a request of the serving stream: 2-D, sixteen subdomains, 200 eigenpairs
        _solve("solve_2d_160", 160, "4x4", 100, 200, 8),
        # the small published configuration: 2-D, Gauss-Legendre nodes, 50 eigenpairs
        _solve("solve_2d_40", 40, "2x2", 51, 50, 4, rule="gauss"),
        # the plain FP64 path, the arm that the mixed one is compared with
        _solve("solve_fp64_3d_12", 12, "2x2x2", 8, 20, 6, precision="fp64"),
        # a new interval on a resident pencil: bordered and interface factors for eight nodes
        dict(name="factor_3d_24", kind="factor", N=24, splits="2x2x2", first=30, nev=50, nodes=8, nrhs=1),
        # a block of right-hand sides of the size of a Krylov block on factors that are kept
        dict(name="resolvent_2d_64", kind="resolvent", N=64, splits="2x2", first=40, nev=81, nodes=8, nrhs=32),
        # pairs whose interface part is known, completed by FP64 subdomain solves
        dict(name="polish_2d_40", kind="polish", N=40, splits="2x2", pairs=16),
        # the check that no eigenvalue was missed
        dict(name="inertia_3d_16", kind="inertia", N=16, splits="2x2x2", index=60),
        # Gram matrix of a Rayleigh-Ritz basis of the benchmark's width
        dict(name="gram_1885", kind="gram", rows=8000, cols=1885),
        # the smallest call: one small update of a device-resident block, ragged in every size
        dict(name="cgemm_250x190x100", kind="cgemm", m=250, n=190, k=100),
        # projected eigenproblems: of the benchmark's Rayleigh-Ritz step and of one subdomain's V_j
        dict(name="eigh_1885", kind="eigh", n=1885),
        dict(name="eigh_120", kind="eigh", n=120),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    return {k: v for k, v in _drawn(rng).items() if k != "name"}


def _drawn(rng):
    kind = rng.choice(["solve", "solve", "solve", "factor", "resolvent", "polish", "inertia", "gram", "cgemm", "eigh"])
    if kind == "solve":
        if rng.random() < 0.15:
            return _solve("", _log_int(rng, 8, 13), "2x2x2", rng.randint(4, 12), rng.randint(10, 24),
                          rng.randint(4, 6), precision="fp64")
        if rng.random() < 0.5:
            splits = rng.choice(["2x2", "4x2", "4x4"])
            N = _log_int(rng, 32, 160)
            groups = "2x2" if splits == "4x4" and rng.random() < 0.5 else ""
            return _solve("", N, splits, rng.randint(11, 100), rng.randint(20, min(200, N)), rng.randint(4, 8),
                          rule=rng.choice(["midpoint", "midpoint", "gauss"]), groups=groups)
        N = _log_int(rng, 12, 30)
        return _solve("", N, rng.choice(["2x2x1", "2x2x2"]), rng.randint(8, 60), rng.randint(20, 60 + 2 * N),
                      rng.randint(6, 8))
    if kind in ("factor", "resolvent"):
        two = rng.random() < 0.5
        c = dict(kind=kind, N=_log_int(rng, 30, 100) if two else _log_int(rng, 10, 24),
                 splits=rng.choice(["2x2", "4x2", "4x4"]) if two else "2x2x2", first=rng.randint(11, 60),
                 nev=rng.randint(20, 80), nodes=rng.randint(4, 8))
        c["nrhs"] = 1 if kind == "factor" else _log_int(rng, 1, 64)
        return c
    if kind == "polish":
        return dict(kind=kind, N=_log_int(rng, 20, 48), splits="2x2", pairs=rng.randint(3, 16))
    if kind == "inertia":
        return dict(kind=kind, N=_log_int(rng, 8, 16), splits="2x2x2", index=rng.randint(10, 100))
    if kind == "gram":
        return dict(kind=kind, rows=_log_int(rng, 500, 16000), cols=_log_int(rng, 32, 1885))
    if kind == "cgemm":
        return dict(kind=kind, m=_log_int(rng, 17, 1024), n=_log_int(rng, 17, 1024), k=_log_int(rng, 8, 128))
    return dict(kind=kind, n=_log_int(rng, 40, 1885))


# --------------------------------------------------------------------------------------
# Q1 box pencils: A = sum_a c_a K (axis a) x M (other axes), M = M x M (x M)
# --------------------------------------------------------------------------------------
def _ints(s):
    return tuple(int(v) for v in s.split("x"))


def _axis(N, h):
    """Eigenvalues and M-orthonormal eigenvectors (columns) of the 1-D pencil on N nodes, spacing h."""
    t = np.arange(1, N + 1) * np.pi / (N + 1)
    lam = (6.0 / h ** 2) * (1.0 - np.cos(t)) / (2.0 + np.cos(t))
    v = np.sin(np.outer(np.arange(1, N + 1), t))
    return lam, v / np.sqrt(h / 6.0 * (4.0 + 2.0 * np.cos(t)) * (N + 1) / 2.0)


def _grid_sum(lams):
    ev = np.zeros(())
    for lam in lams:
        ev = ev[..., None] + lam
    return ev


class _Csr:
    def __init__(self, rowptr, col, val):
        self.rowptr, self.col, self.val = rowptr, col, val


class _Box:
    """The pencil of one seed: coefficients, partition and spectrum."""

    def __init__(self, N, splits, seed, window=None, tries=1):
        self.N, self.dim, self.splits, self.h = N, len(splits), splits, 1.0 / (N + 1)
        rng = np.random.default_rng(seed)
        self.rng = rng
        lam, self.vec = _axis(N, self.h)
        best = -1.0
        for _ in range(tries):  # of a few seeded boxes, the one whose window is best separated
            coef = rng.uniform(0.85, 1.15, self.dim)
            ev = _grid_sum([c * lam for c in coef]).ravel()
            if window is None:
                self.coef, self.ev = coef, ev
                break
            first, nev = window
            low = np.sort(np.partition(ev, first + nev + 1)[: first + nev + 1])[max(0, first - 2):]
            gap = float(np.min(np.diff(low) / low[1:]))
            if gap > best:
                best, self.coef, self.ev = gap, coef, ev
        self.n = N ** self.dim
        blocks, sep = [], []
        for k in splits:  # planes of width one node at floor(i (N+1)/k) - 1
            b, s = np.zeros(N, dtype=np.int64), np.zeros(N, dtype=bool)
            for i in range(1, k):
                c = (i * (N + 1)) // k - 1
                s[c] = True
                b[c + 1:] += 1
            blocks.append(b)
            sep.append(s)
        lab = np.zeros((N,) * self.dim, dtype=np.int64)
        cut = np.zeros((N,) * self.dim, dtype=bool)
        for a, k in enumerate(splits):
            shape = [1] * self.dim
            shape[a] = N
            lab = lab * k + blocks[a].reshape(shape)
            cut |= sep[a].reshape(shape)
        lab[cut] = -1
        self.part, self.p = lab.ravel().astype(np.int32), math.prod(splits)

    def csr(self):
        N, h, d = self.N, self.h, self.dim
        K = {-1: -1.0 / h, 0: 2.0 / h, 1: -1.0 / h}
        M = {-1: h / 6.0, 0: 4.0 * h / 6.0, 1: h / 6.0}
        offs = np.array(np.meshgrid(*[[-1, 0, 1]] * d, indexing="ij")).reshape(d, -1).T
        a = np.array([sum(self.coef[i] * K[o[i]] * math.prod(M[o[j]] for j in range(d) if j != i) for i in range(d))
                      for o in offs])
        m = np.array([math.prod(M[x] for x in o) for o in offs])
        at = np.indices((N,) * d).reshape(d, -1)
        ok = np.ones((self.n, len(offs)), dtype=bool)
        for i in range(d):
            q = at[i][:, None] + offs[:, i][None, :]
            ok &= (q >= 0) & (q < N)
        step = offs @ np.array([N ** (d - 1 - i) for i in range(d)])
        col = (np.arange(self.n)[:, None] + step[None, :])[ok].astype(np.int32)
        rowptr = np.concatenate([[0], np.cumsum(ok.sum(1))]).astype(np.int64)
        va = np.broadcast_to(a, ok.shape)[ok]
        vm = np.broadcast_to(m, ok.shape)[ok]
        return _Csr(rowptr, col, va), _Csr(rowptr, col, vm)

    def interval(self, first, nev):
        """Ends at the midpoints of the gaps around the sorted eigenvalues first .. first+nev-1 (from 1)."""
        e = np.sort(self.ev)
        last = first + nev - 1
        alpha = 0.5 * (e[first - 2] + e[first - 1]) if first > 1 else e[0] - 1.0
        return float(alpha), float(0.5 * (e[last - 1] + e[last]))

    def modes(self, idx):
        """M-orthonormal eigenvectors of the flat spectrum indices idx, as columns."""
        at = np.unravel_index(idx, (self.N,) * self.dim)
        X = np.ones((1, len(idx)))
        for q in at:
            X = (X[:, None, :] * self.vec[:, q][None, :, :]).reshape(-1, len(idx))
        return X

    def perm(self):
        """new index -> original index of the interior-first ordering."""
        return np.argsort(np.where(self.part < 0, self.p, self.part), kind="stable")

    def resolvent(self, z, Rhs):
        """(A - z M)^{-1} Rhs on the interior-first ordering."""
        p = self.perm()
        T = np.empty_like(Rhs)
        T[p] = Rhs
        T = T.reshape((self.N,) * self.dim + (-1,))
        for a in range(self.dim):
            T = np.moveaxis(np.tensordot(self.vec.T, T, axes=(1, a)), 0, a)
        T = T / (self.ev.reshape((self.N,) * self.dim) - z)[..., None]
        for a in range(self.dim):
            T = np.moveaxis(np.tensordot(self.vec, T, axes=(1, a)), 0, a)
        return T.reshape(self.n, -1)[p]

    def sizes(self):
        """Subdomain sizes d_j, their interface couplings s_j (from the grid) and the interface size."""
        d = [int(np.count_nonzero(self.part == j)) for j in range(self.p)]
        lab = self.part.reshape((self.N,) * self.dim)
        s = []
        for j in range(self.p):
            near = lab == j
            for a in range(self.dim):
                near = near | np.roll(near, 1, a) | np.roll(near, -1, a)
            s.append(int(np.count_nonzero(near & (lab == -1))))
        return d, s, int(np.count_nonzero(self.part < 0))


def _box(case, seed):
    window = (case["first"], case["nev"]) if "first" in case else None
    return _Box(case["N"], _ints(case["splits"]), seed, window, tries=8)


def _options(case):
    return R.rfdd_default_options(
        precision=R.RFDD_FP64 if case.get("precision") == "fp64" else R.RFDD_MIXED,
        quad_rule=R.RFDD_GAUSS_LEGENDRE if case.get("rule") == "gauss" else R.RFDD_MIDPOINT)


def _groups(case):
    """Group label of every subdomain, blocks along each axis gathered into contiguous runs."""
    splits, gs = _ints(case["splits"]), _ints(case["groups"])
    lab = np.zeros(splits, dtype=np.int64)
    for a, idx in enumerate(np.indices(splits)):
        lab = lab * gs[a] + (idx * gs[a]) // splits[a]
    return lab.ravel().astype(np.int32)


class _DeviceArray:
    """A raw device pointer of a result, as torch reads it."""

    def __init__(self, address, shape):
        self.__cuda_array_interface__ = dict(shape=shape, typestr="<f8", data=(address, False), version=3)


# --------------------------------------------------------------------------------------
# prepare, run
# --------------------------------------------------------------------------------------
def _polish_pairs(case, box):
    """Pairs with a large interface part and an eigenvalue away from those of the subdomains."""
    cut = [(i * (box.N + 1)) // 2 - 1 for i in (1,)][0]
    sub = [_axis(w, box.h)[0] for w in (cut, box.N - cut - 1)]
    inner = np.concatenate([_grid_sum([c * sub[i] for c, i in zip(box.coef, q)]).ravel()
                            for q in ((0, 0), (0, 1), (1, 0), (1, 1))])
    order = np.argsort(box.ev)[: 40 + 8 * case["pairs"]]
    X = box.modes(order)
    share = np.linalg.norm(X[box.part < 0], axis=0) / np.linalg.norm(X, axis=0)
    far = np.array([np.abs(inner - box.ev[i]).min() / box.ev[i] for i in order])
    good = np.argsort(-np.minimum(far / 1e-2, 1.0) * (share > 0.1), kind="stable")[: case["pairs"]]
    return order[np.sort(good)]


def _shift_gap(case, box):
    """The sorted spectrum and the index before the widest of a few gaps at a seeded place in it."""
    e = np.sort(box.ev)
    i = case["index"] + int(box.rng.integers(0, box.n // 4))
    return e, i + int(np.argmax(np.diff(e[i: i + 6])))


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("solve", "factor", "resolvent", "polish", "inertia"):
        box = _box(case, seed)
        A, M = box.csr()
        h = R.rfdd_setup(A, M, box.part, box.p, _options(case))
        st = dict(kind=kind, h=h)
        if "first" in case:
            st["alpha"], st["beta"] = box.interval(case["first"], case["nev"])
            st["nodes"] = case["nodes"]
        if kind == "solve":
            if case["groups"]:
                R.rfdd_set_interface_groups(h, _groups(case))
            st["probe"] = torch.from_numpy(box.rng.standard_normal(box.n)).cuda()
        elif kind in ("factor", "resolvent"):
            st["z"], st["w"] = R.rfdd_quadrature(st["alpha"], st["beta"], case["nodes"])
            st["rhs"] = (box.rng.standard_normal((box.n, case["nrhs"]))
                         + 1j * box.rng.standard_normal((box.n, case["nrhs"])))
            st["node"] = case["nodes"] // 2
            if kind == "resolvent":
                R.rfdd_factor(h, st["z"], st["w"])
        elif kind == "polish":
            idx = _polish_pairs(case, box)
            X = box.modes(idx)
            inside = box.part >= 0
            X[inside] = box.rng.standard_normal((int(inside.sum()), len(idx)))
            st["lam"], st["X"] = box.ev[idx].copy(), X
        else:
            e, i = _shift_gap(case, box)
            st["sigma"] = float(e[i] + 0.55 * (e[i + 1] - e[i]))
        return st
    g = torch.Generator(device="cuda").manual_seed(int(seed))

    def randn(*shape, dtype=torch.float64):
        return torch.randn(*shape, dtype=dtype, device="cuda", generator=g)

    if kind == "gram":  # a basis and its image under a mass matrix (here diagonal)
        Y = randn(case["rows"], case["cols"])
        D = 0.5 + torch.rand(case["rows"], 1, dtype=torch.float64, device="cuda", generator=g)
        return dict(kind=kind, Y=Y.cpu().numpy(), PY=(Y * D).cpu().numpy(),
                    G=np.zeros((case["cols"], case["cols"])))
    if kind == "cgemm":
        m, n, k = case["m"], case["n"], case["k"]
        return dict(kind=kind, m=m, n=n, k=k, A=randn(m, k, dtype=torch.complex64),
                    B=randn(k, n, dtype=torch.complex64), C=randn(m, n, dtype=torch.complex64))
    n = case["n"]  # eigh: a projected pencil, orthogonal basis, spread spectrum
    q, _ = torch.linalg.qr(randn(n, n))
    lam = torch.cumsum(0.5 + torch.rand(n, dtype=torch.float64, device="cuda", generator=g), 0)
    H = (q * lam) @ q.T
    return dict(kind=kind, H=(0.5 * (H + H.T)).cpu().numpy())


def run(st):
    kind = st["kind"]
    if kind == "solve":
        r = R.rfdd_solve(st["h"], st["alpha"], st["beta"], st["nodes"])
        nev, lam, vec, _ = R.rfdd_result_get(r, device=True)
        X = torch.as_tensor(_DeviceArray(vec, (st["h"].n, nev)), device="cuda")
        # an eigenvector's sign is free: made unique by a fixed probe vector
        X = X * torch.sign(st["probe"] @ X)
        lam = torch.as_tensor(_DeviceArray(lam, (nev,)), device="cuda").clone()
        R.rfdd_release(st["h"])
        return {"evals": lam, "evecs": X}
    if kind == "factor":
        R.rfdd_factor(st["h"], st["z"], st["w"])
        return R.rfdd_shifted_solve(st["h"], st["node"], 2, 0, st["rhs"])
    if kind == "resolvent":
        return R.rfdd_shifted_solve(st["h"], st["node"], 2, 0, st["rhs"])
    if kind == "polish":
        lam, X, _ = R.rfdd_polish(st["h"], st["lam"], st["X"])
        return {"evals": lam, "evecs": X}
    if kind == "inertia":
        return R.rfdd_inertia(st["h"], st["sigma"])
    if kind == "gram":
        return R.rfdd_dgemm(st["Y"], st["PY"], st["G"], ta=True, sym=True)
    if kind == "cgemm":
        C = st["C"].clone()
        R.rfdd_cgemm_noalloc(st["m"], st["n"], st["k"], st["A"].data_ptr(), st["k"], st["B"].data_ptr(), st["n"],
                             C.data_ptr(), st["n"], -1.0, 1.0, torch.cuda.current_stream().cuda_stream)
        return C
    lam, V = R.rfdd_sym_eig(st["H"])
    return {"evals": lam, "evecs": V * np.sign(V[:, :1])}  # the sign that makes the first entry positive


# --------------------------------------------------------------------------------------
# work and exact values
# --------------------------------------------------------------------------------------
def work(case):
    kind = case["kind"]
    if kind in ("solve", "factor", "resolvent", "polish", "inertia"):
        box = _Box(case["N"], _ints(case["splits"]), 0)
        d, s, S = box.sizes()
        nnz, n = 3 ** box.dim * box.n, box.n
    if kind == "inertia":  # real bordered factorisation, then the tridiagonalisation of each block
        fl = sum(2 / 3 * ((x + y) ** 3 - y ** 3) + 4 / 3 * x ** 3 for x, y in zip(d, s)) + 4 / 3 * S ** 3
        return {"bytes": 20 * nnz + 8 * sum((x + y) ** 2 for x, y in zip(d, s)) + 8 * S * S, "flops": fl}
    if kind == "polish":  # one real LU and solve for each pair and subdomain
        return {"bytes": 20 * nnz + case["pairs"] * (8 * sum(x * x for x in d) + 16 * n),
                "flops": case["pairs"] * sum(2 / 3 * x ** 3 for x in d)}
    if kind in ("solve", "factor", "resolvent"):  # complex multiply-add = 8
        real = 16 if case.get("precision") == "fp64" else 8  # bytes of a complex factor entry
        lu = case["nodes"] * (sum(8 / 3 * ((x + y) ** 3 - y ** 3) for x, y in zip(d, s)) + 8 / 3 * S ** 3)
        entries = case["nodes"] * (sum((x + y) ** 2 for x, y in zip(d, s)) + S * S)
        per_rhs = 8 * case["nodes"] * (sum(x * x + 2 * x * y for x, y in zip(d, s)) + S * S)
    if kind == "factor":
        return {"bytes": 20 * nnz + real * entries + 32 * n, "flops": lu}
    if kind == "resolvent":  # one node's factors, and the right-hand sides
        return {"bytes": 20 * nnz + real * entries / case["nodes"] + 32 * n * case["nrhs"],
                "flops": 3 * per_rhs / case["nodes"] * case["nrhs"]}
    if kind == "solve":  # factors written and read, one refined filter application on the pairs
        return {"bytes": 20 * nnz + 2 * real * entries + 8 * n * case["nev"],
                "flops": lu + 2 * per_rhs * case["nev"]}
    if kind == "gram":
        return {"bytes": 16 * case["rows"] * case["cols"] + 8 * case["cols"] ** 2,
                "flops": case["rows"] * case["cols"] * (case["cols"] + 1)}
    if kind == "cgemm":
        m, n, k = case["m"], case["n"], case["k"]
        return {"bytes": 8 * (m * k + k * n + 2 * m * n), "flops": 8 * m * n * k}
    return {"bytes": 16 * case["n"] ** 2, "flops": (4 / 3 + 2) * case["n"] ** 3}


def exact(case, seed):
    kind = case["kind"]
    if kind in ("gram", "cgemm", "eigh"):
        st = prepare(case, seed)
        if kind == "gram":
            G = st["Y"].T @ st["PY"]
            return 0.5 * (G + G.T)
        if kind == "cgemm":
            A, B, C = (st[k].to(torch.complex128) for k in "ABC")
            return C - A @ B
        lam, V = np.linalg.eigh(st["H"])
        V = V.T
        return {"evals": lam, "evecs": V * np.sign(V[:, :1])}
    box = _box(case, seed)
    if kind == "solve":
        idx = np.argsort(box.ev)[case["first"] - 1: case["first"] - 1 + case["nev"]]
        X = box.modes(idx)
        return {"evals": box.ev[idx], "evecs": X * np.sign(box.rng.standard_normal(box.n) @ X)}
    if kind in ("factor", "resolvent"):
        a, b = box.interval(case["first"], case["nev"])
        theta = (case["nodes"] // 2 + 0.5) * np.pi / case["nodes"]  # midpoint rule on the upper half circle
        shape = (box.n, case["nrhs"])
        rhs = box.rng.standard_normal(shape) + 1j * box.rng.standard_normal(shape)
        return box.resolvent(0.5 * (a + b) + 0.5 * (b - a) * np.exp(1j * theta), rhs)
    if kind == "polish":
        idx = _polish_pairs(case, box)
        return {"evals": box.ev[idx], "evecs": box.modes(idx)}
    return _shift_gap(case, box)[1] + 1
