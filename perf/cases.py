"""The work that users of the eigensolver library have it do, as cases that can be timed.

Every case goes through the library's public entry points (the binding of the C ABI) and returns
what they compute.  Matrices are the seeded CI-shaped ones of the benchmark and the tests (rows
sorted by a shell level k of degeneracy (k+1)(k+2)/2, diagonal k + N(0, 0.05^2), couplings
N(0, 0.1^2) on a random tile pattern a quarter full), drawn here on the device.
"""
import ctypes
import math

import numpy as np
import torch

from paper_2305_15552_gb300 import binding

DEV = "cuda"
RHO = 0.25            # fill of an active tile
VALUE_BYTES = {"f64": 8, "f32": 4, "bf16": 2}
TORCH = {"f64": torch.float64, "f32": torch.float32}


# ---------------------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------------------
def listed():
    return [
        # the product of the front phase of the hybrid benchmark: 2M rows, FP32, block 16
        dict(name="spmm_f32_2m", op="spmm", n=2_000_000, per_row=400, block=256, val="f32", vec="f32", nb=16),
        # the product of the plain FP64 workload (20,000 rows): the smallest call, latency counts
        dict(name="spmm_f64_20k", op="spmm", n=20_000, per_row=100, block=64, val="f64", vec="f64", nb=8),
        # the FP64-accurate product that starts and certifies RMM-DIIS: FP32 values, FP64 vectors,
        # a row count that no tile divides
        dict(name="spmm_f32_f64_663k", op="spmm", n=663_527, per_row=300, block=256, val="f32", vec="f64", nb=8),
        # one application of the Chebyshev filter (degree 10) to a block of 16 at the paper's
        # density (197,822 rows, ~1080 nonzeros a row)
        dict(name="filter_f32_198k", op="filter", n=197_822, per_row=1080, block=256, val="f32", vec="f32", nb=16,
             degree=10),
        # a new matrix: its SpMM plan and the first product with it (every member of a family, every
        # instance of a batch pays this once)
        dict(name="plan_f32_1m", op="plan", n=1_000_000, per_row=300, block=256, val="f32", vec="f32", nb=16),
        # Gram product of two blocks as Rayleigh-Ritz forms it, at the benchmark's size
        dict(name="gram_f32_2m", op="gram", n=2_000_000, nb=16, vec="f32"),
        # orthonormalisation of a filtered block (ChebFSI, block Lanczos) at the benchmark's size
        dict(name="cholqr2_f32_2m", op="cholqr2", n=2_000_000, nb=16, vec="f32"),
        # the projected problem of a LOBPCG iteration with block 16: one small latency-bound call
        dict(name="ritz_k48", op="ritz", k=48, nb=16, pencil=True),
        # one training step of the learned preconditioner on a sample of the 1M-row family, 8 columns
        dict(name="train_1m", op="train", n=1_000_000, m=8),
        # the learned preconditioner applied to a residual block (inference)
        dict(name="apply_200k", op="apply", n=199_999, per_row=100, block=256, val="f32", vec="f32", nb=8),
        # whole calls: the FP64 LOBPCG solve of the 20,000-row workload, to pairs that serve as
        # reference vectors or 20 iterations, and the mixed-precision hybrid of the
        # 2M-row benchmark (energies: see run())
        dict(name="lobpcg_f64_20k", op="solve", method="lobpcg", n=20_000, per_row=100, block=64, val="f64",
             vec="f64", n_ev=5, nb=8, tol=1e-8, maxiter=500),
        dict(name="hybrid_f32_2m", op="solve", method="hybrid", n=2_000_000, per_row=400, block=256, val="f32",
             vec="f32", n_ev=8, nb=16, tol=1e-6, maxiter=500),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _matrix_shape(rng, lo, hi, most):
    """Rows spread over [lo, hi] and a mean row count, at most `most` nonzeros in all."""
    n = _log_int(rng, lo, hi)
    block = 64 if n < 60_000 else 256
    per_row = rng.randint(60, 140) if block == 64 else rng.randint(90, 500)
    return dict(n=n, per_row=int(min(per_row, max(80, most // n))), block=block)


def draw(rng):
    op = rng.choice(["spmm", "spmm", "spmm", "filter", "plan", "gram", "cholqr2", "ritz", "train", "apply", "solve"])
    if op == "spmm":
        val, vec = rng.choice([("f32", "f32"), ("f32", "f32"), ("f32", "f64"), ("f64", "f64"), ("bf16", "f32")])
        most = 800_000_000 if val != "f64" and vec != "f64" else 150_000_000
        return dict(op=op, val=val, vec=vec, nb=rng.choice([1, 8, 8, 16, 16]), **_matrix_shape(rng, 20_000, 2_000_000, most))
    if op == "filter":
        val, vec = rng.choice([("f32", "f32"), ("f32", "f32"), ("f64", "f64")])
        return dict(op=op, val=val, vec=vec, nb=rng.choice([8, 16]), degree=rng.randint(8, 24),
                    **_matrix_shape(rng, 20_000, 300_000, 80_000_000 if vec == "f32" else 12_000_000))
    if op == "plan":
        return dict(op=op, val=rng.choice(["f32", "f32", "f64", "bf16"]), vec="f32", nb=8,
                    **_matrix_shape(rng, 20_000, 1_000_000, 300_000_000))
    if op == "gram":
        return dict(op=op, n=_log_int(rng, 20_000, 4_000_000), nb=rng.choice([8, 16, 16]), vec=rng.choice(["f32", "f32", "f64"]))
    if op == "cholqr2":
        return dict(op=op, n=_log_int(rng, 20_000, 4_000_000), nb=rng.choice([5, 8, 10, 16, 16]),
                    vec=rng.choice(["f32", "f32", "f64"]))
    if op == "ritz":
        if rng.random() < 0.5:
            nb = rng.choice([8, 16])
            return dict(op=op, k=nb * rng.choice([2, 3]), nb=nb, pencil=True)
        return dict(op=op, k=rng.randint(40, 400), nb=rng.choice([5, 8, 10]), pencil=False)
    if op == "train":
        return dict(op=op, n=_log_int(rng, 20_000, 1_000_000), m=rng.choice([5, 8, 8, 10]))
    if op == "apply":
        return dict(op=op, val="f32", vec=rng.choice(["f32", "f32", "f64"]), nb=rng.choice([8, 16]),
                    **_matrix_shape(rng, 20_000, 400_000, 40_000_000))
    if rng.random() < 0.5:
        return dict(op="solve", method="lobpcg", val="f64", vec="f64", n_ev=5, nb=8, tol=1e-8, maxiter=500, block=64,
                    n=_log_int(rng, 10_000, 40_000), per_row=rng.randint(60, 140))
    n_ev, nb = rng.choice([(5, 8), (8, 16), (10, 16)])
    return dict(op="solve", method="hybrid", val="f32", vec="f32", n_ev=n_ev, nb=nb, tol=1e-6, maxiter=500,
                **_matrix_shape(rng, 100_000, 2_000_000, 600_000_000))


# ---------------------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------------------
class Csr:
    """Upper triangle on the device: rowptr int64, col int32, val (bf16 as int16 bit patterns)."""

    def __init__(self, n, rowptr, col, val, storage):
        self.n, self.rowptr, self.col, self.val, self.storage = n, rowptr, col, val, storage

    def arrays(self):
        return self.rowptr, self.col, self.val

    def values64(self):
        v = self.val.view(torch.bfloat16) if self.storage == "bf16" else self.val
        return v.double()

    def rows(self):
        return torch.repeat_interleave(torch.arange(self.n, device=DEV), self.rowptr[1:] - self.rowptr[:-1])


def _levels(n):
    k = torch.arange(0, 4 + int((6.0 * n) ** (1.0 / 3.0)), device=DEV, dtype=torch.int64)
    ends = (k + 1) * (k + 2) * (k + 3) // 6
    return torch.searchsorted(ends, torch.arange(n, device=DEV), right=True).double()


def _generator(seed, salt):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 1_000_003 + salt)
    return g


def _matrix(case, seed):
    n, B, st = int(case["n"]), int(case["block"]), case["val"]
    g = _generator(seed, 11)
    nblk = -(-n // B)
    mu = max(0.0, (case["per_row"] / (B * RHO) - 1.0) / 2.0)
    p = min(1.0, 2.0 * mu / (nblk - 1)) if nblk > 1 else 0.0
    active = torch.rand(nblk, nblk, device=DEV, generator=g) < p
    active = torch.triu(active, 1)
    active.fill_diagonal_(True)
    tI, tJ = active.nonzero(as_tuple=True)
    del active
    nt = tI.numel()
    first = torch.searchsorted(tI, torch.arange(nblk + 1, device=DEV))
    ar = torch.arange(B, device=DEV)
    strict = ar[None, :] > ar[:, None]
    per = max(1, (1 << 26) // (B * B))
    masks, counts = [], []
    for a in range(0, nt, per):
        b = min(nt, a + per)
        m = torch.rand(b - a, B, B, device=DEV, generator=g) < RHO
        dg = (tI[a:b] == tJ[a:b]).nonzero(as_tuple=True)[0]
        m[dg] &= strict
        m[dg] |= torch.eye(B, dtype=torch.bool, device=DEV)
        m &= ((tI[a:b, None] * B + ar) < n)[:, :, None]
        m &= ((tJ[a:b, None] * B + ar) < n)[:, None, :]
        masks.append(m)
        counts.append(m.sum(2, dtype=torch.int64))
    cnt = torch.cat(counts)                                        # tile x row
    before = torch.cat([torch.zeros(1, B, dtype=torch.int64, device=DEV), cnt.cumsum(0)])
    rowlen = (before[first[1:]] - before[first[:-1]]).reshape(-1)[:n]
    rowptr = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    rowptr[1:] = rowlen.cumsum(0)
    nnz = int(rowptr[-1])
    start = before[:-1] - before[first[:-1]][tI]                   # entries of the row in earlier tiles
    col = torch.empty(nnz, dtype=torch.int32, device=DEV)
    wide = torch.float64 if st == "f64" else torch.float32
    val = torch.empty(nnz, dtype=wide, device=DEV).normal_(0.0, 0.1, generator=g)
    pad = torch.nn.functional.pad(rowptr[:-1], (0, nblk * B - n))
    for i, m in enumerate(masks):
        a = i * per
        t, r, c = m.nonzero(as_tuple=True)
        cn = cnt[a:a + m.shape[0]].reshape(-1)
        tr = t * B + r
        rank = torch.arange(t.numel(), device=DEV) - (cn.cumsum(0) - cn)[tr]
        dest = pad[tI[a + t] * B + r] + start[a + t, r] + rank
        col[dest] = (tJ[a + t] * B + c).int()
        masks[i] = None
        del t, r, c, tr, rank, dest
    # the diagonal entry is the first of its row
    diag = _levels(n) + 0.05 * torch.randn(n, device=DEV, dtype=torch.float64, generator=g)
    val[rowptr[:-1]] = diag.to(wide)
    if st == "bf16":
        val = val.to(torch.bfloat16).view(torch.int16)
    return Csr(n, rowptr, col, val, st)


def _block(n, k, seed, salt, dtype):
    return torch.randn(n, k, device=DEV, dtype=dtype, generator=_generator(seed, salt))


def _start_block(H, k):
    """The lowest k eigenvectors of the leading 1024 rows, zero-padded (a smaller model space)."""
    m = min(1024, H.n)
    e = int(H.rowptr[m])
    r = torch.repeat_interleave(torch.arange(m, device=DEV), H.rowptr[1:m + 1] - H.rowptr[:m])
    c = H.col[:e].long()
    keep = c < m
    D = torch.zeros(m, m, dtype=torch.float64, device=DEV)
    D[r[keep], c[keep]] = Csr(H.n, None, None, H.val[:e], H.storage).values64()[keep]
    D = torch.triu(D) + torch.triu(D, 1).T
    _, Z = np.linalg.eigh(D.cpu().numpy())
    X0 = torch.zeros(H.n, k, dtype=torch.float64, device=DEV)
    X0[:m] = torch.from_numpy(np.ascontiguousarray(Z[:, :k])).to(DEV)
    return X0


class Handle:
    """A solver handle of the C ABI over a matrix that is on the device already."""

    def __init__(self, H, n_ev, block):
        self.lib, self.n, self.n_ev, self.h = binding.load(), H.n, n_ev, ctypes.c_void_p()
        csr = binding.csr_struct(*H.arrays(), H.storage, H.n, True)
        binding.check(self.lib.eig_create(ctypes.byref(csr), n_ev, block, ctypes.byref(self.h)), "eig_create")

    def solve(self, method, X0, **options):
        o, stats = binding.Opts(), binding.Stats()
        self.lib.eig_default_opts(ctypes.byref(o))
        for k, v in options.items():
            setattr(o, k, v)
        o.X0, o.x0_cols, o.x0_on_device, o.stream = X0.data_ptr(), X0.shape[1], 1, binding.stream_ptr()
        rc = self.lib.eig_solve(self.h, binding.METHODS[method], ctypes.byref(o), ctypes.byref(stats))
        if rc not in (binding.EIG_OK, binding.EIG_ENOT_CONVERGED, binding.EIG_EDUPLICATE):
            raise binding.EigError(rc, "eig_solve")

    def ritz(self, vectors):
        theta = np.zeros(self.n_ev)
        X = torch.empty(self.n, self.n_ev, dtype=torch.float64, device=DEV) if vectors else None
        binding.check(self.lib.eig_ritz(self.h, theta.ctypes.data, X.data_ptr() if vectors else None, None, 1), "eig_ritz")
        return theta, X

    def __del__(self):
        if self.h:
            self.lib.eig_destroy(self.h)
            self.h = None


def _params(seed):
    """Network parameters as after some training: He-normal hidden layers, a small output layer."""
    rng = np.random.default_rng([int(seed), 5])
    p = np.zeros(binding.N_LP_PARAMS)
    p[0:6] = [150.0, 1.5, 150.0, 170.0, 0.0, 0.0]
    p[6:12] = [60.0, 1.0, 60.0, 60.0, 1.0, 10.0]
    p[12:204] = rng.standard_normal(192) * math.sqrt(2.0 / 6)
    p[204:236] = rng.standard_normal(32) * 0.1
    p[236:1260] = rng.standard_normal(1024) * math.sqrt(2.0 / 32)
    p[1260:1292] = rng.standard_normal(32) * 0.1
    p[1292:1325] = rng.standard_normal(33) * 0.05
    return p.astype(np.float32)


def _sample(case, seed):
    """A training sample as eig_lp_sample lays it out: features, residuals, targets, column weights."""
    n, m = case["n"], case["m"]
    g = _generator(seed, 31)
    lev = _levels(n) + 0.05 * torch.randn(n, device=DEV, dtype=torch.float64, generator=g)
    theta = torch.linspace(-0.1, 2.5, m, device=DEV, dtype=torch.float64)
    F = torch.empty(n, m, 6, device=DEV)
    F[:, :, 0] = lev.float()[:, None]
    F[:, :, 1] = theta.float()
    F[:, :, 2] = (lev[:, None] - theta).float()
    F[:, :, 3] = (lev.abs() + 24.0 + torch.randn(n, device=DEV, dtype=torch.float64, generator=g)).float()[:, None]
    F[:, :, 4] = torch.randn(n, m, device=DEV, generator=g)
    F[:, :, 5] = 10.0 * torch.randn(n, m, device=DEV, generator=g)
    r = F[:, :, 4] * (1e-2 / math.sqrt(n))
    den = F[:, :, 2].abs().clamp(min=2.0) * torch.where(F[:, :, 2] < 0, -1.0, 1.0)
    z = r / den * (1.0 + 0.3 * torch.randn(n, m, device=DEV, generator=g))
    colw = 1.0 / (m * z.double().square().sum(0))
    return dict(F=F.reshape(n * m, 6), r=r.reshape(-1).contiguous(), z=z.reshape(-1).contiguous(), colw=colw, n=n, m=m)


def _pencil(case, seed):
    """(S^T H S, S^T S) of a LOBPCG basis S = [X W P] of a diagonal H, or a projected matrix alone."""
    k, nb = case["k"], case["nb"]
    rows = 4 * k + 200
    d = _levels(rows) + 0.05 * _block(rows, 1, seed, 41, torch.float64)[:, 0]
    S, _ = torch.linalg.qr(_block(rows, k, seed, 42, torch.float64))
    if not case["pencil"]:
        return S.T @ (d[:, None] * S), None
    S = S.clone()
    S[:, nb:] = 0.1 * S[:, nb:] + 0.02 * S[:, :nb].repeat(1, k // nb - 1)
    return S.T @ (d[:, None] * S), S.T @ S


def prepare(case, seed):
    op = case["op"]
    s = dict(case=case)
    if op in ("spmm", "filter", "plan", "apply", "solve"):
        H = _matrix(case, seed)
    if op in ("spmm", "filter"):
        s["plan"] = binding.SpmmPlan(H, device_arrays=H.arrays())
        s["X"] = _block(H.n, case["nb"], seed, 2, TORCH[case["vec"]])
    if op == "filter":
        # the filter damps [2.5, lambda_max]: centre and half width of that interval
        ub = float(_levels(H.n)[-1]) + 4.0
        s["c"], s["e"] = 0.5 * (ub + 2.5), 0.5 * (ub - 2.5)
        s["active"] = torch.ones(case["nb"], dtype=torch.int32, device=DEV)
    if op == "plan":
        vec = torch.float64 if case["val"] == "f64" else TORCH[case["vec"]]
        s["H"], s["X"] = H, _block(H.n, case["nb"], seed, 2, vec)
    if op == "apply":
        host = Csr(H.n, *(t.cpu().numpy() for t in H.arrays()), H.storage)
        s["solver"] = binding.Solver(host, min(5, case["nb"]), case["nb"])
        s["params"] = _params(seed)
        s["theta"] = np.linspace(-0.1, 2.5, case["nb"])
        s["R"] = _block(H.n, case["nb"], seed, 3, TORCH[case["vec"]]) * 1e-2
    if op == "solve":
        s["handle"] = Handle(H, case["n_ev"], case["nb"])
        s["X0"] = _start_block(H, case["nb"])
    if op == "gram":
        # Y = H X of a nearly converged block: a multiple of X plus a residual
        s["A"] = _block(case["n"], case["nb"], seed, 4, TORCH[case["vec"]])
        s["B"] = s["A"] * torch.linspace(0.5, 3.0, case["nb"], device=DEV, dtype=s["A"].dtype)
        s["B"] += 0.3 * _block(case["n"], case["nb"], seed, 5, TORCH[case["vec"]])
    if op == "cholqr2":
        # a filtered block: columns of different norms that lean towards the lowest vector
        X = _block(case["n"], case["nb"], seed, 6, TORCH[case["vec"]])
        X += 0.5 * X[:, :1].clone()
        s["X"] = X * torch.logspace(0.0, -2.0, case["nb"], device=DEV, dtype=X.dtype)
        s["Q"] = torch.empty_like(s["X"])
    if op == "ritz":
        s["A"], s["G"] = _pencil(case, seed)
    if op == "train":
        s["sample"] = _sample(case, seed)
        s["p"] = torch.from_numpy(_params(seed)).to(DEV)
        g = _generator(seed, 32)
        s["m1"] = 1e-2 * torch.randn(binding.N_LP_PARAMS, device=DEV, generator=g)
        s["m2"] = 1e-2 * torch.rand(binding.N_LP_PARAMS, device=DEV, generator=g)
        s["grad"] = torch.empty(binding.N_LP_TRAINED + 1, dtype=torch.float64, device=DEV)
        s["ws"] = torch.empty(binding.load().eig_lp_grad_workspace_bytes(), dtype=torch.uint8, device=DEV)
        s["t"] = 20
    return s


# ---------------------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------------------
def run(s):
    case = s["case"]
    op = case["op"]
    if op == "spmm":
        return s["plan"].spmm(s["X"])
    if op == "filter":
        P, X, c, e, act = s["plan"], s["X"], s["c"], s["e"], s["active"]
        Q, W = X, P.spmm_cheb(X, 1.0 / e, c, None, act)
        for _ in range(case["degree"] - 1):
            Q, W = W, P.spmm_cheb(W, 2.0 / e, c, Q, act)
        return W
    if op == "plan":
        P = binding.SpmmPlan(s["H"], device_arrays=s["H"].arrays())
        Y = P.spmm(s["X"])
        P.close()
        return Y
    if op == "gram":
        return binding.gram(s["A"], s["B"])
    if op == "cholqr2":
        s["Q"].copy_(s["X"])               # the entry point works in place
        Q, R = binding.cholqr2(s["Q"])
        return dict(Q=Q, R=R)
    if op == "ritz":
        if case["pencil"]:
            theta, C, info = binding.small_rr(s["A"], s["G"], case["nb"], 1e-10)
            return dict(theta=theta, C=C, info=info)
        w, Z = binding.small_syev(s["A"], case["nb"])
        return dict(w=w, Z=Z)
    if op == "train":
        s["t"] += 1
        binding.lp_grad(s["p"], s["sample"], s["grad"], s["ws"])
        binding.lp_adam(s["p"], s["grad"], s["m1"], s["m2"], s["t"], 1e-3)
        return dict(grad=s["grad"], p=s["p"], m1=s["m1"], m2=s["m2"])
    if op == "apply":
        return s["solver"].lp_apply(s["params"], s["R"], s["theta"])
    # A solve.  LOBPCG returns energies and vectors; an eigenvector is defined up to its sign, so
    # the caller fixes it (largest component positive), and keeps the vectors in FP32, as the start
    # of a larger FP32 solve.  The mixed-precision hybrid stops at a residual of 1e-6, where the
    # energies are exact to the residual's square over the gap but a vector only to the residual
    # over the gap, wherever the last step happens to land: the caller asks for the energies.
    s["handle"].solve(case["method"], s["X0"], tol=case["tol"], vec_type=binding.STORAGE[case["vec"]], switch_res=1e-2,
                      switch_tau=0.0, switch_gap=0.03, rmm_precond=1, maxiter=case["maxiter"])
    theta, X = s["handle"].ritz(case["method"] == "lobpcg")
    if X is None:
        return dict(theta=theta)
    return dict(theta=theta, X=(X * torch.sign(X.gather(0, X.abs().argmax(0, keepdim=True)))).float())


# ---------------------------------------------------------------------------------------
# work
# ---------------------------------------------------------------------------------------
def _nnz(case):
    """Stored nonzeros (upper triangle) of the generator's matrix, in the mean."""
    return 0.5 * case["n"] * (case["per_row"] + 1)


def _product(case, nb, vec_bytes):
    stored = _nnz(case) * (VALUE_BYTES[case["val"]] + 4) + 8 * (case["n"] + 1)
    return stored, 2.0 * case["n"] * nb * vec_bytes, 2.0 * (2 * _nnz(case) - case["n"]) * nb


def work(case):
    op = case["op"]
    vb = VALUE_BYTES[case["vec"]] if "vec" in case else 8
    if op in ("spmm", "plan"):
        mat, vec, fl = _product(case, case["nb"], 8 if op == "plan" and case["val"] == "f64" else vb)
        return dict(bytes=mat + vec, flops=fl)
    if op == "filter":
        # each step needs the whole matrix again; the recurrence reads one block more
        mat, vec, fl = _product(case, case["nb"], vb)
        return dict(bytes=case["degree"] * (mat + 1.5 * vec), flops=case["degree"] * fl)
    if op == "gram":
        return dict(bytes=2 * case["n"] * case["nb"] * vb + 8 * case["nb"] ** 2, flops=2.0 * case["n"] * case["nb"] ** 2)
    if op == "cholqr2":
        return dict(bytes=2 * case["n"] * case["nb"] * vb, flops=6.0 * case["n"] * case["nb"] ** 2)
    if op == "ritz":
        k = case["k"]
        return dict(bytes=8 * k * (k * (2 if case["pencil"] else 1) + case["nb"]), flops=(4.0 / 3.0 + 2.0 * case["pencil"]) * k ** 3)
    if op == "train":
        return dict(bytes=32.0 * case["n"] * case["m"], flops=3 * 2496.0 * case["n"] * case["m"])
    if op == "apply":
        mat, vec, fl = _product(case, case["nb"], vb)
        return dict(bytes=mat + vec + 16 * case["n"], flops=fl + 2516.0 * case["n"] * case["nb"])
    # a solve: at least one product per two digits, each with the matrix once
    mat, vec, fl = _product(case, case["nb"], vb)
    steps = max(4, int(-math.log10(case["tol"])) // 2 * 2)
    return dict(bytes=steps * (mat + 5 * vec), flops=steps * (fl + 20.0 * case["n"] * case["nb"] ** 2))


# ---------------------------------------------------------------------------------------
# the same in 64 bits, with torch alone
# ---------------------------------------------------------------------------------------
def _full(H):
    """Both triangles as a FP64 sparse CSR tensor."""
    r, c, v = H.rows(), H.col.long(), H.values64()
    off = r != c
    A = torch.sparse_coo_tensor(torch.stack([torch.cat([r, c[off]]), torch.cat([c, r[off]])]),
                                torch.cat([v, v[off]]), (H.n, H.n), check_invariants=False)
    return A.coalesce().to_sparse_csr()


def _network(p, F):
    """MLP output o of the feature rows (FP64)."""
    u = (F - p[0:6]) / p[6:12]
    h = torch.relu(u @ p[12:204].view(32, 6).T + p[204:236])
    h = torch.relu(h @ p[236:1260].view(32, 32).T + p[1260:1292])
    return h @ p[1292:1324] + p[1324]


def _jscale(f2):
    return 1.0 / (f2.abs().clamp(min=2.0) * torch.where(f2 < 0, -1.0, 1.0))


def _lanczos(A, v, n_ev, tol, most=700):
    """Lowest n_ev eigenpairs: Lanczos with full reorthogonalisation."""
    n = v.numel()
    V = torch.empty(most + 1, n, dtype=torch.float64, device=DEV)
    V[0] = v / v.norm()
    d, e = [], []
    for j in range(most):
        w = A @ V[j]
        d.append(float(V[j] @ w))
        for _ in range(2):
            w = w - V[:j + 1].T @ (V[:j + 1] @ w)
        e.append(float(w.norm()))
        V[j + 1] = w / e[-1]
        if (j + 1) % 50 == 0:
            T = np.diag(d) + np.diag(e[:-1], 1) + np.diag(e[:-1], -1)
            th, Z = np.linalg.eigh(T)
            if np.all(e[-1] * np.abs(Z[-1, :n_ev]) <= tol):
                return th[:n_ev], V[:j + 1].T @ torch.from_numpy(np.ascontiguousarray(Z[:, :n_ev])).to(DEV)
    return None, None


def exact(case, seed):
    op = case["op"]
    if op in ("spmm", "filter", "plan", "apply", "solve"):
        H = _matrix(case, seed)
        A = _full(H)
    if op in ("spmm", "plan"):
        X = _block(H.n, case["nb"], seed, 2, torch.float64 if case["val"] == "f64" else TORCH[case["vec"]])
        return A @ X.double()
    if op == "filter":
        ub = float(_levels(H.n)[-1]) + 4.0
        c, e = 0.5 * (ub + 2.5), 0.5 * (ub - 2.5)
        Q = _block(H.n, case["nb"], seed, 2, TORCH[case["vec"]]).double()
        W = (A @ Q - c * Q) / e
        for _ in range(case["degree"] - 1):
            Q, W = W, 2.0 * (A @ W - c * W) / e - Q
        return W
    if op == "apply":
        d = H.values64()[H.rowptr[:-1]]
        R = (_block(H.n, case["nb"], seed, 3, TORCH[case["vec"]]) * 1e-2).double()
        th = torch.linspace(-0.1, 2.5, case["nb"], dtype=torch.float64, device=DEV)
        rowabs = torch.sparse_csr_tensor(A.crow_indices(), A.col_indices(), A.values().abs(), A.shape) @ torch.ones(
            H.n, dtype=torch.float64, device=DEV)
        sc = math.sqrt(H.n) / R.norm(dim=0)
        HR = A @ R
        p = torch.from_numpy(_params(seed)).to(DEV).double()
        W = torch.empty_like(R)
        for j in range(case["nb"]):
            F = torch.stack([d, th[j].expand(H.n), d - th[j], rowabs, R[:, j] * sc[j], (HR[:, j] - d * R[:, j]) * sc[j]], 1)
            W[:, j] = _jscale(F[:, 2]) * (1.0 + _network(p, F)) * R[:, j]
        return W
    if op == "solve":
        X0 = _start_block(H, case["nb"])
        theta, X = _lanczos(A, X0[:, :case["n_ev"]].mean(1), case["n_ev"], 1e-11)
        if theta is None:
            return None
        if case["method"] != "lobpcg":
            return dict(theta=theta)
        X = X * torch.sign(X.gather(0, X.abs().argmax(0, keepdim=True)))
        return dict(theta=theta, X=X)
    if op == "gram":
        s = prepare(case, seed)
        return s["A"].double().T @ s["B"].double()
    if op == "cholqr2":
        X = prepare(case, seed)["X"].double()
        R = torch.linalg.cholesky(X.T @ X, upper=True)
        return dict(Q=torch.linalg.solve_triangular(R, X, upper=True, left=False), R=R)
    if op == "ritz":
        A, G = _pencil(case, seed)
        if case["pencil"]:
            L = torch.linalg.cholesky(G)
            Y = torch.linalg.solve_triangular(L, A, upper=False)
            A = torch.linalg.solve_triangular(L, Y.T.contiguous(), upper=False)
            return dict(theta=torch.linalg.eigvalsh(0.5 * (A + A.T))[:case["nb"]], C=None, info=0)
        return dict(w=torch.linalg.eigvalsh(0.5 * (A + A.T))[:case["nb"]], Z=None)
    # train
    s = prepare(case, seed)
    smp = s["sample"]
    p = s["p"].double().requires_grad_(True)
    m1, m2, p0, t = s["m1"].double(), s["m2"].double(), s["p"].double(), s["t"] + 1
    loss = torch.zeros((), dtype=torch.float64, device=DEV)
    for a in range(0, smp["F"].shape[0], 400_000 // smp["m"] * smp["m"]):
        b = a + 400_000 // smp["m"] * smp["m"]
        F, r, z = smp["F"][a:b].double(), smp["r"][a:b].double(), smp["z"][a:b].double()
        w = smp["colw"].repeat(F.shape[0] // smp["m"])
        part = (w * (_jscale(F[:, 2]) * (1.0 + _network(p, F)) * r - z).square()).sum()
        part.backward()
        loss += part.detach()
    g = p.grad.clone()
    a1, a2 = 0.9 * m1 + 0.1 * g, 0.999 * m2 + 0.001 * g * g
    p1 = p0 - 1e-3 * (a1 / (1 - 0.9 ** t)) / ((a2 / (1 - 0.999 ** t)).sqrt() + 1e-8)
    for new, old in ((a1, m1), (a2, m2), (p1, p0)):
        new[:12] = old[:12]                # the feature statistics are not trained
    return dict(grad=torch.cat([g[12:], loss[None]]), p=p1, m1=a1, m2=a2)
