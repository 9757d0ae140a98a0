"""The work that users of this framework have it do, as cases that can be timed
and compared: reconstructions of one scan or of a batch of scans through
sgtv.Handle in its forms, precisions and options, the warm-start network's
inference and training step, and one warm-started solve from counts to image.

A case is a dict of plain values; "kind" says which path it takes:
  scan   one scan: `iters` ADMM iterations, then the image and the objective
         (`evals` times, as a user's traced solve does; `state` returns the
         whole ADMM state as a checkpoint stores it)
  batch  several scans of uneven shapes in one handle, the same pass
  net    the network's forward pass on resident inputs
  train  one training step: loss, gradients and the Adam update
  warm   a scan's counts swapped into a resident instrument, the network's
         start, then plain iterations (the warm-start driver's own calls)

Every pass of scan and batch continues the handle's solve, so a second pass
starts where the first one ended.

Inputs follow the recipe of paper_1601_08201_gb300/synth.py (a shifted coded
aperture, a phantom of rectangles with Gaussian-mixture profiles, Poisson
counts), drawn on the GPU because a full-size matrix is drawn many times.
"""
import math

import numpy as np
import torch

from paper_1601_08201_gb300 import sgtv, synth, warmstart, wsnet

DEV = "cuda" if torch.cuda.is_available() else "cpu"


# ------------------------------------------------------------------------------------------
# the cases

def _scan(name, Nx, Nz, Nq, I, nnz_col, counts, iters, rho=1.0, precision="fp32", single_pass=False, graph=False,
          standard_tv=False, n_dirs=4, n_inner=1, evals=1, state=False, **more):
    c = dict(kind="scan", Nx=Nx, Nz=Nz, Nq=Nq, I=I, nnz_col=nnz_col, counts=counts, rho=rho, precision=precision,
             single_pass=single_pass, graph=graph, standard_tv=standard_tv, n_dirs=n_dirs, n_inner=n_inner,
             iters=iters, evals=evals, state=state, **more)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest solve, with the defaults of the README's first example; a checkpoint of the whole
        # state at its end: launches, small grids and host calls decide
        _scan("tiny_checkpoint", 16, 16, 32, 4096, 64, 50.0, iters=20, rho=256.0, state=True),
        # the shape of the paper's scan (41 x 9 spatial bins, 54 q-bins, 128 x 64 detector), the fastest
        # form: a clinical-size image reconstructed in one go
        _scan("paper_single_pass", 41, 9, 54, 8192, 64, 26.0, iters=104, single_pass=True, graph=True),
        # the checking mode: FP64 everywhere, ragged sizes (no multiple of a warp, a tile or a vector)
        _scan("ragged_fp64", 13, 7, 37, 3001, 50, 30.0, iters=10, rho=256.0, precision="fp64",
              state=True),
        # the other regulariser and the options: per-bin TV, the two-direction stencil, two surrogate steps,
        # more q-bins than a warp keeps in registers, odd sizes
        _scan("standard_tv_options", 45, 31, 150, 70001, 48, 20.0, iters=16, single_pass=True, standard_tv=True,
              n_dirs=2, n_inner=2),
        # the instrument of the warm-start protocol (64^3, one measurement per hyper-voxel) in the plain
        # two-pass form with graphs at the fast penalty, its objective traced every 10 iterations
        _scan("instrument_trace", 64, 64, 64, 262144, 128, 30.0, iters=50, rho=4096.0, graph=True, evals=5),
        # a quarter of the full-size problem with the default options (two passes, no graph)
        _scan("quarter_two_pass", 128, 128, 16, 262144, 256, 20.0, iters=16),
        # BF16 values of A, the precision form, on half the full-size problem
        _scan("half_bf16", 128, 128, 32, 524288, 256, 20.0, iters=16, precision="bf16", single_pass=True, graph=True),
        # the headline: 1M hyper-voxels, 1M measurements, 2^28 nonzeros, FP32, single pass
        _scan("full_single_pass", 128, 128, 64, 1 << 20, 256, 20.0, iters=20, single_pass=True),
        # many scans of uneven shapes in one handle (the batched form's shape ranges, fewer scans)
        dict(name="batch_uneven", kind="batch", scans=6, nx_min=32, nx_max=80, nnz_col=128, precision="fp32",
             single_pass=True, graph=True, iters=16, shapes=3000),
        # the network proposing the start of one scan (inference, one sample)
        dict(name="net_inference", kind="net", H=64, W=64, Q=64, n_dual=0, batch=1),
        # one training step of the protocol: 8 scans, image and dual channels
        dict(name="net_training_step", kind="train", H=64, W=64, Q=64, n_dual=4, batch=8),
        # a whole warm-started solve at the size that the warm-start tests use
        dict(name="warm_solve", kind="warm", Nx=32, Nz=32, Nq=16, nnz_col=64, counts=30.0, rho=4096.0, iters=64),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges (sizes uniform in their logarithm)."""
    u = rng.random()
    if u < 0.6:
        Nx, Nz, Nq = _log_int(rng, 8, 128), _log_int(rng, 7, 128), _log_int(rng, 9, 160)
        J = Nx * Nz * Nq
        I = max(1000, min(1 << 20, int(J * rng.uniform(0.3, 1.2))))
        cap = max(16, min(256, I // 8, (1 << 27) // J))
        nnz_col = _log_int(rng, 16, cap) if cap > 16 else 16
        if J * nnz_col > 1 << 27:  # no dearer than the largest listed case
            Nq = max(9, (1 << 27) // (Nx * Nz * nnz_col))
        precision = rng.choice(["fp32", "fp32", "fp32", "bf16", "fp64"])
        work = Nx * Nz * Nq * nnz_col
        if precision == "fp64" and work > 1 << 25:
            precision = "fp32"
        return _scan(None, Nx, Nz, Nq, I, nnz_col, round(rng.uniform(5.0, 100.0), 1),
                     iters=rng.choice([8, 11, 16, 24]) if work > 1 << 23 else rng.choice([10, 24, 50]),
                     rho=rng.choice([1.0, 1.0, 64.0, 4096.0]), precision=precision,
                     single_pass=rng.random() < 0.6, graph=rng.random() < 0.5, standard_tv=rng.random() < 0.2,
                     n_dirs=rng.choice([4, 4, 4, 2]), n_inner=rng.choice([1, 1, 1, 2]))
    if u < 0.7:
        return dict(kind="batch", scans=rng.randint(2, 6), nx_min=16, nx_max=rng.randint(24, 72),
                    nnz_col=rng.choice([32, 64, 128]), precision=rng.choice(["fp32", "fp32", "bf16"]),
                    single_pass=rng.random() < 0.7, graph=rng.random() < 0.7, iters=rng.choice([8, 11, 16]),
                    shapes=rng.randint(1, 1 << 20))
    H, W = 4 * _log_int(rng, 4, 16), 4 * _log_int(rng, 4, 16)
    Q = _log_int(rng, 12, 64)
    if u < 0.8:
        return dict(kind="net", H=H, W=W, Q=Q, n_dual=rng.choice([0, 2, 4]), batch=rng.randint(1, 8))
    if u < 0.9:
        return dict(kind="train", H=H, W=W, Q=Q, n_dual=rng.choice([0, 4]), batch=rng.randint(2, 8))
    return dict(kind="warm", Nx=H, Nz=W, Nq=_log_int(rng, 12, 48), nnz_col=rng.choice([32, 64]),
                counts=round(rng.uniform(5.0, 100.0), 1), rho=4096.0, iters=rng.choice([32, 64]))


# ------------------------------------------------------------------------------------------
# inputs

def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return g


def _matrix(g, Nx, Nz, Nq, I, nnz_col):
    """A by columns and by rows (tensors on the GPU): every column holds nnz_col
    nonzeros, the set bits of a coded aperture shifted by x from the column's
    window start on, values U(0.1, 1)."""
    code = torch.rand(I, generator=g, device=DEV) < 0.5
    code[:nnz_col] = True  # enough set bits however the code falls
    ones = torch.nonzero(code).reshape(-1)
    n1, ZQ, shift = ones.numel(), Nz * Nq, I // Nx
    J = Nx * ZQ
    start = torch.arange(ZQ, device=DEV) * I // ZQ
    m = torch.arange(nnz_col, device=DEV)
    row = torch.empty((J, nnz_col), dtype=torch.int32, device=DEV)
    for x in range(Nx):
        k0 = torch.searchsorted(ones, (start + x * shift) % I)
        row[x * ZQ:(x + 1) * ZQ] = ((ones[(k0[:, None] + m) % n1] - x * shift) % I).to(torch.int32)
    row = row.sort(dim=1).values
    val = 0.1 + 0.9 * torch.rand((J, nnz_col), generator=g, device=DEV)
    order = row.reshape(-1).sort(stable=True).indices
    rowptr = torch.zeros(I + 1, dtype=torch.int64, device=DEV)
    rowptr[1:] = torch.bincount(row.reshape(-1), minlength=I).cumsum(0)
    col = torch.div(order, nnz_col, rounding_mode="floor").to(torch.int32)
    return row, val, rowptr, col, val.reshape(-1)[order]


def _phantom(rng, Nx, Nz, Nq, regions):
    """Piecewise-constant rectangles over zero, each with a Gaussian-mixture profile in q."""
    f = np.zeros((Nx, Nz, Nq))
    q = np.arange(Nq)
    for _ in range(regions):
        wx = int(rng.integers(max(1, Nx // 8), max(1, Nx // 2) + 1))
        wz = int(rng.integers(max(1, Nz // 8), max(1, Nz // 2) + 1))
        x0, z0 = int(rng.integers(0, Nx - wx + 1)), int(rng.integers(0, Nz - wz + 1))
        mtp = np.zeros(Nq)
        for _ in range(int(rng.integers(2, 5))):
            mu, sigma = rng.uniform(0.0, Nq), rng.uniform(1.0, max(1.0001, Nq / 8.0))
            mtp += rng.uniform(0.5, 1.0) * np.exp(-((q - mu) ** 2) / (2.0 * sigma * sigma))
        f[x0:x0 + wx, z0:z0 + wz, :] = mtp
    return torch.from_numpy(f.reshape(-1)).to(DEV)


def _problem(seed, Nx, Nz, Nq, I, nnz_col, counts, rho, regions=4):
    """A synth.Problem (host arrays, as sgtv.Handle takes them) and A on the GPU."""
    g = _gen(seed)
    row, val, rowptr, col, cval = A = _matrix(g, Nx, Nz, Nq, I, nnz_col)
    f = _phantom(np.random.default_rng(seed), Nx, Nz, Nq, regions)
    J = Nx * Nz * Nq
    Af = torch.segment_reduce(cval.double() * f[col.long()], "sum", lengths=rowptr.diff())
    scale = (counts / 1.1) / float(Af.mean())
    r = 0.1 * float(Af.mean()) * scale
    y = torch.poisson(Af * scale + r, generator=g).float()
    beta = 0.05 * float((val.double() * y.double()[row.long()]).sum(1).max())
    host = lambda t: t.cpu().numpy()  # noqa: E731
    P = synth.Problem(Nx=Nx, Nz=Nz, Nq=Nq, I=I, J=J, nnz=J * nnz_col,
                      csc_colptr=np.arange(0, J * nnz_col + 1, nnz_col, dtype=np.int64), csc_row=host(row.reshape(-1)),
                      csc_val=host(val.reshape(-1)), csr_rowptr=host(rowptr), csr_col=host(col), csr_val=host(cval),
                      y=host(y), b=np.array([r], dtype=np.float32), beta=beta, rho=float(rho),
                      f_true=host((f * scale).float()), seed=seed)
    return P, A


def _counts(seed, P, A, counts):
    """Another scan's counts through the instrument P (as synth.measure draws them)."""
    row, val, rowptr, col, cval = A
    g = _gen(seed)
    f = _phantom(np.random.default_rng(seed), P.Nx, P.Nz, P.Nq, 4)
    Af = torch.segment_reduce(cval.double() * f[col.long()], "sum", lengths=rowptr.diff())
    scale = (counts / 1.1) / float(Af.mean())
    r = 0.1 * float(Af.mean()) * scale
    y = torch.poisson(Af * scale + r, generator=g).float()
    beta = 0.05 * float((val.double() * y.double()[row.long()]).sum(1).max())
    M = synth.Problem(**{**P.__dict__, "y": y.cpu().numpy(), "b": np.array([r], dtype=np.float32), "beta": beta})
    return M


def _batch_problems(case, seed):
    """Scans of uneven shapes: the case fixes the shapes, the seed the contents."""
    rng = np.random.default_rng(case["shapes"])
    out = []
    for k in range(case["scans"]):
        Nx, Nz = (int(rng.integers(case["nx_min"], case["nx_max"] + 1)) for _ in range(2))
        Nq = int(rng.choice([32, 64, 128]))
        counts = float(rng.uniform(5.0, 100.0))
        out.append((Nx, Nz, Nq, counts, seed * 64 + k))
    return out


def _net_layers(Q, n_dual):
    return [(Q + 1, 64), (64, 64), (64, 128), (128, 128), (128, 256), (256, 128), (128, 64), (64, 64),
            (64, Q * (1 + n_dual))]


def _net_params(seed, Q, n_dual):
    """He-initialised weights (the last layer ten times smaller), small biases, in the packed order."""
    rng = np.random.default_rng(seed)
    parts = []
    for l, (ci, co) in enumerate(_net_layers(Q, n_dual)):
        std = math.sqrt(2.0 / (9 * ci)) * (0.1 if l == 8 else 1.0)
        parts += [std * rng.standard_normal(co * ci * 9), 0.02 * rng.standard_normal(co)]
    return np.concatenate(parts).astype(np.float32)


def _net_data(seed, case):
    """Inputs as the driver packs them (a noisy positive image of mean 1 and a constant count-level
    channel) and targets (an image in units of the flat start, a dual within the unit ball)."""
    g = _gen(seed)
    N, Q, H, W = case["batch"], case["Q"], case["H"], case["W"]
    x = torch.empty((N, Q + 1, H, W), device=DEV)
    t = torch.empty((N, Q * (1 + case["n_dual"]), H, W), device=DEV)
    for n in range(N):
        img = _phantom(np.random.default_rng(seed * 16 + n), H, W, Q, 4).reshape(H, W, Q).permute(2, 0, 1).float()
        img = img / img.mean()
        noisy = 0.5 + 0.5 * img + 0.2 * torch.rand((Q, H, W), generator=g, device=DEV)
        x[n, :Q] = noisy / noisy.mean()
        x[n, Q] = 0.4 + 0.5 * torch.rand(1, generator=g, device=DEV)
        t[n, :Q] = img
        t[n, Q:] = 0.2 * torch.randn(t[n, Q:].shape, generator=g, device=DEV)
    return x, t


def _flags(case):
    return ((sgtv.FLAG_SINGLE_PASS if case["single_pass"] else 0) | (sgtv.FLAG_GRAPH if case["graph"] else 0)
            | (sgtv.FLAG_STANDARD_TV if case.get("standard_tv") else 0))


def _weights(case):
    return [1.0, 1.0, 1.0, 1.0] if case["n_dirs"] == 4 else [0.8, 1.25]


def prepare(case, seed):
    kind = case["kind"]
    if kind == "scan":
        P, _ = _problem(seed, *(case[k] for k in ("Nx", "Nz", "Nq", "I", "nnz_col", "counts", "rho")))
        h = sgtv.Handle(P, n_dirs=case["n_dirs"], w=_weights(case), n_inner=case["n_inner"],
                        precision=case["precision"], flags=_flags(case))
        return dict(case=case, h=h, image=np.zeros(P.J, np.float32))
    if kind == "batch":
        Ps = [_problem(s, Nx, Nz, Nq, Nx * Nz * Nq, case["nnz_col"], counts, 1.0)[0]
              for Nx, Nz, Nq, counts, s in _batch_problems(case, seed)]
        h = sgtv.Handle(Ps, precision=case["precision"], flags=_flags(case))
        return dict(case=case, h=h, image=np.zeros(sum(P.J for P in Ps), np.float32))
    if kind == "warm":
        P, A = _problem(seed, case["Nx"], case["Nz"], case["Nq"], case["Nx"] * case["Nz"] * case["Nq"],
                        case["nnz_col"], case["counts"], case["rho"])
        M = _counts(seed + (1 << 20), P, A, case["counts"])
        solver = warmstart.Solver(P, torch, flags=sgtv.FLAG_GRAPH | sgtv.FLAG_SINGLE_PASS, rho=case["rho"])
        net = wsnet.WarmNet(case["Nx"], case["Nz"], case["Nq"], 1, seed=0)
        net.set_params(_net_params(seed, case["Nq"], 0))
        return dict(case=case, solver=solver, net=net, scan=M)
    x, t = _net_data(seed, case)
    net = wsnet.WarmNet(case["H"], case["W"], case["Q"], case["batch"], seed=0, n_dual=case["n_dual"])
    net.set_params(_net_params(seed, case["Q"], case["n_dual"]))
    torch.cuda.synchronize()  # the network runs on its own stream
    return dict(case=case, net=net, x=x, t=t, out=torch.zeros_like(t))


# ------------------------------------------------------------------------------------------
# one pass

def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind in ("scan", "batch"):
        h = state["h"]
        if case.get("state"):
            h.iterate(case["iters"])
            s = h.get_state_f64()
            # the FP32 mode holds its state in 32 bits; a checkpoint stores what is held
            return s if case["precision"] == "fp64" else tuple(np.asarray(a, np.float32) for a in s)
        evals = case.get("evals", 1)
        phis = []
        for _ in range(evals):
            h.iterate(case["iters"] // evals)
            phis.append(h.objective())
        return dict(image=sgtv.get_image(h.h, state["image"]), objective=phis)
    if kind == "net":
        state["net"].forward(state["x"].data_ptr(), case["batch"], state["out"].data_ptr())
        return state["out"]
    if kind == "train":
        net = state["net"]
        loss = net.loss_grad(state["x"].data_ptr(), state["t"].data_ptr(), case["batch"])
        net.adam_step(1e-4)
        return dict(loss=loss, grads=net.get_grads())
    solver, M = state["solver"], state["scan"]
    solver.load(M)
    f0 = warmstart.warm_image(solver, state["net"], M, torch)
    solver.h.warm_start(f0.data_ptr(), 0.0)
    return dict(start=f0, image=solver.solve(case["iters"]))


# ------------------------------------------------------------------------------------------
# what a pass cannot do without

def _scan_work(J, I, nnz, case):
    """Bytes of `iters` iterations: each surrogate step needs A's values once (V bytes per nonzero;
    their positions can be held in far fewer bytes, so none are counted), f in and out, s, y; the
    shrink c in and out, d out, per direction."""
    T = 8 if case["precision"] == "fp64" else 4
    V = {"fp32": 4, "bf16": 2, "fp64": 8}[case["precision"]]
    nd, ni, it = case.get("n_dirs", 4), case.get("n_inner", 1), case["iters"]
    per = ni * (nnz * V + T * (3 * J + I) + T * nd * J) + T * 3 * nd * J
    flops = ni * (4 * nnz + (10 * nd + 12) * J) + 10 * nd * J
    ev = case.get("evals", 1) if not case.get("state") else 0
    return dict(bytes=it * per + ev * (nnz * V + T * (J + I)) + 4 * J, flops=it * flops + ev * 2 * nnz)


def _net_macs(H, W, Q, n_dual):
    px = [1, 1, 4, 4, 16, 16, 4, 1, 1]
    return sum(9 * ci * co * (H * W // p) for (ci, co), p in zip(_net_layers(Q, n_dual), px))


def _net_params_count(Q, n_dual):
    return sum(9 * ci * co + co for ci, co in _net_layers(Q, n_dual))


def work(case):
    kind = case["kind"]
    if kind == "scan":
        J = case["Nx"] * case["Nz"] * case["Nq"]
        return _scan_work(J, case["I"], J * case["nnz_col"], case)
    if kind == "batch":
        J = sum(Nx * Nz * Nq for Nx, Nz, Nq, _, _ in _batch_problems(case, 0))
        return _scan_work(J, J, J * case["nnz_col"], case)
    if kind == "warm":
        J = case["Nx"] * case["Nz"] * case["Nq"]
        w = _scan_work(J, J, J * case["nnz_col"], dict(case, precision="fp32"))
        macs = _net_macs(case["Nx"], case["Nz"], case["Nq"], 0)
        return dict(bytes=w["bytes"] + 2 * _net_params_count(case["Nq"], 0), flops=w["flops"] + 2 * macs)
    H, W, Q, nd, N = (case[k] for k in ("H", "W", "Q", "n_dual", "batch"))
    macs, params = N * _net_macs(H, W, Q, nd), _net_params_count(Q, nd)
    io = 4 * N * H * W * (Q + 1 + Q * (1 + nd))
    if kind == "net":
        return dict(bytes=io + 2 * params, flops=2 * macs)
    first = N * 9 * (Q + 1) * 64 * H * W  # no gradient for the network's input
    return dict(bytes=io + (2 + 4 + 6 * 4) * params, flops=2 * (3 * macs - first))


# ------------------------------------------------------------------------------------------
# the same in 64 bits, in plain torch

def _product(ptr, idx, val, v):
    """Row sums of val * v[idx] over the segments of ptr, at most 2^27 elements at a time."""
    out, n = [], ptr.numel() - 1
    step = max(1, min(n, int((1 << 27) * n // max(1, idx.numel()))))
    for a in range(0, n, step):
        b = min(n, a + step)
        lo, hi = int(ptr[a]), int(ptr[b])
        out.append(torch.segment_reduce(val[lo:hi].double() * v[idx[lo:hi].long()], "sum", lengths=ptr[a:b + 1].diff(),
                                        initial=0.0))
    return torch.cat(out)


def _shift(a, dx, dz):
    """a at the neighbour (x + dx, z + dz), zero outside, on the first two axes."""
    out = torch.zeros_like(a)
    Nx, Nz = a.shape[:2]
    xs, xd = slice(max(0, dx), Nx + min(0, dx)), slice(max(0, -dx), Nx + min(0, -dx))
    zs, zd = slice(max(0, dz), Nz + min(0, dz)), slice(max(0, -dz), Nz + min(0, -dz))
    out[xd, zd] = a[xs, zs]
    return out


class _Solve64:
    """The iteration of include/sgtv.h (Eqs. 5-7) on one scan, dense tensors in 64 bits."""

    def __init__(self, A, P, beta, rho, n_dirs=4, w=(1.0, 1.0, 1.0, 1.0), n_inner=1, per_bin=False, bf16=False):
        self.row, self.val, self.rowptr, self.col, self.cval = A
        if bf16:  # the precision form's matrix is A rounded to BF16
            self.val, self.cval = self.val.bfloat16().float(), self.cval.bfloat16().float()
        self.shape = (P.Nx, P.Nz, P.Nq)
        self.y = torch.from_numpy(P.y).to(DEV).double()
        self.r = float(P.b[0])
        self.beta, self.rho, self.tau, self.n_inner, self.per_bin = beta, rho, beta / rho, n_inner, per_bin
        self.dirs = [(1, 0), (-1, 0), (0, 1), (0, -1)] if n_dirs == 4 else [(1, 0), (0, 1)]
        self.w = list(w)[:n_dirs]
        self.colptr = torch.arange(0, self.val.numel() + 1, self.val.shape[1], device=DEV)
        self.s = self.val.double().sum(1)
        num = float(self.y.sum()) - self.r * self.y.numel()
        num = num if num > 0 else (float(self.y.sum()) or 1.0)
        self.kappa = num / float(self.s.sum())
        self.start(torch.full_like(self.s, self.kappa))

    def back(self, v):
        return _product(self.colptr, self.row.reshape(-1), self.val.reshape(-1), v)

    def grad(self, f):
        f = f.reshape(self.shape)
        return [w * (f - _shift(f, dx, dz)) for w, (dx, dz) in zip(self.w, self.dirs)]

    def start(self, f):
        self.f = f
        self.d = self.grad(f)
        self.c = [torch.zeros_like(v) for v in self.d]

    def iterate(self, n):
        one = torch.ones(self.shape[:2] + (1,), dtype=torch.float64, device=DEV)
        for _ in range(n):
            for _ in range(self.n_inner):
                ybar = _product(self.rowptr, self.col, self.cval, self.f) + self.r
                e = self.back(torch.where(self.y == 0, 0.0, self.y / ybar)).reshape(self.shape)
                f = self.f.reshape(self.shape)
                alpha, gamma = torch.zeros_like(f), torch.zeros_like(f)
                for w, (dx, dz), d, c in zip(self.w, self.dirs, self.d, self.c):
                    u = d - c
                    inF, inB = _shift(one, dx, dz), _shift(one, -dx, -dz)
                    alpha += w * w * (0.5 + 0.5 * inF + inB)
                    gamma += w * (w * inF * (f + _shift(f, dx, dz)) + u)
                    gamma += w * inB * (w * (f + _shift(f, -dx, -dz)) - _shift(u, -dx, -dz))
                alpha, B = self.rho * alpha, self.s.reshape(self.shape) - self.rho * gamma
                disc = torch.sqrt(B * B + 8 * alpha * f * e)
                pos = torch.where(B + disc > 0, 2 * f * e / (B + disc), 0.0)
                self.f = torch.where(B >= 0, pos, (disc - B) / (4 * alpha)).reshape(-1)
            v = [g + c for g, c in zip(self.grad(self.f), self.c)]
            n2 = sum(a * a for a in v)
            n2 = n2 if self.per_bin else n2.sum(2, keepdim=True)
            norm = torch.sqrt(n2)
            k = torch.where(norm > 0, 1 - self.tau / norm, 0.0).clamp(min=0)
            self.d = [k * a for a in v]
            self.c = [a - b for a, b in zip(v, self.d)]

    def objective(self):
        ybar = _product(self.rowptr, self.col, self.cval, self.f) + self.r
        t = torch.where(self.y > 0, self.y * torch.log(torch.where(self.y > 0, self.y, 1.0) / ybar), 0.0)
        n2 = sum(a * a for a in self.grad(self.f))
        tv = float(torch.sqrt(n2 if self.per_bin else n2.sum(2)).sum())
        dev = float((ybar - self.y + t).sum())
        return dev + self.beta * tv, dev, tv


def _net64(params, x, Q, n_dual):
    """The network of include/wsnet.h in 64 bits (weights rounded to BF16, as every kernel uses
    them), from a packed parameter tensor: the output, and the weights as leaves for gradients."""
    F = torch.nn.functional
    leaves, off = [], 0
    for ci, co in _net_layers(Q, n_dual):
        W = params[off:off + 9 * ci * co].bfloat16().double().reshape(co, ci, 3, 3).requires_grad_()
        b = params[off + 9 * ci * co:off + 9 * ci * co + co].double().requires_grad_()
        leaves.append((W, b))
        off += 9 * ci * co + co
    conv = lambda a, l: F.conv2d(a, *leaves[l], padding=1)  # noqa: E731
    up = lambda a: F.interpolate(a, scale_factor=2, mode="nearest")  # noqa: E731
    a2 = conv(conv(x.double(), 0).relu(), 1).relu()
    a4 = conv(conv(F.avg_pool2d(a2, 2), 2).relu(), 3).relu()
    a6 = conv(conv(F.avg_pool2d(a4, 2), 4).relu(), 5).relu()
    a7 = conv(up(a6) + a4, 6).relu()
    z = conv(conv(up(a7) + a2, 7).relu(), 8)
    return torch.cat([F.softplus(z[:, :Q]), z[:, Q:]], 1), leaves


def _solve64_of(case, seed):
    P, A = _problem(seed, *(case[k] for k in ("Nx", "Nz", "Nq", "I", "nnz_col", "counts", "rho")))
    return _Solve64(A, P, P.beta, P.rho, case["n_dirs"], _weights(case), case["n_inner"], case["standard_tv"],
                    case["precision"] == "bf16")


def exact(case, seed):
    kind = case["kind"]
    if kind == "scan":
        S = _solve64_of(case, seed)
        if case["state"]:
            S.iterate(case["iters"])
            return S.f, torch.cat([d.reshape(-1) for d in S.d]), torch.cat([c.reshape(-1) for c in S.c])
        phis = []
        for _ in range(case["evals"]):
            S.iterate(case["iters"] // case["evals"])
            phis.append(tuple(np.float64(v) for v in S.objective()))
        return dict(image=S.f, objective=phis)
    if kind == "batch":
        images, sums = [], np.zeros(3)
        for Nx, Nz, Nq, counts, s in _batch_problems(case, seed):
            P, A = _problem(s, Nx, Nz, Nq, Nx * Nz * Nq, case["nnz_col"], counts, 1.0)
            S = _Solve64(A, P, P.beta, P.rho, bf16=case["precision"] == "bf16")
            S.iterate(case["iters"])
            images.append(S.f)
            sums += S.objective()
        return dict(image=torch.cat(images), objective=[tuple(np.float64(v) for v in sums)])
    if kind == "warm":
        P, A = _problem(seed, case["Nx"], case["Nz"], case["Nq"], case["Nx"] * case["Nz"] * case["Nq"],
                        case["nnz_col"], case["counts"], case["rho"])
        M = _counts(seed + (1 << 20), P, A, case["counts"])
        S = _Solve64(A, M, M.beta, case["rho"])
        bp = S.back(S.y) / S.s
        x = torch.empty((1, P.Nq + 1, P.Nx, P.Nz), dtype=torch.float64, device=DEV)
        x[0, :P.Nq] = (bp / bp.mean()).reshape(S.shape).permute(2, 0, 1)
        x[0, P.Nq] = math.log(max(float(S.y.mean()), 1e-3)) / 5.0
        params = torch.from_numpy(_net_params(seed, P.Nq, 0)).to(DEV)
        with torch.no_grad():
            out, _ = _net64(params, x, P.Nq, 0)
        f0 = S.kappa * out[0].permute(1, 2, 0).reshape(-1)
        S.start(f0)
        S.iterate(case["iters"])
        return dict(start=f0, image=S.f)
    x, t = _net_data(seed, case)
    params = torch.from_numpy(_net_params(seed, case["Q"], case["n_dual"])).to(DEV)
    if kind == "net":
        with torch.no_grad():
            return _net64(params, x, case["Q"], case["n_dual"])[0]
    out, leaves = _net64(params, x, case["Q"], case["n_dual"])
    loss = ((out - t.double()) ** 2).mean()
    loss.backward()
    grads = torch.cat([g.grad.reshape(-1) for pair in leaves for g in pair])
    return dict(loss=np.float64(loss.item()), grads=grads)
