"""The measured workloads: what a user of the library has it do, through its public calls.

Each kind of case is one use of the C ABI's Python binding; ``listed()`` holds one or two sizes of each and
``draw()`` gives others of the same ranges.  ``exact()`` restates the methods in 64 bits with plain torch.
"""
import math
import os

import numpy as np
import torch

import paper_1610_00835_gb300 as P

DEV = "cuda"
F64 = torch.float64
STEPS = 64  # midpoints of the optical-depth march, the library's default


def listed():
    return [
        # The smallest call: one operator apply on a small, odd 2D grid, as a parameter study or a unit test makes it.
        {"name": "apply_47", "kind": "apply", "dim": 2, "n": 47},
        # The homogeneous unit square at 32^2 in FP64 with the closed-form optical depth, solved to 1e-10.
        {"name": "fp64_32", "kind": "fp64", "n": 32, "mu_s": 1.0, "mu_a": 0.1, "tau": "closed", "precond": "none"},
        # The paper's preconditioning experiment (constant mu_s, mu_a = 0.2) at h = 1/128 in FP64, diffusion preconditioner.
        {"name": "fp64_128_diffusion", "kind": "fp64", "n": 128, "mu_s": 40.0, "mu_a": 0.2, "tau": "closed", "precond": "diffusion"},
        # The heterogeneous 128^2 medium, plain: FP64 GMRES to 1e-6, every kernel entry generated on the fly.
        {"name": "solve_128", "kind": "solve", "n": 128},
        # The same medium with the stored symmetric operator: assembly and solve, as for each new medium.
        {"name": "blocks_128", "kind": "blocks", "n": 128},
        # The 32^3 medium: K assembled and one solve to 1e-6.
        {"name": "solve3_32", "kind": "solve3", "n": 32},
        # Step two on the 32^3 medium: the scattering-free sweep on 128 directions.
        {"name": "sweep3_32", "kind": "sweep", "dim": 3, "n": 32, "dirs": 128},
        # 64 sources on one 128^2 medium, solved in lockstep on the tensor-core product (K assembled before).
        {"name": "sources_128_64", "kind": "sources", "n": 128, "count": 64},
        # One source on each of several media of uneven sizes, in one batch (the largest grids keep sigma_t in global memory).
        {"name": "batch_uneven", "kind": "batch", "sizes": "64,97,128,160,200,243"},
        # The learned preconditioner's network on the residuals of 64 sources: BF16 inference.
        {"name": "forward_128_64", "kind": "forward", "n": 128, "batch": 64},
        # Its training: loss and gradient of a batch of 16 images (the optimiser adds one small kernel to this).
        {"name": "grad_128_16", "kind": "grad", "n": 128, "batch": 16},
        # The fast multipole operator of order 6 at 512^2, where dense forms no longer fit: one solve.
        {"name": "fmm_512", "kind": "fmm", "n": 512, "order": 6},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["apply", "fp64", "solve", "blocks", "solve3", "sweep", "sources", "batch", "forward", "grad", "fmm"])
    c = {"kind": kind}
    if kind == "apply":
        c["dim"] = rng.choice([2, 2, 3])
        c["n"] = _log(rng, 12, 243) if c["dim"] == 2 else rng.randint(6, 32)
    elif kind == "fp64":
        c["tau"] = rng.choice(["closed", "closed", "closed", "march"])
        c["n"] = _log(rng, 12, 128) if c["tau"] == "closed" else _log(rng, 12, 40)
        c["mu_s"], c["mu_a"] = round(math.exp(rng.uniform(0.0, math.log(40.0))), 3), round(rng.uniform(0.1, 0.5), 3)
        c["precond"] = rng.choice(["none", "fft", "diffusion"]) if c["tau"] == "closed" else "none"
        if c["precond"] == "none":
            c["mu_s"] = min(c["mu_s"], 8.0)
    elif kind in ("solve", "blocks"):
        c["n"] = _log(rng, 24, 150)
    elif kind == "solve3":
        c["n"] = rng.randint(8, 31)
    elif kind == "sweep":
        c["dim"] = rng.choice([2, 3])
        c["n"], c["dirs"] = (_log(rng, 16, 160), _log(rng, 8, 128)) if c["dim"] == 2 else (rng.randint(10, 32), _log(rng, 8, 128))
    elif kind == "sources":
        c["n"], c["count"] = _log(rng, 24, 128), _log(rng, 2, 128)
    elif kind == "batch":
        ns, left = [], 6e9  # pairs, about the listed batch's
        for _ in range(rng.randint(2, 6)):
            ns.append(_log(rng, 24, max(24, min(243, int(left ** 0.25)))))
            left -= ns[-1] ** 4
        c["sizes"] = ",".join(str(v) for v in ns)
    elif kind == "forward":
        c["n"] = 8 * _log(rng, 4, 32)
        c["batch"] = max(1, min(_log(rng, 1, 64), 64 * 128 * 128 // c["n"] ** 2))
    elif kind == "grad":
        c["n"] = 8 * _log(rng, 4, 16)
        c["batch"] = _log(rng, 2, 16)
    else:
        c["n"], c["order"] = rng.randint(8, 15) << rng.randint(2, 5), rng.choice([4, 6])
    return c


# ---- inputs: the media and sources of the paper's unit-square tests, drawn from the seed

def _centres(dim, n):
    c = (torch.arange(n, dtype=F64, device=DEV) + 0.5) / n
    return torch.stack([a.reshape(-1) for a in torch.meshgrid(*[c] * dim, indexing="ij")][::-1], dim=1)


def _bumps(rng, dim, n, count, amp, base=0.0, width=(0.05, 0.2), centre=(0.2, 0.8)):
    """base + the sum of `count` Gaussian bumps at the cell centres."""
    x = _centres(dim, n)
    v = torch.full((n ** dim,), base, dtype=F64, device=DEV)
    for _ in range(count):
        a, w, c = rng.uniform(*amp), rng.uniform(*width), rng.uniform(*centre, size=dim)
        v += a * torch.exp(-((x - torch.as_tensor(c, device=DEV)) ** 2).sum(1) / (2 * w * w))
    return v


def _source(rng, dim, n):
    return _bumps(rng, dim, n, 2, (0.5, 1.0), width=(0.08, 0.2), centre=(0.3, 0.7))


def _medium(rng, dim, n):
    """sigma_t = 1 + bumps of amplitude 0.5..3 and sigma_s = 0.9 (2D) or 0.8 (3D) sigma_t."""
    st = _bumps(rng, dim, n, 4 if dim == 2 else 6, (0.5, 3.0), base=1.0)
    return st, (0.9 if dim == 2 else 0.8) * st


def _inputs(case, seed):
    """The medium and the source(s) of a case, FP64 on the GPU."""
    rng = np.random.default_rng([seed, 7])
    kind, dim = case["kind"], 3 if case["kind"] == "solve3" else case.get("dim", 2)
    if kind == "batch":
        d = [_medium(rng, 2, int(n)) + (_source(rng, 2, int(n)),) for n in case["sizes"].split(",")]
        return {"media": d}
    n = case["n"]
    if kind == "fp64" and case["tau"] == "closed":
        st = torch.full((n * n,), case["mu_s"] + case["mu_a"], dtype=F64, device=DEV)
        ss = torch.full((n * n,), case["mu_s"], dtype=F64, device=DEV)
    else:
        st, ss = _medium(rng, dim, n)
    if kind == "sources":
        f = torch.stack([_source(rng, 2, n) for _ in range(case["count"])])
    else:
        f = _source(rng, dim, n)
    d = {"dim": dim, "n": n, "st": st, "ss": ss, "f": f}
    if kind == "sweep":
        # an angular density of the solution's size, and the directions (Fibonacci points, or equal angles)
        m = torch.arange(case["dirs"], dtype=F64, device=DEV) + 0.5
        d["U"] = 0.2 * _source(rng, dim, n) + 0.05
        if dim == 2:
            t = 2 * math.pi * m / case["dirs"]
            v = torch.stack([torch.cos(t), torch.sin(t)], 1)
        else:
            z = 1 - 2 * m / case["dirs"]
            t = (m - 0.5) * math.pi * (3 - math.sqrt(5.0))
            s = torch.sqrt(1 - z * z)
            v = torch.stack([s * torch.cos(t), s * torch.sin(t), z], 1)
        d["dirs"] = v.float().contiguous()
    return d


LEVELS, CHANNELS = 4, 32
WEIGHTS = os.path.join(os.path.dirname(os.path.abspath(P.__file__)), "data", "unet_l4_c32.bin")


def _net_inputs(case, seed):
    """Coefficients over 5 and right-hand sides of unit mean square, [B, 3, n, n], and targets [B, n, n]."""
    rng = np.random.default_rng([seed, 11])
    n, B = case["n"], case["batch"]
    x = torch.empty(B, 3, n * n, dtype=torch.float32, device=DEV)
    t = torch.empty(B, n * n, dtype=torch.float32, device=DEV)
    for b in range(B):
        s = math.exp(rng.uniform(math.log(4.0), math.log(16.0)))
        ss = s * _bumps(rng, 2, n, 2, (0.2, 1.0), base=1.0)
        v = _bumps(rng, 2, n, 4, (-1.0, 1.0), width=(0.03, 0.3), centre=(0.1, 0.9))
        x[b, 0], x[b, 1], x[b, 2] = (ss + 0.3) / 5, ss / 5, v / v.square().mean().sqrt()
        t[b] = _bumps(rng, 2, n, 3, (-1.0, 1.0), width=(0.1, 0.3))
    return x.view(B, 3, n, n), t.view(B, n, n)


def _layers():
    """(outputs, inputs, kernel) of every convolution in parameter order."""
    enc = [(CHANNELS, 3 if k == 0 else CHANNELS, 3) for k in range(2 * LEVELS)]
    dec = [(CHANNELS, CHANNELS * (2 if k % 2 == 0 else 1), 3) for k in range(2 * (LEVELS - 1))]
    return enc + dec + [(1, CHANNELS, 1)]


def _init_params(seed):
    """A network at the start of its training: normal weights scaled to the fan-in, small biases."""
    rng = np.random.default_rng([seed, 13])
    out = []
    for co, ci, k in _layers():
        out += [rng.normal(0.0, math.sqrt(2.0 / (ci * k * k)), co * ci * k * k), rng.normal(0.0, 0.01, co)]
    return np.concatenate(out).astype(np.float32)


# ---- the cases through the library's entry points

def prepare(case, seed):
    kind = case["kind"]
    if kind in ("forward", "grad"):
        net = P.vie_unet_create(LEVELS, CHANNELS)
        x, t = _net_inputs(case, seed)
        if kind == "forward":
            P.vie_unet_load(net, WEIGHTS)
        else:
            P.vie_unet_set_params(net, _init_params(seed))
        return {"case": case, "net": net, "x": x, "t": t, "o": torch.empty_like(t)}
    d = _inputs(case, seed)
    if kind == "batch":
        ns = [int(n) for n in case["sizes"].split(",")]
        b = P.vie_batch_create(ns, [m[0].cpu().numpy() for m in d["media"]], [m[1].cpu().numpy() for m in d["media"]])
        g = torch.cat([m[2] for m in d["media"]])
        return {"case": case, "b": b, "g": g, "y": torch.empty_like(g)}
    opts = {}
    if kind == "fp64":
        opts = {"precision": P.VIE_PREC_FP64, "tau_mode": P.VIE_TAU_CLOSED if case["tau"] == "closed" else P.VIE_TAU_MARCH}
    h = P.vie_create(d["dim"], d["n"], d["st"].cpu().numpy(), d["ss"].cpu().numpy(), **opts)
    s = {"case": case, "h": h, "f": d["f"], "U": torch.zeros_like(d["f"])}
    if kind == "fp64" and case["precond"] == "fft":
        P.vie_set_fft_preconditioner(h)
    if kind == "fp64" and case["precond"] == "diffusion":
        P.vie_set_diffusion_preconditioner(h)
    if kind == "sources":
        P.vie_assemble(h, P.VIE_OPERATOR_BF16X3)
    if kind == "fmm":
        P.vie_assemble_fmm(h, case["order"])
    if kind == "sweep":
        s.update(U=d["U"], dirs=d["dirs"], Phi=torch.empty(case["dirs"], d["n"] ** d["dim"], dtype=torch.float32, device=DEV))
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "apply":
        P.vie_apply(s["h"], P.VIE_OP_K_SIGMA_S, s["f"], s["U"])
        return s["U"]
    if kind == "fp64":
        P.vie_solve_gmres(s["h"], s["f"], s["U"], rtol=1e-10)
        return s["U"]
    if kind in ("solve", "fmm"):
        P.vie_solve_gmres(s["h"], s["f"], s["U"], rtol=1e-6)
        return s["U"]
    if kind in ("blocks", "solve3"):
        P.vie_assemble(s["h"], P.VIE_OPERATOR_SYM32 if kind == "blocks" else P.VIE_OPERATOR_FP32)
        P.vie_solve_gmres(s["h"], s["f"], s["U"], rtol=1e-6)
        return s["U"]
    if kind == "sweep":
        P.ert_sweep(s["h"], s["U"], s["f"], s["dirs"], s["Phi"])
        return s["Phi"]
    if kind == "sources":
        P.vie_solve_gmres(s["h"], s["f"], s["U"], rtol=1e-6, nrhs=case["count"])
        return s["U"]
    if kind == "batch":
        P.vie_batch_apply(s["b"], P.VIE_OP_K_SIGMA_S, s["g"], s["y"])
        o = s["b"].offsets
        return [s["y"][o[i]:o[i + 1]] for i in range(len(o) - 1)]
    if kind == "forward":
        P.vie_unet_forward(s["net"], s["x"], s["o"], case["batch"], case["n"], use_bf16=True)
        return s["o"]
    loss, grad = P.vie_unet_loss_grad(s["net"], s["x"], s["t"], case["batch"], case["n"])
    return {"loss": loss, "grad": grad}


# ---- the work of one pass

def _pair_flops(dim, n):
    """Every unordered pair's optical depth: a multiply-add for each cell its midpoints touch, and the entry itself."""
    cells = min(1.11 * n, 200.0) if dim == 2 else 3.44 * n
    return 0.5 * n ** (2 * dim) * (2 * cells + 10)


def work(case):
    kind, n = case["kind"], case.get("n", 0)
    if kind == "apply":
        return {"bytes": 32 * n ** case["dim"], "flops": _pair_flops(case["dim"], n)}
    if kind == "fp64":  # about ten operator products
        per = 2.0 * n ** 4 if case["tau"] == "closed" else 2 * _pair_flops(2, n)
        return {"bytes": 32 * n * n, "flops": 10 * per}
    if kind == "solve":  # about nine operator products
        return {"bytes": 32 * n * n, "flops": 9 * _pair_flops(2, n)}
    if kind == "blocks":  # the entries once, written and read by about nine products
        return {"bytes": 10 * 2.0 * n ** 4, "flops": _pair_flops(2, n) + 18.0 * n ** 4}
    if kind == "solve3":  # K written once and read by about eight products
        return {"bytes": 9 * 4.0 * n ** 6, "flops": _pair_flops(3, n) + 16.0 * n ** 6}
    if kind == "sweep":
        d = case["dim"]
        rays, steps = case["dirs"] * n ** d, 0.9 * n
        return {"bytes": 4 * rays + 32 * n ** d, "flops": rays * steps * (25 if d == 2 else 45)}
    if kind == "sources":  # K (four bytes an entry) read by about nine products
        return {"bytes": 9 * 4.0 * n ** 4 + 16 * case["count"] * n * n, "flops": 9 * 2.0 * n ** 4 * case["count"]}
    if kind == "batch":
        ns = [int(v) for v in case["sizes"].split(",")]
        return {"bytes": sum(32 * v * v for v in ns), "flops": sum(_pair_flops(2, v) for v in ns)}
    if kind in ("forward", "grad"):
        ls = _layers()
        size = [n >> (k // 2) for k in range(2 * LEVELS)] + [n >> (LEVELS - 2 - k // 2) for k in range(2 * (LEVELS - 1))] + [n]
        macs = case["batch"] * sum(co * ci * k * k * m * m for (co, ci, k), m in zip(ls, size))
        par = sum(co * ci * k * k + co for co, ci, k in ls)
        return {"bytes": 16 * case["batch"] * n * n + (4 if kind == "forward" else 8) * par, "flops": (2 if kind == "forward" else 6) * macs}
    b, L = _leaves(n)
    vals = 9 * b * b * n * n + 27 * case["order"] ** 4 * sum(4 ** l for l in range(2, L + 1))
    return {"bytes": 9 * 4.0 * vals, "flops": 9 * 2.0 * vals}


# ---- 64-bit values by plain torch

def _pad(dim, n, st):
    return st.view([1, 1] + [n] * dim)


def _kernel(sig, dim, n, a, d, sigma_c=None):
    """h^d e^{-tau} / (|S^{d-1}| r^{d-1}) from lattice points a to a + d ([pairs, dim]); tau by the march, or sigma_c r."""
    r = d.square().sum(1).sqrt()
    h = 1.0 / n
    if sigma_c is not None:
        tau = sigma_c * h * r
    else:
        tau = torch.zeros_like(r)
        scale = 2.0 / max(n - 1, 1)
        a0, d0 = a * scale - 1, d * scale
        for i in range(STEPS):
            u = torch.add(a0, d0, alpha=(i + 0.5) / STEPS).view([1] * dim + [-1, dim])
            tau += torch.nn.functional.grid_sample(sig, u, mode="bilinear", padding_mode="border", align_corners=True).view(-1)
        tau *= h * r / STEPS
    return h * torch.exp(-tau) / (2 * math.pi * r if dim == 2 else 4 * math.pi * r * r)


def _gauss(m):
    x, w = np.polynomial.legendre.leggauss(m)
    return torch.as_tensor(x, device=DEV), torch.as_tensor(w, device=DEV)


def _self_cell(dim, n, st):
    """The integral of e^{-s|z|} / (|S^{d-1}| |z|^{d-1}) over the own cell, in polar form."""
    x, w = _gauss(48)
    a, q, s = 0.5 / n, 0.25 * math.pi, st[:, None]
    th = 0.5 * q * (x + 1)
    if dim == 2:
        R = a / torch.cos(th)
        return 8 * (0.5 * q * w * -torch.expm1(-s * R) / s).sum(1) / (2 * math.pi)
    rmax = a * torch.sqrt(1 + 1 / torch.cos(th) ** 2)
    rho = (a + 0.5 * (rmax - a)[:, None] * (x + 1)).reshape(-1)
    ww = (0.5 * q * w[:, None] * 0.5 * (rmax - a)[:, None] * w * a).reshape(-1) / rho ** 2
    out = torch.empty_like(st)
    for k in range(0, len(st), 4096):
        sk = st[k:k + 4096, None]
        out[k:k + 4096] = 48 * (ww * -torch.expm1(-sk * rho) / sk).sum(1) / (4 * math.pi)
    return out


def _lattice(dim, n):
    j = torch.arange(n ** dim, device=DEV)
    return torch.stack([(j // n ** k) % n for k in range(dim)], 1).to(F64)


def _dense(dim, n, st, sigma_c=None, chunk=1 << 22):
    """A in 64 bits: every pair once, mirrored, and the self cells on the diagonal."""
    N = n ** dim
    u, sig = _lattice(dim, n), _pad(dim, n, st)
    A = torch.zeros(N, N, dtype=F64, device=DEV)
    rows = max(1, chunk // N)
    for j in range(0, N, rows):
        t = u[j:j + rows]
        k = min(j + rows, N)
        d = (u[None, j:] - t[:, None]).reshape(-1, dim)  # sources from the block's first target on
        d[(d == 0).all(1)] = 1.0  # the diagonal is set below
        v = _kernel(sig, dim, n, t[:, None].expand(-1, N - j, -1).reshape(-1, dim), d, sigma_c).view(k - j, N - j)
        A[j:k, j:] = v
        A[k:, j:k] = v[:, k - j:].T
    A.diagonal().copy_(_self_cell(dim, n, st))
    return A


def _gmres(apply, b, tol=1e-14, m=150):
    """x with apply(x) = b, full GMRES with twice-applied orthogonalisation."""
    x = torch.zeros_like(b)
    for _ in range(3):
        r = b - apply(x)
        beta = r.norm()
        if beta <= tol * b.norm():
            break
        V, H = [r / beta], torch.zeros(m + 1, m, dtype=F64, device=DEV)
        for k in range(m):
            w, B = apply(V[k]), torch.stack(V)
            for _ in range(2):
                c = B @ w
                w = w - B.T @ c
                H[:k + 1, k] += c
            H[k + 1, k] = w.norm()
            V.append(w / H[k + 1, k])
            if k % 4 == 3 or k == m - 1:
                e = torch.zeros(k + 2, dtype=F64, device=DEV)
                e[0] = beta
                Q, R = torch.linalg.qr(H[:k + 2, :k + 1])
                c = Q.T @ e
                if (e - Q @ c).norm() <= tol * b.norm() or H[k + 1, k] <= 1e-14 * beta:
                    break
        x = x + torch.stack(V[:k + 1]).T @ torch.linalg.solve_triangular(R, c[:, None], upper=True)[:, 0]
    return x


def _leaves(n):
    """Leaf size and level of the quadtree: halved while even and the leaves keep 8 cells a side."""
    L = 0
    while n % (2 << L) == 0 and n // (2 << L) >= 8:
        L += 1
    return n >> L, L


def _cheb(p, x, z):
    """S_p(x, z) = 1/p + 2/p sum_k T_k(x) T_k(z), [points, nodes]."""
    k = torch.arange(1, p, dtype=F64, device=DEV)
    tx, tz = torch.cos(k * torch.acos(x.clamp(-1, 1))[:, None]), torch.cos(k * torch.acos(z)[:, None])
    return 1.0 / p + 2.0 / p * tx @ tz.T


def _fmm(n, p, st):
    """v -> A v by the interpolation-based FMM with its near entries and node values in 64 bits."""
    b, L = _leaves(n)
    sig = _pad(2, n, st)
    z = torch.cos((2 * torch.arange(p, dtype=F64, device=DEV) + 1) * math.pi / (2 * p))

    def values(tgt, src, keep):
        """Kernel blocks [boxes, sources, targets] between node sets in lattice coordinates."""
        out = torch.zeros(len(tgt), src.shape[1], tgt.shape[1], dtype=F64, device=DEV)
        for i in range(0, len(tgt), max(1, (1 << 22) // out[0].numel())):
            s = slice(i, i + max(1, (1 << 22) // out[0].numel()))
            d = (src[s][:, :, None] - tgt[s][:, None]).reshape(-1, 2)
            a = tgt[s][:, None].expand(-1, src.shape[1], -1, -1).reshape(-1, 2)
            same = (d == 0).all(1)
            d[same] = 1.0
            v = _kernel(sig, 2, n, a, d)
            v[same] = 0.0
            out[s] = v.view(out[s].shape) * keep[s, None, None]
        return out

    def grid(level):
        nb = 1 << level
        i = torch.arange(nb * nb, device=DEV)
        return nb, torch.stack([i % nb, i // nb], 1)

    def neighbours(level, offs):
        """Index of the box at an offset (per box), and whether it exists."""
        nb, B = grid(level)
        c = B + offs
        ok = ((c >= 0) & (c < nb)).all(1)
        c = c.clamp(0, nb - 1)
        return c[:, 1] * nb + c[:, 0], ok.to(F64)

    k = torch.arange(b * b, device=DEV)
    cell = torch.stack([k % b, k // b], 1)
    nb, B = grid(L)
    cells = (B[:, None] * b + cell[None]).to(F64)
    index = ((B[:, None, 1] * b + cell[None, :, 1]) * n + B[:, None, 0] * b + cell[None, :, 0])
    near = []
    for oy in (-1, 0, 1):
        for ox in (-1, 0, 1):
            nbr, ok = neighbours(L, torch.tensor([ox, oy], device=DEV).expand(len(B), 2))
            near.append((nbr, values(cells, cells[nbr], ok)))
    m = torch.arange(p * p, device=DEV)
    node = torch.stack([z[m % p], z[m // p]], 1)
    far = []
    for level in range(2, L + 1):
        nb, B = grid(level)
        w = n / nb
        pts = (B[:, None] * w + 0.5 * w * (node[None] + 1) - 0.5).to(F64)
        par = B % 2
        offs = [(x, y) for y in range(-3, 4) for x in range(-3, 4) if max(abs(x), abs(y)) > 1]
        lev = []
        for o in offs:
            o = torch.tensor(o, device=DEV)
            nbr, ok = neighbours(level, o.expand(len(B), 2))
            ok = ok * ((o >= -2 - par) & (o <= 3 - par)).all(1)
            at = ok.nonzero()[:, 0]
            if len(at):
                lev.append((at, nbr[at], values(pts[at], pts[nbr[at]], ok[at])))
        far.append(lev)
    c1 = 2 * (torch.arange(b, dtype=F64, device=DEV) + 0.5) / b - 1
    S1 = _cheb(p, c1, z)
    Pm = (S1[k // b][:, :, None] * S1[k % b][:, None, :]).reshape(b * b, p * p)  # [cell, node]
    S2 = [_cheb(p, -1.0 + q + 0.5 * (z + 1), z) for q in (0, 1)]
    C = [torch.einsum("ij,kl->ikjl", S2[q // 2], S2[q % 2]).reshape(p * p, p * p) for q in range(4)]  # [child node, node]
    diag = _self_cell(2, n, st)

    def apply(v):
        s = v[index]
        W = {L: s @ Pm}
        for level in range(L - 1, 1, -1):
            nb, B = grid(level)
            W[level] = sum(W[level + 1][(2 * B[:, 1] + q // 2) * 2 * nb + 2 * B[:, 0] + q % 2] @ C[q] for q in range(4))
        loc = None
        for level in range(2, L + 1):
            nb, B = grid(level)
            new = torch.zeros_like(W[level])
            for at, nbr, K in far[level - 2]:
                new[at] += torch.einsum("bst,bs->bt", K, W[level][nbr])
            if loc is not None:
                up, q = (B[:, 1] // 2) * (nb // 2) + B[:, 0] // 2, B[:, 0] % 2 + 2 * (B[:, 1] % 2)
                for i in range(4):
                    at = (q == i).nonzero()[:, 0]
                    new[at] += loc[up[at]] @ C[i].T
            loc = new
        out = loc @ Pm.T
        for nbr, K in near:
            out += torch.einsum("bst,bs->bt", K, s[nbr])
        y = diag * v
        y[index.reshape(-1)] += out.reshape(-1)
        return y

    return apply


def _net(params, x):
    """The network in 64 bits: parameters as one vector, x [B, 3, n, n]."""
    F, at, ws = torch.nn.functional, 0, []
    for co, ci, k in _layers():
        ws.append((params[at:at + co * ci * k * k].view(co, ci, k, k), params[at + co * ci * k * k:at + co * ci * k * k + co]))
        at += co * ci * k * k + co
    conv = lambda v, l: F.relu(F.conv2d(v, ws[l][0], ws[l][1], padding=1))  # noqa: E731
    e = []
    for l in range(LEVELS):
        x = conv(conv(x if l == 0 else F.avg_pool2d(x, 2), 2 * l), 2 * l + 1)
        e.append(x)
    for k, l in enumerate(range(LEVELS - 2, -1, -1)):
        x = torch.cat([F.interpolate(x, scale_factor=2, mode="nearest"), e[l]], 1)
        x = conv(conv(x, 2 * LEVELS + 2 * k), 2 * LEVELS + 2 * k + 1)
    return F.conv2d(x, *ws[-1])[:, 0]


def _sweep(d):
    """Backward characteristics with the step midpoints frozen, every ray of a direction at once."""
    dim, n = d["dim"], d["n"]
    x = _centres(dim, n)
    sig, q = _pad(dim, n, d["st"]), _pad(dim, n, d["ss"] * d["U"] + d["f"])
    out = []
    for v in d["dirs"].to(F64):
        L = torch.full((len(x),), 2.0, dtype=F64, device=DEV)
        for k in range(dim):
            if v[k] > 0:
                L = torch.minimum(L, x[:, k] / v[k])
            elif v[k] < 0:
                L = torch.minimum(L, (1 - x[:, k]) / -v[k])
        ns = torch.ceil(L * (2.0 * n) - 1e-6).clamp(min=1)
        dl = L / ns
        tau, acc = torch.zeros_like(L), torch.zeros_like(L)
        scale = 2.0 / max(n - 1, 1)
        u0, du = (x * n - 0.5) * scale - 1, -dl[:, None] * v * n * scale
        for s in range(int(ns.max())):
            u = torch.add(u0, du, alpha=s + 0.5).view([1] * dim + [-1, dim])
            sg, qq = (torch.nn.functional.grid_sample(f, u, mode="bilinear", padding_mode="border", align_corners=True).view(-1)
                      for f in (sig, q))
            on = s < ns
            acc = torch.where(on, acc + torch.exp(-tau) * qq * -torch.expm1(-sg * dl) / sg, acc)
            tau = torch.where(on, tau + sg * dl, tau)
        out.append(acc)
    return torch.stack(out)


def exact(case, seed):
    kind = case["kind"]
    if kind in ("forward", "grad"):
        x, t = _net_inputs(case, seed)
        if kind == "forward":
            raw = np.fromfile(WEIGHTS, dtype=np.uint8)
            count = int(raw[16:24].view(np.int64)[0])
            par = torch.as_tensor(raw[24:24 + 4 * count].view(np.float32).astype(np.float64), device=DEV)
            return torch.cat([_net(par, v) for v in x.double().split(8)])
        par = torch.as_tensor(_init_params(seed).astype(np.float64), device=DEV).requires_grad_()
        loss = sum((_net(par, v) - w).square().sum() for v, w in zip(x.double().split(8), t.double().split(8))) / t.numel()
        loss.backward()
        return {"loss": float(loss), "grad": par.grad.cpu().numpy()}
    d = _inputs(case, seed)
    if kind == "sweep":
        return _sweep(d)
    if kind == "batch":  # the media whose dense operator takes seconds at most
        return [_dense(2, math.isqrt(len(m[0])), m[0]) @ (m[1] * m[2]) if len(m[0]) <= 17000 else None for m in d["media"]]
    if kind == "apply" and d["n"] ** d["dim"] > 33000:
        return None
    if kind == "fmm":
        A = _fmm(d["n"], case["order"], d["st"])
    else:
        M = _dense(d["dim"], d["n"], d["st"], float(d["st"][0]) if case.get("tau") == "closed" else None)
        A = lambda v: M @ v  # noqa: E731
    if kind == "apply":
        return A(d["ss"] * d["f"])
    one = lambda f: _gmres(lambda v: v - A(d["ss"] * v), A(f))  # noqa: E731
    return torch.stack([one(f) for f in d["f"]]) if kind == "sources" else one(d["f"])
