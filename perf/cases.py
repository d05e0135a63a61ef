"""Performance cases: what a user of the library has it do, through its public
entry points, with inputs made from a seed and the same results in 64 bits by
plain torch.

A case of kind "level" is one batch of samples of one level
(``Context.run_level_dev``: moment sums and per-sample outputs), "batch" the
samples of all levels of a hierarchy at once (``Context.run_batch_dev``, what
every round of Algorithm 1 runs), "learned" one gradient of the learned level's
network (``Context.surrogate_loss_grad``, what a training step runs).

Workloads, levels, step ratios, particle numbers and observables are those of
``paper_2311_08872_gb300.workloads``.  On the finest grids the horizon T is cut:
a pass there is the same step repeated, and the full horizons take seconds.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2311_08872_gb300 import mlmc_dk, workloads


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # Algorithm 1's default pilot on the coarsest level: the smallest call, launches and latency count
        dict(name="pilot16", kind="level", workload="mlmc16_256", level=0, mc=False, count=256, T=0.02),
        # plain single-level Monte Carlo, 1000 samples on 32^2 (the fine path alone)
        dict(name="mc32", kind="level", workload="mc32", level=0, mc=True, count=1000, T=0.01),
        # a middle level of the five-level hierarchy: fine path and coupled coarse path, one CTA per sample
        dict(name="coupled64", kind="level", workload="mlmc16_256", level=2, mc=False, count=1151, T=0.02),
        # its finest level, where most of the hierarchy's time goes: a sample over a thread-block cluster
        dict(name="coupled256", kind="level", workload="mlmc16_256", level=4, mc=False, count=59, T=0.002),
        # finest level of the low-density hierarchy: grids beyond the registers, densities near zero
        dict(name="stream512", kind="level", workload="lowdens32_512", level=4, mc=False, count=7, T=7.8e-4),
        # finest level of the largest hierarchy: four observables and their ten products
        dict(name="stream1024", kind="level", workload="large32_1024", level=5, mc=False, count=5, T=9.7e-5),
        # finest level of the regular setting on (0, 2 pi)^2 at N = 2e9: fluctuation state about the noise-free path
        dict(name="fluct128", kind="level", workload="paper_reg", level=5, mc=False, count=311, T=1.024),
        # Crank-Nicolson time step: an implicit solve per step
        dict(name="theta128", kind="level", workload="theta16_128", level=3, mc=False, count=75, T=0.02),
        # Fourier coupling, the finest level of the three-level hierarchy
        dict(name="fourier54", kind="level", workload="fourier6_54", level=2, mc=False, count=607, T=0.02),
        # Fourier coupling, the fourth level
        dict(name="fourier162", kind="level", workload="fourier6_162", level=3, mc=False, count=45, T=0.005),
        # all levels of the five-level hierarchy at once, counts in the proportions of its allocation: the whole call
        dict(name="batch16_256", kind="batch", workload="mlmc16_256", scale=16, T=0.004),
        # one training step's gradient of the learned level's network at the training batch size
        dict(name="learned1024", kind="learned", workload="mlmc16_256", batch=1024),
    ]


# per (workload, levels): largest cell-steps of a drawn case, and horizons; the
# implicit and Fourier levels cost more per cell-step, so their cap is lower
_DRAWN = [
    ("mlmc16_256", (0, 1, 2, 3, 4), 5e9, (0.001, 0.02)),
    ("mlmc16_256_sym", (0, 1, 2, 3), 4e9, (0.001, 0.02)),
    ("mc32", (0,), 2e9, (0.004, 0.01)),
    ("lowdens32_512", (1, 2, 3, 4), 4e9, (1e-4, 2e-3)),
    ("large32_1024", (2, 4, 5), 4e9, (9.7e-5, 1.9e-4)),
    ("paper_reg", (1, 2, 3, 4, 5), 4e9, (1.024, 1.024)),
    ("paper_irreg", (3, 4, 5), 4e9, (1.024, 1.024)),
    ("theta16_128", (1, 2, 3), 4e8, (0.005, 0.02)),
    ("implicit16_64", (0, 1, 2), 4e8, (0.01, 0.02)),
    ("fourier6_162", (1, 2, 3), 1e9, (0.003, 0.02)),
    ("paper_reg_fourier", (1, 2), 1e9, (1.024, 1.024)),
]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    u = rng.random()
    if u < 0.08:
        return dict(kind="learned", workload="mlmc16_256", batch=int(_log_uniform(rng, 64, 4096)))
    if u < 0.16:
        return dict(kind="batch", workload="mlmc16_256", scale=int(_log_uniform(rng, 20, 200)),
                    T=_log_uniform(rng, 0.001, 0.004))
    name, levels, cap, (t_lo, t_hi) = rng.choice(_DRAWN)
    level = rng.choice(levels)
    T = _log_uniform(rng, t_lo, t_hi) if t_hi > t_lo else t_hi
    case = dict(kind="level", workload=name, level=level, mc=name == "mc32" or rng.random() < 0.2, count=1, T=T)
    wl = _workload(case)
    n, M, *_ = _grid(wl, level)
    # at least a few samples, at most what the cap on cell-steps and 20000 samples allow
    most = max(3.0, min(20000.0, cap / (float(n) * n * M)))
    case["count"] = int(_log_uniform(rng, min(3.0, most), most + 0.999))
    return case


# ------------------------------------------------------------------ a pass
def _workload(case):
    wl = workloads.get(case["workload"])
    if case["kind"] == "level":
        return wl.with_(T=case["T"], L_max=case["level"])
    if case["kind"] == "batch":
        return wl.with_(T=case["T"])
    return wl.with_(L_max=0)


def _counts(case):
    return [max(2, a // case["scale"]) for a in workloads.get(case["workload"]).alloc]


def prepare(case, seed):
    wl = _workload(case)
    ctx = mlmc_dk.Context.from_workload(wl)
    state = {"case": case, "ctx": ctx, "seed": _philox_seed(seed)}
    if case["kind"] == "level":
        state["sums"] = torch.zeros(mlmc_dk.sums_len(ctx.n_quant), dtype=torch.float64, device="cuda")
        state["samples"] = torch.zeros(case["count"], mlmc_dk.sample_stride(ctx.n_obs), dtype=torch.float64,
                                       device="cuda")
    elif case["kind"] == "batch":
        state["counts"] = _counts(case)
        state["sums"] = torch.zeros(ctx.L_max + 1, mlmc_dk.sums_len(ctx.n_quant), dtype=torch.float64, device="cuda")
    else:
        theta, state["X"], state["T"] = _network(case, seed)
        ctx.surrogate_init(0)
        ctx.surrogate_params(theta)
    return state


def run(state):
    case, ctx = state["case"], state["ctx"]
    if case["kind"] == "learned":
        loss, grad = ctx.surrogate_loss_grad(state["X"], state["T"])
        return {"loss": loss, "grad": grad}
    stream = torch.cuda.current_stream().cuda_stream
    sums = state["sums"]
    if case["kind"] == "batch":
        ctx.run_batch_dev(state["counts"], 0, state["seed"], sums.data_ptr(), stream)
        return {"sums": sums}
    samples = state["samples"]
    ctx.run_level_dev(case["level"], int(case["mc"]), 0, case["count"], state["seed"], sums.data_ptr(),
                      samples.data_ptr(), stream)
    return {"sums": sums, "samples": samples}


# ------------------------------------------------------------------ work
def _grid(wl, level):
    """(n, M, h, tau) of a level: M_0 = ceil(T / (mu h_0^2)) steps on level 0,
    tau falling with the square of h."""
    h0 = wl.length / wl.n0
    M0 = wl.M0 if wl.M0 > 0 else max(1, math.ceil(wl.T / (wl.mu * h0 * h0) * (1.0 - 1e-9)))
    r = wl.ratio ** level
    return wl.n0 * r, M0 * r * r, h0 / r, wl.T / M0 / (r * r)


def _level_work(wl, level, coupled, count, samples):
    n, M, _, _ = _grid(wl, level)
    r = wl.ratio
    K = len(wl.observables)
    Q = K * (K + 1) // 2 if wl.products else K
    # per cell and step: half a Philox call (30), a Box-Muller pair (14), the
    # amplitude and the two transfers (12), two edge fluxes (6) and the update (8)
    fine, coarse = 70.0, 26.0
    if wl.b0 > 0:
        # the implicit solve as a transform pair per step
        fine += 10.0 * math.log2(n)
        coarse += 10.0 * math.log2(n)
    flops = fine * n * n * M * count
    cells = float(n * n)
    if coupled:
        fine_sum = 2.0 * n * n * M * count   # the coupled normals
        flops += fine_sum + coarse * (n // r) ** 2 * (M // (r * r)) * count
        if wl.coupling == 1:
            # a transform of the two summed components per coarse step
            flops += 2.0 * 5.0 * n * n * math.log2(n) * (M // 9) * count
        cells += (n // r) ** 2
    byts = cells * (8 + 4 * K) + 8.0 * (2 + 12 * Q)
    if samples:
        byts += 8.0 * count * (2 * K + 2)
    return byts, flops


def work(case):
    wl = _workload(case)
    if case["kind"] == "learned":
        B, P = case["batch"], 148481
        return {"bytes": 4.0 * (65 * B + 2 * P), "flops": 6.0 * B * P}
    if case["kind"] == "level":
        b, f = _level_work(wl, case["level"], case["level"] > 0 and not case["mc"], case["count"], True)
        return {"bytes": b, "flops": f}
    parts = [_level_work(wl, l, l > 0, c, False) for l, c in enumerate(_counts(case))]
    return {"bytes": sum(p[0] for p in parts), "flops": sum(p[1] for p in parts)}


# ------------------------------------------------------------------ inputs
def _philox_seed(seed):
    return (int(seed) * 0x9E3779B97F4A7C15 + 0x1234567) & 0x7FFFFFFFFFFFFFFF


_WIDTHS = (64, 256, 256, 256, 1)


def _network(case, seed):
    """Network parameters (He-uniform weights, small biases), standardised
    features and targets close to a quadratic of a few of them."""
    g = np.random.default_rng(seed)
    theta = []
    for a, b in zip(_WIDTHS[:-1], _WIDTHS[1:]):
        lim = math.sqrt(6.0 / a)
        theta += [g.uniform(-lim, lim, a * b), g.uniform(-0.05, 0.05, b)]
    X = g.standard_normal((case["batch"], 64)).astype(np.float32)
    T = (0.6 * X[:, 0] - 0.3 * X[:, 5] + 0.05 * (X[:, 2] ** 2 - 1.0) +
         0.01 * g.standard_normal(case["batch"])).astype(np.float32)
    return np.concatenate(theta).astype(np.float32), X, T


# ------------------------------------------------------------------ in 64 bits
def exact(case, seed):
    if case["kind"] == "learned":
        return _exact_gradient(case, seed)
    wl, ps = _workload(case), _philox_seed(seed)
    if case["kind"] == "level":
        if _exact_seconds(wl, case["level"], case["count"]) > 18.0:
            return None
        sums, samples = _exact_level(wl, case["level"], case["mc"], case["count"], ps)
        return {"sums": sums, "samples": samples}
    counts = _counts(case)
    if sum(_exact_seconds(wl, l, c) for l, c in enumerate(counts)) > 18.0:
        return None
    return {"sums": np.stack([_exact_level(wl, l, False, c, ps)[0] for l, c in enumerate(counts)])}


def _exact_seconds(wl, level, count):
    """A rough time of _exact_level on a GPU: launches, or about 1 ns per cell and step."""
    n, M, _, _ = _grid(wl, level)
    return M * max(1.5e-3, 1.0e-9 * count * n * n)


def _exact_gradient(case, seed):
    theta, X, T = (torch.from_numpy(a.astype(np.float64)) for a in _network(case, seed))
    params, off = [], 0
    for a, b in zip(_WIDTHS[:-1], _WIDTHS[1:]):
        params.append(theta[off:off + a * b].reshape(b, a).clone().requires_grad_())
        params.append(theta[off + a * b:off + a * b + b].clone().requires_grad_())
        off += a * b + b
    h = X
    for i in range(0, len(params), 2):
        h = h @ params[i].T + params[i + 1]
        if i + 2 < len(params):
            h = torch.relu(h)
    loss = ((h[:, 0] - T) ** 2).mean()
    loss.backward()
    return {"loss": loss.item(), "grad": torch.cat([p.grad.reshape(-1) for p in params]).numpy()}


def _philox(c0, c1, c2, c3, k0, k1):
    """Philox4x32-10 on int64 tensors that hold 32-bit words."""
    mask = 0xFFFFFFFF
    for r in range(10):
        if r:
            k0, k1 = (k0 + 0x9E3779B9) & mask, (k1 + 0xBB67AE85) & mask
        p0, p1 = c0 * 0xD2511F53, c2 * 0xCD9E8D57
        c0, c1, c2, c3 = ((p1 >> 32) & mask) ^ c1 ^ k0, p1 & mask, ((p0 >> 32) & mask) ^ c3 ^ k1, p0 & mask
    return c0, c1, c2, c3


def _box_muller(a, b):
    u = (a.double() + 1.0) * 2.0 ** -32
    th = (b.double() + 0.5) * (2.0 * math.pi * 2.0 ** -32)
    r = torch.sqrt(-2.0 * torch.log(u))
    return torch.stack((r * torch.cos(th), r * torch.sin(th)))


def _normals(seed, level, tag, ids, m, n, pairs):
    """Standard normals [2 components][sample][n][n] of fine step m."""
    c2 = (ids & 0xFFFFFFFF)[:, None]
    c3 = ((level + 1) | (tag << 8)) | (((ids >> 32) & 0xFFFF) << 16)[:, None]
    x = _philox(pairs[None, :], torch.full_like(c2, m), c2, c3, seed & 0xFFFFFFFF, seed >> 32)
    z = torch.stack((_box_muller(x[0], x[1]), _box_muller(x[2], x[3])), dim=-1)
    return z.reshape(2, ids.numel(), n, n)


def _step(rho, Z, h, tau, N, b0):
    """One step of the scheme (Z: normals of the increments, or None)."""
    lap = (torch.roll(rho, 1, -1) + torch.roll(rho, -1, -1) + torch.roll(rho, 1, -2) + torch.roll(rho, -1, -2) -
           4.0 * rho)
    out = rho + (1.0 - b0) * tau / (2.0 * h * h) * lap
    if Z is not None and N > 0:
        amp = math.sqrt(tau / N) / (2.0 * h * h) * torch.sqrt(torch.clamp(rho, min=0.0))
        f1, f2 = amp * Z[0], amp * Z[1]
        out += torch.roll(f1, -1, -2) - torch.roll(f1, 1, -2) + torch.roll(f2, -1, -1) - torch.roll(f2, 1, -1)
    if b0 > 0:
        n = rho.shape[-1]
        s = torch.sin(math.pi * torch.arange(n, dtype=torch.float64, device=rho.device) / n) ** 2
        den = 1.0 + b0 * 2.0 * tau / (h * h) * (s[:, None] + s[None, :])
        out = torch.fft.irfft2(torch.fft.rfft2(out) / den[:, :n // 2 + 1], s=(n, n))
    return out


def _fourier_restriction(n, device):
    """One axis of the Fourier coupling: the modes that the coarse grid of n/3
    points resolves, its Nyquist mode with weight 2^-1/2 from each alias."""
    nc = n // 3
    K = nc // 2
    xi = torch.arange(-K, K + 1, dtype=torch.float64, device=device)
    w = torch.ones_like(xi)
    w[0] = w[-1] = math.sqrt(0.5)
    y = torch.arange(nc, dtype=torch.float64, device=device) / nc
    x = torch.arange(n, dtype=torch.float64, device=device) / n
    d = y[:, None] - x[None, :]
    return (w * torch.cos(2.0 * math.pi * d[:, :, None] * xi)).sum(-1) / math.sqrt(n * nc)


def _exact_level(wl, level, mc, count, seed):
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    f64 = dict(dtype=torch.float64, device=dev)
    n, M, h, tau = _grid(wl, level)
    r = wl.ratio
    period = r * r
    coupled = level > 0 and not mc
    ids = torch.arange(count, dtype=torch.int64, device=dev)
    pairs = torch.arange(n * n // 2, dtype=torch.int64, device=dev)
    phi_f = torch.as_tensor(np.stack(wl.phi(level)), **f64)
    rho0 = torch.as_tensor(wl.rho0(level), **f64)
    K = phi_f.shape[0]
    rho, bar = rho0.expand(count, n, n).clone(), rho0.clone()
    if coupled:
        nc, hc, tc = n // r, r * h, period * tau
        phi_c = torch.as_tensor(np.stack(wl.phi(level - 1)), **f64)
        rho0c = torch.as_tensor(wl.rho0(level - 1), **f64)
        rho_c, bar_c = rho0c.expand(count, nc, nc).clone(), rho0c.clone()
        acc = torch.zeros(2, count, n, n, **f64) if wl.coupling == 1 else torch.zeros(2, count, nc, nc, **f64)
        P1 = _fourier_restriction(n, dev) if wl.coupling == 1 else None
    for m in range(M):
        Z = _normals(seed, level, int(mc), ids, m, n, pairs)
        rho = _step(rho, Z, h, tau, wl.N, wl.b0)
        bar = _step(bar, None, h, tau, wl.N, wl.b0)
        if coupled:
            acc += Z if wl.coupling == 1 else Z.reshape(2, count, nc, 2, nc, 2).sum((3, 5))
            if (m + 1) % period == 0:
                Zc = P1 @ acc @ P1.T / 3.0 if wl.coupling == 1 else acc / 4.0
                rho_c = _step(rho_c, Zc, hc, tc, wl.N, wl.b0)
                bar_c = _step(bar_c, None, hc, tc, wl.N, wl.b0)
                acc.zero_()
    samples = torch.zeros(count, 2 * K + 2, **f64)
    samples[:, :K] = h * h * torch.einsum("sij,kij->sk", rho - bar, phi_f)
    samples[:, 2 * K] = h * h * rho.sum((1, 2))
    if coupled:
        samples[:, K:2 * K] = hc * hc * torch.einsum("sij,kij->sk", rho_c - bar_c, phi_c)
        samples[:, 2 * K + 1] = hc * hc * rho_c.sum((1, 2))
    sums = [torch.tensor(float(count), **f64), torch.tensor(0.0, **f64)]   # the scheme conserves the mass
    for j in range(K):
        for k in (range(j, K) if wl.products else (j,)):
            df, dc = samples[:, j], samples[:, K + j]
            pf, pc = wl.N * df * samples[:, k], wl.N * dc * samples[:, K + k]
            dp = pf - pc
            sums += [(dp ** e).sum() for e in (1, 2, 3, 4)]
            sums += [pf.sum(), (pf ** 2).sum(), pc.sum(), (pc ** 2).sum()]
            sums += [df.sum(), (df ** 2).sum(), dc.sum(), (dc ** 2).sum()]
    return torch.stack(sums).cpu().numpy(), samples.cpu().numpy()
