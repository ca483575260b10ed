"""Performance cases of the outer step: what a training or merging program has the library do.

Every case is one call of a public entry point of `paper_2607_03011_gb300.isoloco` on a
decoder-shaped parameter set: `outer_step` (IsoLoCo: the converged polar path, the fixed-step
variant, clip_high / clip_low, and bf16 replicas), `outer_step_host`, `diloco_outer_step`
(mean, TIES, DARE) and `iso_c_merge`.  A parameter set is `layers` decoder layers of width d
(four d x d matrices, two d x ff, one ff x d, two vectors of d) and, with vocab > 0, an
embedding and an untied head of vocab x d.  Values follow the paper's setting: theta ~
N(0, 0.02^2), per-worker pseudo-gradients with a shared low-rank part and independent noise
at 1e-3 of theta, and a momentum buffer carried from an earlier step.

The step works in place, so a pass begins from the kept global weights and momentum (the copy
a program holds to start the next round from, or to roll back to): otherwise repeated passes
on the same replicas would drift away from the values a step meets.
"""
from __future__ import annotations

import math

import torch

_THETA_STD = 0.02
_DELTA_STD = 2e-5
_RANK = 32

_LISTED = [
    # The smallest call: the unit-test-sized set, two workers.  Launch and iteration latency.
    dict(name="tiny_k2", op="iso", d=64, ff=256, layers=1, vocab=0, K=2, dtype="f32", momentum=0.9, sparsity=0.0),
    # Odd and ragged sizes: no dimension is a multiple of 8, tensors start at odd offsets.
    dict(name="ragged_k3", op="iso", d=515, ff=1361, layers=3, vocab=5003, K=3, dtype="f32", momentum=0.9,
         sparsity=0.0),
    # The headline: the ~180M set with eight workers, fp32 throughout.
    dict(name="llama_180m_k8", op="iso", d=1024, ff=2816, layers=12, vocab=32000, K=8, dtype="f32", momentum=0.9,
         sparsity=0.0),
    # The largest: the ~1.1B set's width (six of its layers), eight workers.
    dict(name="wide_2048_k8", op="iso", d=2048, ff=5632, layers=6, vocab=32000, K=8, dtype="f32", momentum=0.9,
         sparsity=0.0),
    # The ~3B set's width (one of its layers), four bf16 replicas.
    dict(name="bf16_3072_k4", op="iso", d=3072, ff=8192, layers=1, vocab=32000, K=4, dtype="bf16", momentum=0.9,
         sparsity=0.0),
    # The fixed five-step variant (Sec. 4.3), which a run that cannot wait for convergence picks.
    dict(name="fast_steps_k8", op="fast", d=1024, ff=2816, layers=4, vocab=32000, K=8, dtype="f32", momentum=0.9,
         sparsity=0.0),
    # The spectrum-clipping ablation (Sec. 4.5) on a mid-sized model without its embedding.
    dict(name="clip_high_k8", op="clip_high", d=1024, ff=2816, layers=3, vocab=0, K=8, dtype="f32", momentum=0.9,
         sparsity=0.0),
    # Parameters and replicas that live in host memory (offloaded workers), copies included.
    dict(name="host_k8", op="host", d=1024, ff=2816, layers=2, vocab=0, K=8, dtype="f32", momentum=0.9,
         sparsity=0.0),
    # Iso-C model merging (Eq. 1): four bf16 experts merged into an fp32 base.
    dict(name="merge_bf16_k4", op="merge", d=1024, ff=2816, layers=6, vocab=32000, K=4, dtype="bf16", momentum=0.0,
         sparsity=0.0),
    # DiLoCo's own step (Alg. 1) on the ~180M set: one streaming pass.
    dict(name="diloco_180m_k8", op="mean", d=1024, ff=2816, layers=12, vocab=32000, K=8, dtype="f32", momentum=0.9,
         sparsity=0.0),
    # TIES aggregation (Sec. 3.2) at the paper's sparsity.
    dict(name="ties_180m_k8", op="ties", d=1024, ff=2816, layers=12, vocab=32000, K=8, dtype="f32", momentum=0.9,
         sparsity=0.1),
    # DARE aggregation with many bf16 replicas and an odd number of parameters.
    dict(name="dare_bf16_k16", op="dare", d=1021, ff=2777, layers=6, vocab=10007, K=16, dtype="bf16", momentum=0.0,
         sparsity=0.3),
]


def listed():
    return [dict(c) for c in _LISTED]


def _shapes(case):
    d, ff, vocab = case["d"], case["ff"], case["vocab"]
    s = [(vocab, d)] if vocab else []
    for _ in range(case["layers"]):
        s += [(d, 0), (d, d), (d, d), (d, d), (d, d), (d, 0), (d, ff), (d, ff), (ff, d)]
    if vocab:
        s.append((vocab, d))
    return s


def _table(case):
    table, off = [], 0
    for r, c in _shapes(case):
        table.append((off, r, c))
        off += r * (c or 1)
    return table, off


def _polar_flops(r, c):
    """Multiply-adds x 2 of one polar factor by odd quintic steps, symmetric products counted once:
    7 steps, or 12 for a near-square matrix; on the n x n side where that is less."""
    m, n = max(r, c), min(r, c)
    steps = 12 if (m - n) * 16 < n else 7
    direct = steps * (m * n * n + n ** 3 + 2 * m * n * n)
    gram = m * n * n + steps * (2 * n ** 3 + n ** 3 + n ** 3 + 2 * n ** 3) + 2 * m * n * n
    return float(min(direct, gram))


def work(case):
    table, n = _table(case)
    eb = 4 if case["dtype"] == "f32" else 2
    op = case["op"]
    # replicas, theta and momentum in; theta and momentum out (merge: base in, merged out)
    nbytes = case["K"] * n * eb + (8 * n if op == "merge" else 16 * n)
    flops = 0.0
    if op in ("iso", "clip_high", "clip_low", "host", "merge"):
        flops = sum(_polar_flops(r, c) for _, r, c in table if c)
    if op in ("clip_high", "clip_low"):
        # H = Q^T Delta, the polar factor of the n x n H / sigma_bar - I, and Q S'
        flops += sum(_polar_flops(min(r, c), min(r, c)) + 3.0 * r * c * min(r, c) for _, r, c in table if c)
    if op == "fast":
        flops = sum(5.0 * (3.0 * r * c * min(r, c) + min(r, c) ** 3) for _, r, c in table if c)
    return {"bytes": float(nbytes), "flops": float(flops)}


def _cost(case):
    w = work(case)
    return w["bytes"] / 6e12 + w["flops"] / 7e14


def draw(rng):
    """Widths from 24 to 3072 over their logarithm, one in two odd; every entry point and option."""
    most = _cost(next(c for c in _LISTED if c["name"] == "wide_2048_k8"))
    while True:
        op = rng.choice(["iso", "iso", "iso", "iso", "fast", "clip_high", "clip_low", "host", "merge", "mean", "ties",
                         "dare"])
        d = int(round(math.exp(rng.uniform(math.log(24), math.log(3072)))))
        d = d | 1 if rng.random() < 0.5 else max(24, d // 64 * 64 or d // 8 * 8)
        ff = max(32, int(d * rng.uniform(2.0, 4.0)))
        ff = ff | 1 if rng.random() < 0.5 else (ff // 8 * 8)
        layers = int(round(math.exp(rng.uniform(0.0, math.log(16)))))
        vocab = rng.choice([0, 0, d * rng.randint(2, 6) + rng.randint(0, 9), 10007, 32000])
        case = dict(op=op, d=d, ff=ff, layers=layers, vocab=vocab, K=rng.choice([1, 2, 3, 4, 6, 8, 8, 12, 16]),
                    dtype=rng.choice(["f32", "f32", "bf16"]), momentum=rng.choice([0.0, 0.9]),
                    sparsity=rng.choice([0.05, 0.1, 0.3, 0.5]) if op in ("ties", "dare") else 0.0)
        _, n = _table(case)
        # room for three states, and host buffers quick to make
        if _cost(case) <= most and n * (case["K"] * 4 + 40) <= 30e9 and (op != "host" or n * case["K"] <= 3e8):
            return case


def _inputs(case, seed):
    """theta, momentum [n] fp32 and K replicas (every buffer 16-byte aligned), on the GPU."""
    table, n = _table(case)
    dev = torch.device("cuda")
    g = torch.Generator(device=dev)
    g.manual_seed(int(seed))
    theta = torch.randn(n, generator=g, device=dev) * _THETA_STD
    mom = torch.randn(n, generator=g, device=dev) * _DELTA_STD
    shared = torch.empty(n, device=dev)
    for off, r, c in table:
        if c:
            rk = min(_RANK, r, c)
            a = torch.randn(r, rk, generator=g, device=dev)
            b = torch.randn(c, rk, generator=g, device=dev)
            shared[off:off + r * c] = (a @ b.T).reshape(-1) * (_DELTA_STD / math.sqrt(rk))
        else:
            shared[off:off + r] = torch.randn(r, generator=g, device=dev) * _DELTA_STD
    dt = torch.float32 if case["dtype"] == "f32" else torch.bfloat16
    reps = []
    for _ in range(case["K"]):
        x = torch.randn(n, generator=g, device=dev)
        x.mul_(_DELTA_STD).add_(shared).neg_().add_(theta)
        reps.append(x.to(dt))
    return table, n, theta, mom, reps


def prepare(case, seed):
    from paper_2607_03011_gb300 import isoloco

    table, n, theta, mom, reps = _inputs(case, seed)
    op = case["op"]
    kw = dict(outer_lr=0.7, momentum=case["momentum"])
    if op == "fast":
        kw["fast_steps"] = 5
    elif op in ("clip_high", "clip_low"):
        kw["spectrum_kind"] = 1 if op == "clip_high" else 2
    elif op in ("ties", "dare"):
        kw.update(aggregator=1 if op == "ties" else 2, sparsity=case["sparsity"], seed=11)
    st = dict(op=op, theta0=theta, mom0=mom, reps=reps, opts=isoloco.make_opts(**kw),
              plan=isoloco.Plan(table, n, case["K"], reps[0].dtype))
    if op == "merge":
        st["out"] = torch.empty_like(theta)
    elif op == "host":
        st["reps"] = [r.cpu().pin_memory() for r in reps]
        st["theta"], st["mom"] = theta.cpu().pin_memory(), mom.cpu().pin_memory()
    else:
        st["theta"], st["mom"] = theta.clone(), mom.clone()
    return st


def run(st):
    op, plan = st["op"], st["plan"]
    if op == "merge":
        plan.iso_c_merge(st["theta0"], st["reps"], 1.0, st["out"])
        return st["out"]
    theta, mom = st["theta"], st["mom"]
    theta.copy_(st["theta0"], non_blocking=True)
    mom.copy_(st["mom0"], non_blocking=True)
    if op == "host":
        plan.outer_step_host(theta, mom, st["reps"], st["opts"])
    elif op in ("mean", "ties", "dare"):
        plan.diloco_outer_step(theta, mom, st["reps"], st["opts"])
    else:
        plan.outer_step(theta, mom, st["reps"], st["opts"])
    return theta, mom


def tolerance(case):
    op = case["op"]
    if op == "mean" or op == "dare":
        return {"rel": 1e-6, "max": 1e-4}  # 32-bit sums of K terms, cancellation in mu B + U included
    if op == "ties":
        # 32-bit sums decide an entry's sign: where positive and negative mass nearly cancel it flips
        return {"rel": 2e-3, "max": 0.99}
    if op == "merge":
        return {"rel": 1e-5, "max": 1e-3}  # Iso-C's error relative to the base it is added to
    if op in ("clip_high", "clip_low"):
        return {"rel": 5e-4, "max": 0.02}  # three passes per product: 1e-5 to 1e-4 in U
    # Iso-C from 16-bit hi + lo operand planes: up to 1e-3 in U, less in mu B + U
    return {"rel": 2e-3, "max": 0.05}


# ------------------------------------------------------------------ the same in 64 bits
def _polar64(a):
    """Orthogonal polar factor: scaled Newton (Higham 1986) on a square matrix; a rectangular one goes
    through the triangular factor of its Gram matrix (these are well conditioned)."""
    if a.shape[0] < a.shape[1]:
        return _polar64(a.mT).mT
    if a.shape[0] > a.shape[1] and (a.shape[0] - a.shape[1]) * 16 >= a.shape[1]:
        r = torch.linalg.cholesky((a.mT @ a) / a.square().sum()).mT
        return torch.linalg.solve_triangular(r, a / a.norm(), upper=True, left=False) @ _polar64(r)
    if a.shape[0] > a.shape[1]:
        q, r = torch.linalg.qr(a)
        return q @ _polar64(r)
    x = a / a.norm()
    for _ in range(40):
        y = torch.linalg.inv(x)
        g = ((torch.linalg.matrix_norm(y, 1) * torch.linalg.matrix_norm(y, math.inf)) /
             (torch.linalg.matrix_norm(x, 1) * torch.linalg.matrix_norm(x, math.inf))) ** 0.25
        nx = 0.5 * (g * x + y.mT / g)
        done = (nx - x).norm() <= 1e-9 * nx.norm()
        x = nx
        if done:
            break
    # one unscaled step: quadratic convergence leaves rounding only
    return 0.5 * (x + torch.linalg.inv(x).mT)


# the first five steps of the standard quintic schedule, which define the fixed-step variant
_QUINTIC = [(8.1554822, -22.4715242, 15.8685976), (4.03306695, -2.79585802, 0.50982817),
            (3.88173828, -2.75072926, 0.513786618), (3.35469155, -2.50666689, 0.509138704),
            (2.33843651, -1.69909139, 0.420275305)]


def _direction64(op, delta):
    """The update direction of one matrix: Iso-C, its fixed-step form, or the clipped spectrum."""
    r = min(delta.shape)
    if op == "fast":
        t = delta if delta.shape[0] >= delta.shape[1] else delta.mT
        x = t / (t.mT @ t).norm().sqrt()
        for a, b, c in _QUINTIC:
            g = x.mT @ x
            x = a * x + x @ (b * g + c * (g @ g))
        x = x if delta.shape[0] >= delta.shape[1] else x.mT
        return delta.norm() / math.sqrt(r) * x
    q = _polar64(delta)
    sbar = (q * delta).sum() / r
    if op not in ("clip_high", "clip_low"):
        return sbar * q
    tall = delta.shape[0] >= delta.shape[1]
    h = q.mT @ delta if tall else delta @ q.mT
    s, v = torch.linalg.eigh(0.5 * (h + h.mT))
    f = (v * (torch.clamp(s, max=sbar) if op == "clip_high" else torch.clamp(s, min=sbar))) @ v.mT
    return q @ f if tall else f @ q


def _splitmix_top24(z):
    """Top 24 bits of SplitMix64's mix of z (int64 bit patterns)."""
    def shr(x, k):
        return (x >> k) & ((1 << (64 - k)) - 1)

    def c64(v):
        return v - (1 << 64) if v >= 1 << 63 else v

    z = (z ^ shr(z, 30)) * c64(0xBF58476D1CE4E5B9)
    z = (z ^ shr(z, 27)) * c64(0x94D049BB133111EB)
    return shr(z ^ shr(z, 31), 40)


def _sum64(op, case, n, theta, reps):
    """The aggregated pseudo-gradient over all entries."""
    K = case["K"]
    p = float(torch.tensor(case["sparsity"], dtype=torch.float32))  # the option is a 32-bit float
    if op == "ties":
        keep = n - int(math.floor(p * n))
        pos = torch.zeros(n, dtype=torch.float64, device=theta.device)
        neg = torch.zeros_like(pos)
        cp = torch.zeros(n, dtype=torch.int32, device=theta.device)
        cn = torch.zeros_like(cp)
        for r in reps:
            dl = theta - r.float()
            thr = dl.abs().sort(descending=True).values[keep - 1]
            dl = torch.where(dl.abs() >= thr, dl, torch.zeros_like(dl)).double()
            pos += dl.clamp(min=0)
            neg += dl.clamp(max=0)
            cp += dl > 0
            cn += dl < 0
        s = pos + neg
        return torch.where(s > 0, pos / cp.clamp(min=1), torch.where(s < 0, neg / cn.clamp(min=1), torch.zeros_like(s)))
    acc = torch.zeros(n, dtype=torch.float64, device=theta.device)
    pthr = int(math.ceil(p * (1 << 24)))
    for k, r in enumerate(reps):
        dl = theta.double() - r.double()
        if op == "dare":
            gamma = 0x9E3779B97F4A7C15 - (1 << 64)
            idx = torch.arange(k * n + 1, (k + 1) * n + 1, dtype=torch.int64, device=theta.device)
            dl = torch.where(_splitmix_top24(idx * gamma + 11) >= pthr, dl / (1.0 - p), torch.zeros_like(dl))
            del idx
        acc += dl
    return acc if op == "merge" else acc / K


def exact(case, seed):
    op = case["op"]
    if op not in ("mean", "ties", "dare"):
        # seconds: the inverses and eigenvectors of the n x n matrices in 64 bits
        t = sum(((r * c * min(r, c) if op == "fast" else 0) + min(r, c) ** 3) * 1e-10 for _, r, c in _table(case)[0] if c)
        if t * (4 if op in ("clip_high", "clip_low") else 1) > 20.0:
            return None
    table, n, theta, mom, reps = _inputs(case, seed)
    d = _sum64(op, case, n, theta, reps)
    del reps
    if op not in ("mean", "ties", "dare"):
        sign = -1.0 if op == "merge" else 1.0
        for off, r, c in table:
            if c:
                d[off:off + r * c] = _direction64(op, d[off:off + r * c].view(r, c)).reshape(-1)
        d *= sign
    if op == "merge":
        return theta.double() + d
    mu = case["momentum"]
    mu = float(torch.tensor(mu, dtype=torch.float32))
    eta = float(torch.tensor(0.7, dtype=torch.float32))
    b = mu * mom.double() + d
    return theta.double() - eta * (d + mu * b), b
