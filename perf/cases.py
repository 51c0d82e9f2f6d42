"""The workloads this library is timed on.

A case is one call (or one short sequence of calls) of the public interface on inputs of a
stated size: characterising a target (descriptor), the loss and its gradient, one Adam
iteration, a differentiable descriptor inside somebody else's autograd graph, a batch of
mixed jobs, a short reconstruction.  Inputs are what these calls meet: two-phase media
(thresholded periodic Gaussian random fields) as targets, and fields somewhere on the way
from the uniform random start to such a medium.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2103_09686_gb300 as dm
from paper_2103_09686_gb300 import autograd as dm_autograd

SOFT, IDENTITY = "soft", "identity"


def _case(name, call, shape, window, levels=1, descriptor="s2", threshold=SOFT, phases=1, count=1, iters=1):
    c = {"call": call, "ndim": len(shape), "levels": levels, "descriptor": descriptor, "threshold": threshold,
         "phases": phases, "count": count, "iters": iters}
    for a in range(3):
        c["n%d" % a] = int(shape[a]) if a < len(shape) else 0
        c["w%d" % a] = int(window[a]) if a < len(window) else 0
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest call: characterise a 32^2 patch; launches and latency are all of it
        _case("descriptor_32", "descriptor", (32, 32), (4, 4)),
        # one reconstruction iteration of the paper's 64^2 media
        _case("adam_64", "adam", (64, 64), (16, 16)),
        # an image that is no power of two in either axis, cut from a larger micrograph
        _case("loss_grad_odd", "loss_grad", (255, 381), (25, 31)),
        # the descriptor as a layer of another program's loss: autograd forward and backward
        _case("autograd_256", "autograd", (256, 256), (32, 32), levels=3),
        # the headline: one iteration of a 512^2 reconstruction over three multigrid levels
        _case("adam_512", "adam", (512, 512), (64, 64), levels=3),
        # a large micrograph characterised once, short range, levels down to 64^2
        _case("descriptor_1024", "descriptor", (1024, 1024), (16, 16), levels=5),
        # a served 3-D job
        _case("adam_3d_64", "adam", (64, 64, 64), (8, 8, 8), levels=2),
        # the largest 3-D medium
        _case("loss_grad_3d_128", "loss_grad", (128, 128, 128), (24, 24, 24), levels=2),
        # mixed jobs of a server advanced together, one iteration each
        _case("adam_batch_24", "adam_batch", (64, 512), (16, 64), count=24),
        # three phases: all nine cross-correlations
        _case("adam_phases_3", "adam", (512, 512), (64, 64), levels=3, phases=3),
        # the three-point descriptor of the paper's checkerboards, two multigrid levels
        _case("adam_s3_128", "adam", (128, 128), (31, 31), levels=2, descriptor="s3"),
        # the identity-threshold ablation on the large 3-D medium
        _case("identity_3d_128", "loss_grad", (128, 128, 128), (24, 24, 24), threshold=IDENTITY),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["s2", "s2", "s2", "s2_3d", "s2_3d", "batch", "phases", "s3", "identity", "tilde", "reconstruct"])
    call = rng.choice(["descriptor", "loss_grad", "adam", "autograd"])
    levels = rng.choice([1, 1, 2, 3])
    if kind in ("s2", "tilde"):
        step = 1 << (levels - 1)
        wmax = rng.choice([8, 16, 32, 64])
        shape = [max(step, _log_int(rng, 24, 1024) // step * step) for _ in range(2)]
        window = [max(1, min(_log_int(rng, 2, wmax), (n >> (levels - 1)) // 2)) for n in shape]
        return _case(None, call, shape, window, levels, descriptor="s2" if kind == "s2" else "tilde")
    if kind == "s2_3d":
        levels = min(levels, 2)
        step = 1 << (levels - 1)
        shape = [max(step, _log_int(rng, 12, 128) // step * step) for _ in range(3)]
        window = [max(1, min(_log_int(rng, 1, 16), (n >> (levels - 1)) // 2)) for n in shape]
        return _case(None, call, shape, window, levels)
    if kind == "batch":
        lo = rng.choice([32, 64])
        hi = rng.choice([128, 256, 512])
        wlo = rng.randint(4, 16)
        return _case(None, "adam_batch", (lo, hi), (wlo, rng.randint(wlo, 64)), count=rng.randint(2, 24))
    if kind == "phases":
        step = 1 << (levels - 1)
        shape = [max(step, _log_int(rng, 32, 384) // step * step) for _ in range(2)]
        window = [max(1, min(_log_int(rng, 2, 48), (n >> (levels - 1)) // 2)) for n in shape]
        return _case(None, rng.choice(["descriptor", "loss_grad", "adam"]), shape, window, levels,
                     phases=rng.randint(2, 3))
    if kind == "s3":
        levels = min(levels, 2)
        step = 1 << (levels - 1)
        shape = [max(step, _log_int(rng, 24, 160) // step * step) for _ in range(2)]
        window = [max(1, min(_log_int(rng, 4, 31), (n >> (levels - 1)) // 2)) for n in shape]
        return _case(None, rng.choice(["descriptor", "loss_grad", "adam"]), shape, window, levels, descriptor="s3")
    if kind == "identity":
        n = rng.choice([32, 48, 64, 80, 96, 128])
        w = rng.randint(1, min(24, n // 2))
        return _case(None, rng.choice(["descriptor", "loss_grad", "autograd"]), (n, n, n), (w, w, w),
                     threshold=IDENTITY)
    n = [_log_int(rng, 24, 160) for _ in range(2)]
    w = [max(1, min(_log_int(rng, 4, 31), a // 2)) for a in n]
    return _case(None, "reconstruct", n, w, iters=rng.randint(4, 12))


# ----------------------------------------------------------------------------- inputs

LR = 1e-3


def _problem(c):
    nd = c["ndim"]
    shape = tuple(c["n%d" % a] for a in range(nd))
    window = tuple(c["w%d" % a] for a in range(nd))
    kind = {"s2": dm.DMCR_DESC_S2, "s3": dm.DMCR_DESC_S3, "tilde": dm.DMCR_DESC_S2_TILDE}[c["descriptor"]]
    return dm.Params(shape=shape, window=window, levels=c["levels"], descriptor=kind, phases=c["phases"],
                     threshold=dm.DMCR_IDENTITY if c["threshold"] == IDENTITY else dm.DMCR_SOFT)


def _problems(c):
    """The instances of a case: one, or `count` square 2-D jobs of mixed size and window."""
    if c["call"] != "adam_batch":
        return [_problem(c)]
    # sizes and windows belong to the case; only the contents of the fields follow the seed
    rng = np.random.default_rng(c["count"] * 1000 + c["n0"] + c["n1"] + c["w0"] + c["w1"])
    sizes = [n for n in (32, 64, 96, 128, 256, 512) if c["n0"] <= n <= c["n1"]]
    out = []
    for _ in range(c["count"]):
        n = int(rng.choice(sizes))
        w = int(min(rng.integers(c["w0"], c["w1"] + 1), n // 2))
        out.append(dm.Params(shape=(n, n), window=(w, w)))
    return out


def _medium(shape, gen, phases):
    """Indicator(s) of a periodic Gaussian random field cut at quantiles (FP32, on the GPU)."""
    noise = torch.randn(shape, generator=gen, device="cuda", dtype=torch.float32)
    kern = torch.ones(shape, device="cuda", dtype=torch.float32)
    for a, n in enumerate(shape):
        x = torch.arange(n, device="cuda", dtype=torch.float32)
        x = torch.minimum(x, n - x)
        k = torch.exp(-x * x / (2.0 * max(n / 32.0, 1.5) ** 2))
        kern = kern * k.reshape([-1 if b == a else 1 for b in range(len(shape))])
    g = torch.fft.ifftn(torch.fft.fftn(noise) * torch.fft.fftn(kern)).real
    flat = g.reshape(-1)
    if phases == 1:
        cut = torch.sort(flat).values[int(0.65 * (flat.numel() - 1))]
        return (g > cut).float().contiguous()
    order = torch.sort(flat).values
    cuts = [order[int((k + 1) / phases * (flat.numel() - 1))] for k in range(phases - 1)]
    label = torch.zeros(shape, device="cuda", dtype=torch.int64)
    for q in cuts:
        label += (g > q).long()
    return torch.stack([(label == k).float() for k in range(phases)]).contiguous()


def _inputs(c, seed):
    """(problems, target media, fields): the field lies between the uniform start and a medium
    of the same statistics, as in the course of a reconstruction."""
    ps = _problems(c)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed) * 7919 + 17)
    targets, fields = [], []
    for p in ps:
        targets.append(_medium(p.shape, gen, p.phases))
        start = torch.rand(targets[-1].shape, generator=gen, device="cuda", dtype=torch.float32)
        other = _medium(p.shape, gen, p.phases)
        blend = 0.0 if p.descriptor == dm.DMCR_DESC_S3 else 0.4
        fields.append((start + blend * (other - start)).contiguous())
    return ps, targets, fields


def _target(p, medium):
    """The target descriptor a program has in hand: that of a medium, in FP32.  A medium's
    pooled levels hold few distinct values v_a, so S_bar(r) = sum_ab F(v_a, v_b) C_ab(r) with
    the correlations C_ab of their indicators (transforms, 64 bits)."""
    if p.descriptor == dm.DMCR_DESC_S3:
        return _exact_descriptor(p, medium.double()).float()
    alpha, c1, c3 = _constants()
    shifts = torch.tensor(_half_window(p.window), device="cuda")
    out = []
    for lev, fs in enumerate(_levels(medium.double(), p)):
        n = fs[0].shape
        values = [torch.unique(f) for f in fs]
        hats = [[torch.fft.fftn((f == v).double()) for v in vs] for f, vs in zip(fs, values)]
        at = tuple(shifts[:, a] % n[a] for a in range(3))
        for ha, va in zip(hats, values):
            for hb, vb in zip(hats, values):
                mean = 0.5 * (va[:, None] + vb[None, :])
                f = mean if p.threshold == dm.DMCR_IDENTITY else c1 * torch.sigmoid(alpha * (mean - 0.75)) + c3
                f = (f * f).tolist()
                power = torch.zeros_like(ha[0])
                for i, x in enumerate(ha):
                    power += x.conj() * sum(f[i][j] * y for j, y in enumerate(hb))
                s = torch.fft.ifftn(power).real[at] * (_weight(p, lev) / fs[0].numel())
                out.append(_tilde(p, s))
    return torch.cat(out).float()


def prepare(case, seed):
    ps, targets, fields = _inputs(case, seed)
    call = case["call"]
    st = {"call": call, "ps": ps, "fields": fields, "p": ps[0], "field": fields[0]}
    if call == "descriptor":
        st["field"] = targets[0]
        st["desc"] = torch.empty(dm.dmcr_descriptor_length(ps[0]), device="cuda")
        st["ws"] = dm.workspace(ps[0])
        return st
    if call == "autograd":
        gen = torch.Generator(device="cuda")
        gen.manual_seed(int(seed) + 5)
        st["field"] = fields[0].requires_grad_(True)
        st["up"] = torch.randn(case["levels"] * _khalf(ps[0].window), generator=gen, device="cuda")
        return st
    st["targets"] = [_target(p, t) for p, t in zip(ps, targets)]
    st["target"] = st["targets"][0]
    st["loss"] = torch.empty(len(dm.OUT_NAMES) * len(ps), device="cuda")
    if call == "loss_grad":
        st["grad"] = torch.empty_like(fields[0])
        st["ws"] = dm.workspace(ps[0])
        return st
    st["ms"] = [torch.zeros_like(f) for f in fields]
    st["vs"] = [torch.zeros_like(f) for f in fields]
    st["steps"] = [0] * len(ps)
    st["opts"] = dm.ReconOpts(lr=LR, max_iters=case["iters"], check_every=case["iters"], report_rounded=False)
    st["ws"] = dm.batch_workspace(ps) if call == "adam_batch" else dm.workspace(ps[0])
    return st


def run(state):
    s = state
    call, p = s["call"], s["p"]
    if call == "descriptor":
        dm.dmcr_descriptor(p, s["field"], s["desc"], s["ws"])
        return {"desc": s["desc"]}
    if call == "autograd":
        f = s["field"]
        f.grad = None
        desc = dm_autograd.s2_descriptor(f, p)
        desc.backward(s["up"])
        return {"desc": desc.detach(), "grad": f.grad}
    if call == "loss_grad":
        dm.dmcr_loss_grad(p, dm.LossOpts(), s["field"], s["target"], s["loss"], s["grad"], None, s["ws"])
        return {"loss": s["loss"], "grad": s["grad"]}
    if call == "adam":
        s["steps"][0] = dm.dmcr_adam_step(p, s["opts"], s["target"], s["field"], s["ms"][0], s["vs"][0],
                                          s["steps"][0], s["loss"], s["ws"])
        return {"loss": s["loss"], "field": s["field"], "m": s["ms"][0], "v": s["vs"][0]}
    if call == "adam_batch":
        s["steps"] = dm.dmcr_adam_step_batched(s["ps"], s["opts"], s["targets"], s["fields"], s["ms"], s["vs"],
                                               s["steps"], s["loss"], s["ws"])
        cat = lambda ts: torch.cat([t.reshape(-1) for t in ts])   # noqa: E731
        return {"loss": s["loss"], "field": cat(s["fields"]), "m": cat(s["ms"]), "v": cat(s["vs"])}
    rep, s["steps"][0] = dm.dmcr_reconstruct(p, s["opts"], s["target"], s["field"], s["ms"][0], s["vs"][0],
                                             s["steps"][0], ws=s["ws"])
    return {"L": rep["L"], "rel_err": rep["rel_err"], "field": s["field"], "m": s["ms"][0], "v": s["vs"][0]}


# ----------------------------------------------------------------------------- work

def _khalf(window):
    k = 1
    for w in window:
        k *= 2 * w + 1
    return (k + 1) // 2


def work(case):
    """Bytes: the field (and target, gradient or Adam state) once in and once out.  Operations:
    a correlation over N positions cannot do with less than a transform there and back
    (5 N log2 N each), its gradient the same again; the three-point matrix is a product of an
    N x K ensemble with itself, its gradient another."""
    call = case["call"]
    back = call != "descriptor"
    nbytes = flops = 0.0
    for p in _problems(case):
        k = _khalf(p.window)
        ph = max(1, p.phases)
        n1 = float(np.prod(p.shape))
        length = 0
        for lev in range(p.levels):
            n = float(np.prod([a >> lev for a in p.shape]))
            if p.descriptor == dm.DMCR_DESC_S3:
                length += k * k
                flops += (1 + 2 * back) * n * k * k
            else:
                length += ph * ph * k
                flops += ph * (4 if back else 2) * 5 * n * math.log2(max(n, 2))
        per_field = {"descriptor": 1, "autograd": 2, "loss_grad": 2}.get(call, 6)
        nbytes += 4.0 * (per_field * ph * n1 + length * (2 if call == "autograd" else 1))
    return {"bytes": nbytes * case["iters"], "flops": flops * case["iters"]}


# ----------------------------------------------------------------------------- 64-bit values

def _constants(alpha=10.0):
    s0 = 1.0 / (1.0 + math.exp(0.75 * alpha))
    s1 = 1.0 / (1.0 + math.exp(-0.25 * alpha))
    c1 = 1.0 / (s1 - s0)
    return alpha, c1, -c1 * s0


def _half_window(window):
    """Shifts of the half window in the library's order (3-D tuples)."""
    w = [0] * (3 - len(window)) + list(window)
    out = [(0, 0, x) for x in range(w[2] + 1)]
    out += [(0, y, x) for y in range(1, w[1] + 1) for x in range(-w[2], w[2] + 1)]
    out += [(z, y, x) for z in range(1, w[0] + 1) for y in range(-w[1], w[1] + 1) for x in range(-w[2], w[2] + 1)]
    return out


class _Pairs:
    """Values of the pairs (x, x + r) of one field with another (tips), in FP64, for runs of
    shifts that differ in rx alone: tensors (run, n0, n1, n2)."""

    def __init__(self, tail, tip, window, identity):
        self.identity = identity
        self.alpha, self.c1, self.c3 = _constants()
        self.n = tail.shape
        self.w = [0] * (3 - len(window)) + list(window)
        if identity:
            self.a, b = 0.5 * tail, 0.5 * tip
        else:
            self.a = torch.exp(-0.5 * self.alpha * tail + 0.75 * self.alpha)
            b = torch.exp(-0.5 * self.alpha * tip)
        for a in range(3):
            w = self.w[a]
            if w:
                b = torch.cat([b.narrow(a, self.n[a] - w, w), b, b.narrow(a, 0, w)], a)
        self.b = b.contiguous()

    def value(self, r, count=1):
        """s (the mean itself for the identity threshold) of the pairs of the shifts
        (r0, r1, r2 .. r2 + count - 1)."""
        s = self.b.stride()
        off = sum((self.w[a] + r[a]) * s[a] for a in range(3))
        tip = self.b.as_strided((count,) + tuple(self.n), (1,) + tuple(s), off)
        return self.a + tip if self.identity else (self.a * tip).add_(1.0).reciprocal_()

    def f(self, v):
        return v if self.identity else v.mul(self.c1).add_(self.c3)

    def ff(self, v):
        """f f' of the pair's mean."""
        if self.identity:
            return v
        return (v.mul(self.c1).add_(self.c3)).mul_(v).mul_((1.0 - v).mul_(self.c1 * self.alpha))


def _runs(shifts, n):
    """Runs (first index, first shift, count) of consecutive rx, at most about 2^24 pairs each."""
    most = max(1, (1 << 24) // n)
    i = 0
    while i < len(shifts):
        j = i + 1
        while j < len(shifts) and j - i < most and shifts[j][:2] == shifts[i][:2]:
            j += 1
        yield i, shifts[i], j - i
        i = j


def _embed(t):
    return t.reshape((1,) * (3 - t.dim()) + tuple(t.shape))


def _pool(t, nd):
    s = t.shape
    if nd == 2:
        return t.reshape(s[0], s[1] // 2, 2, s[2] // 2, 2).mean((2, 4))
    return t.reshape(s[0] // 2, 2, s[1] // 2, 2, s[2] // 2, 2).mean((1, 3, 5))


def _unpool(g, nd):
    for a in ((1, 2) if nd == 2 else (0, 1, 2)):
        g = g.repeat_interleave(2, a)
    return g / (2 ** nd)


def _levels(field, p):
    """Per level and phase the pooled field (FP64, 3-D embedded)."""
    nd = len(p.shape)
    cur = [_embed(f) for f in (field if p.phases > 1 else [field])]
    out = []
    for _ in range(p.levels):
        out.append(cur)
        cur = [_pool(t, nd) for t in cur] if len(out) < p.levels else cur
    return out


def _weight(p, lev):
    return 2.0 ** (len(p.shape) / 2.0 * lev)


def _s3_ensemble(f, p, shifts):
    pr = _Pairs(f, f, p.window, False)
    return pr, torch.cat([pr.f(pr.value(r, m)).reshape(m, -1) for _, r, m in _runs(shifts, f.numel())])


def _exact_descriptor(p, field):
    shifts = _half_window(p.window)
    ident = p.threshold == dm.DMCR_IDENTITY
    out = []
    for lev, fs in enumerate(_levels(field, p)):
        w = _weight(p, lev)
        if p.descriptor == dm.DMCR_DESC_S3:
            _, e = _s3_ensemble(fs[0], p, shifts)
            out.append((w / fs[0].numel() * (e @ e.T)).reshape(-1))
            continue
        for tail in fs:
            for tip in fs:
                pr = _Pairs(tail, tip, p.window, ident)
                s = torch.empty(len(shifts), dtype=torch.float64, device="cuda")
                for k, r, m in _runs(shifts, tail.numel()):
                    v = pr.f(pr.value(r, m)).reshape(m, -1)
                    s[k:k + m] = (v * v).sum(1)
                out.append(_tilde(p, s * (w / tail.numel())))
    return torch.cat(out)


def _tilde_q():
    alpha, c1, c3 = _constants()
    return 2.0 * (c1 / (1.0 + math.exp(0.25 * alpha)) + c3) ** 2


def _tilde(p, s):
    """One level's block of the corrected descriptor from S_bar2."""
    if p.descriptor != dm.DMCR_DESC_S2_TILDE:
        return s
    return torch.cat([s[:1], (s[1:] - _tilde_q() * s[0]) / (1.0 - _tilde_q())])


def _exact_vjp(p, field, up):
    """(dD/dM)^T up."""
    nd = len(p.shape)
    shifts = _half_window(p.window)
    ident = p.threshold == dm.DMCR_IDENTITY
    k = len(shifts)
    total = [torch.zeros_like(t) for t in _levels(field, p)[0]]
    off = 0
    for lev, fs in enumerate(_levels(field, p)):
        w = _weight(p, lev)
        grads = [torch.zeros_like(t) for t in fs]
        if p.descriptor == dm.DMCR_DESC_S3:
            pr, e = _s3_ensemble(fs[0], p, shifts)
            g = up[off:off + k * k].reshape(k, k)
            off += k * k
            back = (w / fs[0].numel()) * ((g + g.T) @ e)          # dL/de, K x N
            for i, r in enumerate(shifts):
                s = pr.value(r)[0]
                c = 0.5 * back[i].reshape(fs[0].shape) * (s * (1.0 - s)).mul_(pr.c1 * pr.alpha)
                grads[0] += c + torch.roll(c, r, (0, 1, 2))
        else:
            for a, tail in enumerate(fs):
                for b, tip in enumerate(fs):
                    u = up[off:off + k]
                    off += k
                    if p.descriptor == dm.DMCR_DESC_S2_TILDE:
                        q = _tilde_q()
                        u = torch.cat([u[:1] - q / (1.0 - q) * u[1:].sum(), u[1:] / (1.0 - q)])
                    u = u * (w / tail.numel())
                    # the tails' share of every pair, then the tips' (their tail lies at -r;
                    # a run of consecutive rx is passed backwards)
                    there = _Pairs(tail, tip, p.window, ident)
                    back = _Pairs(tip, tail, p.window, ident)
                    for i, r, m in _runs(shifts, tail.numel()):
                        um = u[i:i + m]
                        grads[a] += torch.tensordot(um, there.ff(there.value(r, m)), 1)
                        last = (-r[0], -r[1], -(r[2] + m - 1))
                        grads[b] += torch.tensordot(um.flip(0), back.ff(back.value(last, m)), 1)
        for a, g in enumerate(grads):
            for _ in range(lev):
                g = _unpool(g, nd)
            total[a] += g
    out = torch.stack([t.reshape(p.shape) for t in total])
    return out if p.phases > 1 else out[0]


def _exact_loss_grad(p, field, target):
    """The six loss values and the gradient of L = E (1 + lambda0 E_bc), lambda0 = N."""
    d = _exact_descriptor(p, field)
    rho = d - target
    n = float(np.prod(p.shape))
    e = torch.linalg.norm(rho)
    over, under = (field - 1.0).clamp_min(0.0), (-field).clamp_min(0.0)
    ebc = ((over * over).sum() + (under * under).sum()) / (n * n)
    lam = n * e
    loss = torch.stack([e, e * e, ebc, lam, e + lam * ebc, e / torch.linalg.norm(target)])
    g = _exact_vjp(p, field, rho / e * (1.0 + n * ebc)) + 2.0 * lam / (n * n) * (over - under)
    return loss, g


def exact(case, seed):
    ps, targets, fields = _inputs(case, seed)
    call = case["call"]
    if call == "descriptor":
        return {"desc": _exact_descriptor(ps[0], targets[0].double())}
    if call == "autograd":
        gen = torch.Generator(device="cuda")
        gen.manual_seed(int(seed) + 5)
        up = torch.randn(case["levels"] * _khalf(ps[0].window), generator=gen, device="cuda").double()
        f = fields[0].double()
        return {"desc": _exact_descriptor(ps[0], f), "grad": _exact_vjp(ps[0], f, up)}
    if call == "reconstruct":
        return None
    losses, outs = [], []
    for p, t, f in zip(ps, targets, fields):
        want = _target(p, t).double()
        loss, g = _exact_loss_grad(p, f.double(), want)
        losses.append(loss)
        outs.append((f.double(), g))
    if call == "loss_grad":
        return {"loss": losses[0], "grad": outs[0][1]}
    # one Adam step from zero moments (Keras form)
    b1, b2, eps = 0.9, 0.999, 1e-7
    ms = [(1.0 - b1) * g for _, g in outs]
    vs = [(1.0 - b2) * g * g for _, g in outs]
    lr_t = LR * math.sqrt(1.0 - b2) / (1.0 - b1)
    new = [f - lr_t * m / (torch.sqrt(v) + eps) for (f, _), m, v in zip(outs, ms, vs)]
    if call == "adam":
        return {"loss": losses[0], "field": new[0], "m": ms[0], "v": vs[0]}
    cat = lambda ts: torch.cat([t.reshape(-1) for t in ts])   # noqa: E731
    return {"loss": torch.cat(losses), "field": cat(new), "m": cat(ms), "v": cat(vs)}
