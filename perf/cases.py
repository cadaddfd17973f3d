"""The calls a user of this library makes, as measurable cases.

Each case is one pass through the public entry points of ``paper_2602_06895_gb300.ps``:

* ``generate``   Philox -> weighted events of a channel set (Program.generate, or an executor replay),
                 FP64 and mixed precision, compiled and interpreted programs;
* ``adapt``      one VEGAS training iteration (generation with the training histogram, then the rebin);
* ``flow``       sampling from the coupling flow; ``flow_train`` a training step's gradients on the map's
                 weights;
* ``reweight``   global multichannel weights of given events: inverse maps, densities, combination;
* ``unweight``   the maximum weight with a bounded over-weight share, then accept/reject.

The sizes are those of the library's benchmark configurations (1e5 events at 2->2, 1e7 at 2->4, 4e6 of
the six 2->5 channels, chunks of 2^22 at 2->8, flow batches of 2^16, 1e6 reweighted, 1e7 unweighted).
``exact`` evaluates the same methods from their formulas with torch in 64 bits.
"""
import math
from functools import lru_cache

import numpy as np
import torch

from paper_2602_06895_gb300 import ps
from paper_2602_06895_gb300 import workloads as W

DEV = "cuda"
F64 = torch.float64
M32 = 0xFFFFFFFF

# elementary floating-point operations of one event (sums, products, quotients, roots and one per
# function call), counted on the formulas; the SDE sum of the multichannel sets included
_OPS = {"2to2": 50, "2to4": 460, "2to5": 1300, "2to8": 3600}


def listed():
    return [
        # a quick look at a fixed-energy process: the smallest call, latency counts
        {"name": "gen_2to2_f64", "kind": "generate", "set": "2to2", "events": 100_000, "precision": "f64",
         "jit": False, "replay": False, "store": "all"},
        # production of a sample of the W W process with the compiled FP64 program
        {"name": "gen_2to4_f64", "kind": "generate", "set": "2to4", "events": 10_000_000, "precision": "f64",
         "jit": True, "replay": False, "store": "all"},
        # the same without waiting for a compiler: the interpreter is what program_for gives by default
        {"name": "gen_2to4_interp", "kind": "generate", "set": "2to4", "events": 999_983, "precision": "f64",
         "jit": False, "replay": False, "store": "all"},
        # production in mixed precision
        {"name": "gen_2to4_mixed", "kind": "generate", "set": "2to4", "events": 10_000_000, "precision": "mixed",
         "jit": True, "replay": False, "store": "all"},
        # an integration of six channels with t-chains and uneven shares: weights and shares are stored
        {"name": "gen_2to5_f64", "kind": "generate", "set": "2to5", "events": 4_000_000, "precision": "f64",
         "jit": True, "replay": False, "store": "weights"},
        # a chunk of a streamed 24-channel run, replayed from its executor: the FP64 integration, and
        # the production of event records in mixed precision
        {"name": "gen_2to8_f64", "kind": "generate", "set": "2to8", "events": 1 << 22, "precision": "f64",
         "jit": True, "replay": True, "store": "weights"},
        {"name": "gen_2to8_mixed", "kind": "generate", "set": "2to8", "events": 1 << 22, "precision": "mixed",
         "jit": True, "replay": True, "store": "all"},
        # one iteration of VEGAS training before a production
        {"name": "adapt_2to4", "kind": "adapt", "events": 1_000_000, "jit": True},
        # inference sampling from a trained flow
        {"name": "flow_sample", "kind": "flow", "events": 1 << 20, "layers": 6, "bins": 16},
        # a flow training step: sample, map, loss and gradients
        {"name": "flow_train", "kind": "flow_train", "events": 1 << 16, "layers": 6, "bins": 16},
        # events of one channel reweighted with the densities of all six
        {"name": "reweight_2to5", "kind": "reweight", "events": 1_000_000, "channel": 1},
        # unweighting of a 2->4 sample
        {"name": "unweight", "kind": "unweight", "events": 10_000_000, "eps": 1e-3},
    ]


def draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["generate"] * 6 + ["adapt", "flow", "flow_train", "reweight", "unweight"])
    if kind == "generate":
        sel = rng.choice(["2to2", "2to4", "2to4", "2to5", "2to8"])
        top = {"2to2": 1_000_000, "2to4": 10_000_000, "2to5": 4_000_000, "2to8": 1 << 22}[sel]
        jit = sel == "2to8" or rng.random() < 0.7
        precision = rng.choice(["f64", "f64", "mixed"])
        return {"kind": kind, "set": sel, "events": size(1000, top if jit else min(top, 2_000_000)),
                "precision": precision, "jit": jit, "replay": rng.random() < 0.4,
                "store": "weights" if precision == "f64" and sel in ("2to5", "2to8") else "all"}
    if kind == "adapt":
        return {"kind": kind, "events": size(10_000, 2_000_000), "jit": rng.random() < 0.7}
    if kind == "flow":
        return {"kind": kind, "events": size(1000, 1 << 20), "layers": rng.randint(3, 6), "bins": 16}
    if kind == "flow_train":
        return {"kind": kind, "events": size(1000, 1 << 16), "layers": rng.randint(3, 6), "bins": 16}
    if kind == "reweight":
        return {"kind": kind, "events": size(1000, 1_000_000), "channel": rng.randint(0, 5)}
    return {"kind": kind, "events": size(1000, 10_000_000), "eps": rng.choice([0.0, 1e-4, 1e-3, 1e-2])}


# --------------------------------------------------------------------------------------------
# what a user has in hand
# --------------------------------------------------------------------------------------------
def _channels(name):
    if name == "2to2":
        return [W.two_body_fixed()]
    if name == "2to4":
        return [W.ww_hadronic()]
    if name == "2to5":
        return W.multichannel_2to5()
    return W.channels_2to8()


def _split(name, n, n_ch):
    """Event counts per channel: the uneven shares of the 2->5 set, else even ones."""
    if name == "2to5":
        tot = sum(W.MULTICHANNEL_EVENTS)
        ev = [n * c // tot for c in W.MULTICHANNEL_EVENTS]
        ev[-1] += n - sum(ev)
        return ev
    return [n // n_ch + (1 if c < n % n_ch else 0) for c in range(n_ch)]


def _grid(seed, dims, bins):
    """Edges of an adapted-looking VEGAS grid: bin widths that vary smoothly by a factor of a few."""
    rng = np.random.default_rng(seed)
    x = (np.arange(bins) + 0.5) / bins
    e = np.zeros((dims, bins + 1))
    for j in range(dims):
        a, b, c = rng.uniform(-0.6, 0.6, 3)
        w = np.exp(a * np.cos(np.pi * x) + b * np.cos(2 * np.pi * x) + c * np.sin(3 * np.pi * x))
        e[j, 1:] = np.cumsum(w) / np.sum(w)
        e[j, -1] = 1.0
    return e


def _flow_params(flow, seed):
    """Parameters of the size a trained flow has, in the logical layout."""
    rng = np.random.default_rng(seed)
    masks = [flow.mask(l) for l in range(flow.n_layers)]
    layout, n = ps.flow_param_layout(flow.dims, flow.n_layers, flow.bins, flow.hidden, masks)
    p = np.zeros(n, dtype=np.float32)
    for lay in layout:
        for name, (o, shape) in lay.items():
            size = int(np.prod(shape))
            if name in ("W1", "W2"):
                v = rng.uniform(-1, 1, size) / math.sqrt(shape[1])
            else:
                v = rng.normal(0, {"W3": 0.05, "b3": 0.2}.get(name, 0.1), size)
            p[o:o + size] = v
    return p


def _weights(n, seed):
    """Event weights as a 2->4 sample has them: a narrow bulk with a tail, a few cut events."""
    g = torch.Generator(device=DEV).manual_seed(seed)
    w = torch.exp(0.35 * torch.randn(n, generator=g, device=DEV, dtype=F64)) * 1.2e-8
    w[torch.rand(n, generator=g, device=DEV) < 1e-3] = 0.0
    return w


def prepare(case, seed):
    kind, n = case["kind"], case["events"]
    s = {"case": case, "seed": seed}
    if kind == "generate":
        chans = _channels(case["set"])
        n_ch, mixed = len(chans), case["precision"] == "mixed"
        prog = ps.program_for(chans, precision=case["precision"], jit=case["jit"],
                              ctas_per_sm=4 if mixed and case["set"] == "2to8" else 0)
        if case["set"] == "2to4":
            prog.set_vegas(0, _grid(seed, 8, 64))
        ev = _split(case["set"], n, n_ch)
        whole = case["store"] == "all"
        out, ws = prog.alloc(ev, chans[0]["n"] + 2 if whole else 0, x=whole and chans[0]["hadronic"],
                             alpha=chans[0]["integrand"] == "pdf_sde")
        if case["store"] == "weights":  # an output that is not given is not written
            out = {k: out[k] for k in ("weight", "alpha")}
        s.update(prog=prog, ev=ev, out=out, ws=ws)
        if case["replay"]:
            s["exec"] = prog.exec_create(ev, out, ws)
    elif kind == "adapt":
        prog = ps.program_for([W.ww_hadronic()], jit=case["jit"])
        prog.set_vegas(0, _grid(seed, 8, 64))
        prog.vegas_training(True)
        out, ws = prog.alloc([n], 6)
        s.update(prog=prog, out=out, ws=ws, done=0)
    elif kind in ("flow", "flow_train"):
        d = W.n_random_dims(W.ww_hadronic())
        flow = ps.Flow(d, case["layers"], case["bins"], 128, max_batch=n if kind == "flow_train" else 1 << 16,
                       init_seed=seed)
        flow.set_params(_flow_params(flow, seed))
        s.update(flow=flow, r=torch.empty((d, n), dtype=F64, device=DEV),
                 logdet=torch.empty(n, dtype=F64, device=DEV))
        if kind == "flow_train":
            prog = ps.program_for([W.ww_hadronic()], jit=True)
            prog.set_vegas(0, _grid(seed, 8, 64))
            s["prog"] = prog
            s["out"], s["ws"] = prog.alloc([n], 6)
    elif kind == "reweight":
        chans = W.multichannel_2to5()
        dens = [dict(c, integrand="none") for c in chans]
        prog, dprog = ps.program_for(chans), ps.program_for(dens, jit=True)
        ev = _reweight_events(case, seed)
        m = len(chans)
        # one workspace per channel; rows of J begin at multiples of 16 bytes, as the map's outputs want
        ws = [dprog.alloc([n if k == j else 0 for k in range(m)], 0, x=False)[1] for j in range(m)]
        s.update(chans=chans, prog=prog, dprog=dprog, mom=ev["momenta"], x1=ev["x1"], x2=ev["x2"], ws=ws,
                 J=torch.empty((m, n + n % 2), dtype=F64, device=DEV)[:, :n],
                 P=torch.empty((m, n), dtype=F64, device=DEV),
                 r=[torch.empty((W.n_random_dims(c), n), dtype=F64, device=DEV) for c in chans],
                 w=torch.empty(n, dtype=F64, device=DEV))
    else:
        s.update(w=_weights(n, seed), u=ps.Unweighter(n), idx=torch.zeros(n, dtype=torch.int64, device=DEV),
                 w_out=torch.zeros(n, dtype=F64, device=DEV))
    return s


def _table(stats):
    return np.array([[c[k] for k in ("n", "n_nonzero", "sum_w", "sum_w2", "max_w")] for c in stats])


def run(s):
    case, seed, n = s["case"], s["seed"], s["case"]["events"]
    kind = case["kind"]
    if kind == "generate":
        if case["replay"]:
            s["exec"].launch(seed)  # a stream of chunks reads its statistics once, at its end
            return s["out"]
        s["prog"].generate(s["ev"], seed, s["out"], s["ws"])
        return {"events": s["out"], "stats": _table(s["prog"].stats())}
    if kind == "adapt":
        s["prog"].generate([n], seed, s["out"], s["ws"], event_offset=s["done"])
        s["done"] += n
        s["prog"].vegas_adapt(0)
        return {"weight": s["out"]["weight"], "grid": s["prog"].get_vegas(0, 8, 64), "stats": _table(s["prog"].stats())}
    if kind == "flow":
        s["flow"].generate(n, seed, s["r"], s["logdet"])
        return {"r": s["r"], "logdet": s["logdet"]}
    if kind == "flow_train":
        s["flow"].sample(n, seed, s["r"], s["logdet"])
        s["prog"].map(0, s["r"], s["out"], s["ws"])
        loss, grads = s["flow"].gradients(s["out"]["weight"])
        return {"r": s["r"], "logdet": s["logdet"], "weight": s["out"]["weight"], "loss": loss, "grads": grads}
    if kind == "reweight":
        m = len(s["chans"])
        for j, ch in enumerate(s["chans"]):
            ps.inverse_map(s["prog"], j, ch, s["mom"], s["x1"], s["x2"], s["r"][j], s["P"][j])
            # the density is all that is wanted of the forward map: only its weight is stored
            s["dprog"].map(j, s["r"][j], {"weight": s["J"][j]}, s["ws"][j])
        ps.global_weights(s["J"], [1.0 / m] * m, s["w"], P=s["P"], x1=s["x1"], x2=s["x2"], pdf=s["chans"][0]["pdf"])
        return {"J": s["J"], "P": s["P"], "w": s["w"]}  # the points r are on the way
    s["u"].max_weight(s["w"], case["eps"])
    s["u"].select(s["w"], seed, s["idx"], s["w_out"])
    return {"max": s["u"].result, "idx": s["idx"], "w": s["w_out"], "n": s["u"].n_accepted}


def work(case):
    kind, n = case["kind"], case["events"]
    if kind == "generate":
        legs = {"2to2": 4, "2to4": 6, "2to5": 7, "2to8": 10}[case["set"]]
        fp = 4 if case["precision"] == "mixed" else 8
        extra = {"2to2": 0, "2to4": 2, "2to5": 3, "2to8": 3}[case["set"]]
        if case["store"] == "weights":
            return {"bytes": n * 16, "flops": n * _OPS[case["set"]]}
        return {"bytes": n * ((4 * legs + extra) * fp + 8), "flops": n * _OPS[case["set"]]}
    if kind == "adapt":
        return {"bytes": n * (6 * 4 + 3) * 8, "flops": n * _OPS["2to4"]}
    d, nets = 10, 0
    for l in range(case.get("layers", 0)):
        nb = len(_mask(d, l))
        nets += 2 * ((d - nb) * 128 + 128 * 128 + 128 * nb * (3 * case["bins"] + 1))
    if kind == "flow":
        return {"bytes": n * (d + 1) * 8, "flops": n * nets}
    if kind == "flow_train":
        return {"bytes": n * (2 * d + 30) * 8, "flops": 3 * n * nets + n * _OPS["2to4"]}
    if kind == "reweight":
        m = 6
        return {"bytes": n * 8 * (30 + m * 2 + 1), "flops": m * n * 2 * 700}
    return {"bytes": n * 8 + 0.2 * n * 16, "flops": 3 * n}


# --------------------------------------------------------------------------------------------
# the methods in 64 bits, from their formulas
# --------------------------------------------------------------------------------------------
def _philox(ev, c2, c3, seed):
    """Philox4x32-10 (Salmon et al., SC'11) on 64-bit integer tensors: the four output words."""
    c = [ev & M32, (ev >> 32) & M32, torch.full_like(ev, c2), torch.full_like(ev, c3)]
    k0, k1 = seed & M32, (seed >> 32) & M32
    for _ in range(10):
        p0, p1 = c[0] * 0xD2511F53, c[2] * 0xCD9E8D57  # the product wraps to its 64 bits
        c = [((p1 >> 32) & M32) ^ c[1] ^ k0, p1 & M32, ((p0 >> 32) & M32) ^ c[3] ^ k1, p0 & M32]
        k0, k1 = (k0 + 0x9E3779B9) & M32, (k1 + 0xBB67AE85) & M32
    return c


def _points(n, first, channel, seed, d, mixed=False):
    """The d uniform numbers of events first .. first+n-1: 52 bits each, 23 in mixed programs."""
    ev = torch.arange(first, first + n, device=DEV, dtype=torch.int64)
    out = []
    for j in range(0, d, 2):
        o = _philox(ev, channel, j // 2, seed)
        for hi, lo in ((o[1], o[0]), (o[3], o[2])):
            if mixed:
                out.append(((hi >> 9).double() + 0.5) * 2.0 ** -23)
            else:
                out.append((((hi << 20) | (lo >> 12)).double() + 0.5) * 2.0 ** -52)
    return out[:d]


def _where(c, a, b):
    return torch.where(c, torch.as_tensor(a, dtype=F64, device=DEV), torch.as_tensor(b, dtype=F64, device=DEV))


def _t(v):
    return torch.as_tensor(v, dtype=F64, device=DEV)


def _map_nu(r, m, nu, lo_, hi_, a):
    lo_, hi_ = _t(lo_), _t(hi_)
    m2 = m * m if m > 0 else -a
    lo, hi, w = lo_ - m2, hi_ - m2, 1.0 - nu
    L = torch.log1p((hi_ - lo_) / lo)
    if nu == 1.0:
        e = torch.expm1(r * L)
        x, jac = lo_ + lo * e, lo * (1 + e) * L
    elif nu < 1.0:
        rho = torch.expm1(w * L)
        z = r * rho
        e = torch.expm1(torch.log1p(z) / w)
        x, jac = lo_ + lo * e, lo * (1 + e) * rho / (w * (1 + z))
    else:
        rho = torch.expm1(-w * L)
        z = (1 - r) * rho
        xm = hi * torch.exp(torch.log1p(z) / w)
        x, jac = m2 + xm, -xm * rho / (w * (1 + z))
    ok = (lo > 0) & (hi >= lo)
    return _where(ok, torch.minimum(torch.maximum(x, lo_), hi_), lo_), _where(ok, jac, 0.0)


def _map_bw(r, M, G, lo_, hi_):
    lo_, hi_ = _t(lo_), _t(hi_)
    mg, m2 = M * G, M * M
    a, b = (lo_ - m2) / mg, (hi_ - m2) / mg
    D = torch.atan2((hi_ - lo_) / mg, 1 + a * b)
    u = torch.atan(a) + D * r
    low, high = u < -math.pi / 4, u > math.pi / 4
    T = torch.tan(_where(low, D * r, _where(high, D * (1 - r), u)))
    den = _where(low, 1 - a * T, _where(high, 1 + b * T, 1.0))
    num = _where(low, T * (1 + a * a), _where(high, b - T, T))
    k = _where(low, 1 + a * a, _where(high, 1 + b * b, 1.0))
    x = _where(low, lo_, m2) + mg * num / den
    jac = D * mg * k * (1 + T * T) / (den * den)
    ok = hi_ >= lo_
    return _where(ok, torch.minimum(torch.maximum(x, lo_), hi_), lo_), _where(ok, jac, 0.0)


def _invariant(r, M, G, nu, lo_, hi_, a):
    return _map_bw(r, M, G, lo_, hi_) if G > 0 else _map_nu(r, M, nu, lo_, hi_, a)


def _kallen(x, y, z):
    """(x - y - z)^2 - 4 y z without cancellation, clamped at zero."""
    x, y, z = torch.broadcast_tensors(_t(x), _t(y), _t(z))
    ry, rz = torch.sqrt(y.clamp(min=0)), torch.sqrt(z.clamp(min=0))
    pos = (x - (ry + rz) ** 2) * (x - (ry - rz) ** 2)
    neg = x * x - 2 * x * (y + z) + (z - y) ** 2
    mix = (x - y - z) ** 2 - 4 * y * z
    return _where((y >= 0) & (z >= 0), pos, _where((y <= 0) & (z <= 0), neg, mix)).clamp(min=0)


def _t_range(s, mA2, mB2, m1, m2):
    m12, m22 = m1 * m1, m2 * m2
    A = mA2 + m12 - (s + mA2 - mB2) * (s + m12 - m22) / (2 * s)
    lam = _kallen(s, mA2, mB2) * ((s - (m1 + m2) ** 2) * (s - (m1 - m2) ** 2)).clamp(min=0)
    B = torch.sqrt(lam) / (2 * s)
    prod = (m12 - mA2) * (m22 - mB2) + (m12 * mB2 - m22 * mA2) * (m12 - m22 - mA2 + mB2) / s
    big = _where(A <= 0, A - B, A + B)
    small = _where(big != 0, prod / _where(big != 0, big, 1.0), 0.0)
    return -_where(A <= 0, small, big), -_where(A <= 0, big, small), B


def _boost(p, q, m, sign):
    """p from the rest frame of q (sign +1), or into it (sign -1); momenta are tuples (E, x, y, z)."""
    qp = q[1] * p[1] + q[2] * p[2] + q[3] * p[3]
    c = qp / (m * (q[0] + m)) + sign * p[0] / m
    return ((q[0] * p[0] + sign * qp) / m, p[1] + q[1] * c, p[2] + q[2] * c, p[3] + q[3] * c)


def _add(a, b, s=1.0):
    return tuple(x + s * y for x, y in zip(a, b))


def _sq(p):
    return p[0] * p[0] - p[1] * p[1] - p[2] * p[2] - p[3] * p[3]


def _axis(a):
    """cos, sin of the polar angle and of the azimuth of a three-momentum."""
    pt = torch.sqrt(a[1] * a[1] + a[2] * a[2])
    p = torch.sqrt(pt * pt + a[3] * a[3])
    on = pt > 0
    ipt = 1 / _where(on, pt, 1.0)
    return a[3] / p, pt / p, _where(on, a[1] * ipt, 1.0), _where(on, a[2] * ipt, 0.0)


def _two_to_two(rphi, pA, pB, tabs, m1, m2, s, mA2, mB2):
    p0, m0 = _add(pA, pB), torch.sqrt(s)
    cA, sA, cp, sp = _axis(_boost(pA, p0, m0, -1))
    lo, hi, B = _t_range(s, mA2, mB2, m1, m2)
    near = tabs - lo <= hi - tabs
    f = _where(B > 0, _where(near, tabs - lo, hi - tabs) / _where(B > 0, B, 1.0), 1.0)
    omc, opc = _where(near, f, 2 - f), _where(near, 2 - f, f)
    cth, sth = _where(omc <= opc, 1 - omc, opc - 1), torch.sqrt((omc * opc).clamp(min=0))
    phi = 2 * math.pi * rphi
    lam = ((s - (m1 + m2) ** 2) * (s - (m1 - m2) ** 2)).clamp(min=0)
    p = torch.sqrt(lam) / (2 * m0)
    e1, e2 = (s + m1 * m1 - m2 * m2) / (2 * m0), (s + m2 * m2 - m1 * m1) / (2 * m0)
    vx, vy, vz = p * sth * torch.cos(phi), p * sth * torch.sin(phi), p * cth
    rx, rz = cA * vx + sA * vz, -sA * vx + cA * vz
    q1 = (e1, cp * rx - sp * vy, sp * rx + cp * vy, rz)
    q2 = (e2, -q1[1], -q1[2], -q1[3])
    return _boost(q1, p0, m0, 1), _boost(q2, p0, m0, 1), 0.5 * math.pi / torch.sqrt(_kallen(s, mA2, mB2))


def _two_body(rphi, rth, s0, m1, m2, p0):
    m0 = torch.sqrt(s0)
    lam = ((s0 - (m1 + m2) ** 2) * (s0 - (m1 - m2) ** 2)).clamp(min=0)
    sl = torch.sqrt(lam)
    p = sl / (2 * m0)
    cth, sth, phi = 2 * rth - 1, 2 * torch.sqrt(rth * (1 - rth)), 2 * math.pi * rphi
    q1 = ((s0 + m1 * m1 - m2 * m2) / (2 * m0), p * sth * torch.cos(phi), p * sth * torch.sin(phi), p * cth)
    q2 = ((s0 + m2 * m2 - m1 * m1) / (2 * m0), -q1[1], -q1[2], -q1[3])
    if p0 is not None:
        q1, q2 = _boost(q1, p0, m0, 1), _boost(q2, p0, m0, 1)
    return q1, q2, 0.5 * math.pi * sl / s0


class _Topo:
    """A channel's tree: leaves, parents, t-chain order and the layout of its random dimensions."""

    def __init__(self, ch):
        self.ch, self.nd = ch, ch["nodes"]
        self.parent = {k: j for j, nd in enumerate(self.nd) for k in nd.get("children", [])}
        self.leaves = [self._leaves(j) for j in range(len(self.nd))]
        root = self.nd[0]
        self.kappa = len(root["children"]) - 1 if root["kind"] == "tchain" else 0
        self.pre = [j for j in self._walk(0) if self.nd[j]["kind"] == "decay"]
        left, right, self.order = 0, self.kappa, {}
        for i in range(1, self.kappa):
            if ch["tside"][i - 1] == 0:
                self.order[i], left = left, left + 1
            else:
                self.order[i], right = right, right - 1
        self.order[self.kappa], self.order[self.kappa + 1] = left, right
        names = ["shat"] if ch["hadronic"] else []
        names += [("s", j) for j in ch["sorder"]] + [("ts", i) for i in range(1, self.kappa)]
        names += ["x"] if ch["hadronic"] else []
        for i in range(1, self.kappa + 1):
            names += [("tphi", i), ("tt", i)]
        for j in self.pre:
            names += [("phi", j), ("th", j)]
        self.dim = {k: i for i, k in enumerate(names)}

    def _walk(self, j):
        yield j
        for c in self.nd[j].get("children", []):
            yield from self._walk(c)

    def _leaves(self, j):
        if self.nd[j]["kind"] == "leaf":
            return [self.nd[j]["leaf"]]
        return [x for c in self.nd[j]["children"] for x in self._leaves(c)]

    def bounds(self, j, s, known):
        """Smallest and largest mass of node j given the invariants sampled before it."""
        def least(k):
            if self.nd[k]["kind"] == "leaf":
                return _t(self.nd[k]["mass"])
            if k in known:
                return torch.sqrt(s[k])
            return sum(least(c) for c in self.nd[k]["children"])

        off, cur = _t(0.0), j
        while True:
            p = self.parent[cur]
            off = off + sum(least(c) for c in self.nd[p]["children"] if c != cur)
            if p in known:
                break
            cur = p
        lo = least(j)
        return lo, torch.maximum(torch.sqrt(s[p]) - off, lo)

    def props(self):
        """Propagators of the SDE weight: ("s", leaves, M, G), ("t", leaves of the legs before it, M)."""
        out = [("s", self.leaves[j], nd["M"], nd["G"]) for j, nd in enumerate(self.nd)
               if j and nd["kind"] == "decay" and nd["sde"]]
        legs = self.nd[0]["children"]
        for k in range(self.kappa):
            out.append(("t", [x for c in legs[:k + 1] for x in self.leaves[c]], self.ch["Mt"], 0.0))
        return out

    def mass(self, j, s):
        return _t(self.nd[j]["mass"]) if self.nd[j]["kind"] == "leaf" else torch.sqrt(s[j])


def _sde(props, rec):
    """Product of propagators of one channel from the event record [p_a, p_b, p_1 ..]."""
    P = 1.0
    for kind, legs, M, G in props:
        q = rec[0] if kind == "t" else tuple(torch.zeros_like(c) for c in rec[0])
        for i in legs:
            q = _add(q, rec[2 + i], -1.0 if kind == "t" else 1.0)
        P = P / ((_sq(q) - M * M) ** 2 + (M * G) ** 2)
    return P


def _forward(chans, which, r, grid=None):
    """The channel map of points r (a list of tensors): event record, x1, x2, weight, alpha."""
    ch = chans[which]
    T = _Topo(ch)
    nd, D = T.nd, T.dim
    r = [x if torch.is_tensor(x) else _t(x) for x in r]
    n = ch["n"]
    w = torch.full_like(r[0], (2 * math.pi) ** (4 - 3 * n))
    if ch["vegas_dims"]:
        nb = ch["vegas_bins"]
        for j in range(ch["vegas_dims"]):
            e = _t(np.arange(nb + 1) / nb if grid is None else grid[j])
            y = r[j] * nb
            k = y.long().clamp(0, nb - 1)
            wd = e[k + 1] - e[k]
            r[j] = e[k] + (y - k) * wd
            w = w * (nb * wd)
    s, known, P = {}, {0}, 1.0
    if ch["hadronic"]:
        m = sum(x["mass"] for x in nd if x["kind"] == "leaf")
        sh = ch["shat"]
        s[0], j = _invariant(r[D["shat"]], sh["M"], sh["G"], sh["nu"], m * m, ch["S"], ch["a"])
        w = w * j
    else:
        s[0] = torch.full_like(r[0], ch["sqrt_s"] ** 2)
    for j in ch["sorder"]:
        lo, hi = T.bounds(j, s, known)
        s[j], jac = _invariant(r[D[("s", j)]], nd[j]["M"], nd[j]["G"], nd[j]["nu"], lo * lo, hi * hi, ch["a"])
        known.add(j)
        w = w * jac
        if nd[j]["sde"]:
            P = P / ((s[j] - nd[j]["M"] ** 2) ** 2 + (nd[j]["M"] * nd[j]["G"]) ** 2)
    legs, kappa, st = nd[0]["children"], T.kappa, {0: s[0]}
    left, right = 0, kappa
    for i in range(1, kappa):
        if ch["tside"][i - 1] == 0:
            left += 1
        else:
            right -= 1
        lo = sum(T.mass(legs[k], s) for k in range(left, right + 1)) ** 2
        hi = torch.maximum((torch.sqrt(st[i - 1]) - T.mass(legs[T.order[i]], s)).clamp(min=0) ** 2, lo)
        st[i], jac = _map_nu(r[D[("ts", i)]], 0.0, ch["ts_nu"], lo, hi, ch["a"])
        w = w * jac
    x1 = x2 = None
    if ch["hadronic"]:
        tau = s[0] / ch["S"]
        L = torch.log(tau)
        x1 = torch.exp(r[D["x"]] * L)
        x2 = tau / x1
        w = w * (-L / ch["S"])
    h, zero = 0.5 * torch.sqrt(s[0]), torch.zeros_like(s[0])
    pa, pb = (h, zero, zero, h), (h, zero, zero, -h)
    mom = {}
    pA, pB, mA2, mB2, cur = pa, pb, zero, zero, s[0]
    for i in range(1, kappa + 1):
        side = ch["tside"][i - 1] if i < kappa else 0
        l1 = legs[T.order[i]]
        m1 = T.mass(l1, s)
        m2 = T.mass(legs[T.order[i + 1]], s) if i == kappa else torch.sqrt(st[i])
        if i < kappa and side == 1:
            m1, m2 = m2, m1
        lo, hi, _ = _t_range(cur, mA2, mB2, m1, m2)
        lo = lo.clamp(min=0)
        t, jt = _map_nu(r[D[("tt", i)]], 0.0, ch["t_nu"], lo, torch.maximum(hi, lo), ch["a"])
        q1, q2, jb = _two_to_two(r[D[("tphi", i)]], pA, pB, t, m1, m2, cur, mA2, mB2)
        w = w * (jt * jb)
        P = P / ((t + ch["Mt"] ** 2) ** 2)
        if i == kappa:
            mom[l1], mom[legs[T.order[i + 1]]] = q1, q2
        elif side == 0:
            mom[l1], pA, mA2, cur = q1, _add(pA, q1, -1.0), -t, st[i]
        else:
            mom[l1], pB, mB2, cur = q2, _add(pB, q2, -1.0), -t, st[i]
    for j in T.pre:
        c1, c2 = nd[j]["children"]
        mom[c1], mom[c2], jac = _two_body(r[D[("phi", j)]], r[D[("th", j)]], s[j], T.mass(c1, s), T.mass(c2, s),
                                          None if j == 0 else mom[j])
        w = w * jac
    rec = [pa, pb] + [None] * n
    for j, x in enumerate(nd):
        if x["kind"] == "leaf":
            rec[2 + x["leaf"]] = mom[j]
    if ch["hadronic"]:
        rho = torch.sqrt(x1 / x2)
        rec = [(0.5 * (rho * (p[0] + p[3]) + (p[0] - p[3]) / rho), p[1], p[2],
                0.5 * (rho * (p[0] + p[3]) - (p[0] - p[3]) / rho)) for p in rec]
    alpha = None
    a, b = ch["pdf"]
    if ch["integrand"] == "one_plus_cos2":
        p = rec[2]
        w = w * (1 + p[3] ** 2 / (p[1] ** 2 + p[2] ** 2 + p[3] ** 2))
    elif ch["integrand"] == "pdf_props":
        w = w * P * tau ** a * ((1 - x1) * (1 - x2)) ** b
    elif ch["integrand"] == "pdf_sde":
        tot = P
        for c, other in enumerate(chans):
            if c != which:
                tot = tot + _sde(_Topo(other).props(), rec)
        alpha = P / tot
        w = w * P * tau ** a * ((1 - x1) * (1 - x2)) ** b
    bad = ~torch.isfinite(w)
    for p in rec:
        for c in p:
            bad = bad | ~torch.isfinite(c)
    if x1 is not None:
        bad = bad | ~((x1 > 0) & (x1 <= 1) & (x2 > 0) & (x2 <= 1))
    return rec, x1, x2, _where(bad, 0.0, w), alpha


def _stats(w):
    return {"n": float(w.numel()), "n_nonzero": float((w != 0).sum()), "sum_w": float(w.sum()),
            "sum_w2": float((w * w).sum()), "max_w": float(w.max().clamp(min=0)) if w.numel() else 0.0}


def _rows(rec):
    return torch.stack([c for p in rec for c in p])


def _exact_generate(case, seed):
    chans = _channels(case["set"])
    ev = _split(case["set"], case["events"], len(chans))
    mixed = case["precision"] == "mixed"
    mom, x1, x2, w, al, stats = [], [], [], [], [], []
    for c, ch in enumerate(chans):
        grid = _grid(seed, 8, 64) if case["set"] == "2to4" else None
        d = len(_Topo(ch).dim)
        rows = [[], [], [], [], []]
        for lo in range(0, ev[c], 1 << 21):
            m = min(1 << 21, ev[c] - lo)
            got = _forward(chans, c, _points(m, lo, c, seed, d, mixed), grid)
            for k, v in enumerate((_rows(got[0]),) + got[1:]):
                if v is not None:
                    rows[k].append(v.float() if mixed and k != 3 else v)
        cat = [torch.cat(v, dim=-1) if v else None for v in rows]
        for to, v in zip((mom, x1, x2, w, al), cat):
            if v is not None:
                to.append(v)
        stats.append(_stats(cat[3]) if cat[3] is not None else
                     {"n": 0.0, "n_nonzero": 0.0, "sum_w": 0.0, "sum_w2": 0.0, "max_w": 0.0})
    out = {"weight": torch.cat(w)}
    for k, v in (("momenta", mom), ("x1", x1), ("x2", x2), ("alpha", al)):
        if v and (case["store"] == "all" or k == "alpha"):
            out[k] = torch.cat(v, dim=-1)
    return out if case["replay"] else {"events": out, "stats": _table(stats)}


def _rebin(h, e, alpha):
    """Lepage's refinement of one row of edges from its importance histogram."""
    n = len(h)
    imp = np.array([np.mean(h[max(k - 1, 0):k + 2]) for k in range(n)])
    if not imp.sum() > 0:
        return e.copy()
    d = imp / imp.sum()
    m = np.zeros(n)
    on = (d > 0) & (d < 1)
    m[on] = ((1 - d[on]) / -np.log(d[on])) ** alpha
    m[d >= 1] = 1.0
    cum = np.concatenate([[0.0], np.cumsum(m)])
    out = np.interp(cum[-1] * np.arange(n + 1) / n, cum, e)
    out[0], out[-1] = e[0], e[-1]
    return out


def _exact_adapt(case, seed):
    ch, n, grid = W.ww_hadronic(), case["events"], _grid(seed, 8, 64)
    r = _points(n, 0, 0, seed, 10)
    w = _forward([ch], 0, list(r), grid)[3]
    new = np.zeros_like(grid)
    for j in range(8):
        k = (r[j] * 64).long().clamp(0, 63)
        h = torch.zeros(64, dtype=F64, device=DEV).index_add_(0, k, w * w).cpu().numpy()
        new[j] = _rebin(h, grid[j], 1.5)
    return {"weight": w, "grid": new, "stats": _table([_stats(w)])}


def _mask(d, layer):
    """Transformed dims of a coupling layer (d <= 16): one bit of the dim index, flipped in turn."""
    nb = max(1, math.ceil(math.log2(d)))
    return [j for j in range(d) if ((j >> (layer % nb)) & 1) != (layer // nb) % 2]


def _flow_layers(case, seed):
    class Shape:  # what _flow_params reads of a flow
        dims, n_layers, bins, hidden = 10, case["layers"], case["bins"], 128
        mask = staticmethod(lambda l: _mask(10, l))

    p = torch.as_tensor(_flow_params(Shape, seed), device=DEV).double()
    return p, Shape


def _net(p, o, shape):
    size = shape[0] * (shape[1] if len(shape) > 1 else 1)
    return p[o:o + size].reshape(shape)


def _unpack(p, d, layer, o, K, H):
    """Weights of one layer from offset o: W1, b1, W2, b2, W3, b3; and the next offset."""
    nb = len(_mask(d, layer))
    got = []
    for shape in ((H, d - nb), (H,), (H, H), (H,), (nb * (3 * K + 1), H), (nb * (3 * K + 1),)):
        got.append(_net(p, o, shape))
        o += math.prod(shape)
    return got, o


def _spline_params(x, net, nb, K):
    W1, b1, W2, b2, W3, b3 = net
    silu = torch.nn.functional.silu
    raw = (silu(silu(x @ W1.T + b1) @ W2.T + b2) @ W3.T + b3).reshape(x.shape[0], nb, 3 * K + 1)
    w = 1e-3 + (1 - K * 1e-3) * torch.softmax(raw[..., :K], -1)
    h = 1e-3 + (1 - K * 1e-3) * torch.softmax(raw[..., K:2 * K], -1)
    return w, h, 1e-3 + torch.nn.functional.softplus(raw[..., 2 * K:])


def _bin(v, w, h, dv, of_x):
    xk, yk = torch.cumsum(w, -1) - w, torch.cumsum(h, -1) - h
    k = ((v.unsqueeze(-1) >= (xk if of_x else yk)).sum(-1) - 1).clamp(0, w.shape[-1] - 1)
    g = lambda t, i: torch.gather(t, -1, i.unsqueeze(-1)).squeeze(-1)
    return g(xk, k), g(w, k), g(yk, k), g(h, k), g(dv, k), g(dv, k + 1)


def _rq(x, par):
    """Rational-quadratic spline (Durkan et al. 2019) of x in its bin: y and dy/dx."""
    x0, wk, y0, hk, d0, d1 = par
    xi, s = (x - x0) / wk, hk / wk
    om = xi * (1 - xi)
    den = s + (d1 + d0 - 2 * s) * om
    return y0 + hk * (s * xi * xi + d0 * om) / den, s * s * (d1 * xi * xi + 2 * s * om + d0 * (1 - xi) ** 2) / den ** 2


def _flow_forward(p, z, layers, K):
    x, ld, o = z.clone(), torch.zeros(z.shape[0], dtype=F64, device=DEV), 0
    d = z.shape[1]
    for l in range(layers):
        tb = _mask(d, l)
        ta = [j for j in range(d) if j not in tb]
        net, o = _unpack(p, d, l, o, K, 128)
        w, h, dv = _spline_params(x[:, ta], net, len(tb), K)
        y, dy = _rq(x[:, tb], _bin(x[:, tb], w, h, dv, True))
        x = x.clone()
        x[:, tb] = y
        ld = ld + torch.log(dy).sum(1)
    return x, ld


def _flow_logq(p, r, layers, K):
    """log g(r) = -log |dr/dz| by the inverse flow, differentiable in p."""
    d, offs, o = r.shape[1], [], 0
    for l in range(layers):
        net, o = _unpack(p, d, l, o, K, 128)
        offs.append(net)
    x, lq = r, 0.0
    for l in reversed(range(layers)):
        tb = _mask(d, l)
        ta = [j for j in range(d) if j not in tb]
        w, h, dv = _spline_params(x[:, ta], offs[l], len(tb), K)
        y = x[:, tb]
        par = _bin(y, w, h, dv, False)
        x0, wk, y0, hk, d0, d1 = par
        s, dy = hk / wk, y - y0
        a = hk * (s - d0) + dy * (d1 + d0 - 2 * s)
        b = hk * d0 - dy * (d1 + d0 - 2 * s)
        c = -s * dy
        xb = x0 + wk * 2 * c / (-b - torch.sqrt(b * b - 4 * a * c))
        lq = lq - torch.log(_rq(xb, par)[1]).sum(1)
        x = x.clone()
        x[:, tb] = xb
    return lq


def _flow_points(case, seed):
    n, d = case["events"], 10
    ev = torch.arange(n, device=DEV, dtype=torch.int64)
    z = []
    for i in range(d // 2):
        o = _philox(ev, 0x466C6F77, i, seed)
        z += [((o[k] >> 9).double() + 0.5) * 2.0 ** -23 for k in (0, 1)]
    p, _ = _flow_layers(case, seed)
    z = torch.stack(z, 1)
    r, ld = [], []
    for lo in range(0, n, 1 << 17):
        a, b = _flow_forward(p, z[lo:lo + (1 << 17)], case["layers"], case["bins"])
        r.append(a.clamp(1e-7, 1 - 1e-7))
        ld.append(b)
    return p, torch.cat(r), torch.cat(ld)


def _exact_flow(case, seed):
    _, r, ld = _flow_points(case, seed)
    return {"r": r.T.contiguous(), "logdet": ld}


def _exact_flow_train(case, seed):
    p, r, ld = _flow_points(case, seed)
    w_map = _forward([W.ww_hadronic()], 0, list(r.T.contiguous()), _grid(seed, 8, 64))[3]
    w = w_map * torch.exp(ld)
    p.requires_grad_(True)
    tot, loss = w.sum(), 0.0
    for lo in range(0, r.shape[0], 1 << 14):
        part = -(w[lo:lo + (1 << 14)] / tot * _flow_logq(p, r[lo:lo + (1 << 14)], case["layers"], case["bins"])).sum()
        part.backward()
        loss += float(part.detach())
    return {"r": r.T.contiguous(), "logdet": ld, "weight": w_map, "loss": loss, "grads": p.grad}


def _inv_nu(x, m, nu, lo_, hi_, a):
    lo_, hi_ = _t(lo_), _t(hi_)
    m2 = m * m if m > 0 else -a
    lo, hi, w = lo_ - m2, hi_ - m2, 1.0 - nu
    L, l = torch.log1p((hi_ - lo_) / lo), torch.log1p((x - lo_) / lo)
    if nu == 1.0:
        return l / L
    if nu < 1.0:
        return torch.expm1(w * l) / torch.expm1(w * L)
    return 1 - torch.expm1(w * torch.log((x - m2) / hi)) / torch.expm1(-w * L)


def _inv_bw(x, M, G, lo_, hi_):
    lo_, hi_ = _t(lo_), _t(hi_)
    mg, m2 = M * G, M * M
    a, b, t = (lo_ - m2) / mg, (hi_ - m2) / mg, (x - m2) / mg
    D = torch.atan2((hi_ - lo_) / mg, 1 + a * b)
    return _where(x - lo_ <= hi_ - x, torch.atan2((x - lo_) / mg, 1 + a * t) / D,
                  1 - torch.atan2((hi_ - x) / mg, 1 + b * t) / D)


def _inv_invariant(x, M, G, nu, lo_, hi_, a):
    return _inv_bw(x, M, G, lo_, hi_) if G > 0 else _inv_nu(x, M, nu, lo_, hi_, a)


def _turn(y, x):
    ph = torch.atan2(y, x) / (2 * math.pi)
    return _where(ph < 0, ph + 1, ph)


def _inverse(ch, rec, x1, x2):
    """The random numbers that the channel maps to an event record in the lab frame."""
    T = _Topo(ch)
    nd, D, n = T.nd, T.dim, ch["n"]
    rho = torch.sqrt(x1 / x2)
    q = [(0.5 * ((p[0] + p[3]) / rho + rho * (p[0] - p[3])), p[1], p[2],
          0.5 * ((p[0] + p[3]) / rho - rho * (p[0] - p[3]))) for p in rec]
    ml = {x["leaf"]: x["mass"] for x in nd if x["kind"] == "leaf"}
    ap = [torch.sqrt(p[1] ** 2 + p[2] ** 2 + p[3] ** 2) for p in q[2:]]
    dirs = [(p[1] / a, p[2] / a, p[3] / a) for p, a in zip(q[2:], ap)]
    pn, s, r = {}, {}, [None] * len(D)
    for j, x in enumerate(nd):
        if j == 0:
            continue
        acc, s2 = None, 0.0
        for u, i in enumerate(T.leaves[j]):
            acc = q[2 + i] if acc is None else _add(acc, q[2 + i])
            s2 = s2 + ml[i] ** 2
            for k in T.leaves[j][u + 1:]:
                d2 = sum((a - b) ** 2 for a, b in zip(dirs[i], dirs[k]))
                s2 = s2 + 2 * (ml[i] ** 2 * ap[k] ** 2 + ml[k] ** 2 * ap[i] ** 2 + ml[i] ** 2 * ml[k] ** 2) / (
                    q[2 + i][0] * q[2 + k][0] + ap[i] * ap[k]) + ap[i] * ap[k] * d2
        pn[j], s[j] = acc, s2 if x["kind"] == "decay" else _t(x["mass"] ** 2)
    s[0] = x1 * x2 * ch["S"]
    m, sh = sum(ml.values()), ch["shat"]
    r[D["shat"]] = _inv_invariant(s[0], sh["M"], sh["G"], sh["nu"], m * m, ch["S"], ch["a"])
    r[D["x"]] = torch.log(x1) / torch.log(s[0] / ch["S"])
    known = {0}
    for j in ch["sorder"]:
        lo, hi = T.bounds(j, s, known)
        known.add(j)
        r[D[("s", j)]] = _inv_invariant(s[j], nd[j]["M"], nd[j]["G"], nd[j]["nu"], lo * lo, hi * hi, ch["a"])
    legs, kappa, st = nd[0]["children"], T.kappa, {0: s[0]}
    left, right = 0, kappa
    for i in range(1, kappa):
        if ch["tside"][i - 1] == 0:
            left += 1
        else:
            right -= 1
        c = pn[legs[left]]
        for k in range(left + 1, right + 1):
            c = _add(c, pn[legs[k]])
        lo = sum(T.mass(legs[k], s) for k in range(left, right + 1)) ** 2
        st[i] = _sq(c)
        hi = torch.maximum((torch.sqrt(st[i - 1]) - T.mass(legs[T.order[i]], s)).clamp(min=0) ** 2, lo)
        r[D[("ts", i)]] = _inv_nu(st[i], 0.0, ch["ts_nu"], lo, hi, ch["a"])
    h, zero = 0.5 * torch.sqrt(s[0]), torch.zeros_like(s[0])
    pA, pB, mA2, mB2, cur = (h, zero, zero, h), (h, zero, zero, -h), zero, zero, s[0]
    for i in range(1, kappa + 1):
        side = ch["tside"][i - 1] if i < kappa else 0
        leg = legs[T.order[i]]
        m1 = T.mass(leg, s)
        m2 = T.mass(legs[T.order[i + 1]], s) if i == kappa else torch.sqrt(st[i])
        q1 = pn[leg]
        if i < kappa and side == 1:
            m1, m2 = m2, m1
            q1 = _add(_add(pA, pB), pn[leg], -1.0)
        t = -_sq(_add(pA, q1, -1.0))
        lo, hi, _ = _t_range(cur, mA2, mB2, m1, m2)
        lo = lo.clamp(min=0)
        r[D[("tt", i)]] = _inv_nu(t, 0.0, ch["t_nu"], lo, torch.maximum(hi, lo), ch["a"])
        p0, m0 = _add(pA, pB), torch.sqrt(cur)
        cA, sA, cp, sp = _axis(_boost(pA, p0, m0, -1))
        b = _boost(q1, p0, m0, -1)
        v1, v2 = cp * b[1] + sp * b[2], -sp * b[1] + cp * b[2]
        r[D[("tphi", i)]] = _turn(v2, cA * v1 - sA * b[3])
        if i < kappa and side == 0:
            pA, mA2, cur = _add(pA, q1, -1.0), -t, st[i]
        elif i < kappa:
            pB, mB2, cur = _add(pB, pn[leg], -1.0), -t, st[i]
    for j in T.pre:
        c1 = nd[j]["children"][0]
        b = pn[c1] if j == 0 else _boost(pn[c1], pn[j], torch.sqrt(s[j]), -1)
        pt2 = b[1] ** 2 + b[2] ** 2
        pa = torch.sqrt(pt2 + b[3] ** 2)
        up = b[3] >= 0
        half = 0.5 * pt2 / (pa * (pa + b[3].abs()))
        r[D[("th", j)]] = _where(up, 1 - half, half)
        r[D[("phi", j)]] = _turn(b[2], b[1])
    return r


@lru_cache(maxsize=1)
def _reweight_record(n, channel, seed):
    chans = W.multichannel_2to5()
    d = len(_Topo(chans[channel]).dim)
    return _forward(chans, channel, _points(n, 0, channel, seed, d))[:3]


def _reweight_events(case, seed):
    """Events of one channel of the 2->5 set, as a file of events would hold them."""
    rec, x1, x2 = _reweight_record(case["events"], case["channel"], seed)
    return {"momenta": _rows(rec), "x1": x1.clone(), "x2": x2.clone()}


def _exact_reweight(case, seed):
    chans = W.multichannel_2to5()
    rec, x1, x2 = _reweight_record(case["events"], case["channel"], seed)
    J, P = [], []
    for j, ch in enumerate(chans):
        r = _inverse(ch, rec, x1, x2)
        J.append(_forward([dict(ch, integrand="none")], 0, r)[3])
        P.append(_sde(_Topo(ch).props(), rec))
    J, P = torch.stack(J), torch.stack(P)
    g = (_where(J > 0, 1 / _where(J > 0, J, 1.0), 0.0) / len(chans)).sum(0)
    a, b = chans[0]["pdf"]
    f = P.sum(0) * (x1 * x2) ** a * ((1 - x1) * (1 - x2)) ** b
    return {"J": J, "P": P, "w": _where(g > 0, f / _where(g > 0, g, 1.0), 0.0)}


def _exact_unweight(case, seed):
    n, eps = case["events"], case["eps"]
    w = _weights(n, seed)
    v = torch.sort(w, descending=True).values
    S = v.sum()
    cum = torch.cumsum(v, 0)
    k = torch.arange(1, n + 1, device=DEV, dtype=F64)
    t = float(v[0])
    if eps > 0:
        # the excess over t = v[k] is cum[k-1] - k v[k]: the root lies below the last one not above eps S
        over = cum[:-1] - k[:-1] * v[1:]
        m = int((over <= eps * S).sum())
        t = float((cum[m] - eps * S) / (m + 1)) if m < n else 0.0
    ev = torch.arange(n, device=DEV, dtype=torch.int64)
    o = _philox(ev, 0x556E7700, 0, seed)
    u = (((o[1] << 20) | (o[0] >> 12)).double() + 0.5) * 2.0 ** -52
    keep = torch.nonzero(u * t < w).squeeze(1)
    out = torch.zeros(n, dtype=F64, device=DEV)
    out[:keep.numel()] = w[keep].clamp(min=t)
    return {"max": torch.tensor([t, float(S), float(v[0]), float((w > t).sum()), 0.0], dtype=F64), "idx": None,
            "w": out, "n": None}


def exact(case, seed):
    return {"generate": _exact_generate, "adapt": _exact_adapt, "flow": _exact_flow, "flow_train": _exact_flow_train,
            "reweight": _exact_reweight, "unweight": _exact_unweight}[case["kind"]](case, seed)
