"""The calls of this framework whose speed is measured: Monte Carlo prices and
pathwise sensitivities under a bilinear local-volatility grid, each through the
entry point a program calls. Inputs come from a seed; ``exact`` restates the
estimators in plain torch, in 64 bits, path for path on the same counters.
"""
import math

import numpy as np
import torch

from paper_2002_02481_gb300 import lv
from paper_2002_02481_gb300.autograd import lv_price

# Path-steps (paths x time steps) up to which the 64-bit restatement stays
# well under 20 seconds.
EXACT_PATH_STEPS = 1.4e9


def listed():
    small = dict(grid="skew", n_spot=20, n_time=10, s_lo=50.0, s_hi=200.0, t_hi=1.0, T=1.0, r=0.0, phi=1)
    paper = dict(grid="skew", n_spot=30, n_time=60, s_lo=20.0, s_hi=300.0, t_hi=3.0, T=3.0, r=0.0, phi=1)
    return [
        # a quote: one option priced and read back, the smallest call (latency and launches count)
        dict(name="price_small", kind="price", n_steps=52, n_paths=16384, **small),
        # its hedge: the price, delta and 200 vega buckets of the same option
        dict(name="greeks_small", kind="greeks", n_steps=52, n_paths=16384, **small),
        # one step of a fit through torch.autograd: forward and backward on a float32 grid
        dict(name="autograd_step", kind="autograd", n_steps=156, n_paths=65536, **paper),
        # the paper's own run: 1,800 vegas on 500,000 paths, a recalibrated grid in, results on the host
        dict(name="greeks_500k", kind="recalibrated", n_steps=156, n_paths=500000, **paper),
        # the benchmark's run: results stay on the device
        dict(name="greeks_1m", kind="greeks_device", n_steps=156, n_paths=1 << 20, **paper),
        # forward-only pricing at the benchmark's size
        dict(name="price_1m", kind="price", n_steps=156, n_paths=1 << 20, **paper),
        # a put under the other readings: Euler on S, spot weight linear in ln S
        dict(name="greeks_euler_s", kind="greeks_device", n_steps=156, n_paths=300001, interp=1, scheme=1,
             **{**paper, "phi": -1, "r": 0.02}),
        # end-of-day sensitivities of a put with rho and the maturity sensitivity
        dict(name="greeks_ext", kind="ext", n_steps=156, n_paths=1 << 19, **{**paper, "phi": -1, "r": 0.03}),
        # second-order buckets for a vega hedge's delta
        dict(name="vanna_1m", kind="vanna", n_steps=156, n_paths=1 << 20, **paper),
        # the binary64 run that states the other calls' rounding
        dict(name="greeks_fp64", kind="fp64", n_steps=156, n_paths=1 << 16, **paper),
        # a desk: 8 surfaces x 64 options, aggregated risk per surface
        dict(name="book_risk", kind="book_risk", n_surf=8, per_surface=64, log2_lo=14.0, log2_hi=20.0, r=0.01,
             **{k: paper[k] for k in ("grid", "n_spot", "n_time", "s_lo", "s_hi", "t_hi")}),
        # a long-dated option on a fine grid with daily steps: the largest call
        dict(name="greeks_large", kind="greeks", grid="skew", n_spot=100, n_time=100, s_lo=20.0, s_hi=300.0, t_hi=5.0,
             T=5.0, r=0.0, phi=1, n_steps=1260, n_paths=1 << 26),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["price", "greeks", "greeks", "greeks_device", "recalibrated", "autograd", "ext", "vanna", "fp64",
                       "book", "book_risk", "tangent", "kahan"])
    c = dict(kind=kind, grid=rng.choice(["skew", "skew", "uneven"]), n_spot=_log_int(rng, 5, 100),
             n_time=_log_int(rng, 2, 100), r=rng.choice([0.0, 0.01, 0.03]))
    c["t_hi"] = rng.choice([1.0, 3.0, 5.0])
    c["s_lo"], c["s_hi"] = rng.choice([(50.0, 200.0), (20.0, 300.0)])
    if kind in ("book", "book_risk"):
        c.update(n_surf=rng.randint(1, 8), per_surface=rng.randint(2, 24), log2_lo=rng.uniform(10.0, 14.0),
                 log2_hi=rng.uniform(14.5, 18.0))
        return c
    c.update(T=c["t_hi"] * rng.choice([1.0, 0.5, 0.9]), phi=rng.choice([1, -1]), n_steps=_log_int(rng, 12, 1260))
    if kind in ("price", "greeks", "greeks_device", "recalibrated", "ext", "kahan"):
        c.update(interp=rng.choice([0, 0, 1]), scheme=rng.choice([0, 0, 1]))
    most = {"fp64": 4e7, "autograd": 4e8}.get(kind, 4e9)
    c["n_paths"] = max(1, min(_log_int(rng, 1 << 11, 1 << 22) - rng.randint(0, 37), int(most / c["n_steps"])))
    return c


# ------------------------------------------------------------------ inputs

def _grid(case, rng):
    """Spot nodes, time nodes and sigma: a seeded smooth skew on log-spaced
    nodes, or the same skew on irregular ones."""
    I, J = case["n_spot"], case["n_time"]
    base, slope = rng.uniform(0.15, 0.30), rng.uniform(-0.15, -0.05)
    if case["grid"] == "uneven":
        gaps = rng.uniform(0.4, 1.6, size=I - 1)
        x = np.concatenate([[0.0], np.cumsum(gaps)]) / gaps.sum()
        gaps = rng.uniform(0.4, 1.6, size=J - 1)
        t = case["t_hi"] * np.concatenate([[0.0], np.cumsum(gaps)]) / gaps.sum()
    else:
        x = np.arange(I, dtype=np.float64) / (I - 1)
        t = np.linspace(0.0, case["t_hi"], J)
    s = case["s_lo"] * (case["s_hi"] / case["s_lo"]) ** x
    sig = base + slope * np.log(s[:, None] / 100.0) + 0.02 * t[None, :] + rng.normal(0.0, 0.005, size=(I, J))
    return s, t, np.clip(sig, 0.05, 0.6)


def _inputs(case, seed):
    """Host-side inputs of a case: surfaces, options and the Monte Carlo seed."""
    rng = np.random.Generator(np.random.PCG64(seed))
    d = dict(seed=int(rng.integers(1, 1 << 62)), S0=float(rng.uniform(95.0, 105.0)))
    if case["kind"] in ("book", "book_risk"):
        d["surfs"] = [_grid(case, rng) for _ in range(case["n_surf"])]
        mats = [m for m in (0.25, 0.5, 1.0, 2.0, 3.0) if m <= case["t_hi"]]
        d["weights"] = rng.uniform(-2.0, 2.0, size=case["n_surf"] * case["per_surface"])
        # the book's make-up (surface, type, maturity, path count) is the case's, not the seed's
        fixed = np.random.Generator(np.random.PCG64(7))
        d["items"] = []
        for s in range(case["n_surf"]):
            for _ in range(case["per_surface"]):
                T = float(mats[fixed.integers(0, len(mats))])
                d["items"].append(_Item(s, 1 if fixed.uniform() < 0.5 else -1, float(rng.uniform(60.0, 140.0)), T,
                                        int(round(52 * T)), int(2.0 ** fixed.uniform(case["log2_lo"], case["log2_hi"])),
                                        len(d["items"])))
        return d
    d["K"] = float(rng.uniform(95.0, 105.0))
    d["spot"], d["time"], d["sigma"] = _grid(case, rng)
    if case["kind"] == "autograd":
        d["sigma"] = d["sigma"].astype(np.float32)
    return d


class _Item:
    def __init__(self, surface, phi, K, T, n_steps, n_paths, stream_id):
        self.surface, self.phi, self.K, self.T = surface, phi, K, T
        self.n_steps, self.n_paths, self.stream_id = n_steps, n_paths, stream_id


def prepare(case, seed):
    d = _inputs(case, seed)
    kind = case["kind"]
    if kind in ("book", "book_risk"):
        surfs = [lv.Surface(*g) for g in d["surfs"]]
        book = lv.Book(surfs, d["items"])
        if kind == "book_risk":
            book.set_weights(d["weights"])
        return dict(kind=kind, surfs=surfs, book=book, args=(d["S0"], case["r"], d["seed"]))
    s = lv.Surface(d["spot"], d["time"], d["sigma"])
    s.set_option_type(case["phi"])
    s.set_interpolation(case.get("interp", 0))
    s.set_scheme(case.get("scheme", 0))
    if kind == "tangent":
        s.set_adjoint_method(lv.LV_ADJ_TANGENT)
    if kind == "kahan":
        s.set_accumulation(lv.LV_ACC_KAHAN)
    s.set_stream(torch.cuda.current_stream().cuda_stream)
    st = dict(kind=kind, surf=s, args=(d["S0"], case["r"], d["K"], case["T"], case["n_steps"], case["n_paths"],
                                       d["seed"]))
    if kind == "autograd":
        st["S0"] = torch.tensor(d["S0"], dtype=torch.float64, requires_grad=True)
        st["sigma"] = torch.tensor(d["sigma"], device="cuda", requires_grad=True)
    if kind == "recalibrated":
        st["sigma"] = d["sigma"]
    if kind in ("greeks_device", "fp64"):
        st["out"] = torch.empty(3 + s.IJ, dtype=torch.float64, device="cuda")
    return st


def run(state):
    kind, a = state["kind"], state["args"]
    if kind == "book":
        return state["book"].run(*a)
    if kind == "book_risk":
        return state["book"].run_risk(*a)
    s = state["surf"]
    if kind == "price":
        return s.price(*a)
    if kind == "recalibrated":
        s.set_sigma(state["sigma"])
        return s.price_greeks(*a)
    if kind in ("greeks", "tangent", "kahan"):
        return s.price_greeks(*a)
    if kind == "greeks_device":
        s.price_greeks_device(*a, state["out"].data_ptr())
        return state["out"]
    if kind == "fp64":
        s.price_greeks_fp64_device(*a, state["out"].data_ptr())
        return state["out"]
    if kind == "ext":
        return s.price_greeks_ext(*a)
    if kind == "vanna":
        return s.price_greeks_vanna(*a)
    S0, sigma = state["S0"], state["sigma"]
    S0.grad = sigma.grad = None
    price = lv_price(S0, sigma, s, *a[1:])
    price.backward()
    return price.detach(), S0.grad, sigma.grad


# ------------------------------------------------------------------ work

def _path_steps(case):
    if case["kind"] in ("book", "book_risk"):
        return float(sum(o.n_steps * o.n_paths for o in _inputs(case, 1)["items"]))
    return float(case["n_steps"]) * case["n_paths"]


def work(case):
    """Arithmetic a path-step cannot do without: 36 operations forward
    (Philox, Box-Muller, the bilinear lookup, the Euler step) and, for the
    half of the paths that end in the money, 19 backward; the grid in and the
    results out."""
    ops = 36.0 if case["kind"] == "price" else 36.0 + 19.0 * 0.5
    nodes = case["n_spot"] * case["n_time"]
    if case["kind"] == "book":
        values = nodes * case["n_surf"] * (1 + case["per_surface"])
    elif case["kind"] == "book_risk":
        values = 2 * nodes * case["n_surf"]
    else:
        values = nodes if case["kind"] == "price" else 2 * nodes
    return {"bytes": 8.0 * (values + 16), "flops": ops * _path_steps(case)}


# ------------------------------------------------------------------ 64 bits

_M32 = 0xFFFFFFFF


def _normals(seed, stream_id, p0, m, n_steps, dev):
    """Standard normals [n_steps, m] of paths p0 .. p0 + m: Philox4x32-10 on
    (block, path, stream, 0) and Box-Muller on 23-bit uniforms."""
    B = (n_steps + 3) // 4
    p = torch.arange(p0, p0 + m, dtype=torch.int64, device=dev)[None, :]
    blk = torch.arange(B, dtype=torch.int64, device=dev)[:, None]
    c0 = blk.expand(B, m)
    c1 = (p & _M32).expand(B, m)
    c2 = (((p >> 32) & 0xFFFF) | (stream_id << 16)).expand(B, m)
    c3 = torch.zeros(B, m, dtype=torch.int64, device=dev)
    k0, k1 = seed & _M32, (seed >> 32) & _M32
    for _ in range(10):
        q0, q1 = c0 * 0xD2511F53, c2 * 0xCD9E8D57
        c0, c1, c2, c3 = ((q1 >> 32) & _M32) ^ c1 ^ k0, q1 & _M32, ((q0 >> 32) & _M32) ^ c3 ^ k1, q0 & _M32
        k0, k1 = (k0 + 0x9E3779B9) & _M32, (k1 + 0xBB67AE85) & _M32
    z = torch.empty(B, 4, m, dtype=torch.float64, device=dev)
    for h, (wa, wb) in enumerate(((c0, c1), (c2, c3))):
        rho = torch.sqrt(-2.0 * torch.log(((wa >> 9).double() + 0.5) * 2.0 ** -23))
        ang = (2.0 * math.pi) * (((wb >> 9).double() + 0.5) * 2.0 ** -23)
        z[:, 2 * h], z[:, 2 * h + 1] = rho * torch.cos(ang), rho * torch.sin(ang)
    return z.reshape(4 * B, m)[:n_steps]


def _sums(g, S0, r, K, T, N, n_paths, seed, phi, interp=0, scheme=0, stream_id=0, want="greeks"):
    """Sums over paths of V, V^2, x_bar_0 (= S0 d V / d S0), and of the bucket
    terms [I, J] (vegas, or with want = "vanna" the second-order terms), d V /
    d r and d V / d T."""
    dev = torch.device("cuda")
    s, tau, sig = (torch.as_tensor(np.asarray(v, dtype=np.float64), device=dev) for v in g)
    I, J = sig.shape
    nodes = torch.log(s) if interp else s
    dt = T / N
    sq = math.sqrt(dt)
    tn = np.arange(N) * dt
    th = np.asarray(g[1], dtype=np.float64)
    jn = np.clip(np.searchsorted(th, tn, side="right") - 1, 0, J - 2)
    vn = np.clip((tn - th[jn]) / (th[jn + 1] - th[jn]), 0.0, 1.0)
    out = torch.zeros(5, dtype=torch.float64, device=dev)
    buckets = torch.zeros(I * J, dtype=torch.float64, device=dev)
    disc = math.exp(-r * T)
    chunk = max(32, int(6e7 // N))
    for p0 in range(0, n_paths, chunk):
        m = min(chunk, n_paths - p0)
        Z = _normals(seed, stream_id, p0, m, N, dev)
        x = torch.full((m,), S0 if scheme else math.log(S0), dtype=torch.float64, device=dev)
        keep = []

        def at(n, x):
            S = x if scheme else torch.exp(x)
            i = (torch.searchsorted(s, S, right=True) - 1).clamp_(0, I - 2)
            c = torch.log(S.clamp(min=1e-300)) if interp else S
            w = nodes[i + 1] - nodes[i]
            u = ((c - nodes[i]) / w).clamp_(0.0, 1.0)
            lo, hi, v = sig[:, jn[n]], sig[:, jn[n] + 1], float(vn[n])
            dlo, dhi = lo[i + 1] - lo[i], hi[i + 1] - hi[i]
            inside = ((S >= s[0]) & (S <= s[-1])).double()
            kap = inside * ((1.0 - v) * dlo + v * dhi) / w * (1.0 if interp else S)
            top, bot = lo[i] + u * dlo, hi[i] + u * dhi
            return S, i, u, v, (1.0 - v) * top + v * bot, kap, bot - top, inside * (1.0 if interp else S) / w

        for n in range(N):
            if want != "price":
                keep.append(x)
            _, _, _, _, sg, _, _, _ = at(n, x)
            if scheme:
                x = x * (1.0 + r * dt + sg * sq * Z[n])
            else:
                x = x + (r - 0.5 * sg * sg) * dt + sg * sq * Z[n]
        SN = x if scheme else torch.exp(x)
        itm = phi * (SN - K)
        V = disc * itm.clamp(min=0.0)
        out[0] += V.sum()
        out[1] += (V * V).sum()
        if want == "price":
            continue
        live = torch.nonzero(itm > 0.0).reshape(-1)
        # x_bar_N: d V / d x_N on ln S, d V / d S_N under Euler on S
        xb = torch.full_like(SN[live], disc * phi) if scheme else disc * phi * SN[live]
        if want == "vanna":     # the pathwise delta first: x_bar_0 = x_bar_N prod (1 + g_n)
            D = torch.ones_like(xb)
            for n in range(N):
                _, _, _, _, sg, kap, _, _ = at(n, keep[n][live])
                D = D * (1.0 + (sq * Z[n][live] - sg * dt) * kap)
            xb = xb * D
            out[2] += xb.sum()
        if want == "ext":
            out[3] += (-T * V).sum()
            out[4] += (-r * V).sum()
        for n in range(N - 1, -1, -1):
            z = Z[n][live]
            S, i, u, v, sg, kap, dsig_t, sdu = at(n, keep[n][live])
            if want == "vanna":
                h = sq * z - sg * dt
                f = 1.0 + h * kap
                q = xb / S0 * ((z * z - 1.0) / sg - sq * z * (1.0 + kap / (sg * f)))
                e = xb / S0 * (h / f) * sdu
            else:
                if scheme:
                    h = S * sq * z
                    f = 1.0 + r * dt + sq * z * (sg + kap)
                else:
                    h = sq * z - sg * dt
                    f = 1.0 + h * kap
                q, e = xb * h, 0.0
                if want == "ext":
                    wt = th[jn[n] + 1] - th[jn[n]]
                    ds = dsig_t / wt if th[0] <= tn[n] < th[-1] else 0.0 * dsig_t
                    ar = S * dt if scheme else dt
                    am = S * (r + sg * z / (2.0 * sq)) if scheme else (r - 0.5 * sg * sg) + sg * z / (2.0 * sq)
                    out[3] += (xb * ar).sum()
                    out[4] += (xb * (am / N + h * ds * (n / N))).sum()
                xb = xb * f
            k = i * J + int(jn[n])
            a, b = q * (1.0 - v), q * v
            ea, eb = e * (1.0 - v), e * v
            for off, val in ((J, a * u + ea), (0, a * (1.0 - u) - ea), (J + 1, b * u + eb), (1, b * (1.0 - u) - eb)):
                buckets += torch.bincount(k + off, weights=val, minlength=I * J)
        if want != "vanna":
            out[2] += (xb * (S0 if scheme else 1.0)).sum()
    o = [float(v) for v in out.cpu()]
    return o, buckets.reshape(I, J).cpu().numpy()


def _stderr(o, P):
    mean = o[0] / P
    var = (o[1] / P - mean * mean) * P / (P - 1.0) if P > 1 else 0.0
    return math.sqrt(max(var, 0.0) / P)


def exact(case, seed):
    if _path_steps(case) > EXACT_PATH_STEPS:
        return None
    d = _inputs(case, seed)
    kind = case["kind"]
    if kind in ("book", "book_risk"):
        blocks, risk = [], [[0.0, 0.0, 0.0, 0.0] for _ in d["surfs"]]
        for q, it in enumerate(d["items"]):
            o, b = _sums(d["surfs"][it.surface], d["S0"], case["r"], it.K, it.T, it.n_steps, it.n_paths, d["seed"],
                         it.phi, stream_id=it.stream_id)
            P, w = it.n_paths, d["weights"][q]
            p, dl, se, v = o[0] / P, o[2] / (P * d["S0"]), _stderr(o, P), b / P
            blocks.append(np.concatenate([[p, dl, se], v.reshape(-1)]))
            t = risk[it.surface]
            risk[it.surface] = [t[0] + w * p, t[1] + w * dl, t[2] + (w * se) ** 2, t[3] + w * v]
        if kind == "book":
            return np.concatenate(blocks)
        return np.concatenate([np.concatenate([[t[0], t[1], math.sqrt(t[2])], np.reshape(t[3], -1)]) for t in risk])
    want = {"price": "price", "ext": "ext", "vanna": "vanna"}.get(kind, "greeks")
    P, S0 = case["n_paths"], d["S0"]
    o, b = _sums((d["spot"], d["time"], d["sigma"]), S0, case["r"], d["K"], case["T"], case["n_steps"], P, d["seed"],
                 case["phi"], case.get("interp", 0), case.get("scheme", 0), want=want)
    price, delta = o[0] / P, o[2] / (P * S0)
    if kind == "price":
        return price, _stderr(o, P)
    if kind == "ext":
        return price, delta, b / P, o[3] / P, o[4] / P
    if kind in ("greeks_device", "fp64"):
        return torch.from_numpy(np.concatenate([[price, delta, _stderr(o, P)], (b / P).reshape(-1)]))
    if kind == "autograd":
        return (torch.tensor(price, dtype=torch.float64), torch.tensor(delta, dtype=torch.float64),
                torch.from_numpy(b / P))
    return price, delta, b / P
