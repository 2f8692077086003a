"""Workloads of the parallel multicanonical simulation, measured through its public API.

Each case is one call (or one turn of the loop) that a program using the package makes:
a weight iteration driven by hand, a whole weight iteration on the host or on the device,
a production run, a batch of instances, a read of the configurations.  The instances hold
walkers that have already been spread over the energies by weights close to the
reciprocal density of states, as they are in the middle of a run.
"""
import math
import random

import numpy as np

from paper_1707_00919_gb300 import muca as M

# Integer operations of one attempted flip: Philox4x32-10 (78 per four words) and the
# flip itself (own spin, four comparisons, count, threshold, compare, update, record).
OPS_PER_ATTEMPT = 35
MAX_ATTEMPTS = 3.0e9          # of a drawn case; the largest listed case runs 4.7e9
NUMPY_SECONDS = 8.0           # exact() simulates a case in numpy when that stays below


# ---------------------------------------------------------------------------------
# cases
# ---------------------------------------------------------------------------------
def listed():
    return [
        # The smallest simulation: 128 walkers at L = 8, one weight iteration of 31
        # thermalization and 100 recorded sweeps.  One block per few SMs: launch, weights
        # upload and the latency of one walker's chain.
        dict(name="step_l8_w128", kind="step", L=8, W=128, layout="int8", order="typewriter",
             therm=31 * 64, rec=100 * 64, window=0, settle=60),
        # An early iteration of the paper's schedule (30 w attempts of thermalization, few
        # recorded ones, starting and ending inside a sweep), the walkers in a window of
        # 60 energies: short launches, any attempt range.
        dict(name="early_l16_w4096", kind="step", L=16, W=4096, layout="int8", order="typewriter",
             therm=1800, rec=15, window=60, settle=4),
        # The headline workload: L = 32, 16384 walkers, 31 + 10 sweeps.
        dict(name="step_l32_w16384", kind="step", L=32, W=16384, layout="int8", order="typewriter",
             therm=31 * 1024, rec=10 * 1024, window=0, settle=1200),
        # Production at the default walker count of a GB300 (full occupancy at L = 32):
        # recorded sweeps only but for the lead.
        dict(name="production_l32_w48640", kind="production", L=32, W=48640, layout="packed", order="typewriter",
             therm=20, rec=100, settle=800),
        # L = 64, 32768 walkers, bit-packed: one weight iteration of 31 + 4 sweeps, the
        # largest state.
        dict(name="step_l64_w32768", kind="step", L=64, W=32768, layout="packed", order="typewriter",
             therm=31 * 4096, rec=4 * 4096, window=0, settle=600),
        # The paper's own update order (one random site sequence for all walkers).
        dict(name="random_l32_w16384", kind="step", L=32, W=16384, layout="int8", order="random",
             therm=31 * 1024, rec=10 * 1024, window=0, settle=300),
        # A late iteration of the paper's schedule with few walkers, as a served request
        # runs hundreds of times: thirty sweeps of thermalization and ninety recorded ones
        # that start and end inside a sweep, on 32 warps.
        dict(name="paper_l48_w1024", kind="step", L=48, W=1024, layout="int8", order="typewriter",
             therm=69150, rec=215807, window=0, settle=200),
        # Weight iteration on the host from ln W = 0, a fixed number of iterations.
        dict(name="iterate_l16_w4096", kind="iterate", L=16, W=4096, layout="int8", order="typewriter",
             therm=31, rec=10, iterations=40, settle=1),
        # The same with its host steps on the device, a walker count that is no multiple
        # of a warp.
        dict(name="device_l24_w5003", kind="device", L=24, W=5003, layout="packed", order="typewriter",
             therm=31, rec=10, iterations=12, settle=1),
        # A lattice size without a kernel of its own.
        dict(name="step_l40_w4096", kind="step", L=40, W=4096, layout="int8", order="typewriter",
             therm=8 * 1600, rec=4 * 1600, window=0, settle=100),
        # Twelve instances of uneven size in one launch per weight iteration.
        dict(name="batch_12", kind="batch", n=12, mix=1234, wmax=16384, layout="int8", therm=31, rec=10,
             iterations=1, settle=1),
        # Configurations read out between sweeps (magnetisation, correlation functions).
        dict(name="snapshot_l32_w16384", kind="snapshot", L=32, W=16384, layout="int8", order="typewriter",
             rec=5, settle=300),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "production", "iterate", "device", "batch", "snapshot"])
    layout = rng.choice(["int8", "packed"])
    if kind == "batch":
        return dict(kind=kind, n=rng.randint(3, 14), mix=rng.randint(0, 9999), wmax=_log_int(rng, 1024, 12000),
                    layout=layout, therm=rng.randint(10, 31), rec=rng.randint(2, 10), iterations=1, settle=1)
    L = rng.choice([8, 16, 16, 24, 32, 32, 32, 48, 64, 64, 4 * rng.randint(1, 16)])
    N = L * L
    # whole blocks in half of the cases, any count in the others
    W = _log_int(rng, 100, 60000)
    if rng.random() < 0.5:
        W = max(128, W // 128 * 128)
    order = "random" if kind in ("step", "production") and rng.random() < 0.2 else "typewriter"
    special = L in (8, 16, 24, 32, 48, 64)
    # attempts per walker: the slower kernels and the longer chains get fewer
    most = MAX_ATTEMPTS * (1.0 if special and order == "typewriter" else 0.12) / W
    most = min(most, 3.0e5)
    if kind == "step":
        if rng.random() < 0.5:   # whole sweeps
            rec = rng.randint(1, 20)
            therm = rng.choice([0, 5, 31])
            while (therm + rec) * N > most and therm + rec > 2:
                therm, rec = therm // 2, max(1, rec // 2)
            therm, rec, window = therm * N, rec * N, 0
        else:                    # the paper's schedule at some width
            w = _log_int(rng, 10, N + 1) if N > 10 else 10
            therm = int(min(30 * w, most * 0.6))
            rec = int(min(math.floor(6.0 * w ** 2.25 / W) + 1, most * 0.4 + 1))
            window = w
        settle = max(1, min(200, int(most / N)))
        return dict(kind=kind, L=L, W=W, layout=layout, order=order, therm=therm, rec=rec, window=window,
                    settle=settle)
    sweeps = max(2, min(120, int(most / N)))
    if kind == "production":
        return dict(kind=kind, L=L, W=W, layout=layout, order=order, therm=rng.randint(0, sweeps // 2),
                    rec=rng.randint(max(1, sweeps // 2), sweeps), settle=sweeps)
    if kind == "snapshot":
        W = min(W, 80_000_000 // N)
        return dict(kind=kind, L=L, W=W, layout=layout, order=order, rec=rng.randint(1, min(5, sweeps)),
                    settle=sweeps)
    iterations = rng.randint(2, 20)
    while iterations > 2 and iterations * 12 > sweeps * 10:
        iterations -= 1
    return dict(kind=kind, L=L, W=W, layout=layout, order=order, therm=max(1, min(31, sweeps // iterations)),
                rec=rng.randint(1, 10), iterations=iterations, settle=1)


def _batch_specs(case):
    rng = random.Random(case["mix"])
    return [(rng.choice([16, 24, 32, 48, 64]), rng.randint(512, case["wmax"])) for _ in range(case["n"])]


# ---------------------------------------------------------------------------------
# weights: minus Onsager's entropy of the infinite square lattice
# ---------------------------------------------------------------------------------
_ENTROPY = None


def _entropy():
    """(energies per spin, entropies per spin) of the infinite lattice, u from -2 to 2."""
    global _ENTROPY
    if _ENTROPY is None:
        beta = np.linspace(0.0, 2.5, 2501)
        theta = (np.arange(2000) + 0.5) * (np.pi / 2 / 2000)
        kappa = 2.0 * np.sinh(2 * beta) / np.cosh(2 * beta) ** 2
        root = np.sqrt(np.maximum(0.0, 1.0 - (kappa[:, None] * np.sin(theta)[None, :]) ** 2))
        ln_z = np.log(2.0 * np.cosh(2 * beta)) + np.mean(np.log(0.5 * (1.0 + root)), axis=1) / 2.0
        u = -np.gradient(ln_z, beta)
        s = ln_z + beta * u
        u, s = u[::-1], np.maximum(s[::-1], 0.0)
        keep = np.concatenate([[True], np.diff(np.maximum.accumulate(u)) > 0]) & (u > -2.0)
        u, s = np.concatenate([[-2.0], u[keep]]), np.concatenate([[0.0], s[keep]])
        _ENTROPY = np.concatenate([u[:-1], [0.0], -u[:-1][::-1]]), np.concatenate([s[:-1], [math.log(2.0)], s[:-1][::-1]])
    return _ENTROPY


def _weights(L, window):
    """ln W(e) close to -ln g(e); with a window, only inside the window around the centre
    and constant outside it, as the recursion leaves them before the range is covered."""
    N = L * L
    u, s = _entropy()
    e = np.arange(N + 1)
    lnW = -N * np.interp(-2.0 + 4.0 * e / N, u, s)
    if window:
        lo, hi = max(0, N // 2 - window // 2), min(N, N // 2 + window // 2)
        lnW[:lo], lnW[hi + 1:] = lnW[lo], lnW[hi]
    return lnW


# ---------------------------------------------------------------------------------
# preparation and one pass
# ---------------------------------------------------------------------------------
def _layout(case):
    return M.MUCA_LAYOUT_PACKED if case["layout"] == "packed" else M.MUCA_LAYOUT_INT8


def prepare(case, seed):
    if case["kind"] == "batch":
        inst = []
        for i, (L, W) in enumerate(_batch_specs(case)):
            m = M.Muca(L, W, seed * 1000 + i, _layout(case))
            m.sweep(case["settle"], record=False)
            inst.append(m)
        return dict(case=case, inst=inst, batch=M.Batch(inst),
                    params=M.make_params(therm_sweeps=case["therm"], sweeps_per_iter=case["rec"],
                                         max_iterations=case["iterations"], flat_threshold=2.0))
    m = M.Muca(case["L"], case["W"], seed, _layout(case))
    state = dict(case=case, m=m)
    if case["kind"] in ("iterate", "device"):
        m.sweep(case["settle"], record=False)
        # a threshold that min/mean cannot reach: the number of iterations is the case's
        state["params"] = M.make_params(therm_sweeps=case["therm"], sweeps_per_iter=case["rec"],
                                        max_iterations=case["iterations"], flat_threshold=2.0)
        state["zero"] = np.zeros(m.n_bins)
        return state
    state["lnW"] = _weights(case["L"], case.get("window", 0))
    m.set_weights(state["lnW"])
    if case["order"] == "random":
        m.site_order = M.MUCA_ORDER_RANDOM
    m.sweep(case["settle"], record=False)
    m.synchronize()
    return state


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "batch":
        state["batch"].iterate_until_flat(state["params"])
        return {"lnW": [m.get_weights() for m in state["inst"]], "H": [m.get_histogram() for m in state["inst"]],
                "energies": [m.get_energies() for m in state["inst"]]}
    m = state["m"]
    if kind == "step":
        # one weight iteration in the caller's hands: weights, sampling, histogram,
        # flatness, Eq. (4)
        lnW = state["lnW"].copy()
        m.set_weights(lnW)
        m.thermalize_and_record(case["therm"], case["rec"])
        H = m.get_histogram()
        flat = M.muca_flatness(m.L, H, measures=("min_over_mean",))["min_over_mean"]
        M.muca_update_weights(m.L, lnW, H)
        state["lnW"] = lnW
        return {"H": H, "flat": flat, "lnW": lnW, "energies": m.get_energies()}
    if kind == "production":
        H, ln_g = m.production(case["therm"], case["rec"])
        return {"H": H, "ln_g": ln_g, "energies": m.get_energies()}
    if kind == "snapshot":
        m.sweep(case["rec"], record=True)
        return {"lattice": m.get_lattice(), "energies": m.get_energies()}
    m.set_weights(state["zero"])
    if kind == "iterate":
        st = m.iterate_until_flat(state["params"])
    else:
        st = m.iterate_device(state["params"], 8)
    return {"lnW": m.get_weights(), "H": m.get_histogram(), "metric": st.last_metric, "energies": m.get_energies()}


# ---------------------------------------------------------------------------------
# work that a pass cannot do without
# ---------------------------------------------------------------------------------
def _attempts(case):
    """(L, W, attempts per walker) of every instance of the case."""
    if case["kind"] == "batch":
        n = (case["therm"] + case["rec"]) * case["iterations"]
        return [(L, W, n * L * L) for L, W in _batch_specs(case)]
    L, W, N = case["L"], case["W"], case["L"] ** 2
    if case["kind"] == "step":
        n = case["therm"] + case["rec"]
    elif case["kind"] == "snapshot":
        n = case["rec"] * N
    else:
        n = (case["therm"] + case["rec"]) * case.get("iterations", 1) * N
    return [(L, W, n)]


def work(case):
    nbytes = flops = 0
    for L, W, n in _attempts(case):
        N = L * L
        lattice = W * (N if case["layout"] == "int8" else L * (4 if L <= 32 else 8))
        # lattices and energies in and out, weights in, histogram out
        nbytes += 2 * lattice + 8 * W + 16 * (N + 1)
        if case["kind"] == "snapshot":
            nbytes += W * N
        flops += OPS_PER_ATTEMPT * W * n
    return {"bytes": nbytes, "flops": flops}


# ---------------------------------------------------------------------------------
# the same chain in numpy
# ---------------------------------------------------------------------------------
def _philox(c0, c1, c2, c3, seed):
    """Philox4x32-10 on counters of uint64 arrays (values below 2^32), four words each."""
    mask = np.uint64(0xFFFFFFFF)
    k0, k1 = seed & 0xFFFFFFFF, (seed >> 32) & 0xFFFFFFFF
    x = [np.asarray(v, dtype=np.uint64) for v in (c0, c1, c2, c3)]
    for _ in range(10):
        p0, p1 = x[0] * np.uint64(0xD2511F53), x[2] * np.uint64(0xCD9E8D57)
        x = [(p1 >> np.uint64(32)) ^ x[1] ^ np.uint64(k0), p1 & mask,
             (p0 >> np.uint64(32)) ^ x[3] ^ np.uint64(k1), p0 & mask]
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return x


def _thresholds(lnW):
    """T[e, k] as uint64, an always-accept entry as 2^32."""
    nb = len(lnW)
    T = np.zeros((nb, 5), dtype=np.uint64)
    for k in range(5):
        to = np.arange(nb) + 2 - k
        ok = (to >= 0) & (to < nb)
        dw = np.where(ok, lnW[np.clip(to, 0, nb - 1)] - lnW, -np.inf)
        t = np.minimum(np.floor(np.exp(np.minimum(dw, 0.0)) * 2.0 ** 32), 2.0 ** 32 - 1)
        T[:, k] = np.where(dw >= 0, 2.0 ** 32, np.where(t == 2.0 ** 32 - 1, 2.0 ** 32, t)).astype(np.uint64)
    return T


class _Walkers:
    """All walkers of an instance, advanced attempt by attempt (typewriter order)."""

    def __init__(self, L, W, seed):
        self.L, self.W, self.seed, self.t = L, W, seed, 0
        self.N = N = L * L
        self.w = np.arange(W, dtype=np.uint64)
        s = np.empty((N, W), dtype=np.int8)
        for b in range(N // 4):
            for u, q in enumerate(_philox(np.full(W, b), np.zeros(W), self.w, np.ones(W), seed)):
                s[4 * b + u] = (q >> np.uint64(31)) != 0
        g = s.reshape(L, L, W)
        self.e = ((g != np.roll(g, -1, 0)).sum((0, 1)) + (g != np.roll(g, -1, 1)).sum((0, 1))) // 2
        self.s = s

    def advance(self, lnW, n, record):
        L, N, s = self.L, self.N, self.s
        T = _thresholds(lnW).reshape(-1)
        H = np.zeros(N + 1, dtype=np.uint64)
        q = None
        for t in range(self.t, self.t + n):
            if q is None or t % 4 == 0:
                q = _philox(np.full(self.W, t >> 2), np.zeros(self.W), self.w, np.zeros(self.W), self.seed)
            y, x = divmod(t % N, L)
            c = s[y * L + x]
            k = ((c ^ s[(y - 1) % L * L + x]) + (c ^ s[(y + 1) % L * L + x]) + (c ^ s[y * L + (x - 1) % L]) +
                 (c ^ s[y * L + (x + 1) % L]))
            acc = q[t % 4] < T[self.e * 5 + k]
            c ^= acc.astype(np.int8)
            self.e = self.e + np.where(acc, 2 - k, 0)
            if record:
                H += np.bincount(self.e, minlength=N + 1).astype(np.uint64)
        self.t += n
        return H


def exact(case, seed):
    """The outputs of the first pass for a single typewriter-order instance that numpy can
    follow in a few seconds; None otherwise."""
    if case["kind"] not in ("step", "production") or case["order"] != "typewriter":
        return None
    L, W, n = _attempts(case)[0]
    N = L * L
    if (n + case["settle"] * N) * (1.0e-4 + W * 6.0e-8) > NUMPY_SECONDS:
        return None
    walkers = _Walkers(L, W, seed)
    lnW = _weights(L, case.get("window", 0))
    walkers.advance(lnW, case["settle"] * N, False)
    unit = 1 if case["kind"] == "step" else N
    walkers.advance(lnW, case["therm"] * unit, False)
    H = walkers.advance(lnW, case["rec"] * unit, True)
    seen = H > 0
    with np.errstate(divide="ignore"):
        lnH = np.log(H.astype(np.float64))
    energies = walkers.e.astype(np.int32)
    if case["kind"] == "production":
        ln_g = np.where(seen, lnH - lnW, -np.inf)
        top = ln_g.max()
        ln_g = ln_g + N * math.log(2.0) - (top + math.log(np.exp(ln_g - top).sum()))
        return {"H": H, "ln_g": ln_g, "energies": energies}
    inside = np.ones(N + 1, dtype=bool)
    inside[[1, N - 1]] = False
    flat = float(H[inside].min()) / (float(H[inside].sum()) / (N - 1))
    return {"H": H, "flat": flat, "lnW": np.where(seen, lnW - np.where(seen, lnH, 0.0), lnW), "energies": energies}
