"""Performance cases of the batched low-rank update library.

Each case is one unit of work as a variational or projector Monte Carlo
program hands it to the library, through the public Python binding:

  sweep    a run of Monte Carlo steps (form the move operands, propose the
           ratio, accept, commit the occupation), then the log-value, the sign
           and the inverse that the sweep's measurements read;
  refresh  rebuild A^{-1}, log-value and sign from the current configuration
           and read the drift, the log-value and the inverse;
  ragged   walkers of uneven n and rank k through the persistent step: one
           differentiated proposal (log ratio and its adjoint), then accepted
           steps;
  orbital  the log ratio of backflow-style updates, differentiated through the
           orbital matrix shared by all walkers;
  slog     the standalone differentiable batch of log|det| / log|pf|.

Walkers sit on 2n sites that come in pairs, one pair per orbital, with one
site of each pair occupied; the orbital (pairing) matrix couples each site to
its own orbital (partner) and, by Gaussian entries of variance ~1/n, to all
others.  A move takes a particle to the other site of its pair.  That is the
configuration set a sampler equilibrated in |psi|^2 visits: ratios of order
one, matrices away from the nodes, rows and columns in random order so that
the eliminations have to pivot.
"""
import math
import random

import torch

from paper_2602_05255_gb300 import lrugb

DTYPES = {"f64": torch.float64, "c128": torch.complex128, "f32": torch.float32, "c64": torch.complex64}
BYTES = {"f64": 8, "c128": 16, "f32": 4, "c64": 8}
FLUSH = {"native": lrugb.FLUSH_NATIVE, "split": lrugb.FLUSH_SPLIT, "df": lrugb.FLUSH_DF}
ARITH = {"native": lrugb.ARITH_NATIVE, "df": lrugb.ARITH_DF}
DEV = "cuda"


def listed():
    return [
        # one walker, 64 particles, one step: the latency of a single small call chain (single-walker debugging,
        # correlated sampling of one configuration)
        {"name": "det_step_1x64", "task": "sweep", "kind": "det", "walkers": 1, "n": 64, "k": 1, "dtype": "f64",
         "delay": 0, "flush": "native", "arith": "native", "steps": 1},
        # the headline workload: 1024 walkers of 1024 particles, delayed updates in the form the autotuner picks
        {"name": "det_sweep_1024x1024", "task": "sweep", "kind": "det", "walkers": 1024, "n": 1024, "k": 1,
         "dtype": "f64", "delay": 16, "flush": "split", "arith": "df", "steps": 16},
        # its periodic refresh (every 128 steps), with the drift read as the default does
        {"name": "det_refresh_512x1024", "task": "refresh", "kind": "det", "walkers": 512, "n": 1024, "dtype": "f64"},
        # plain updates with every option at its default, at an n no tile divides
        {"name": "det_plain_384x500", "task": "sweep", "kind": "det", "walkers": 384, "n": 500, "k": 1,
         "dtype": "f64", "delay": 0, "flush": "native", "arith": "native", "steps": 8},
        # complex orbitals (twisted boundaries, magnetic fields), delayed, default precision
        {"name": "det_c128_sweep_512x512", "task": "sweep", "kind": "det", "walkers": 512, "n": 512, "k": 1,
         "dtype": "c128", "delay": 16, "flush": "native", "arith": "native", "steps": 16},
        # and the refresh of complex walkers
        {"name": "det_c128_refresh_256x512", "task": "refresh", "kind": "det", "walkers": 256, "n": 512,
         "dtype": "c128"},
        # the Pfaffian workload: 1024 walkers, n = 256 on 512 sites, row-and-column moves, K = 8
        {"name": "pf_sweep_1024x256", "task": "sweep", "kind": "pf", "walkers": 1024, "n": 256, "k": 1,
         "dtype": "f64", "delay": 8, "flush": "split", "arith": "df", "steps": 8},
        # start (or refresh) of the Pfaffian walkers: inverse and Pfaffian from scratch
        {"name": "pf_refresh_1024x256", "task": "refresh", "kind": "pf", "walkers": 1024, "n": 256, "dtype": "f64"},
        # few large walkers, two-electron moves: the precision workload's shape
        {"name": "det_two_64x2048", "task": "sweep", "kind": "det", "walkers": 64, "n": 2048, "k": 2, "dtype": "f64",
         "delay": 32, "flush": "split", "arith": "native", "steps": 32},
        # walkers of uneven size and rank in single precision complex: gradient of one proposal, then four steps
        {"name": "ragged_c64_512", "task": "ragged", "walkers": 512, "sizes": "128,256,512,1024", "ranks": "1,2,4,8",
         "dtype": "c64", "delay": 4, "steps": 4},
        # wave-function optimisation: gradient of the log ratios with respect to the shared orbitals and U, V
        {"name": "orbital_grad_512x256", "task": "orbital", "walkers": 512, "n": 256, "k": 2, "dtype": "f64"},
        # standalone differentiable log-determinants of a training batch, at an n no tile divides
        {"name": "slogdet_grad_256x500", "task": "slog", "kind": "det", "walkers": 256, "n": 500, "dtype": "f64"},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    task = rng.choice(["sweep", "sweep", "sweep", "refresh", "refresh", "ragged", "orbital", "slog"])
    if task == "ragged":
        sizes = sorted({_log_int(rng, 24, 700) for _ in range(rng.randint(2, 4))})
        ranks = sorted({rng.randint(1, 8) for _ in range(rng.randint(2, 3))})
        mean = sum(s * s for s in sizes) / len(sizes)
        return {"task": task, "walkers": max(4, min(_log_int(rng, 8, 1024), int(2 ** 26 / mean))),
                "sizes": ",".join(map(str, sizes)), "ranks": ",".join(map(str, ranks)),
                "dtype": rng.choice(["f64", "c128", "c64"]), "delay": rng.choice([0, 4]), "steps": 4}
    dtype = rng.choice(["f64", "f64", "f64", "c128", "f32", "c64"])
    n = _log_int(rng, 48, 1024)
    if n >= 128 and rng.random() < 0.5:
        n = n // 128 * 128
    kind = rng.choice(["det", "det", "pf"])
    if kind == "pf":
        n = min(512, n) // 2 * 2
    heavy = 4 if dtype == "c128" else 1
    walkers = _log_int(rng, 1, 1024)
    if task == "orbital":
        n = min(n, 512)
        return {"task": task, "walkers": max(1, min(walkers, int(2 ** 25 / heavy / n ** 2))), "n": n,
                "k": rng.choice([1, 2, 4]), "dtype": dtype}
    if task in ("refresh", "slog"):
        cap = int(2 ** 35 / heavy / n ** 3)
        return {"task": task, "kind": kind, "walkers": max(1, min(walkers, cap)), "n": n, "dtype": dtype}
    walkers = max(1, min(walkers, int(2 ** 28 / heavy / n ** 2), int(2 ** 37 / heavy / n ** 3)))
    k = rng.choice([1, 1, 1, 2])
    delay = rng.choice([0, 4, 8, 16])
    tiles = n % 128 == 0 and dtype == "f64" and delay > 0
    flush = rng.choice(["split", "native", "df"] if tiles else ["native"])
    arith = rng.choice(["df", "native"]) if dtype == "f64" else "native"
    return {"task": task, "kind": kind, "walkers": walkers, "n": n, "k": k, "dtype": dtype, "delay": delay,
            "flush": flush, "arith": arith, "steps": rng.choice([4, 8, 16])}


# ---- inputs -------------------------------------------------------------------


def _generator(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _normal(gen, shape, dtype):
    """Standard normal entries (complex: E|z|^2 = 1); drawn in double, so that every dtype sees the same numbers."""
    wide = torch.complex128 if dtype.is_complex else torch.float64
    return torch.randn(shape, generator=gen, device=DEV, dtype=wide)


def _phases(gen, shape, dtype):
    """Random signs, or unit phases for complex dtypes."""
    z = _normal(gen, shape, dtype)
    return z / z.abs()


def _scrambled(gen, n):
    return torch.rand(n, generator=gen, device=DEV).argsort()


def _orbitals(gen, n, dtype):
    """2n x n orbital matrix: sites 2j and 2j + 1 carry orbital pi(j) and noise of standard deviation 0.7 / sqrt(n)."""
    phi = _normal(gen, (2 * n, n), dtype) * (0.7 / math.sqrt(n))
    column = _scrambled(gen, n).repeat_interleave(2)
    phi[torch.arange(2 * n, device=DEV), column] += _phases(gen, (2 * n,), dtype)
    return phi.to(dtype)


def _pairing(gen, n, dtype):
    """2n x 2n skew pairing matrix: the sites of pairs j and j + n/2 are coupled, plus skew noise."""
    g = _normal(gen, (2 * n, 2 * n), dtype) * (0.25 / math.sqrt(n))
    f = torch.triu(g - g.T, 1)
    half = n // 2
    j = torch.arange(half, device=DEV)
    for a in (0, 1):
        for b in (0, 1):
            f[2 * j + a, 2 * (j + half) + b] += 1.0
    return (f - f.T).to(dtype)


def _occupation(gen, walkers, n):
    """walkers x n int32: one site of every pair, in an order of each walker's own."""
    order = torch.rand(walkers, n, generator=gen, device=DEV).argsort(dim=1)
    side = torch.randint(0, 2, (walkers, n), generator=gen, device=DEV)
    return (2 * order + side).to(torch.int32)


def _moves(gen, occ, steps, k):
    """slot, forward, back: steps x walkers x k int32; every slot of a walker moves at most once, to its pair's other
    site, so a pass over the moves and a pass back restore the occupation."""
    walkers, n = occ.shape
    slot = torch.rand(walkers, n, generator=gen, device=DEV).argsort(dim=1)[:, torch.arange(steps * k, device=DEV) % n]
    back = occ.long().gather(1, slot)
    lay = lambda x: x.reshape(walkers, steps, k).transpose(0, 1).contiguous().to(torch.int32)  # noqa: E731
    return lay(slot), lay(back ^ 1), lay(back)


def _steps(case):
    """Steps of a sweep: as many as its particles allow without one moving twice."""
    return max(1, min(case["steps"], case["n"] // case["k"]))


def _signed_permutation_plus_noise(gen, walkers, n, dtype):
    a = _normal(gen, (walkers, n, n), dtype) * (0.7 / math.sqrt(n))
    at = torch.rand(walkers, n, generator=gen, device=DEV).argsort(dim=1)
    a.scatter_add_(2, at[..., None], _phases(gen, (walkers, n, 1), dtype))
    return a


def _geometry(case):
    """n and k of every walker of a ragged case: a property of the case, not of the seed."""
    r = random.Random(len(case["sizes"]) * 1000 + case["walkers"])
    sizes, ranks = ([int(x) for x in case[key].split(",")] for key in ("sizes", "ranks"))
    n = [r.choice(sizes) for _ in range(case["walkers"])]
    k = [r.choice(ranks) for _ in range(case["walkers"])]
    k[0] = max(ranks)
    return n, k, max(ranks)


def _ragged_inputs(case, seed):
    """Per class of equal (n, k): walkers, A (w, n, n), U, V (vectors, steps + 1 of each), g; all in 64 bits."""
    gen, dtype = _generator(seed), DTYPES[case["dtype"]]
    n_w, k_w, _ = _geometry(case)
    classes = []
    for n, k in sorted(set(zip(n_w, k_w))):
        who = [w for w in range(case["walkers"]) if (n_w[w], k_w[w]) == (n, k)]
        a = _signed_permutation_plus_noise(gen, len(who), n, dtype)
        u, v = (_normal(gen, (case["steps"] + 1, len(who), k, n), dtype) / math.sqrt(n) for _ in range(2))
        classes.append((n, k, who, a, u, v, _normal(gen, (len(who),), dtype)))
    return classes


def _offsets(values):
    out, at = [], 0
    for x in values:
        out.append(at)
        at += x
    return out, at


def _flat(case, classes, pick, size):
    """Walker after walker in one tensor: pick(class) is (w, m) for its walkers, of which size(n, k_max) slots are
    reserved."""
    n_w, _, kmax = _geometry(case)
    at, total = _offsets([size(n, kmax) for n in n_w])
    out = torch.zeros(total, dtype=DTYPES[case["dtype"]], device=DEV)
    for c in classes:
        rows = pick(c).to(out.dtype)
        for i, w in enumerate(c[2]):
            out[at[w]:at[w] + rows.shape[1]] = rows[i]
    return out


def prepare(case, seed):
    task, dtype = case["task"], DTYPES[case["dtype"]]
    gen = _generator(seed)
    if task in ("sweep", "refresh"):
        w, n, pf = case["walkers"], case["n"], case["kind"] == "pf"
        source = (_pairing if pf else _orbitals)(gen, n, dtype)
        occ = _occupation(gen, w, n)
        more = {} if task == "refresh" else {"k": case["k"], "delay": case["delay"], "flush": FLUSH[case["flush"]],
                                             "arith": ARITH[case["arith"]]}
        st = lrugb.LowRankState(case["kind"], w, n, dtype=dtype, **more)
        st.init((st.gather_pairs if pf else st.gather_rows)(source, occ))
        state = {"task": task, "pf": pf, "st": st, "source": source, "turn": 0}
        if task == "refresh":
            slot, forward, _ = _moves(gen, occ, max(1, n // 4), 1)
            moved = occ.scatter(1, slot[..., 0].T.long(), forward[..., 0].T)
            return {**state, "occ": [moved.contiguous(), occ]}
        slot, forward, back = _moves(gen, occ, _steps(case), case["k"])
        return {**state, "k": case["k"], "occ": occ, "slot": slot, "new": [forward, back]}
    if task == "ragged":
        n_w, k_w, kmax = _geometry(case)
        classes = _ragged_inputs(case, seed)
        st = lrugb.LowRankState("det", case["walkers"], n_w, k=kmax, dtype=dtype, delay=case["delay"], k_per_walker=k_w)
        st.init(_flat(case, classes, lambda c: c[3].flatten(1), lambda n, k: n * n))
        vectors = lambda which, t: _flat(case, classes, lambda c: c[which][t].flatten(1), lambda n, k: n * k)  # noqa: E731
        u = [vectors(4, t) for t in range(case["steps"] + 1)]
        v = [vectors(5, t) for t in range(case["steps"] + 1)]
        g = torch.zeros(case["walkers"], dtype=dtype, device=DEV)
        for c in classes:
            g[torch.tensor(c[2], device=DEV)] = c[6].to(dtype)
        return {"task": task, "st": st, "u": [u, [-x for x in u]], "v": v, "g": g, "turn": 0}
    w, n = case["walkers"], case["n"]
    if task == "orbital":
        phi, rows = _orbitals(gen, n, dtype), _occupation(gen, w, n)
        u, v = ((_normal(gen, (w, case["k"], n), dtype) / math.sqrt(n)).to(dtype) for _ in range(2))
        g = _normal(gen, (w,), dtype).to(dtype)
        st = lrugb.LowRankState("det", w, n, k=case["k"], dtype=dtype)
        st.init(st.gather_rows(phi, rows))
        return {"task": task, "st": st, "phi": phi.requires_grad_(), "rows": rows, "u": u.requires_grad_(),
                "v": v.requires_grad_(), "g": g}
    if case["kind"] == "pf":
        f = _pairing(gen, n, dtype)
        at = _occupation(gen, w, n).long()
        a = f[at[:, :, None], at[:, None, :]]
    else:
        a = _signed_permutation_plus_noise(gen, w, n, dtype).to(dtype)
    g = torch.randn(w, generator=gen, device=DEV, dtype=torch.float64)
    return {"task": task, "f": lrugb.slogpf if case["kind"] == "pf" else lrugb.slogdet,
            "a": a.contiguous().requires_grad_(), "g": g}


# ---- one pass -----------------------------------------------------------------


def run(state):
    return {"sweep": _sweep, "refresh": _refresh, "ragged": _ragged, "orbital": _orbital, "slog": _slog}[state["task"]](state)


def _sweep(state):
    st, k, occ, slot = state["st"], state["k"], state["occ"], state["slot"]
    new = state["new"][state["turn"]]
    state["turn"] ^= 1
    ratios, status = [], []
    for t in range(slot.shape[0]):
        if state["pf"]:
            b, idx = st.form_pf_moves(state["source"], occ, slot[t], new[t])
            r, s = st.propose_pf(lrugb.Operand(dense=b, idx=idx, onehot_mask=((1 << k) - 1) << k))
        else:
            v, idx = st.form_row_moves(state["source"], occ, slot[t], new[t])
            r, s = st.propose_det(lrugb.Operand(idx=idx, onehot_mask=(1 << k) - 1), lrugb.Operand(dense=v))
        st.accept()
        st.commit_moves(occ, slot[t], new[t])
        ratios.append(r)
        status.append(s)
    logabs, sign = st.logvalue()
    return {"ratio": torch.stack(ratios), "status": torch.stack(status), "logabs": logabs, "sign": sign,
            "inverse": st.inverse()}


def _refresh(state):
    st, occ = state["st"], state["occ"][state["turn"]]
    state["turn"] ^= 1
    drift = st.refresh((st.gather_pairs if state["pf"] else st.gather_rows)(state["source"], occ))
    logabs, sign = st.logvalue()
    return {"drift": drift, "logabs": logabs, "sign": sign, "inverse": st.inverse()}


def _ragged(state):
    st, u, v = state["st"], state["u"][state["turn"]], state["v"]
    state["turn"] ^= 1
    st.step_persistent(lrugb.Operand(dense=u[0]), lrugb.Operand(dense=v[0]), accept=False)
    log_ratio = st.log_ratio()
    g_u, g_v, g_a = st.backward_det(state["g"])
    ratios, accepted = [], []
    for t in range(1, len(u)):
        r, _, acc = st.step_persistent(lrugb.Operand(dense=u[t]), lrugb.Operand(dense=v[t]))
        ratios.append(r)
        accepted.append(acc)
    logabs, sign = st.logvalue()
    return {"log_ratio": log_ratio, "g_u": g_u, "g_v": g_v, "g_a": g_a, "ratio": torch.stack(ratios),
            "accepted": torch.stack(accepted), "logabs": logabs, "sign": sign, "inverse": st.inverse()}


def _orbital(state):
    log_ratio = lrugb.orbital_log_ratio(state["st"], state["phi"], state["rows"], state["u"], state["v"])
    grads = torch.autograd.grad(log_ratio, (state["phi"], state["u"], state["v"]), state["g"])
    return {"log_ratio": log_ratio.detach(), "g_phi": grads[0], "g_u": grads[1], "g_v": grads[2]}


def _slog(state):
    sign, logabs = state["f"](state["a"])
    (g_a,) = torch.autograd.grad(logabs, (state["a"],), state["g"])
    return {"sign": sign.detach(), "logabs": logabs.detach(), "g_a": g_a}


# ---- what a pass cannot do without ---------------------------------------------


def work(case):
    """Bytes: the inverse has to be read once for every dense vector that meets it step by step, and written once (kept
    state and returned copy); matrices and gradients once.  Flops: the matrix-vector products of those steps, n^3-type
    eliminations at their textbook count; complex products count four."""
    task, b = case["task"], BYTES[case["dtype"]]
    mul = 8 if case["dtype"] in ("c128", "c64") else 2
    if task == "ragged":
        n_w, k_w, _ = _geometry(case)
        steps = case["steps"]
        squares, vectors = sum(n * n for n in n_w), sum(n * k for n, k in zip(n_w, k_w))
        rank = sum(n * n * k for n, k in zip(n_w, k_w))
        # per proposal X = A^{-1} U and Y = V A^{-1} share one read of A^{-1}; gA and the copy are written
        return {"bytes": b * ((steps + 4) * squares + 2 * (steps + 2) * vectors),
                "flops": mul * rank * (2 * steps + 3 + steps)}
    w, n = case["walkers"], case["n"]
    if task == "orbital":
        k = case["k"]
        return {"bytes": b * (w * n * n + 4 * w * k * n + 2 * 2 * n * n), "flops": mul * w * k * n * n * 3}
    if task == "slog":
        return {"bytes": b * w * n * n * 2, "flops": mul * w * n ** 3}
    if task == "refresh":
        pf = mul * w * n ** 3 / 3 if case["kind"] == "pf" else 0
        return {"bytes": b * w * n * n * 4, "flops": mul * w * n ** 3 + pf}
    steps, k = _steps(case), case["k"]
    return {"bytes": b * w * n * n * (steps + 3) + b * w * n * k * steps * 3, "flops": mul * w * n * n * k * steps * 2}


# ---- the same in 64 bits with torch alone ---------------------------------------


def _inverse(a):
    """Inverses of a batch, a few at a time (bounded workspace)."""
    step = max(1, int(2 ** 27 / a.shape[-1] ** 2))
    return torch.cat([torch.linalg.inv(x) for x in a.split(step)])


def _factored(a):
    """Sign, log|det| and inverse of a batch from one factorisation."""
    eye = torch.eye(a.shape[-1], device=DEV, dtype=a.dtype)
    sign, logabs, inverse = [], [], []
    for x in a.split(max(1, int(2 ** 27 / a.shape[-1] ** 2))):
        lu, pivots = torch.linalg.lu_factor(x)
        d = lu.diagonal(dim1=1, dim2=2)
        swaps = (pivots != torch.arange(1, a.shape[-1] + 1, device=DEV)).sum(1) % 2
        sign.append((d / d.abs()).prod(1) * (1 - 2 * swaps))
        logabs.append(d.abs().log().sum(1))
        inverse.append(torch.linalg.lu_solve(lu, pivots, eye.expand_as(x)))
    return torch.cat(sign), torch.cat(logabs), torch.cat(inverse)


def _log(z):
    return torch.log(z) if z.is_complex() else torch.log(z.abs())


def _matrices(pf, source, occ):
    return source[occ[:, :, None], occ[:, None, :]] if pf else source[occ]


def _pf_small(m):
    """Pfaffian of a batch of 2 x 2 or 4 x 4 skew matrices."""
    if m.shape[-1] == 2:
        return m[:, 0, 1]
    return m[:, 0, 1] * m[:, 2, 3] - m[:, 0, 2] * m[:, 1, 3] + m[:, 0, 3] * m[:, 1, 2]


def exact(case, seed):
    task, dtype = case["task"], DTYPES[case["dtype"]]
    gen = _generator(seed)
    wide = torch.complex128 if dtype.is_complex else torch.float64
    if task == "ragged":
        return _exact_ragged(case, seed, wide)
    w, n = case["walkers"], case["n"]
    cost = w * n ** 3 * (4 if dtype.is_complex else 1)
    if cost > 2 ** 40.1 or (task == "sweep" and case["kind"] == "pf" and cost * _steps(case) > 2 ** 38):
        return None
    if task in ("sweep", "refresh"):
        pf = case["kind"] == "pf"
        source = (_pairing if pf else _orbitals)(gen, n, dtype).to(wide)
        occ = _occupation(gen, w, n)
        if task == "refresh":
            slot, forward, _ = _moves(gen, occ, max(1, n // 4), 1)
            moved = occ.scatter(1, slot[..., 0].T.long(), forward[..., 0].T).long()
            sign, logabs, inverse = _factored(_matrices(pf, source, moved))
            before = _inverse(_matrices(pf, source, occ.long()))
            norm = lambda x: torch.linalg.vector_norm(x, dim=(1, 2))  # noqa: E731
            return {"drift": norm(before - inverse) / norm(inverse), "logabs": logabs / 2 if pf else logabs,
                    "sign": None if pf else sign, "inverse": inverse}
        slot, forward, _ = (x.long() for x in _moves(gen, occ, _steps(case), case["k"]))
        return _exact_sweep(pf, source, occ.long(), slot, forward)
    if task == "orbital":
        phi, rows = _orbitals(gen, n, dtype).to(wide), _occupation(gen, w, n).long()
        u, v = ((_normal(gen, (w, case["k"], n), dtype) / math.sqrt(n)).to(dtype).to(wide) for _ in range(2))
        g = _normal(gen, (w,), dtype).to(dtype).to(wide)
        log_ratio, g_u, g_v, g_a = _adjoint(_inverse(phi[rows]), u, v, g)
        return {"log_ratio": log_ratio, "g_phi": torch.zeros_like(phi).index_add_(0, rows.flatten(), g_a.flatten(0, 1)),
                "g_u": g_u, "g_v": g_v}
    if case["kind"] == "pf":
        f = _pairing(gen, n, dtype)
        at = _occupation(gen, w, n).long()
        a = f[at[:, :, None], at[:, None, :]].to(wide)
    else:
        a = _signed_permutation_plus_noise(gen, w, n, dtype).to(dtype).to(wide)
    g = torch.randn(w, generator=gen, device=DEV, dtype=torch.float64)
    sign, logabs = torch.linalg.slogdet(a)
    half = 0.5 if case["kind"] == "pf" else 1.0
    return {"sign": None if half < 1 else sign, "logabs": half * logabs,
            "g_a": half * g[:, None, None] * _inverse(a).conj().transpose(1, 2)}


def _exact_sweep(pf, source, occ, slot, new):
    """The ratios one after the other, and the state behind the last."""
    steps, w, k = slot.shape
    ratios, now = [], occ.clone()
    if not pf:
        # det A_t / det A_0 = det(I + V A_0^{-1} E) over the first t moves
        v = torch.stack([source[new[t]] - source[occ.gather(1, slot[t])] for t in range(steps)], 1).flatten(1, 2)
        cols = slot.transpose(0, 1).flatten(1)
        e = torch.zeros(w, occ.shape[1], steps * k, device=DEV, dtype=source.dtype).scatter_(1, cols[:, None, :], 1.0)
        core = torch.eye(steps * k, device=DEV, dtype=source.dtype) + v @ torch.linalg.solve(_matrices(pf, source, occ), e)
        minors = [torch.linalg.det(core[:, :t * k, :t * k].contiguous()) for t in range(1, steps + 1)]
        ratios = [m / p for m, p in zip(minors, [torch.ones_like(minors[0])] + minors[:-1])]
        now.scatter_(1, cols, new.transpose(0, 1).flatten(1))
    else:
        # a congruence by what the k moved particles change: pf(J + B^T A^{-1} B) / pf(J)
        for t in range(steps):
            a = _matrices(True, source, now)
            nxt = now.scatter(1, slot[t], new[t])
            change = _matrices(True, source, nxt) - a
            e = torch.zeros(w, k, a.shape[1], device=DEV, dtype=a.dtype).scatter_(2, slot[t][..., None], 1.0)
            # rows of the change at the moved particles; the part among them is counted once
            x = change.gather(1, slot[t][..., None].expand(-1, -1, a.shape[1])).clone()
            for p in range(k):
                for q in range(p):
                    x[:, p].scatter_(1, slot[t][:, q:q + 1], 0.0)
            b = torch.cat([x, e], 1).transpose(1, 2)
            j = torch.zeros(2 * k, 2 * k, device=DEV, dtype=a.dtype)
            j[:k, k:], j[k:, :k] = torch.eye(k, device=DEV), -torch.eye(k, device=DEV)
            m = j + b.transpose(1, 2) @ torch.linalg.solve(a, b)
            ratios.append(_pf_small((m - m.transpose(1, 2)) / 2) / _pf_small(j[None]))
            now = nxt
    sign, logabs, inverse = _factored(_matrices(pf, source, now))
    return {"ratio": torch.stack(ratios), "status": None, "logabs": logabs / 2 if pf else logabs,
            "sign": None if pf else sign, "inverse": inverse}


def _adjoint(inverse, u, v, g):
    """log det(I + V A^{-1} U) and its vector-Jacobian products with g (u, v: walkers x k x n vectors)."""
    x, y = inverse @ u.transpose(1, 2), v @ inverse
    core = torch.eye(u.shape[1], device=DEV, dtype=u.dtype) + v @ x
    ry, xr = torch.linalg.solve(core, y), torch.linalg.solve(core.transpose(1, 2), x.transpose(1, 2))
    weigh = lambda t: g[:, None, None] * t.conj()  # noqa: E731
    return _log(torch.linalg.det(core)), weigh(ry), weigh(xr), -weigh((x @ ry).transpose(1, 2))


def _exact_ragged(case, seed, wide):
    n_w, k_w, kmax = _geometry(case)
    dtype, steps, w = DTYPES[case["dtype"]], case["steps"], case["walkers"]
    mats, total = _offsets([n * n for n in n_w])
    vecs, length = _offsets([n * kmax for n in n_w])
    zeros = lambda *shape: torch.zeros(shape, dtype=wide, device=DEV)  # noqa: E731
    out = {"log_ratio": zeros(w), "g_u": zeros(length), "g_v": zeros(length), "g_a": zeros(total),
           "ratio": zeros(steps, w), "accepted": None, "logabs": torch.zeros(w, dtype=torch.float64, device=DEV),
           "sign": zeros(w), "inverse": zeros(total)}
    for n, k, who, *tensors in _ragged_inputs(case, seed):
        a, u, v, g = (x.to(dtype).to(wide) for x in tensors)
        at = torch.tensor(who, device=DEV)
        inverse = _inverse(a)
        out["log_ratio"][at], g_u, g_v, g_a = _adjoint(inverse, u[0], v[0], g)
        out["sign"][at], out["logabs"][at] = torch.linalg.slogdet(a)
        for t in range(1, steps + 1):
            x, y = inverse @ u[t].transpose(1, 2), v[t] @ inverse
            core = torch.eye(k, device=DEV, dtype=wide) + v[t] @ x
            ratio = torch.linalg.det(core)
            inverse = inverse - x @ torch.linalg.solve(core, y)
            out["ratio"][t - 1, at] = ratio
            out["sign"][at] *= ratio / ratio.abs()
            out["logabs"][at] += ratio.abs().log()
        for i, walker in enumerate(who):
            out["g_u"][vecs[walker]:vecs[walker] + k * n] = g_u[i].flatten()
            out["g_v"][vecs[walker]:vecs[walker] + k * n] = g_v[i].flatten()
            out["g_a"][mats[walker]:mats[walker] + n * n] = g_a[i].flatten()
            out["inverse"][mats[walker]:mats[walker] + n * n] = inverse[i].flatten()
    return out
