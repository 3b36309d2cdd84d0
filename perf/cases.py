"""The decoding work that the framework's speed is judged on, each case through the public entry points.

Kinds of case (key "kind"):
  siso      sogrand_decode: soft-output decoding of independent component words
  plain     product_decode: block-turbo decoding, one launch per half iteration
  batched   product_decode(persistent=True): the same in one launch, square or row code x column code
  gldpc     gldpc_decode: QC-GLDPC frames (rows and wrapped diagonals)
  mixed     product_decode_mixed: frames of three codes in one launch
  host      product_decode_host: host buffers in, host buffers out
  serve     Server: a burst of requests of four codes, submitted together and waited for

Inputs are random codewords over BPSK/AWGN at the Eb/N0 the decoders run at, one value per word or frame drawn
uniformly from [lo, hi] dB.
"""
import functools
import math

import numpy as np
import torch

import paper_2310_10737_gb300 as sg

DEV = "cuda"
# primitive polynomials and error-correcting capability of the extended BCH components
SPECS = {"8_4": (8, 0b1011, 1), "16_11": (16, 0b10011, 1), "16_7": (16, 0b10011, 2), "32_26": (32, 0b100101, 1),
         "64_57": (64, 0b1000011, 1), "64_51": (64, 0b1000011, 2), "128_120": (128, 0b10001001, 1)}
MIX = ("32_26", "64_51", "128_120")            # the mixed batch, in 4:2:1 proportion
SERVED = ("32_26", "64_57", "64_51", "128_120")  # the codes a server registers


def listed():
    return [
        # one receiver's block of short words, a call every few microseconds: launch and call overhead
        dict(name="siso small", kind="siso", code="32_26", short=0, words=64, L=1, cap=10000, thr=0.0, apriori=False,
             lo=3.0, hi=3.0),
        # an ordinary batch of component words over the operating range, lists of 4
        dict(name="siso ordinary", kind="siso", code="64_57", short=0, words=20000, L=4, cap=10000, thr=0.0,
             apriori=False, lo=2.0, hi=5.0),
        # one half iteration of somebody's own iterative receiver: long words, a-priori LLRs, the paper's list rule
        dict(name="siso a-priori", kind="siso", code="128_120", short=0, words=5003, L=4, cap=10000, thr=1e-5,
             apriori=True, lo=2.5, hi=4.0),
        # the component simulation: a million words of one code in one launch, cap 10^5
        dict(name="siso million", kind="siso", code="64_57", short=0, words=1000000, L=4, cap=100000, thr=0.0,
             apriori=False, lo=2.0, hi=5.0),
        # the plain method as the paper states it: 200 frames, 4 iterations, one launch per half
        dict(name="plain", kind="plain", code="32_26", short=0, frames=200, L=4, cap=10000, thr=0.0, alpha=0.5,
             iters=4, lo=3.0, hi=3.0),
        # one frame that somebody waits for
        dict(name="batched one frame", kind="batched", code="64_57", col="64_57", short=0, frames=1, L=4, cap=10000,
             thr=0.0, alpha=0.5, iters=20, lo=3.0, hi=3.0),
        # the headline workload: a large batch of eBCH(64,57)^2 over 2.5-4 dB
        dict(name="batched large", kind="batched", code="64_57", col="64_57", short=0, frames=20000, L=4, cap=10000,
             thr=0.0, alpha=0.5, iters=20, lo=2.5, hi=4.0),
        # rate adaptation: shortened (60,53) rows, (64,51) columns, a ragged batch with the paper's list rule
        dict(name="batched rectangular", kind="batched", code="64_57", col="64_51", short=4, frames=401, L=4,
             cap=10000, thr=1e-5, alpha=0.5, iters=20, lo=2.5, hi=4.0),
        # the paper's QC-GLDPC code at its operating point
        dict(name="gldpc", kind="gldpc", code="32_26", short=0, frames=2000, L=4, cap=10000, thr=1e-5, alpha=0.6,
             iters=20, lo=2.25, hi=3.0),
        # codes of uneven length in one launch, 4:2:1
        dict(name="mixed", kind="mixed", frames=2800, L=4, cap=10000, thr=0.0, alpha=0.5, iters=20, lo=2.5, hi=4.0),
        # a receiver on host buffers: copies in and out count
        dict(name="host", kind="host", code="64_57", col="64_57", short=0, frames=6000, L=4, cap=10000, thr=0.0,
             alpha=0.5, iters=20, lo=2.5, hi=4.0),
        # serving: a burst of requests of 1-64 frames of four codes
        dict(name="serve", kind="serve", requests=24, most=64, epoch=16, L=4, cap=10000, thr=0.0, alpha=0.5, iters=20,
             lo=2.5, hi=4.0),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("siso", "siso", "siso", "batched", "batched", "batched", "plain", "gldpc", "mixed", "host", "serve"))
    L = rng.choice((1, 2, 4, 4, 4, 8, 16))
    thr = rng.choice((0.0, 0.0, 0.0, 1e-4, 1e-5, 1e-6))
    lo = rng.uniform(2.0, 3.5)
    c = dict(kind=kind, L=L, cap=_log_int(rng, 500, 10000), thr=thr)
    if kind == "siso":
        code = rng.choice(("16_11", "32_26", "64_57", "64_57", "64_51", "128_120"))
        lo = rng.uniform(2.0, 4.0)
        return dict(c, code=code, short=rng.choice((0, 0, rng.randint(1, 5))),
                    words=_log_int(rng, 32, {"64_51": 20000, "128_120": 100000}.get(code, 200000)),
                    cap=min(c["cap"], 16000 if code != "16_11" else 400), apriori=rng.random() < 0.4, lo=lo,
                    hi=lo + rng.uniform(0.0, 1.5))
    c.update(L=min(L, 4), alpha=rng.choice((0.5, 0.5, 0.6)), iters=rng.choice((4, 10, 20)), lo=max(lo, 2.5),
             hi=max(lo, 2.5) + rng.uniform(0.0, 1.0))
    if kind == "plain":
        return dict(c, code=rng.choice(("32_26", "64_57")), short=rng.choice((0, 3)), frames=_log_int(rng, 1, 2000))
    if kind == "gldpc":
        return dict(c, code="32_26", short=0, alpha=0.6, frames=_log_int(rng, 1, 8000))
    if kind == "mixed":
        return dict(c, frames=_log_int(rng, 7, 2800))
    if kind == "serve":
        return dict(c, requests=rng.randint(1, 32), most=rng.choice((4, 16, 64)), epoch=rng.choice((2, 8, 16)))
    code, col, short = rng.choice((("32_26", "32_26", 0), ("64_57", "64_57", 0), ("64_57", "64_57", 0),
                                   ("64_57", "64_57", 4), ("64_51", "64_51", 0), ("64_57", "64_51", 0),
                                   ("128_120", "128_120", 0)))
    most = {"32_26": 20000, "64_57": 10000}.get(col, 1000)
    return dict(c, code=code, col=col, short=short, frames=_log_int(rng, 1, most))


# ---------------------------------------------------------------------------
# codes: parity checks, generators, and the handles that a program keeps
# ---------------------------------------------------------------------------
def _nullspace(H):
    """A basis (rows) of {x : H x = 0 over GF(2)}."""
    M, pivots = np.array(H, np.uint8), []
    for col in range(M.shape[1]):
        r = len(pivots)
        if r == M.shape[0]:
            break
        nz = np.nonzero(M[r:, col])[0]
        if not nz.size:
            continue
        M[[r, r + nz[0]]] = M[[r + nz[0], r]]
        hit = M[:, col].astype(bool)
        hit[r] = False
        M[hit] ^= M[r]
        pivots.append(col)
    free = np.setdiff1d(np.arange(M.shape[1]), pivots)
    G = np.zeros((free.size, M.shape[1]), np.uint8)
    G[np.arange(free.size), free] = 1
    G[:, pivots] = M[:len(pivots), free].T
    return G


@functools.lru_cache(None)
def _parity(name, short=0):
    """Parity-check matrix of an extended BCH code (columns alpha^i, alpha^3i, ..., then the overall parity),
    shortened by its first `short` positions."""
    n, poly, t = SPECS[name]
    m = n.bit_length() - 1
    exp = [1]
    for _ in range(n - 2):
        x = exp[-1] << 1
        exp.append(x ^ poly if x & n else x)
    H = np.zeros((t * m + 1, n), np.uint8)
    for i in range(n - 1):
        for j in range(t):
            v = exp[((2 * j + 1) * i) % (n - 1)]
            H[j * m:(j + 1) * m, i] = [(v >> b) & 1 for b in range(m)]
    H[-1] = 1
    return np.ascontiguousarray(H[:, short:])


@functools.lru_cache(None)
def _generator(name, short=0, diag=False):
    H = _parity(name, short)
    if diag:  # every row and every wrapped diagonal of the n x n array a component word
        m, n = H.shape
        X = np.zeros((2 * n * m, n * n), np.uint8)
        for w in range(n):
            X[w * m:(w + 1) * m, w * n:(w + 1) * n] = H
            X[(n + w) * m:(n + w + 1) * m][:, [((w + j) % n) * n + j for j in range(n)]] = H
        H = X
    return torch.from_numpy(_nullspace(H)).to(DEV, torch.float32)


@functools.lru_cache(None)
def _handle(name, short, cap):
    """The code object of a program: made once, its order tables covering the cap."""
    c = sg.Code(_parity(name, short))
    c.reserve(cap)
    return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _sigma2(case, count, rate, g):
    db = case["lo"] + (case["hi"] - case["lo"]) * torch.rand(count, generator=g, device=DEV)
    return 1.0 / (2.0 * rate * 10.0 ** (db / 10.0))


def _bits(G, count, g):
    u = torch.randint(0, 2, (count, G.shape[0]), generator=g, device=DEV).float()
    return torch.remainder(u @ G, 2.0)


def _llr(x, s2, g):
    s2 = s2.view(-1, *([1] * (x.dim() - 1)))
    y = (1.0 - 2.0 * x) + torch.sqrt(s2) * torch.randn(x.shape, generator=g, device=DEV)
    return (2.0 * y / s2).contiguous()


def _frames(case, code, short, col, col_short, count, g):
    """Product-code frames [count, n_col, n_row]."""
    Gr, Gc = _generator(code, short), _generator(col, col_short)
    (kr, nr), (kc, nc) = Gr.shape, Gc.shape
    out = torch.empty((count, nc, nr), device=DEV)
    s2 = _sigma2(case, count, kr * kc / (nr * nc), g)
    for f in range(0, count, 4096):
        k = min(4096, count - f)
        u = torch.randint(0, 2, (k, kc, kr), generator=g, device=DEV).float()
        x = torch.remainder(Gc.T @ torch.remainder(u @ Gr, 2.0), 2.0)
        out[f:f + k] = _llr(x, s2[f:f + k], g)
    return out


def _words(case, seed):
    g = torch.Generator(device=DEV).manual_seed(seed)
    G = _generator(case["code"], case["short"])
    x = _bits(G, case["words"], g)
    s2 = _sigma2(case, case["words"], G.shape[0] / G.shape[1], g)
    ch = _llr(x, s2, g)
    # a-priori LLRs as an earlier half iteration leaves them: a second, weaker look at the same bits, scaled
    a = (0.5 * _llr(x, 2.0 * s2, g)).contiguous() if case["apriori"] else None
    return ch, a


def _split(frames):
    """4:2:1, at least one frame of each code."""
    a, b = max(1, 4 * frames // 7), max(1, 2 * frames // 7)
    return a, b, max(1, frames - a - b)


def prepare(case, seed):
    g = torch.Generator(device=DEV).manual_seed(seed)
    kind, s = case["kind"], {"case": case}
    if kind == "siso":
        s["code"] = _handle(case["code"], case["short"], case["cap"])
        s["ch"], s["a"] = _words(case, seed)
    elif kind == "mixed":
        s["groups"] = [(_handle(c, 0, case["cap"]), _frames(case, c, 0, c, 0, k, g))
                       for c, k in zip(MIX, _split(case["frames"]))]
    elif kind == "gldpc":
        G = _generator(case["code"], 0, True)
        n = math.isqrt(G.shape[1])
        x = _bits(G, case["frames"], g).view(-1, n, n)
        s["code"] = _handle(case["code"], 0, case["cap"])
        s["llr"] = _llr(x, _sigma2(case, case["frames"], G.shape[0] / (n * n), g), g)
    elif kind == "serve":
        r = np.random.RandomState(1000 * case["requests"] + case["most"])  # the mix of requests is the case's own
        codes = [_handle(c, 0, case["cap"]) for c in SERVED]
        s["server"] = sg.Server(codes, [case["requests"] * case["most"]] * len(codes), L=case["L"],
                                query_cap=case["cap"], thr=case["thr"], alpha=case["alpha"], max_iter=case["iters"],
                                epoch_halves=case["epoch"])
        s["requests"] = []
        for _ in range(case["requests"]):
            k, f = r.randint(len(SERVED)), r.randint(1, case["most"] + 1)
            n = codes[k].n
            s["requests"].append((k, _frames(case, SERVED[k], 0, SERVED[k], 0, f, g).cpu().pin_memory(),
                                  _host_out(f, n, n)))
    else:
        short = case["short"]
        col = case.get("col", case["code"])
        # a shortened code with itself as the column code stays square; with another, only the rows are shortened
        col_short = short if col == case["code"] else 0
        s["code"] = _handle(case["code"], short, case["cap"])
        s["col"] = _handle(col, col_short, case["cap"])
        s["llr"] = _frames(case, case["code"], short, col, col_short, case["frames"], g)
        if kind == "host":
            s["llr"] = s["llr"].cpu().pin_memory()
            s["out"] = _host_out(case["frames"], s["col"].n, s["code"].n)
    return s


def _host_out(frames, nc, nr):
    return dict(bits=torch.empty((frames, (nr * nc + 7) // 8), dtype=torch.uint8).pin_memory(),
                half_iters=torch.empty(frames, dtype=torch.int32).pin_memory(),
                status=torch.empty(frames, dtype=torch.uint8).pin_memory(),
                queries=torch.empty(frames, dtype=torch.int64).pin_memory())


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def _tensors(out):
    """What the call decoded and counted (without the call's own timings)."""
    return {k: v for k, v in out.items() if k not in ("timing_ms", "launches")}


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "siso":
        return sg.sogrand_decode(state["code"], state["ch"], state["a"], L=case["L"], query_cap=case["cap"],
                                 thr=case["thr"])
    p = dict(L=case["L"], query_cap=case["cap"], thr=case["thr"], alpha=case["alpha"], max_iter=case["iters"])
    if kind == "mixed":
        outs, info = sg.product_decode_mixed(state["groups"], **p)
        return [_tensors(o) for o in outs] + [_tensors(info)]
    if kind == "gldpc":
        return _tensors(sg.gldpc_decode(state["code"], state["llr"], **p))
    if kind == "serve":
        server = state["server"]
        tickets = [server.submit(k, llr, out)[0] for k, llr, out in state["requests"]]
        for t in tickets:
            if not server.wait(t)[0]:
                raise RuntimeError("a request did not finish")
        return {key: torch.cat([out[key].flatten() for _, _, out in state["requests"]])
                for key in ("bits", "half_iters", "status", "queries")}
    if kind == "host":
        return sg.product_decode_host(state["code"], state["llr"], out=state["out"], col_code=state["col"], **p)
    return _tensors(sg.product_decode(state["code"], state["llr"], col_code=state["col"],
                                      persistent=kind == "batched", **p))


# Codebook queries of an average word (per half iteration for the frames) and half iterations of an average frame, over
# the declared Eb/N0 with lists of 4; each query takes about six XORs and products.
QUERIES = {"8_4": 20, "16_11": 60, "16_7": 200, "32_26": 200, "64_57": 400, "64_51": 9000, "128_120": 900}
HALVES = 4


def work(case):
    kind = case["kind"]
    if kind == "siso":
        n, m = SPECS[case["code"]][0] - case["short"], (SPECS[case["code"]][0] + 63) // 64
        w = case["words"]
        out = n * 9 + 4 + 8 + 4 + case["L"] * (8 * m + 4)
        return {"bytes": w * (n * (8 if case["apriori"] else 4) + out),
                "flops": 6 * w * min(case["cap"], QUERIES[case["code"]] * case["L"] / 4)}

    def frames(code, col, short, count):
        nr, nc = SPECS[code][0] - short, SPECS[col][0]
        # LLRs in, bits and the frame's counters out; the decoded words' queries
        return (count * (4 * nr * nc + nr * nc / 8 + 29),
                6 * count * HALVES * max(nr, nc) * min(case["cap"], max(QUERIES[code], QUERIES[col]) * case["L"] / 4))

    if kind == "mixed":
        each = [frames(c, c, 0, k) for c, k in zip(MIX, _split(case["frames"]))]
    elif kind == "serve":
        each = [frames(c, c, 0, case["requests"] * (case["most"] + 1) / 2 / len(SERVED)) for c in SERVED]
    else:
        each = [frames(case["code"], case.get("col", case["code"]), case["short"], case["frames"])]
    return {"bytes": sum(b for b, _ in each), "flops": sum(f for _, f in each)}


# ---------------------------------------------------------------------------
# the soft outputs in 64 bits
# ---------------------------------------------------------------------------
@functools.lru_cache(None)
def _subsets(w, m, lo, n):
    """The w-subsets of {lo..n} with sum m, in lexicographic order, as tuples."""
    if w == 0:
        return [()] if m == 0 else []
    got = []
    for r in range(lo, n + 1):
        if m < w * r + w * (w - 1) // 2:
            break
        if m - r > (w - 1) * n - (w - 1) * (w - 2) // 2:
            continue
        got += [(r,) + t for t in _subsets(w - 1, m - r, r + 1, n)]
    return got


@functools.lru_cache(None)
def _order(n, c, parity, most):
    """The first `most` patterns of one parity by cost = rank sum + c weight, then weight, then lexicographic rank
    vector: 0-based ranks [patterns, 15], n in the unused places, and the weights."""
    got = []
    for cost in range(n * (n + 1) // 2 + c * n + 1):
        for w in range(parity, min(n, 15) + 1, 2):
            m = cost - c * w
            if m < w * (w + 1) // 2:
                break
            got += _subsets(w, m, 1, n)
        if len(got) >= most:
            break
    got = got[:most]
    e = np.full((len(got), 15), n, np.int64)
    for i, t in enumerate(got):
        e[i, :len(t)] = np.array(t, np.int64) - 1
    top = max(1, max(len(t) for t in got))
    return torch.from_numpy(e[:, :top]).to(DEV), torch.tensor([len(t) for t in got], device=DEV)


def exact(case, seed):
    """SOGRAND's soft outputs (even codes: the search and the soft output within the parity class of the hard
    decision), the masses in 64 bits.  None for the frames, whose outputs are whole numbers, and for batches that would
    take long."""
    if case["kind"] != "siso" or case["words"] > 25000 or (case["code"] == "64_51" and case["words"] > 3000):
        return None
    ch, a = _words(case, seed)
    lam = ch + a if a is not None else ch
    H = _parity(case["code"], case["short"])
    m, n = H.shape
    W, L, cap = case["words"], case["L"], min(case["cap"], 1 << (n - 1))
    k = n - m
    log_phi = (k * math.log(2) + math.log1p(-2.0 ** -k)) - ((n - 1) * math.log(2) + math.log1p(-2.0 ** (1 - n)))
    hcol = torch.tensor([sum(int(H[t, i]) << t for t in range(m)) for i in range(n)], device=DEV)
    mag, perm = torch.sort(lam.abs(), dim=1, stable=True)
    y = (lam < 0).long()
    s0 = torch.zeros(W, dtype=torch.long, device=DEV)
    for i in range(n):
        s0 ^= y[:, i] * hcol[i]
    par = y.sum(1) & 1
    qa = torch.clamp(torch.floor(mag.double() * 256 + 0.5), max=2.0 ** 20 - 1).long()
    r = torch.arange(1, n + 1, device=DEV)
    sx, sxx, sy, sxy = n * (n + 1) // 2, n * (n + 1) * (2 * n + 1) // 6, qa.sum(1), (qa * r).sum(1)
    nb = n * sxy - sx * sy
    top = 2 * (sy * (n * sxx - sx * sx) - nb * sx) + n * nb
    c = torch.where((nb > 0) & (top >= 0), torch.div(top, (2 * n * nb).clamp(min=1), rounding_mode="floor"), 0)
    c = c.clamp(0, n)
    t = torch.cat([torch.exp(-mag.double()), torch.ones((W, 1), device=DEV, dtype=torch.float64)], 1)
    h = torch.cat([hcol[perm], torch.zeros((W, 1), device=DEV, dtype=torch.long)], 1)
    u, b = torch.zeros(W, device=DEV, dtype=torch.float64), torch.zeros(W, device=DEV, dtype=torch.float64)
    for e in range(n):  # the nonzero patterns' mass: even part, odd part
        u, b = u + b * t[:, e], b + t[:, e] + u * t[:, e]
    total = torch.where(par == 0, u, b)
    app = lam.double().clone()
    pm = torch.ones(W, device=DEV, dtype=torch.float64)
    lapp = torch.zeros((W, L), device=DEV, dtype=torch.float64)
    rank_of = torch.argsort(perm, dim=1)  # bit -> rank
    kind_of = c * 2 + par
    for kd in torch.unique(kind_of).tolist():
        todo = torch.nonzero(kind_of == kd).flatten()
        for most in (min(cap, 1500), cap):
            E, wt = _order(n, kd // 2, kd % 2, most)
            Q = E.shape[0]
            step = max(1, 3_000_000 // (Q * E.shape[1]))
            late = []
            for at in range(0, todo.numel(), step):
                ids = todo[at:at + step]
                syn, mass = s0[ids][:, None].expand(-1, Q).clone(), torch.ones((ids.numel(), Q), device=DEV, dtype=torch.float64)
                for x in range(E.shape[1]):
                    syn ^= h[ids][:, E[:, x]]
                    mass *= t[ids][:, E[:, x]]
                hit = syn == 0
                nth = hit.long().cumsum(1)
                done = nth[:, -1] >= L
                queried = torch.where(wt > 0, mass, 0.0).cumsum(1)
                place = [torch.where(nth[:, -1] > l, (nth == l + 1).long().argmax(1), Q) for l in range(L)]
                p = torch.stack([torch.where(q < Q, mass.gather(1, q.clamp(max=Q - 1)[:, None])[:, 0], 0.0) for q in place], 1)
                stop = torch.where(done, place[L - 1], Q - 1)
                used = torch.where(done, L, nth[:, -1])
                if case["thr"] > 0:  # the list rule, checked at each listed word
                    found = torch.zeros_like(done)
                    for l in range(L):
                        q = place[l].clamp(max=Q - 1)
                        rest = (total[ids] - queried.gather(1, q[:, None])[:, 0]).clamp(min=0) * math.exp(log_phi)
                        low = (place[l] < Q) & (rest / (rest + p[:, :l + 1].sum(1)) < case["thr"]) & ~found
                        stop, used = torch.where(low, q, stop), torch.where(low, l + 1, used)
                        found |= low
                    done |= found
                if most < cap:
                    late.append(ids[~done])
                else:
                    done |= True
                p = torch.where(torch.arange(L, device=DEV) < used[:, None], p, 0.0)
                rest = (total[ids] - queried.gather(1, stop[:, None])[:, 0]).clamp(min=0) * math.exp(log_phi)
                D = rest + p.sum(1)
                x = lam[ids].double()
                some = done & (used > 0)
                a0, a1 = (rest / D)[:, None] * torch.sigmoid(x), (rest / D)[:, None] * torch.sigmoid(-x)
                for l in range(L):
                    ranks = E[place[l].clamp(max=Q - 1)]
                    flip = (rank_of[ids][:, :, None] == ranks[:, None, :]).any(2)
                    one = (y[ids].bool() ^ flip)
                    w = (p[:, l] / D)[:, None]
                    a0, a1 = a0 + torch.where(one, 0.0, w), a1 + torch.where(one, w, 0.0)
                app[ids[some]] = torch.log(a0 / a1)[some]
                pm[ids[some]] = (rest / D)[some]
                lapp[ids[some]] = (p / D[:, None])[some]
            if most == cap:
                break
            todo = torch.cat(late)
            if not todo.numel():
                break
    return dict(hard=None, llr_app=app, llr_ext=torch.where((lapp.sum(1) > 0)[:, None], app - lam.double(), 0.0),
                p_miss=pm, queries=None, list_words=None, list_app=lapp, list_count=None)
