"""Performance cases: the calls that a program using this library spends its time in, and their exact results.

Each case is one pass through the public entry points of ``paper_0908_4403_gb300.heget``: cross sections (one call, a
replayed graph, with per-event weights, a mixed batch), |M|^2 of given momenta, phase-space generation and
distributions.  Sizes are those of the benchmark's workloads and of the tests, with smaller and ragged ones beside
them.  ``exact`` restates the same quantities in plain torch, in 64 bits, from their definitions.

A case's fields:
  kind       xsec | xsec_sync | graph | amp2 | phase_space | hist | batch
  n, N       photons and points (batch: the requests are spread over N points at most each)
  precision  32 or 64
  alg        "tree" (the default ordering sum) or "subset"
  sampler    "fixed" (500 GeV), "uniform" (200 .. 2000 GeV) or "toy" (14 TeV toy PDF, floor 100 GeV)
  weights    xsec: also return every event's weight
  mask       amp2: evaluate the helicities with lambda_1 = +1 only (else all)
"""
import ctypes
import math

import torch

from paper_0908_4403_gb300 import heget as H

ALPHA, QU, PT_MIN, ETA_MAX, DR_MIN = 1 / 137.035999, 2 / 3, 20.0, 2.5, 0.4
HIST_SPECS = [(H.HEGET_OBS_PT_MAX, 40, 20.0, 820.0), (H.HEGET_OBS_PT, 40, 20.0, 820.0),
              (H.HEGET_OBS_ETA, 50, -2.5, 2.5), (H.HEGET_OBS_DR, 48, 0.4, 5.2), (H.HEGET_OBS_DR_MIN, 48, 0.4, 5.2)]


def _case(name, kind, n, N, precision=32, alg="tree", sampler="toy", weights=False, mask=False):
    return {"name": name, "kind": kind, "n": n, "N": N, "precision": precision, "alg": alg, "sampler": sampler,
            "weights": weights, "mask": mask}


def listed():
    return [
        # the smallest call: a quick estimate at a fixed energy, waited for (an adaptive loop's inner step)
        _case("xsec_n2_1k", "xsec_sync", 2, 1000, sampler="fixed"),
        # the step of a Monte Carlo loop over seeds, captured once and replayed; a ragged size
        _case("graph_n3_10k", "graph", 3, 10007),
        # the two-photon check workload: FP64, fixed energy
        _case("xsec_n2_64k_fp64", "xsec", 2, 65536, precision=64, sampler="fixed"),
        # the headline step: four photons, toy PDF, a million points
        _case("xsec_n4_1m", "xsec", 4, 1048576),
        # the plain FP64 arm of the same workload, with every event's weight kept for an analysis
        _case("xsec_n4_256k_fp64_weights", "xsec", 4, 262144, precision=64, weights=True),
        # six photons by the ordering tree (the default)
        _case("xsec_n6_256k", "xsec", 6, 262144),
        # eight photons, uniform energies, by the subset recursion
        _case("xsec_n8_64k_subset", "xsec", 8, 65536, alg="subset", sampler="uniform"),
        # |M|^2 of a program's own events (another generator's), one polarisation of the first photon, odd row count
        _case("amp2_n5_50k_mask", "amp2", 5, 50001, mask=True),
        # |M|^2 in FP64 of seven-photon events: the accuracy reference of a reweighting
        _case("amp2_n7_20k_fp64_subset", "amp2", 7, 20011, precision=64, alg="subset"),
        # unweighted phase-space points written out for another program: every output
        _case("phase_space_n5_500k", "phase_space", 5, 500000),
        # five distributions of the headline step's events from their weights
        _case("hist_n4_1m", "hist", 4, 1048576),
        # one batch of a serving loop: 24 requests of mixed n, size and precision
        _case("batch_mix", "batch", 8, 65536, alg="subset"),
    ]


# rough cost of one point, nanoseconds, for bounding the drawn sizes (largest listed case: about 4.5 ms)
_TREE_NS = {2: 2, 3: 2.5, 4: 3, 5: 5, 6: 20, 7: 220, 8: 2600}
_SUBSET_NS = {2: 3, 3: 3, 4: 4, 5: 5, 6: 8, 7: 16, 8: 40}
_FP64_NS = {2: 6, 3: 10, 4: 20, 5: 60, 6: 90, 7: 250, 8: 700}


def _draw_size(rng, lo, hi):
    N = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    return N | 1 if rng.random() < 0.5 else N


def draw(rng):
    kind = rng.choice(["xsec", "xsec", "xsec", "xsec_sync", "graph", "amp2", "amp2", "phase_space", "hist", "batch"])
    n = rng.randint(2, 8)
    precision = rng.choice([32, 32, 64])
    # what users pick: the tree by default in FP32, the recursion for many photons and for FP64 beyond five
    alg = "subset" if (n >= 7 or (precision == 64 and n >= 6)) else rng.choice(["tree", "tree", "subset"])
    sampler = rng.choice(["toy", "toy", "uniform", "fixed"])
    ns = _FP64_NS[n] if precision == 64 else (_TREE_NS if alg == "tree" else _SUBSET_NS)[n]
    if kind == "amp2":
        ns *= 4   # every row is evaluated; a tenth or more of the generated points are not
    elif kind in ("phase_space", "hist"):
        precision, alg, ns = 64 if kind == "phase_space" else 32, "tree" if n <= 6 else "subset", 4 + n
        if kind == "hist":
            sampler = rng.choice(["toy", "uniform"])
    elif kind == "batch":
        # FP32 and FP64 requests of every n
        c = _case("", "batch", 8, _draw_size(rng, 2000, 65536), alg="subset")
        del c["name"]
        return c
    hi = min(1048576, 4.0e6 / ns)
    c = _case("", kind, n, _draw_size(rng, 500, max(600, hi)), precision=precision, alg=alg, sampler=sampler,
              weights=kind == "xsec" and precision == 64 and rng.random() < 0.5,
              mask=kind == "amp2" and rng.random() < 0.3)
    del c["name"]
    return c


# ---------------------------------------------------------------------------------------------------------------------
# the calls
# ---------------------------------------------------------------------------------------------------------------------

class _State:
    """What a program keeps between calls: a context (or graph) and its device buffers."""

    def __init__(self, case, seed):
        self.kind = case["kind"]
        self.n, self.N = int(case["n"]), int(case["N"])
        self.precision = int(case["precision"])
        self.seed = _stream_seed(seed)
        self.sampler = _sampler(case["sampler"])
        self.ctx = H.heget_create(torch.cuda.current_device())
        self.graph = None
        H.heget_set_algorithm(self.ctx, H.HEGET_ALG_SUBSET if case["alg"] == "subset" else H.HEGET_ALG_TREE)

    def __del__(self):
        if self.graph is not None:
            H.heget_graph_destroy(self.graph)
        H.heget_destroy(self.ctx)


def _stream_seed(seed):
    return (0x0908440300000001 + int(seed) * 0x9E3779B97F4A7C15) % (1 << 64)


def _sampler(name):
    if name == "fixed":
        return H.sampler_fixed(500.0)
    return H.sampler_uniform(200.0, 2000.0) if name == "uniform" else H.sampler_toy_pdf()


def _result_buffer(*count):
    """Device room for one result (or for `count` of them), and its fields: doubles (sigma, error, sums, acceptance: each by
    itself, they differ by orders of magnitude) and counts."""
    assert ctypes.sizeof(H.heget_xsec_result) == 80
    b = torch.zeros(*count, 10, dtype=torch.float64, device="cuda")
    return b, {"values": [b[..., k] for k in range(5)], "counts": b.view(torch.int64)[..., 6:]}


def _columns(hist):
    """Every histogram's bins of sum w and of sum w^2, as views."""
    out, at = [], 0
    for q in HIST_SPECS:
        rows = hist[at:at + 2 * (q[1] + 2)].view(-1, 2)
        out += [rows[:, 0], rows[:, 1]]
        at += rows.numel()
    return out


def _batch_requests(case, seed):
    """24 requests: n in 2..8, FP32 and FP64 alike, N log-uniform from 1000 up to the case's, smaller from n = 7 on in FP64."""
    g = torch.Generator().manual_seed(7)   # the mix of a case is fixed by its size; the events change with the seed
    reqs = []
    for k in range(24):
        n = 2 + k % 7
        precision = 64 if (k // 7) % 2 else 32
        u = float(torch.rand(1, generator=g, dtype=torch.float64))
        N = int(1000 * (int(case["N"]) / 1000.0) ** u)
        if precision == 64 and n >= 6:
            N = max(500, N // 8)
        reqs.append({"n": n, "precision": precision, "seed": (_stream_seed(seed) + 977 * k) % (1 << 64), "i0": 4096 * k,
                     "N": N})
    return reqs


def prepare(case, seed):
    s = _State(case, seed)
    kind, n, N = s.kind, s.n, s.N
    if kind in ("xsec", "graph"):
        s.result, s.out = _result_buffer()
        s.w = torch.empty(N, dtype=torch.float64, device="cuda") if case["weights"] else None
        if s.w is not None:
            s.out["weights"] = s.w
        if kind == "graph":
            s.graph = H.heget_graph_xsec(s.ctx, n, N, s.sampler, s.precision, s.result)
    elif kind == "amp2":
        s.mom = _events(case, seed)
        s.amp2 = torch.empty(N, dtype=torch.float64, device="cuda")
        s.mask = _helicity_mask(n) if case["mask"] else None
    elif kind == "phase_space":
        f = dict(dtype=torch.float64, device="cuda")
        s.out = {"momenta": torch.empty(N, n + 2, 4, **f), "weights": torch.empty(N, **f), "sqrt_s": torch.empty(N, **f),
                 "y": torch.empty(N, **f), "mask": torch.empty(N, dtype=torch.uint8, device="cuda"),
                 "tries": torch.empty(N, dtype=torch.int32, device="cuda")}
    elif kind == "hist":
        s.w = torch.empty(N, dtype=torch.float64, device="cuda")
        result, _ = _result_buffer()
        H.heget_xsec_async(s.ctx, n, s.seed, 0, N, s.sampler, s.precision, result, w_out=s.w)
        s.hist = torch.empty(H.hist_bins(HIST_SPECS), dtype=torch.float64, device="cuda")
        s.out = _columns(s.hist)
    elif kind == "batch":
        s.requests, s.out = _batch_requests(case, seed), []
        for a in range(2, 9):
            mine = [q for q in s.requests if q["n"] == a]
            rows, fields = _result_buffer(len(mine))
            s.out.append(fields)
            for q, row in zip(mine, rows):
                q["sampler"], q["result_dev"] = s.sampler, row
    return s


def run(s):
    if s.kind == "xsec":
        H.heget_xsec_async(s.ctx, s.n, s.seed, 0, s.N, s.sampler, s.precision, s.result, w_out=s.w)
        return s.out
    if s.kind == "xsec_sync":
        r = H.heget_xsec(s.ctx, s.n, s.N, s.seed, s.sampler, s.precision)
        return {"values": [r.sigma_fb, r.err_fb, r.sum_w, r.sum_w2, r.accept],
                "counts": [r.n_pass, r.n_total, r.n_tries, r.n_escalated]}
    if s.kind == "graph":
        H.heget_graph_launch(s.graph, s.seed)
        return s.out
    if s.kind == "amp2":
        H.heget_amp2(s.ctx, s.n, s.N, s.mom, s.amp2, hel_mask=s.mask, precision=s.precision)
        return s.amp2
    if s.kind == "phase_space":
        o = s.out
        H.heget_phase_space_ex(s.ctx, s.seed, 0, s.N, s.n, s.sampler, momenta=o["momenta"], weights=o["weights"],
                               sqrt_s=o["sqrt_s"], y=o["y"], mask=o["mask"], tries=o["tries"])
        return o
    if s.kind == "hist":
        H.heget_hist(s.ctx, s.n, s.seed, 0, s.N, s.sampler, s.w, HIST_SPECS, s.hist)
        return s.out
    H.heget_xsec_batch(s.ctx, s.requests)
    return s.out


# ---------------------------------------------------------------------------------------------------------------------
# work
# ---------------------------------------------------------------------------------------------------------------------

# share of the generated points that pass the cuts (toy PDF and uniform energies alike, to a few per cent)
_PASS = {2: 0.9, 3: 0.7, 4: 0.57, 5: 0.45, 6: 0.34, 7: 0.3, 8: 0.26}


def _amp_flops(n):
    """Flops of one point's helicity sum with the orderings regrouped by photon set and met in the middle: the fewest of
    the ways known to this library."""
    m = n // 2
    f = sum(math.comb(n, k) * 2 ** k * (12 * k + 12 if k > 1 else 12) for k in range(1, m + 1))
    f += sum(math.comb(n, k) * 2 ** k * (12 * k + 12 if k > 1 else 12) for k in range(1, n - m))
    f += math.comb(n, n - m) * 2 ** (n - m) * 12 * (n - m) + math.comb(n, m) * 2 ** n * 8
    return 2.0 * f


def _gen_flops(n):
    """Sampler, RAMBO and cuts of one point: about 45 operations a photon, 10 a pair, 60 besides."""
    return 60.0 + 45.0 * n + 10.0 * n * (n - 1) / 2


def _xsec_work(n, N):
    return {"bytes": 80.0, "flops": N * (_gen_flops(n) + _PASS[n] * _amp_flops(n))}


def work(case):
    kind, n, N = case["kind"], int(case["n"]), int(case["N"])
    if kind in ("xsec", "xsec_sync", "graph"):
        w = _xsec_work(n, N)
        w["bytes"] += 8.0 * N if case["weights"] else 0.0
        return w
    if kind == "amp2":
        return {"bytes": N * (32.0 * (n + 2) + 8.0), "flops": N * _amp_flops(n) * (0.5 if case["mask"] else 1.0)}
    if kind == "phase_space":
        return {"bytes": N * (32.0 * (n + 2) + 29.0), "flops": N * _gen_flops(n)}
    if kind == "hist":
        # only the events with a weight need their observables
        return {"bytes": 8.0 * N + 16.0 * sum(q[1] + 2 for q in HIST_SPECS),
                "flops": N * _PASS[n] * (_gen_flops(n) + 25.0 * n + 10.0 * n * (n - 1))}
    parts = [_xsec_work(q["n"], q["N"]) for q in _batch_requests(case, 0)]
    return {"bytes": sum(p["bytes"] for p in parts), "flops": sum(p["flops"] for p in parts)}


# ---------------------------------------------------------------------------------------------------------------------
# the same quantities in plain torch, 64 bits
# ---------------------------------------------------------------------------------------------------------------------

def _philox(c0, c1, c2, c3, seed):
    """Philox4x32-10 on int64 tensors (or ints) holding 32-bit words."""
    k0, k1 = seed & 0xFFFFFFFF, seed >> 32

    def mul(a, m):
        low = (a & 0xFFFF) * m
        high = (a >> 16) * m + (low >> 16)
        return high >> 16, ((high << 16) | (low & 0xFFFF)) & 0xFFFFFFFF
    for _ in range(10):
        h0, l0 = mul(c0, 0xD2511F53)
        h1, l1 = mul(c2, 0xCD9E8D57)
        c0, c1, c2, c3 = h1 ^ c1 ^ k0, l1, h0 ^ c3 ^ k1, l0
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return c0, c1, c2, c3


def _uniform(lo, hi):
    m = (hi << 20) | (lo >> 12)
    return (2 * m + 1).double() * 2.0 ** -53   # (2 m + 1) has 53 bits: exact


def _draws(i, block, tag, seed):
    """Draws 2 block and 2 block + 1 of stream `tag` of the points i."""
    z = torch.zeros_like(i)
    w = _philox(i & 0xFFFFFFFF, i >> 32, z + block, z + tag, seed)
    return _uniform(w[0], w[1]), _uniform(w[2], w[3])


def _toy(i, seed):
    """(x1, x2, attempts) of the toy PDF x^-1/2 (1-x)^3 with sqrt(x1 x2) 14 TeV > 100 GeV, by rejection."""
    N = i.numel()
    x = torch.zeros(2, N, dtype=torch.float64, device=i.device)
    tries = torch.ones(N, dtype=torch.int64, device=i.device)
    blk = torch.zeros(N, dtype=torch.int64, device=i.device)
    at = torch.zeros(N, dtype=torch.int64, device=i.device)    # which of the two fractions is being drawn
    live = torch.arange(N, device=i.device)
    while live.numel():
        u, v = _draws(i[live], blk[live], 0, seed)
        blk[live] += 1
        om = 1.0 - u * u
        hit = v < om * om * om
        won, u = live[hit], u[hit]
        which = at[won]
        x[which, won] = u * u
        at[won] = which + 1
        both = won[which == 1]
        low = ~(14000.0 * torch.sqrt(x[0, both] * x[1, both]) > 100.0)
        tries[both[low]] += 1
        at[both[low]] = 0
        live = live[at[live] < 2]
    return x[0], x[1], tries


def _rambo(r, rs):
    """n massless momenta [N, n, 4] of total (rs, 0, 0, 0) from uniforms r [4, N, n]."""
    c, phi = 2.0 * r[0] - 1.0, 2.0 * math.pi * r[1]
    q0 = -torch.log(r[2] * r[3])
    s = torch.sqrt(1.0 - c * c)
    q = torch.stack([q0, q0 * s * torch.cos(phi), q0 * s * torch.sin(phi), q0 * c], -1)
    Q = q.sum(1)
    M = torch.sqrt(Q[:, 0] ** 2 - (Q[:, 1:] ** 2).sum(-1))
    b = -Q[:, 1:] / M[:, None]
    gamma, a, x = Q[:, 0] / M, M / (M + Q[:, 0]), rs / M
    bq = (b[:, None] * q[..., 1:]).sum(-1)
    e = x[:, None] * (gamma[:, None] * q[..., 0] + bq)
    v = x[:, None, None] * (q[..., 1:] + b[:, None] * (q[..., 0] + a[:, None] * bq)[..., None])
    return torch.cat([e[..., None], v], -1)


def _pass(k, y):
    """Cuts on photons k [N, n, 4] with boost rapidity y, strict."""
    n = k.shape[1]
    pt = torch.sqrt(k[..., 1] ** 2 + k[..., 2] ** 2)
    eta, phi = torch.asinh(k[..., 3] / pt) + y[:, None], torch.atan2(k[..., 2], k[..., 1])
    ok = ((pt > PT_MIN) & (eta.abs() < ETA_MAX)).all(1)
    dr = []
    for i in range(n):
        for j in range(i + 1, n):
            d = (phi[:, i] - phi[:, j]).abs()
            d = torch.where(d > math.pi, 2 * math.pi - d, d)
            dr.append(torch.sqrt((eta[:, i] - eta[:, j]) ** 2 + d * d))
            ok &= dr[-1] > DR_MIN
    return ok, pt, eta, torch.stack(dr, 1)


def _generate(n, i, sampler, seed):
    """Events i of a stream: sqrt(s-hat), y, attempts, photons [N, n, 4]."""
    one = torch.ones(i.numel(), dtype=torch.float64, device=i.device)
    y, tries = torch.zeros_like(one), torch.ones_like(i)
    if sampler == "fixed":
        rs = 500.0 * one
    elif sampler == "uniform":
        rs = 200.0 + 1800.0 * _draws(i, 0, 0, seed)[0]
    else:
        x1, x2, tries = _toy(i, seed)
        rs, y = 14000.0 * torch.sqrt(x1 * x2), 0.5 * torch.log(x1 / x2)
    r = [sum((list(_draws(i, 2 * a + h, 1, seed)) for h in (0, 1)), []) for a in range(n)]
    return rs, y, tries, _rambo(torch.stack([torch.stack([ra[d] for ra in r], 1) for d in range(4)]), rs)


def _helicity_sum(k, E1, E2, wh, chunk=1 << 22):
    """sum_h wh[h] |A_h|^2 of events with photons k [N, n, 4], in units of sqrt(s-hat), over the photon helicities h for
    a right-handed quark along +z (energy E1) and its antiquark along -z (E2): the ordering sum built up over photon sets,
    massless chiral chain in two components."""
    N, n = k.shape[:2]
    rows = max(1, chunk // 3 ** n)
    if N > rows:
        return torch.cat([_helicity_sum(k[a:a + rows], E1[a:a + rows], E2[a:a + rows], wh, chunk) for a in range(0, N, rows)])
    p = k[..., 1:].norm(dim=-1)
    c = k[..., 3] / p
    pt = torch.sqrt(k[..., 1] ** 2 + k[..., 2] ** 2)
    s, ephi = pt / p, torch.complex(k[..., 1] / pt, k[..., 2] / pt)
    E = []   # E[i][lambda]: eps*(k_i, lambda) . sigma as a 2x2 matrix [N, 2, 2]
    for i in range(n):
        E.append([])
        for lam in (-1.0, 1.0):
            e00 = torch.complex(-lam * s[:, i], torch.zeros_like(s[:, i]))
            e01, e10 = -(1 - lam * c[:, i]) * ephi[:, i].conj(), (1 + lam * c[:, i]) * ephi[:, i]
            E[i].append(torch.stack([torch.stack([e00, e01], -1), torch.stack([e10, -e00], -1)], -2) / math.sqrt(2.0))
    cur = {0: torch.zeros(N, 1, 2, dtype=torch.complex128, device=k.device)}
    cur[0][:, 0, 1] = torch.sqrt(2.0 * E2)        # vbar: only its second entry
    full = (1 << n) - 1
    for size in range(1, n + 1):
        new = {}
        for S in range(1, full + 1):
            ph = [i for i in range(n) if S >> i & 1]
            if len(ph) != size:
                continue
            J = torch.zeros([N] + [2] * size + [2], dtype=torch.complex128, device=k.device)
            for pos, i in enumerate(ph):
                prev = cur[S & ~(1 << i)].reshape([N] + [2] * (size - 1) + [2])
                for lam in (0, 1):
                    r = (prev.reshape(N, -1, 2) @ E[i][lam]).reshape(prev.shape)
                    J.select(1 + pos, lam).add_(r)
            J = J.reshape(N, -1, 2)
            if S != full:
                q = k[:, ph].sum(1)
                q0, q3 = q[:, 0] - E2, q[:, 3] + E2
                t = q0 * q0 - q[:, 1] ** 2 - q[:, 2] ** 2 - q3 * q3
                A, D, B = (q0 + q3) / t, (q0 - q3) / t, torch.complex(q[:, 1] / t, q[:, 2] / t)
                J = torch.stack([J[..., 0] * A[:, None] + J[..., 1] * B[:, None],
                                 J[..., 0] * B.conj()[:, None] + J[..., 1] * D[:, None]], -1)
            new[S] = J
        cur = new
    amp = cur[full][..., 0] * torch.sqrt(2.0 * E1)[:, None]       # u(p1): only its first entry
    # axes: photon 0's helicity varies slowest; wh is indexed by bits with photon 0 lowest
    order = [sum(((h >> (n - 1 - i)) & 1) << i for i in range(n)) for h in range(1 << n)]
    return (amp.abs() ** 2 * wh[torch.tensor(order, device=k.device)]).sum(1)


def _coupling(n):
    return (4 * math.pi * ALPHA * QU * QU) ** n


def _volume(n):
    return (2 * math.pi) ** (4 - 3 * n) * (math.pi / 2) ** (n - 1) / (math.factorial(n - 1) * math.factorial(n - 2))


def _exact_events(n, N, sampler, seed, i0=0):
    """Generated events, their cuts and their weights in fb."""
    i = torch.arange(i0, i0 + N, dtype=torch.int64, device="cuda")
    rs, y, tries, k = _generate(n, i, sampler, seed)
    ok, pt, eta, dr = _pass(k, y)
    kk, half = k[ok] / rs[ok][:, None, None], torch.full((int(ok.sum()),), 0.5, dtype=torch.float64, device="cuda")
    S = _helicity_sum(kk, half, half, torch.full((1 << n,), 2.0, dtype=torch.float64, device="cuda"))
    w = torch.zeros(N, dtype=torch.float64, device="cuda")
    w[ok] = _coupling(n) * _volume(n) / (24 * math.factorial(n)) * 0.3893793721e12 * S / rs[ok] ** 2
    return {"w": w, "ok": ok, "tries": tries, "rs": rs, "pt": pt, "eta": eta, "dr": dr}


def _exact_result(n, N, sampler, seed, i0=0):
    ev = _exact_events(n, N, sampler, seed, i0)
    w, tries = ev["w"], int(ev["tries"].sum())
    sw, sw2 = math.fsum(w.tolist()), math.fsum((w * w).tolist())
    mean, accept = sw / N, N / tries
    scale = 2.0 * accept if sampler == "toy" else 1.0
    err = scale * math.sqrt(max(0.0, (sw2 - sw * mean) / (N - 1)) / N) if N > 1 else 0.0
    return [scale * mean, err, sw, sw2, accept], [int(ev["ok"].sum()), N, tries, 0], w


def _fields(values, counts):
    return {"values": [torch.tensor(v, dtype=torch.float64) for v in values],
            "counts": torch.tensor(counts, dtype=torch.int64)}


def _events(case, seed):
    """Another generator's events [N, n + 2, 4] (GeV): flat phase space that passes the cuts, unequal beam fractions."""
    n, N = int(case["n"]), int(case["N"])
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    rows, have = [], 0
    while have < N:
        m = int(1.2 * (N - have) / _PASS[n]) + 64
        rs = 200.0 + 1800.0 * torch.rand(m, generator=g, device="cuda", dtype=torch.float64)
        r = torch.rand(4, m, n, generator=g, device="cuda", dtype=torch.float64).clamp_(min=1e-12, max=1 - 1e-12)
        k = _rambo(r, rs)
        ok, _, _, _ = _pass(k, torch.zeros_like(rs))
        p = torch.zeros(m, 2, 4, device="cuda", dtype=torch.float64)
        p[:, :, 0] = 0.5 * rs[:, None]
        p[:, 0, 3], p[:, 1, 3] = 0.5 * rs, -0.5 * rs
        rows.append(torch.cat([p, k], 1)[ok])
        have += rows[-1].shape[0]
    return torch.cat(rows)[:N].contiguous()


def _helicity_mask(n):
    """The combinations with lambda_1 = +1 (bit 2 of the index), as 32-bit words."""
    words = [0] * max(1, (1 << (n + 2)) // 32)
    for h in range(1 << (n + 2)):
        if h >> 2 & 1:
            words[h >> 5] |= 1 << (h & 31)
    return torch.tensor([w - (1 << 32) if w >> 31 else w for w in words], dtype=torch.int32, device="cuda")


def _exact_amp2(case, seed):
    n = int(case["n"])
    mom = _events(case, seed)
    # weight of photon helicities h of the right-handed quark: itself and its parity image
    wh = [2.0] * (1 << n)
    if case["mask"]:
        wh = [float(h & 1) + float(~h & 1) for h in range(1 << n)]
    s = 4.0 * mom[:, 0, 0] * mom[:, 1, 0]
    rs = torch.sqrt(s)
    S = _helicity_sum(mom[:, 2:] / rs[:, None, None], mom[:, 0, 0] / rs, mom[:, 1, 0] / rs,
                      torch.tensor(wh, dtype=torch.float64, device="cuda"))
    return _coupling(n) * s ** (2 - n) * S


def _exact_hist(case, seed):
    n, N = int(case["n"]), int(case["N"])
    ev = _exact_events(n, N, case["sampler"], _stream_seed(seed))
    x = {H.HEGET_OBS_PT_MAX: ev["pt"].amax(1, keepdim=True), H.HEGET_OBS_PT: ev["pt"], H.HEGET_OBS_ETA: ev["eta"],
         H.HEGET_OBS_DR: ev["dr"], H.HEGET_OBS_DR_MIN: ev["dr"].amin(1, keepdim=True)}
    out = []
    for obs, nbins, lo, hi in HIST_SPECS:
        v = x[obs][ev["ok"]]
        w = ev["w"][ev["ok"]][:, None].expand_as(v).reshape(-1)
        b = 1 + torch.floor((v - lo) * (nbins / (hi - lo)))
        b = b.clamp(0, nbins + 1).long().reshape(-1)
        h = torch.zeros(nbins + 2, 2, dtype=torch.float64, device="cuda")
        h[:, 0].index_add_(0, b, w)
        h[:, 1].index_add_(0, b, w * w)
        out += [h[:, 0], h[:, 1]]
    return out


def _exact_seconds(n, N):
    """Rough time of exact() for N generated events (the ordering sum over photon sets runs for those that pass)."""
    return 1.0 + N * (2e-7 * n + _PASS[n] * 3 ** n * 4e-9)


def exact(case, seed):
    kind, n, N = case["kind"], int(case["n"]), int(case["N"])
    sampler, stream = case["sampler"], _stream_seed(seed)
    if kind == "batch":
        if sum(_exact_seconds(q["n"], q["N"]) for q in _batch_requests(case, seed)) - 23.0 > 18.0:
            return None
        out = []
        for a in range(2, 9):
            each = [_exact_result(a, q["N"], sampler, q["seed"], q["i0"]) for q in _batch_requests(case, seed) if q["n"] == a]
            out.append(_fields(list(zip(*[e[0] for e in each])), [e[1] for e in each]))
        return out
    if _exact_seconds(n, N / _PASS[n] if kind == "amp2" else N) > 18.0:
        return None
    if kind == "amp2":
        return _exact_amp2(case, seed)
    if kind == "hist":
        return _exact_hist(case, seed)
    if kind == "phase_space":
        rs, y, tries, k = _generate(n, torch.arange(N, dtype=torch.int64, device="cuda"), sampler, stream)
        ok = _pass(k, y)[0]
        p = torch.zeros(N, 2, 4, device="cuda", dtype=torch.float64)
        p[:, :, 0] = 0.5 * rs[:, None]
        p[:, 0, 3], p[:, 1, 3] = 0.5 * rs, -0.5 * rs
        return {"momenta": torch.cat([p, k], 1), "weights": _volume(n) * (rs * rs) ** (n - 2), "sqrt_s": rs, "y": y,
                "mask": ok.to(torch.uint8), "tries": tries.to(torch.int32)}
    values, counts, w = _exact_result(n, N, sampler, stream)
    if kind == "xsec_sync":
        return {"values": values, "counts": counts}
    out = _fields(values, counts)
    if case["weights"]:
        out["weights"] = w
    return out
