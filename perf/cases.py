"""Timed cases of the connectivity update: what a program that uses this framework has it
do, through the public entry points of ``paper_2509_26193_gb300.relearn`` and
``differentiable``.

A structural-plasticity simulation alternates many electrical steps (spike or rate
delivery over the synapse store) with connectivity updates (deletion, partner search,
acceptance) on a spatial octree that is rebuilt when neurons move or a new network
starts. The layouts are the ones of ``workloads.py`` (uniform cube, Gaussian clusters,
layered slab, batch of uneven cubes), drawn here with torch on the GPU so that large
networks are made quickly; sizes, densities, sigma and theta follow that module, the
tests and ``bench.py``.
"""
import math

import torch

from paper_2509_26193_gb300 import differentiable as D
from paper_2509_26193_gb300 import relearn as R

ALL = 1 << 20  # retracting this many elements breaks every synapse of a neuron
MORTON_MAX = 1 << 20  # RELEARN_NOALLOC_MAX_NEURONS


def listed():
    return [
        # smallest call: one update of a small cube on a standing tree (the smallest
        # network of the batch workload); launches and latency count
        dict(name="cube_1k", kind="step", layout="cube", n=1000, theta=0.3, updates=1,
             rebuild=False, retract=False),
        # the exact O(n^2) draw (theta = 0) on the small parity network
        dict(name="cube_4k_exact", kind="step", layout="cube", n=4096, theta=0.0, updates=1,
             rebuild=False, retract=False),
        # an ordinary network of the tests' size, odd count: a new tree, then three plasticity
        # steps with partial retraction between them
        dict(name="clusters_50k", kind="step", layout="clusters", n=50021, theta=0.3, updates=3,
             rebuild=True, retract=True),
        # a finer criterion (theta 0.2) on a ragged medium network, standing tree
        dict(name="clusters_300k_fine", kind="step", layout="clusters", n=300007, theta=0.2,
             updates=2, rebuild=False, retract=True),
        # the benchmark's step: 2^20 clustered neurons, new tree, ten updates that fill the
        # network up, each followed by spike delivery, then a full deletion
        dict(name="clusters_1m", kind="step", layout="clusters", n=1 << 20, theta=0.3,
             updates=10, rebuild=True, retract=False),
        # the largest network: a 2^24 layered slab, new tree and one update
        dict(name="slab_16m", kind="step", layout="slab", n=1 << 24, theta=0.3, updates=1,
             rebuild=True, retract=False),
        # excitatory and inhibitory dendrite pools
        dict(name="typed_200k", kind="typed", layout="clusters", n=200003, theta=0.3, updates=1,
             rebuild=False, retract=False),
        # a parameter study: many independent uneven networks in one build and update,
        # each with its own sigma
        dict(name="batch_64", kind="batch", networks=64, n_max=250000, theta=0.3),
        # between two connectivity updates: spikes and firing rates over a formed network
        dict(name="deliver_1m", kind="deliver", n=1 << 20),
        # one training step of the differentiable form, benchmark size and a small odd one
        dict(name="length_256k", kind="length", n=1 << 18, theta=0.3),
        dict(name="length_5k", kind="length", n=5003, theta=0.3),
        # spatial order alone, for callers that own all memory
        dict(name="morton_700k", kind="morton", n=700001),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the ranges that the listed ones stand for."""
    kind = rng.choice(["step", "step", "step", "step", "typed", "batch", "deliver", "length",
                       "length", "morton"])
    if kind in ("step", "typed"):
        layout = rng.choice(["cube", "clusters", "clusters", "slab"])
        n = _log(rng, 1000, 2000000 if layout != "slab" else 4000000)
        theta = 0.0 if kind == "step" and n <= 8000 and rng.random() < 0.3 \
            else round(rng.uniform(0.2, 0.5), 3)
        return dict(kind=kind, layout=layout, n=n, theta=theta,
                    updates=rng.randint(1, 4) if kind == "step" else 1,
                    rebuild=rng.random() < 0.5,
                    retract=kind == "step" and rng.random() < 0.5)
    if kind == "batch":
        return dict(kind=kind, networks=rng.randint(2, 128), n_max=_log(rng, 4000, 250000),
                    theta=round(rng.uniform(0.2, 0.5), 3))
    if kind == "deliver":
        return dict(kind=kind, n=_log(rng, 20000, 2000000))
    if kind == "length":
        n = _log(rng, 2000, 300000)
        theta = 0.0 if n < 6000 and rng.random() < 0.3 else round(rng.uniform(0.25, 0.5), 3)
        return dict(kind=kind, n=n, theta=theta)
    return dict(kind=kind, n=_log(rng, 1000, MORTON_MAX))



# ------------------------------------------------------------------------- inputs
def _gen(seed, stream=0):
    return torch.Generator(device="cuda").manual_seed(1000003 * int(seed) + stream)


def _rand(g, *shape):
    return torch.rand(*shape, generator=g, device="cuda", dtype=torch.float64)


def _poisson(g, lam, n, hi=8):
    rate = torch.full((n,), float(lam), device="cuda")
    return torch.poisson(rate, generator=g).clamp_(max=hi).to(torch.int32)


def _positions(layout, n, g):
    """Float32 coordinates and the layout's sigma, in micrometres (see workloads.py)."""
    if layout == "cube":  # 4096 neurons per cubic millimetre
        p = _rand(g, 3, n) * (1000.0 * (n / 4096.0) ** (1.0 / 3.0))
        sigma = 750.0
    elif layout == "clusters":  # 2^14 neurons per Gaussian cluster (std 300), 64 in 10 mm
        k = max(4, round(n / 16384))
        centres = _rand(g, 3, k) * (10000.0 * (k / 64.0) ** (1.0 / 3.0))
        owner = torch.arange(n, device="cuda") % k
        noise = torch.randn(3, n, generator=g, device="cuda", dtype=torch.float64)
        p = centres[:, owner] + 300.0 * noise
        sigma = 750.0
    else:  # slab: ten layers of uneven shares, 20 x 20 x 2.5 mm at 2^24 neurons
        edge = 20000.0 * (n / float(1 << 24)) ** 0.5
        share = 1.0 + 0.6 * (_rand(g, 10) - 0.5)
        layer = torch.searchsorted(torch.cumsum(share / share.sum(), 0), _rand(g, n)).clamp_(max=9)
        p = _rand(g, 3, n)
        p[0] *= edge
        p[1] *= edge
        p[2] = (layer + p[2]) * 250.0
        sigma = 1000.0
    p = p.to(torch.float32)
    return p[0].clone(), p[1].clone(), p[2].clone(), sigma


def _vacancies(layout, n, g):
    if layout == "cube" and n <= 4096:
        return torch.randint(0, 5, (n,), generator=g, device="cuda", dtype=torch.int32)
    return _poisson(g, 1.0 if layout == "slab" else 2.0, n)


def _types(n, g):
    return (_rand(g, n) < 0.2).to(torch.uint8)


def _batch_sizes(case):
    """Network sizes, log-uniform in [1000, n_max] (the study's, the same for every seed),
    and their offsets (host)."""
    g = torch.Generator().manual_seed(7919 * case["networks"] + case["n_max"])
    u = torch.rand(case["networks"], generator=g, dtype=torch.float64)
    lo, hi = math.log(1000.0), math.log(float(case["n_max"]))
    sizes = torch.exp(lo + (hi - lo) * u).round().to(torch.int64)
    off = torch.cat([torch.zeros(1, dtype=torch.int64), torch.cumsum(sizes, 0)])
    return sizes, off.numpy()


class _State:
    pass


def prepare(case, seed):
    s = _State()
    s.case, s.seed = case, int(seed)
    g = _gen(seed)
    kind = case["kind"]
    if kind == "morton":
        n = case["n"]
        s.x, s.y, s.z, _ = _positions("clusters", n, g)
        s.codes = torch.empty(n, dtype=torch.int32, device="cuda")
        s.perm = torch.empty(n, dtype=torch.int32, device="cuda")
        return s
    if kind == "length":
        n = case["n"]
        side = 4000.0 * (n / float(1 << 18)) ** (1.0 / 3.0)  # differentiable_cube's density
        p = (_rand(g, 3, n) * side).to(torch.float32)
        s.x, s.y, s.z = (p[k].clone().requires_grad_(True) for k in range(3))
        s.sigma = torch.tensor([800.0], device="cuda", requires_grad=True)
        s.ax, s.de = _poisson(g, 2.0, n), _poisson(g, 2.0, n)
        s.ctx = R.relearn_create(n, 64)
        return s
    if kind == "batch":
        sizes, s.offsets = _batch_sizes(case)
        n = int(s.offsets[-1])
        sz = sizes.cuda()
        owner = torch.repeat_interleave(torch.arange(len(sizes), device="cuda"), sz)
        side = (sz.to(torch.float64) / 4096.0) ** (1.0 / 3.0) * 1000.0
        p = (_rand(g, 3, n) * side[owner]).to(torch.float32)
        s.x, s.y, s.z = p[0].clone(), p[1].clone(), p[2].clone()
        s.net_sigma = (500.0 + 500.0 * _rand(g, len(sizes))).to(torch.float32)
        s.ax0, s.de0 = _poisson(g, 2.0, n), _poisson(g, 2.0, n)
        s.type = _types(n, g)
    else:
        n = case["n"]
        layout = case.get("layout", "clusters")
        s.x, s.y, s.z, s.sigma = _positions(layout, n, g)
        s.ax0, s.de0 = _vacancies(layout, n, g), _vacancies(layout, n, g)
        s.type = _types(n, g)
    q = int(s.ax0.sum())
    s.ax, s.de = s.ax0.clone(), s.de0.clone()
    s.input = torch.zeros(n, dtype=torch.int32, device="cuda")
    s.all = torch.full((n,), ALL, dtype=torch.int32, device="cuda")
    if kind == "batch":
        s.ctx = R.relearn_create_batched(n, q + 1024, case["networks"], q + 1024)
        return s
    # retracted bound elements become vacant at the partner, so a later update can search
    # for at most twice the first one's elements
    s.ctx = R.relearn_create(n, 2 * q + 1024, 2 * q + 1024)
    R.relearn_build_octree(s.ctx, s.x, s.y, s.z)
    if kind == "deliver":
        prm = R.params(s.sigma, 0.3, s.seed, 0)
        R.relearn_update_connectivity(s.ctx, prm, s.ax, s.de, s.type)
        s.spiked = (_rand(g, n) < 0.05).to(torch.uint8)
        s.rate = (0.1 * _rand(g, n)).to(torch.float32)
        s.input2 = torch.zeros(n, dtype=torch.int32, device="cuda")
        return s
    if kind == "typed":
        s.di0 = _vacancies(layout, n, g)
        s.di = s.di0.clone()
    s.spiked = (_rand(g, case["updates"], n) < 0.05).to(torch.uint8)
    s.ra, s.rd = _poisson(g, 0.5, n), _poisson(g, 0.5, n)
    return s


# ---------------------------------------------------------------------------- run
def _run_step(s):
    c = s.case
    s.ax.copy_(s.ax0)  # the element model's vacancies
    s.de.copy_(s.de0)
    if c["rebuild"]:
        R.relearn_build_octree(s.ctx, s.x, s.y, s.z)
    for u in range(c["updates"]):
        prm = R.params(s.sigma, c["theta"], s.seed, u)
        R.relearn_update_connectivity(s.ctx, prm, s.ax, s.de, s.type)
        R.relearn_deliver_spikes(s.ctx, s.spiked[u], s.input)
        if c["retract"] and u + 1 < c["updates"]:
            prm = R.params(s.sigma, c["theta"], s.seed, 1000 + u)
            R.relearn_delete_synapses(s.ctx, prm, s.ra, s.rd, s.ax, s.de)
    out = [s.ax.clone(), s.de.clone(), s.input.clone()]
    # the network returns to empty
    R.relearn_delete_synapses(s.ctx, R.params(s.sigma, c["theta"], s.seed, 9999), s.all, s.all,
                              s.ax, s.de)
    return out + [s.ax, s.de]


def _run_typed(s):
    c = s.case
    s.ax.copy_(s.ax0)
    s.de.copy_(s.de0)
    s.di.copy_(s.di0)
    if c["rebuild"]:
        R.relearn_build_octree(s.ctx, s.x, s.y, s.z)
    prm = R.params(s.sigma, c["theta"], s.seed, 0)
    R.relearn_update_connectivity_typed(s.ctx, prm, s.ax, s.de, s.di, s.type)
    R.relearn_deliver_spikes(s.ctx, s.spiked[0], s.input)
    out = [s.ax.clone(), s.de.clone(), s.di, s.input]
    R.relearn_delete_synapses(s.ctx, R.params(s.sigma, c["theta"], s.seed, 9999), s.all, s.all,
                              s.ax, s.de)
    return out + [s.ax, s.de]


def _run_batch(s):
    c = s.case
    s.ax.copy_(s.ax0)
    s.de.copy_(s.de0)
    R.relearn_build_octree_batch(s.ctx, s.offsets, s.x, s.y, s.z)
    prm = R.params(0.0, c["theta"], s.seed, 1, net_sigma=s.net_sigma)
    R.relearn_update_connectivity(s.ctx, prm, s.ax, s.de, s.type)
    R.relearn_deliver_spikes(s.ctx, s.type, s.input)  # inhibitory neurons fire
    out = [s.ax.clone(), s.de.clone(), s.input]
    prm = R.params(0.0, c["theta"], s.seed, 999, net_sigma=s.net_sigma)
    R.relearn_delete_synapses(s.ctx, prm, s.all, s.all, s.ax, s.de)
    return out + [s.ax, s.de]


def run(s):
    kind = s.case["kind"]
    if kind == "step":
        return _run_step(s)
    if kind == "typed":
        return _run_typed(s)
    if kind == "batch":
        return _run_batch(s)
    if kind == "deliver":
        R.relearn_deliver_spikes(s.ctx, s.spiked, s.input)
        R.relearn_deliver_rates(s.ctx, s.rate, s.seed, 7, s.input2)
        return [s.input, s.input2]
    if kind == "length":
        for t in (s.x, s.y, s.z, s.sigma):
            t.grad = None
        mean = D.mean_synapse_length(s.ctx, s.x, s.y, s.z, s.sigma, s.ax, s.de,
                                     s.case["theta"])
        mean.backward()
        return [mean.detach(), s.x.grad, s.y.grad, s.z.grad, s.sigma.grad]
    R.relearn_morton_order_noalloc(s.x, s.y, s.z, s.codes, s.perm)
    return [s.codes, s.perm]


# --------------------------------------------------------------------------- work
# Share of the neurons with a vacant axonal element, and the number of sources of the
# updates that follow as a share of the first one's (the network fills up; the clustered
# benchmark: 907k, 425k, 162k, 62k, 24k, ... sources).
_ACTIVE = {"cube": 0.86, "clusters": 0.865, "slab": 0.63}
_LATER = (1.0, 0.47, 0.18, 0.07, 0.027, 0.012, 0.006, 0.004, 0.003, 0.002)


def _candidates(layout, n, theta):
    """Candidates of one source's root frontier: about 2,440 in the 2^18 cube at theta 0.3
    (measured by the library's counters), growing as theta^-2 and with the number of
    shells, 1.2 times that in the clusters, five times in the wide flat slab."""
    if theta == 0.0:
        return n
    f = 2440.0 * (0.3 / theta) ** 2 * {"cube": 1.0, "clusters": 1.2, "slab": 5.0}[layout]
    return min(float(n), f * min(1.6, max(0.3, math.log(n / 500.0) / math.log(524.0))))


def work(case):
    """Inputs read once, outputs written once; 15 flop per root-frontier candidate of every
    source of a search (distance, criterion, exponent, count, running sum), 52 in the
    differentiable form's two passes."""
    kind = case["kind"]
    if kind == "morton":
        return {"bytes": 20.0 * case["n"], "flops": 12.0 * case["n"]}
    if kind == "deliver":
        n = case["n"]
        syn = 1.7 * n
        # spikes: sources, and the targets and signs of the 5 % that fire; rates: all of it
        return {"bytes": syn * (4 + 0.05 * 5 + 9) + n * (1 + 4 + 4 + 4), "flops": 2.0 * syn}
    if kind == "length":
        n = case["n"]
        f = _candidates("cube", n, case["theta"])
        return {"bytes": n * (12 + 8 + 12), "flops": 52.0 * f * 0.86 * n}
    if kind == "batch":
        n = float(_batch_sizes(case)[1][-1])
        f = _candidates("cube", n / case["networks"], case["theta"])
        return {"bytes": n * (12 + 8 + 1 + 8 + 4 + 8) + 1.7 * n * 9,
                "flops": 15.0 * f * 0.86 * n}
    n, lay = case["n"], case["layout"]
    f = _candidates(lay, n, case["theta"])
    later = sum(_LATER[:case["updates"]])
    if case["retract"]:  # retraction and its returned vacancies keep more sources active
        later += 0.4 * (case["updates"] - 1)
    vac = 1.0 if lay == "slab" else 2.0
    per_update = n * (8 + 8 + 1 + 1 + 4)
    return {"bytes": case["updates"] * per_update + n * (12 if case["rebuild"] else 0)
            + 0.85 * vac * n * 9 * 2 + n * 24,
            "flops": 15.0 * f * _ACTIVE[lay] * n * later}


# -------------------------------------------------------------------------- exact
def exact(case, seed):
    """The differentiable form in 64 bits; every other path returns integers."""
    if case["kind"] != "length":
        return None
    s = prepare(case, seed)
    pos = torch.stack([s.x, s.y, s.z]).detach()
    return _mean_length64(pos, s.ax, s.de, 800.0, case["theta"])


def _spread(v):
    out = torch.zeros_like(v)
    for b in range(10):
        out |= ((v >> b) & 1) << (3 * b)
    return out


def _mean_length64(pos, vac_ax, vac_de, sigma, theta):
    """Mean expected synapse length over every source's root frontier and its gradient,
    plain torch in float64. The octree cells are the ten-bit Morton cells (their FP32
    quantisation is part of the method's definition); a cell is accepted when its length
    is less than theta times the distance to its count-weighted centroid, a cell of one
    neuron and the neurons of a depth-10 cell always; the criterion is constant in the
    gradient. A source's own neuron is no candidate."""
    dev = pos.device
    n = pos.shape[1]
    lo, hi = pos.amin(1), pos.amax(1)
    inv = torch.where(hi > lo, 1.0 / (hi - lo), torch.zeros_like(lo))
    q = (((pos - lo[:, None]) * inv[:, None]) * 1024.0).clamp(0.0, 1023.0).to(torch.int64)
    code = _spread(q[0]) | (_spread(q[1]) << 1) | (_spread(q[2]) << 2)
    code, order = torch.sort(code, stable=True)
    x = pos[:, order].to(torch.float64).t().contiguous()  # [n, 3], Morton order
    w = vac_de[order].to(torch.float64)
    m = vac_ax[order].to(torch.float64)
    ext = float((hi.to(torch.float64) - lo.to(torch.float64)).max())
    # levels 0 .. 10: cells; level 11: the single neurons
    cells = []
    for d in range(12):
        if d <= 10:
            key, cell, size = torch.unique_consecutive(code >> (3 * (10 - d)), return_inverse=True,
                                                       return_counts=True)
        else:
            cell, size = torch.arange(n, device=dev), torch.ones(n, dtype=torch.int64, device=dev)
        first = torch.cumsum(size, 0) - size
        k = size.numel()
        cnt = torch.zeros(k, dtype=torch.float64, device=dev).index_add_(0, cell, w)
        cen = torch.zeros(k, 3, dtype=torch.float64, device=dev).index_add_(
            0, cell, x * w[:, None]) / cnt.clamp(min=1.0)[:, None]
        cells.append((cell, size, first, cnt, cen))
    kids = []  # per level: first child cell and number of children in the next level
    for d in range(11):
        first = cells[d][2]
        c0 = cells[d + 1][0][first]
        nxt = torch.cat([c0[1:], torch.tensor([cells[d + 1][1].numel()], device=dev)])
        kids.append((c0, nxt - c0))
    src = torch.nonzero(m > 0).flatten()
    k2 = 1.0 / (sigma * sigma)
    G = [torch.zeros(c[1].numel(), 3, dtype=torch.float64, device=dev) for c in cells]
    gdir = torch.zeros(n, 3, dtype=torch.float64, device=dev)
    sum_ml = torch.zeros((), dtype=torch.float64, device=dev)
    sum_m = torch.zeros((), dtype=torch.float64, device=dev)
    gsig = torch.zeros((), dtype=torch.float64, device=dev)
    chunk = max(1, min(4096, (1 << 25) // max(1, n) if theta == 0.0 else 4096))
    for a in range(0, src.numel(), chunk):
        ids = src[a:a + chunk]
        B = ids.numel()
        row = torch.arange(B, device=dev)
        node = torch.zeros(B, dtype=torch.int64, device=dev)  # the root is expanded
        taken = []
        for d in range(11):
            c0, nk = kids[d]
            rep = nk[node]
            row = torch.repeat_interleave(row, rep)
            start = torch.cumsum(rep, 0) - rep
            node = torch.repeat_interleave(c0[node] - start, rep) + torch.arange(
                row.numel(), device=dev)
            cell, size, first, cnt, cen = cells[d + 1]
            keep = cnt[node] > 0
            row, node = row[keep], node[keep]
            r = x[ids[row]] - cen[node]
            D2 = (r * r).sum(1)
            length = ext / float(1 << (d + 1)) if d < 10 else 0.0
            single = size[node] == 1
            acc = single | (length * length < theta * theta * D2)
            own = single & (first[node] == ids[row])
            t = acc & ~own
            taken.append((d + 1, row[t], node[t], r[t], D2[t]))
            row, node = row[~acc], node[~acc]
        S = torch.zeros(B, dtype=torch.float64, device=dev)
        A = torch.zeros_like(S)
        Dq = torch.zeros_like(S)
        att = []
        for d, ro, no, r, D2 in taken:
            e = cells[d][3][no] * torch.exp(-D2 * k2)
            att.append(e)
            S.index_add_(0, ro, e)
            A.index_add_(0, ro, e * D2.sqrt())
            Dq.index_add_(0, ro, e * D2)
        ok = S > 0
        inv_s = torch.where(ok, 1.0 / S.clamp(min=1e-300), torch.zeros_like(S))
        ell, dbar = A * inv_s, Dq * inv_s
        ms = torch.where(ok, m[ids], torch.zeros_like(S))
        sum_ml += (ms * ell).sum()
        sum_m += ms.sum()
        for (d, ro, no, r, D2), e in zip(taken, att):
            qk = e * inv_s[ro]
            dist = D2.sqrt()
            dl = dist - ell[ro]
            gsig += (ms[ro] * qk * dl * (D2 - dbar[ro])).sum()
            inv_d = torch.where(dist > 0, 1.0 / dist.clamp(min=1e-300), torch.zeros_like(dist))
            g = (ms[ro] * qk * (2.0 * k2 * dl - inv_d))[:, None] * r
            G[d].index_add_(0, no, g)
            gdir.index_add_(0, ids[ro], -g)
    for d in range(1, 12):
        cell, size, first, cnt, cen = cells[d]
        gdir += w[:, None] * (G[d] / cnt.clamp(min=1.0)[:, None])[cell]
    g = torch.empty_like(gdir)
    g[order] = gdir / sum_m
    mean = sum_ml / sum_m
    gs = gsig * (2.0 / (sigma ** 3)) / sum_m
    return [mean, g[:, 0].contiguous(), g[:, 1].contiguous(), g[:, 2].contiguous(), gs.reshape(1)]
