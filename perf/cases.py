"""Performance cases of the framework: whole calls as a user's program makes them.

A case names an entry point ("step": set_Y, step, get_Y and the velocity;
"grad": set_Y, grad; "kl": the differentiable KL, forward and backward), the
problem size and the options of the context.  Sizes are those of
`inputs.WORKLOADS`, of the tests and of `bench.py`.

Inputs: the affinities have the shape of the symmetrised kNN graphs of
`inputs.affinities_csr` (k = 90, or 3 x perplexity, one-sided neighbours per
point, ~135 entries per row of uneven length, columns scattered over the whole
index range, values falling off with a perplexity of about k / 3), made on the
device from the seed: the points of a hidden ring, grouped by cluster, are
joined to the next k positions on either side at random.  Embeddings are Y0 ~
N(0, 1e-4 I) (rho = 0) or clusters spread over the disk up to hyperbolic radius
rho, as in `inputs.spread_embedding`.
"""
import math

import numpy as np
import torch

from paper_2401_13708_gb300 import HyperbolicTSNE
from paper_2401_13708_gb300.autograd import kl_divergence

LEVELS = 29  # tree depth of the method's polar quadtree keys


def _case(name, **kw):
    c = {"name": name, "entry": "step", "n": 2000, "k": 90, "clusters": 10, "rho": 0.0, "precision": "fp32",
         "theta": 0.5, "iters": 1, "exaggeration": 1.0, "momentum": 0.8, "segments": 1, "graphs": False,
         "host": False, "split_rule": "equal_length", "grad_form": "exact", "metric_pow": 1, "use_gains": False}
    c.update(kw)
    return c


def listed():
    return [
        # the exact float64 gradient of a small embedding: checking a run, or an optimiser of the user's own
        _case("grad_exact_f64_2000", entry="grad", precision="fp64", theta=0.0, rho=6.0),
        # the README's program on the small mixture: numpy in and out, ten iterations at a time between two looks
        _case("step_f32_2000", iters=10, exaggeration=12.0, momentum=0.5, graphs=True, host=True),
        # the same in float64
        _case("step_f64_2000", iters=10, precision="fp64", exaggeration=12.0, momentum=0.5),
        # KL as a loss in a torch program, at its default theta = 0: forward and backward, a ragged size
        _case("kl_exact_f32_8191", entry="kl", n=8191, theta=0.0, rho=6.0),
        # one Barnes-Hut gradient for an optimiser of the user's own, a ragged size
        _case("grad_f32_20011", entry="grad", n=20011, clusters=20, rho=6.0),
        # the MNIST-shaped embedding, early exaggeration, five iterations between two looks
        _case("step_f32_70000", n=70000, iters=5, exaggeration=12.0, momentum=0.5),
        # one iteration of it in float64, later on
        _case("step_f64_70000", n=70000, precision="fp64", rho=6.0),
        # the hierarchical data at the most accurate theta in use, spread over the disk
        _case("step_f32_131071_fine", n=131071, clusters=64, theta=0.2, rho=8.0),
        # the same with equal-area cells at the default theta, all optimiser options on
        _case("step_f32_131071_area", n=131071, clusters=64, rho=8.0, split_rule="equal_area", use_gains=True),
        # 64 embeddings of 500 to 20,000 points in one context, replayed as graphs
        _case("step_f32_batch64", n=376430, segments=64, iters=2, exaggeration=12.0, momentum=0.5, graphs=True),
        # the single-cell-sized embedding at its start
        _case("step_f32_1m_start", n=1000000, clusters=200, exaggeration=12.0, momentum=0.5),
        # and later on, spread over the disk up to the rim
        _case("step_f32_1m_spread", n=1000000, clusters=200, rho=12.0),
    ]


def draw(rng):
    c = _case("")
    del c["name"]
    kind = rng.choice(["step", "step", "step", "grad", "kl"])
    f64 = rng.random() < 0.3
    theta = rng.choice([0.0, 0.2, 0.3, 0.5, 0.5, 0.5, 0.8, 1.0])
    top = 1000000 if theta >= 0.5 else 200000
    if f64:
        top = 50000 if theta >= 0.5 else 6000
    if theta == 0.0:
        top = 4000 if f64 else 16000
    c.update(entry=kind, precision="fp64" if f64 else "fp32", theta=theta)
    c["split_rule"] = rng.choice(["equal_length"] * 4 + ["equal_area"])
    if c["split_rule"] == "equal_area":  # (its walks are several times longer)
        top = min(top, 3000 if f64 else 40000 if theta >= 0.5 else 8000)
    n = int(round(math.exp(rng.uniform(math.log(500), math.log(top)))))
    c["n"] = n
    c["k"] = rng.choice([30, 90, 90, 150])
    c["clusters"] = 10 if n < 20000 else rng.choice([20, 64, 200])
    c["rho"] = rng.choice([0.0, 4.0, 6.0, 8.0, 10.0]) if theta != 0.0 or kind != "step" else 6.0
    c["grad_form"] = rng.choice(["exact"] * 4 + ["paper"])
    if kind == "step":
        c["iters"] = 1 if n > 100000 or f64 else rng.randint(1, 6)
        c["exaggeration"], c["momentum"] = rng.choice([(12.0, 0.5), (1.0, 0.8)])
        c["metric_pow"] = rng.choice([1, 1, 1, 2])
        c["use_gains"] = rng.random() < 0.25
        c["graphs"] = rng.random() < 0.5
        c["host"] = rng.random() < 0.2
        if n > 20000 and not f64 and theta >= 0.5 and rng.random() < 0.3:
            c["segments"] = rng.randint(2, max(2, min(64, n // 2000)))
    return c


# ---- inputs ------------------------------------------------------------------

def _offsets(case, seed):
    """Segment boundaries: log-uniform sizes between 1 and 40, scaled to n."""
    ns, n = case["segments"], case["n"]
    if ns == 1:
        return np.array([0, n], dtype=np.int64)
    rng = np.random.default_rng(seed + 17)
    w = np.exp(rng.uniform(0.0, math.log(40.0), size=ns))
    least = min(400, n // ns)
    s = least + np.floor(w / w.sum() * (n - least * ns)).astype(np.int64)
    s[-1] += n - s.sum()
    return np.concatenate([[0], np.cumsum(s)]).astype(np.int64)


def _inputs(case, seed):
    """Affinities (CSR) and embedding on the device."""
    dev = torch.device("cuda")
    gen = torch.Generator(device=dev).manual_seed(int(seed))
    n = case["n"]
    off = _offsets(case, seed)
    sizes = torch.as_tensor(np.diff(off), device=dev)
    seg = torch.repeat_interleave(torch.arange(len(sizes), device=dev), sizes)
    lo = torch.as_tensor(off[:-1], device=dev)[seg]
    size = sizes[seg]
    k = int(min(case["k"], (int(sizes.min()) - 1) // 3))

    # Zipf clusters; ring[q] = the point at ring position q (a segment's points stay in its range)
    w = 1.0 / torch.arange(1, case["clusters"] + 1, device=dev, dtype=torch.float64)
    label = torch.multinomial(w, n, replacement=True, generator=gen) if case["clusters"] > 1 else torch.zeros(
        n, dtype=torch.int64, device=dev)
    jitter = torch.rand(n, generator=gen, device=dev, dtype=torch.float64)
    ring = torch.argsort((seg * case["clusters"] + label).double() + jitter)

    # sign[q, t]: whether q took the position t + 1 after it, or the one before it
    value = torch.float64 if case["precision"] == "fp64" else torch.float32
    d = torch.cat([torch.arange(-k, 0, device=dev), torch.arange(1, k + 1, device=dev)])
    sign = torch.rand(n, k, generator=gen, device=dev) < 0.5
    weight = torch.exp(-torch.arange(1, k + 1, device=dev, dtype=torch.float64) * (3.0 * math.e / k))
    weight = (weight / weight.sum() / 2.0).float()
    rows, cols, vals = torch.empty(n, dtype=torch.int64, device=dev), [], []
    for a in range(0, n, 1 << 17):
        q = torch.arange(a, min(n, a + (1 << 17)), device=dev)
        j = lo[q, None] + (q[:, None] - lo[q, None] + d) % size[q, None]
        t = d.abs() - 1
        mine = torch.where(d > 0, sign[q][:, t], ~sign[q][:, t])
        theirs = torch.where(d > 0, ~sign[j, t], sign[j, t])
        amount = mine.float() + theirs.float()
        j = torch.where(amount > 0, ring[j], n)
        v = amount * weight[t] / size[q, None].float()
        j, order = torch.sort(j, dim=1)
        v = torch.gather(v, 1, order)
        rows[q] = (j < n).sum(1)
        cols.append(j.to(torch.int32))
        vals.append(v)
    cols, vals = torch.cat(cols), torch.cat(vals)
    back = torch.empty_like(ring)
    back[ring] = torch.arange(n, device=dev)
    indptr = torch.zeros(n + 1, dtype=torch.int64, device=dev)
    indptr[1:] = torch.cumsum(rows[back], 0)
    indices, values = [], []
    for a in range(0, n, 1 << 17):  # rows in point order
        b = back[a:a + (1 << 17)]
        c = cols[b]
        keep = c < n
        indices.append(c[keep])
        values.append(vals[b][keep].to(value))
    indices, values = torch.cat(indices), torch.cat(values)

    if case["rho"] == 0.0:
        y = torch.randn(n, 2, generator=gen, device=dev, dtype=torch.float64) * 1e-2
    else:
        m = case["segments"] * case["clusters"]
        at = seg * case["clusters"] + label
        rc = (1.0 + (case["rho"] - 1.0) * torch.rand(m, generator=gen, device=dev, dtype=torch.float64))[at]
        pc = (2.0 * math.pi * torch.rand(m, generator=gen, device=dev, dtype=torch.float64))[at]
        z = torch.randn(n, 2, generator=gen, device=dev, dtype=torch.float64)
        r = torch.tanh((rc + 0.6 * z[:, 0]).abs() / 2.0).clamp(max=1.0 - 1e-4)
        phi = pc + 0.6 * z[:, 1] / torch.sinh(rc.clamp(min=0.5))
        y = torch.stack([r * torch.cos(phi), r * torch.sin(phi)], 1)
    return off, indptr, indices, values, y.contiguous()


def prepare(case, seed):
    off, indptr, indices, values, y = _inputs(case, seed)
    model = HyperbolicTSNE(precision=case["precision"], split_rule=case["split_rule"], grad_form=case["grad_form"],
                           metric_pow=case["metric_pow"], use_gains=case["use_gains"])
    model.set_P(indptr, indices, values)
    model.set_Y(y)
    if case["segments"] > 1:  # the paper's lr = n / 12000 per embedding
        model.set_segments(off, np.diff(off) / 12000.0)
    if case["graphs"]:
        model.set_graphs(True)
    state = {"case": case, "model": model, "y": y, "lr": 1.0 if case["segments"] > 1 else case["n"] / 12000.0}
    if case["host"]:
        state["y"] = y.cpu().numpy()
        state["out"], state["vel"] = np.empty_like(state["y"]), np.empty_like(state["y"])
    else:
        state["out"], state["vel"] = torch.empty_like(y), torch.empty_like(y)
    return state


def run(state):
    c, model = state["case"], state["model"]
    if c["entry"] == "kl":
        y = state["y"] if not c["host"] else torch.from_numpy(state["y"])
        y = y.detach().requires_grad_()
        loss = kl_divergence(y, model, c["theta"])
        loss.backward()
        return {"loss": loss.detach(), "grad": y.grad}
    model.set_Y(state["y"])
    if c["entry"] == "grad":
        g, z = model.grad(c["theta"], c["exaggeration"], out=state["out"])
        return {"grad": g, "Z": z}
    model.step(c["iters"], c["theta"], c["exaggeration"], state["lr"], c["momentum"])
    y = model.get_Y(out=state["out"])
    vel, _, _ = model.get_state(vel=state["vel"], with_gains=False)
    return {"Y": y, "velocity": vel}


def work(case):
    """Operations: 28 per interaction of the repulsive sum and 35 per stored
    affinity; interactions per point: n - 1, or about 11 log2(n) / theta^2 for
    the tree (868 counted at n = 1,000,000 and theta = 0.5).  Bytes: the
    affinities and the embedding in, the results out."""
    n, theta = case["n"], case["theta"]
    nnz = n * case["k"] * 1.5
    per = n - 1 if theta == 0.0 else min(n - 1, 11.0 * math.log2(n / case["segments"]) / theta ** 2)
    value = 8 if case["precision"] == "fp64" else 4
    return {"bytes": nnz * (4 + value) + 8 * n + 16 * n * 3, "flops": case["iters"] * (28.0 * n * per + 35.0 * nnz)}


# ---- the same results in 64 bits ------------------------------------------------

def _pair(delta, paper):
    """w, w^2 d / sinh d and w d / sinh d of delta = cosh(d) - 1 (without the d in the paper's printed form)."""
    delta = delta.clamp(min=1e-300)
    t = torch.sqrt(delta * (delta + 2.0))
    d = torch.log1p(delta + t)
    w = 1.0 / (1.0 + d * d)
    f = 1.0 / t if paper else d / t
    return w, w * w * f, w * f


def _add_pairs(acc, y, il, i, yj, ilj, count, paper, which):
    """acc[i] += (k Delta, k s, count w) of the pairs (i, j), in slices."""
    for a in range(0, i.numel(), 1 << 25):
        s_ = slice(a, a + (1 << 25))
        p, q = i[s_], y[i[s_]]
        dl = q - yj[s_]
        s = dl[:, 0] * dl[:, 0] + dl[:, 1] * dl[:, 1]
        w, rep, att = _pair(2.0 * s * il[p] * ilj[s_], paper)
        m = count[s_] if torch.is_tensor(count) else count
        k = m * (rep if which == "rep" else att) * ilj[s_]
        acc.index_add_(0, p, torch.stack([k * dl[:, 0], k * dl[:, 1], k * s, m * w], 1))


def _force(acc, y, il):
    f = 4.0 * il[:, None] * (acc[:, :2] + (il * acc[:, 2])[:, None] * y)
    return f, acc[:, 3]


def _exact_repulsion(y, il, seg, paper):
    n = y.shape[0]
    out = torch.empty(n, 4, dtype=y.dtype, device=y.device)
    step = max(1, (1 << 25) // n)
    for a in range(0, n, step):
        b = min(n, a + step)
        dl = y[a:b, None, :] - y[None, :, :]
        s = dl[..., 0] ** 2 + dl[..., 1] ** 2
        w, rep, _ = _pair(2.0 * s * il[a:b, None] * il[None, :], paper)
        keep = (seg[a:b, None] == seg[None, :])
        keep[torch.arange(b - a), torch.arange(a, b)] = False
        w = torch.where(keep, w, 0.0)
        k = torch.where(keep, rep * il[None, :], 0.0)
        out[a:b] = torch.stack([(k * dl[..., 0]).sum(1), (k * dl[..., 1]).sum(1), (k * s).sum(1), w.sum(1)], 1)
    return out


def _spread(v):
    for s, m in ((16, 0x0000FFFF0000FFFF), (8, 0x00FF00FF00FF00FF), (4, 0x0F0F0F0F0F0F0F0F), (2, 0x3333333333333333),
                 (1, 0x5555555555555555)):
        v = (v | (v << s)) & m
    return v


def _squeeze(v):
    v = v & 0x5555555555555555
    for s, m in ((1, 0x3333333333333333), (2, 0x0F0F0F0F0F0F0F0F), (4, 0x00FF00FF00FF00FF), (8, 0x0000FFFF0000FFFF),
                 (16, 0x00000000FFFFFFFF)):
        v = (v | (v >> s)) & m
    return v


def _tree_repulsion(y, il, off, seg, theta, area, paper):
    """Barnes-Hut sums over the polar quadtree, level by level: the pairs
    (point, cell) not yet accepted go on to the cell's children."""
    dev, n, ns = y.device, y.shape[0], len(off) - 1
    n2 = y[:, 0] * y[:, 0] + y[:, 1] * y[:, 1]
    c = (1.0 + n2) / (1.0 - n2) if area else torch.sqrt(n2)
    lo = torch.stack([c[off[s]:off[s + 1]].min() for s in range(ns)])
    hi = torch.stack([c[off[s]:off[s + 1]].max() for s in range(ns)])
    span = hi - lo
    rh = torch.where(span[seg] > 0, (c - lo[seg]) / torch.where(span > 0, span, 1.0)[seg], 0.0)
    phi = torch.atan2(y[:, 1], y[:, 0])
    phi = torch.where(phi < 0, phi + 2.0 * math.pi, phi) / (2.0 * math.pi)
    top = (1 << LEVELS) - 1
    qa, qb = ((torch.floor(u * float(1 << LEVELS)).to(torch.int64)).clamp(0, top) for u in (rh, phi))
    key = (_spread(qa) << 1) | _spread(qb)
    order = torch.argsort(key, stable=True)
    order = order[torch.argsort(seg[order], stable=True)]
    ks, sg, ys, ils = key[order], seg[order], y[order], il[order]
    gam = (1.0 + n2[order]) / (1.0 - n2[order])
    terms = torch.stack([gam, 2.0 * ys[:, 0] / (1.0 - n2[order]), 2.0 * ys[:, 1] / (1.0 - n2[order])], 1)

    def dist(ra, rb, dr, sh):
        s = dr * dr + 4.0 * ra * rb * sh * sh
        x = 2.0 * s / ((1.0 - ra) * (1.0 + ra) * (1.0 - rb) * (1.0 + rb))
        return torch.log1p(x + torch.sqrt(x * (x + 2.0)))

    levels = []
    for ell in range(LEVELS + 1):
        pre = ks >> (2 * (LEVELS - ell))
        new = torch.ones(n, dtype=torch.bool, device=dev)
        new[1:] = (pre[1:] != pre[:-1]) | (sg[1:] != sg[:-1])
        first = torch.nonzero(new).flatten()
        cell = torch.cumsum(new, 0) - 1
        m = first.numel()
        count = torch.diff(torch.cat([first, torch.tensor([n], device=dev)]))
        sums = torch.zeros(m, 3, dtype=y.dtype, device=dev).index_add_(0, cell, terms)
        mid = sums[:, 1:] / sums[:, :1]
        yc = mid / (1.0 + torch.sqrt((1.0 - (mid * mid).sum(1)).clamp(min=0.0)))[:, None]
        one = count == 1
        yc = torch.where(one[:, None], ys[first], yc)
        ilc = torch.where(one, ils[first], 1.0 / (1.0 - (yc * yc).sum(1)))
        a, sc = _squeeze(pre[first] >> 1).double(), 2.0 ** -ell
        sp, l0 = span[sg[first]], lo[sg[first]]
        c0, c1, dc = l0 + sp * (a * sc), l0 + sp * ((a + 1.0) * sc), sp * sc
        if area:
            r0, r1 = torch.sqrt((c0 - 1.0) / (c0 + 1.0)), torch.sqrt((c1 - 1.0) / (c1 + 1.0))
            rs = r0 + r1
            dr = torch.where(rs > 0, 2.0 * dc / ((c0 + 1.0) * (c1 + 1.0) * torch.where(rs > 0, rs, 1.0)), 0.0)
        else:
            r0, r1, dr = c0, c1, dc
        sh = math.sin(math.pi * sc)
        rc = torch.maximum(torch.maximum(dist(r0, r1, dr, sh), dist(r0, r1, dr, 0.0)), dist(r1, r1, 0.0 * dr, sh))
        thr = 2.0 * torch.sinh(rc / (2.0 * theta)) ** 2
        if ell == 0:
            thr = torch.full_like(thr, math.inf)
        levels.append((first, count, yc, ilc, thr, cell))
        if m == n:
            break
    acc = torch.zeros(n, 4, dtype=y.dtype, device=dev)  # by sorted position
    step = max(1, min(n, int(4e7 * theta * theta / 200.0) + 1))
    for a in range(0, n, step):
        i = torch.arange(a, min(n, a + step), device=dev)
        ce = levels[0][5][i]
        for ell, (first, count, yc, ilc, thr, cell) in enumerate(levels):
            one = count[ce] == 1
            own = one & (first[ce] == i)
            dl = ys[i] - yc[ce]
            delta = 2.0 * (dl * dl).sum(1) * ils[i] * ilc[ce]
            take = (one & ~own) | (~one & (delta > thr[ce]))
            _add_pairs(acc, ys, ils, i[take], yc[ce[take]], ilc[ce[take]], count[ce[take]].double(), paper, "rep")
            left = ~take & ~own
            i, ce = i[left], ce[left]
            if i.numel() == 0:
                break
            last = ell == len(levels) - 1  # a bucket's points, or the cell's children
            begin = first[ce] if last else levels[ell + 1][5][first[ce]]
            kids = count[ce] if last else levels[ell + 1][5][first[ce] + count[ce] - 1] - begin + 1
            i = torch.repeat_interleave(i, kids)
            ramp = torch.arange(i.numel(), device=dev) - torch.repeat_interleave(torch.cumsum(kids, 0) - kids, kids)
            ce = torch.repeat_interleave(begin, kids) + ramp
            if last:
                far = ce != i
                _add_pairs(acc, ys, ils, i[far], ys[ce[far]], ils[ce[far]], 1.0, paper, "rep")
    out = torch.empty_like(acc)
    out[order] = acc
    return out


def _gradient(case, y, off, seg, edges):
    """Euclidean gradient, Z per segment and the attractive sums' pieces at y."""
    paper = case["grad_form"] == "paper"
    il = 1.0 / (1.0 - (y * y).sum(1))
    if case["theta"] == 0.0:
        acc = _exact_repulsion(y, il, seg, paper)
    else:
        acc = _tree_repulsion(y, il, off, seg, case["theta"], case["split_rule"] == "equal_area", paper)
    rep, zi = _force(acc, y, il)
    z = torch.zeros(len(off) - 1, dtype=y.dtype, device=y.device).index_add_(0, seg, zi)
    i, j, v = edges
    acc = torch.zeros_like(acc)
    for a in range(0, i.numel(), 1 << 25):
        b = slice(a, a + (1 << 25))
        jj = j[b].long()
        _add_pairs(acc, y, il, i[b], y[jj], il[jj], v[b].double(), paper, "att")
    att, _ = _force(acc, y, il)
    return 4.0 * (case["exaggeration"] * att - rep / z[seg][:, None]), z


def exact(case, seed):
    off, indptr, indices, values, y = _inputs(case, seed)
    dev, n = y.device, case["n"]
    seg = torch.repeat_interleave(torch.arange(len(off) - 1, device=dev), torch.as_tensor(np.diff(off), device=dev))
    edges = (torch.repeat_interleave(torch.arange(n, device=dev), torch.diff(indptr)), indices, values)
    if case["entry"] == "grad":
        g, z = _gradient(case, y, off, seg, edges)
        return {"grad": g, "Z": float(z[0])}
    if case["entry"] == "kl":
        g, z = _gradient(dict(case, exaggeration=1.0), y, off, seg, edges)
        i, j, p = edges[0], edges[1].long(), edges[2].double()
        n2 = (y * y).sum(1)
        delta = 2.0 * ((y[i] - y[j]) ** 2).sum(1) / ((1.0 - n2[i]) * (1.0 - n2[j]))
        w, _, _ = _pair(delta, False)
        return {"loss": (p * (torch.log(p) - torch.log(w))).sum() + p.sum() * torch.log(z[0]), "grad": g}
    lr = torch.full((n,), case["n"] / 12000.0, dtype=y.dtype, device=dev)
    if case["segments"] > 1:
        lr = torch.as_tensor(np.diff(off) / 12000.0, device=dev)[seg]
    vel, gains = torch.zeros_like(y), torch.ones_like(y)
    for _ in range(case["iters"]):
        g, _ = _gradient(case, y, off, seg, edges)
        n2 = (y * y).sum(1, keepdim=True)
        a = 1.0 - n2
        if case["use_gains"]:
            gains = torch.where((g > 0) == (vel > 0), gains * 0.8, gains + 0.2).clamp(min=0.01)
        vel = case["momentum"] * vel - lr[:, None] * gains * (g * (0.5 * a) ** case["metric_pow"])
        norm = torch.sqrt((vel * vel).sum(1, keepdim=True))
        u = torch.where(norm > 0, torch.tanh(norm / a) / torch.where(norm > 0, norm, 1.0), 0.0) * vel
        pu, nu = (y * u).sum(1, keepdim=True), (u * u).sum(1, keepdim=True)
        q = ((1.0 + 2.0 * pu + nu) * y + a * u) / (1.0 + 2.0 * pu + n2 * nu)
        r = torch.sqrt((q * q).sum(1, keepdim=True))
        y = torch.where(r >= 1.0 - 0.5e-5, q * ((1.0 - 1e-5) / r), q)
    return {"Y": y, "velocity": vel}
