"""What the library is timed on: the calls that a program using it makes, over the sizes it meets.

A case is one call of a kind:

  new      an alpha complex of atoms in device memory: context, build, every list (rows, Size, flags)
  rebuild  a further build of a context that the program keeps
  host     atoms in host memory in, every list in host memory out (options host_results)
  batch    many molecules of uneven sizes in one context
  sweep    one build at alpha = 1, then the sub-complexes at smaller alphas
  train    a training step: filtration values as an autograd function, a loss, gradients of the inputs
  moved    fixed combinatorics: the values at moved atoms and the gradient for given weights
  chunked  a molecule in host memory built slab by slab, the whole result in host memory

Atoms are drawn like the synthetic molecules of the tests: random sequential addition at 0.05 atoms/A^3 with
1.3 A between centres in a ball (or the shell between radii 320 and 361 A), element radii C/N/O/S, with or
without a 1.4 A probe; or a particle cloud, a jittered lattice with radii over a factor of 8. Centres and
radii are multiples of 1/1024 A, which is what the library quantises to. The molecule is the case's own; the
seed gives its pose (place, axes, mirror images) and the order of its atoms, as files of one molecule differ.
So the lists have the same lengths for every seed, and other rows and values in every place.
"""
import math

import numpy as np
import torch

import paper_1908_05944_gb300 as ac

DENSITY = 0.05                            # atoms per A^3
SEPARATION2 = math.ceil((1.3 * 1024) ** 2)  # quanta^2
RADII = {"vdw": (1741, 1587, 1556, 1843), "probe": (3174, 3021, 2990, 3277)}  # C N O S, quanta of 1/1024 A
ELEMENTS = (0.63, 0.80, 0.99)             # cumulative shares of C, N, O
SHELL = (320.0, 361.0)                    # radii of the capsid-like shell of 3,000,000 atoms
SWEEP = (0.0, 0.25, 0.6)                  # alphas below the built one

# rows of the complex per atom (vertices, edges, triangles, tetrahedra) by input (measured on the synthetic inputs)
PER_ATOM = {("vdw", 0.0): (1.0, 2.9, 1.7, 0.27), ("vdw", 1.0): (1.0, 4.3, 4.1, 1.1), ("probe", 0.0): (1.0, 7.5, 12.7, 6.2),
            ("particles", 0.0): (0.45, 2.4, 3.5, 1.6)}
ROW_BYTES = (13, 17, 21, 25)              # indices, one FP64 value, one flag


def listed():
    return [
        # a small protein, once: latency and launches (the paper's smallest structures hold 1,500 atoms)
        {"name": "globule2k_vdw", "kind": "new", "n": 2000, "radii": "vdw", "alpha": 0.0, "precision": "filtered"},
        # the headline molecule: a large complex with solvent-probe radii, from device memory, lists back
        {"name": "globule100k_probe", "kind": "new", "n": 100000, "radii": "probe", "alpha": 0.0, "precision": "filtered"},
        # the largest single build: a virus capsid
        {"name": "shell3m_probe", "kind": "new", "n": 3000000, "radii": "probe", "alpha": 0.0, "precision": "filtered"},
        # the plain FP64 option on the headline molecule
        {"name": "globule100k_plain_fp64", "kind": "new", "n": 100000, "radii": "probe", "alpha": 0.0, "precision": "plain"},
        # particles with widely spread radii (neighbour counts from a few to over a hundred)
        {"name": "particles100k", "kind": "new", "n": 100000, "radii": "particles", "alpha": 0.0, "precision": "filtered"},
        # a kept context built again
        {"name": "rebuild100k_probe", "kind": "rebuild", "n": 100000, "radii": "probe", "alpha": 0.0},
        # a service: host arrays in, host lists out
        {"name": "host100k_probe", "kind": "host", "n": 100000, "radii": "probe", "alpha": 0.0},
        # a screening run: many molecules at once, sizes log-uniform in [500, 50,000]
        {"name": "batch64_probe", "kind": "batch", "n_mol": 64, "lo": 500, "hi": 50000, "radii": "probe", "alpha": 0.0},
        # void and pocket analysis: one build at alpha = 1 and three smaller alphas from it
        {"name": "sweep20k_vdw", "kind": "sweep", "n": 20011, "radii": "vdw", "alpha": 1.0},
        # one optimisation step through the filtration values
        {"name": "train20k_probe", "kind": "train", "n": 20000, "radii": "probe", "alpha": 0.0},
        # values and gradient at moved atoms with the combinatorics of an earlier build
        {"name": "moved100k_probe", "kind": "moved", "n": 100000, "radii": "probe", "alpha": 0.0},
        # out-of-core: slabs of 100,000 atoms of a molecule in host memory
        {"name": "chunked300k_probe", "kind": "chunked", "n": 300007, "radii": "probe", "alpha": 0.0, "slab": 100000},
    ]


def _size(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["new", "new", "new", "rebuild", "host", "batch", "sweep", "train", "moved", "chunked"])
    radii = rng.choice(["vdw", "probe", "probe"])
    if kind == "new":
        form = rng.choice(["filtered", "filtered", "plain", "particles"])
        if form == "plain":
            return {"kind": kind, "n": _size(rng, 500, 100000), "radii": radii, "alpha": 0.0, "precision": "plain"}
        if form == "particles":
            return {"kind": kind, "n": _size(rng, 500, 100000), "radii": "particles", "alpha": 0.0, "precision": "filtered"}
        alpha = round(rng.uniform(0.0, 1.0), 3) if radii == "vdw" and rng.random() < 0.5 else 0.0
        return {"kind": kind, "n": _size(rng, 500, 2500000), "radii": radii, "alpha": alpha, "precision": "filtered"}
    if kind == "batch":
        lo = _size(rng, 100, 3000)
        return {"kind": kind, "n_mol": _size(rng, 2, 128), "lo": lo, "hi": lo * rng.randint(2, 16), "radii": radii, "alpha": 0.0}
    if kind == "sweep":
        return {"kind": kind, "n": _size(rng, 500, 100000), "radii": "vdw", "alpha": 1.0}
    if kind == "chunked":
        n = _size(rng, 20000, 400000)
        return {"kind": kind, "n": n, "radii": radii, "alpha": 0.0, "slab": max(5000, int(n * rng.uniform(0.2, 0.6)))}
    hi = {"rebuild": 1000000, "host": 300000, "train": 100000, "moved": 200000}[kind]
    return {"kind": kind, "n": _size(rng, 500, hi), "radii": radii, "alpha": 0.0}


# ---------------------------------------------------------------------------
# inputs


def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _points(g, n, r_in, r_out, dev):
    """n quantised centres by random sequential addition, a round of draws at a time: a draw stays if it is
    far enough from every accepted centre and from every earlier draw of its round."""
    cell = 768  # quanta: two points of one cell are always too close
    side = 2 * (int(math.ceil(r_out * 1024)) // cell + 4)
    table = torch.full((side * side * side,), -1, dtype=torch.int32, device=dev)
    pts = torch.zeros((n, 3), dtype=torch.int64, device=dev)
    have = 0
    near = torch.tensor([(z * side + y) * side + x for x in range(-2, 3) for y in range(-2, 3) for z in range(-2, 3)
                         if (x, y, z) != (0, 0, 0)], device=dev)
    while have < n:
        m = int(1.6 * (n - have)) + 64
        d = torch.randn((m, 3), dtype=torch.float64, device=dev, generator=g)
        u = torch.rand(m, dtype=torch.float64, device=dev, generator=g)
        r = ((r_out ** 3 - r_in ** 3) * u + r_in ** 3) ** (1.0 / 3.0)
        q = torch.round(d / d.norm(dim=1, keepdim=True) * r[:, None] * 1024).to(torch.int64)
        c = torch.div(q, cell, rounding_mode="floor") + side // 2
        key = (c[:, 2] * side + c[:, 1]) * side + c[:, 0]
        # this round's draws enter the table as n + their number: the earliest of a cell, in empty cells only
        first = torch.full_like(table, 0x7fffffff)
        first.scatter_reduce_(0, key, torch.arange(n, n + m, dtype=torch.int32, device=dev), "amin")
        free = table < 0
        table = torch.where(free & (first != 0x7fffffff), first, table)
        del first, free
        ok = table[key].to(torch.int64) == torch.arange(n, n + m, device=dev)
        both = torch.cat([pts, q])
        own = torch.arange(n, n + m, device=dev)[ok]
        k, p = key[ok], q[ok]
        good = torch.ones(len(own), dtype=torch.bool, device=dev)
        for j in range(0, len(own), 1 << 18):
            t = slice(j, j + (1 << 18))
            o = table[k[t, None] + near].to(torch.int64)
            e = both[o.clamp(min=0)] - p[t, None]
            good[t] = ~((o >= 0) & (o < own[t, None]) & ((e * e).sum(2) < SEPARATION2)).any(1)
        table[k] = -1
        k, p = k[good][: n - have], p[good][: n - have]
        pts[have:have + len(p)] = p
        table[k] = torch.arange(have, have + len(p), dtype=torch.int32, device=dev)
        have += len(p)
    return pts


def _molecule(n, radii, seed, dev):
    """Quantised atoms: centres (n, 3) and radii (n,), int64, in 1/1024 A."""
    g = torch.Generator(device=dev)
    g.manual_seed(seed)
    if radii == "particles":
        m = max(1, math.ceil(n ** (1.0 / 3.0) - 1e-9))
        k = torch.arange(n, device=dev)
        lattice = torch.stack([k % m, (k // m) % m, k // (m * m)], 1).to(torch.float64)
        u = torch.rand((n, 4), dtype=torch.float64, device=dev, generator=g)
        xyz = lattice + (u[:, :3] - 0.5) * 0.8
        return torch.round(xyz * 1024).to(torch.int64), torch.round(0.25 * 8.0 ** u[:, 3] * 1024).to(torch.int64)
    if n >= 1500000:  # the shell's thickness, its outer radius by the number of atoms
        vol, t = n / DENSITY, SHELL[1] - SHELL[0]
        # 4 pi / 3 (R^3 - (R - t)^3) = vol
        R = t / 2 + math.sqrt(max(0.0, vol / (4 * math.pi * t) - t * t / 12))
        pts = _points(g, n, R - t, R, dev)
    else:
        pts = _points(g, n, 0.0, (3 * n / (4 * math.pi * DENSITY)) ** (1.0 / 3.0), dev)
    u = torch.rand(n, dtype=torch.float64, device=dev, generator=g)
    e = torch.bucketize(u, torch.tensor(ELEMENTS, dtype=torch.float64, device=dev))
    return pts, torch.tensor(RADII[radii], dtype=torch.int64, device=dev)[e]


def _atoms(n, radii, number, seed, dev):
    """A molecule in the seed's pose and order of atoms."""
    pts, rad = _molecule(n, radii, number, dev)
    rng = np.random.default_rng(seed)
    sign = torch.as_tensor(rng.choice([-1, 1], 3), device=dev)
    move = torch.as_tensor(rng.integers(-51200, 51201, 3), device=dev)
    pts = pts[:, torch.as_tensor(rng.permutation(3), device=dev)] * sign + move
    g = torch.Generator(device=dev)
    g.manual_seed(seed)
    o = torch.randperm(n, device=dev, generator=g)
    return pts[o].contiguous(), rad[o].contiguous()


def _batch_sizes(case):
    rng = np.random.default_rng(case["n_mol"] * 1000003 + case["lo"])
    return np.round(np.exp(rng.uniform(math.log(case["lo"]), math.log(case["hi"]), case["n_mol"]))).astype(np.int64)


def _input(case, seed, dev):
    """Quantised atoms of a case and, for a batch, the offsets of its molecules."""
    if case["kind"] != "batch":
        return (*_atoms(case["n"], case["radii"], case["n"], seed, dev), None)
    sizes = _batch_sizes(case)
    mols = [_atoms(int(n), case["radii"], m, seed * 4096 + m, dev) for m, n in enumerate(sizes)]
    return torch.cat([m[0] for m in mols]), torch.cat([m[1] for m in mols]), np.concatenate([[0], np.cumsum(sizes)])


def _moves(case, seed, n, dev):
    g = torch.Generator(device=dev)
    g.manual_seed(seed + 77)
    dx = 1e-3 * torch.randn((n, 3), dtype=torch.float64, device=dev, generator=g)
    dr = 1e-4 * torch.randn(n, dtype=torch.float64, device=dev, generator=g)
    return dx, dr


def _weights(seed, counts, dev):
    g = torch.Generator(device=dev)
    g.manual_seed(seed + 78)
    return [torch.randn(m, dtype=torch.float64, device=dev, generator=g) for m in counts]


def prepare(case, seed):
    dev = _device()
    q, rq, off = _input(case, seed, dev)
    c, r = q.to(torch.float64) / 1024.0, rq.to(torch.float64) / 1024.0
    kind = case["kind"]
    s = {"kind": kind, "alpha": case["alpha"], "c": c, "r": r}
    if kind == "new":
        s["precision"] = ac.AC_PRECISION_PLAIN_FP64 if case["precision"] == "plain" else ac.AC_PRECISION_FILTERED
    elif kind == "batch":
        s["offsets"] = off
    elif kind in ("host", "chunked"):
        s["c"], s["r"] = c.cpu(), r.cpu()
        if kind == "host":  # a service receives into page-locked memory
            s["c"], s["r"] = s["c"].pin_memory(), s["r"].pin_memory()
            s["cx"] = None
        else:
            s["slab"] = case["slab"]
    elif kind == "train":
        s["c"], s["r"] = c.requires_grad_(), r.requires_grad_()
    elif kind in ("rebuild", "moved"):
        s["cx"] = ac.AlphaComplex(c, r, case["alpha"]).build()
        if kind == "rebuild":
            s["cx"].build()
        else:
            dx, dr = _moves(case, seed, len(r), dev)
            s["c2"], s["r2"] = c + dx, r + dr
            s["w"] = _weights(seed, [s["cx"].count(d) for d in range(4)], dev)
    return s


def _lists(cx, copy=True):
    return {"rows": [cx.simplices(d, copy=copy) for d in range(4)], "values": [cx.filtration_values(d, copy=copy) for d in range(4)],
            "attached": [cx.attached(d, copy=copy) for d in range(4)]}


def run(s):
    kind = s["kind"]
    if kind == "new":
        return _lists(ac.alpha_complex(s["c"], s["r"], s["alpha"], precision=s["precision"]))
    if kind == "rebuild":
        return _lists(s["cx"].build(), copy=False)
    if kind == "host":
        # the lists stay in the context's page-locked memory until the next request replaces it
        s["cx"] = cx = ac.AlphaComplex(s["c"], s["r"], s["alpha"], ac.options(host_results=True)).build()
        got = [cx.host_lists(d, copy=False) for d in range(4)]
        return {"rows": [t for t, _, _ in got], "values": [f for _, f, _ in got], "attached": [a for _, _, a in got]}
    if kind == "batch":
        # every molecule's lists, in the molecules' order
        cx = ac.AlphaComplex(s["c"], s["r"], s["alpha"], offsets=s["offsets"]).build()
        out = {"rows": [], "values": [], "attached": []}
        for d in range(4):
            mols = range(cx.n_mol)
            out["rows"].append(torch.cat([cx.simplices(d, m, copy=False) for m in mols]))
            out["values"].append(torch.cat([cx.filtration_values(d, m, copy=False) for m in mols]))
            out["attached"].append(torch.cat([cx.attached(d, m, copy=False) for m in mols]))
        return out
    if kind == "sweep":
        cx = ac.alpha_complex(s["c"], s["r"], s["alpha"])
        return {"whole": _lists(cx), "sub": [cx.subcomplex(a) for a in SWEEP]}
    if kind == "train":
        c, r = s["c"], s["r"]
        c.grad = r.grad = None
        f = ac.AlphaFiltration.apply(c, r, s["alpha"])
        sum((x * x).sum() for x in f).backward()
        return {"values": [x.detach() for x in f], "dcentres": c.grad, "dradii": r.grad}
    if kind == "moved":
        dc, dr = s["cx"].backward(s["w"])
        return {"values": s["cx"].eval_filtration(s["c2"], s["r2"]), "dcentres": dc, "dradii": dr}
    if kind == "chunked":
        cx = ac.ChunkedComplex(s["c"], s["r"], s["alpha"], max_core_atoms=s["slab"])
        out = {"rows": [cx.simplices(d) for d in range(4)], "values": [cx.filtration_values(d) for d in range(4)],
               "attached": [cx.attached(d) for d in range(4)]}
        cx.close()
        return out
    raise ValueError(kind)


def work(case):
    kind, radii, alpha = case["kind"], case["radii"], case["alpha"]
    n = int(_batch_sizes(case).sum()) if kind == "batch" else case["n"]
    lo, hi = PER_ATOM.get((radii, 0.0)), PER_ATOM.get((radii, 1.0), PER_ATOM.get((radii, 0.0)))
    rows = [n * (a + (b - a) * alpha) for a, b in zip(lo, hi)]
    lists = sum(m * b for m, b in zip(rows, ROW_BYTES))
    # a simplex of the complex: its orthocentre and value (about 60 operations), and an empty-orthosphere test
    # (8 operations) against each of about 20 balls that touch all of its vertices
    flops = sum(rows) * (60 + 20 * 8)
    if kind == "moved":
        # read: both sets of atoms, each row with its source, the weights; written: values and gradients
        return {"bytes": 2 * 32 * n + sum(m * (4 * (d + 1) + 9 + 8 + 8) for d, m in enumerate(rows)) + 32 * n, "flops": sum(rows) * 2 * 100}
    if kind == "train":
        return {"bytes": 64 * n + 24 * sum(rows), "flops": flops + sum(rows) * 100}
    if kind == "sweep":
        # a sub-complex reads every row and value once more and writes those that stay (at most all of them)
        return {"bytes": 32 * n + lists + len(SWEEP) * 1.5 * sum(m * (4 * (d + 1) + 8) for d, m in enumerate(rows)), "flops": flops}
    return {"bytes": 32 * n + lists, "flops": flops}


# ---------------------------------------------------------------------------
# the definition in 64 bits: integers for what is an integer, double precision for the rest

STEP = 1 << 22


def _dot(a, b):
    return (a * b).sum(-1)


def _cross(a, b):
    return torch.stack([a[..., 1] * b[..., 2] - a[..., 2] * b[..., 1], a[..., 2] * b[..., 0] - a[..., 0] * b[..., 2],
                        a[..., 0] * b[..., 1] - a[..., 1] * b[..., 0]], -1)


def _ortho(P, W, rows):
    """Orthocentre relative to the first vertex (y), its power (OrthoSize), barycentric
    coordinates of the orthocentre; rows (m, k) of indices. Integer inputs are carried as integers up to the minors."""
    p0, w0 = P[rows[:, 0]], W[rows[:, 0]]
    k = rows.shape[1]
    f = torch.float64
    if k == 1:
        z = torch.zeros((len(rows), 3), dtype=f, device=rows.device)
        return z, -w0.to(f), torch.ones((len(rows), 1), dtype=f, device=rows.device)
    q = [P[rows[:, j]] - p0 for j in range(1, k)]
    a = [_dot(q[j - 1], q[j - 1]) - W[rows[:, j]] + w0 for j in range(1, k)]
    if k == 2:
        D = _dot(q[0], q[0]).to(f)
        mu = [a[0].to(f) / (2 * D)]
        y = mu[0][:, None] * q[0].to(f)
    elif k == 3:
        g11, g22, g12 = _dot(q[0], q[0]), _dot(q[1], q[1]), _dot(q[0], q[1])
        det = (g11 * g22 - g12 * g12).to(f)
        mu = [(g22 * a[0] - g12 * a[1]).to(f) / (2 * det), (g11 * a[1] - g12 * a[0]).to(f) / (2 * det)]
        y = mu[0][:, None] * q[0].to(f) + mu[1][:, None] * q[1].to(f)
    else:
        C = [_cross(q[1], q[2]), _cross(q[2], q[0]), _cross(q[0], q[1])]
        D = _dot(q[0], C[0]).to(f)
        N = (a[0][:, None] * C[0] + a[1][:, None] * C[1] + a[2][:, None] * C[2]).to(f)
        y = N / (2 * D)[:, None]
        mu = [_dot(c.to(f), y) / D for c in C]
    lam = torch.stack([1 - sum(mu)] + mu, 1)
    return y, _dot(y, y) - w0.to(f), lam


def _meeting(P, S, mol):
    """Ordered pairs (i, x), sorted by i, of atoms of one molecule whose grown balls (squared radii S) meet."""
    dev, n = P.device, len(P)
    h = max(1, int(math.ceil(2 * math.sqrt(max(1.0, float(S.max()))))))
    c = torch.div(P - P.min(0).values, h, rounding_mode="floor") + 1
    dim = c.max(0).values + 2
    key = ((mol * dim[2] + c[:, 2]) * dim[1] + c[:, 1]) * dim[0] + c[:, 0]
    order = torch.argsort(key)
    sk = key[order]
    out_i, out_x = [], []
    for i0 in range(0, n, 1 << 18):
        ids = torch.arange(i0, min(n, i0 + (1 << 18)), device=dev)
        for dz in (-1, 0, 1):
            for dy in (-1, 0, 1):
                k = key[ids] + (dz * dim[1] + dy) * dim[0]
                a, b = torch.searchsorted(sk, k - 1), torch.searchsorted(sk, k + 1, right=True)
                m = b - a
                i = torch.repeat_interleave(ids, m)
                x = order[torch.arange(len(i), device=dev) - torch.repeat_interleave(torch.cumsum(m, 0) - m, m) + torch.repeat_interleave(a, m)]
                D = _dot(P[i] - P[x], P[i] - P[x])
                t = D - S[i] - S[x]
                ok = (i != x) & (mol[i] == mol[x]) & (S[i] >= 0) & (S[x] >= 0) & ((t <= 0) | (t * t <= 4 * S[i] * S[x]))
                out_i.append(i[ok])
                out_x.append(x[ok])
    i, x = torch.cat(out_i), torch.cat(out_x)
    D = _dot(P[i] - P[x], P[i] - P[x])
    o = torch.argsort(D, stable=True)
    o = o[torch.argsort(i[o], stable=True)]
    return i[o], x[o]


def _empty(P, W, rows, y, start, deg, nbr):
    """Whether no ball is nearer (in power) to a simplex's orthocentre than its vertices: the neighbours of the
    first vertex are tried in order of distance, and a simplex leaves at its first violator."""
    keep = torch.ones(len(rows), dtype=torch.bool, device=rows.device)
    live = torch.arange(len(rows), device=rows.device)
    j = 0
    while len(live):
        i = rows[live, 0]
        live = live[deg[i] > j]
        if not len(live):
            break
        i = rows[live, 0]
        x = nbr[start[i] + j]
        q = P[x] - P[i]
        a = _dot(q, q) - W[x] + W[i]
        delta = a.to(torch.float64) - 2 * _dot(q.to(torch.float64), y[live])
        bad = (delta < 0) & ~(rows[live] == x[:, None]).any(1)
        keep[live[bad]] = False
        live = live[~bad]
        j += 1
    return keep


def _pairs_within(group, m_total, dev):
    """All pairs (a, b), a before b, of positions within equal runs of a sorted array."""
    _, cnt = torch.unique_consecutive(group, return_counts=True)
    end = torch.repeat_interleave(torch.cumsum(cnt, 0), cnt)
    pos = torch.arange(m_total, device=dev)
    m = end - pos - 1
    a = torch.repeat_interleave(pos, m)
    b = torch.arange(len(a), device=dev) - torch.repeat_interleave(torch.cumsum(m, 0) - m, m) + a + 1
    return a, b


def _lex(rows, n):
    """Rows in lexicographic order (the order)."""
    o = torch.arange(len(rows), device=rows.device)
    for k in reversed(range(rows.shape[1])):
        o = o[torch.argsort(rows[o, k], stable=True)]
    return o


def _complex64(P, W, A, mol):
    """The alpha complex by its definition: per dimension rows, Size (quanta^2), attached, source (dim, row)."""
    dev, n = P.device, len(P)
    f64 = torch.float64
    S = W + A
    i, x = _meeting(P, S, mol)
    deg = torch.bincount(i, minlength=n)
    start = torch.cumsum(deg, 0) - deg
    # potential simplices: orthocentre in the closed alpha-grown balls
    D = _dot(P[i] - P[x], P[i] - P[x])
    t = D + W[i] - W[x]
    e = (i < x) & (t * t <= 4 * D * S[i])
    edges = torch.stack([i[e], x[e]], 1)
    edges = edges[torch.argsort(edges[:, 0] * n + edges[:, 1])]
    ekey = edges[:, 0] * n + edges[:, 1]

    def has(keys, k):
        at = torch.searchsorted(keys, k).clamp(max=max(0, len(keys) - 1))
        return keys[at] == k if len(keys) else torch.zeros_like(k, dtype=torch.bool)

    def potential(base, prefix, extra):
        """Rows base[a] + last entry of base[b] over pairs of equal prefix, kept if `extra` and the alpha bound hold."""
        got, gy, go = [], [], []
        if not len(base):
            z = torch.zeros((0, base.shape[1] + 1), dtype=torch.int64, device=dev)
            return z, torch.zeros((0, 3), dtype=f64, device=dev), torch.zeros(0, dtype=f64, device=dev)
        _, cnt = torch.unique_consecutive(prefix, return_counts=True)
        bound = torch.cumsum(cnt, 0)
        work_ = torch.cumsum(cnt * (cnt - 1) // 2, 0)
        g0 = 0
        while g0 < len(cnt):
            done = int(work_[g0 - 1]) if g0 else 0
            g1 = max(g0 + 1, int(torch.searchsorted(work_, done + STEP, right=True)))
            r0, r1 = (int(bound[g0 - 1]) if g0 else 0), int(bound[g1 - 1])
            a, b = _pairs_within(prefix[r0:r1], r1 - r0, dev)
            rows = torch.cat([base[r0 + a], base[r0 + b][:, -1:]], 1)
            rows = rows[extra(rows)]
            y, os, _ = _ortho(P, W, rows)
            ok = os <= A  # not finite for degenerate tuples: false, or a NaN, which is false too
            got.append(rows[ok])
            gy.append(y[ok])
            go.append(os[ok])
            g0 = g1
        return torch.cat(got), torch.cat(gy), torch.cat(go)

    tris, ty, tos = potential(edges, edges[:, 0], lambda r: has(ekey, r[:, 1] * n + r[:, 2]))
    o = _lex(tris, n)
    tris, ty, tos = tris[o], ty[o], tos[o]
    tets, qy, qos = potential(tris, tris[:, 0] * n + tris[:, 1], lambda r: has(ekey, r[:, 2] * n + r[:, 3]))

    def kept(rows, y):
        m = torch.ones(len(rows), dtype=torch.bool, device=dev)
        for k in range(0, len(rows), STEP):
            m[k:k + STEP] = _empty(P, W, rows[k:k + STEP], y[k:k + STEP], start, deg, x)
        return m

    ey, eos, _ = _ortho(P, W, edges)
    # an edge's test in integers: a_x |q|^2 - a (q . q_x), so that only exact ties are left to the order of input
    free = [None, None, tris[kept(tris, ty)], tets[kept(tets, qy)]]
    free[1] = edges[kept(edges, ey)]
    a_at = _dot(P[i] - P[x], P[i] - P[x]) - W[x] + W[i]
    vbad = torch.zeros(n, dtype=torch.bool, device=dev)
    vbad[i[(a_at < 0) | ((a_at == 0) & (x < i))]] = True
    free[0] = torch.arange(n, device=dev)[~vbad & (S >= 0)][:, None]
    out = [None] * 4
    up = None
    for d in (3, 2, 1, 0):
        rows, flag = free[d], torch.ones(len(free[d]), dtype=torch.int64, device=dev)
        if up is not None and len(up[0]):
            faces = torch.cat([up[0][:, [j for j in range(d + 2) if j != drop]] for drop in range(d + 2)])
            rows = torch.cat([rows, faces])
            flag = torch.cat([flag, torch.zeros(len(faces), dtype=torch.int64, device=dev)])
        o = torch.argsort(flag, descending=True, stable=True)
        o = o[_lex(rows[o], n)]
        srt = rows[o]
        new = torch.ones(len(srt), dtype=torch.bool, device=dev)
        new[1:] = (srt[1:] != srt[:-1]).any(1)
        row_of = torch.empty(len(srt), dtype=torch.int64, device=dev)
        row_of[o] = torch.cumsum(new.to(torch.int64), 0) - 1
        K, att = srt[new], flag[o][new] == 0
        _, os, _ = _ortho(P, W, K)
        size, sd, si = os.clone(), torch.full((len(K),), d, device=dev), torch.arange(len(K), device=dev)
        if up is not None and len(up[0]):
            m = len(up[0])
            fr = row_of[len(free[d]):]           # the row of each facet
            cof = torch.arange(m, device=dev).repeat(d + 2)
            best = torch.full((len(K),), math.inf, dtype=f64, device=dev).scatter_reduce(0, fr, up[1][cof], "amin")
            at = up[1][cof] == best[fr]
            arg = torch.full((len(K),), 1 << 40, device=dev).scatter_reduce(0, fr[at], cof[at], "amin")
            size[att] = best[att]
            sd[att], si[att] = up[3][arg[att]], up[4][arg[att]]
        out[d] = (K, size, att, sd, si)
        up = out[d]
    return out


def _gradient(P, W, K, w):
    """d/dp, d/dr of sum w . Size with the combinatorics fixed (A^2, A)."""
    dev = P.device
    X, R = P.to(torch.float64) / 1024, torch.sqrt(W.to(torch.float64)) / 1024
    dX, dR = torch.zeros_like(X), torch.zeros_like(R)
    tot = [torch.zeros(len(k[0]), dtype=torch.float64, device=dev) for k in K]
    for d in range(4):
        for s in range(4):
            m = K[d][3] == s
            tot[s].index_add_(0, K[d][4][m], w[d][m])
    for s in range(4):
        rows = K[s][0]
        y, _, lam = _ortho(P, W, rows)
        c = X[rows[:, 0]] + y / 1024
        for k in range(s + 1):
            g = 2 * tot[s] * lam[:, k]
            dX.index_add_(0, rows[:, k], g[:, None] * (X[rows[:, k]] - c))
            dR.index_add_(0, rows[:, k], -g * R[rows[:, k]])
    return dX, dR


def exact(case, seed):
    kind = case["kind"]
    dev = _device()
    n = int(_batch_sizes(case).sum()) if kind == "batch" else case["n"]
    if n > 800000:
        return None
    P, rq, off = _input(case, seed, dev)
    W = rq * rq
    mol = torch.zeros(n, dtype=torch.int64, device=dev)
    if off is not None:
        mol = torch.repeat_interleave(torch.arange(len(off) - 1, device=dev), torch.as_tensor(np.diff(off), device=dev))
    K = _complex64(P, W, int(round(case["alpha"] * 1048576)), mol)
    values = [k[1] / 1048576 for k in K]
    lists = {"rows": [None] * 4, "values": values, "attached": [None] * 4}
    if kind == "sweep":
        return {"whole": lists, "sub": [[(None, v[v <= a]) for v in values] for a in SWEEP]}
    if kind == "train":
        dX, dR = _gradient(P, W, K, [2 * v for v in values])
        return {"values": values, "dcentres": dX, "dradii": dR}
    if kind == "moved":
        dX, dR = _gradient(P, W, K, _weights(seed, [len(v) for v in values], dev))
        dx, dr = _moves(case, seed, n, dev)
        X2, R2 = P.to(torch.float64) / 1024 + dx, rq.to(torch.float64) / 1024 + dr
        own = [_ortho(X2, R2 * R2, k[0])[1] for k in K]
        moved = []
        for k in K:
            v = torch.zeros(len(k[0]), dtype=torch.float64, device=dev)
            for s in range(4):
                m = k[3] == s
                v[m] = own[s][k[4][m]]
            moved.append(v)
        return {"values": moved, "dcentres": dX, "dradii": dR}
    return lists  # a batch's: those of all molecules one after another
