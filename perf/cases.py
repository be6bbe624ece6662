"""Performance cases of the library: what a simulation that uses it spends its time on.

Each case is one call (or the pair pattern + values) through the public entry points of
``paper_2008_00409_gb300.pcloth``, at the sizes of the repository's own workloads (64 x 64
up to three stacked 526 x 526 sheets, garments of 2e3 .. 1e5 triangles, the 708 x 708 warm
start cloth, mini-batches of 65,536 rows):

  spmv       y = A x on an assembled system, difference form
  assemble   one step's pattern and values
  solve      Jacobi-PCG (mixed precision) on a given system
  step       one whole time step
  batch      one time step of many garments as one batched system
  proximity  the vertex-triangle pairs closer than the contact thickness
  infer      the learned warm start's guess for every vertex
  train      one Adam step of the learned warm start on a mini-batch

Meshes, states, contact pairs and systems are made here with torch from the seed alone;
the FP64 assembly below (membrane, bending, contact, gravity, pins: the definitions in
include/pcloth.h) makes the systems that `spmv` and `solve` get and is what `exact`
answers for `assemble` and the steps. Solves whose states are rough (z-jitter of 0.1 mm,
condition number about 1e6) run to a relative residual of 1e-9, so that the solution is
determined to FP32 accuracy; steps start from smooth states and use the tolerances of the
benchmark (1e-6) or of the tests (1e-9).
"""
from __future__ import annotations

import math

import torch

from paper_2008_00409_gb300 import pcloth as pc
from paper_2008_00409_gb300.workloads import Material

DEV = "cuda"
H_STEP = 1.0 / 200.0

# --------------------------------------------------------------------------- the cases


def listed():
    return [
        # a small cloth's product: launch and latency (4,096 rows)
        {"name": "spmv_64", "kind": "spmv", "nx": 64, "ny": 64, "layers": 1, "contacts": 0.0},
        # the product at the paper's scale (830,028 rows, 11M blocks): memory bandwidth
        {"name": "spmv_stack526", "kind": "spmv", "nx": 526, "ny": 526, "layers": 3, "contacts": 0.05},
        # a small cloth's assembly, contacts changing the pattern
        {"name": "assemble_64", "kind": "assemble", "nx": 64, "ny": 64, "layers": 1, "contacts": 0.02},
        # assembly at the paper's scale
        {"name": "assemble_stack526", "kind": "assemble", "nx": 526, "ny": 526, "layers": 3, "contacts": 0.05},
        # an interactive cloth's solve (one thread-block cluster holds it)
        {"name": "solve_64", "kind": "solve", "nx": 64, "ny": 64, "layers": 1, "contacts": 0.0, "block": False},
        # one garment of 40k triangles, ragged grid, contacts
        {"name": "solve_garment", "kind": "solve", "nx": 151, "ny": 133, "layers": 1, "contacts": 0.01,
         "block": False},
        # a 520k-triangle cloth with 2% contacts
        {"name": "solve_512", "kind": "solve", "nx": 512, "ny": 512, "layers": 1, "contacts": 0.02, "block": False},
        # the headline step: three stacked sheets, 1.65M triangles, 5% interlayer contacts
        {"name": "step_stack526", "kind": "step", "nx": 526, "ny": 526, "layers": 3, "contacts": 0.05, "tol": 1e-6},
        # 16 garments of 2e3 .. 1e5 triangles advanced together
        {"name": "batch_16", "kind": "batch", "count": 16, "side_min": 33, "side_max": 225, "contacts": 0.01,
         "tol": 1e-9},
        # thickness contacts of three sheets 0.5 mm apart
        {"name": "proximity_stack301", "kind": "proximity", "nx": 301, "ny": 301, "layers": 3},
        # the learned guess for a 708 x 708 cloth
        {"name": "infer_708", "kind": "infer", "rows": 708 * 708},
        # one training step of the learned guess
        {"name": "train_65536", "kind": "train", "batch": 65536, "rows": 1 << 21},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["spmv", "assemble", "solve", "solve", "step", "batch", "proximity", "infer", "train"])
    if kind == "infer":
        return {"kind": kind, "rows": _log(rng, 1000, 708 * 708)}
    if kind == "train":
        return {"kind": kind, "batch": _log(rng, 2000, 65536), "rows": _log(rng, 1 << 17, 1 << 21)}
    if kind == "batch":
        return {"kind": kind, "count": rng.randint(2, 16), "side_min": _log(rng, 20, 60),
                "side_max": _log(rng, 61, 225), "contacts": round(rng.uniform(0.0, 0.02), 4), "tol": 1e-9}
    if kind == "proximity":
        n = _log(rng, 40, 301)
        return {"kind": kind, "nx": n, "ny": max(3, int(n * rng.uniform(0.7, 1.0))), "layers": rng.randint(2, 3)}
    if kind == "solve":
        n = _log(rng, 24, 512)
        layers = rng.choice([1, 1, 2]) if n <= 300 else 1
        return {"kind": kind, "nx": n, "ny": max(16, int(n * rng.uniform(0.7, 1.0))), "layers": layers,
                "contacts": round(rng.uniform(0.0, 0.04), 4), "block": rng.random() < 0.2}
    layers = rng.randint(1, 3)
    n = _log(rng, 24, 526)
    case = {"kind": kind, "nx": n, "ny": max(16, int(n * rng.uniform(0.7, 1.0))), "layers": layers,
            "contacts": round(rng.uniform(0.0, 0.05), 4)}
    if kind == "step":
        case["tol"] = 1e-6 if layers > 1 else 1e-9
    return case


# --------------------------------------------------------------------------- meshes and states


def _pieces(case):
    """(nx, ny, z) of every grid piece."""
    if case["kind"] == "batch":
        n, a, b = case["count"], case["side_min"], case["side_max"]
        sides = [int(round(a * (b / a) ** (k / max(1, n - 1)))) for k in range(n)]
        return [(s, s, 0.0) for s in sides]
    return [(case["nx"], case["ny"], 5e-4 * k) for k in range(case["layers"])]


def _counts(case):
    """Vertices, triangles, hinges, blocks of the mesh pattern (regular-grid closed form) and contact pairs."""
    V = T = H = B = P = 0
    for nx, ny, _ in _pieces(case):
        v, t = nx * ny, 2 * (nx - 1) * (ny - 1)
        e = (nx - 1) * ny + nx * (ny - 1) + (nx - 1) * (ny - 1)
        h = e - 2 * (nx - 1) - 2 * (ny - 1)
        V, T, H, B = V + v, T + t, H + h, B + v + 2 * e + 2 * h
        P += int(round(case.get("contacts", 0.0) * v))
    return V, T, H, B, P


def _capacity(case):
    """Room for the blocks of any cloth of the case: a flipped diagonal adds none."""
    _, _, _, blocks, pairs = _counts(case)
    return (blocks + 6 * pairs + 3) // 4 * 4


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _rand(g, *shape):
    return torch.rand(*shape, generator=g, device=DEV, dtype=torch.float64)


def _mesh(case, g):
    """Rest positions (FP32), triangles, pins, pieces: grids 1 m wide, interior vertices
    moved in the plane by up to 0.2 of the spacing, a tenth of the diagonals flipped, two
    corners of each piece pinned."""
    rests, tris, pins, pieces = [], [], [], []
    vb = 0
    for nx, ny, z in _pieces(case):
        dx = 1.0 / (nx - 1)
        j, i = torch.meshgrid(torch.arange(ny, device=DEV), torch.arange(nx, device=DEV), indexing="ij")
        inner = ((i > 0) & (i < nx - 1) & (j > 0) & (j < ny - 1)).double()
        off = (2.0 * _rand(g, 2, ny, nx) - 1.0) * 0.2 * dx * inner
        rests.append(torch.stack([i * dx + off[0], j * dx + off[1], torch.full_like(off[0], z)], -1).reshape(-1, 3))
        flip = (_rand(g, ny - 1, nx - 1) < 0.1)[..., None]
        v00 = (j * nx + i)[:-1, :-1]
        v10, v01, v11 = v00 + 1, v00 + nx, v00 + nx + 1
        t0 = torch.where(flip, torch.stack([v00, v10, v01], -1), torch.stack([v00, v10, v11], -1))
        t1 = torch.where(flip, torch.stack([v10, v11, v01], -1), torch.stack([v00, v11, v01], -1))
        tris.append(torch.stack([t0, t1], 2).reshape(-1, 3) + vb)
        pins += [vb + (ny - 1) * nx, vb + ny * nx - 1]
        pieces.append((nx, ny, vb, flip[..., 0]))
        vb += nx * ny
    return (torch.cat(rests).float().contiguous(), torch.cat(tris).int().contiguous(),
            torch.tensor(pins, dtype=torch.int32, device=DEV), pieces)


def _contacts(case, pieces, g):
    """Contact pairs, sorted by vertex: with a triangle of a neighbouring sheet at the same
    place (stacked sheets), or with one two to eight cells away on the same piece."""
    frac = case.get("contacts", 0.0)
    pairs = []
    for k, (nx, ny, vb, _) in enumerate(pieces):
        n = int(round(frac * nx * ny))
        if n == 0:
            continue
        local = torch.sort(torch.randperm(nx * ny, generator=g, device=DEV)[:n])[0]
        i, j = local % nx, local // nx
        r = _rand(g, 5, n)
        if case.get("layers", 1) > 1:
            other = 1 if k == 0 else k - 1 if k == len(pieces) - 1 else None
            o = torch.full_like(i, other) if other is not None else torch.where(r[0] < 0.5, k - 1, k + 1)
            qi = (i - (r[1] < 0.5).long()).clamp(0, nx - 2)
            qj = (j - (r[2] < 0.5).long()).clamp(0, ny - 2)
            base = torch.tensor([p[2] for p in pieces], device=DEV)[o]
            flips = torch.stack([p[3] for p in pieces])[o, qj, qi]
        else:
            reach = [max(2, min(8, m // 3)) for m in (nx, ny)]
            d = [(2 + (r[1 + a] * (reach[a] - 1)).long()) * torch.where(r[3 + a] < 0.5, -1, 1) for a in (0, 1)]
            qi = torch.where((i + d[0] >= 0) & (i + d[0] <= nx - 2), i + d[0], i - d[0]).clamp(0, nx - 2)
            qj = torch.where((j + d[1] >= 0) & (j + d[1] <= ny - 2), j + d[1], j - d[1]).clamp(0, ny - 2)
            base, flips = vb, pieces[k][3][qj, qi]
        v00 = qj * nx + qi
        v10, v01, v11 = v00 + 1, v00 + nx, v00 + nx + 1
        up = _rand(g, n) < 0.5
        a = torch.where(up & flips, v10, v00)
        b = torch.where(up, v11, v10)
        c = torch.where(up | flips, v01, v11)
        pairs.append(torch.stack([local + vb, a + base, b + base, c + base], -1))
    if not pairs:
        return None, None
    p = torch.cat(pairs).int().contiguous()
    e = -torch.log1p(-_rand(g, p.shape[0], 3)).clamp_min(1e-12)
    return p, (e / e.sum(1, keepdim=True)).float().contiguous()


def _state(rest, g, rough):
    """Positions and velocities: `rough` adds a z-jitter of N(0, 0.1 mm) at rest; otherwise a
    cloth in smooth motion (long waves of 0.2 mm, velocities of a few cm/s)."""
    r = rest.double()
    if rough:
        x = r.clone()
        x[:, 2] += 1e-4 * torch.randn(r.shape[0], generator=g, device=DEV, dtype=torch.float64)
        return x.float().contiguous(), torch.zeros_like(rest)
    ph = 2.0 * math.pi * _rand(g, 6)
    wave = torch.sin(4.0 * r[:, 0] + ph[0]) * torch.sin(3.0 * r[:, 1] + ph[1])
    x = r.clone()
    x[:, 2] += 2e-4 * wave
    v = torch.stack([0.01 * torch.sin(2.0 * r[:, 1] + ph[2]), 0.01 * torch.sin(2.0 * r[:, 0] + ph[3]),
                     -0.05 + 0.02 * torch.sin(3.0 * r[:, 0] + ph[4]) * torch.sin(2.0 * r[:, 1] + ph[5])], -1)
    return x.float().contiguous(), v.float().contiguous()


# --------------------------------------------------------------------------- the system in 64 bits


def _sum_by(key, val):
    """Sorted distinct keys and, for each, the sum of its rows of val in order of appearance (the same every time)."""
    key, order = torch.sort(key, stable=True)
    first = torch.ones_like(key, dtype=torch.bool)
    first[1:] = key[1:] != key[:-1]
    start = torch.nonzero(first)[:, 0]
    count = torch.diff(start, append=torch.tensor([key.numel()], device=DEV))
    out = val[order[start]]
    live = torch.nonzero(count > 1)[:, 0]
    k = 1
    while live.numel():
        out[live] += val[order[start[live] + k]]
        k += 1
        live = live[count[live] > k]
    return key[start], out


def _outer(a, b):
    return a[..., :, None] * b[..., None, :]


def _angle(x1, x2, x3, x4):
    n1 = torch.linalg.cross(x1 - x3, x1 - x4)
    n2 = torch.linalg.cross(x2 - x4, x2 - x3)
    e = x4 - x3
    le = e.norm(dim=1, keepdim=True)
    s1, s2 = n1.square().sum(1, keepdim=True), n2.square().sum(1, keepdim=True)
    th = torch.atan2((torch.linalg.cross(n1, n2) * e / le).sum(1) / (s1 * s2).sqrt()[:, 0],
                     (n1 * n2).sum(1) / (s1 * s2).sqrt()[:, 0])
    d = lambda u: (u * e).sum(1, keepdim=True) / le  # noqa: E731
    grad = -torch.stack([le / s1 * n1, le / s2 * n2, d(x1 - x4) / s1 * n1 + d(x2 - x4) / s2 * n2,
                         -d(x1 - x3) / s1 * n1 - d(x2 - x3) / s2 * n2], 1)
    return th, grad


def _system64(rest, tris, pins, x, v, pairs, w):
    """row_ptr, col_idx, A, b and the difference-form diagonal of one step, in FP64."""
    mat, h = Material(), H_STEP
    V = rest.shape[0]
    R, X, U, t = rest.double(), x.double(), v.double(), tris.long()
    idx, blocks, force = [], [], []  # per element kind: vertices, h^2 K blocks, right-hand sides

    # membrane: St. Venant-Kirchhoff, stress clamped to its positive part in the Hessian
    e1, e2 = R[t[:, 1]] - R[t[:, 0]], R[t[:, 2]] - R[t[:, 0]]
    n = torch.linalg.cross(e1, e2)
    area, l1 = 0.5 * n.norm(dim=1), e1.norm(dim=1)
    u = e1 / l1[:, None]
    d01, d11 = (e2 * u).sum(1), (e2 * torch.linalg.cross(n / n.norm(dim=1, keepdim=True), u)).sum(1)
    g1 = torch.stack([1.0 / l1, -d01 / (l1 * d11)], 1)
    g2 = torch.stack([torch.zeros_like(l1), 1.0 / d11], 1)
    gr = torch.stack([-g1 - g2, g1, g2], 1)
    mu, lam = mat.young / (2 * (1 + mat.poisson)), mat.young * mat.poisson / (1 - mat.poisson ** 2)
    F = torch.einsum("tka,tkc->tac", X[t], gr)
    G = 0.5 * (F.transpose(1, 2) @ F - torch.eye(2, device=DEV, dtype=torch.float64))
    tr = G[:, 0, 0] + G[:, 1, 1]
    S = 2 * mu * G + lam * tr[:, None, None] * torch.eye(2, device=DEV, dtype=torch.float64)
    m, dev = 0.5 * (S[:, 0, 0] + S[:, 1, 1]), S.clone()
    dev[:, 0, 0] -= m
    dev[:, 1, 1] -= m
    rad = (dev[:, 0, 0] ** 2 + S[:, 0, 1] ** 2).sqrt()
    unit = dev / rad.clamp_min(1e-300)[:, None, None]
    p1, p2 = (m + rad).clamp_min(0.0), (m - rad).clamp_min(0.0)
    Sp = 0.5 * (p1 + p2)[:, None, None] * torch.eye(2, device=DEV, dtype=torch.float64) + \
        0.5 * (p1 - p2)[:, None, None] * unit
    f = -area[:, None, None] * torch.einsum("tab,tbc,tkc->tka", F, S, gr)
    Fg = torch.einsum("tac,tkc->tka", F, gr)
    gg = torch.einsum("tkc,tlc->tkl", gr, gr)
    gSg = torch.einsum("tkc,tcd,tld->tkl", gr, Sp, gr)
    K = (gSg[..., None, None] * torch.eye(3, device=DEV, dtype=torch.float64)
         + mu * torch.einsum("tla,tkb->tklab", Fg, Fg) + lam * torch.einsum("tka,tlb->tklab", Fg, Fg)
         + mu * gg[..., None, None] * (F @ F.transpose(1, 2))[:, None, None])
    K *= (h * h * area)[:, None, None, None, None]
    idx.append(t)
    blocks.append(K)
    force.append(h * f - torch.einsum("tklab,tlb->tka", K, U[t]))
    mass = _sum_by(t.reshape(-1), (mat.rho * area / 3.0)[:, None].expand(-1, 3).reshape(-1, 1))
    mass = torch.zeros(V, device=DEV, dtype=torch.float64).index_copy(0, mass[0], mass[1][:, 0])

    # bending: the two triangles of every interior edge
    a, b, o = t.reshape(-1), t[:, [1, 2, 0]].reshape(-1), t[:, [2, 0, 1]].reshape(-1)
    key, order = torch.sort(torch.minimum(a, b) * V + torch.maximum(a, b), stable=True)
    s = torch.nonzero(key[1:] == key[:-1])[:, 0]
    h0, h1 = order[s], order[s + 1]
    hv = torch.stack([o[h0], o[h1], a[h0], b[h0]], 1)
    coef = 3.0 * (R[hv[:, 3]] - R[hv[:, 2]]).square().sum(1) / (area[h0 // 3] + area[h1 // 3])
    th0, _ = _angle(*(R[hv[:, k]] for k in range(4)))
    th, grad = _angle(*(X[hv[:, k]] for k in range(4)))
    k2 = 2.0 * mat.k_bend * coef
    q = (h * k2.sqrt())[:, None, None] * grad
    qv = (q * U[hv]).sum((1, 2))
    idx.append(hv)
    blocks.append(_outer(q[:, :, None, :].expand(-1, -1, 4, -1).reshape(-1, 3),
                         q[:, None, :, :].expand(-1, 4, -1, -1).reshape(-1, 3)).reshape(-1, 4, 4, 3, 3))
    force.append((-h * k2 * (th - th0))[:, None, None] * grad - q * qv[:, None, None])

    # contact: hold penalty along the partner triangle's normal
    if pairs is not None:
        pv = pairs.long()
        n = torch.linalg.cross(X[pv[:, 2]] - X[pv[:, 1]], X[pv[:, 3]] - X[pv[:, 1]])
        n = n / n.norm(dim=1, keepdim=True)
        sw = torch.cat([torch.ones_like(w[:, :1]), -w], 1).double()
        qc = h * math.sqrt(mat.k_contact) * sw[..., None] * n[:, None, :]
        idx.append(pv)
        blocks.append(_outer(qc[:, :, None, :].expand(-1, -1, 4, -1).reshape(-1, 3),
                             qc[:, None, :, :].expand(-1, 4, -1, -1).reshape(-1, 3)).reshape(-1, 4, 4, 3, 3))
        force.append(-qc * (qc * U[pv]).sum((1, 2))[:, None, None])

    # upper blocks (row <= column), their mirror images, the diagonal
    keys, vals = [torch.arange(V, device=DEV) * (V + 1)], [torch.zeros(V, 9, device=DEV, dtype=torch.float64)]
    for vid, blk in zip(idx, blocks):
        for k in range(vid.shape[1]):
            for l in range(k, vid.shape[1]):
                swap = (vid[:, k] > vid[:, l])[:, None, None]
                keys.append(torch.minimum(vid[:, k], vid[:, l]) * V + torch.maximum(vid[:, k], vid[:, l]))
                vals.append(torch.where(swap, blk[:, k, l].transpose(1, 2), blk[:, k, l]).reshape(-1, 9))
    del blocks, blk
    ukey, ublk = _sum_by(torch.cat(keys), torch.cat(vals))
    del keys, vals
    r, c = ukey // V, ukey % V
    low = torch.nonzero(r != c)[:, 0]
    key, order = torch.sort(torch.cat([ukey, c[low] * V + r[low]]))
    A = torch.cat([ublk, ublk[low].reshape(-1, 3, 3).transpose(1, 2).reshape(-1, 9)])[order]
    r, c = key // V, key % V
    row_ptr = torch.searchsorted(r, torch.arange(V + 1, device=DEV)).int()
    pinned = torch.zeros(V, dtype=torch.bool, device=DEV)
    pinned[pins.long()] = True
    eye = torch.eye(3, device=DEV, dtype=torch.float64).reshape(9)
    dres = mass[:, None] * eye
    near = torch.nonzero(pinned[c] & ~pinned[r])[:, 0]
    if near.numel():
        kk, ss = _sum_by(r[near], A[near])
        dres[kk] -= ss
    A[pinned[r] | pinned[c]] = 0.0
    dg = torch.nonzero(r == c)[:, 0]
    A[dg] += mass[:, None] * eye
    kk, ss = _sum_by(torch.cat([i.reshape(-1) for i in idx]), torch.cat([q.reshape(-1, 3) for q in force]))
    b = h * mass[:, None] * torch.tensor(mat.gravity, device=DEV, dtype=torch.float64)
    b[kk] += ss
    b[pinned] = 0.0
    return row_ptr, c.int(), A, b, dres


def _operator64(row_ptr, col_idx, A, dres):
    """The difference-form operator D_i p_i + sum_j A_ij (p_j - p_i) as a scalar CSR matrix, and its diagonal."""
    V, nb = row_ptr.numel() - 1, row_ptr.long().diff()
    r = torch.repeat_interleave(torch.arange(V, device=DEV), nb)
    dg = torch.nonzero(r == col_idx)[:, 0]
    A = A.double().clone().reshape(-1, 9)
    A[dg] = 0.0
    total = torch.zeros(V, 9, device=DEV, dtype=torch.float64)
    kk, ss = _sum_by(r, A)
    total[kk] = ss
    A[dg] = dres.double().reshape(V, 9) - total
    s0 = row_ptr[:-1].long()
    k = torch.arange(r.numel(), device=DEV) - s0[r]
    cols = torch.empty(9 * r.numel(), device=DEV, dtype=torch.int32)
    vals = torch.empty(9 * r.numel(), device=DEV, dtype=torch.float64)
    for a in range(3):
        for b in range(3):
            at = 9 * s0[r] + a * 3 * nb[r] + 3 * k + b
            cols[at] = 3 * col_idx + b
            vals[at] = A[:, 3 * a + b]
    crow = torch.zeros(3 * V + 1, device=DEV, dtype=torch.int32)
    crow[1:] = torch.cumsum((3 * nb).repeat_interleave(3), 0).int()
    return torch.sparse_csr_tensor(crow, cols, vals, (3 * V, 3 * V)), A[dg][:, [0, 4, 8]].reshape(-1)


def _solve64(row_ptr, col_idx, A, dres, b, tol=1e-12, limit=30000):
    """Jacobi-PCG in FP64."""
    M, d = _operator64(row_ptr, col_idx, A, dres)
    r = b.double().reshape(-1).clone()
    x = torch.zeros_like(r)
    z = r / d
    p, rz, stop = z.clone(), r @ z, tol * r.norm()
    for it in range(limit):
        q = M @ p
        al = rz / (p @ q)
        x += al * p
        r -= al * q
        z = r / d
        rz, old = r @ z, rz
        p = z + (rz / old) * p
        if it % 64 == 63 and bool(r.norm() <= stop):
            break
    return x.reshape(-1, 3)


# --------------------------------------------------------------------------- prepare, run, exact


def _opts(tol, block=False):
    return pc.solve_opts(tol=tol, max_iter=40000, precision=pc.PC_PREC_MIXED,
                         precond=pc.PC_PRECOND_BLOCK if block else pc.PC_PRECOND_JACOBI)


def _cloth(case, seed):
    g = _gen(seed)
    rest, tris, pins, pieces = _mesh(case, g)
    pairs, w = _contacts(case, pieces, g)
    x, v = _state(rest, g, case["kind"] in ("spmv", "assemble", "solve"))
    return {"rest": rest, "tris": tris, "pins": pins, "pieces": pieces, "pairs": pairs, "w": w, "x0": x, "v0": v,
            "g": g}


class _Context:
    """A library context that is released with the state that holds it."""

    def __init__(self, s, material, max_contacts):
        self.h = None
        self.h = pc.pc_create(s["rest"].shape[0], s["tris"].shape[0], s["tris"], s["rest"], s["pins"], material,
                              max_contacts)

    def __del__(self):
        if self.h is not None:
            pc.pc_destroy(self.h)


def _mlp(case, seed):
    """Rows of features and solutions at the scales of a falling cloth, a network and its statistics."""
    g, n = _gen(seed), case["rows"]
    f = lambda *s: torch.randn(*s, generator=g, device=DEV)  # noqa: E731
    scale = torch.tensor([0.3] * 3 + [0.05] * 3 + [2.0] * 3 + [0.05] * 3, device=DEV)
    feat = f(n, 12) * scale
    target = 0.05 * torch.tanh(feat[:, :3] + 0.5 * feat[:, 6:9]) + feat[:, 3:6] + 0.01 * f(n, 3)
    parts = []
    for fan_out, fan_in in ((64, 12), (64, 64), (3, 64)):
        parts += [(2.0 * torch.rand(fan_out * fan_in, generator=g, device=DEV) - 1.0) * math.sqrt(6.0 / fan_in),
                  0.1 * f(fan_out)]
    rows = torch.randint(0, n, (case.get("batch", 1),), generator=g, device=DEV, dtype=torch.int32)
    resid = (target - feat[:, 3:6]).double()
    stats = torch.cat([feat.double().mean(0), feat.double().std(0), resid.mean(0), resid.std(0)]).float()
    return {"feat": feat, "target": target, "params": torch.cat(parts), "stats": stats, "rows": rows,
            "fixed": (torch.rand(n, generator=g, device=DEV) < 1e-4).to(torch.uint8)}


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("infer", "train"):
        s = _mlp(case, seed)
        s["kind"], s["n"] = kind, case["rows"] if kind == "infer" else case["batch"]
        if kind == "infer":
            s["prev"], s["out"] = s["feat"][:, 3:6].contiguous(), torch.empty(case["rows"], 3, device=DEV)
        else:
            s["mlp"], s["opts"] = pc.pc_mlp_create(), pc.adam_opts(1e-3)
        return s
    s = _cloth(case, seed)
    s["kind"] = kind
    V, npairs = s["rest"].shape[0], 0 if s["pairs"] is None else s["pairs"].shape[0]
    material = Material(contact_thickness=5.5e-4) if kind == "proximity" else Material()
    s["ctx"] = _Context(s, material, npairs if kind != "proximity" else 6 * V)
    if kind == "proximity":
        s["x0"][:, 2] += 2e-5 * torch.randn(V, generator=s["g"], device=DEV)
        s["out"] = (torch.zeros(6 * V, 4, dtype=torch.int32, device=DEV), torch.zeros(6 * V, 3, device=DEV))
    elif kind in ("spmv", "solve"):
        s["row_ptr"], col, A, b, dres = _system64(s["rest"], s["tris"], s["pins"], s["x0"], s["v0"], s["pairs"], s["w"])
        s["nnzb"] = col.numel()
        cap = (s["nnzb"] + 3) // 4 * 4
        s["col_idx"] = torch.zeros(cap, dtype=torch.int32, device=DEV)
        s["col_idx"][: s["nnzb"]] = col
        s["vals"] = torch.zeros(9 * cap, device=DEV)
        s["vals"][: 9 * s["nnzb"]] = A.float().reshape(-1)
        s["b"], s["dres"] = b.float().reshape(-1), dres.float().reshape(-1)
        if kind == "spmv":
            s["p"] = torch.randn(3 * V, generator=s["g"], device=DEV)
        else:
            s["opts"] = _opts(1e-9, case["block"])
        s["out"] = torch.empty(3 * V, device=DEV)
    elif kind == "assemble":
        cap = _capacity(case)
        s["row_ptr"] = torch.zeros(V + 1, dtype=torch.int32, device=DEV)
        s["col_idx"] = torch.zeros(cap, dtype=torch.int32, device=DEV)
        s["vals"], s["b"], s["dres"] = (torch.zeros(k, device=DEV) for k in (9 * cap, 3 * V, 9 * V))
    else:
        s["x"], s["v"], s["dv"] = s["x0"].clone(), s["v0"].clone(), torch.empty(3 * V, device=DEV)
        o = pc.pc_step_opts()
        o.h, o.solve, o.warm_start = H_STEP, _opts(case["tol"]), pc.PC_WARM_ZERO
        s["opts"] = o
        s["inst"] = [p[2] for p in s["pieces"]] + [V]
    return s


def run(s):
    kind = s["kind"]
    if kind == "infer":
        pc.pc_mlp_infer(s["n"], s["params"], s["stats"], s["feat"], s["prev"], s["fixed"], s["out"])
        return s["out"]
    if kind == "train":
        pc.pc_mlp_train_step(s["mlp"], s["n"], s["rows"], s["params"], s["stats"], s["feat"], s["target"], s["opts"])
        return s["params"]
    ctx = s["ctx"].h
    if kind == "spmv":
        pc.pc_bsr_spmv(ctx, s["row_ptr"], s["col_idx"], s["nnzb"], s["vals"], s["dres"], s["p"], s["out"])
        return s["out"]
    if kind == "assemble":
        n = pc.pc_assemble_pattern(ctx, s["pairs"], s["w"], s["row_ptr"], s["col_idx"])
        pc.pc_assemble_values(ctx, s["row_ptr"], s["col_idx"], n, s["x0"], s["v0"], s["pairs"], s["w"], H_STEP,
                              s["vals"], s["b"], s["dres"])
        return {"nnzb": n, "row_ptr": s["row_ptr"], "col_idx": s["col_idx"], "vals": s["vals"], "b": s["b"],
                "dres": s["dres"]}
    if kind == "solve":
        s["out"].zero_()
        pc.pc_pcg_solve(ctx, s["row_ptr"], s["col_idx"], s["nnzb"], s["vals"], s["dres"], s["b"], s["out"], s["opts"])
        return s["out"]
    if kind == "proximity":
        n = pc.pc_proximity_query(ctx, s["x0"], 5.5e-4, *s["out"])
        return {"n": n, "pairs": s["out"][0], "w": s["out"][1]}
    # one time step from the same state each time
    s["x"].copy_(s["x0"])
    s["v"].copy_(s["v0"])
    if kind == "batch":
        pc.pc_step_batched(ctx, s["x"], s["v"], s["pairs"], s["w"], s["inst"], s["opts"])
        return {"x": s["x"], "v": s["v"]}
    pc.pc_step(ctx, s["x"], s["v"], s["pairs"], s["w"], s["opts"], dv_out=s["dv"])
    return {"x": s["x"], "v": s["v"], "dv": s["dv"]}


def _layers(p):
    p, out, o = p.double(), [], 0
    for fan_out, fan_in in ((64, 12), (64, 64), (3, 64)):
        out.append((p[o:o + fan_out * fan_in].reshape(fan_out, fan_in), p[o + fan_out * fan_in:o + fan_out * (fan_in + 1)]))
        o += fan_out * (fan_in + 1)
    return out


def _network(p, x):
    (w1, b1), (w2, b2), (w3, b3) = _layers(p)
    return torch.relu(torch.relu(x @ w1.T + b1) @ w2.T + b2) @ w3.T + b3


def exact(case, seed):
    kind = case["kind"]
    if kind == "proximity":  # membership and weights are defined by FP32 decisions, reproducible bit for bit
        return None
    if kind in ("infer", "train"):
        s = _mlp(case, seed)
        st = s["stats"].double()
        if kind == "infer":
            y = _network(s["params"], (s["feat"].double() - st[:12]) / st[12:24]) * st[27:] + st[24:27]
            y += s["feat"][:, 3:6].double()
            y[s["fixed"] != 0] = 0.0
            return y
        at = s["rows"].long()
        p = s["params"].double().requires_grad_(True)
        feat, target = s["feat"][at].double(), s["target"][at].double()
        y = _network(p, (feat - st[:12]) / st[12:24])
        loss = 0.5 * (y - (target - feat[:, 3:6] - st[24:27]) / st[27:]).square().sum() / y.shape[0]
        gr, = torch.autograd.grad(loss, p)
        return p.detach() - 1e-3 * gr / (gr.abs() + 1e-8)
    s = _cloth(case, seed)
    row_ptr, col, A, b, dres = _system64(s["rest"], s["tris"], s["pins"], s["x0"], s["v0"], s["pairs"], s["w"])
    if kind == "spmv":
        M, _ = _operator64(row_ptr, col, A.float(), dres.float())
        return M @ torch.randn(3 * s["rest"].shape[0], generator=s["g"], device=DEV).double()
    if kind == "assemble":
        vals = torch.zeros(9 * _capacity(case), device=DEV, dtype=torch.float64)
        vals[: A.numel()] = A.reshape(-1)
        return {"nnzb": None, "row_ptr": None, "col_idx": None, "vals": vals, "b": b.reshape(-1),
                "dres": dres.reshape(-1)}
    if kind == "solve":
        return _solve64(row_ptr, col, A.float(), dres.float(), b.float()).reshape(-1)
    dv = _solve64(row_ptr, col, A, dres, b)
    v = s["v0"].double() + dv
    out = {"x": s["x0"].double() + H_STEP * v, "v": v}
    return out if kind == "batch" else out | {"dv": dv.reshape(-1)}


def work(case):
    """Each input read once, each output written once; the products of a solve by the
    iterations that such grids take (about 14 per vertex of their longer side)."""
    kind = case["kind"]
    if kind == "infer":
        return {"bytes": case["rows"] * (12 + 3 + 3) * 4 + case["rows"], "flops": case["rows"] * 2 * (768 + 4096 + 192)}
    if kind == "train":
        return {"bytes": case["batch"] * (12 + 3 + 1) * 4, "flops": case["batch"] * 6 * (768 + 4096 + 192)}
    V, T, H, B, P = _counts(case)
    nnzb = B + 6 * P
    mesh = 56 * T + 24 * H + 4 * V + 28 * P
    if kind == "proximity":
        return {"bytes": 12 * V + 12 * T + 28 * 4 * V, "flops": 100 * 4 * V}
    if kind == "spmv":
        return {"bytes": 40 * nnzb + 64 * V, "flops": 18 * nnzb}
    if kind == "assemble":
        return {"bytes": mesh + 24 * V + 40 * nnzb + 52 * V, "flops": 600 * T + 400 * H + 9 * (9 * T + 16 * H)}
    iters = 14 * max(max(nx, ny) for nx, ny, _ in _pieces(case))
    if kind == "batch":
        iters = iters // 2
    flops = iters * (18 * nnzb + 30 * V)
    if kind == "solve":
        return {"bytes": 40 * nnzb + 72 * V, "flops": flops}
    return {"bytes": mesh + 48 * V, "flops": flops}
