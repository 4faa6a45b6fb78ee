"""The workloads whose speed matters to users of the library, each through its public entry points.

Point sets are drawn on the GPU from the seed: the halo / filament / background mixture that stands for an N-body
snapshot (60 % in NFW halos, 25 % along filaments, 15 % uniform), the halo + uniform mixture of the differentiable
workload, uniform points, and batches of independent bounded NFW halos.  A case is one kind of call at one size:

  noalloc   volumes of a small set by the entry point that allocates nothing (latency)
  build     cells of one set and what a snapshot analysis takes from them: volumes, neighbour lists, densities,
            gradients, and, with G > 0, densities on a G^3 grid; with "adjoint", also the volume adjoint
  sets      many independent bounded halos of uneven sizes in one batched build
  autograd  forward and backward of a loss on the densities through torch.autograd
  rebuild   new positions in an existing handle (an optimisation or time step), volumes and moments
  products  everything an analysis asks of a handle it already has
  voxels    the exact volume-averaged grid and the weighted centroidal gradient of an existing handle
  owned     one rank's brick of a decomposed set: cells of its own particles, bounded by buffer particles
"""
import math

import numpy as np
import torch

from paper_1601_06429_gb300 import autograd
from paper_1601_06429_gb300 import binding as vt

# ---------------------------------------------------------------- the cases


def listed():
    return [
        # a small set inside a host loop that may not allocate: launches and synchronisation count
        {"name": "noalloc_1000", "kind": "noalloc", "n": 1000, "points": "uniform", "dtype": "f32", "periodic": True},
        # the smallest configuration, in FP64, with every output
        {"name": "uniform_4096_f64", "kind": "build", "n": 4096, "points": "uniform", "dtype": "f64",
         "precision": "filter32", "periodic": True, "G": 32, "adjoint": False},
        # the FP64-geometry clipper, for users who want volumes to 1e-6
        {"name": "clustered_30011_plain64", "kind": "build", "n": 30011, "points": "clustered", "dtype": "f32",
         "precision": "plain64", "periodic": True, "G": 0, "adjoint": False},
        # an ordinary sub-volume, ragged size
        {"name": "clustered_65537", "kind": "build", "n": 65537, "points": "clustered", "dtype": "f32",
         "precision": "filter32", "periodic": True, "G": 64, "adjoint": True},
        # a whole simulation box with all outputs and a 256^3 grid
        {"name": "clustered_2m", "kind": "build", "n": 2097152, "points": "clustered", "dtype": "f32",
         "precision": "filter32", "periodic": True, "G": 256, "adjoint": False},
        # the headline step: 256^3 particles, all outputs, grid and adjoint
        {"name": "clustered_16m", "kind": "build", "n": 16777216, "points": "clustered", "dtype": "f32",
         "precision": "filter32", "periodic": True, "G": 256, "adjoint": True},
        # independent halos of 64 to 65536 particles (a halo catalogue), one batched build
        {"name": "halo_sets_400", "kind": "sets", "sets": 400, "nmin": 64, "nmax": 65536, "dtype": "f32"},
        # a loss on the densities, differentiated with respect to the positions
        {"name": "autograd_1m", "kind": "autograd", "n": 1048576, "dtype": "f32"},
        # one step of an optimisation that keeps its handle
        {"name": "rebuild_200k", "kind": "rebuild", "n": 200003, "dtype": "f32"},
        # the per-particle products of a handle, each asked for once
        {"name": "products_1m", "kind": "products", "n": 1000003, "dtype": "f32"},
        # mass-conserving gridding (about one voxel per four particles) and the weighted energy gradient
        {"name": "voxels_128k", "kind": "voxels", "n": 131072, "dtype": "f32", "G": 32},
        # one rank of a decomposed snapshot: a third of its points are buffer particles
        {"name": "owned_300k", "kind": "owned", "n": 300007, "dtype": "f32"},
    ]


def draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["noalloc", "build", "build", "build", "sets", "autograd", "rebuild", "products", "voxels", "owned"])
    if kind == "noalloc":
        points = rng.choice(["uniform", "clustered"])
        # a clustered set this small has cells wider than a quarter of a periodic box: bounded
        return {"kind": kind, "n": size(600, 8192), "points": points, "dtype": rng.choice(["f32", "f64"]),
                "periodic": points == "uniform" and rng.random() < 0.7}
    if kind == "build":
        prec = rng.choice(["filter32", "filter32", "filter32", "plain64"])
        n = size(2000, 200000 if prec == "plain64" else 6000000)
        points = rng.choice(["clustered", "clustered", "uniform"])
        return {"kind": kind, "n": n, "points": points, "dtype": rng.choice(["f32", "f32", "f64"]), "precision": prec,
                "periodic": (points == "uniform" or n > 20000) and rng.random() < 0.75,
                "G": rng.choice([0, 24, 60, 128]), "adjoint": rng.random() < 0.5}
    if kind == "sets":
        return {"kind": kind, "sets": size(4, 500), "nmin": size(30, 200), "nmax": size(2000, 65536), "dtype": "f32"}
    if kind == "voxels":
        n = size(25000, 200000)
        return {"kind": kind, "n": n, "dtype": "f32", "G": int(n ** (1.0 / 3.0) * rng.uniform(0.3, 0.7))}
    lo, hi = {"autograd": (10000, 2000000), "rebuild": (10000, 2000000), "products": (25000, 3000000),
              "owned": (25000, 1500000)}[kind]
    return {"kind": kind, "n": size(lo, hi), "dtype": rng.choice(["f32", "f32", "f64"])}


# ---------------------------------------------------------------- point sets, on the GPU, from the seed


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _rand(g, *shape):
    return torch.rand(*shape, generator=g, device="cuda", dtype=torch.float64)


def _directions(g, n):
    v = torch.randn(n, 3, generator=g, device="cuda", dtype=torch.float64)
    return v / v.norm(dim=1, keepdim=True)


def _nfw_radii(g, conc):
    """r / r_vir of NFW profiles of concentration conc (one per point), by bisection of the enclosed mass."""
    def mass(x):
        return torch.log1p(x) - x / (1.0 + x)

    want = _rand(g, len(conc)) * mass(conc)
    lo, hi = torch.zeros_like(conc), conc.clone()
    for _ in range(40):
        mid = 0.5 * (lo + hi)
        below = mass(mid) < want
        lo, hi = torch.where(below, mid, lo), torch.where(below, hi, mid)
    return 0.5 * (lo + hi) / conc


def _halo_points(g, n, n_halo, L, nbar):
    """n points in n_halo NFW halos: masses from a power law of slope -1.9 over three decades, at least 20 points
    each, virial radii from an overdensity of 200."""
    n_halo = max(1, min(n_halo, n // 40))
    a = -0.9
    m = (1.0 + _rand(g, n_halo) * (1000.0 ** a - 1.0)) ** (1.0 / a)
    cnt = 20 + torch.floor(m / m.sum() * (n - 20 * n_halo)).long()
    cnt[torch.argmax(m)] += n - int(cnt.sum())
    hid = torch.repeat_interleave(torch.arange(n_halo, device="cuda"), cnt)
    conc = 5.0 + 10.0 * _rand(g, n_halo)
    rvir = (3.0 * cnt / (4.0 * math.pi * 200.0 * nbar)) ** (1.0 / 3.0)
    r = _nfw_radii(g, conc[hid]) * rvir[hid]
    return (_rand(g, n_halo, 3) * L)[hid] + r[:, None] * _directions(g, n)


def _filament_points(g, n, n_fil, L):
    """n points along n_fil straight filaments of length 5 to 20, Gaussian cross-section of width 0.5."""
    fid = torch.randint(n_fil, (n,), generator=g, device="cuda")
    length = 5.0 + 15.0 * _rand(g, n_fil)
    d = _directions(g, n_fil)[fid]
    off = torch.randn(n, 3, generator=g, device="cuda", dtype=torch.float64) * 0.5
    off -= (off * d).sum(1, keepdim=True) * d
    return (_rand(g, n_fil, 3) * L)[fid] + (_rand(g, n) * length[fid])[:, None] * d + off


def _distinct(x, lo, L, g):
    """x with the repeated positions replaced by uniform ones (two particles never share a position)."""
    for _ in range(20):
        b = (x.view(torch.int32).long() if x.dtype == torch.float32 else x.view(torch.int64))
        h = (b[:, 0] * 73856093) ^ (b[:, 1] * 19349669 + 7) ^ (b[:, 2] * 83492791 * 31)
        s, order = torch.sort(h)
        again = order[1:][s[1:] == s[:-1]]
        if not len(again):
            break
        x[again] = (lo + _rand(g, len(again), 3) * L).to(x.dtype)
    return x


def _points(case, seed, points, n, L):
    """[n, 3] points in the periodic box [0, L), in a random order."""
    g = _gen(seed)
    nbar = n / L ** 3
    share = min(1.0, n / 2097152.0)
    if points == "uniform":
        x = _rand(g, n, 3) * L
    elif points == "halo_mix":
        nh = int(0.3 * n)
        x = torch.cat([_halo_points(g, nh, max(1, round(2000 * share)), L, nbar), _rand(g, n - nh, 3) * L])
    else:
        nh, nf = int(0.6 * n), int(0.25 * n)
        x = torch.cat([_halo_points(g, nh, max(1, round(2000 * share)), L, nbar),
                       _filament_points(g, nf, max(1, round(1000 * share)), L),
                       _rand(g, n - nh - nf, 3) * L])
    x = x[torch.randperm(n, generator=g, device="cuda")]
    dt = torch.float32 if case["dtype"] == "f32" else torch.float64
    x = (x - L * torch.floor(x / L)).to(dt)
    x[x >= L] = 0
    return _distinct(x.contiguous(), 0.0, L, g)


def _box_side(n):
    """Side of a box of the reference density: 2,097,152 points in 100^3, representable in FP32."""
    return float(np.float32(100.0 * (n / 2097152.0) ** (1.0 / 3.0)))


def _halo_sets(case, seed):
    """Independent NFW halos of log-uniform sizes (the case's, whatever the seed), each in its own box [-1, 1]^3."""
    r = np.random.Generator(np.random.Philox(case["sets"]))
    sizes = np.floor(np.exp(r.uniform(np.log(case["nmin"]), np.log(case["nmax"]), case["sets"]))).astype(np.int64)
    off = np.concatenate([[0], np.cumsum(sizes)])
    g = _gen(seed)
    n = int(off[-1])
    sid = torch.repeat_interleave(torch.arange(case["sets"], device="cuda"), torch.from_numpy(sizes).cuda())
    conc = 5.0 + 10.0 * _rand(g, case["sets"])
    x = _nfw_radii(g, conc[sid])[:, None] * _directions(g, n)
    x = x.clamp(-1.0, 1.0).to(torch.float32).contiguous()
    # repeated positions: distinct over all sets, which is more than is needed
    return _distinct(x, -1.0, 2.0, g), off


# ---------------------------------------------------------------- one case: its state and one pass


def _csr_buffers(pos):
    """Room for volumes and neighbour lists, kept by the caller: 18 neighbours a particle (15.5 on average)."""
    n = len(pos)
    return (torch.zeros(n, dtype=pos.dtype, device="cuda"), torch.zeros(n + 1, dtype=torch.int64, device="cuda"),
            torch.zeros(18 * n, dtype=torch.int32, device="cuda"))


def prepare(case, seed):
    kind = case["kind"]
    s = {"kind": kind, "case": dict(case)}
    if kind == "sets":
        s["pos"], s["off"] = _halo_sets(case, seed)
        s["csr"] = _csr_buffers(s["pos"])
        s["boxes"] = np.tile(np.array([-1.0, -1.0, -1.0, 1.0, 1.0, 1.0]), (case["sets"], 1))
        return s
    n = case["n"]
    L = 1.0 if kind in ("autograd", "rebuild") or case.get("points") == "uniform" else _box_side(n)
    points = case.get("points") or ("halo_mix" if kind in ("autograd", "rebuild") else "clustered")
    s["L"] = L
    s["lo"], s["hi"] = (0.0, 0.0, 0.0), (L, L, L)
    pos = s["pos"] = _points(case, seed, points, n, L)
    g = _gen(seed + 1000003)
    s["w"] = torch.rand(n, generator=g, device="cuda", dtype=pos.dtype)
    if kind in ("build", "products", "owned"):
        s["csr"] = _csr_buffers(pos)
    if kind == "noalloc":
        s["vol"] = torch.empty(n, dtype=pos.dtype, device="cuda")
    elif kind == "rebuild":
        # the handle was built on other positions of the same particles
        s["h"] = vt.vt_build(_points(case, seed + 500009, points, n, L), None, s["lo"], s["hi"], True)
        s["vol"] = torch.empty(n, dtype=pos.dtype, device="cuda")
        s["cen"] = torch.empty(n, 3, dtype=pos.dtype, device="cuda")
        s["energy"] = torch.empty(n, dtype=pos.dtype, device="cuda")
    elif kind in ("products", "voxels"):
        s["mass"] = 0.5 + s["w"]
        s["h"] = vt.vt_build(pos, s["mass"], s["lo"], s["hi"], True)
    elif kind == "owned":
        # the brick is the part x < 2L/3; its own particles come first, the others are its buffer
        own = pos[:, 0] < 2.0 * L / 3.0
        s["pos"] = torch.cat([pos[own], pos[~own]]).contiguous()
        s["n_owned"] = int(own.sum())
    return s


def run(s):
    kind, case, pos = s["kind"], s["case"], s["pos"]
    if kind == "noalloc":
        vt.vt_volumes_noalloc(pos, s["lo"], s["hi"], case["periodic"], s["vol"])
        return {"vol": s["vol"]}
    if kind == "build":
        h = vt.vt_build(pos, None, s["lo"], s["hi"], case["periodic"], case["precision"])
        vol, off, ids = s["csr"]
        vt.vt_cells(h, vol, off, ids)
        out = {"vol": vol, "off": off, "ids": ids, "dens": vt.density(h), "grad": vt.gradient(h)}
        if case["G"]:
            out["grid"] = vt.grid_density(h, case["G"])
        if case["adjoint"]:
            out["adjoint"] = vt.backward(h, s["w"], 0.0)
        vt.vt_destroy(h)
        return out
    if kind == "sets":
        h = vt.vt_build_batched(pos, s["off"], s["boxes"])
        vol, off, ids = s["csr"]
        vt.vt_cells(h, vol, off, ids)
        out = {"vol": vol, "off": off, "ids": ids, "dens": vt.density(h)}
        vt.vt_destroy(h)
        return out
    if kind == "autograd":
        x = pos.detach().requires_grad_(True)
        vol, energy = autograd.cells(x, s["lo"], s["hi"])
        loss = (s["w"] * torch.log(1.0 / vol)).sum() + 0.5 * energy.sum()
        (grad,) = torch.autograd.grad(loss, x)
        return {"vol": vol.detach(), "energy": energy.detach(), "grad": grad}
    if kind == "rebuild":
        vt.vt_rebuild(s["h"], pos)
        vt.vt_cells(s["h"], s["vol"])
        vt.vt_moments(s["h"], s["cen"], s["energy"])
        return {"vol": s["vol"], "cen": s["cen"], "energy": s["energy"]}
    h = s.get("h")
    if kind == "products":
        vol, off, ids = s["csr"]
        vt.vt_cells(h, vol, off, ids)
        cen, energy = vt.moments(h)
        return {"vol": vol, "off": off, "ids": ids, "dens": vt.density(h), "grad": vt.gradient(h),
                "grad_gg": vt.gradient_gg(h), "cen": cen, "energy": energy, "adjoint": vt.backward(h, s["w"], 0.25),
                "radius": vt.cell_radius(h)}
    if kind == "voxels":
        return {"grid": vt.grid_density_volume(h, case["G"]), "weighted": vt.backward_weighted(h, s["w"])}
    h = vt.vt_build_owned(pos, s["n_owned"], None, s["lo"], s["hi"], True)
    vol, off, ids = s["csr"]
    vt.vt_cells(h, vol, off, ids)
    out = {"vol": vol, "off": off, "ids": ids, "dens": vt.density(h), "radius": vt.cell_radius(h)}
    vt.vt_destroy(h)
    return out


def work(case):
    """Bytes read and written once, and the clipping's arithmetic: per cell about 163 sites examined against 26.7
    vertices (6 flops each), 40 flops a vertex and 30 a facet, 27.7 kflop in all; 15.4 neighbours a cell."""
    kind = case["kind"]
    if kind == "sets":
        span = math.log(case["nmax"] / case["nmin"]) if case["nmax"] > case["nmin"] else 1.0
        n = case["sets"] * (case["nmax"] - case["nmin"]) / span
    else:
        n = case["n"]
    b = 4 if case["dtype"] == "f32" else 8
    clip, facets = 27700.0 * n, 15.4 * n
    if kind == "noalloc":
        return {"bytes": 4 * b * n, "flops": clip}
    if kind == "build":
        return {"bytes": n * (8 * b + 8) + 4 * facets + b * case["G"] ** 3 + (4 * b * n if case["adjoint"] else 0),
                "flops": clip}
    if kind == "sets":
        return {"bytes": n * (5 * b + 8) + 4 * facets, "flops": clip}
    if kind == "autograd":
        return {"bytes": n * 9 * b, "flops": clip}
    if kind == "rebuild":
        return {"bytes": n * 8 * b, "flops": clip}
    if kind == "products":
        return {"bytes": n * (19 * b + 8 + 40) + (32 + 4) * facets, "flops": 60.0 * facets}
    if kind == "voxels":
        return {"bytes": n * (4 * b + 40) + 32 * facets + b * case["G"] ** 3, "flops": 2 * 4000.0 * n}
    return {"bytes": n * (6 * b + 8) + 4 * facets * 2 / 3, "flops": clip * 2 / 3}


# ---------------------------------------------------------------- the same in 64 bits, for small sets


def _cells64(x, L, periodic, most=640):
    """Voronoi cells of x [n, 3] (float64, box [0, L)) by clipping every cell with its neighbours' bisectors in order
    of distance, all cells in step: (volume [n], cell, neighbour, displacement of every facet); None if `most`
    nearest neighbours do not bound a cell."""
    n, dev, T = len(x), x.device, 96
    m = min(most, n - 1)
    disp = torch.empty(n, m, 3, dtype=torch.float64, device=dev)
    nbr = torch.empty(n, m, dtype=torch.long, device=dev)
    for a in range(0, n, 1024):
        d = x[None, :, :] - x[a:a + 1024, None, :]
        if periodic:
            d = d - L * torch.round(d / L)
        d2 = (d * d).sum(-1)
        d2[torch.arange(len(d2), device=dev), torch.arange(a, a + len(d2), device=dev)] = math.inf
        _, k = torch.topk(d2, m, dim=1, largest=False)
        nbr[a:a + 1024] = k
        disp[a:a + 1024] = torch.gather(d, 1, k[:, :, None].expand(-1, -1, 3))
    # planes n.y <= h: six walls, then the bisectors
    P = torch.zeros(n, m + 6, 4, dtype=torch.float64, device=dev)
    for w in range(6):
        P[:, w, w // 2] = 1.0 if w % 2 == 0 else -1.0
        P[:, w, 3] = 0.5 * L if periodic else (L - x[:, w // 2] if w % 2 == 0 else x[:, w // 2])
    P[:, 6:, :3] = disp
    P[:, 6:, 3] = 0.5 * (disp * disp).sum(-1)

    def vertex(c, t):
        A = P[c[:, None], t.reshape(len(c), -1)].reshape(len(c), -1, 3, 4)
        na, nb, nc = A[:, :, 0, :3], A[:, :, 1, :3], A[:, :, 2, :3]
        bc, ca, ab = torch.linalg.cross(nb, nc), torch.linalg.cross(nc, na), torch.linalg.cross(na, nb)
        det = (na * bc).sum(-1, keepdim=True)
        det = torch.where(det == 0, torch.full_like(det, 1e-300), det)
        return (A[:, :, 0, 3:] * bc + A[:, :, 1, 3:] * ca + A[:, :, 2, 3:] * ab) / det

    tri = torch.zeros(n, T, 3, dtype=torch.long, device=dev)
    live = torch.zeros(n, T, dtype=torch.bool, device=dev)
    for k in range(8):
        X, Y, Z = k & 1, 2 + ((k >> 1) & 1), 4 + ((k >> 2) & 1)
        flip = bin(k).count("1") % 2 == 1
        tri[:, k] = torch.tensor([X, Z, Y] if flip else [X, Y, Z], device=dev)
        live[:, k] = True
    every = torch.arange(n, device=dev)
    V = vertex(every, tri)
    for k in range(6, m + 6):
        R2 = torch.where(live, (V * V).sum(-1), torch.zeros((), dtype=torch.float64, device=dev)).amax(1)
        act = torch.nonzero(2.0 * P[:, k, 3] < 4.0 * R2).flatten()
        if not len(act):
            break
        out = ((V[act] * P[act, k, None, :3]).sum(-1) > P[act, k, 3:]) & live[act]
        hit = out.any(1)
        c, out = act[hit], out[hit]
        if not len(c):
            continue
        r = int(out.sum(1).amax())
        first = torch.argsort((~out).to(torch.int8), dim=1, stable=True)[:, :r]
        gone = torch.gather(out, 1, first)
        t = torch.gather(tri[c], 1, first[:, :, None].expand(-1, -1, 3))
        e0 = t.reshape(len(c), -1)
        e1 = t.roll(-1, dims=2).reshape(len(c), -1)
        ok = gone[:, :, None].expand(-1, -1, 3).reshape(len(c), -1)
        code = torch.where(ok, e0 * 4096 + e1, torch.full_like(e0, -1))
        back = torch.where(ok, e1 * 4096 + e0, torch.full_like(e0, -2))
        edge = ok & ~(code[:, :, None] == back[:, None, :]).any(2)
        b = int(edge.sum(1).amax())
        pick = torch.argsort((~edge).to(torch.int8), dim=1, stable=True)[:, :b]
        new = torch.stack([torch.gather(e0, 1, pick), torch.gather(e1, 1, pick), torch.full_like(pick, k)], -1)
        isnew = torch.gather(edge, 1, pick)
        live[c] &= ~out
        free = torch.argsort(live[c].to(torch.int8), dim=1, stable=True)[:, :b]
        if bool((torch.gather(live[c], 1, free) & isnew).any()):
            return None
        vn = vertex(c, new)
        row, col = torch.nonzero(isnew, as_tuple=True)
        slot = free[row, col]
        tri[c[row], slot] = new[row, col]
        V[c[row], slot] = vn[row, col]
        live[c[row], slot] = True
    else:
        R2 = torch.where(live, (V * V).sum(-1), torch.zeros((), dtype=torch.float64, device=dev)).amax(1)
        if m < n - 1 and bool((2.0 * P[:, -1, 3] < 4.0 * R2).any()):
            return None
    # facets: the vertices of each (cell, plane), in order around it
    ci, ti = torch.nonzero(live, as_tuple=True)
    cell = ci.repeat_interleave(3)
    plane = tri[ci, ti].reshape(-1)
    v = V[ci, ti].repeat_interleave(3, dim=0)
    nrm = P[cell, plane, :3]
    nrm = nrm / nrm.norm(dim=1, keepdim=True)
    key = cell * (m + 6) + plane
    uniq, seg = torch.unique(key, return_inverse=True)
    cnt = torch.bincount(seg, minlength=len(uniq)).to(torch.float64)
    cen = torch.zeros(len(uniq), 3, dtype=torch.float64, device=dev).index_add_(0, seg, v) / cnt[:, None]
    q = v - cen[seg]
    ax = torch.where((nrm[:, :1].abs() < 0.6), torch.tensor([[1.0, 0, 0]], dtype=torch.float64, device=dev),
                     torch.tensor([[0, 1.0, 0]], dtype=torch.float64, device=dev))
    u1 = torch.linalg.cross(nrm, ax)
    u1 = u1 / u1.norm(dim=1, keepdim=True)
    u2 = torch.linalg.cross(nrm, u1)
    a, b = (q * u1).sum(1), (q * u2).sum(1)
    o = torch.argsort(torch.atan2(b, a))
    o = o[torch.argsort(seg[o], stable=True)]
    seg, a, b, cell, plane = seg[o], a[o], b[o], cell[o], plane[o]
    start = torch.cat([torch.tensor([0], device=dev), torch.nonzero(seg[1:] != seg[:-1]).flatten() + 1])
    nxt = torch.arange(1, len(seg) + 1, device=dev)
    nxt[torch.cat([start[1:], torch.tensor([len(seg)], device=dev)]) - 1] = start
    area = torch.zeros(len(uniq), dtype=torch.float64, device=dev).index_add_(0, seg, 0.5 * (a * b[nxt] - a[nxt] * b))
    fc, fp = uniq // (m + 6), uniq % (m + 6)
    dist = P[fc, fp, 3] / P[fc, fp, :3].norm(dim=1)
    vol = torch.zeros(n, dtype=torch.float64, device=dev).index_add_(0, fc, dist * area / 3.0)
    real = fp >= 6
    return vol, fc[real], nbr[fc[real], fp[real] - 6], P[fc[real], fp[real], :3]


def exact(case, seed):
    if case["kind"] not in ("noalloc", "build") or case["n"] > 6000:
        return None
    s = prepare(case, seed)
    x, L = s["pos"].double(), s["L"]
    got = _cells64(x, L, case["periodic"])
    if got is None:
        return None
    vol, i, j, d = got
    if case["kind"] == "noalloc":
        return {"vol": vol}
    dens = 1.0 / vol
    M = torch.zeros(len(x), 3, 3, dtype=torch.float64, device=x.device)
    M.index_add_(0, i, d[:, :, None] * d[:, None, :])
    rhs = torch.zeros(len(x), 3, dtype=torch.float64, device=x.device).index_add_(0, i, d * (dens[j] - dens[i])[:, None])
    out = {"vol": vol, "off": None, "ids": None, "dens": dens, "grad": torch.linalg.solve(M, rhs)}
    G = case["G"]
    if G:
        c = (torch.arange(G, device=x.device, dtype=torch.float64) + 0.5) * (L / G)
        grid = torch.empty(G, G, G, dtype=torch.float64, device=x.device)
        for a in range(G):
            q = torch.stack([c[None, :].expand(G, G), c[:, None].expand(G, G), c[a].expand(G, G)], -1).reshape(-1, 3)
            best = torch.empty(len(q), dtype=torch.long, device=x.device)
            for k in range(0, len(q), 1024):
                e = x[None] - q[k:k + 1024, None]
                if case["periodic"]:
                    e = e - L * torch.round(e / L)
                best[k:k + 1024] = (e * e).sum(-1).argmin(1)
            grid[a] = dens[best].reshape(G, G)
        out["grid"] = grid
    if case["adjoint"]:
        out["adjoint"] = None
    return out
