"""The work that users of this library have it do, as cases that can be timed.

A case is a plain dict; ``prepare`` makes what a program holds before the call
(meshes, start coordinates, batches, a server), ``run`` is one pass through the
public entry points and returns the results, ``work`` says what the pass cannot
do without, and ``exact`` computes the results with plain torch in FP64.

Kinds of case:

* ``steady``: a mesh is created once and smoothed again and again: new start
  coordinates in, passes, coordinates out (all on the device);
* ``oneshot``: one request from host arrays: create, smooth, coordinates back
  to host memory, destroy;
* ``batch``: many meshes of uneven size, one ``Batch`` call;
* ``serve``: a burst of requests to a running ``Server``;
* ``histogram``: the quality histogram of a mesh.

The grids are those of ``meshgen`` (random diagonals, interior jitter, outer
ring fixed, optionally clustered towards seeded centres; Morton or random
numbering), made on the GPU because the numpy construction takes minutes at
the largest size; the Delaunay meshes come from ``meshgen`` itself.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import meshgen
import paper_1502_00355_gb300 as sls

DEV = "cuda"
OPTIONS = ("layout", "copy_back", "strict", "record_accept", "form", "precision", "skip_unchanged")
DEFAULTS = {"mesh": "grid", "jitter": 0.35, "pull": 0.0, "numbering": "morton", "tol": 0.0}


def listed():
    return [
        # the paper's small mesh: 4,096 nodes, where a pass is mostly launch and latency
        {"name": "small_64", "kind": "steady", "nx": 64, "ny": 64, "jitter": 0.3, "passes": 10},
        # the paper's own largest mesh, 100,000 Delaunay points, smoothed to the tolerance
        {"name": "delaunay_100k", "kind": "steady", "mesh": "delaunay", "n": 100000, "passes": 200, "tol": 1e-9,
         "expect": 88},
        # a mesh as it comes out of a mesher that does not order its nodes, odd sizes, separate x and y
        # arrays, decisions wanted
        {"name": "random_1009x701_soa", "kind": "steady", "nx": 1009, "ny": 701, "numbering": "random",
         "layout": "soa", "record_accept": True, "passes": 50},
        # the medium configuration: 1024 x 1024, 100 passes
        {"name": "medium_1024", "kind": "steady", "nx": 1024, "ny": 1024, "passes": 100},
        # the benchmark: 4096 x 4096, clustered, to the tolerance
        {"name": "large_4096", "kind": "steady", "nx": 4096, "ny": 4096, "pull": 0.05, "passes": 200, "tol": 1e-9,
         "expect": 77},
        # Form B (in place, coloured), which users take because it needs fewer sweeps
        {"name": "form_b_1500x1100", "kind": "steady", "nx": 1500, "ny": 1100, "pull": 0.05, "form": "B",
         "passes": 200, "tol": 1e-9, "expect": 38},
        # the paper's precision
        {"name": "binary32_2048", "kind": "steady", "nx": 2048, "ny": 2048, "precision": 32, "passes": 50},
        # one small request from start to end: a mesh of a few thousand nodes, smoothed once and thrown away
        {"name": "oneshot_150x111", "kind": "oneshot", "nx": 150, "ny": 111, "passes": 20},
        # one large request from pinned host arrays (how the end-to-end benchmark feeds the library)
        {"name": "oneshot_2048", "kind": "oneshot", "nx": 2048, "ny": 2048, "pull": 0.05, "pinned": True,
         "passes": 200, "tol": 1e-9, "expect": 76},
        # the batched workload's distribution (1K to 256K nodes, 10 to 100 passes each), 48 meshes
        {"name": "batch_48", "kind": "batch", "count": 48, "lo": 1024, "hi": 262144, "jitter": 0.3,
         "lo_passes": 10, "hi_passes": 100},
        # a burst of served requests, 1K to 256K nodes, caps 10 to 200, tolerance on
        {"name": "serve_24", "kind": "serve", "count": 24, "lo": 1024, "hi": 262144, "jitter": 0.3,
         "lo_passes": 10, "hi_passes": 200, "tol": 1e-9},
        # mesh quality report before and after smoothing
        {"name": "histogram_2048", "kind": "histogram", "nx": 2048, "ny": 2048, "pull": 0.05, "bins": 20},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_grid(rng, lo, hi):
    n = _log_int(rng, lo, hi)
    ny = max(3, int(round(math.sqrt(n / rng.uniform(1.0, 4.0)))))
    return {"nx": max(3, int(round(n / ny))), "ny": ny}


def draw(rng):
    kind = rng.choice(["steady", "steady", "steady", "oneshot", "batch", "serve", "histogram"])
    if kind in ("batch", "serve"):
        hi = _log_int(rng, 16384, 262144)
        c = {"kind": kind, "count": rng.randint(5, 40), "lo": 1024, "hi": hi, "jitter": 0.3,
             "lo_passes": 10, "hi_passes": rng.randint(20, 150), "tol": rng.choice([0.0, 1e-9])}
        return c
    if kind == "histogram":
        return {"kind": kind, **_draw_grid(rng, 4000, 8000000), "pull": rng.choice([0.0, 0.05]),
                "bins": rng.choice([10, 20, 33, 256])}
    if kind == "oneshot":
        c = {"kind": kind, **_draw_grid(rng, 1000, 4000000), "passes": _log_int(rng, 5, 100),
             "numbering": rng.choice(["morton", "morton", "random"]), "pinned": rng.random() < 0.5}
        return c
    c = {"kind": kind, "passes": _log_int(rng, 5, 100)}
    if rng.random() < 0.25:
        c.update({"mesh": "delaunay", "n": _log_int(rng, 1000, 100000)})
    else:
        c.update({**_draw_grid(rng, 1000, 6000000), "jitter": rng.choice([0.3, 0.35]),
                  "pull": rng.choice([0.0, 0.05])})
    c["numbering"] = rng.choice(["morton", "morton", "random"])
    if rng.random() < 0.3:
        c["tol"] = rng.choice([1e-9, 1e-4])
        c["passes"] = max(c["passes"], 20)
    option = rng.choice(["", "", "", "layout", "copy_back", "strict", "accept", "form", "precision", "skip", "noalloc"])
    if option == "layout":
        c["layout"] = "soa"
    elif option == "accept":
        c["record_accept"] = True
    elif option == "form":
        c["form"] = "B"
    elif option == "precision":
        c["precision"] = 32
    elif option == "skip":
        c["skip_unchanged"] = True
    elif option == "noalloc":
        c["noalloc"] = True
    elif option:
        c[option] = True
    return c


# --- inputs -----------------------------------------------------------------

def _interleave(v):
    for s, m in ((16, 0x0000FFFF0000FFFF), (8, 0x00FF00FF00FF00FF), (4, 0x0F0F0F0F0F0F0F0F),
                 (2, 0x3333333333333333), (1, 0x5555555555555555)):
        v = (v | (v << s)) & m
    return v


def _grid(nx, ny, jitter, pull, numbering, seed):
    """(xy float64 (n, 2), tri int32 (m, 3), boundary uint8 (n,)) on the GPU."""
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    h = 1.0 / (ny - 1)
    j, i = torch.meshgrid(torch.arange(ny, device=DEV), torch.arange(nx, device=DEV), indexing="ij")
    i, j = i.reshape(-1), j.reshape(-1)
    n = nx * ny
    fixed = (i == 0) | (i == nx - 1) | (j == 0) | (j == ny - 1)
    free = ~fixed
    xy = torch.stack([i.double() * h, j.double() * h], 1)
    noise = (torch.rand(n, 2, dtype=torch.float64, device=DEV, generator=g) * 2.0 - 1.0) * (jitter * h)
    xy = torch.where(free[:, None], xy + noise, xy)
    if pull > 0.0:
        # a share of the interior nodes moves towards the nearest of 1,024 centres, by at most 2h
        inner = free.nonzero()[:, 0]
        k = int(round(pull * inner.numel()))
        chosen = inner[torch.rand(inner.numel(), device=DEV, generator=g).argsort(stable=True)[:k]]
        scale = torch.tensor([(nx - 1) * h, (ny - 1) * h], dtype=torch.float64, device=DEV)
        centres = torch.rand(1024, 2, dtype=torch.float64, device=DEV, generator=g) * scale
        lam = torch.rand(k, 1, dtype=torch.float64, device=DEV, generator=g) * 0.5 + 0.25
        for at in range(0, k, 65536):
            p = xy[chosen[at:at + 65536]]
            near = ((p[:, None, 0] - centres[None, :, 0]) ** 2 + (p[:, None, 1] - centres[None, :, 1]) ** 2).argmin(1)
            step = lam[at:at + 65536] * (centres[near] - p)
            length = step.square().sum(1, keepdim=True).sqrt()
            xy[chosen[at:at + 65536]] = p + step * torch.where(length > 2 * h, 2 * h / length.clamp_min(1e-300), 1.0)
    if numbering == "random":
        rank = torch.rand(n, dtype=torch.float64, device=DEV, generator=g).argsort(stable=True).argsort()
    else:
        rank = (_interleave(i) | (_interleave(j) << 1)).argsort(stable=True).argsort()
    diag = torch.rand((nx - 1) * (ny - 1), device=DEV, generator=g) < 0.5
    qj, qi = torch.meshgrid(torch.arange(ny - 1, device=DEV), torch.arange(nx - 1, device=DEV), indexing="ij")
    v00 = (qj * nx + qi).reshape(-1)
    v10, v01, v11 = v00 + 1, v00 + nx, v00 + nx + 1
    tri = torch.stack([v00, v10, torch.where(diag, v01, v11), torch.where(diag, v10, v00), v11, v01], 1).reshape(-1, 3)
    out = torch.empty_like(xy)
    out[rank] = xy
    boundary = torch.empty(n, dtype=torch.uint8, device=DEV)
    boundary[rank] = fixed.to(torch.uint8)
    return out, rank[tri].to(torch.int32), boundary


def _inputs(case, seed):
    c = {**DEFAULTS, **case}
    if c["mesh"] == "delaunay":
        m = meshgen.delaunay_random(c["n"], seed, numbering=c["numbering"])
        return torch.from_numpy(m.xy).to(DEV), torch.from_numpy(m.tri).to(DEV), torch.from_numpy(m.boundary).to(DEV)
    return _grid(c["nx"], c["ny"], c["jitter"], c["pull"], c["numbering"], seed)


def _specs(case, seed):
    """Per mesh of a batch or a burst: (nx, ny, passes, seed).  The sizes and
    passes belong to the case, the coordinates and diagonals to the seed."""
    rng = np.random.default_rng([case["count"], case["lo"], case["hi"], case["hi_passes"]])
    out = []
    for k in range(case["count"]):
        n = math.exp(rng.uniform(math.log(case["lo"]), math.log(case["hi"])))
        ny = max(3, int(round(math.sqrt(n / rng.uniform(1.0, 4.0)))))
        out.append((max(3, int(round(n / ny))), ny, int(rng.integers(case["lo_passes"], case["hi_passes"] + 1)),
                    seed * 1000 + k))
    return out


def _many(case, seed):
    return [(_grid(nx, ny, case["jitter"], 0.0, "morton", s), passes) for nx, ny, passes, s in _specs(case, seed)]


def _host(t, pinned=False):
    return (t.cpu().pin_memory() if pinned else t.cpu()).numpy()


def _options(case):
    return {k: case[k] for k in OPTIONS if k in case}


# --- one pass ---------------------------------------------------------------

def prepare(case, seed):
    kind = case["kind"]
    s = {"case": case, "kind": kind}
    if kind == "batch":
        s["meshes"], s["passes"] = [], []
        for (xy, tri, boundary), passes in _many(case, seed):
            s["meshes"].append(sls.Mesh(_host(xy), _host(tri), _host(boundary), numbering="grouped"))
            s["passes"].append(passes)
        s["batch"] = sls.Batch(s["meshes"], s["passes"], [case.get("tol", 0.0)] * len(s["meshes"]))
        return s
    if kind == "serve":
        s["requests"] = [(_host(xy), _host(tri), _host(boundary), passes)
                         for (xy, tri, boundary), passes in _many(case, seed)]
        s["server"] = sls.Server()
        return s
    xy, tri, boundary = _inputs(case, seed)
    if kind == "oneshot":
        pinned = bool(case.get("pinned"))
        s["args"] = (_host(xy, pinned), _host(tri, pinned), _host(boundary, pinned))
        s["out"] = _host(torch.empty_like(xy), pinned)
        return s
    s["mesh"] = sls.Mesh(_host(xy), _host(tri), _host(boundary), **_options(case))
    if kind == "steady":
        s["start"] = xy
        if case.get("noalloc"):
            s["work"], s["out"] = torch.empty_like(xy), torch.empty_like(xy)
    return s


def _numbers(infos):
    """Per mesh: iterations, accepted nodes of the last pass, whether the
    tolerance stopped it; and the largest squared move of the last pass."""
    return (np.array([[i["iterations"], i["accepted_last"], i["converged"]] for i in infos], np.int64),
            np.array([i["maxd2_last"] for i in infos]))


def run(s):
    case, kind = s["case"], s["kind"]
    tol = case.get("tol", 0.0)
    if kind == "steady":
        mesh = s["mesh"]
        if case.get("noalloc"):
            s["work"].copy_(s["start"])
            torch.cuda.current_stream().synchronize()  # the call reads its buffers on the mesh's stream
            info = mesh.smooth_noalloc(s["work"], s["out"], case["passes"], tol)
            return (s["out"], *_numbers([info]))
        mesh.set_coords(s["start"])
        info = mesh.smooth(case["passes"], tol)
        out = (mesh.coords_device(), *_numbers([info]))
        return out + (mesh.accept_mask(),) if case.get("record_accept") else out
    if kind == "oneshot":
        with sls.Mesh(*s["args"]) as mesh:
            info = mesh.smooth(case["passes"], tol)
            return (mesh.coords(s["out"]), *_numbers([info]))
    if kind == "batch":
        s["batch"].reset()
        infos = s["batch"].smooth()
        return ([m.coords_device() for m in s["meshes"]], *_numbers(infos))
    if kind == "serve":
        server = s["server"]
        jobs = [server.submit(xy, tri, boundary, passes, tol) for xy, tri, boundary, passes in s["requests"]]
        done = [server.wait(j) for j in jobs]
        return ([d[0] for d in done], *_numbers([d[1] for d in done]))
    counts, qmin, qmean = s["mesh"].histogram(case["bins"])
    return counts, qmin, qmean


# --- what a pass cannot do without --------------------------------------------

def work(case):
    """Per node-update: its coordinates read and written, its neighbour ids
    (six on average) read; per triangle evaluation (two of each of a node's six
    triangles) about 30 operations, and 17 for the centre and the move.  Each
    call besides: coordinates in and out; one-shot calls: the triangles too,
    read once and turned into the neighbour lists."""
    kind = case["kind"]

    def passes_of(cap):
        return min(cap, case.get("expect", 60)) if case.get("tol", 0.0) > 0.0 else cap

    if kind in ("batch", "serve"):
        todo = [(nx * ny, passes_of(p)) for nx, ny, p, _ in _specs(case, 0)]
    elif kind == "histogram":
        n = case["nx"] * case["ny"]
        return {"bytes": n * 16 + 2 * n * 12, "flops": 2 * n * 32}
    else:
        todo = [(case["n"] if case.get("mesh") == "delaunay" else case["nx"] * case["ny"], passes_of(case["passes"]))]
    width = 4 if case.get("precision") == 32 else 8
    call = 32 + (24 + 28 if kind in ("oneshot", "serve") else 0)
    return {"bytes": sum(n * (p * (4 * width + 24) + call) for n, p in todo),
            "flops": sum(n * p * 377 for n, p in todo)}


# --- the same results in plain torch, FP64 -------------------------------------

def _rank_in_row(row, n):
    """Position of every entry within its run of equal, ascending row values; and the runs' lengths."""
    count = torch.bincount(row, minlength=n)
    start = torch.cumsum(count, 0) - count
    return torch.arange(row.numel(), device=row.device) - start[row], count


class _Exact:
    """Smart Laplacian smoothing with separate FP64 torch operations: the
    neighbours summed in ascending (x, y, id) of the start coordinates."""

    def __init__(self, xy, tri, boundary):
        self.n, self.tri = xy.shape[0], tri.long()
        a, b, c = self.tri.unbind(1)
        key = torch.cat([a, b, b, c, c, a]) * self.n + torch.cat([b, a, c, b, a, c])
        key = torch.unique(key)
        i, j = self._order(xy, key)
        at, self.deg = _rank_in_row(i, self.n)
        self.nb = torch.zeros(int(self.deg.max()), self.n, dtype=torch.int64, device=xy.device)
        self.nb[at, i] = j
        corner = self.tri.reshape(-1)
        o = corner.argsort(stable=True)
        at, self.ntri = _rank_in_row(corner[o], self.n)
        self.inc = torch.zeros(int(self.ntri.max()), self.n, dtype=torch.int64, device=xy.device)
        self.inc[at, corner[o]] = o // 3
        self.free = (boundary == 0) & (self.ntri > 0)
        ext = xy.max(0).values - xy.min(0).values
        self.diag = math.sqrt(float(ext[0]) * float(ext[0]) + float(ext[1]) * float(ext[1]))

    def _order(self, xy, key):
        i, j = key // self.n, key % self.n
        for column in (1, 0):  # ids are ascending already; stable sorts by y, then x, then node
            o = xy[j, column].argsort(stable=True)
            i, j = i[o], j[o]
        o = i.argsort(stable=True)
        return i[o], j[o]

    @staticmethod
    def alpha(p, q, r):
        e1, e2, e3 = q - p, r - p, r - q
        cross = e1[:, 0] * e2[:, 1] - e1[:, 1] * e2[:, 0]
        l1 = e1[:, 0] * e1[:, 0] + e1[:, 1] * e1[:, 1]
        l2 = e2[:, 0] * e2[:, 0] + e2[:, 1] * e2[:, 1]
        l3 = e3[:, 0] * e3[:, 0] + e3[:, 1] * e3[:, 1]
        s = (l1 + l2) + l3
        return torch.where(s > 0.0, cross * 3.4641016151377544 / torch.where(s > 0.0, s, 1.0), 0.0)

    def update(self, x, nodes, strict):
        """(new coordinates, accepted, squared move) of the listed nodes."""
        deg, ntri = self.deg[nodes], self.ntri[nodes]
        c = x[self.nb[0, nodes]]
        for k in range(1, self.nb.shape[0]):
            c = torch.where((k < deg)[:, None], c + x[self.nb[k, nodes]], c)
        c = c / deg[:, None].double()
        p = x[nodes]
        old, new = None, None
        for k in range(self.inc.shape[0]):
            v = self.tri[self.inc[k, nodes]]
            q = [x[v[:, s]] for s in range(3)]
            a_old = self.alpha(*q)
            a_new = self.alpha(*[torch.where((v[:, s] == nodes)[:, None], c, q[s]) for s in range(3)])
            on = k < ntri
            old = a_old if old is None else torch.where(on, torch.minimum(old, a_old), old)
            new = a_new if new is None else torch.where(on, torch.minimum(new, a_new), new)
        ok = new > old if strict else new >= old
        d = c - p
        d2 = d[:, 0] * d[:, 0] + d[:, 1] * d[:, 1]
        return torch.where(ok[:, None], c, p), ok, torch.where(ok, d2, 0.0)

    def colours(self):
        """Jones-Plassmann classes: priority splitmix64(150200355 + id), ties by id."""
        def shr(v, k):
            return (v >> k) & ((1 << (64 - k)) - 1)

        def signed(v):
            return v - (1 << 64) if v >= 1 << 63 else v

        z = torch.arange(self.n, device=self.deg.device) + 150200355 + signed(0x9E3779B97F4A7C15)
        z = (z ^ shr(z, 30)) * signed(0xBF58476D1CE4E5B9)
        z = (z ^ shr(z, 27)) * signed(0x94D049BB133111EB)
        z = (z ^ shr(z, 31)) ^ signed(1 << 63)  # signed comparisons now order as unsigned ones
        colour = torch.where(self.free, -1, -2)
        ids = torch.arange(self.n, device=z.device)
        while bool((colour == -1).any()):
            left = (colour == -1).nonzero()[:, 0]
            win = torch.ones_like(left, dtype=torch.bool)
            used = torch.zeros_like(left)
            for k in range(self.nb.shape[0]):
                j = self.nb[k, left]
                on, cj = k < self.deg[left], colour[j]
                beaten = (z[j] > z[left]) | ((z[j] == z[left]) & (ids[j] > left))
                win &= ~(on & (cj == -1) & beaten)
                used |= torch.where(on & (cj >= 0), torch.ones_like(used) << cj.clamp_min(0), 0)
            pick = torch.zeros_like(left)
            for k in range(62, -1, -1):
                pick = torch.where((used >> k) & 1 == 0, k, pick)
            colour[left[win]] = pick[win]
        return [(colour == k).nonzero()[:, 0] for k in range(int(colour.max()) + 1)]

    def smooth(self, x, passes, tol, form="A", strict=False):
        classes = self.colours() if form == "B" else [self.free.nonzero()[:, 0]]
        t = tol * self.diag
        mask = torch.zeros(self.n, dtype=torch.uint8, device=x.device)
        x = x.clone()
        done, accepted, largest, stopped = 0, 0, 0.0, 0
        while done < passes and not stopped:
            accepted, largest = 0, 0.0
            for nodes in classes:
                if nodes.numel() == 0:
                    continue
                got, ok, d2 = self.update(x, nodes, strict)
                x[nodes] = got
                mask[nodes] = ok.to(torch.uint8)
                accepted += int(ok.sum())
                largest = max(largest, float(d2.max()))
            done += 1
            stopped = int(tol > 0.0 and largest < t * t)
        return x, [done, accepted, stopped], largest, mask


def exact(case, seed):
    kind = case["kind"]
    tol = case.get("tol", 0.0)
    if kind in ("batch", "serve"):
        got = [_Exact(*inputs).smooth(inputs[0], passes, tol) for inputs, passes in _many(case, seed)]
        return [g[0] for g in got], np.array([g[1] for g in got], np.int64), np.array([g[2] for g in got])
    xy, tri, boundary = _inputs(case, seed)
    if kind == "histogram":
        q = _Exact.alpha(*[xy[tri[:, k].long()] for k in range(3)])
        bins = ((q + 1.0) / 2.0 * case["bins"]).floor().clamp(0, case["bins"] - 1).long()
        return torch.bincount(bins, minlength=case["bins"]), float(q.min()), float(q.mean())
    if case.get("precision") == 32:
        xy = xy.float().double()  # the coordinates that such a mesh holds
    x, numbers, largest, mask = _Exact(xy, tri, boundary).smooth(xy, case["passes"], tol, case.get("form", "A"),
                                                                 bool(case.get("strict")))
    if case.get("precision") == 32:
        # a different computation: only the coordinates have a 64-bit counterpart
        return x, None, None
    out = (x, np.array([numbers], np.int64), np.array([largest]))
    return out + (mask,) if case.get("record_accept") else out
