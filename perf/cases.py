"""Timed cases of the irradiance library: what a planner has it do, through the public calls.

Every case works on a room made from its sizes and a seed: an axis-aligned shell with furniture boxes,
meshed in cells of edge `h` (two triangles each, in Z-order, tangentially jittered), as the rooms of the
tests and the benchmark are.  The sizes fix the number of triangles; the seed moves the furniture, the
jitter, the candidate positions, the dwell times and the lamp power.

    kind      one pass
    matrix    the irradiance matrix of one room for one lamp (with visibility words where `vis`)
    batch     several rooms x lamp designs in one persistent launch
    fluence   the fluence of every patch for `nvec` dwell-time vectors, and its covered fraction
    streamed  the same fluence without storing the matrix
    plan      a changed room from the start: build, matrix, fluence, coverage
    area      the patch-mean irradiance (solid angles)
    raster    the visibility-cube estimator at `R` pixels a face edge
    propose   the learned proposal: features, scores, and the selection of the kept candidates
    train     four training steps of the scorer, and the gradients of the last
"""
import functools
import math

import numpy as np
import torch

import paper_2103_14137_gb300 as uvc
from paper_2103_14137_gb300 import proposal

HEIGHT = 3.0              # rooms are 3 m high
MU_MIN = 100.0            # J/m^2
KEEP = 0.2                # kept fraction of the proposal
EXACT_TESTS = 4e9         # segment-triangle tests that exact() may make by brute force


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------

def listed():
    """Twelve cases over the sizes of the tests (988 triangles) to the large floors (hundreds of thousands)."""
    return [
        # the smallest call: one point lamp in a small room, all patches, where launches and latency count
        dict(name="tiny_matrix", kind="matrix", layout="ward", W=4.0, D=4.0, h=0.42, beds=1, patch="tri", np=0,
             nc=200, lamp="point", K=1, vis=True),
        # the headline: a hospital ward with a vertical line lamp, every patch against every candidate
        dict(name="ward_matrix", kind="matrix", layout="ward", W=10.0, D=8.0, h=0.1165, beds=6, patch="split", np=0,
             nc=2000, lamp="line", K=8, vis=True),
        # a lamp that is no vertical line (a horizontal tube on an arm), odd sizes, no visibility words
        dict(name="tube_matrix", kind="matrix", layout="ward", W=7.3, D=5.1, h=0.13, beds=3, patch="tri", np=12345,
             nc=333, lamp="tube", K=6, vis=False),
        # rooms of uneven size x lamp designs (K = 4, 8, 12), as a robot-design comparison runs them
        dict(name="batch_rooms", kind="batch", rooms=3, designs=4, h=0.16, np=9273, nc=260),
        # evaluating 16 plans on the ward with the stored matrix (rows on 16-byte boundaries)
        dict(name="ward_fluence", kind="fluence", layout="ward", W=10.0, D=8.0, h=0.1165, beds=6, patch="split", np=0,
             nc=2000, nvec=16, pad=4),
        # the same for a middling room whose matrix has an odd row length, and an odd number of plans
        dict(name="odd_fluence", kind="fluence", layout="ward", W=6.1, D=5.3, h=0.16, beds=2, patch="tri", np=9273,
             nc=697, nvec=37, pad=1),
        # a floor of rooms whose matrix is not kept: fluence of 64 plans straight from the geometry
        dict(name="floor_streamed", kind="streamed", layout="floor", W=18.0, D=18.0, h=0.075, beds=6, patch="quad",
             np=0, nc=250, lamp="line", K=8, nvec=64),
        # furniture was moved: the whole path once, for a few candidates (the build weighs most)
        dict(name="replan", kind="plan", layout="ward", W=8.0, D=6.0, h=0.12, beds=4, patch="split", np=0, nc=64,
             lamp="line", K=8, nvec=4),
        # patch means instead of centroid samples, for a shortlist of candidates
        dict(name="ward_area", kind="area", layout="ward", W=10.0, D=8.0, h=0.1165, beds=6, patch="split", np=0,
             nc=100, lamp="line", K=8),
        # the paper's own estimator at its own resolution, for a handful of candidates
        dict(name="ward_raster", kind="raster", layout="ward", W=10.0, D=8.0, h=0.1165, beds=6, patch="quad", np=0,
             nc=5, lamp="line", K=8, R=512),
        # scoring and selecting the candidates of a room before its matrix is computed
        dict(name="propose", kind="propose", layout="ward", W=10.0, D=8.0, h=0.1165, beds=6, patch="split", np=0,
             nc=2000, sketch=511),
        # fitting the scorer: forward, backward and Adam on its usual batch
        dict(name="train", kind="train", B=4096, in_dim=114, hidden=256),
    ]


def _logu(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    """One more case of the same ranges: the kind first, then sizes spread over the logarithm of their range."""
    kind = rng.choice(["matrix", "matrix", "batch", "fluence", "fluence", "streamed", "plan", "area", "raster", "propose",
                       "train"])
    if kind == "train":
        return dict(kind=kind, B=int(_logu(rng, 257, 8192)), in_dim=rng.choice([66, 114]), hidden=rng.choice([64, 256]))
    if kind == "batch":
        return dict(kind=kind, rooms=rng.randint(2, 4), designs=rng.randint(2, 6), h=round(_logu(rng, 0.14, 0.3), 3),
                    np=int(_logu(rng, 1500, 12000)), nc=int(_logu(rng, 60, 400)))
    c = dict(kind=kind, layout="ward", W=round(rng.uniform(4.0, 10.0), 1), D=round(rng.uniform(4.0, 8.0), 1),
             h=round(_logu(rng, 0.1165, 0.4), 3), beds=rng.randint(1, 6), patch=rng.choice(["tri", "split", "quad"]),
             np=0)
    tris = _triangles(c)
    if rng.random() < 0.5:   # a subset of the patches, odd counts among them
        c["np"] = max(300, int(tris * rng.uniform(0.2, 0.48)))
    patches = c["np"] or {"tri": tris, "split": 2 * tris, "quad": tris // 2}[c["patch"]]
    lamp = rng.choice(["point", "line", "line", "line", "tube"])
    K = 1 if lamp == "point" else rng.choice([4, 8, 12])
    if kind == "fluence":
        return dict(c, nc=min(int(_logu(rng, 40, 3000)), int(2.0e8 / patches)), nvec=rng.randint(1, 64),
                    pad=rng.choice([1, 4]))
    if kind == "propose":
        return dict(c, nc=int(_logu(rng, 200, 3000)), sketch=rng.randint(40, 700))
    if kind == "raster":
        return dict(c, nc=rng.randint(1, 5), lamp=lamp, K=K, R=rng.choice([64, 200, 256, 512]))
    pairs = {"matrix": 1.5e8, "streamed": 5e7, "plan": 1e7, "area": 8e6}[kind]
    if lamp == "tube":
        pairs /= 4
    c = dict(c, nc=max(8, min(int(_logu(rng, 20, 2000)), int(pairs / patches))), lamp=lamp, K=K)
    if kind == "matrix":
        return dict(c, vis=rng.random() < 0.5)
    if kind in ("streamed", "plan"):
        return dict(c, nvec=rng.randint(1, 64 if kind == "streamed" else 16))
    return c


# ---------------------------------------------------------------------------
# rooms
# ---------------------------------------------------------------------------

def _boxes(case, rng):
    """Furniture boxes (lo, hi); their sizes follow from the case alone, the seed only shifts them."""
    W, D = case["W"], case["D"]
    out = []
    if case["layout"] == "floor":   # rooms of 3 m along both sides of a corridor: walls with door gaps, a bed each
        n, mid, t = int(W // 3.0), D / 2, 0.1
        for side in (-1, 1):
            y = mid + side * 1.5 - (t if side < 0 else 0.0)
            for r in range(n):
                x0 = 3.0 * r + (1.05 if r else 0.05) + rng.uniform(0.0, 0.1)
                out.append((np.array([x0, y, 0.0]), np.array([x0 + (1.8 if r else 1.0), y + t, 2.9])))
            y0, y1 = (0.02, mid - 1.62) if side < 0 else (mid + 1.62, D - 0.02)
            for r in range(1, n):
                out.append((np.array([3.0 * r - t / 2, y0, 0.0]), np.array([3.0 * r + t / 2, y1, 2.9])))
            for r in range(n):
                x0, yb = 3.0 * r + 0.5 + rng.uniform(0.0, 0.3), (0.4 if side < 0 else D - 2.6) + rng.uniform(0.0, 0.2)
                out.append((np.array([x0, yb, 0.0]), np.array([x0 + 1.0, yb + 2.0, 0.6])))
        return out
    for b in range(case["beds"]):   # beds along the long walls, a cabinet beside every other, partitions between bays
        side, r = b % 2, b // 2
        room_left = W - (0.5 + 3.1 * r)
        if room_left < 2.0:
            break
        bx = 0.35 + 3.1 * r + rng.uniform(0.0, 0.15)
        off = 0.05 + rng.uniform(0.0, 0.05)
        y0 = off if side == 0 else D - off - min(2.0, 0.4 * D)
        out.append((np.array([bx, y0, 0.0]), np.array([bx + 1.0, y0 + min(2.0, 0.4 * D), 0.6])))
        if b % 2 == 0:
            out.append((np.array([bx + 1.2, 0.06, 0.0]), np.array([bx + 1.8, 0.56, 1.8])))
        elif room_left > 3.1:
            out.append((np.array([bx + 2.4, 0.42 * D, 0.0]), np.array([bx + 2.5, 0.58 * D, 2.0])))
    return out


def _counts(lo, hi, h):
    ext = np.round(np.asarray(hi) - np.asarray(lo), 6)   # the seed's shift of a box must not change its cells
    return np.maximum(1, np.floor(ext / h + 0.499).astype(np.int64))


def _triangles(case):
    """Triangles of the case's room (the same for every seed)."""
    n = 0
    for lo, hi, inward in [(np.zeros(3), np.array([case["W"], case["D"], HEIGHT]), True)] + [
            (lo, hi, False) for lo, hi in _boxes(case, np.random.default_rng(0))]:
        c = _counts(lo, hi, case["h"])
        n += 2 * int((2 if inward else 1) * c[0] * c[1] + 2 * c[1] * c[2] + 2 * c[0] * c[2])
    return n


def _spread(x):
    x = x.astype(np.uint64)
    for s, m in ((8, 0x00FF00FF), (4, 0x0F0F0F0F), (2, 0x33333333), (1, 0x55555555)):
        x = (x | (x << np.uint64(s))) & np.uint64(m)
    return x


def _box_faces(lo, hi, h, inward, rng):
    """Corner quads (cells, 4, 3) of a box's faces, wound counter-clockwise seen from the free side, and their
    normals; furniture stands on the floor and has no bottom face."""
    n, ext = _counts(lo, hi, h), hi - lo
    for k in range(3):
        u, v = (k + 1) % 3, (k + 2) % 3
        for side in (0, 1):
            if not inward and k == 2 and side == 0:
                continue
            P = np.empty((n[u] + 1, n[v] + 1, 3))
            P[..., k] = (lo, hi)[side][k]
            P[..., u] = (lo[u] + ext[u] * np.arange(n[u] + 1) / n[u])[:, None]
            P[..., v] = (lo[v] + ext[v] * np.arange(n[v] + 1) / n[v])[None, :]
            if n[u] > 1 and n[v] > 1:   # inner vertices move inside the face's plane
                P[1:-1, 1:-1][..., [u, v]] += rng.uniform(-0.08 * h, 0.08 * h, (n[u] - 1, n[v] - 1, 2))
            a, b = (x.ravel() for x in np.meshgrid(np.arange(n[u]), np.arange(n[v]), indexing="ij"))
            order = np.argsort(_spread(a) | (_spread(b) << np.uint64(1)), kind="stable")
            a, b = a[order], b[order]
            sign = (1.0 if side else -1.0) * (-1.0 if inward else 1.0)
            q = np.stack([P[a, b], P[a + 1, b], P[a + 1, b + 1], P[a, b + 1]], 1)
            nrm = np.zeros(3)
            nrm[k] = sign
            yield (q if sign > 0 else q[:, ::-1]), nrm


def _area(t):
    return 0.5 * np.linalg.norm(np.cross(t[:, 1] - t[:, 0], t[:, 2] - t[:, 0]), axis=1)


def _room(case, seed):
    """The room's arrays (NumPy): triangles, patches and the list of its boxes."""
    rng = np.random.default_rng(seed)
    boxes = _boxes(case, rng)
    quads, nrm = [], []
    shell = (np.zeros(3), np.array([case["W"], case["D"], HEIGHT]))
    for (lo, hi), inward in [(shell, True)] + [(b, False) for b in boxes]:
        for q, n in _box_faces(lo, hi, case["h"], inward, rng):
            quads.append(q)
            nrm.append(np.repeat(n[None], q.shape[0], 0))
    quads, nrm = np.concatenate(quads), np.concatenate(nrm)
    verts = quads.reshape(-1, 3)
    base = 4 * np.arange(quads.shape[0])[:, None]
    tris = np.concatenate([base + [[0, 1, 2]], base + [[0, 2, 3]]], 1).reshape(-1, 3)
    tnrm, T = np.repeat(nrm, 2, 0), verts[tris]
    if case["patch"] == "quad":
        ptri = T.reshape(-1, 2, 3, 3)
        excl = np.arange(T.shape[0]).reshape(-1, 2)
        pn = nrm
    else:
        par = np.arange(T.shape[0])
        if case["patch"] == "split":   # halved at the midpoint of the longest edge (the diagonal, corner 2 to 0)
            even = (par % 2 == 0)[:, None]
            d, o = np.where(even, T[:, 2], T[:, 1]), np.where(even, T[:, 1], T[:, 2])
            m = 0.5 * (T[:, 0] + d)
            T = np.stack([np.stack([T[:, 0], o, m], 1), np.stack([o, d, m], 1)], 1).reshape(-1, 3, 3)
            par = np.repeat(par, 2)
        ptri = np.concatenate([T[:, None], np.zeros_like(T)[:, None]], 1)
        excl = np.stack([par, np.full_like(par, -1)], 1)
        pn = tnrm[par]
    a0, a1 = _area(ptri[:, 0]), _area(ptri[:, 1])
    cen = (ptri[:, 0].mean(1) * a0[:, None] + ptri[:, 1].mean(1) * a1[:, None]) / (a0 + a1)[:, None]
    keep = np.arange(cen.shape[0])
    if case["np"] and case["np"] < keep.size:
        keep = np.sort(rng.choice(keep.size, case["np"], replace=False))
    f32 = lambda x: np.ascontiguousarray(x, np.float32)  # noqa: E731
    return dict(verts=f32(verts), tris=np.ascontiguousarray(tris, np.int32), tnrm=f32(tnrm), cen=f32(cen[keep]),
                nrm=f32(pn[keep]), area=f32((a0 + a1)[keep]), excl=np.ascontiguousarray(excl[keep], np.int32),
                ptri=f32(ptri[keep]), boxes=boxes)


def _candidates(case, room, n, zb, length, rng):
    """n lamp positions on a free floor grid, 0.15 m clear of the furniture, in grid order height by height."""
    W, D = case["W"], case["D"]
    step = min(0.4, math.sqrt(W * D * len(zb) / (1.6 * n)))
    while True:
        out = []
        for z in zb:
            g = [np.arange(0.2, e - 0.2 + 1e-9, step) for e in (W, D)]
            xy = np.stack([x.ravel() for x in np.meshgrid(*g, indexing="ij")], 1)
            ok = np.ones(xy.shape[0], bool)
            for lo, hi in room["boxes"]:
                if z < hi[2] + 0.15:
                    ok &= ~((xy > lo[:2] - 0.15).all(1) & (xy < hi[:2] + 0.15).all(1))
            out.append(np.concatenate([xy[ok], np.full((int(ok.sum()), 1), z)], 1))
        c = np.concatenate(out)
        if c.shape[0] >= n:
            break
        step *= 0.8
    pick = np.sort(rng.choice(c.shape[0], n, replace=False))
    return np.ascontiguousarray(c[pick], np.float32)


def _lamp(kind, K, power, length=1.2):
    if kind == "point":
        return uvc.point_lamp(power)
    off = np.zeros((K, 3))
    off[:, 2 if kind == "line" else 0] = length * (np.arange(K) + 0.5) / K - (0.0 if kind == "line" else length / 2)
    return uvc.Lamp(off, np.full(K, 1.0 / K), power)


def _cuda(x):
    return torch.from_numpy(x).cuda()


def _device_room(room):
    return {k: _cuda(v) for k, v in room.items() if k != "boxes"}


def _build(g):
    return uvc.build_scene(g["verts"], g["tris"], g["cen"], g["nrm"], g["area"], g["excl"])


def _sampled_matrix(g, cand, gen, rows, lda):
    """A matrix as the library stores them, in plain torch: the inverse-square law with about half of the
    facing pairs dark, in a buffer of `lda` columns."""
    n = g["cen"].shape[0]
    A = torch.zeros((rows, lda), device="cuda")
    for i in range(0, rows, 256):
        v = cand[i:i + 256, None, :] - g["cen"][None]
        d2 = (v * v).sum(-1)
        cos = (v * g["nrm"][None]).sum(-1).clamp_min(0) / d2.sqrt()
        lit = torch.rand(cos.shape, device="cuda", generator=gen) < 0.5
        A[i:i + 256, :n] = 120.0 / (4 * math.pi) * cos / d2 * lit
    return A


# ---------------------------------------------------------------------------
# preparing and running
# ---------------------------------------------------------------------------

def prepare(case, seed):
    kind, rng = case["kind"], np.random.default_rng([seed, 1])
    power = float(rng.uniform(80.0, 160.0))
    s = dict(kind=kind, case=case)
    if kind == "train":
        B, d, H = case["B"], case["in_dim"], case["hidden"]
        s["mlp"] = uvc.Mlp(d, H, max_batch=B, seed=seed)
        s["batches"] = [(_cuda(rng.standard_normal((B, d), np.float32)), _cuda(rng.random(B, np.float32) ** 8),
                         _cuda(rng.uniform(0.5, 4.0, B).astype(np.float32) / B)) for _ in range(4)]
        return s
    if kind == "batch":
        jobs, lamps, s["keep"] = [], [], []
        for L, K in ((0.6, 4), (1.2, 8), (1.8, 12)):
            lamps.append(_lamp("line", K, power, L))
        for c in _batch_rooms(case):
            room = _room(c, seed)
            scene = _build(_device_room(room))
            for d in range(case["designs"]):
                cand = _cuda(_candidates(c, room, c["nc"], [(0.3, 0.5, 0.8, 1.1)[d % 4]], (0.6, 1.2, 1.8)[d % 3], rng))
                jobs.append((scene, cand, d % 3, torch.empty((c["nc"], scene.np), device="cuda"), None))
        s["batch"], s["out"] = uvc.Batch(jobs, lamps), [j[3] for j in jobs]
        return s
    room = _room(case, seed)
    g = s["room"] = _device_room(room)
    cand = s["cand"] = _cuda(_candidates(case, room, case["nc"], (0.5, 1.0, 1.5) if case["nc"] > 300 else (0.5, 1.0), 1.2, rng))
    nc, np_ = cand.shape[0], g["cen"].shape[0]
    if "lamp" in case:
        s["lamp"] = _lamp(case["lamp"], case["K"], power)
    if "nvec" in case:
        s["t"] = _cuda(rng.uniform(0.0, 60.0 / max(1, nc // 200), (case["nvec"], nc)).astype(np.float32))
    if kind != "plan":
        s["scene"] = _build(g)
    if kind in ("matrix", "area", "plan"):
        s["A"] = torch.empty((nc, np_ if kind != "plan" else (np_ + 3) // 4 * 4), device="cuda")
    if kind == "matrix" and case["vis"]:
        s["vis"] = torch.empty((case["K"], nc, (np_ + 31) // 32), dtype=torch.int32, device="cuda")
    if kind == "fluence":
        gen = torch.Generator("cuda").manual_seed(seed)
        lda = -(-np_ // case["pad"]) * case["pad"]
        s["A"] = _sampled_matrix(g, cand, gen, nc, lda + (lda + 1) % 2 * (case["pad"] == 1))   # odd rows where pad is 1
    if kind in ("fluence", "streamed"):
        s["mu"] = torch.empty((case["nvec"], np_), device="cuda")
    if kind == "raster":
        s["work"] = uvc.raster_workspace(s["scene"], s["lamp"], case["R"], nc)
        s["A"] = torch.empty((nc, s["scene"].nt), device="cuda")
    if kind == "propose":
        gen = torch.Generator("cuda").manual_seed(seed)
        pick = torch.from_numpy(np.sort(rng.choice(np_, min(case["sketch"], np_), replace=False))).cuda()
        probe = {k: g[k][pick].contiguous() for k in ("cen", "nrm", "area")}
        s["A"], s["parea"] = _sampled_matrix(probe, cand, gen, nc, pick.numel()), probe["area"]
        s["scorer"] = _scorer(nc)
        s["rank"] = torch.randn(nc, device="cuda", generator=gen)
    return s


def _batch_rooms(case):
    """Uneven rooms: each has half as many more candidates and coarser or finer cells than the one before."""
    return [dict(layout="ward", W=4.5 + 1.9 * r, D=4.2 + 1.1 * r, h=case["h"] * (1.0, 0.8, 1.25, 0.9)[r], beds=1 + r,
                 patch=("tri", "split", "quad", "tri")[r], np=(0 if r == 1 else case["np"] // (1, 1, 2, 3)[r]),
                 nc=case["nc"] * (2 + r) // 2) for r in range(case["rooms"])]


@functools.lru_cache(maxsize=4)
def _scorer(nc):
    return proposal.Scorer.load(max_batch=nc)


def run(s):
    kind = s["kind"]
    if kind == "matrix":
        A, vis = uvc.irradiance_matrix(s["scene"], s["cand"], s["lamp"], A=s["A"], vis=s.get("vis"))
        return [A] if vis is None else [A, vis]
    if kind == "batch":
        s["batch"].launch()
        return s["out"]
    if kind == "fluence":
        mu = uvc.fluence(s["scene"], s["A"], s["t"], mu=s["mu"])
        return [mu, *uvc.coverage(s["scene"], mu, MU_MIN)]
    if kind == "streamed":
        return [uvc.fluence_streamed(s["scene"], s["cand"], s["lamp"], s["t"], mu=s["mu"])]
    if kind == "plan":
        scene = _build(s["room"])
        A, _ = uvc.irradiance_matrix(scene, s["cand"], s["lamp"], A=s["A"])
        mu = uvc.fluence(scene, A, s["t"])
        cov = uvc.coverage(scene, mu, MU_MIN)
        scene.free()
        return [A[:, :mu.shape[1]], mu, *cov]
    if kind == "area":
        return list(uvc.irradiance_area_mean(s["scene"], s["cand"], s["lamp"], s["room"]["ptri"], A=s["A"], with_closed=True))
    if kind == "raster":
        return [uvc.irradiance_raster(s["scene"], s["room"]["tnrm"], s["cand"], s["lamp"], R=s["case"]["R"], A=s["A"],
                                      workspace=s["work"])]
    if kind == "propose":
        feat = proposal.features(s["scene"], s["cand"], s["A"], s["parea"])
        logit = s["scorer"].scores(feat)
        # the selection ranks scores that are held fixed: its whole numbers must not hang on a logit's last bit
        score = s["rank"].clone()
        uvc.mark_best(s["A"], score, rare=proposal.rare_count(score.shape[0]))
        idx, kept = uvc.select_top(score, proposal.keep_count(score.shape[0], KEEP), cand=s["cand"])
        return dict(feat=feat, logit=logit, idx=idx, kept=kept, lost=uvc.probe_lost(s["A"], idx, s["parea"]))
    # so small a learning rate leaves the FP32 weights as they are: every pass does the same steps
    losses = [s["mlp"].train_step(x, y, w, 1e-30) for x, y, w in s["batches"]]
    return [torch.cat(losses), s["mlp"].grads()]


# ---------------------------------------------------------------------------
# work and exact values
# ---------------------------------------------------------------------------

def work(case):
    """Inputs read once and outputs written once; 60 operations per facing test and Eq. (7) term of a source and
    patch (both sides of the geometry), products and sums for the dense parts."""
    kind = case["kind"]
    if kind == "train":
        B, P, H = case["B"], case["in_dim"], case["hidden"]
        n = P * H + H * H + 3 * H + 1
        return dict(bytes=4.0 * (4 * B * (P + 2) + 4 * 4 * n), flops=4.0 * 2 * B * (2 * P * H + 3 * H * H + 3 * H))
    if kind == "batch":
        b = f = 0.0
        for c in _batch_rooms(case):
            nt, np_ = _sizes(c)
            for d in range(case["designs"]):
                b += 4.0 * c["nc"] * np_ + 48.0 * nt + 40.0 * np_
                f += 60.0 * (4, 8, 12)[d % 3] * c["nc"] * np_
        return dict(bytes=b, flops=f)
    nt, np_ = _sizes(case)
    nc, K, nvec = case["nc"], case.get("K", 1), case.get("nvec", 1)
    scene, pairs = 48.0 * nt + 40.0 * np_ + 12.0 * nc, float(nc) * np_
    if kind == "fluence":
        return dict(bytes=4.0 * (pairs + nvec * (nc + 2 * np_)) + 4.0 * np_, flops=2.0 * pairs * nvec)
    if kind == "streamed":
        return dict(bytes=scene + 4.0 * nvec * (nc + np_), flops=pairs * (60.0 * K + 2.0 * nvec))
    if kind == "raster":
        pix = 6.0 * case["R"] ** 2 * K * nc
        return dict(bytes=48.0 * nt + 12.0 * nt + 4.0 * nc * nt, flops=40.0 * pix + 60.0 * K * nc * nt)
    if kind == "propose":
        return dict(bytes=scene + 4.0 * (nc * (114 + case["sketch"]) + 2 * nc), flops=10.0 * pairs + 2.0 * nc * (114 + 257) * 256)
    out = 4.0 * pairs
    if kind == "matrix" and case["vis"]:
        out += 4.0 * K * nc * ((np_ + 31) // 32)
    if kind == "area":
        return dict(bytes=scene + 72.0 * np_ + out + pairs, flops=pairs * K * 160.0)
    if kind == "plan":
        return dict(bytes=2 * scene + out + 4.0 * nvec * (nc + 2 * np_), flops=pairs * (60.0 * K + 2.0 * nvec))
    return dict(bytes=scene + out, flops=60.0 * K * pairs)


def _sizes(case):
    nt = _triangles(case)
    np_ = {"tri": nt, "split": 2 * nt, "quad": nt // 2}[case["patch"]]
    return nt, min(np_, case["np"] or np_)


def _visible(o, p, T, excl):
    """(len(o), len(p)) truths in 64 bits: no triangle of T but a patch's own meets the open segment from o to p."""
    e1, e2 = T[:, 1] - T[:, 0], T[:, 2] - T[:, 0]
    out = torch.ones((o.shape[0], p.shape[0]), dtype=torch.bool, device="cuda")
    own = torch.arange(T.shape[0], device="cuda")
    n = max(1, int(2e7 // (p.shape[0] * T.shape[0]))) if T.shape[0] else o.shape[0]
    step = max(1, int(2e7 // (n * T.shape[0])))
    for i in range(0, o.shape[0], n):
        for j in range(0, p.shape[0], step):
            d = p[None, j:j + step] - o[i:i + n, None]                       # (n, step, 3)
            s = o[i:i + n, None, None] - T[None, None, :, 0]                 # (n, 1, nt, 3)
            h = torch.cross(d[:, :, None].expand(-1, -1, T.shape[0], -1), e2.expand(d.shape[0], d.shape[1], -1, -1), -1)
            det = (h * e1).sum(-1)
            q = torch.cross(s, e1.expand(s.shape[0], 1, -1, -1), -1)
            u, v = (s * h).sum(-1) / det, (q * d[:, :, None]).sum(-1) / det
            t = (q * e2).sum(-1) / det
            hit = (u >= 0) & (v >= 0) & (u + v <= 1) & (t > 0) & (t < 1)
            hit &= (excl[j:j + step, :1] != own) & (excl[j:j + step, 1:] != own)
            out[i:i + n, j:j + step] = ~hit.any(-1)
    return out


def _exact_matrix(s):
    g, lamp = s["room"], s["lamp"]
    T = g["verts"].double()[g["tris"].long()]
    p, n = g["cen"].double(), g["nrm"].double()
    A = torch.zeros((s["cand"].shape[0], p.shape[0]), dtype=torch.float64, device="cuda")
    for off, w in zip(lamp.offsets, lamp.weights):
        o = (s["cand"] + torch.from_numpy(off).cuda()).double()              # a source sits at the FP32 sum
        v = o[:, None] - p[None]
        d = v.norm(dim=-1)
        E = (v * n[None]).sum(-1).clamp_min(0) * (float(w) * lamp.power) / (4 * math.pi * d ** 3)
        A += E * _visible(o, p, T, g["excl"])
    return A


def _cover(mu, area):
    a = area.double()
    ok = (mu >= MU_MIN).double()
    return [(ok @ a) / a.sum(), ok.mean(1)]


def _exact_train(s):
    m = s["mlp"]
    P = {k: torch.from_numpy(np.array(v)).cuda().double().requires_grad_() for k, v in m.split(m.params()).items()}
    losses = []
    for x, y, w in s["batches"]:
        for v in P.values():
            v.grad = None
        z = torch.relu(torch.relu(x.double() @ P["W1"][:m.in_dim] + P["b1"]) @ P["W2"] + P["b2"]) @ P["w3"] + P["b3"]
        loss = (w.double() * (torch.nn.functional.softplus(z) - y.double() * z)).sum()
        loss.backward()
        losses.append(loss.detach()[None])
    return [torch.cat(losses), torch.cat([v.grad.reshape(-1) for v in P.values()]).cpu().numpy()]


def _nearest(c, T):
    """Distance of each point to its nearest triangle: inside the prism over it the plane's, else an edge's."""
    a, b, d = T[:, 0], T[:, 1], T[:, 2]
    nrm = torch.cross(b - a, d - a, -1)
    nrm = nrm / nrm.norm(dim=-1, keepdim=True)
    out = []
    for i in range(0, c.shape[0], 64):
        p = c[i:i + 64, None]
        inside = torch.ones((p.shape[0], T.shape[0]), dtype=torch.bool, device=c.device)
        best = torch.full(inside.shape, math.inf, dtype=torch.float64, device=c.device)
        for q, r in ((a, b), (b, d), (d, a)):
            e, v = r - q, p - q
            inside &= (torch.cross(e[None].expand_as(v), v, -1) * nrm).sum(-1) >= 0
            t = ((v * e).sum(-1) / (e * e).sum(-1)).clamp(0, 1)
            best = torch.minimum(best, (v - t[..., None] * e).norm(dim=-1))
        best = torch.where(inside, ((p - a) * nrm).sum(-1).abs(), best)
        out.append(best.min(1).values)
    return torch.cat(out)


def _exact_propose(s):
    """The features' definition in 64 bits (bins decided there too), and the scorer's network on them."""
    g, nc = s["room"], s["cand"].shape[0]
    c, area = s["cand"].double(), g["area"].double()
    k = np.arange(1, 64)
    edges = torch.from_numpy(((0.1 * 250.0 ** (k / 64)) ** 2).astype(np.float32)).cuda().double()
    feat = torch.zeros((nc, 114), dtype=torch.float64, device="cuda")
    for i in range(0, nc, 256):
        d2 = (c[i:i + 256, None] - g["cen"].double()[None]).square().sum(-1)
        feat[i:i + 256].scatter_add_(1, torch.bucketize(d2, edges, right=True), area.expand_as(d2))
    feat /= area.sum()
    feat[:, 64] = _nearest(c, g["verts"].double()[g["tris"].long()])
    feat[:, 65] = c[:, 2]
    A, a = s["A"].double(), s["parea"].double()
    best = A.max(0).values
    lit = best > 0
    A, a, best = A[:, lit], a[lit], best[lit]
    hard = (torch.floor(torch.log2(best / ((a * best).sum() / a.sum()))) + 4).clamp(0, 7).long()
    eff = torch.bucketize(A / best, torch.tensor([0.5, 0.7, 0.8, 0.9, 0.95], dtype=torch.float64, device="cuda"), right=True)
    feat.scatter_add_(1, 66 + 6 * hard + eff, (a / a.sum()).expand_as(A))
    m = s["scorer"].mlp
    P = {k: torch.from_numpy(np.array(v)).cuda().double() for k, v in m.split(s["scorer"].flat).items()}
    z = torch.relu(torch.relu(feat @ P["W1"][:114] + P["b1"]) @ P["W2"] + P["b2"]) @ P["w3"] + P["b3"]
    return dict(feat=feat, logit=z, idx=None, kept=None, lost=None)


def exact(case, seed):
    """What run() returns, in 64 bits.  Visibility by brute force: None where that takes too many tests (the
    rasteriser, the solid angles and the batches always do)."""
    kind = case["kind"]
    if kind in ("batch", "area", "raster"):
        return None
    if kind in ("matrix", "streamed", "plan"):
        nt, np_ = _sizes(case)
        if float(nt) * np_ * case["nc"] * case["K"] > EXACT_TESTS:
            return None
    s = prepare(case, seed)
    if kind == "train":
        return _exact_train(s)
    if kind == "propose":
        return _exact_propose(s)
    if kind == "fluence":
        mu = s["t"].double() @ s["A"][:, :s["mu"].shape[1]].double()
        return [mu, *_cover(mu, s["room"]["area"])]
    A = _exact_matrix(s)
    if kind == "matrix":
        return [A, None]
    mu = s["t"].double() @ A
    return [mu] if kind == "streamed" else [A, mu, *_cover(mu, s["room"]["area"])]
