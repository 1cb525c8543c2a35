"""The work that users of the library have it do, as measurable cases.

Every case goes through the package's public entry points: building hash codes
and lookup tables, matching one pair, a few pairs, an exhaustive or an uneven
pair list, with the epipolar band, with the mutual check and the Hamming
threshold, one pair per launch, end to end from host memory, and the first
stage of Ga-CasHash.  Sizes are those of the repository's configurations: one
pair of 2,000 x 2,000; 100 images of 4,000..12,000 features with all pairs;
images of 1,000..20,000 features (log-uniform) with 30 neighbours each; pinhole
views of 200,000 points with about 8,000 key-points each.

A case's image sizes (and, for views, its cameras) follow from its "layout"
number; the descriptors, noise, projection matrix and random words follow from
the seed given to prepare().
"""
import math

import numpy as np
import torch

import paper_1805_08995_gb300 as ch

DIM = 128
BF16, FP32 = ch.CASHASH_BF16, ch.CASHASH_FP32
BATCHED, PER_PAIR = ch.CASHASH_SCHED_PERSISTENT, ch.CASHASH_SCHED_PER_PAIR
NO_TAU = 128


def _case(name, op, images, **over):
    c = {"name": name, "op": op, "images": images, "n_images": 2, "lo": 2000, "hi": 2000, "layout": 1,
         "code_bits": 128, "n_tables": 6, "bits": 8, "top_k": 10, "tau": NO_TAU, "flags": 0,
         "precision": BF16, "schedule": BATCHED, "epi_px": -1.0}
    c.update(over)
    return c


def listed():
    return [
        # One pair handed over on its own, as by an interactive tool: plan, match and release in a call.
        _case("pair_once", "pairs", "all"),
        # Hash codes and tables of two small images, each frame of a live pipeline (default FP32 projection).
        _case("build_pair", "build", "all", precision=FP32),
        # A dozen images of a small object, every pair, the plan kept: too few pairs to fill the GPU.
        _case("few_pairs", "match", "all", n_images=12, lo=1000, hi=5000, layout=2),
        # Hash codes of an ordinary photo collection with the default FP32 projection.
        _case("build_fp32", "build", "all", n_images=40, lo=4000, hi=12000, layout=3, precision=FP32),
        # Hash codes of the exhaustive set below with the tensor-core projection.
        _case("build_bf16", "build", "all", n_images=100, lo=4000, hi=12000, layout=4),
        # The headline workload: 100 images of about 8k features, all 4,950 pairs.
        _case("exhaustive", "match", "all", n_images=100, lo=4000, hi=12000, layout=4),
        # A photo collection with uneven images and a sparse neighbour graph.
        _case("uneven", "match", "graph", n_images=400, lo=1000, hi=20000, layout=5),
        # Guided matching inside a 4 px epipolar band along a camera path (about 8k key-points a view).
        _case("views_band", "match", "views", n_images=160, layout=6, epi_px=4.0),
        # Mutual check and the Hamming threshold of Sec. 6, as a precision-minded reconstruction asks for.
        _case("mutual_tau", "match", "all", n_images=30, lo=2000, hi=6000, layout=7, flags=ch.CASHASH_FLAG_MUTUAL,
              tau=50),
        # The schedule that launches one kernel per pair.
        _case("per_pair", "match", "all", n_images=16, lo=2000, hi=9000, layout=8, schedule=PER_PAIR,
              precision=FP32),
        # End to end from pinned host descriptors to host match lists.
        _case("run_host", "host", "all", n_images=24, lo=4000, hi=12000, layout=9),
        # First stage of Ga-CasHash: top-scale subsets, their matches, fundamental matrices.
        _case("ga_stage1", "ga", "views", n_images=60, layout=10),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: sizes over the whole range of the listed ones, and the options users set."""
    op = rng.choice(["pairs", "build", "match", "match", "match", "band", "per_pair", "host", "ga"])
    opt = dict(layout=rng.randrange(1, 1 << 30))
    if op in ("band", "ga"):
        n = _log_int(rng, 8, 160 if op == "band" else 100)
        return dict(_case("", "match" if op == "band" else "ga", "views", n_images=n,
                          epi_px=4.0 if op == "band" else -1.0, **opt))
    opt.update(precision=rng.choice([FP32, BF16]), top_k=rng.choice([4, 10, 10, 16]),
               n_tables=rng.choice([4, 6, 6, 8]), code_bits=rng.choice([64, 128, 128]))
    if op != "build" and rng.random() < 0.3:
        opt["tau"] = rng.choice([40, 50, 60])
    if op == "pairs":
        a, b = sorted((_log_int(rng, 500, 20000), _log_int(rng, 500, 20000)))
        return dict(_case("", "pairs", "all", lo=a, hi=b, **opt))
    if op == "build":
        n = _log_int(rng, 2, 100)
        return dict(_case("", "build", "all", n_images=n, lo=1000, hi=_log_int(rng, 1001, 16000), **opt))
    if op == "per_pair":
        return dict(_case("", "match", "all", n_images=rng.randrange(2, 17), lo=1000, hi=rng.randrange(1001, 12001),
                          schedule=PER_PAIR, **opt))
    if op == "host":
        return dict(_case("", "host", "all", n_images=rng.randrange(2, 30), lo=1000,
                          hi=_log_int(rng, 1001, 12000), **opt))
    if rng.random() < 0.4:
        c = _case("", "match", "graph", n_images=_log_int(rng, 40, 400), lo=rng.choice([500, 1000, 3000]),
                  hi=rng.randrange(5000, 20001), **opt)
        while _candidates(c) > MOST_CANDIDATES:
            c["n_images"] = c["n_images"] * 3 // 4
        return c
    lo, hi = rng.choice([500, 1000, 4000]), rng.randrange(4001, 12001)
    n = _log_int(rng, 3, 70)
    if n <= 40 and rng.random() < 0.4:
        opt["flags"] = rng.choice([ch.CASHASH_FLAG_MUTUAL, ch.CASHASH_FLAG_ACCEPT_SINGLE])
    return dict(_case("", "match", "all", n_images=n, lo=lo, hi=hi, **opt))


# ---------------------------------------------------------------------------
# layouts: image sizes, pair lists, cameras
# ---------------------------------------------------------------------------

def _offsets(sizes):
    off = np.zeros(len(sizes) + 1, np.uint64)
    off[1:] = np.cumsum(np.asarray(sizes, np.uint64))
    return off


def _layout(case):
    """Image sizes, pair list and, per image, the images it shares points with ("all" and "graph")."""
    rng = np.random.default_rng([case["layout"], 11])
    n, lo, hi = case["n_images"], case["lo"], case["hi"]
    if case["images"] == "all":
        sizes = np.array([lo, hi]) if n == 2 else rng.integers(lo, hi + 1, size=n)
        pairs = np.stack(np.triu_indices(n, 1), axis=1)
        step = np.array([-5, -4, -3, -2, -1, 1, 2, 3, 4, 5])
        near = (np.arange(n)[:, None] + step[None, :]) % n
        near = np.where(near == np.arange(n)[:, None], (near + 1) % n, near)
    else:
        sizes = np.rint(np.exp(rng.uniform(math.log(lo), math.log(hi), size=n))).astype(np.int64)
        k = min(30, n - 1)
        near = np.argsort(rng.random((n, n)) + 2.0 * np.eye(n), axis=1)[:, :k]
        i = np.repeat(np.arange(n), k)
        j = near.ravel()
        pairs = np.unique(np.stack([np.minimum(i, j), np.maximum(i, j)], axis=1), axis=0)
    return sizes, pairs.astype(np.uint32), near


VIEW_POINTS, WIDTH, HEIGHT, FOCAL = 200_000, 1920, 1080, 1000.0


def _cameras(case):
    """Cameras on a helix around the unit cube's centre, looking along the path."""
    n = case["n_images"]
    rng = np.random.default_rng([case["layout"], 12])
    cams = []
    for i in range(n):
        th = 4 * math.pi * i / 500
        pos = np.array([0.5 + 0.25 * math.cos(th), 0.5 + 0.25 * math.sin(th), 0.5 + 0.5 * (i / 499 - 0.5)])
        pos += rng.normal(0, 0.01, 3)
        fwd = np.array([-math.sin(th), math.cos(th), 0.0])
        up = np.array([0.0, 0.0, 1.0])
        axis = rng.normal(0, 0.05, 3)
        ang = float(np.linalg.norm(axis))
        kx, ky, kz = axis / ang
        K = np.array([[0, -kz, ky], [kz, 0, -kx], [-ky, kx, 0]])
        rot = np.eye(3) + math.sin(ang) * K + (1 - math.cos(ang)) * (K @ K)
        Rw = rot @ np.stack([np.cross(fwd, up), -up, fwd])
        cams.append((Rw, -Rw @ pos))
    return cams


def _view_F(cams, pairs):
    """Fundamental matrices (x_candidate^T F x_query = 0) of the view pairs."""
    Kinv = np.linalg.inv(np.array([[FOCAL, 0, WIDTH / 2], [0, FOCAL, HEIGHT / 2], [0, 0, 1.0]]))
    F = np.zeros((len(pairs), 9))
    for p, (a, b) in enumerate(pairs):
        Rr = cams[b][0] @ cams[a][0].T
        tr = cams[b][1] - Rr @ cams[a][1]
        tx = np.array([[0, -tr[2], tr[1]], [tr[2], 0, -tr[0]], [-tr[1], tr[0], 0]])
        Fm = Kinv.T @ tx @ Rr @ Kinv
        F[p] = (Fm / np.linalg.norm(Fm)).ravel()
    return F


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _sift(g, n):
    """SIFT-like uint8 descriptors: |N(0,1)|, unit norm, clipped at 0.2, unit norm, times 512, rounded."""
    out = torch.empty((n, DIM), dtype=torch.uint8, device="cuda")
    for s in range(0, n, 1 << 20):
        x = torch.randn((min(1 << 20, n - s), DIM), generator=g, device="cuda").abs_()
        x /= x.norm(dim=1, keepdim=True)
        x.clamp_(max=0.2)
        x /= x.norm(dim=1, keepdim=True)
        out[s:s + len(x)] = (x * 512.0).round_().clamp_(0, 255).to(torch.uint8)
    return out


def _noisy(g, rows):
    """The same points seen again: N(0, 8^2) per component, rounded and clipped."""
    out = torch.empty_like(rows)
    for s in range(0, len(rows), 1 << 20):
        r = rows[s:s + (1 << 20)]
        x = torch.randn(r.shape, generator=g, device="cuda").mul_(8.0).add_(r)
        out[s:s + len(r)] = x.round_().clamp_(0, 255).to(torch.uint8)
    return out


def _photo_desc(g, sizes, near):
    """Descriptors of images of which 30 % are noisy copies of fresh descriptors of a neighbour image."""
    n = int(sizes.sum())
    fresh = _sift(g, n)
    img = torch.from_numpy(np.repeat(np.arange(len(sizes)), sizes)).cuda()
    copy = torch.rand(n, generator=g, device="cuda") < 0.3
    src_rows = torch.nonzero(~copy).ravel()
    cnt = torch.bincount(img[src_rows], minlength=len(sizes))
    first = torch.cumsum(cnt, 0) - cnt
    dst = torch.nonzero(copy).ravel()
    nb = torch.from_numpy(np.ascontiguousarray(near)).cuda()
    pick = torch.randint(0, near.shape[1], (len(dst),), generator=g, device="cuda")
    src = nb[img[dst], pick]
    u = torch.rand(len(dst), generator=g, device="cuda", dtype=torch.float64)
    row = src_rows[first[src] + torch.minimum((u * cnt[src]).long(), cnt[src] - 1)]
    fresh[dst] = _noisy(g, fresh[row])
    return fresh


def _views(case, g):
    """Key-points, descriptors and scales of the views, their pair list (20 % overlap) and F.  The scene and
    the cameras follow from the layout; noise, clutter and descriptors from the generator."""
    cams = _cameras(case)
    n = case["n_images"]
    scene = _gen(case["layout"])
    X = torch.rand((VIEW_POINTS, 3), generator=scene, device="cuda", dtype=torch.float64)
    unit = 1.6 * 0.2 * 2.0 ** torch.clamp(-torch.log1p(-torch.rand(VIEW_POINTS, generator=scene, device="cuda",
                                                                   dtype=torch.float64)), max=5.0)
    seen = torch.zeros((n, VIEW_POINTS), device="cuda")
    uv, sc = [], []
    for i, (Rw, t) in enumerate(cams):
        Y = X @ torch.from_numpy(Rw.T.copy()).cuda() + torch.from_numpy(t).cuda()
        z = Y[:, 2]
        p = Y[:, :2] / z[:, None] * FOCAL + torch.tensor([WIDTH / 2, HEIGHT / 2], device="cuda")
        ok = (z > 0.02) & (z < 0.355) & (p[:, 0] >= 0) & (p[:, 0] < WIDTH) & (p[:, 1] >= 0) & (p[:, 1] < HEIGHT)
        seen[i] = ok
        uv.append(p[ok])
        sc.append(unit[ok] / z[ok])
    both = seen @ seen.T
    n_vis = both.diagonal().cpu().numpy().astype(np.int64)
    both = both.cpu().numpy()
    need = 0.2 * np.maximum(1, np.minimum(n_vis[:, None], n_vis[None, :]))
    pairs = np.argwhere(np.triu(both >= need, 1)).astype(np.uint32)
    view, point = torch.nonzero(seen, as_tuple=True)
    n_cl = np.rint(n_vis * 0.3 / 0.7).astype(np.int64)
    n_clutter, n_real = int(n_cl.sum()), len(view)
    desc = torch.cat([_noisy(g, _sift(g, VIEW_POINTS)[point]), _sift(g, n_clutter)])
    kp = torch.cat([torch.cat(uv) + torch.randn((n_real, 2), generator=g, device="cuda", dtype=torch.float64),
                    torch.rand((n_clutter, 2), generator=g, device="cuda", dtype=torch.float64)
                    * torch.tensor([WIDTH, HEIGHT], device="cuda", dtype=torch.float64)])
    noise = torch.exp(0.1 * torch.randn(n_real, generator=g, device="cuda", dtype=torch.float64))
    e = -torch.log1p(-torch.rand(n_clutter, generator=g, device="cuda", dtype=torch.float64))
    scale = torch.cat([torch.cat(sc) * noise, 1.6 * 2.0 ** torch.clamp(e, max=5.0)])
    view = torch.cat([view, torch.from_numpy(np.repeat(np.arange(n), n_cl)).cuda()])
    order = torch.argsort(view + torch.rand(len(view), generator=g, device="cuda", dtype=torch.float64))
    return (n_vis + n_cl, pairs, desc[order].contiguous(), kp[order].float().contiguous(),
            scale[order].float().contiguous(), _view_F(cams, pairs))


def _inputs(case, seed):
    g = _gen(seed)
    d = {"R": np.random.default_rng([seed, 13]).standard_normal(
        (case["code_bits"] + case["n_tables"] * case["bits"], DIM)), "kpts": None, "scale": None, "F": None}
    if case["images"] == "views":
        sizes, d["pairs"], d["desc"], d["kpts"], d["scale"], F = _views(case, g)
        d["F"] = torch.from_numpy(F).cuda()
    else:
        sizes, d["pairs"], near = _layout(case)
        d["desc"] = _photo_desc(g, sizes, near)
    d["off"] = _offsets(sizes)
    if case["op"] == "ga":
        d["words"] = torch.randint(-2 ** 31, 2 ** 31, (len(d["pairs"]), 256, 8), generator=g, device="cuda").int()
    return d


def _capacity(case, off, pairs):
    """Room for the match lists: every query for short lists and overlapping views, else an eighth of them."""
    queries = int((off[pairs[:, 0].astype(np.int64) + 1] - off[pairs[:, 0].astype(np.int64)]).sum())
    return queries if len(pairs) < 200 or case["images"] == "views" else queries // 8


def prepare(case, seed):
    d = _inputs(case, seed)
    p = ch.cashash_default_params(code_bits=case["code_bits"], n_tables=case["n_tables"],
                                  bits_per_table=case["bits"], top_k=case["top_k"], tau=case["tau"],
                                  flags=case["flags"], precision=case["precision"], schedule=case["schedule"],
                                  epi_px=case["epi_px"])
    st = {"op": case["op"], "pairs": d["pairs"], "ctx": ch.cashash_create(p, d["R"])}
    st["cap"] = _capacity(case, d["off"], d["pairs"])
    if case["op"] == "host":
        st.update(desc=d["desc"].cpu().pin_memory(), off=d["off"], moff=np.zeros(len(d["pairs"]) + 1, np.uint64),
                  mt=np.zeros((st["cap"], 2), np.uint32))
        return st
    st["set"] = ch.DeviceSet(p, d["off"], d["desc"], d["kpts"])
    if case["op"] == "build":
        return st
    ch.cashash_build_codes(st["ctx"], st["set"])
    if case["op"] == "ga":
        st.update(scale=d["scale"], words=d["words"], mean=ch.cashash_get_mean(st["ctx"]))
        return st
    st.update(F=d["F"] if case["epi_px"] >= 0 else None,
              moff=torch.zeros(len(d["pairs"]) + 1, dtype=torch.int64, device="cuda"),
              mt=torch.zeros((st["cap"], 2), dtype=torch.int32, device="cuda"))
    if case["op"] == "match":
        st["plan"] = ch.cashash_plan_create(st["ctx"], st["set"], d["pairs"])
    return st


def run(state):
    op, ctx = state["op"], state["ctx"]
    if op == "build":
        s = state["set"]
        ch.cashash_build_codes(ctx, s)
        return {"codes": s.codes, "buckets": s.buckets, "sqnorm": s.sqnorm}
    if op == "host":
        ch.cashash_run_host(ctx, state["desc"], state["off"], state["pairs"], state["cap"], match_off=state["moff"],
                            matches=state["mt"])
        return {"match_off": state["moff"], "matches": state["mt"]}
    if op == "ga":
        F, info = ch.cashash_ga_stage1(ctx, state["set"], state["scale"], state["mean"], state["pairs"],
                                       state["words"])
        return {"F": F, "info": info}
    if op == "pairs":
        ch.cashash_match_pairs(ctx, state["set"], state["pairs"], state["moff"], state["mt"], state["cap"],
                               F=state["F"])
    else:
        ch.cashash_match_plan(ctx, state["plan"], state["moff"], state["mt"], state["cap"], F=state["F"])
    return {"match_off": state["moff"], "matches": state["mt"]}


# ---------------------------------------------------------------------------
# the work a pass cannot do without
# ---------------------------------------------------------------------------

VIEW_KPTS, VIEW_NEIGHBOURS = 7950, 28   # per view of the camera path above, on average


def _candidates(case):
    sizes, pairs, _ = _layout(case)
    return float((sizes[pairs[:, 0]] * sizes[pairs[:, 1]]).sum()) * case["n_tables"] / (1 << case["bits"])


MOST_CANDIDATES = 9.0e9   # of a drawn pair list: below the largest listed one's


def work(case):
    """Bytes: every input read once, every output written once.  Flops: the projection (2 x rows x 128 per
    feature) and one Hamming distance (2 x code bits) per candidate that shares a bucket with its query, at
    the number of candidates of evenly filled buckets; squared distances of the k ranked candidates."""
    T, k, nb = case["n_tables"], case["top_k"], float(1 << case["bits"])
    rows = case["code_bits"] + T * case["bits"]
    if case["images"] == "views":
        n = case["n_images"]
        P = n * VIEW_NEIGHBOURS * max(0.2, 1 - 14 / n)
        share = 0.2 if case["op"] == "ga" else 1.0
        N, Q = n * VIEW_KPTS * share, P * VIEW_KPTS * share
        cand = Q * T * VIEW_KPTS * share / nb
    else:
        sizes, pairs, _ = _layout(case)
        P, N = len(pairs), float(sizes.sum())
        sa, sb = sizes[pairs[:, 0]].astype(float), sizes[pairs[:, 1]].astype(float)
        Q, cand = float(sa.sum()), _candidates(case)
        if case["flags"] & ch.CASHASH_FLAG_MUTUAL:
            Q, cand = Q + float(sb.sum()), 2 * cand
    build = {"bytes": N * (DIM + 16 + 8 + 4 + T * 20), "flops": N * 2 * rows * DIM}
    match = {"bytes": N * (DIM + 16 + 8 + 4 + T * 20) + 8 * (P + 1),
             "flops": cand * 2 * case["code_bits"] + Q * k * 2 * DIM}
    if case["epi_px"] >= 0:
        match["bytes"] += N * 8 + P * 72
    if case["op"] == "build":
        return build
    if case["op"] in ("host", "ga"):
        return {"bytes": build["bytes"] + match["bytes"], "flops": build["flops"] + match["flops"]}
    return match


# ---------------------------------------------------------------------------
# the results in 64 bits, by plain torch and numpy
# ---------------------------------------------------------------------------

def _exact_codes(desc, mu, R, case):
    """Bits of the projections: codes [n][code_bits] and short codes [n][tables] (int64)."""
    n, cb, T, m = len(desc), case["code_bits"], case["n_tables"], case["bits"]
    bits = torch.empty((n, R.shape[0]), dtype=torch.bool, device="cuda")
    Rt = torch.from_numpy(np.ascontiguousarray(R.T)).cuda()
    for s in range(0, n, 1 << 18):
        bits[s:s + (1 << 18)] = (desc[s:s + (1 << 18)].double() - mu) @ Rt > 0
    w = 2 ** torch.arange(m, device="cuda")
    return bits[:, :cb], (bits[:, cb:].reshape(n, T, m).long() * w).sum(-1)


def _mean(desc):
    return desc.sum(0, dtype=torch.int64).double() / max(len(desc), 1)


def _exact_pair(A, B, case, F=None):
    """Matches of one pair as an array over the queries: candidate index or -1.  A and B hold the images'
    descriptors, code bits, short codes and key-points."""
    k, cb = case["top_k"], case["code_bits"]
    nB = len(B[0])
    out = torch.full((len(A[0]),), -1, dtype=torch.int64, device="cuda")
    big = 1 << 40
    for s in range(0, len(out), 4096):
        a = [x[s:s + 4096] if x is not None else None for x in A]
        H = ((cb - (2.0 * a[1].float() - 1) @ (2.0 * B[1].float() - 1).T) / 2).long()
        ok = torch.zeros_like(H, dtype=torch.bool)
        for t in range(case["n_tables"]):
            ok |= a[2][:, t, None] == B[2][None, :, t]
        ok &= H <= case["tau"]
        if F is not None:
            f, x, y = F.tolist(), a[3][:, 0].double(), a[3][:, 1].double()
            la, lb, lc = (((f[3 * r] * x + f[3 * r + 1] * y) + f[3 * r + 2])[:, None] for r in range(3))
            num = (la * B[3][None, :, 0].double() + lb * B[3][None, :, 1].double()) + lc
            ok &= num * num <= case["epi_px"] ** 2 * (la * la + lb * lb)
        key = torch.where(ok, H * (1 << 24) + torch.arange(nB, device="cuda"), big)
        key = torch.topk(key, min(k, nB), dim=1, largest=False).values
        j = key % (1 << 24) * (key < big)
        da, db = a[0].double()[:, None, :], B[0][j].double()
        d = ((da - db) ** 2).sum(-1).long()
        dj = torch.where(key < big, d * (1 << 24) + j, big * (1 << 20)).sort(dim=1).values
        n = (key < big).sum(1)
        d1 = dj[:, 0] >> 24
        d2 = dj[:, min(1, dj.shape[1] - 1)] >> 24
        hit = (n >= 2) & (25 * d1 < 16 * d2)
        if case["flags"] & ch.CASHASH_FLAG_ACCEPT_SINGLE:
            hit |= n == 1
        out[s:s + 4096] = torch.where(hit, dj[:, 0] % (1 << 24), -1)
    return out


def _exact_matches(d, case):
    """Per pair: the matched (query, candidate) rows."""
    mu = _mean(d["desc"])
    code, short = _exact_codes(d["desc"], mu, d["R"], case)
    return _match_lists(d["desc"], code, short, d["kpts"], d["off"], d["pairs"], case,
                        d["F"] if case["epi_px"] >= 0 else None)


def _match_lists(desc, code, short, kpts, off, pairs, case, F):
    o = off.astype(np.int64)

    def image(i):
        r = slice(o[i], o[i + 1])
        return [desc[r], code[r], short[r], kpts[r] if kpts is not None else None]

    out = []
    for p, (a, b) in enumerate(pairs.astype(np.int64)):
        A, B = image(a), image(b)
        Fp = None if F is None else F[p].reshape(3, 3)
        m = _exact_pair(A, B, case, None if Fp is None else Fp.ravel())
        q = torch.nonzero(m >= 0).ravel()
        if case["flags"] & ch.CASHASH_FLAG_MUTUAL:
            back = _exact_pair(B, A, case, None if Fp is None else Fp.T.ravel())
            q = q[back[m[q]] == q]
        out.append(torch.stack([q, m[q]], dim=1))
    return out


def _sampson2(F, xa, xb):
    Fx, Ft = xa @ F.T, xb @ F
    return (xb * Fx).sum(1) ** 2 / (Fx[:, 0] ** 2 + Fx[:, 1] ** 2 + Ft[:, 0] ** 2 + Ft[:, 1] ** 2)


def _low_rank(F):
    U, S, V = np.linalg.svd(F)
    S[..., 2] = 0
    return (U * S[..., None, :]) @ V


def _exact_F(pa, pb, words):
    """RANSAC over normalised 8-point samples with the documented draws, batches and stop; the refit on the
    winner's inliers, unit norm, its largest entry positive.  Returns F and the five info words."""
    m = len(pa)
    if m < 16:
        return np.zeros(9), [m, 0, -1, 0, 0]
    xa, xb = np.c_[pa, np.ones(m)], np.c_[pb, np.ones(m)]
    Ts = []
    for p in (pa, pb):
        c = p.mean(0)
        s = math.sqrt(2) / np.sqrt(((p - c) ** 2).sum(1)).mean()
        Ts.append(np.array([[s, 0, -s * c[0]], [0, s, -s * c[1]], [0, 0, 1]]))
    rows = np.einsum("ni,nj->nij", xb @ Ts[1].T, xa @ Ts[0].T).reshape(m, 9)
    best, best_h, best_F, done = -1, -1, None, 0
    while done < 256:
        idx = []
        for h in range(done, done + 32):
            left = list(range(m)) if m < 64 else None
            got = []
            for k in range(8):
                r = (int(words[h, k]) * (m - k)) >> 32
                if left is not None:
                    got.append(left.pop(r))
                else:
                    for g in sorted(got):
                        r += g <= r
                    got.append(r)
            idx.append(got)
        null = np.linalg.svd(rows[np.array(idx)])[2][:, -1].reshape(-1, 3, 3)
        Fs = Ts[1].T @ _low_rank(null) @ Ts[0]
        for h, F in enumerate(Fs):
            n = int((_sampson2(F, xa, xb) <= 9.0).sum())
            if n > best:
                best, best_h, best_F = n, done + h, F
        done += 32
        if (1 - (best / m) ** 8) ** done <= 1 - 0.99:
            break
    inl = _sampson2(best_F, xa, xb) <= 9.0
    if inl.sum() >= 8:
        best_F = Ts[1].T @ _low_rank(np.linalg.svd(rows[inl])[2][-1].reshape(3, 3)) @ Ts[0]
    f = (best_F / np.linalg.norm(best_F)).ravel()
    f *= math.copysign(1.0, f[np.argmax(np.abs(f))])
    n = int((_sampson2(f.reshape(3, 3), xa, xb) <= 9.0).sum())
    return f, [m, n, best_h, int(3 * n >= 2 * m), done]


def _exact_ga(d, case):
    off = d["off"].astype(np.int64)
    scale = d["scale"].cpu().numpy()
    sel, sub = [], [0]
    for i in range(len(off) - 1):
        n = off[i + 1] - off[i]
        k = -(-n * 20 // 100)
        order = np.lexsort((np.arange(n), -scale[off[i]:off[i + 1]].astype(np.float64)))
        sel.append(np.sort(order[:k]) + off[i])
        sub.append(sub[-1] + k)
    pick = torch.from_numpy(np.concatenate(sel)).cuda()
    desc = d["desc"][pick]
    code, short = _exact_codes(desc, _mean(d["desc"]), d["R"], case)
    sub = np.array(sub, np.uint64)
    kp = d["kpts"][pick].cpu().numpy().astype(np.float64)
    words = d["words"].cpu().numpy().view(np.uint32)
    F, info = [], []
    for p, mt in enumerate(_match_lists(desc, code, short, None, sub, d["pairs"], case, None)):
        a, b = (int(sub[i]) for i in d["pairs"][p])
        q = mt.cpu().numpy()
        f, w = _exact_F(kp[a + q[:, 0]], kp[b + q[:, 1]], words[p])
        F.append(f)
        info.append(w)
    return {"F": torch.from_numpy(np.array(F)).cuda(), "info": torch.tensor(info, dtype=torch.int32, device="cuda")}


def exact(case, seed):
    """What run() returns, from float64 projections and dense comparisons of whole images; None where a pair
    list is too long for that."""
    if case["op"] == "ga" and case["n_images"] > 60:
        return None
    if case["op"] in ("match", "pairs", "host"):
        w = work(case)["flops"] * 2.0 ** case["bits"] / (2 * case["code_bits"] * case["n_tables"])
        if w > 1.5e10:
            return None
    d = _inputs(case, seed)
    if case["op"] == "ga":
        return _exact_ga(d, case)
    if case["op"] == "build":
        code, short = _exact_codes(d["desc"], _mean(d["desc"]), d["R"], case)
        n = len(code)
        w = torch.zeros((n, 4), dtype=torch.int64, device="cuda")
        shift = 2 ** torch.arange(32, device="cuda")
        for k in range(case["code_bits"] // 32):
            w[:, k] = (code[:, 32 * k:32 * k + 32].long() * shift).sum(1)
        bk = torch.zeros((n, 8), dtype=torch.uint8, device="cuda")
        bk[:, :case["n_tables"]] = short.to(torch.uint8)
        sq = (d["desc"].int() ** 2).sum(1, dtype=torch.int64)
        return {"codes": (w - (w >> 31) * 2 ** 32).int(), "buckets": bk, "sqnorm": sq.int()}
    lists = _exact_matches(d, case)
    off = np.zeros(len(lists) + 1, np.int64)
    off[1:] = np.cumsum([len(x) for x in lists])
    mt = torch.cat(lists) if lists else torch.zeros((0, 2), dtype=torch.int64, device="cuda")
    full = torch.zeros((_capacity(case, d["off"], d["pairs"]), 2), dtype=torch.int32, device="cuda")
    full[:len(mt)] = mt.int()
    if case["op"] == "host":
        return {"match_off": off.astype(np.uint64), "matches": full.cpu().numpy().view(np.uint32)}
    return {"match_off": torch.from_numpy(off).cuda(), "matches": full}
