"""The work that users of this library have it do, as cases that can be timed and compared.

Every case is one public call, or the short chain of calls that a program makes with it: a
sparse uplift of a scene (each of its forms), a rendered view with the decode and the text query,
a training step's forward and backward, and the Top-K filter of an accumulator.  Scenes, cameras,
region maps and codes are drawn on the GPU with the shapes and distributions of this repository's
synthetic workloads (blob or uniform Gaussians, log-scales N(-4, 0.5), opacities sigmoid(N(0, 1.5)),
cameras on a band of radius 3, Voronoi region maps, Dirichlet region codes).

Top-K atom ids are returned where they come from a given accumulator.  An uplift returns the
accumulator itself and the coefficients: two runs of one uplift add in another order, so atoms of
equal coefficients (to FP32 rounding) change places in the id list from run to run.

`exact` composites in 64 bits with plain torch: tiles of 16 x 16 pixels, 32 list entries at a time.
"""
import math
import random
from types import SimpleNamespace

import numpy as np
import torch

import paper_2605_13600_gb300 as gb
from paper_2605_13600_gb300.autograd import SparseRender

DEV = "cuda"
TILE = 16


def listed():
    return [
        # the smallest uplift: a preview of 8 thumbnails (the repository's 10k-Gaussian workload); launches count
        dict(name="uplift_thumbnails", kind="uplift", form="views", n=10_000, V=8, W=160, H=120, R=32, C=64, s=4, K=4,
             layout="uniform"),
        # a room-sized object scan with the paper's codebook (64 atoms, 4 per code), default form of the wrapper
        dict(name="uplift_room", kind="uplift", form="views", n=300_000, V=24, W=640, H=480, R=100, C=64, s=4, K=4,
             layout="blobs"),
        # the repository's headline: 1M Gaussians, 200 views, the chunked form
        dict(name="uplift_scene", kind="uplift", form="chunked", n=1_000_000, V=200, W=988, H=731, R=200, C=256, s=8,
             K=8, layout="blobs"),
        # region maps that stay in pinned host memory and are staged while views compute
        dict(name="uplift_host_maps", kind="uplift", form="host", n=1_000_000, V=25, W=988, H=731, R=200, C=256, s=8,
             K=8, layout="blobs"),
        # the three semantic levels of one scene in one pass
        dict(name="uplift_levels", kind="levels", n=500_000, V=12, W=800, H=600, R=200, C=256, s=8, K=8,
             layout="blobs"),
        # many scenes of uneven size through one captured graph
        dict(name="uplift_batch", kind="batch", scenes=5, n=80_000, n_max=900_000, V=8, W=648, H=484, R=200, C=256, s=8,
             K=8, layout="blobs"),
        # a small preview frame in FP32 codes, as an interactive viewer asks for it
        dict(name="render_preview", kind="render", n=10_000, W=161, H=119, C=64, K=4, dtype="f32", layout="uniform"),
        # a served 1080p frame: rendered bf16 codes, then features and the similarity to 32 phrases in one call
        dict(name="frame_query_1080p", kind="frame", n=1_000_000, W=1920, H=1080, C=256, K=8, D=512, Q=32, canon=0,
             layout="blobs"),
        # training through the render: forward and gradients of one 800 x 600 view
        dict(name="train_render", kind="train_render", n=500_000, W=800, H=600, C=256, K=8, layout="blobs"),
        # the other half of that step: decode, region loss and its gradient back to the codes
        dict(name="train_head", kind="train_head", W=800, H=600, C=256, D=512, R=200, s=8),
        # decode, similarity and relevancy of a cropped window of pixels as separate calls, FP32 codes
        dict(name="query_crop", kind="query", P=1221, C=64, D=512, Q=16, canon=4, dtype="f32"),
        # the Top-K, the entropy and the entropy filter of a finished accumulator
        dict(name="topk_filter", kind="topk", n=1_000_000, C=256, K=8),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["uplift", "uplift", "uplift", "levels", "batch", "render", "frame", "train_render",
                       "train_head", "query", "topk"])
    W = rng.randint(150, 1300)
    H = max(100, min(980, int(W * rng.uniform(0.55, 0.8))))
    C, K = rng.choice([(32, 4), (64, 4), (64, 8), (128, 8), (200, 6), (256, 8)])
    layout = rng.choice(["blobs", "blobs", "uniform"])
    if kind == "uplift":
        form = rng.choice(["views", "chunked", "host", "compensated"])
        return dict(kind=kind, form=form, n=_log(rng, 5_000, 1_000_000), V=_log(rng, 1, 40), W=W, H=H,
                    R=rng.randint(8, 200), C=C, s=K, K=K, layout=layout)
    if kind == "levels":
        return dict(kind=kind, n=_log(rng, 10_000, 600_000), V=_log(rng, 1, 12), W=W, H=H, R=rng.randint(40, 200), C=C,
                    s=K, K=K, layout=layout)
    if kind == "batch":
        n = _log(rng, 10_000, 200_000)
        return dict(kind=kind, scenes=rng.randint(2, 6), n=n, n_max=n * rng.randint(1, 5), V=rng.randint(2, 10), W=W,
                    H=H, R=rng.randint(8, 200), C=C, s=K, K=K, layout=layout)
    if kind == "render":
        return dict(kind=kind, n=_log(rng, 5_000, 1_000_000), W=W, H=H, C=C, K=K, dtype=rng.choice(["f32", "bf16"]),
                    layout=layout)
    if kind == "frame":
        return dict(kind=kind, n=_log(rng, 20_000, 1_000_000), W=W, H=H, C=C, K=K, D=rng.choice([256, 512, 768]),
                    Q=rng.choice([16, 32]), canon=rng.choice([0, 4]), layout=layout)
    if kind == "train_render":
        return dict(kind=kind, n=_log(rng, 10_000, 600_000), W=min(W, 1000), H=min(H, 750), C=C, K=K, layout=layout)
    if kind == "train_head":
        return dict(kind=kind, W=min(W, 1000), H=min(H, 750), C=rng.choice([64, 128, 256]), D=rng.choice([256, 512, 768]),
                    R=rng.randint(8, 200), s=K)
    if kind == "query":
        return dict(kind=kind, P=_log(rng, 500, 1_000_000), C=rng.choice([64, 128, 256]), D=rng.choice([256, 512, 768]),
                    Q=rng.choice([16, 32]), canon=4, dtype=rng.choice(["f32", "bf16"]))
    return dict(kind=kind, n=_log(rng, 5_000, 1_000_000), C=C, K=K)


# ---------------------------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------------------------

def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed) & 0x7FFFFFFF)


def _scene(g, n, layout):
    def normal(*shape):
        return torch.randn(*shape, generator=g, device=DEV)

    blob = torch.zeros(n, dtype=torch.int64, device=DEV)
    if layout == "uniform":
        means = torch.rand(n, 3, generator=g, device=DEV) * 2 - 1
    else:
        centres = torch.rand(64, 3, generator=g, device=DEV) * 2 - 1
        blob = torch.randint(0, 64, (n,), generator=g, device=DEV)
        means = centres[blob] + 0.2 * normal(n, 3)
    return SimpleNamespace(n=n, means=means.contiguous(), scales=torch.exp(0.5 * normal(n, 3) - 4.0),
                           quats=torch.nn.functional.normalize(normal(n, 4), dim=1),
                           opacity=torch.sigmoid(1.5 * normal(n)), blob=blob)


def _cameras(rnd, V, W, H):
    """Pinhole cameras on a sphere band of radius 3 (elevation -20 to 30 degrees), looking at the origin, 60 degrees."""
    f = W / (2.0 * math.tan(math.radians(60.0) / 2.0))
    cams = []
    for k in range(V):
        el, az = math.radians(rnd.uniform(-20.0, 30.0)), 2.0 * math.pi * (k + rnd.random()) / V
        c = 3.0 * np.array([math.cos(el) * math.cos(az), math.cos(el) * math.sin(az), math.sin(el)])
        z = -c / np.linalg.norm(c)
        x = np.cross(z, [0.0, 0.0, 1.0])
        x /= np.linalg.norm(x)
        R = np.stack([x, np.cross(z, x), z])
        vm = np.concatenate([R, (-R @ c)[:, None]], axis=1).reshape(12).astype(np.float32)
        cams.append(SimpleNamespace(viewmat=vm, fx=float(np.float32(f)), fy=float(np.float32(f)), cx=W / 2.0, cy=H / 2.0,
                                    width=W, height=H))
    return cams


def _regions(g, R, W, H):
    """Voronoi partition of one view into R cells (squared distances are exact in FP32 at these sizes)."""
    sx = torch.randint(0, W, (R,), generator=g, device=DEV).float()
    sy = torch.randint(0, H, (R,), generator=g, device=DEV).float()
    dx = (torch.arange(W, device=DEV).float()[:, None] - sx) ** 2
    dy = (torch.arange(H, device=DEV).float()[:, None] - sy) ** 2
    return (dy[:, None, :] + dx[None, :, :]).argmin(dim=2).to(torch.int32).reshape(-1)


def _codes(g, rows, C, s):
    """s distinct atoms per row with Dirichlet(1) coefficients."""
    idx = torch.rand(rows, C, generator=g, device=DEV).topk(s, dim=1).indices.to(torch.int32)
    w = torch.empty(rows, s, device=DEV).exponential_(generator=g)
    return idx.contiguous(), w / w.sum(dim=1, keepdim=True)


def _workload(g, rnd, case, n, V, scene=None, cams=None):
    W, H, R, C, s = case["W"], case["H"], case["R"], case["C"], case["s"]
    scene = scene or _scene(g, n, case["layout"])
    cams = cams or _cameras(rnd, V, W, H)
    maps = torch.empty(V * W * H, dtype=torch.int32, device=DEV)
    for v in range(V):
        maps[v * W * H:(v + 1) * W * H] = _regions(g, R, W, H) + v * R
    ci, cv = _codes(g, R * V, C, s)
    offs = np.arange(V + 1, dtype=np.int64) * (W * H)
    return SimpleNamespace(scene=scene, cams=cams, region_maps=maps, map_offsets=offs, code_idx=ci, code_val=cv, C=C,
                           s=s, K=case["K"])


def _gaussian_codes(g, scene, C, K):
    """K-sparse codes as an uplift leaves them: descending, summing to one, the atoms of a blob from its own pool of 32;
    5% of the Gaussians were never seen and hold the padding (-1, 0)."""
    pool = torch.rand(64, C, generator=g, device=DEV).topk(min(32, C), dim=1).indices
    pick = torch.rand(scene.n, pool.shape[1], generator=g, device=DEV).topk(K, dim=1).indices
    idx = torch.gather(pool[scene.blob], 1, pick).to(torch.int32)
    val = torch.empty(scene.n, K, device=DEV).exponential_(generator=g).sort(dim=1, descending=True).values
    val = val / val.sum(dim=1, keepdim=True)
    unseen = torch.rand(scene.n, generator=g, device=DEV) < 0.05
    idx[unseen] = -1
    val[unseen] = 0.0
    return idx.cpu().numpy(), val.cpu().numpy()


def _unit(g, rows, dim):
    return torch.nn.functional.normalize(torch.randn(rows, dim, generator=g, device=DEV), dim=1)


def _rendered_like(g, P, C):
    """Rows like rendered codes: a few dozen atoms per pixel, total weight up to one."""
    x = torch.empty(P, C, device=DEV).exponential_(generator=g)
    x *= torch.rand(P, C, generator=g, device=DEV) < 0.15
    return x / x.sum(dim=1, keepdim=True).clamp_min(1e-3) * torch.rand(P, 1, generator=g, device=DEV)


def _batch_sizes(case):
    B, n0, n1 = case["scenes"], case["n"], case["n_max"]
    return [(int(n0 * (n1 / n0) ** (b / max(1, B - 1))), case["V"] + (b * 3) % 5) for b in range(B)]


def prepare(case, seed):
    g, rnd, kind = _gen(seed), random.Random(seed), case["kind"]
    if kind == "uplift":
        wl = _workload(g, rnd, case, case["n"], case["V"])
        up = gb.Uplift(wl, chunked=case["form"] in ("chunked", "host"), compensated=case["form"] == "compensated")
        host = wl.region_maps.cpu().pin_memory() if case["form"] == "host" else None
        return dict(case=case, wls=[wl], up=up, host=host)
    if kind == "levels":
        base = _workload(g, rnd, case, case["n"], case["V"])
        wls = [base]
        for div in (2, 4):  # coarser levels merge the cells of the finest one
            R = case["R"] // div
            per = case["W"] * case["H"]
            view = torch.arange(case["V"], device=DEV, dtype=torch.int32).repeat_interleave(per)
            cell = (base.region_maps - view * case["R"]) // div
            ci, cv = _codes(g, (R + 1) * case["V"], case["C"], case["s"])
            wls.append(SimpleNamespace(**{**vars(base), "region_maps": cell + view * (R + 1), "code_idx": ci,
                                          "code_val": cv}))
        return dict(case=case, wls=wls, up=gb.LevelUplift(wls))
    if kind == "batch":
        wls = [_workload(g, rnd, case, n, V) for n, V in _batch_sizes(case)]
        return dict(case=case, wls=wls, up=gb.BatchedUplift(wls))
    if kind in ("render", "frame", "train_render"):
        scene = _scene(g, case["n"], case["layout"])
        cam = _cameras(rnd, 1, case["W"], case["H"])[0]
        idx, val = _gaussian_codes(g, scene, case["C"], case["K"])
        r = gb.Render(scene, idx, val, case["C"], [cam])
        P = case["W"] * case["H"]
        st = dict(case=case, r=r, cam=cam, scene=scene)
        if kind == "train_render":
            st["opacity"] = scene.opacity.clone().requires_grad_()
            st["val"] = r.topk_val.clone().requires_grad_()
            st["grad"] = torch.randn(case["H"], case["W"], case["C"], generator=g, device=DEV)
            return st
        bf16 = kind == "frame" or case["dtype"] == "bf16"
        st["out"] = r.outputs(cam, dtype=torch.bfloat16 if bf16 else torch.float32)
        if kind == "frame":
            D, Q, canon = case["D"], case["Q"], case["canon"]
            st["codebook"], st["text"] = _unit(g, case["C"], D), _unit(g, Q, D)
            st["features"] = torch.empty(P, D, dtype=torch.bfloat16, device=DEV)
            st["norm2"] = torch.empty(P, device=DEV)
            st["answer"] = torch.empty(P, Q - canon, device=DEV)
            st["ws"] = torch.empty(gb.scoup_decode_query_workspace_size(P, case["C"], D, Q), dtype=torch.uint8, device=DEV)
        return st
    if kind == "train_head":
        P, C, D, R = case["W"] * case["H"], case["C"], case["D"], case["R"]
        ci, cv = _codes(g, R, C, case["s"])
        return dict(case=case, codes=_rendered_like(g, P, C), codebook=_unit(g, C, D), ci=ci, cv=cv,
                    regions=_regions(g, R, case["W"], case["H"]),
                    feats=torch.empty(P, D, dtype=torch.bfloat16, device=DEV),
                    dfeats=torch.empty(P, D, dtype=torch.bfloat16, device=DEV),
                    dcodes=torch.empty(P, C, device=DEV), loss=torch.zeros((), dtype=torch.float64, device=DEV))
    if kind == "query":
        P, C, D, Q, canon = case["P"], case["C"], case["D"], case["Q"], case["canon"]
        codes = _rendered_like(g, P, C)
        return dict(case=case, codes=codes.bfloat16() if case["dtype"] == "bf16" else codes, codebook=_unit(g, C, D),
                    text=_unit(g, Q, D), feats=torch.empty(P, D, dtype=torch.bfloat16, device=DEV),
                    norm2=torch.empty(P, device=DEV), sim=torch.empty(P, Q, device=DEV),
                    rel=torch.empty(P, Q - canon, device=DEV))
    if kind == "topk":
        n, C, K = case["n"], case["C"], case["K"]
        # rows of a finished uplift: a third of the atoms hold weight, a fifth of the Gaussians was never seen
        acc = torch.empty(n, C, device=DEV).exponential_(generator=g)
        acc *= torch.rand(n, C, generator=g, device=DEV) < 0.6 * torch.rand(n, 1, generator=g, device=DEV)
        acc *= (torch.rand(n, 1, generator=g, device=DEV) > 0.2)
        return dict(case=case, acc=acc, idx=torch.empty(n, K, dtype=torch.int32, device=DEV),
                    val=torch.empty(n, K, device=DEV), entropy=torch.empty(n, device=DEV),
                    keep=torch.empty(n, dtype=torch.uint8, device=DEV),
                    ws=torch.empty(gb.scoup_entropy_filter_workspace_size(), dtype=torch.uint8, device=DEV))
    raise ValueError(kind)


# ---------------------------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------------------------

def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "uplift":
        up = st["up"]
        if st["host"] is not None:
            up.run_host_maps(st["host"], stats=False)
        else:
            up.run(stats=False)
        # the compensated form keeps the running sums first (their terms are what rounding left over)
        return {"accum": up.accum[0] if up.compensated else up.accum, "topk_val": up.topk_val}
    if kind == "levels":
        st["up"].run(stats=False)
        return {"accum": st["up"].accum, "topk_val": st["up"].topk_val}
    if kind == "batch":
        st["up"].run()
        return {"accum": list(st["up"].accum), "topk_val": list(st["up"].topk_val)}
    if kind == "render":
        out, _ = st["r"].run(0, out=st["out"], stats=False)
        return {"codes": out[0], "T": out[1]}
    if kind == "frame":
        out, _ = st["r"].run(0, out=st["out"], stats=False)
        gb.scoup_decode_query(out[0].view(-1, case["C"]), st["codebook"], st["text"], st["answer"],
                              n_canon=case["canon"], features=st["features"], feat_norm2=st["norm2"],
                              workspace=st["ws"])
        return {"codes": out[0], "T": out[1], "features": st["features"], "norm2": st["norm2"], "answer": st["answer"]}
    if kind == "train_render":
        codes = SparseRender.apply(st["opacity"], st["val"], st["r"], 0)
        d_op, d_val = torch.autograd.grad(codes, (st["opacity"], st["val"]), st["grad"])
        return {"codes": codes.detach(), "d_opacity": d_op, "d_val": d_val}
    if kind == "train_head":
        gb.scoup_decode(st["codes"], st["codebook"], st["feats"])
        st["loss"].zero_()
        gb.scoup_region_l2_grad(st["feats"], st["regions"], st["ci"], st["cv"], st["codebook"], st["dfeats"], st["loss"])
        gb.scoup_decode_backward(st["dfeats"], st["codebook"], st["dcodes"])
        return {"features": st["feats"], "dfeatures": st["dfeats"], "dcodes": st["dcodes"], "loss": st["loss"].float()}
    if kind == "query":
        gb.scoup_decode(st["codes"], st["codebook"], st["feats"], feat_norm2=st["norm2"])
        gb.scoup_similarity(st["feats"], st["text"], st["sim"], feat_norm2=st["norm2"])
        gb.scoup_relevancy(st["sim"], case["canon"], st["rel"])
        return {"features": st["feats"], "norm2": st["norm2"], "similarity": st["sim"], "relevancy": st["rel"]}
    gb.scoup_topk_entropy(st["acc"], case["K"], st["idx"], st["val"], st["entropy"])
    gb.scoup_entropy_filter(st["entropy"], case["n"] // 2, st["idx"], st["val"], st["keep"], workspace=st["ws"])
    return {"idx": st["idx"], "val": st["val"], "entropy": st["entropy"], "keep": st["keep"]}


# ---------------------------------------------------------------------------------------------
# work that a pass cannot do without
# ---------------------------------------------------------------------------------------------

PAIRS, PAIR_FLOPS = 60, 15  # (Gaussian, pixel) pairs a pixel looks at before it is opaque, and the operations of one


def work(case):
    kind = case["kind"]
    if kind in ("uplift", "levels", "batch"):
        L = 3 if kind == "levels" else 1
        sizes = _batch_sizes(case) if kind == "batch" else [(case["n"], case["V"])]
        px, C, K = case["W"] * case["H"], case["C"], case["K"]
        nbytes = sum(44 * n + L * (4 * px * V + 8 * case["R"] * V * case["s"] + 4 * n * C + 8 * n * K) for n, V in sizes)
        return {"bytes": nbytes, "flops": sum(PAIRS * PAIR_FLOPS * px * V for _, V in sizes)}
    if kind in ("render", "frame", "train_render"):
        n, px, C, K = case["n"], case["W"] * case["H"], case["C"], case["K"]
        nbytes, flops = 44 * n + 8 * n * K, PAIRS * PAIR_FLOPS * px
        if kind == "render":
            return {"bytes": nbytes + px * (C * (2 if case["dtype"] == "bf16" else 4) + 8), "flops": flops}
        if kind == "frame":
            D, Q = case["D"], case["Q"]
            return {"bytes": nbytes + px * (2 * C + 8 + 2 * D + 4 + 4 * (Q - case["canon"])) + 4 * D * (C + Q),
                    "flops": flops + 2.0 * px * C * (D + Q)}
        return {"bytes": 2 * nbytes + px * 8 * C + 4 * n * (K + 1), "flops": 3 * flops}
    if kind == "train_head":
        P, C, D = case["W"] * case["H"], case["C"], case["D"]
        return {"bytes": P * (4 * C + 2 * D + 2 * D + 4 * C + 4) + 4 * C * D, "flops": 4.0 * P * C * D}
    if kind == "query":
        P, C, D, Q = case["P"], case["C"], case["D"], case["Q"]
        return {"bytes": P * ((2 if case["dtype"] == "bf16" else 4) * C + 2 * D + 4 + 4 * Q + 4 * (Q - case["canon"])),
                "flops": 2.0 * P * D * (C + Q)}
    n, C, K = case["n"], case["C"], case["K"]
    return {"bytes": n * (4 * C + 8 * K + 4 + 1), "flops": 4.0 * n * C}


# ---------------------------------------------------------------------------------------------
# the same in 64 bits
# ---------------------------------------------------------------------------------------------

def _project(scene, cam):
    """Standard 3DGS projection: pixel means, conics, depth, tile rectangles [x0, y0, x1, y1) (empty if culled)."""
    W = torch.tensor(np.asarray(cam.viewmat, np.float64).reshape(3, 4), device=DEV)
    t = scene.means.double() @ W[:, :3].T + W[:, 3]
    q = torch.nn.functional.normalize(scene.quats.double(), dim=1)
    w, x, y, z = q.unbind(1)
    rot = torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                       2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                       2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)], 1).view(-1, 3, 3)
    M = rot * scene.scales.double()[:, None, :]
    cov = M @ M.transpose(1, 2)
    tz = t[:, 2].clamp_min(1e-6)
    lx, ly = 1.3 * 0.5 * cam.width / cam.fx, 1.3 * 0.5 * cam.height / cam.fy
    tx, ty = (t[:, 0] / tz).clamp(-lx, lx) * tz, (t[:, 1] / tz).clamp(-ly, ly) * tz
    zero = torch.zeros_like(tz)
    J = torch.stack([cam.fx / tz, zero, -cam.fx * tx / tz ** 2, zero, cam.fy / tz, -cam.fy * ty / tz ** 2], 1)
    A = J.view(-1, 2, 3) @ W[:, :3]
    c2 = A @ cov @ A.transpose(1, 2)
    a, b, c = c2[:, 0, 0] + 0.3, c2[:, 0, 1], c2[:, 1, 1] + 0.3
    det = a * c - b * b
    mid = 0.5 * (a + c)
    r = torch.ceil(3.0 * torch.sqrt(mid + torch.sqrt((mid * mid - det).clamp_min(0.1))))
    mx, my = cam.fx * t[:, 0] / tz + cam.cx - 0.5, cam.fy * t[:, 1] / tz + cam.cy - 0.5
    gx, gy = -(-cam.width // TILE), -(-cam.height // TILE)

    def clip(v, hi):
        return torch.floor(v / TILE).clamp(0, hi).long()

    x0, x1, y0, y1 = clip(mx - r, gx), clip(mx + r + 15, gx), clip(my - r, gy), clip(my + r + 15, gy)
    ok = (t[:, 2] > 0.2) & (det > 0) & (x1 > x0) & (y1 > y0)
    x1, y1 = torch.where(ok, x1, x0), torch.where(ok, y1, y0)
    return SimpleNamespace(mx=mx, my=my, qa=-0.5 * c / det, qb=b / det, qc=-0.5 * a / det, z=t[:, 2], x0=x0, y0=y0,
                           x1=x1, y1=y1, gx=gx, gy=gy)


def _tile_lists(p):
    """Gaussians of every tile front to back (ids, packed) and the tiles' first positions."""
    w = p.x1 - p.x0
    cnt = w * (p.y1 - p.y0)
    order = torch.argsort(p.z, stable=True)
    order = order[cnt[order] > 0]
    ids = torch.repeat_interleave(order, cnt[order])
    first = torch.cumsum(cnt[order], 0) - cnt[order]
    k = torch.arange(ids.numel(), device=DEV) - torch.repeat_interleave(first, cnt[order])
    tile = (p.y0[ids] + k // w[ids]) * p.gx + p.x0[ids] + k % w[ids]
    tile, perm = torch.sort(tile, stable=True)
    return ids[perm], torch.searchsorted(tile, torch.arange(p.gx * p.gy + 1, device=DEV))


def _composite(scene, cam, visit):
    """Front to back over all tiles, 32 entries at a time: visit(tiles, ids, weight, alpha, gauss, T_before) with the
    weights e [tiles, 32, 256]; returns the final transmittance [tiles, 256]."""
    p = _project(scene, cam)
    ids, start = _tile_lists(p)
    o = scene.opacity.double()
    n_tiles = p.gx * p.gy
    px = torch.arange(256, device=DEV)
    T = torch.ones(n_tiles, 256, dtype=torch.float64, device=DEV)
    tt = torch.arange(n_tiles, device=DEV)
    X = ((tt % p.gx) * TILE)[:, None] + px % TILE
    Y = ((tt // p.gx) * TILE)[:, None] + px // TILE
    done = (X >= cam.width) | (Y >= cam.height)
    at = 0
    while ids.numel():
        act = tt[(start[1:] - start[:-1] > at) & ~done.all(dim=1)]
        if not act.numel():
            break
        pos = start[act][:, None] + at + torch.arange(32, device=DEV)
        real = pos < start[act + 1][:, None]
        g = torch.where(real, ids[pos.clamp_max(ids.numel() - 1)], 0)
        dx = p.mx[g][:, :, None] - X[act][:, None, :]
        dy = p.my[g][:, :, None] - Y[act][:, None, :]
        power = p.qa[g][:, :, None] * dx * dx + p.qb[g][:, :, None] * dx * dy + p.qc[g][:, :, None] * dy * dy
        G = torch.exp(power)
        alpha = (o[g][:, :, None] * G).clamp_max(0.99)
        alpha = torch.where((alpha >= 1.0 / 255.0) & (power <= 0) & real[:, :, None] & ~done[act][:, None, :], alpha, 0.0)
        after = T[act][:, None, :] * torch.cumprod(1.0 - alpha, dim=1)
        take = after >= 1e-4
        before = torch.cat([T[act][:, None, :], after[:, :-1]], dim=1)
        visit(act, g, torch.where(take, alpha * before, 0.0), alpha, G, before)
        T[act] = torch.where(take, after, 1.0).amin(dim=1).minimum(T[act])
        done[act] |= ~take[:, -1]
        at += 32
    return T


def _untile(x, cam):
    """[tiles, 256, ...] to [H, W, ...]."""
    gx, gy = -(-cam.width // TILE), -(-cam.height // TILE)
    x = x.view(gy, gx, TILE, TILE, *x.shape[2:]).transpose(1, 2).reshape(gy * TILE, gx * TILE, *x.shape[2:])
    return x[:cam.height, :cam.width].contiguous()


def _tiled(x, cam, fill=0):
    """[H, W, ...] to [tiles, 256, ...]."""
    gx, gy = -(-cam.width // TILE), -(-cam.height // TILE)
    full = torch.full((gy * TILE, gx * TILE, *x.shape[2:]), fill, dtype=x.dtype, device=DEV)
    full[:cam.height, :cam.width] = x
    return full.view(gy, TILE, gx, TILE, *x.shape[2:]).transpose(1, 2).reshape(gy * gx, TILE * TILE, *x.shape[2:])


def _dense(idx, val, C):
    """Sparse rows [n, s] (atom -1: padding) to dense [n, C], FP64."""
    out = torch.zeros(idx.shape[0], C, dtype=torch.float64, device=DEV)
    return out.scatter_add_(1, idx.long().clamp_min(0), torch.where(idx >= 0, val.double(), 0.0))


def _exact_uplift(wls, K):
    """accum [n, L C] and the Top-K coefficients [L, n, K] of workloads that share scene and views."""
    base = wls[0]
    n, C = base.scene.n, base.C
    acc = torch.zeros(n, len(wls) * C, dtype=torch.float64, device=DEV)
    tables = [_dense(w.code_idx, w.code_val, C) for w in wls]
    for v, cam in enumerate(base.cams):
        lo, hi = int(base.map_offsets[v]), int(base.map_offsets[v + 1])
        pix = [_tiled(w.region_maps[lo:hi].view(cam.height, cam.width).long(), cam) for w in wls]

        def visit(act, g, e, *_):
            per = torch.cat([torch.bmm(e, t[m[act]]) for t, m in zip(tables, pix)], dim=2)
            acc.index_add_(0, g.reshape(-1), per.view(-1, per.shape[2]))

        _composite(base.scene, cam, visit)
    top = [acc[:, l * C:(l + 1) * C].topk(K, dim=1).values for l in range(len(wls))]
    return acc, torch.stack([t / t.sum(dim=1, keepdim=True).clamp_min(1e-300) for t in top])


def _exact_render(st):
    case, cam, r = st["case"], st["cam"], st["r"]
    table = _dense(r.topk_idx, r.topk_val, case["C"])
    n_tiles = -(-cam.width // TILE) * -(-cam.height // TILE)
    What = torch.zeros(n_tiles, 256, case["C"], dtype=torch.float64, device=DEV)

    def visit(act, g, e, *_):
        What[act] += torch.bmm(e.transpose(1, 2), table[g])

    T = _composite(st["scene"], cam, visit)
    return _untile(What, cam), _untile(T, cam)


def _exact_gradients(st):
    case, cam, r = st["case"], st["cam"], st["r"]
    table = _dense(r.topk_idx, r.topk_val, case["C"])
    grad = _tiled(st["grad"].double(), cam)
    S = torch.zeros(grad.shape[0], 256, dtype=torch.float64, device=DEV)
    front = torch.zeros_like(S)
    d_op = torch.zeros(case["n"], dtype=torch.float64, device=DEV)
    d_val = torch.zeros(case["n"], case["K"], dtype=torch.float64, device=DEV)
    atoms = r.topk_idx.long()

    def total(act, g, e, *_):
        S[act] += (e * torch.bmm(table[g], grad[act].transpose(1, 2))).sum(dim=1)

    def gradients(act, g, e, alpha, G, before):
        gw = torch.bmm(table[g], grad[act].transpose(1, 2))
        upto = front[act][:, None, :] + torch.cumsum(e * gw, dim=1)
        d_alpha = before * gw - (S[act][:, None, :] - upto) / (1.0 - alpha)
        d_alpha = torch.where((e > 0) & (alpha < 0.99), G * d_alpha, 0.0)
        front[act] = upto[:, -1]
        d_op.index_add_(0, g.reshape(-1), d_alpha.sum(dim=2).view(-1))
        per_atom = torch.bmm(e, grad[act])
        a = atoms[g]
        d = torch.where(a >= 0, torch.gather(per_atom, 2, a.clamp_min(0)), 0.0)
        d_val.index_add_(0, g.reshape(-1), d.view(-1, case["K"]))

    _composite(st["scene"], cam, total)
    _composite(st["scene"], cam, gradients)
    return d_op, d_val


def _cosines(F, text):
    n = F.norm(dim=1, keepdim=True).clamp_min(1e-300) * text.double().norm(dim=1)
    return F @ text.double().T / n


def _relevancy(sim, canon, alpha=10.0):
    worst = sim[:, :canon].amax(dim=1, keepdim=True)
    return torch.sigmoid(alpha * (sim[:, canon:] - worst))


def exact(case, seed):
    kind = case["kind"]
    if kind in ("uplift", "levels", "batch"):
        sizes = _batch_sizes(case) if kind == "batch" else [(case["n"], case["V"])]
        if sum(V * (case["W"] * case["H"] * case["C"] * (3 if kind == "levels" else 1) + 100 * n) for n, V in sizes) > 8e9:
            return None  # over about 20 seconds
    st = prepare(case, seed)
    if kind == "uplift":
        acc, top = _exact_uplift(st["wls"], case["K"])
        return {"accum": acc, "topk_val": top[0]}
    if kind == "levels":
        acc, top = _exact_uplift(st["wls"], case["K"])
        return {"accum": acc, "topk_val": top}
    if kind == "batch":
        both = [_exact_uplift([w], case["K"]) for w in st["wls"]]
        return {"accum": [a for a, _ in both], "topk_val": [t[0] for _, t in both]}
    if kind == "render":
        What, T = _exact_render(st)
        return {"codes": What, "T": T}
    if kind == "frame":
        What, T = _exact_render(st)
        F = What.view(-1, case["C"]) @ st["codebook"].double()
        sim = _cosines(F, st["text"])
        return {"codes": What, "T": T, "features": F, "norm2": F.square().sum(dim=1),
                "answer": _relevancy(sim, case["canon"]) if case["canon"] else sim}
    if kind == "train_render":
        d_op, d_val = _exact_gradients(st)
        return {"codes": _exact_render(st)[0], "d_opacity": d_op, "d_val": d_val}
    if kind == "train_head":
        cb = st["codebook"].double()
        F = st["codes"].double() @ cb
        d = F - (_dense(st["ci"], st["cv"], case["C"]) @ cb)[st["regions"].long()]
        return {"features": F, "dfeatures": 2 * d, "dcodes": 2 * d @ cb.T, "loss": d.square().sum()}
    if kind == "query":
        F = st["codes"].double() @ st["codebook"].double()
        sim = _cosines(F, st["text"])
        return {"features": F, "norm2": F.square().sum(dim=1), "similarity": sim,
                "relevancy": _relevancy(sim, case["canon"])}
    a = st["acc"].double()
    p = a / a.sum(dim=1, keepdim=True).clamp_min(1e-300)
    ent = -torch.where(a > 0, p * torch.log(p.clamp_min(1e-300)), 0.0).sum(dim=1)
    top = a.topk(case["K"], dim=1).values
    top = top / top.sum(dim=1, keepdim=True).clamp_min(1e-300)
    kept = torch.zeros(case["n"], dtype=torch.bool, device=DEV)
    kept[torch.argsort(ent, stable=True)[:case["n"] // 2]] = True
    return {"idx": None, "val": torch.where(kept[:, None], top, 0.0), "entropy": ent, "keep": None}
