"""The work a user of this library has it do, as timed cases.

Every case goes through the public entry points of the package
(``gazecut.solve_pair``, ``solve_costs``, ``solve_level1``, ``solve_level2``,
``gs_solve_batched``, ``learn.hinge_loss`` and the data-term / adjoint calls)
on synthetic rectified pairs from the package's seeded scene generator, with
the sizes, truncations and weights of its workloads.  The buffers a program
keeps between frames are made in ``prepare``; the images are new for each seed.

Left out: the fixed-sweep mode (its labels depend on the interleaving of
concurrent tiles, so no two runs can be compared value by value) and the
solver state itself (opaque, and one of many maximum flows).
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_1803_01516_gb300 import autotune, learn, metrics, synth
from paper_1803_01516_gb300 import gazecut as gc

THETA = (0.95, 0.9, 40.0, 10.0)      # w1, w2, tau, lambda part of the way through learning
SCALE = 256.0                        # int32 quantisation of the learned data term


def listed():
    return [
        # a thumbnail or a region of interest: one call is all latency (64x48, 16 depth numbers)
        {"name": "tiny-64x48x16", "kind": "pair", "w": 64, "h": 48, "D": 16, "opts": "default",
         "scene": "rects", "tau": 30, "lam": 8},
        # the headline: one 384x288 frame, 16 depth numbers, tuned options, buffers kept
        {"name": "main-384x288x16", "kind": "pair", "w": 384, "h": 288, "D": 16, "opts": "tuned",
         "scene": "layers", "tau": 30, "lam": 10},
        # the paper's colour data term on the same frame size (sum of absolute differences, 0..765)
        {"name": "colour-384x288x16", "kind": "rgb", "w": 384, "h": 288, "D": 16, "opts": "tuned",
         "scene": "layers", "tau": 765, "lam": 14},
        # an odd crop by a caller who keeps nothing and gives no options
        {"name": "crop-333x251x23", "kind": "pair", "w": 333, "h": 251, "D": 23, "opts": "none",
         "scene": "layers", "tau": 30, "lam": 10},
        # a larger frame with a long depth range
        {"name": "vga-640x480x64", "kind": "pair", "w": 640, "h": 480, "D": 64, "opts": "tuned",
         "scene": "layers", "tau": 30, "lam": 10},
        # the largest: a 960x540 frame of slanted planes
        {"name": "planes-960x540x48", "kind": "pair", "w": 960, "h": 540, "D": 48, "opts": "tuned",
         "scene": "planes", "tau": 40, "lam": 12},
        # an offline job: pairs of uneven size and depth range in one batched call
        {"name": "batch-12-uneven", "kind": "batch", "pairs": 12, "sizes_seed": 4000},
        # one sample of a training step: structured hinge loss, forward and backward
        {"name": "train-384x288x32", "kind": "train", "w": 384, "h": 288, "D": 32},
        # the approximate modes of the paper on the headline frame
        {"name": "level1-384x288x16-b2", "kind": "level1", "w": 384, "h": 288, "D": 16, "b": 2},
        {"name": "level2-384x288x16-b3", "kind": "level2", "w": 384, "h": 288, "D": 16, "b": 3},
        # the learned data term, the energy of a labeling and its adjoint with
        # respect to every data cost and weight (a matching cost trained from outside)
        {"name": "adjoint-1280x720x64", "kind": "adjoint", "w": 1280, "h": 720, "D": 64},
    ]


def _log_int(rng: random.Random, lo: int, hi: int) -> int:
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    kind = rng.choice(["pair", "pair", "pair", "rgb", "batch", "train", "level1", "level2",
                       "adjoint"])
    if kind == "batch":
        return {"kind": kind, "pairs": _log_int(rng, 2, 12), "sizes_seed": rng.randrange(1 << 30)}
    top = {"pair": 12.0e6, "adjoint": 50.0e6}.get(kind, 4.0e6)      # graph nodes at most
    while True:
        D = _log_int(rng, 8, 64)
        w, h = _log_int(rng, 64, 960), _log_int(rng, 48, 720)
        ng = w - 2 * (D - 1)
        if ng >= 16 and 2.0e4 <= ng * h * (D - 1) <= top:
            break
    c = {"kind": kind, "w": w, "h": h, "D": D}
    if kind == "pair":
        c.update(opts=rng.choice(["tuned", "default", "none"]),
                 scene=rng.choice(["rects", "layers", "layers", "planes"]), tau=rng.randint(20, 40),
                 lam=rng.randint(6, 14))
    elif kind == "rgb":
        c.update(opts="tuned", scene="layers", tau=765, lam=rng.randint(10, 20))
    elif kind in ("level1", "level2"):
        c.update(b=rng.choice([2, 3]))
    return c


def _pair(w, h, D, scene, tau, lam, seed, rgb=False):
    md = min(2 * (D - 1), 40)
    wl = synth.Workload("case", w, h, D, tau=tau, lam=lam, sigma=2.0 if scene != "layers" else 3.0,
                        scene=scene, n_layers=12 if scene == "planes" else 5,
                        n_slanted=12 if scene == "planes" else 2,
                        max_disp=2 * (D - 1) if scene == "planes" else md,
                        rect_disps=(2, max(3, md // 2), max(4, md - 2)), seed_base=seed)
    L, R, dR = (synth.make_pair_rgb if rgb else synth.make_pair)(wl, 0)
    return torch.from_numpy(L).cuda(), torch.from_numpy(R).cuda(), dR


def _batch_sizes(case):
    rng = random.Random(case["sizes_seed"])
    out = []
    for _ in range(case["pairs"]):
        D = rng.randint(16, 64)
        out.append((max(rng.randint(160, 640), 2 * (D - 1) + 8), rng.randint(120, 480), D))
    return out


def prepare(case, seed):
    kind = case["kind"]
    s = {"kind": kind}
    if kind == "batch":
        sizes = _batch_sizes(case)
        ps = [gc.Params(w=w, h=h, D=D, tau=30, lam=10) for w, h, D in sizes]
        s["batch"] = gc.Batch(ps, [autotune.tuned_opts(p) for p in ps])
        imgs = [_pair(w, h, D, "layers", 30, 10, seed * 100 + i)
                for i, (w, h, D) in enumerate(sizes)]
        s["L"], s["R"] = [x[0] for x in imgs], [x[1] for x in imgs]
        return s
    w, h, D = case["w"], case["h"], case["D"]
    if kind in ("train", "adjoint"):
        L, R, dR = _pair(w, h, D, "layers", 30, 8, seed)
        gt = torch.from_numpy(metrics.gt_depth(dR, D, 2 * (D - 1))).cuda()
        if kind == "train":
            p = gc.Params(w=w, h=h, D=D, tau=0, lam=0, inhibit=1023 * int(SCALE))
            s["pr"] = learn.problem(L, R, p, autotune.tuned_opts(p))
            s["theta"] = torch.tensor(THETA, dtype=torch.float64, requires_grad=True)
        else:
            p = gc.Params(w=w, h=h, D=D, tau=0, lam=int(SCALE * THETA[3]), inhibit=1023 * int(SCALE))
            n = h * p.ng * D
            s.update(L=L, R=R, p=p, cost=torch.empty(n, dtype=torch.int32, device="cuda"),
                     dcost=torch.empty(n, dtype=torch.float32, device="cuda"),
                     counts=torch.zeros(2, dtype=torch.int64, device="cuda"),
                     sums=torch.zeros(3, dtype=torch.int64, device="cuda"),
                     energy=torch.zeros(1, dtype=torch.int64, device="cuda"))
        s["gt"] = gt
        return s
    if kind in ("level1", "level2"):
        L, R, _ = _pair(w, h, D, "layers", 30, 10, seed)
        p = gc.Params(w=w, h=h, D=D, tau=30, lam=10)
        o = autotune.tuned_opts(p)
        oc = autotune.tuned_opts(gc.gs_delegate_params(p, case["b"]))
        s.update(L=L, R=R, p=p, o=o, b=case["b"], bufs=gc.Level1Buffers(p, case["b"], o, oc),
                 cost=torch.empty(h * p.ng * D, dtype=torch.int32, device="cuda"))
        return s
    L, R, _ = _pair(w, h, D, case["scene"], case["tau"], case["lam"], seed, kind == "rgb")
    p = gc.Params(w=w, h=h, D=D, tau=case["tau"], lam=case["lam"])
    s.update(L=L, R=R, p=p, o=None, buf=None)
    if case["opts"] != "none":
        s["o"] = autotune.tuned_opts(p) if case["opts"] == "tuned" else gc.SolveOpts()
        s["buf"] = gc.Buffers(p, s["o"])
    return s


def run(s):
    kind = s["kind"]
    if kind == "pair":
        labels, flow, status = gc.solve_pair(s["L"], s["R"], s["p"], s["o"], s["buf"])
        return {"labels": labels, "flow": flow, "status": status}
    if kind == "rgb":
        gc.gs_stereo_cost_volume_rgb(s["L"], s["R"], s["p"], s["buf"].cost)
        labels, flow, status = gc.solve_costs(s["buf"].cost, s["p"], s["o"], s["buf"])
        return {"labels": labels, "flow": flow, "status": status}
    if kind == "batch":
        gc.gs_solve_batched(s["batch"], s["L"], s["R"])
        return [{"labels": b.labels, "flow": b.flow, "status": b.status} for b in s["batch"].bufs]
    if kind in ("level1", "level2"):
        gc.gs_stereo_cost_volume(s["L"], s["R"], s["p"], s["cost"])
        if kind == "level1":
            labels, coarse, status = gc.solve_level1(s["cost"], s["p"], s["b"], s["o"], s["bufs"])
        else:
            labels, coarse, status = gc.solve_level2(s["cost"], s["p"], s["b"], 2, s["o"], s["bufs"])
        return {"labels": labels, "coarse": coarse, "status": status}
    if kind == "train":
        loss = learn.hinge_loss(s["theta"], s["pr"], s["gt"], SCALE)
        (grad,) = torch.autograd.grad(loss, s["theta"])
        return {"loss": loss.detach(), "grad": grad, "labels": s["pr"].buf.labels}
    w1, w2, tau, _ = THETA
    p = s["p"]
    gc.gs_stereo_cost_volume_f32(s["L"], s["R"], p, w1, w2, tau, SCALE, s["cost"])
    gc.gs_energy(s["cost"], s["gt"], p, s["energy"])
    gc.gs_energy_backward(s["gt"], p, 0.5, s["dcost"], s["counts"])
    gc.gs_cost_volume_f32_backward(s["L"], s["R"], p, w1, w2, tau, s["gt"], s["sums"])
    return {k: s[k] for k in ("cost", "energy", "dcost", "counts", "sums")}


def work(case):
    """Images read once, results written once; a handful of operations per cross point."""
    if case["kind"] == "batch":
        one = [work({"kind": "pair", "w": w, "h": h, "D": D}) for w, h, D in _batch_sizes(case)]
        return {k: sum(x[k] for x in one) for k in ("bytes", "flops")}
    w, h, D = case["w"], case["h"], case["D"]
    sites = (w - 2 * (D - 1)) * h
    ch = 3 if case["kind"] == "rgb" else 1
    images = 2 * w * h * ch
    if case["kind"] == "adjoint":
        return {"bytes": images + 4 * sites + 8 * sites * D + 48, "flops": 12 * sites * D}
    if case["kind"] == "train":
        return {"bytes": images + 8 * sites + 48, "flops": 24 * sites * D}
    extra = 4 * sites // case["b"] ** 2 if "b" in case else 0
    return {"bytes": images + 4 * sites + extra + 12, "flops": (3 * ch + 4) * sites * D}


def exact(case, seed):
    """Labels, flows, energies and counts are whole numbers (None: nothing to
    round).  The adjoint with respect to the data costs is computed here."""
    if case["kind"] != "adjoint":
        return None
    s = prepare(case, seed)
    p, gt = s["p"], s["gt"].long()
    d = torch.zeros((p.h, p.ng, p.D), dtype=torch.float64, device="cuda")
    d.scatter_(2, gt.unsqueeze(-1), 0.5)
    jumps = [(gt[:, 1:] - gt[:, :-1]).abs(), (gt[1:] - gt[:-1]).abs()]
    counts = torch.stack([sum(j.sum() for j in jumps), sum((j - 1).clamp(min=0).sum() for j in jumps)])
    return {"cost": None, "energy": None, "dcost": d.reshape(-1), "counts": counts, "sums": None}
