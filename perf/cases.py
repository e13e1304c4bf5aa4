"""What is timed when the library is tuned: the calls that a program running FDA makes, over the
sizes that the library is built for.

A case names one use of the public entry points (``use``), the model dimension ``d``, the number of
workers ``K``, the sketch ``l`` x ``m``, the layout of the K x d model tensor (``packed``: rows at a
pitch of d, as ``torch.empty(K, d)`` gives them, so that the rows of a ragged d are not 16-byte
aligned; else rows padded to 32 elements) and the drift of the workers.  Sizes and drifts are those
of the synthetic workloads (LeNet-5, a small CNN, VGG16*, DenseNet121, DenseNet201, ConvNeXt-Large)
and everything between them.

Uses
    step    one step of SketchFDA that does not fire: local states with a sketch, the estimate read
            back by the host, which decides (nearly every step of a run)
    linear  the same for LinearFDA (norm and projection, no sketch)
    mean    the same from the averaged state (``fda_mean_state``)
    round   states with norm, projection and sketch, the estimate left on the device, the average
            gated by it; fires every time (Theta = 0) and leaves the workers' rows to the caller
    sync    the model average with broadcast, without the monitoring around it
    hook    ``fda_local_state_linear_noalloc``, as a hook inside a training step calls it
    host    ``fda_round_host``: a whole round on pinned host buffers, fires every time
    rounds  the multi-round driver with an in-place optimiser stand-in; every third step fires
"""
import math

import numpy as np
import torch

import fda_synth as S
import paper_2405_20988_b200 as F

STEPS = 12                      # steps of one pass of the multi-round driver
SIGMA_W0 = 0.05                 # spread of the last global model
SKETCH, LINEAR = F.FDA_STATE_NORM | F.FDA_STATE_SKETCH, F.FDA_STATE_NORM | F.FDA_STATE_LINEAR
LARGEST = 197_767_336 * 8       # K * d of the largest case


def _case(name, use, d, K, l=5, m=250, packed=False, drift="iid"):
    return {"name": name, "use": use, "d": d, "K": K, "l": l, "m": m, "packed": packed, "drift": drift}


def listed():
    return [
        # the smallest model of the paper, LeNet-5: launches and latency count
        _case("lenet5 step", "step", 61_706, 5, packed=True),
        # the same through the driver, with its optimiser steps and synchronisations
        _case("lenet5 rounds", "rounds", 61_706, 5),
        # a small CNN with both kinds of summary, synchronising every round, rows as torch packs them
        _case("smallcnn round", "round", 1_199_882, 10, packed=True, drift="shared"),
        # the same model held by a program in host memory
        _case("smallcnn host", "host", 1_199_882, 10, drift="shared"),
        # VGG16* with a sketch larger than the recommended one
        _case("vgg16star 8x1000 step", "step", 2_600_000, 20, 8, 1000, drift="shared"),
        # DenseNet121, thirty workers that drift at very different rates
        _case("densenet121 step", "step", 6_964_106, 30, drift="scaled"),
        # LinearFDA on it (a context without a sketch), ragged rows
        _case("densenet121 linear", "linear", 6_964_106, 30, 0, 1, packed=True, drift="scaled"),
        # the allocation-free call on it, from inside a training step
        _case("densenet121 hook", "hook", 6_964_106, 30, packed=True, drift="scaled"),
        # DenseNet201, the most workers, heavy-tailed drift, a sketch with more rows and columns
        _case("densenet201 step", "step", 20_013_928, 60, 7, 500, drift="heavy"),
        _case("densenet201 mean", "mean", 20_013_928, 60, 7, 500, drift="heavy"),
        # ConvNeXt-Large, the largest model: the monitoring pass and the model average
        _case("convnext step", "step", 197_767_336, 8),
        _case("convnext sync", "sync", 197_767_336, 8),
    ]


def _spread(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    use = rng.choice(["step", "step", "step", "linear", "mean", "mean", "round", "sync", "hook", "host", "rounds"])
    l, m = rng.choice([(5, 250), (5, 250), (5, 250), (7, 500), (8, 1000), (3, 100)])
    if use in ("linear", "hook"):
        l, m = 0, 1                     # no sketch
    K = rng.randint(3, 60)
    # elements a case may have: all of them stay below the largest listed one, those with larger
    # sketches, many steps or copies over the host's bus well below
    most = {"host": 24_000_000, "rounds": 20_000_000}.get(use, LARGEST)
    if (l, m) == (8, 1000):
        most = min(most, 150_000_000)
    elif (l, m) == (7, 500):
        most = min(most, 1_200_000_000)
    d = _spread(rng, 60_000, most // K) if most // K > 60_000 else 60_000
    return {"use": use, "d": d, "K": K, "l": l, "m": m, "packed": rng.random() < 0.5,
            "drift": "iid" if use == "rounds" else rng.choice(["iid", "shared", "scaled", "heavy"])}


def _models(case, gen, w_t0):
    """K x d view of the drifted models, drawn on the device."""
    d, K, drift = case["d"], case["K"], case["drift"]
    w = torch.empty((K, d if case["packed"] else S.row_stride(d)), device="cuda")[:, :d]
    shared = torch.randn(d, device="cuda", generator=gen) * S.SHARED_SIGMA if drift == "shared" else None
    scales = torch.rand(K, generator=gen, device="cuda").tolist() if drift == "scaled" else None
    for k in range(K):
        row = w[k]
        sigma = 1e-3
        if drift == "scaled":
            sigma = S.SCALE_LO * (S.SCALE_HI / S.SCALE_LO) ** scales[k]
        elif d > 100_000_000:
            sigma = 1e-4
        row.normal_(0.0, sigma, generator=gen)
        if drift == "shared":
            row += shared
        elif drift == "heavy":          # one coordinate in a hundred follows Student's t with two degrees of freedom
            mask = torch.rand(d, device="cuda", generator=gen) < S.HEAVY_FRACTION
            n = int(mask.sum())
            t = torch.randn(n, device="cuda", generator=gen)
            t /= (-torch.log(1.0 - torch.rand(n, device="cuda", generator=gen))).clamp_(min=1e-12).sqrt_()
            row[mask] = t * S.HEAVY_SCALE
        row += w_t0
    return w


def prepare(case, seed):
    d, K, l, m, use = case["d"], case["K"], case["l"], case["m"], case["use"]
    gen = torch.Generator(device="cuda").manual_seed(seed)
    s = {"use": use, "K": K}
    s["w_t0"] = torch.randn(d, device="cuda", generator=gen) * SIGMA_W0
    if use == "rounds":                 # all workers start from the last global model
        s["w"] = torch.empty((K, d if case["packed"] else S.row_stride(d)), device="cuda")[:, :d]
        s["w"].copy_(s["w_t0"])
        s["delta"] = torch.randn((K, d), device="cuda", generator=gen) * 1e-3
        s["theta"] = 5e-6 * d           # three steps in one direction fire, two do not
    else:
        s["w"] = _models(case, gen, s["w_t0"])
    if use in ("linear", "round", "hook", "host"):
        xi = torch.randn(d, device="cuda", generator=gen)
        s["xi"] = xi / xi.norm()
    if use == "hook":
        s["states"] = torch.empty((K, 2), device="cuda")
        return s
    s["ctx"] = F.FdaContext(l, m, S.hash_coefficients(seed, l), d_max=d, K_max=K)
    s["epsilon"] = float(np.float32(0.06 * math.sqrt(250.0 / m)))
    if use == "host":
        for name in ("w_t0", "xi"):
            s[name] = s[name].cpu().pin_memory()
        host = torch.empty((K, s["w"].stride(0)), pin_memory=True)[:, :d]
        host.copy_(s["w"])
        s["w"] = host
        s["states"] = torch.empty((K, s["ctx"].state_len), pin_memory=True)
    elif use not in ("sync", "rounds"):
        s["states"] = torch.empty((1 if use == "mean" else K, s["ctx"].state_len), device="cuda")
        s["est"] = s["ctx"].new_estimate_buffer()
    return s


def _host_estimate(est):
    e = est.as_dict()
    return {"values": np.array([e["mean_sq"], e["est"], e["H"]], dtype=np.float32), "rows": e["rows"],
            "trigger": int(e["trigger"])}


def _device_estimate(buf):
    f = buf.view(torch.float32)
    return {"values": f[:4], "rows": f[6:], "trigger": buf[16:24].view(torch.int32)}


def _drift(delta):
    def step(t, w):                     # three steps forward, three back
        w.add_(delta, alpha=1.0 if t % 6 < 3 else -1.0)
    return step


def run(s):
    use, w, w_t0 = s["use"], s["w"], s["w_t0"]
    if use == "hook":
        F.fda_local_state_linear_noalloc(w, w_t0, s["xi"], LINEAR, s["states"])
        return s["states"]
    ctx, K = s["ctx"], s["K"]
    if use == "step":
        ctx.fda_local_state(w, w_t0, None, SKETCH, s["states"])
        est = ctx.fda_combine_estimate(s["states"], K, F.FDA_VARIANT_SKETCH, s["epsilon"], 1e9, s["est"])
        return {"states": s["states"], "estimate": _host_estimate(est)}
    if use == "linear":
        ctx.fda_local_state(w, w_t0, s["xi"], LINEAR, s["states"])
        est = ctx.fda_combine_estimate(s["states"], K, F.FDA_VARIANT_LINEAR, 0.0, 1e9, s["est"])
        return {"states": s["states"], "estimate": _host_estimate(est)}
    if use == "mean":
        ctx.fda_mean_state(w, w_t0, None, SKETCH, s["states"])
        est = ctx.fda_combine_estimate(s["states"], 1, F.FDA_VARIANT_SKETCH, s["epsilon"], 1e9, s["est"])
        return {"states": s["states"], "estimate": _host_estimate(est)}
    if use == "round":
        ctx.fda_local_state(w, w_t0, s["xi"], SKETCH | LINEAR, s["states"])
        ctx.fda_combine_estimate(s["states"], K, F.FDA_VARIANT_SKETCH, s["epsilon"], 0.0, s["est"], want_host=False)
        ctx.fda_average_models(w, w_t0, s["est"], 0)
        return {"states": s["states"], "estimate": _device_estimate(s["est"]), "w_t0": w_t0}
    if use == "sync":
        ctx.fda_average_models(w, w_t0, None, F.FDA_AVG_BROADCAST)
        return {"w": w, "w_t0": w_t0}
    if use == "host":
        est = ctx.fda_round_host(w, w_t0, s["xi"], SKETCH | LINEAR, F.FDA_VARIANT_SKETCH, s["epsilon"], 0.0, 0,
                                 s["states"])
        return {"states": s["states"], "estimate": _host_estimate(est), "w_t0": w_t0}
    out = F.run_rounds(ctx, w, w_t0, None, STEPS, _drift(s["delta"]), F.FDA_VARIANT_SKETCH, s["epsilon"], s["theta"])
    return {"H": np.array(out["H"], dtype=np.float32), "syncs": np.array(out["syncs"]), "w": w, "w_t0": w_t0}


def work(case):
    d, K, l, m, use = case["d"], case["K"], case["l"], case["m"], case["use"]
    n = float(K) * d
    states = K * (2 + l * m)
    sketch = 3.0 * n + float(l) * n              # drift, square, sum; one addition per row
    if use == "step":
        return {"bytes": 4.0 * (n + d + 2 * states), "flops": sketch}
    if use == "linear":
        return {"bytes": 4.0 * (n + 2 * d + 2 * states), "flops": 5.0 * n}
    if use == "hook":
        return {"bytes": 4.0 * (n + 2 * d + 2 * K), "flops": 5.0 * n}
    if use == "mean":
        return {"bytes": 4.0 * (n + d + 2 * (2 + l * m)), "flops": 4.0 * n + float(l) * d}
    if use == "sync":
        return {"bytes": 4.0 * (2 * n + d), "flops": n}
    if use in ("round", "host"):                 # the models and vectors read once, the new global model written
        return {"bytes": 4.0 * (n + 3 * d + 2 * states), "flops": sketch + 3.0 * n}
    # rounds: per step the drift is applied (two reads, a write) and the states are formed; every
    # third step averages and broadcasts
    return {"bytes": 4.0 * STEPS * (3 * n + n + d + 2 * states) + 4.0 * (STEPS // 3) * (2 * n + d),
            "flops": STEPS * (2.0 * n + sketch) + (STEPS // 3) * n}


def tolerance(case):
    # sums of 32-bit floats in another order; the largest difference is taken against the root mean
    # square of an output, which a single cell or projection may lie well below
    return {"rel": 1e-5, "max": 1e-4}
