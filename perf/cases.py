"""What a user of this library has it compute, as measurable cases.

A case is a dict of plain values.  ``kind`` says which entry point it goes
through:

  frame     HRC.forward: one lit frame (a renderer's inner loop)
  grad      fluence() and its backward: one step of inverse rendering
  bounce    fluence_bounces() and its backward: a step through K bounces
  batch     BatchedHRC.forward: many scenes of uneven size at once
  batchgrad BatchedHRC.forward and .backward: the same with gradients

Sizes and scene contents are those of ``scenes.py`` and of the benchmark
(64^2 .. 2048^2, 1 to 4 channels, fp32 and the 16-bit storage modes, the
options cross blur, environment map and per-channel extinction).
``exact`` is the method in float64 torch: sorted ray clipping for levels
0..2, Eqs. 18-20 upwards, Eqs. 13-17 downwards, gradients by autograd.
"""
import math
import random

import numpy as np
import torch

from paper_2505_02041_gb300 import HRC, BatchedHRC, fluence, fluence_bounces, scenes


# ---------------------------------------------------------------------------
# The cases
# ---------------------------------------------------------------------------
def listed():
    return [
        # a thumbnail or a game tile: the smallest scene of the tests, where launches and latency count
        dict(name="frame_disks64", kind="frame", scene="disks", W=64, H=64, C=1, prec="fp32"),
        # one step of inverse rendering at the size of the differentiable workload
        dict(name="grad_fog256", kind="grad", scene="fog", W=256, H=256, C=1, prec="fp32"),
        # an interactive RGB frame
        dict(name="frame_fog512", kind="frame", scene="fog", W=512, H=512, C=3, prec="fp32"),
        # a window of odd size, lit from outside, with the blur on: no extent divides a tile, the trace
        # cannot use tensor copies
        dict(name="frame_odd_env_blur", kind="frame", scene="volumetric", W=1021, H=763, C=3, prec="fp32", env=64,
             blur=True),
        # the headline frame, in the configuration that the autotuner picks, as a frame loop runs it
        dict(name="frame_vol1024", kind="frame", scene="volumetric", W=1024, H=1024, C=3, prec="fp32", tuned=True),
        # the same frame in 16-bit storage
        dict(name="frame_vol1024_bf16", kind="frame", scene="volumetric", W=1024, H=1024, C=3, prec="bf16",
             tuned=True),
        # a large frame
        dict(name="frame_fog2048", kind="frame", scene="fog", W=2048, H=2048, C=3, prec="fp32"),
        # a training step at the headline size
        dict(name="grad_vol1024", kind="grad", scene="volumetric", W=1024, H=1024, C=3, prec="fp32"),
        # a training step with coloured fog (extinction per channel) and the blur on
        dict(name="grad_channels512", kind="grad", scene="fog", W=512, H=512, C=3, prec="fp32", channels=True,
             blur=True),
        # scattering media: two bounces, differentiated through both
        dict(name="bounce_fog512", kind="bounce", scene="fog", W=512, H=512, C=3, prec="fp32", bounces=2),
        # many small scenes: a tile set or a data generator
        dict(name="batch_small_bf16", kind="batch", scene="fog", scenes=96, lo=64, hi=256, pick=5, C=3, prec="bf16",
             tuned=True),
        # a training batch of uneven scenes
        dict(name="batchgrad_mixed_bf16", kind="batchgrad", scene="fog", scenes=12, lo=128, hi=1024, pick=4, C=3,
             prec="bf16", tuned=True),
    ]


def draw(rng):
    most = max(_ops(c) for c in listed())
    while True:
        c = _draw(rng)
        if _ops(c) <= most:
            return c


def _draw(rng):
    def size(lo, hi):
        n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
        return n if rng.random() < 0.6 else max(lo, n // 32 * 32)

    kind = rng.choice(["frame", "frame", "frame", "grad", "grad", "bounce", "batch", "batchgrad"])
    prec = rng.choice(["fp32", "fp32", "fp16", "bf16"])
    if kind in ("batch", "batchgrad"):
        hi = rng.choice([256, 512, 1024])
        return dict(kind=kind, scene="fog", scenes=rng.randint(3, 96 if hi == 256 else 16), lo=64, hi=hi,
                    pick=rng.randint(0, 999), C=rng.choice([1, 3, 3]), prec=prec, tuned=rng.random() < 0.5)
    W = size(48, 2048 if kind == "frame" else 1024)
    H = max(48, min(2048, int(W * rng.uniform(0.5, 2.0)))) if rng.random() < 0.7 else W
    c = dict(kind=kind, scene=rng.choice(["fog", "volumetric", "disks"]), W=W, H=H, C=rng.choice([1, 2, 3, 3, 3, 4]),
             prec=prec)
    if kind != "frame" and c["scene"] == "disks":
        c["scene"] = "fog"
    if rng.random() < 0.25:
        c["blur"] = True
    if kind == "bounce":
        c["bounces"] = rng.randint(1, 3)
    elif rng.random() < 0.2:
        c["env"] = rng.choice([16, 64, 250])
    if c["C"] > 1 and W <= 1024 and rng.random() < 0.15:
        c["channels"] = True
    if kind == "frame" and W * H <= 1 << 20 and rng.random() < 0.3:
        c["tuned"] = True
    return c


def _sizes(case):
    """(W, H) of every scene of a case."""
    if "scenes" not in case:
        return [(case["W"], case["H"])]
    g = random.Random(case["pick"])
    steps = [n for n in (64, 128, 256, 512, 1024) if case["lo"] <= n <= case["hi"]]
    return [(g.choice(steps), g.choice(steps)) if g.random() < 0.25 else (n, n)
            for n in (g.choice(steps) for _ in range(case["scenes"]))]


def _levels(U):
    N = 0
    while (1 << N) < U:
        N += 1
    return N


def _ops(case):
    """Arithmetic of one pass: every entry of T_n and R_n of the four frames,
    with its merges (2 C + 1 operations each, plus the average at odd
    directions); a backward counts twice its forward; K bounces K + 1 passes
    whose backward recomputes K of them."""
    C = case["C"]
    total = 0.0
    for W, H in _sizes(case):
        for U, V in ((W, H), (H, W)):
            for n in range(_levels(U) + 1):
                merges = 1.5 if n >= 3 else (1 << n) + 2.0
                total += 2.0 * U * V * (1 + 0.5 ** n) * merges * (2 * C + 1)      # T_n
                total += 2.0 * U * V * 2 * (3 * C + 1)                            # R_n: two edges
    if case.get("channels"):
        total *= C * 3.0 / (2 * C + 1)
    if case["kind"] in ("grad", "batchgrad"):
        total *= 3
    if case["kind"] == "bounce":
        total *= 4 * case["bounces"] + 3
    return total


def work(case):
    C = case["C"]
    pix = sum(W * H for W, H in _sizes(case))
    sig = C if case.get("channels") else 1
    planes = 2 * C + sig                                   # e, sigma, F
    if case["kind"] in ("grad", "batchgrad"):
        planes += 2 * C + sig                              # dL/dF, dL/de, dL/dsigma
    if case["kind"] == "bounce":
        planes += 4 * C + sig                              # albedo, dL/dF, dL/de, dL/dsigma, dL/dalbedo
    return {"bytes": 4.0 * pix * planes, "flops": _ops(case)}


# ---------------------------------------------------------------------------
# Inputs and passes
# ---------------------------------------------------------------------------
def _scene(case, W, H, seed):
    if case["scene"] == "disks":
        return scenes.scene_disks_boxes(W, H, case["C"], seed)
    if case["scene"] == "fog":
        return scenes.scene_disks_rects_fog(W, H, case["C"], seed)
    return scenes.scene_volumetric_walls(W, H, case["C"], seed)


def _inputs(case, seed):
    """Host float32 arrays: per scene (e, sigma), and what the kind adds."""
    g = np.random.Generator(np.random.PCG64([seed, 11]))
    out = []
    for k, (W, H) in enumerate(_sizes(case)):
        e, s = _scene(case, W, H, seed * 1000 + k)
        d = dict(e=e, s=s)
        if case.get("channels"):
            d["s"] = np.stack([s * np.float32(f) for f in (1.0, 0.5, 2.0, 0.8)[: case["C"]]])
        if case["kind"] in ("grad", "bounce", "batchgrad"):
            d["g"] = g.standard_normal(e.shape, dtype=np.float32)
        if case["kind"] == "bounce":
            d["a"] = g.uniform(0.2, 0.8, size=e.shape).astype(np.float32)
        out.append(d)
    env = None
    if case.get("env"):
        M = case["env"]
        th = 2 * np.pi * (np.arange(M) + 0.5) / M
        env = np.stack([0.4 + 0.3 * np.cos(th - g.uniform(0, 6)) for _ in range(case["C"])]).astype(np.float32)
    return out, env


def prepare(case, seed):
    ins, env = _inputs(case, seed)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    st = dict(kind=case["kind"])
    if case["kind"] in ("batch", "batchgrad"):
        b = BatchedHRC(_sizes(case), case["C"], precision=case["prec"])
        st["h"] = b
        st["e"], st["s"] = b.pack([dev(d["e"]) for d in ins], [dev(d["s"]) for d in ins])
        st["F"] = torch.empty_like(st["e"])
        if case.get("tuned"):
            b.autotune(st["e"], st["s"])
        if case["kind"] == "batchgrad":
            st["g"] = torch.cat([dev(d["g"]).reshape(-1) for d in ins])
            st["ge"], st["gs"] = torch.empty_like(st["e"]), torch.empty_like(st["s"])
        return st
    h = HRC(case["W"], case["H"], case["C"], precision=case["prec"])
    if case.get("channels"):
        h.set_channel_extinction(True)
    if case.get("blur"):
        h.set_cross_blur(True)
    if case["kind"] == "bounce":
        h.reserve_bounces(case["bounces"])
    if env is not None:
        h.set_environment(dev(env))
    if case.get("tuned"):
        h.autotune()
    d = ins[0]
    st["h"] = h
    st["e"], st["s"] = dev(d["e"]), dev(d["s"])
    if case["kind"] == "frame":
        st["F"] = torch.empty_like(st["e"])
    else:
        st["g"] = dev(d["g"])
        for k in ("e", "s"):
            st[k].requires_grad_(True)
        if case["kind"] == "bounce":
            st["a"] = dev(d["a"]).requires_grad_(True)
            st["K"] = case["bounces"]
    return st


def run(st):
    h, kind = st["h"], st["kind"]
    if kind in ("frame", "batch"):
        return {"F": h.forward(st["e"], st["s"], st["F"])}
    if kind == "batchgrad":
        F = h.forward(st["e"], st["s"], st["F"])
        ge, gs = h.backward(st["g"], st["ge"], st["gs"])
        return {"F": F, "ge": ge, "gs": gs}
    if kind == "grad":
        F = fluence(h, st["e"], st["s"])
        ge, gs = torch.autograd.grad(F, (st["e"], st["s"]), st["g"])
        return {"F": F.detach(), "ge": ge, "gs": gs}
    F = fluence_bounces(h, st["e"], st["s"], st["a"], st["K"])
    ge, gs, ga = torch.autograd.grad(F, (st["e"], st["s"], st["a"]), st["g"])
    return {"F": F.detach(), "ge": ge, "gs": gs, "ga": ga}


# ---------------------------------------------------------------------------
# The method in float64 torch
# ---------------------------------------------------------------------------
def exact(case, seed):
    ins, env = _inputs(case, seed)
    device = "cuda" if torch.cuda.is_available() else "cpu"
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(device=device, dtype=torch.float64)
    env = None if env is None else dev(env)
    res = []
    for d in ins:
        e, s = dev(d["e"]), dev(d["s"])
        want = [e, s]
        a = None
        if "a" in d:
            a = dev(d["a"])
            want.append(a)
        grads = "g" in d
        for t in want:
            t.requires_grad_(grads)
        with torch.set_grad_enabled(grads):
            F = _lighting(e, s, env, case.get("blur"))
            for _ in range(case.get("bounces", 0)):
                F = _lighting(e + a * s * F / (2 * math.pi), s, env, case.get("blur"))
        r = {"F": F.detach()}
        if grads:
            r.update(zip(("ge", "gs", "ga"), torch.autograd.grad(F, want, dev(d["g"]))))
        res.append(r)
    if "scenes" in case:
        return {k: torch.cat([r[k].reshape(-1) for r in res]) for k in res[0]}
    return res[0]


def _lighting(e, s, env, blur):
    """F of Algorithm 1 (with Eq. 21 when asked) for e [C][H][W], s [H][W] or [C][H][W]."""
    if s.dim() == 3:
        return torch.cat([_lighting(e[c:c + 1], s[c], None if env is None else env[c:c + 1], blur)
                          for c in range(e.shape[0])])
    F = 0
    for q in range(4):
        eq, sq = (e, s) if q < 2 else (e.transpose(-1, -2), s.transpose(-1, -2))      # [.., v, u]
        if q in (1, 3):
            eq, sq = eq.flip(-1), sq.flip(-1)
        f = _frame(eq.transpose(-1, -2), sq.transpose(-1, -2), q, env).transpose(-1, -2)
        if q in (1, 3):
            f = f.flip(-1)
        F = F + (f if q < 2 else f.transpose(-1, -2))
    return _blur(F, s) if blur else F


def _frame(e, s, q, env):
    """R_0(u + 1, v) of one quadrant frame, e [C][U][V], s [U][V]."""
    C, U, V = e.shape
    N = _levels(U)
    envs = _env_levels(env, q, N, C, e)
    if N == 0:
        return envs[0].expand(C, U, V)
    T = [_trace(e, s, n) for n in range(min(2, N) + 1)]
    for n in range(3, N + 1):
        T.append(_extend(T[-1], n))
    v = torch.arange(V, device=e.device)

    def shifted(rows, off, fill):           # rows [..][K][V], row k read at v + off[k]
        i = v[None, :] + off[:, None]
        ok = (i >= 0) & (i < V)
        r = rows.gather(-1, i.clamp(0, V - 1).expand(rows.shape))
        return torch.where(ok, r, fill)

    R = None                                # R_N: the environment
    for n in range(N - 1, -1, -1):
        Un, S = -(-U >> n), 1 << n
        U1 = -(-U >> (n + 1))
        ev = envs[n + 1][:, None, :, None]  # [C][1][2S][1]
        i = torch.arange(S, device=e.device)
        arcs = torch.tensor([math.atan2(2 * (j + 1) - 2 * S, 2 * S) - math.atan2(2 * j - 2 * S, 2 * S)
                             for j in range(2 * S)], dtype=torch.float64, device=e.device)
        R1 = ev.expand(C, U1 + 1, 2 * S, V) if R is None else torch.cat([R, ev.expand(C, 1, 2 * S, V)], 1)
        odd = even = 0
        nodd, neven = Un // 2, (Un + 1) // 2
        for sg in (1, 0):
            j, kk = 2 * i + sg, i + sg
            A, fill = arcs[j][:, None], ev[:, :, j]
            t = T[n][:, 1:2 * nodd:2][:, :, kk]                                       # Eq. 14
            far = shifted(R1[:, 1:nodd + 1][:, :, j], 2 * kk - S, fill)
            odd = odd + A * t[:C] + t[C:] * far
            t = T[n + 1][:, :neven][:, :, 2 * kk]                                      # Eqs. 15-17
            far = shifted(R1[:, 1:neven + 1][:, :, j], 4 * kk - 2 * S, fill)
            even = even + 0.5 * (R1[:, :neven][:, :, j] + A * t[:C] + t[C:] * far)
        R = even.new_zeros(C, Un, S, V)
        R[:, 0::2] = even
        R[:, 1::2] = odd
    last = envs[0][:, None, :, None].expand(C, 1, 1, V)
    return torch.cat([R[:, 1:], last], 1)[:, :, 0]


def _trace(e, s, n):
    """T_n [C + 1][U_n][2^n + 1][V] (radiances, transmittance) by clipping."""
    C, U, V = e.shape
    a, P = 1 << n, (1 << n) + 1
    Un = -(-U >> n)
    ep = torch.nn.functional.pad(e, (P, P, 0, a * Un + P - U))
    sp = torch.nn.functional.pad(s, (P, P, 0, a * Un + P - U))
    rows = []
    for k in range(a + 1):
        b = 2 * k - a
        ts = {0.0, 1.0} | {(2 * g - 1) / (2 * a) for g in range(1, a + 1)}
        ts = sorted(ts | {(2 * m - 1) / (2 * abs(b)) for m in range(1, abs(b) + 1)})
        L, t = e.new_zeros(C, Un, V), e.new_ones(Un, V)
        for t0, t1 in zip(ts, ts[1:]):
            if t1 - t0 < 1e-12:
                continue
            mid = 0.5 * (t0 + t1)
            du, dv, ln = math.floor(0.5 + a * mid), math.floor(0.5 + b * mid), (t1 - t0) * math.hypot(a, b)
            cut = (slice(du, du + a * Un, a), slice(P + dv, P + dv + V))
            sg = sp[cut]
            tau = sg * ln
            small = tau.abs() < 1e-4
            safe = torch.where(small, torch.ones_like(sg), sg)
            w = torch.where(small, ln * (1 - tau / 2 + tau * tau / 6 - tau ** 3 / 24),
                            -torch.expm1(-safe * ln) / safe)
            L = L + t * w * ep[(slice(None),) + cut]
            t = t * torch.exp(-tau)
        rows.append(torch.cat([L, t[None]]))
    return torch.stack(rows, 2)


def _extend(T, n):
    """T_n from T_{n-1} (Eqs. 18-20)."""
    C, Um, _, V = T.shape[0] - 1, T.shape[1], T.shape[2], T.shape[3]
    Un, h = -(-Um >> 1), 1 << (n - 1)
    vac = T.new_zeros(C + 1, 1, 1, 1)
    vac[C] = 1
    if Um < 2 * Un:
        T = torch.cat([T, vac.expand(C + 1, 1, T.shape[2], V)], 1)
    near, far = T[:, 0::2], T[:, 1::2]
    v = torch.arange(V, device=T.device)

    def merged(kn, kf, off):
        i = v[None, :] + off[:, None]
        f = far[:, :, kf]
        f = torch.where((i >= 0) & (i < V), f.gather(-1, i.clamp(0, V - 1).expand(f.shape)), vac)
        r = near[:, :, kn]
        return torch.cat([r[:C] + r[C:] * f[:C], r[C:] * f[C:]])

    kk = torch.arange(h + 1, device=T.device)
    kp, km = kk[1:], kk[:-1]
    out = T.new_zeros(C + 1, Un, 2 * h + 1, V)
    out[:, :, 0::2] = merged(kk, kk, 2 * kk - h)
    out[:, :, 1::2] = 0.5 * (merged(km, kp, 2 * km - h) + merged(kp, km, 2 * kp - h))
    return out


def _env_levels(env, q, N, C, like):
    """Value of cone j outside the grid, [C][2^n] for n = 0 .. N (zero without a map)."""
    if env is None:
        return [like.new_zeros(C, 1 << n) for n in range(N + 1)]
    S, M = 1 << N, env.shape[1]
    du, top = float(S), []
    for j in range(S):
        arc = math.atan2(2 * (j + 1) - S, S) - math.atan2(2 * j - S, S)
        dv = 2 * (j + 0.5) - S
        x, y = ((du, dv), (-du, dv), (dv, du), (dv, -du))[q]
        f = math.atan2(y, x) / (2 * math.pi) * M - 0.5
        m = math.floor(f)
        top.append(arc * ((1 - (f - m)) * env[:, m % M] + (f - m) * env[:, (m + 1) % M]))
    vals = [torch.stack(top, 1)]
    for _ in range(N):
        vals.append(vals[-1][:, 0::2] + vals[-1][:, 1::2])
    return vals[::-1]


def _blur(F, s):
    """Eq. 21 leaving out neighbours whose opacity differs by more than 1/2."""
    alpha = 1 - torch.exp(-s.detach())
    pad = torch.nn.functional.pad
    Fp, ap = pad(F, (1, 1, 1, 1)), pad(alpha, (1, 1, 1, 1), value=9.0)
    H, W = s.shape
    acc, wgt = 4 * F, 4.0
    for dy, dx in ((0, 1), (2, 1), (1, 0), (1, 2)):
        keep = ((ap[dy:dy + H, dx:dx + W] - alpha).abs() <= 0.5).to(F.dtype)
        acc = acc + keep * Fp[:, dy:dy + H, dx:dx + W]
        wgt = wgt + keep
    return acc / wgt
