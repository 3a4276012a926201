"""The work a user of this library has it do, as cases that can be timed and compared.

Every case calls the public entry points through the binding (``paper_2606_14173_gb300.hpt``): traces
of the seeded scenes, cache bakes, angular-spectrum propagation and phase-only encoding.  Scenes,
render settings and sizes are those of the benchmark configurations, the serving stream and the
tests; ``draw`` spreads over the ranges between them.

A program keeps one library context for its device, so the cases of a process share one; scenes,
output buffers and input fields belong to the state of a case.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2606_14173_gb300 import hpt, scenes as S

_ctx = None


def _context():
    global _ctx
    if _ctx is None:
        _ctx = hpt.Context(torch.cuda.current_device())
    return _ctx


class _SceneHandle:
    """An uploaded scene, released with the state that holds it."""

    def __init__(self, scene):
        self.ctx = _context()
        self.sid = self.ctx.upload_scene(scene)

    def __del__(self):
        try:
            self.ctx.release_scene(self.sid)
        except Exception:
            pass


# ------------------------------------------------------------------------------------ cases
def _trace(name, scene, **kw):
    base = dict(name=name, op="trace", scene=scene, W=256, H=256, rgb=True, spp=16, depth=4, K=8, fp64=False,
                pose=False, phase="hash", host=False)
    base.update(kw)
    return base


def listed():
    return [
        # configuration 0: two emissive textures, one wavelength, direct emission only
        _trace("quads_256", "quads", rgb=False, depth=1, K=1),
        # an interactive preview of a ragged size (the tests' crop): launches and latency count
        _trace("spheres_preview", "spheres", W=203, H=117, spp=8, K=4),
        # a small request of the serving stream: 512 x 512, an eye offset and a focal depth
        _trace("spheres_request", "spheres", W=512, H=512, spp=16, K=4, pose=True),
        # the headline frame: 1080p, RGB, 64 samples, eight holograms from one path set
        _trace("spheres_1080p", "spheres", W=1920, H=1080, spp=64),
        # the plain double-precision form of the coherent chain on a band of that frame
        _trace("spheres_fp64_band", "spheres", W=1920, H=270, spp=16, fp64=True),
        # the 185k-triangle scene with its resident ambient cache, an SLM crop at 3.74 um
        _trace("slabs_cache", "slabs", W=960, H=540, spp=32),
        # Gaussian-random-field phases: the maps of a new phase seed, then the frame that uses them
        _trace("spheres_grf", "spheres", W=640, H=360, spp=8, phase="grf"),
        # the ambient cache of a scene, baked on the device
        dict(name="bake_64", op="bake", scene="spheres", res=64, spp=16, depth=4),
        # the second stage of the two-stage scheme: the headline frame's fields to the SLM
        dict(name="asm_1080p", op="asm", W=1920, H=1080, rgb=True, K=8),
        # a single ragged field set, as the tests carry it
        dict(name="asm_small", op="asm", W=300, H=200, rgb=True, K=2),
        # the largest SLM, one hologram
        dict(name="asm_4k", op="asm", W=3840, H=2160, rgb=True, K=1),
        # gradient steps of the phase-only encoding
        dict(name="encode_1080p", op="encode", W=1920, H=1080, iters=10),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["trace", "trace", "trace", "bake", "asm", "asm", "encode"])
    if op == "trace":
        W, H = _log_int(rng, 64, 1920), _log_int(rng, 48, 1080)
        scene = rng.choice(["quads", "spheres", "spheres", "slabs"])
        c = _trace("", scene, W=W, H=H, rgb=rng.random() < 0.75, spp=_log_int(rng, 4, 64),
                   depth=rng.choice([1, 2, 3, 4, 4, 4, 6]), K=rng.choice([1, 2, 3, 4, 8]), fp64=rng.random() < 0.2,
                   pose=rng.random() < 0.3, phase=rng.choice(["hash", "hash", "zero", "grf"]), host=rng.random() < 0.15)
        # no more path samples than the headline frame's share for this kind of scene
        cap = {"quads": 2.0e8, "spheres": 2.0e8, "slabs": 1.0e8}[scene] / (1.5 if c["depth"] > 4 or c["fp64"] else 1.0)
        while _samples(c) > cap and c["spp"] > 4:
            c["spp"] = max(4, c["spp"] // 2)
    elif op == "bake":
        c = dict(op="bake", scene=rng.choice(["spheres", "slabs"]), res=_log_int(rng, 16, 96),
                 spp=_log_int(rng, 4, 32), depth=rng.choice([2, 3, 4]))
    elif op == "asm":
        c = dict(op="asm", W=_log_int(rng, 33, 3840), H=_log_int(rng, 17, 2160), rgb=rng.random() < 0.6,
                 K=rng.choice([1, 2, 3, 8, 11]))
    else:
        c = dict(op="encode", W=_log_int(rng, 65, 1920), H=_log_int(rng, 49, 1080), iters=rng.choice([5, 10, 20]))
    c.pop("name", None)
    return c


def _samples(case):
    return case["W"] * case["H"] * (3 if case["rgb"] else 1) * case["spp"]


# ----------------------------------------------------------------------------------- inputs
_SCENES = {"quads": (S.config0_scene, 1000), "spheres": (S.config1_scene, 1001), "slabs": (S.config3_scene, 1003)}
_SCENE_KEY = {"quads": "cfg0", "spheres": "cfg1", "slabs": "cfg3"}
_RENDER = {"quads": S.config0_render, "spheres": S.config1_render, "slabs": S.config3_render}
_GRF_NX, _GRF_NY = 4096, 2048        # the grid of the phase maps, as the benchmark builds them
_PITCH, _Z = 6.4e-6, 80e-3           # SLM pitch and recording-plane distance of the propagation cases


def _scene(case, seed):
    make, base = _SCENES[case["scene"]]
    return make(seed=base + seed)


def _lambdas(case):
    return S.RGB_LAMBDAS if case.get("rgb", True) else (520e-9,)


def _render(case, seed):
    T = np.eye(4)
    if case["pose"]:
        # an eye offset and a focal depth, drawn as the serving stream draws them
        rng = np.random.default_rng([seed, 1])
        dx, dy = rng.uniform(-5e-3, 5e-3, 2)
        T = S.pose_T(dx, dy, S.SCENE_MEDIAN_DEPTH[_SCENE_KEY[case["scene"]]] - rng.uniform(5e-3, 30e-3))
    return _RENDER[case["scene"]](
        W=case["W"], H=case["H"], lambdas=_lambdas(case), channels=(0, 1, 2) if case["rgb"] else (1,), spp=case["spp"],
        max_depth=case["depth"], K=case["K"], T=T, seed=1 + seed, phase_seed=2 + seed,
        phase_mode={"hash": S.PHASE_HASH, "zero": S.PHASE_ZERO, "grf": S.PHASE_GRF}[case["phase"]])


def _fields(case, seed, shape):
    """Speckle fields, as a trace with random facet phases leaves them: circular complex normal."""
    g = torch.Generator(device="cuda").manual_seed(7919 * seed + 13)
    return torch.view_as_complex(torch.randn(shape + (2,), generator=g, device="cuda", dtype=torch.float32))


def _target(case, seed):
    """A target field for the encoding: a smooth positive amplitude with a random phase (a traced hologram's statistics)."""
    g = torch.Generator(device="cuda").manual_seed(104729 * seed + 29)
    H, W = case["H"], case["W"]
    low = torch.rand((1, 1, 9, 9), generator=g, device="cuda", dtype=torch.float32)
    amp = 0.2 + torch.nn.functional.interpolate(low, size=(H, W), mode="bilinear", align_corners=True)[0, 0]
    ph = torch.rand((2, H, W), generator=g, device="cuda", dtype=torch.float32) * (2 * math.pi)
    return torch.polar(amp, ph[0]).contiguous(), ph[1].contiguous()


def prepare(case, seed):
    op = case["op"]
    st = {"case": case, "op": op, "ctx": _context()}
    if op in ("trace", "bake"):
        scene = _scene(case, seed)
        st["scene"] = _SceneHandle(scene)
    if op == "trace":
        st["r"] = r = _render(case, seed)
        if case["host"]:
            st["out"] = torch.empty(r.out_shape(), dtype=torch.complex64, pin_memory=True)
        else:
            st["out"] = torch.empty(r.out_shape(), dtype=torch.complex64, device="cuda")
        st["prec"] = hpt.PREC_FP64 if case["fp64"] else hpt.PREC_DF32
    elif op == "bake":
        st["lo"], st["hi"] = scene.verts.min(0), scene.verts.max(0)
        st["seed"] = 5 + seed
    elif op == "asm":
        st["U"] = _fields(case, seed, (len(_lambdas(case)), case["K"], case["H"], case["W"]))
        st["out"] = torch.empty_like(st["U"])
    else:
        st["target"], st["phi0"] = _target(case, seed)
        st["phi"] = torch.empty_like(st["phi0"])
    return st


def run(st):
    case, ctx = st["case"], st["ctx"]
    stream = torch.cuda.current_stream().cuda_stream
    if st["op"] == "trace":
        r, sid, out = st["r"], st["scene"].sid, st["out"]
        if case["phase"] == "grf":
            r.grf = ctx.grf_build(r.phase_seed, r.K, _GRF_NX, _GRF_NY, r.pitch, stream=stream)
        if case["host"]:
            ctx.trace_host(sid, r, out.numpy(), precision=st["prec"], stream=stream)
        else:
            ctx.trace(sid, r, out, precision=st["prec"], stream=stream)
        return out
    if st["op"] == "bake":
        return ctx.cache_bake(st["scene"].sid, case["res"], st["lo"], st["hi"], case["spp"], case["depth"],
                              seed=st["seed"], stream=stream)
    if st["op"] == "asm":
        return ctx.asm_propagate(st["U"], _lambdas(case), _PITCH, _Z, out=st["out"], stream=stream)
    st["phi"].copy_(st["phi0"])
    losses = ctx.phase_encode(st["target"], st["phi"], 520e-9, _PITCH, _Z, case["iters"], 0.2, stream=stream)
    # the loss sums float32 fields: it is kept, as they are, in float32
    return {"phi": st["phi"], "losses": losses.astype(np.float32)}


# ------------------------------------------------------------------------------------- work
# float operations of one path sample on each scene (box tests at 20, triangle tests at 30, a vertex at
# 120 and a coherent refinement at 400, as the work counters find them), before the holograms' phasors
_FLOPS = {"quads": 600.0, "spheres": 2400.0, "slabs": 4200.0}
_TRIS = {"quads": 4, "spheres": 23044, "slabs": 185204}


def _pads(W, H):
    return tuple(1 << max(1, math.ceil(math.log2(2 * n))) for n in (W, H))


def _fft_flops(W, H):
    """One padded propagation: the window's rows and every padded column, there and back."""
    Wp, Hp = _pads(W, H)
    return 2 * 5 * (H * Wp * math.log2(Wp) + Wp * Hp * math.log2(Hp)) + 6 * Wp * Hp


def work(case):
    op = case["op"]
    if op == "trace":
        nl = 3 if case["rgb"] else 1
        n = _samples(case)
        deep = min(1.0, 0.4 + 0.15 * case["depth"])
        return {"bytes": 8 * nl * case["K"] * case["W"] * case["H"] + 100 * _TRIS[case["scene"]],
                "flops": n * (_FLOPS[case["scene"]] * deep + 25 * case["K"])}
    if op == "bake":
        n = case["res"] ** 3
        return {"bytes": 12 * n + 100 * _TRIS[case["scene"]], "flops": 3 * n * case["spp"] * _FLOPS[case["scene"]]}
    if op == "asm":
        f = (3 if case["rgb"] else 1) * case["K"]
        return {"bytes": 16 * f * case["W"] * case["H"], "flops": f * _fft_flops(case["W"], case["H"])}
    n = case["W"] * case["H"]
    return {"bytes": 16 * n, "flops": case["iters"] * (2 * _fft_flops(case["W"], case["H"]) + 60 * n)}


# ------------------------------------------------------------------------------------ exact
def _asm64(U, lams, z):
    """Zero-padded angular-spectrum propagation in 64 bits with torch.fft: U [n_lambda][K][H][W]."""
    H, W = U.shape[-2:]
    Wp, Hp = _pads(W, H)
    ox, oy = (Wp - W) // 2, (Hp - H) // 2
    fx = torch.fft.fftfreq(Wp, _PITCH, device=U.device, dtype=torch.float64)
    fy = torch.fft.fftfreq(Hp, _PITCH, device=U.device, dtype=torch.float64)
    out = torch.empty(U.shape, dtype=torch.complex128, device=U.device)
    for l, lam in enumerate(lams):
        a = 1.0 / lam ** 2 - fx[None, :] ** 2 - fy[:, None] ** 2
        turns = z * torch.sqrt(a.clamp_min(0.0))
        turns -= torch.floor(turns)
        h = torch.where(a > 0, torch.polar(torch.ones_like(turns), 2 * math.pi * turns), 0.0)
        del a, turns
        for k in range(U.shape[1]):
            P = torch.zeros((Hp, Wp), dtype=torch.complex128, device=U.device)
            P[oy:oy + H, ox:ox + W] = U[l, k]
            out[l, k] = torch.fft.ifft2(torch.fft.fft2(P) * h)[oy:oy + H, ox:ox + W]
    return out


def _encode64(target, phi, iters, lr):
    """Gradient steps on the phase, L = sum |s A - T|^2 with A = ASM_z(exp(i phi)), s = <A, T> / <A, A>."""
    T, phi, losses = target.to(torch.complex128), phi.to(torch.float64), []
    for _ in range(iters):
        u = torch.polar(torch.ones_like(phi), phi)
        A = _asm64(u[None, None], (520e-9,), _Z)[0, 0]
        s = (A.conj() * T).sum() / (A.abs() ** 2).sum()
        R = s * A - T
        losses.append(float((R.abs() ** 2).sum()))
        G = _asm64((s.conj() * R)[None, None], (520e-9,), -_Z)[0, 0]
        phi = phi + 2.0 * lr * (u * G.conj()).imag
    return {"phi": phi, "losses": np.array(losses)}


def _philox(c, key):
    """Philox4x32-10 (Salmon et al., SC'11) of counters c (four int64 tensors)."""
    m32 = 0xFFFFFFFF
    k0, k1 = key & m32, (key >> 32) & m32
    c = list(c)

    def mul(a, x):  # 32 x 32 -> (high, low) words in int64 without overflow
        lo = (a & 0xFFFF) * x
        hi = (a >> 16) * x + (lo >> 16)
        return (hi >> 16) & m32, ((hi & 0xFFFF) << 16 | (lo & 0xFFFF)) & m32

    for r in range(10):
        if r:
            k0, k1 = (k0 + 0x9E3779B9) & m32, (k1 + 0xBB67AE85) & m32
        h0, l0 = mul(0xD2511F53, c[0])
        h1, l1 = mul(0xCD9E8D57, c[2])
        c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
    return c


def _quads64(case, seed):
    """The two-quad scene in 64 bits: cone rays meet the front or the back quad, whose texture is the
    radiance; U_m = (1/(i lambda)) mean sqrt(L) cos(theta) r / (pdf cos(theta_P)) exp(i(k r + phi_m)), cos(theta_P)
    = cos(theta) as the quads lie across the axis."""
    sc, r = _scene(case, seed), _render(case, seed)
    dev = "cuda"
    quads = []
    for q in range(2):
        v = sc.verts[4 * q:4 * q + 4].astype(np.float64)
        off, w, h = (int(x) for x in sc.tex_info[q])
        tex = torch.tensor(sc.tex_data[off:off + w * h * 3].reshape(h, w, 3), dtype=torch.float64, device=dev)
        quads.append((v[0], v[1, 0] - v[0, 0], v[3, 1] - v[0, 1], tex))
    t0, t1, t2 = (float(x) for x in r.T[:3, 3])   # the poses drawn here are translations
    out = torch.empty(r.out_shape(), dtype=torch.complex128, device=dev)
    pix = torch.arange(r.W * r.H, device=dev)
    x = ((pix % r.W) + 0.5 - 0.5 * r.W) * r.pitch - t0
    y = ((pix // r.W) + 0.5 - 0.5 * r.H) * r.pitch - t1
    for l, lam in enumerate(r.lambdas):
        hc = 2.0 * math.sin(0.5 * math.asin(lam / (2.0 * r.pitch))) ** 2
        pdf = 1.0 / (2.0 * math.pi * hc)
        acc = [torch.zeros(r.W * r.H, dtype=torch.complex128, device=dev) for _ in range(r.K)]
        for s in range(r.spp):
            c = [pix, torch.full_like(pix, s), torch.zeros_like(pix), torch.full_like(pix, (l << 16) | 0xFFFF)]
            d = _philox(c, r.seed)
            u0, u1 = ((d[i] >> 8).double() / 16777216.0 for i in (0, 1))
            s1 = hc * u0
            ct, sn = 1.0 - s1, torch.sqrt(s1 * (2.0 - s1))
            dx, dy = sn * torch.cos(2 * math.pi * u1), sn * torch.sin(2 * math.pi * u1)
            L = torch.zeros_like(ct)
            R = torch.zeros_like(ct)
            P = [torch.zeros_like(ct) for _ in range(3)]
            free = torch.ones_like(pix, dtype=torch.bool)
            for v0, eu, ev, tex in quads:
                t = (v0[2] + t2) / ct
                px, py = x + dx * t, y + dy * t
                a, b = (px - v0[0]) / eu, (py - v0[1]) / ev
                hit = free & (a >= 0) & (a <= 1) & (b >= 0) & (b <= 1) & (t > 0)
                free &= ~hit
                gx, gy = a * tex.shape[1] - 0.5, b * tex.shape[0] - 0.5
                i, j = torch.floor(gx), torch.floor(gy)
                fx, fy = gx - i, gy - j
                i0, i1 = (k.long().clamp(0, tex.shape[1] - 1) for k in (i, i + 1))
                j0, j1 = (k.long().clamp(0, tex.shape[0] - 1) for k in (j, j + 1))
                tc = tex[:, :, r.channels[l]]
                val = (tc[j0, i0] * (1 - fx) + tc[j0, i1] * fx) * (1 - fy) + (tc[j1, i0] * (1 - fx) + tc[j1, i1] * fx) * fy
                L, R = torch.where(hit, val, L), torch.where(hit, t, R)
                for k, pk in enumerate((px, py, torch.full_like(px, v0[2]))):
                    P[k] = torch.where(hit, pk, P[k])
            cells = [torch.floor(p / r.facet_size).long() & 0xFFFFFFFF for p in P]
            turns = R / lam
            turns = turns - torch.floor(turns)
            amp = torch.sqrt(L) * R / (pdf * lam)
            for m in range(r.K):
                u = 0.0
                if r.phase_mode == S.PHASE_HASH:
                    o = _philox(cells + [torch.full_like(pix, (l << 16) | (m >> 2))], r.phase_seed)
                    u = (o[m & 3] >> 8).double() / 16777216.0
                acc[m] += -1j * torch.polar(amp, 2 * math.pi * (turns + u))
        for m in range(r.K):
            out[l, m] = (acc[m] / r.spp).reshape(r.H, r.W)
    return out


def exact(case, seed):
    op = case["op"]
    if op == "asm":
        Wp, Hp = _pads(case["W"], case["H"])
        if Wp * Hp * case["K"] > 2 ** 28:
            return None
        shape = (len(_lambdas(case)), case["K"], case["H"], case["W"])
        return _asm64(_fields(case, seed, shape), _lambdas(case), _Z)
    if op == "encode":
        return _encode64(*_target(case, seed), case["iters"], 0.2)
    if op == "trace" and case["scene"] == "quads" and case["phase"] != "grf" and _samples(case) * case["K"] < 2 ** 28:
        return _quads64(case, seed)
    # the other scenes have no closed form: mirrors, lenses and rough surfaces through a mesh
    return None
