"""The work that users of the library have it do, as measurable cases.

A case names a kind of call (``KINDS``) and a system size.  Systems are the repository's own
configurations (``scao_tiny``, ``mcao_20m``, ``eelt_mcao``) or the 39 m one scaled to another number
of subapertures, guide stars, layers and DMs.  Inputs are drawn with torch from the seed: von Karman
screens, and a control matrix that is the scaled transpose of the geometric interaction matrix, which
keeps a loop stable without the library's own calibration.  ``exact`` restates each kind in 64 bits.
"""
import math

import numpy as np
import torch

from paper_1608_00386_gb300 import inputs, mcao

DTYPES = {"float32": mcao.DTYPE_F32, "bfloat16": mcao.DTYPE_BF16, "fp8_e4m3": mcao.DTYPE_FP8_E4M3}
ESIZE = {"float32": 4, "bfloat16": 2, "fp8_e4m3": 1}
# subapertures across the pupil whose science transform (16 points per subaperture) factors in 2, 3, 5
SUBS = [8, 9, 10, 12, 15, 16, 18, 20, 24, 25, 27, 30, 32, 36, 40, 45, 48, 50, 54, 60, 64, 72, 75, 80]


def listed():
    return [
        # the smallest loop (one natural star, 16 x 16): each step's commands and Strehl read back, as a
        # real-time study does; latency and launches count
        {"name": "step_8m", "kind": "step", "system": "scao_tiny", "dtype": "float32", "noise": False},
        # the ordinary loop: three laser stars, photon and read noise
        {"name": "step_20m", "kind": "step", "system": "mcao_20m", "dtype": "float32", "noise": True},
        # the largest loop, the benchmark's workload: six laser and three natural stars, 1.8 GB of control matrix
        {"name": "step_39m", "kind": "step", "system": "eelt_mcao", "dtype": "float32", "noise": True},
        # Monte-Carlo statistics: 16 realizations together, reduced-precision control matrix
        {"name": "batch_39m", "kind": "batch", "system": "eelt_mcao", "dtype": "bfloat16", "noise": True,
         "n_real": 16, "n_steps": 2},
        # a short exposure read out whole at its end: the PSF image, Strehl, commands and slopes
        {"name": "exposure_39m", "kind": "exposure", "system": "eelt_mcao", "dtype": "bfloat16", "noise": True,
         "n_steps": 20},
        # a calibration measurement at given commands with the wide-field laser-star sensors
        {"name": "measure_wide", "kind": "measure", "system": "scaled", "n_sub": 40, "n_lgs": 3, "n_ngs": 1,
         "n_layers": 5, "n_dms": 2, "screen": 2048, "wide": True, "noise": False},
        # the largest calibration: the whole interaction matrix (55608 x 8051)
        {"name": "interaction_39m", "kind": "interaction", "system": "eelt_mcao", "noise": False},
        # gradient-based tuning: slopes forward, command gradient backward through autograd
        {"name": "gradient_20m", "kind": "gradient", "system": "mcao_20m", "noise": False, "wrt": "commands",
         "n_vec": 1},
        # the control matrix applied to 16 slope vectors at once
        {"name": "product_39m", "kind": "product", "system": "eelt_mcao", "dtype": "float32", "noise": False,
         "n_real": 16},
        # the real-time controller's update on its own buffers
        {"name": "noalloc_39m", "kind": "noalloc", "n_cmd": 8051, "n_slopes": 55608},
        # the ten screens of the 39 m system
        {"name": "screens_2048", "kind": "screens", "screen": 2048, "n_layers": 10},
        # the ordinary system's control matrix by regularised least squares
        {"name": "tikhonov_20m", "kind": "tikhonov", "system": "mcao_20m", "noise": False, "fp64": False},
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _draw_system(rng, most, wide=False):
    x = _log(rng, SUBS[0], most)
    return {"system": "scaled", "n_sub": min(SUBS, key=lambda s: abs(math.log(s / x))), "n_lgs": rng.randint(1, 6 if most == 80 else 3),
            "n_ngs": rng.randint(0, 3), "n_layers": rng.randint(1, 10), "n_dms": rng.randint(1, 3),
            "screen": rng.choice([512, 750, 1000, 1024, 1536, 2048]), "wide": wide}


def draw(rng):
    kind = rng.choice(["step", "step", "batch", "exposure", "measure", "interaction", "gradient", "product", "noalloc",
                       "screens", "tikhonov"])
    if kind == "noalloc":
        return {"kind": kind, "n_cmd": int(_log(rng, 40, 8051)), "n_slopes": int(_log(rng, 60, 55608))}
    if kind == "screens":
        n = min((2 ** a * 3 ** b * 5 ** c for a in range(13) for b in range(4) for c in range(4)
                 if 64 <= 2 ** a * 3 ** b * 5 ** c <= 4096), key=lambda m, x=_log(rng, 64, 4096): abs(m - x))
        return {"kind": kind, "screen": n, "n_layers": rng.randint(1, max(1, min(10, 10 * 2048 ** 2 // n ** 2)))}
    case = {"kind": kind, "noise": rng.random() < 0.75}
    if kind in ("interaction", "gradient", "measure", "product", "tikhonov"):
        case["noise"] = False
    if kind == "measure":
        wide = rng.random() < 0.5
        case.update(_draw_system(rng, 40 if wide else 80, wide))
    else:
        case.update(_draw_system(rng, 40 if kind in ("gradient", "tikhonov") else 80))
    if kind in ("step", "batch", "exposure", "product"):
        case["dtype"] = rng.choice(list(ESIZE))
    if kind in ("batch", "product"):
        case["n_real"] = rng.randint(2, 16 if case["n_sub"] > 32 else 40)
    if kind in ("batch", "exposure"):
        case["n_steps"] = rng.randint(1, 2 if kind == "batch" else 20)
    if kind == "gradient":
        case["wrt"] = rng.choice(["commands", "all"])
        case["n_vec"] = 1 if case["wrt"] == "commands" else rng.randint(1, 4)
    if kind == "tikhonov":
        case["fp64"] = rng.random() < 0.25
    return case


# ------------------------------------------------------------------------------------------
# systems and inputs
# ------------------------------------------------------------------------------------------
def _system(case):
    if case["system"] != "scaled":
        return getattr(inputs, case["system"])(noise=case["noise"])
    cfg = inputs.eelt_mcao(noise=case["noise"], screen_n=case["screen"], n_layers=case["n_layers"])
    n_sub, npx = case["n_sub"], 16 if case["wide"] else 8
    cfg["D"] = 0.4875 * n_sub
    lgs, ngs = cfg["wfs"][:6][:case["n_lgs"]], cfg["wfs"][6:][:case["n_ngs"]]
    for w in lgs:
        w.update(n_sub=n_sub, n_px=npx)
    cfg["wfs"] = lgs + ngs
    cfg["science"][0]["n_px"] = 8 * n_sub
    for lay in cfg["layers"]:
        lay["pixel"] = 0.4875 / 8
    cfg["dms"] = [inputs.dm_spec(cfg, *p) for p in ((0.0, 0.4875), (4000.0, 1.0), (12700.0, 1.19))[:case["n_dms"]]]
    return cfg


def _pupil(cfg, n):
    x = (np.arange(n) - 0.5 * (n - 1)) * (cfg["D"] / n)
    r2 = x[None, :] ** 2 + x[:, None] ** 2
    return ((r2 <= 0.25 * cfg["D"] ** 2) & (r2 >= 0.25 * cfg["obstruction"] ** 2 * cfg["D"] ** 2)).astype(np.float64)


def _valid(cfg, w):
    """(column, row) of every valid subaperture of a sensor, in row-major order."""
    n, p = w["n_sub"], w["n_px"]
    frac = _pupil(cfg, n * p).reshape(n, p, n, p).mean(axis=(1, 3))
    sy, sx = np.nonzero(frac >= w["valid_thr"])
    return sx, sy


def _n_slopes(cfg):
    return sum(2 * len(_valid(cfg, w)[0]) for w in cfg["wfs"])


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _normal(shape, sigma, gen):
    return torch.randn(shape, generator=gen, device="cuda") * sigma


def _screens(cfg, gen):
    """Periodic von Karman screens of every layer (float32, on the GPU)."""
    out = []
    for lay in cfg["layers"]:
        n = lay["n"]
        f = torch.fft.fftfreq(n, d=lay["pixel"], device="cuda")
        k2 = f[:, None] ** 2 + f[None, :] ** 2
        amp = torch.sqrt(0.023 * lay["r0"] ** (-5 / 3) * (k2 + lay["L0"] ** -2) ** (-11 / 6)) / (n * lay["pixel"])
        amp[0, 0] = 0.0
        c = torch.complex(_normal((n, n), 1.0, gen), _normal((n, n), 1.0, gen)) * amp
        out.append((torch.fft.ifft2(c).real * n * n).contiguous())
    return out


def _geometric(cfg):
    """Geometric interaction matrix (slope of each Gaussian influence function at each subaperture's
    projected centre, in detector pixels), transposed: [n_commands][n_slopes], zero where the
    influence is below 1e-10."""
    out = torch.zeros((inputs.n_commands(cfg), _n_slopes(cfg)), device="cuda")
    col = 0
    for w in cfg["wfs"]:
        sx, sy = _valid(cfg, w)
        d = cfg["D"] / w["n_sub"]
        px = cfg["lambda_ref"] / w["lambda"] * w["n_fft"] * (d / w["n_px"]) / (2 * math.pi * w["n_bin"])
        row = 0
        for m in cfg["dms"]:
            f = 1 - m["alt"] / w["height"] if w["type"] == "lgs" else 1.0
            ay, ax = np.nonzero(m["valid"])
            a = [torch.tensor((q - 0.5 * (m[n] - 1)) * m["pitch"], dtype=torch.float32, device="cuda")
                 for q, n in ((ax, "nx"), (ay, "ny"))]
            p = [torch.tensor((q - 0.5 * (w["n_sub"] - 1)) * d * f + m["alt"] * t, dtype=torch.float32, device="cuda")
                 for q, t in ((sx, w["theta"][0]), (sy, w["theta"][1]))]
            s2 = m["pitch"] ** 2 / (2 * math.log(1 / m["coupling"]))
            dx, dy = p[0][None, :] - a[0][:, None], p[1][None, :] - a[1][:, None]
            g = torch.exp(-(dx * dx + dy * dy) / (2 * s2))
            g = torch.where(g < 1e-10, 0.0, g) * (px * f / s2)
            nv = len(sx)
            out[row:row + len(ax), col:col + nv] = -dx * g
            out[row:row + len(ax), col + nv:col + 2 * nv] = -dy * g
            row += len(ax)
        col += 2 * nv
    return out


def _control(cfg):
    """Gradient-descent control matrix: the geometric transpose over the bound of its squared norm."""
    R = _geometric(cfg)
    return R.mul_(1.0 / float(R.abs().sum(0).max() * R.abs().sum(1).max()))


def _tikhonov_input(cfg, seed):
    """An interaction matrix [n_slopes][n_commands] with a calibration's one per cent of gain errors."""
    D = _geometric(cfg).T.contiguous()
    return D.mul_(1 + _normal(D.shape, 0.01, _generator(seed)))


def _draws(case, cfg, seed):
    """What a case needs beside its screens: commands, slope vectors."""
    gen = _generator(seed + 1)
    if case["kind"] in ("measure", "gradient"):
        c = _normal((inputs.n_commands(cfg),), 0.5, gen)
        return c, _normal((case.get("n_vec", 1), _n_slopes(cfg)), 1.0, gen)
    return _normal((case["n_real"], _n_slopes(cfg)), 0.5, gen)


def _noalloc_inputs(case, seed):
    gen = _generator(seed)
    ld = (case["n_slopes"] + 3) // 4 * 4
    return (_normal((case["n_cmd"], ld), 1e-4, gen)[:, :case["n_slopes"]], _normal((case["n_slopes"],), 0.5, gen),
            _normal((case["n_cmd"],), 1.0, gen))


def prepare(case, seed):
    kind = case["kind"]
    if kind == "noalloc":
        R, s, c = _noalloc_inputs(case, seed)
        return {"kind": kind, "R": R, "s": s, "c": c}
    if kind == "screens":
        return {"kind": kind, "n": case["screen"], "count": case["n_layers"], "seed": seed}
    cfg = _system(case)
    if kind == "tikhonov":
        return {"kind": kind, "D": _tikhonov_input(cfg, seed), "fp64": case["fp64"]}
    cfg["seed"] = seed
    n_real = case.get("n_real", 1)
    # on the caller's stream, so that passes follow one another as the steps of one loop do
    sim = mcao.Sim(cfg, n_real=n_real, stream=torch.cuda.current_stream())
    state = {"kind": kind, "sim": sim, "n_real": n_real, "n_steps": case.get("n_steps", 1)}
    if kind != "product":
        screens = _screens(cfg, _generator(seed))
        for r in range(n_real):   # realizations: the same screens a fraction of their period apart
            sim.load_atmosphere([torch.roll(s, r * s.shape[1] // n_real, 1) if r else s for s in screens], realization=r)
        sim.set_realization(0)
    sim.load_dms()
    if kind in ("step", "batch", "exposure", "product"):
        sim.load_reconstructor(_control(cfg), dtype=DTYPES[case["dtype"]])
        state["commands"] = torch.empty((n_real, inputs.n_commands(cfg)), pin_memory=True)
        state["strehl"] = torch.empty((n_real, 1, 2), dtype=torch.float64, pin_memory=True)
    if kind in ("measure", "gradient"):
        c, state["g"] = _draws(case, cfg, seed)
        state["wrt"] = case.get("wrt")
        state["c"] = c.cpu().numpy() if kind == "measure" or case["wrt"] == "all" else c.requires_grad_()
        if kind == "gradient":
            sim.set_commands(c.detach().cpu().numpy())
    if kind == "product":
        state["s"] = _draws(case, cfg, seed)
    torch.cuda.synchronize()   # the simulation's streams do not wait on torch's
    return state


def run(state):
    kind = state["kind"]
    if kind == "noalloc":
        mcao.reconstruct_noalloc(state["R"], state["s"], state["c"], 0.5)
        return state["c"]
    if kind == "screens":
        return [mcao.generate_screen(state["n"], 0.0609375, 0.157, 25.0, state["seed"] + i) for i in range(state["count"])]
    if kind == "tikhonov":
        return mcao.tikhonov_reconstructor(state["D"], 1e-2, fp64=state["fp64"])
    sim = state["sim"]
    if kind in ("step", "batch"):
        sim.step(state["n_steps"])
        for r in range(state["n_real"]):
            sim.set_realization(r)
            sim.read_async(state["commands"][r], state["strehl"][r])
        return {"commands": state["commands"], "strehl": state["strehl"]}
    if kind == "exposure":
        sim.reset_psf()
        sim.step(state["n_steps"])
        image, sr_long, sr_last = sim.psf(0)
        return {"psf": image, "strehl": [sr_long, sr_last], "commands": sim.commands(), "slopes": sim.slopes()}
    if kind == "measure":
        sim.set_commands(state["c"])
        return sim.measure()
    if kind == "interaction":
        return sim.interaction_matrix()
    if kind == "product":
        return sim.reconstruct_batch(state["s"])
    if state["wrt"] == "all":
        return sim.slopes_vjp(state["g"], commands=True, phase=True, layers=True)
    s = mcao.sensing(sim, state["c"])
    return s.detach(), torch.autograd.grad(s, state["c"], state["g"][0])[0]


def work(case):
    kind = case["kind"]
    if kind == "noalloc":
        n = case["n_cmd"] * case["n_slopes"]
        return {"bytes": 4 * (n + case["n_slopes"] + 2 * case["n_cmd"]), "flops": 2 * n}
    if kind == "screens":
        n = case["screen"] ** 2 * case["n_layers"]
        return {"bytes": 4 * n, "flops": 5 * n * math.log2(case["screen"] ** 2)}
    cfg = _system(case)
    nc, ns = inputs.n_commands(cfg), _n_slopes(cfg)
    if kind == "tikhonov":
        # Gram matrix, Cholesky inverse and product over the nonzero entries of D
        nnz = float((_geometric(cfg) != 0).sum())
        return {"bytes": 4 * nnz + (8 if case["fp64"] else 4) * nc * ns, "flops": nnz / ns * nnz + nc ** 3 + 2 * nc * nnz}
    real, steps = case.get("n_real", 1), case.get("n_steps", 1)
    if kind == "product":
        return {"bytes": ESIZE[case["dtype"]] * nc * ns + 4 * real * (nc + ns), "flops": 2 * real * nc * ns}
    grids = len(cfg["layers"]) + len(cfg["dms"])
    read = 4 * sum(min(lay["n"], cfg["D"] / lay["pixel"]) ** 2 for lay in cfg["layers"])
    surf = 4 * sum(d["surf_n"] ** 2 for d in cfg["dms"])
    sense = sum(len(_valid(cfg, w)[0]) * (12 * grids * w["n_px"] ** 2 + 5 * w["n_fft"] ** 2 * math.log2(w["n_fft"] ** 2))
                for w in cfg["wfs"])
    if kind == "measure":
        return {"bytes": read + surf + 4 * (nc + ns), "flops": sense}
    if kind == "interaction":
        return {"bytes": read + surf + 4 * (nc + nc * ns), "flops": 3 * sense}
    if kind == "gradient":
        more = 0 if case["wrt"] == "commands" else 4 * case["n_vec"] * (
            sum((w["n_sub"] * w["n_px"]) ** 2 for w in cfg["wfs"]) + sum(lay["n"] ** 2 for lay in cfg["layers"]))
        return {"bytes": read + surf + 4 * (nc + ns) * (1 + case["n_vec"]) + more, "flops": (3 + case["n_vec"]) * sense}
    m2 = (cfg["science"][0]["n_px"] * cfg["science"][0]["pad"]) ** 2
    one = {"bytes": ESIZE[case["dtype"]] * nc * ns + real * (read + surf + 4 * (ns + 2 * nc) + 16 * m2),
           "flops": real * (2 * nc * ns + sense + 5 * m2 * math.log2(m2))}
    end = 8 * m2 if kind == "exposure" else 0
    return {"bytes": steps * one["bytes"] + end, "flops": steps * one["flops"]}


# ------------------------------------------------------------------------------------------
# the same in 64 bits
# ------------------------------------------------------------------------------------------
def _axis64(x, n, periodic):
    i = torch.floor(x)
    t, i = x - i, i.long()
    if periodic:
        return i % n, (i + 1) % n, t
    t = torch.where(i < 0, 0.0, torch.where(i >= n - 1, 1.0, t))
    i = i.clamp(0, n - 2)
    return i, i + 1, t


def _view64(cfg, w, alt):
    """Positions (x, y) of a sensor's pupil samples projected to an altitude."""
    n = w["n_sub"] * w["n_px"]
    f = 1 - alt / w["height"] if w["type"] == "lgs" else 1.0
    x = (torch.arange(n, device="cuda", dtype=torch.float64) - 0.5 * (n - 1)) * (cfg["D"] / n) * f
    return x + alt * w["theta"][0], x + alt * w["theta"][1]


def _dm_rows64(cfg, w, m):
    """Influence of a DM's actuator columns / rows on a sensor's pupil columns / rows."""
    s2 = m["pitch"] ** 2 / (2 * math.log(1 / m["coupling"]))
    g = []
    for x, na in zip(_view64(cfg, w, m["alt"]), (m["nx"], m["ny"])):
        i0, i1, t = _axis64(x / m["surf_dx"] + 0.5 * (m["surf_n"] - 1), m["surf_n"], False)
        at = lambda i: (i.double() - 0.5 * (m["surf_n"] - 1)) * m["surf_dx"]  # noqa: E731
        a = (torch.arange(na, device="cuda", dtype=torch.float64) - 0.5 * (na - 1)) * m["pitch"]
        e = [torch.exp(-((at(i)[:, None] - a) ** 2) / (2 * s2)) for i in (i0, i1)]
        g.append((1 - t)[:, None] * e[0] + t[:, None] * e[1])
    return g


def _phase64(cfg, w, screens, commands):
    """Residual phase of a sensor's pupil at step 0."""
    out = 0.0
    for lay, s in zip(cfg["layers"], screens):
        x, y = (q / lay["pixel"] + 0.5 * (lay["n"] - 1) for q in _view64(cfg, w, lay["alt"]))
        (x0, x1, tx), (y0, y1, ty) = _axis64(x, lay["n"], True), _axis64(y, lay["n"], True)
        rows = (1 - ty)[:, None] * s[y0] + ty[:, None] * s[y1]
        out = out + (1 - tx) * rows[:, x0] + tx * rows[:, x1]
    at = 0
    for m in cfg["dms"]:
        gx, gy = _dm_rows64(cfg, w, m)
        v = torch.tensor(m["valid"] != 0, device="cuda")
        n = int(v.sum())
        C = torch.zeros(v.shape, dtype=torch.float64, device="cuda").masked_scatter(v, commands[at:at + n])
        out = out - gy @ C @ gx.T
        at += n
    return out


def _spots64(cfg, w, phase):
    """(x slopes, y slopes) of the valid subapertures from the pupil phase."""
    sx, sy = _valid(cfg, w)
    p, N, b = w["n_px"], w["n_fft"], w["n_bin"]
    at = (torch.tensor(sy, device="cuda"), slice(None), torch.tensor(sx, device="cuda"))
    blocks = lambda q: q.reshape(w["n_sub"], p, w["n_sub"], p)[at]  # noqa: E731
    r = torch.arange(p, device="cuda", dtype=torch.float64)
    phi = blocks(phase) * (cfg["lambda_ref"] / w["lambda"]) - math.pi * (r[:, None] + r[None, :]) / N
    E = torch.polar(blocks(torch.tensor(_pupil(cfg, w["n_sub"] * p), device="cuda")), phi)
    F = torch.fft.fft2(E, s=(N, N))
    I = F.real ** 2 + F.imag ** 2
    if w["type"] == "lgs" and w["na_fwhm"] > 0:
        d = cfg["D"] / w["n_sub"]
        cx, cy = ((torch.tensor(q, device="cuda") - 0.5 * (w["n_sub"] - 1)) * d - o for q, o in zip((sx, sy), w["launch"]))
        dist = torch.hypot(cx, cy)
        sig = dist * w["na_fwhm"] / w["height"] ** 2 / math.sqrt(8 * math.log(2)) / (w["lambda"] / (N * d / p))
        u = torch.fft.fftfreq(N, d=1.0 / N, device="cuda", dtype=torch.float64)
        near = torch.where(dist > 0, dist, 1.0)
        t = u[None, None, :] * (cx / near)[:, None, None] + u[None, :, None] * (cy / near)[:, None, None]
        I = torch.fft.ifft2(torch.fft.fft2(I) * torch.exp(-2 * math.pi ** 2 * (sig[:, None, None] * t / N) ** 2)).real
    det = torch.roll(I, (N // 2, N // 2), (1, 2)).reshape(-1, N // b, b, N // b, b).sum((2, 4))
    c = torch.arange(N // b, device="cuda", dtype=torch.float64) - 0.5 * (N // b - 1)
    tot = det.sum((1, 2))
    return (det * c).sum((1, 2)) / tot, (det * c[:, None]).sum((1, 2)) / tot


def _slopes64(cfg, screens, commands):
    return torch.cat([s for w in cfg["wfs"] for s in _spots64(cfg, w, _phase64(cfg, w, screens, commands))])


def _philox64(counter, seed):
    """Words 0 and 1 of Philox4x32-10 at counter (k, 0, 0, 1)."""
    M = 0xFFFFFFFF

    def mul(a, x):   # 32 x 32 -> (high, low) without leaving signed 64 bits
        lo, hi = a * (x & 0xFFFF), a * (x >> 16)
        t = hi + (lo >> 16)
        return t >> 16, ((t & 0xFFFF) << 16) | (lo & 0xFFFF)
    c = [counter, torch.zeros_like(counter), torch.zeros_like(counter), torch.ones_like(counter)]
    k = [seed & M, seed >> 32 & M]
    for _ in range(10):
        (h0, l0), (h1, l1) = mul(0xD2511F53, c[0]), mul(0xCD9E8D57, c[2])
        c = [h1 ^ c[1] ^ k[0], l1, h0 ^ c[3] ^ k[1], l0]
        k = [(k[0] + 0x9E3779B9) & M, (k[1] + 0xBB67AE85) & M]
    return c[0], c[1]


def _screen64(n, pixel, r0, L0, seed):
    k = torch.arange(n * n, device="cuda", dtype=torch.int64)
    u, v = (((q >> 8).double() + 0.5) / 2 ** 24 for q in _philox64(k, seed))
    z = torch.polar(torch.sqrt(-2 * torch.log(u)), 2 * math.pi * v).reshape(n, n)
    f = torch.fft.fftfreq(n, d=pixel, device="cuda", dtype=torch.float64)
    k2 = f[:, None] ** 2 + f[None, :] ** 2
    amp = torch.sqrt(0.023 * r0 ** (-5 / 3) * (k2 + L0 ** -2) ** (-11 / 6)) / (n * pixel)
    amp[0, 0] = 0.0
    return torch.fft.ifft2(z * amp).real * n * n


def _matrix64(cfg, screens):
    """Jacobian of the slopes with respect to the commands at zero commands."""
    c = torch.zeros(inputs.n_commands(cfg), dtype=torch.float64, device="cuda")
    rows = []
    for w in cfg["wfs"]:
        sx, sy = (torch.tensor(q, device="cuda") for q in _valid(cfg, w))
        p, n = w["n_px"], w["n_sub"]
        phase = _phase64(cfg, w, screens, c).requires_grad_()
        for s in _spots64(cfg, w, phase):   # subapertures do not share samples: one backward pass has them all
            L = torch.autograd.grad(s.sum(), phase, retain_graph=True)[0].reshape(n, p, n, p)[sy, :, sx]
            cols = []
            for m in cfg["dms"]:
                gx, gy = _dm_rows64(cfg, w, m)
                gx, gy = gx.reshape(n, p, -1)[sx], gy.reshape(n, p, -1)[sy]
                D = torch.einsum("syb,sya->sba", gy, torch.einsum("syx,sxa->sya", L, gx))
                cols.append(-D[:, torch.tensor(m["valid"] != 0, device="cuda")])
            rows.append(torch.cat(cols, 1))
    return torch.cat(rows)


def _stored64(R, dtype):
    """The control matrix's values as the library stores them."""
    if dtype == "bfloat16":
        return R.bfloat16()
    if dtype == "fp8_e4m3":
        scale = R.abs().amax(1, keepdim=True) / 448
        scale = torch.where(scale < 2.0 ** -126, 1.0, scale)
        return (R / scale).to(torch.float8_e4m3fn).double() * scale.double()
    return R


def exact(case, seed):
    kind = case["kind"]
    if kind == "noalloc":
        R, s, c = _noalloc_inputs(case, seed)
        return c.double() + 0.5 * (R.double() @ s.double())
    if kind == "screens":
        return [_screen64(case["screen"], 0.0609375, 0.157, 25.0, seed + i) for i in range(case["n_layers"])]
    cfg = _system(case)
    if kind == "tikhonov":
        D = _tikhonov_input(cfg, seed).double()
        G = D.T @ D
        lam = 1e-2 * float(G.diagonal().sum()) / G.shape[0]
        G.diagonal().add_(lam)
        return -torch.cholesky_solve(D.T, torch.linalg.cholesky(G)), lam
    if kind == "product":
        R, s = _stored64(_control(cfg), case["dtype"]), _draws(case, cfg, seed).double()
        return torch.cat([s @ r.double().T for r in R.split(512)], 1)
    if kind in ("batch", "exposure") or case["noise"]:
        return None   # noise turns the last bit of an intensity into whole counts
    screens = [s.double() for s in _screens(cfg, _generator(seed))]
    if kind == "interaction":
        return _matrix64(cfg, screens)
    if kind == "step":
        c = torch.zeros(inputs.n_commands(cfg), dtype=torch.float64, device="cuda")
        s = _slopes64(cfg, screens, c)
        R = _stored64(_control(cfg), case["dtype"])
        q = cfg["science"][0]
        star = dict(type="ngs", theta=q["theta"], n_sub=q["n_px"] // 8, n_px=8)
        phi = _phase64(cfg, star, screens, c) * (cfg["lambda_ref"] / q["lambda"])
        A = torch.tensor(_pupil(cfg, q["n_px"]), device="cuda")
        sr = float((torch.polar(A, phi).sum().abs() / A.sum()) ** 2)
        return {"commands": torch.cat([cfg["gain"] * (r.double() @ s) for r in R.split(512)])[None], "strehl": np.array([[[sr, sr]]])}
    c, g = _draws(case, cfg, seed)
    if kind == "measure":
        return _slopes64(cfg, screens, c.double())
    c = c.double().requires_grad_()
    if case["wrt"] == "commands":
        s = _slopes64(cfg, screens, c)
        return s.detach(), torch.autograd.grad(s, c, g[0].double())[0]
    for q in screens:
        q.requires_grad_()
    phases = [_phase64(cfg, w, screens, c) for w in cfg["wfs"]]
    s = torch.cat([v for w, phase in zip(cfg["wfs"], phases) for v in _spots64(cfg, w, phase)])
    rows = [torch.autograd.grad(s, [c] + phases + screens, v.double(), retain_graph=True) for v in g]
    n = 1 + len(phases)
    return (torch.stack([r[0] for r in rows]), torch.stack([torch.cat([q.reshape(-1) for q in r[1:n]]) for r in rows]),
            torch.stack([torch.cat([q.reshape(-1) for q in r[n:]]) for r in rows]))
