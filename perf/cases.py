"""What the performance of the LSRTM operators is measured on.

Each case is one pass of a user's program through the public entry points of
`paper_2508_10405_gb300`, at the sizes of this repository's workloads (the
presets of `lsrtm_inputs`, the options of `bench.py`), with the record length
of the long surveys cut so that a pass stays below half a second: every time
step of a record costs the same.

    listed()            the cases
    draw(rng)           one more case of the same ranges
    prepare(case, seed) inputs and operator handle on the GPU
    run(state)          one pass
    work(case)          bytes and operations a pass cannot do without
    exact(case, seed)   the outputs of run() in 64 bits, by plain torch
"""
import math

import numpy as np
import torch

import paper_2508_10405_gb300 as gb

BANDS = {"fp32": gb.BAND_FP32, "bf16": gb.BAND_BF16, "fp16": gb.BAND_FP16}
TIME_KINDS = ("born", "adjoint", "autograd", "psf", "cg", "model")


# --------------------------------------------------------------------------
# Cases
# --------------------------------------------------------------------------

def _survey(name, kind, *, nz, nx, ny=1, dx, dt, nt, order, f0, shots, vmin=1500.0, vmax=2500.0, npml=20, rec_step=1,
            bands="fp32", fs=False, window=0, spacing=20, iters=2, recon="boundary"):
    c = {"name": name} if name else {}
    c |= dict(kind=kind, nz=nz, ny=ny, nx=nx, dx=dx, dt=dt, nt=nt, order=order, npml=npml, f0=f0, shots=shots,
             vmin=vmin, vmax=vmax, rec_step=rec_step, bands=bands, fs=fs, window=window, recon=recon)
    if kind == "psf":
        c["spacing"] = spacing
    if kind == "cg":
        c["iters"] = iters
    return c


def listed():
    return [
        # the smallest call: Born modelling of one shot on a 101 x 101 grid (order 4, full 1000-step record);
        # a few thousand cells per time step, so launches and latency count
        _survey("born_1shot_101", "born", nz=101, nx=101, dx=10.0, dt=1e-3, nt=1000, order=4, f0=15.0, shots=1),
        # the differentiation path: 16 shots on 200 x 200 through the autograd Function, forward and backward
        _survey("autograd_16shot_200", "autograd", nz=200, nx=200, dx=10.0, dt=1e-3, nt=750, order=4, f0=12.0,
                shots=16),
        # one L of the 2D survey that the benchmark inverts: 96 shots, 384 x 1152, order 8, a receiver in every cell
        _survey("born_96shot_384x1152", "born", nz=384, nx=1152, dx=8.0, dt=0.8e-3, nt=256, order=8, f0=15.0, shots=96,
                vmax=4700.0),
        # one L^T of the same survey with FP16 boundary bands (bench.py's storage); the bands of the background are
        # kept by the handle as in a CG loop
        _survey("adjoint_96shot_384x1152", "adjoint", nz=384, nx=1152, dx=8.0, dt=0.8e-3, nt=256, order=8, f0=15.0,
                shots=96, vmax=4700.0, bands="fp16"),
        # PSF probe L^T L comb of the marine line: 120 shots of uneven aperture windows and streamer lengths
        _survey("psf_120shot_windows", "psf", nz=300, nx=2000, dx=12.5, dt=1e-3, nt=200, order=8, f0=20.0, shots=120,
                vmax=3200.0, window=100, spacing=20),
        # a whole call: CGNR on a free-surface survey of odd size, receivers on every second cell
        _survey("cg_12shot_free_surface", "cg", nz=187, nx=411, dx=10.0, dt=1e-3, nt=400, order=8, f0=15.0, shots=12,
                vmax=3500.0, rec_step=2, fs=True, iters=2),
        # data-domain input: nonlinear modelling of 48 shots and the muted residual against observed records
        _survey("model_mute_48shot", "model", nz=384, nx=1152, dx=8.0, dt=0.8e-3, nt=384, order=8, f0=15.0, shots=48,
                vmax=4700.0),
        # one L of the 3D survey (dipping layers, 128 x 256 x 256), two of its shots
        _survey("born_3d_2shot", "born", nz=128, ny=256, nx=256, dx=12.5, dt=1e-3, nt=96, order=8, f0=20.0, shots=2,
                vmax=3500.0, rec_step=2),
        # one L^T of the 3D survey with BF16 bands
        _survey("adjoint_3d_2shot", "adjoint", nz=128, ny=256, nx=256, dx=12.5, dt=1e-3, nt=96, order=8, f0=20.0,
                shots=2, vmax=3500.0, rec_step=2, bands="bf16"),
        # image-domain CGNR with the interpolated PSF Hessian on the marine-line image, both parameters
        dict(name="psf_cg_300x2000", kind="psf_cg", nz=300, nx=2000, spacing=20, iters=6, mask=3),
        # Wiener deblurring of the marine-line image (the Fourier form)
        dict(name="wiener_300x2000", kind="wiener", nz=300, nx=2000, spacing=20, eps=1e-3),
        # the space-domain 11 x 11 deblurring filters of the same image
        dict(name="deblur_300x2000", kind="deblur", nz=300, nx=2000, spacing=20, flen=11, eps=1e-3),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("born", "adjoint", "born", "adjoint", "autograd", "psf", "cg", "model", "born3", "adjoint3",
                       "psf_cg", "wiener", "deblur"))
    if kind in ("psf_cg", "wiener", "deblur"):
        s = rng.choice((12, 15, 16, 20, 20))
        c = dict(kind=kind, nz=rng.randint(90, 300), nx=_log(rng, 200, 2000), spacing=s)
        if kind == "psf_cg":
            return c | dict(iters=rng.randint(2, 6), mask=rng.choice((1, 2, 3, 3)))
        c["eps"] = rng.choice((1e-3, 3e-3, 1e-2))
        return c | dict(flen=rng.choice((7, 9, 11))) if kind == "deblur" else c
    if kind in ("born3", "adjoint3"):
        order = rng.choice((4, 8))
        return _survey("", kind[:-1], nz=rng.randint(40, 128), ny=rng.randint(48, 200), nx=rng.randint(48, 256), dx=12.5,
                       dt=1e-3, nt=rng.randint(60, 96), order=order, f0=20.0, shots=rng.randint(1, 2), vmax=3500.0,
                       npml=rng.choice((10, 16, 20)), rec_step=rng.choice((1, 2, 3)),
                       bands=rng.choice(("fp32", "bf16", "fp16")))
    order = rng.choice((4, 8, 8))
    nz, nx = _log(rng, 80, 384), _log(rng, 90, 1152)
    cells = (nz + 40) * (nx + 40)
    fs = kind != "psf" and rng.random() < 0.25
    if kind in ("autograd", "cg"):
        top, nt = 4e6, rng.randint(200, 500)
    else:
        top, nt = 2.2e7, rng.randint(200, 600 if cells < 2e5 else 250)
    shots = max(1, min(_log(rng, 1, 96), int(top / cells)))
    vmax = rng.choice((2500.0, 3500.0, 4700.0))
    recon = "checkpoint" if kind == "adjoint" and not fs and rng.random() < 0.25 else "boundary"
    return _survey("", kind, nz=nz, nx=nx, dx=10.0, dt=0.9e-3, nt=nt, order=order, f0=15.0, shots=shots, vmax=vmax,
                   npml=rng.choice((12, 20, 20, 25)), rec_step=rng.choice((1, 1, 2, 5)),
                   bands=rng.choice(("fp32", "fp16", "bf16")), fs=fs, window=rng.randint(30, 100) if kind == "psf" else 0,
                   spacing=rng.choice((12, 15, 20)), iters=rng.randint(1, 2), recon=recon)


# --------------------------------------------------------------------------
# Inputs
# --------------------------------------------------------------------------

def _gen(seed):
    g = torch.Generator()
    g.manual_seed(int(seed) * 7919 + 17)
    return g


def _uniform(g, lo, hi, n):
    return (lo + (hi - lo) * torch.rand(n, generator=g, dtype=torch.float64)).tolist()


def _earth(case, seed):
    """Smoothed layered velocity, Gardner density and reflectors on the layer boundaries (dln Vp, dln Ip)."""
    g = _gen(seed)
    nz, ny, nx = case["nz"], case["ny"], case["nx"]
    f = dict(device="cuda", dtype=torch.float64)
    z = torch.arange(nz, **f).view(nz, 1, 1)
    y = (torch.arange(ny, **f) / max(ny - 1, 1)).view(1, ny, 1)
    x = (torch.arange(nx, **f) / max(nx - 1, 1)).view(1, 1, nx)
    vmin, vmax, n = case["vmin"], case["vmax"], 8
    vp = vmin + 0.8 * (vmax - vmin) * (z / max(nz - 1, 1)) + 0 * x + 0 * y
    dm = torch.zeros((2, nz, ny, nx), **f)
    # layer boundaries from just below the receivers (reached within a short record) to the bottom
    depth = [math.exp(u) / nz for u in _uniform(g, math.log(9.0), math.log(0.95 * nz), n - 2)] + [12.0 / nz, 25.0 / nz]
    dip, phase = _uniform(g, -0.12, 0.12, n), _uniform(g, 0, 2 * math.pi, n)
    jump, a, b = _uniform(g, -0.06, 0.12, n), _uniform(g, -0.08, 0.08, n), _uniform(g, -0.08, 0.08, n)
    for k in range(n):
        surf = nz * depth[k] * (1 + dip[k] * (x - 0.5) + 0.5 * dip[k] * (y - 0.5)
                                + 0.05 * torch.sin(2 * math.pi * (2 * x + y) + phase[k]))
        vp = vp + 0.5 * jump[k] * (vmax - vmin) * (1 + torch.tanh((z - surf) / 12.0))
        bump = torch.exp(-0.5 * ((z - surf) / 0.8) ** 2)
        dm[0] += a[k] * bump
        dm[1] += b[k] * bump
    vp = vp.clamp(vmin, vmax)
    rho = 310.0 * vp ** 0.25
    dm = dm * (z >= 6)   # no reflector through the sources and receivers
    shape = (nz, nx) if ny == 1 else (nz, ny, nx)
    return (vp.float().view(shape).contiguous(), rho.float().view(shape).contiguous(),
            dm.float().view((2,) + shape).contiguous())


def _geometry(case, seed):
    """Sources along the surface, receivers on every rec_step-th surface cell, or a towed streamer of uneven length
    with its aperture window."""
    g = _gen(seed + 1)
    nz, ny, nx, S, st = case["nz"], case["ny"], case["nx"], case["shots"], case["rec_step"]
    jit = torch.rand(S, generator=g, dtype=torch.float64).numpy()
    if ny > 1:
        side = int(math.ceil(math.sqrt(S)))
        src = [(1 * ny + int((k // side + 0.5 + 0.3 * (jit[k] - 0.5)) * ny / side)) * nx + int((k % side + 0.5) * nx / side)
               for k in range(S)]
        ry, rx = np.meshgrid(np.arange(0, ny, st), np.arange(0, nx, st), indexing="ij")
        rec = ((1 * ny + ry) * nx + rx).ravel()
        return dict(src_idx=np.array(src, np.int32), rec_ptr=(np.arange(S + 1) * rec.size).astype(np.int32),
                    rec_idx=np.tile(rec, S).astype(np.int32))
    xs = np.clip(((np.arange(S) + 0.2 + 0.6 * jit) * nx / S).astype(np.int64), 0, nx - 1)
    row = 2 * nx
    if not case["window"]:
        rec = row + np.arange(0, nx, st)
        return dict(src_idx=(row + xs).astype(np.int32), rec_ptr=(np.arange(S + 1) * rec.size).astype(np.int32),
                    rec_idx=np.tile(rec, S).astype(np.int32))
    ptr, idx, x0, wn = [0], [], [], []
    chan = torch.randint(120, 241, (S,), generator=g).numpy()
    for k in range(S):
        rx = xs[k] + 4 + 2 * np.arange(min(int(chan[k]), max(1, nx // 4)))
        rx = rx[rx < nx] if (rx < nx).any() else xs[k:k + 1]
        lo, hi = max(0, int(xs[k]) - case["window"]), min(nx, int(rx.max()) + case["window"] + 1)
        idx.append(row + rx)
        ptr.append(ptr[-1] + rx.size)
        x0.append(lo)
        wn.append(hi - lo)
    return dict(src_idx=(row + xs).astype(np.int32), rec_ptr=np.array(ptr, np.int32),
                rec_idx=np.concatenate(idx).astype(np.int32), win_x0=np.array(x0, np.int32), win_nx=np.array(wn, np.int32))


def _ricker(case):
    t = np.arange(case["nt"]) * case["dt"] - 1.0 / case["f0"]
    a = (math.pi * case["f0"] * t) ** 2
    return ((1 - 2 * a) * np.exp(-a)).astype(np.float32)


def _records(case, geom, seed, scale):
    """Records with a few reflection-like events: hyperbolae of random depth, velocity and strength."""
    g = _gen(seed + 2)
    nx, ny, dx = case["nx"], case["ny"], case["dx"]
    rec = torch.from_numpy(geom["rec_idx"].astype(np.int64)).cuda()
    cnt = torch.from_numpy(np.diff(geom["rec_ptr"]).astype(np.int64)).cuda()
    src = torch.repeat_interleave(torch.from_numpy(geom["src_idx"].astype(np.int64)).cuda(), cnt)
    off2 = (((rec % nx) - (src % nx)).float() * dx) ** 2
    off2 = off2 + ((((rec // nx) % ny) - ((src // nx) % ny)).float() * dx) ** 2
    t = (torch.arange(case["nt"], device="cuda", dtype=torch.float32) + 1) * case["dt"]
    d = torch.zeros((rec.numel(), case["nt"]), device="cuda", dtype=torch.float32)
    T = case["nt"] * case["dt"]
    for t0, v, a in zip(_uniform(g, 0.3 * T, 0.9 * T, 3), _uniform(g, 1600.0, 2600.0, 3), _uniform(g, 0.3, 1.0, 3)):
        u = (math.pi * case["f0"] * (t[None, :] - torch.sqrt(t0 * t0 + off2 / (v * v))[:, None])) ** 2
        d += a * scale * (1 - 2 * u) * torch.exp(-u)
    return d


def _image_inputs(case, seed):
    """Migrated image of thin dipping reflectors and its blurred, dimmed remigration, both parameters."""
    g = _gen(seed)
    nz, nx = case["nz"], case["nx"]
    f = dict(device="cuda", dtype=torch.float64)
    z, x = torch.arange(nz, **f).view(nz, 1), torch.arange(nx, **f).view(1, nx)
    depth = z / max(nz - 1, 1)
    m, b = torch.zeros((2, nz, nx), **f), torch.zeros((2, nz, nx), **f)
    n = 30
    at, dip = _uniform(g, 0.03, 0.97, n), _uniform(g, -0.12, 0.12, n)
    amp = [_uniform(g, -0.1, 0.1, n) for _ in range(2)]
    for k in range(n):
        u = (z - (at[k] * nz + dip[k] * (x - nx / 2))) ** 2
        wide = 0.6 + 2.0 * depth
        line, blur = torch.exp(-0.5 * u / 0.36), torch.exp(-0.5 * u / (0.36 + wide ** 2)) * (0.6 / torch.sqrt(0.36 + wide ** 2))
        for q in range(2):
            m[q] += amp[q][k] * line
            b[q] += amp[q][k] * blur * (1 - 0.5 * depth)
    noise = torch.randn((2, nz, nx), generator=g, dtype=torch.float64).cuda()
    b += 0.01 * b.abs().amax(dim=(1, 2), keepdim=True) * noise
    return m.float(), b.float()


def _psf_inputs(case, seed):
    """PSF images of the Vp and Ip combs: a tilted band-limited blob around every node, weaker across parameters."""
    g = _gen(seed + 3)
    nz, nx, s = case["nz"], case["nx"], case["spacing"]
    f = dict(device="cuda", dtype=torch.float64)
    nkz, nkx = (nz - 1 - s // 2) // s + 1, (nx - 1 - s // 2) // s + 1
    z, x = torch.arange(nz, **f), torch.arange(nx, **f)
    kz, kx = ((z - s // 2 + s // 2) // s).clamp(0, nkz - 1).long(), ((x - s // 2 + s // 2) // s).clamp(0, nkx - 1).long()
    dz, dx = (z - (s // 2 + kz * s)).view(nz, 1), (x - (s // 2 + kx * s)).view(1, nx)
    depth = (z / max(nz - 1, 1)).view(nz, 1)
    out = []
    for j in range(2):
        q = []
        for i in range(2):
            r = torch.rand((3, nkz, nkx), generator=g, dtype=torch.float64).cuda()[:, kz][:, :, kx]
            sig, tilt, a = (0.08 + 0.08 * depth) * s * (0.85 + 0.3 * r[0]), 0.8 * (r[1] - 0.5), (1 - 0.6 * depth) * (0.8 + 0.4 * r[2])
            u = (dz * torch.cos(tilt) + dx * torch.sin(tilt)) / sig
            v = (dx * torch.cos(tilt) - dz * torch.sin(tilt)) / (2 * sig)
            e = torch.exp(-0.5 * (u * u + v * v))
            q.append(a * e * (1 - u * u) if i == j else 0.3 * a * e * u)
        out.append(torch.stack(q).float().contiguous())
    return out


def _handle(case, vp, rho, geom):
    nd = 3 if case["ny"] > 1 else 2
    recon = gb.RECON_CHECKPOINT if case["recon"] == "checkpoint" else gb.RECON_AUTO
    return gb.Lsrtm(ndim=nd, nz=case["nz"], ny=case["ny"], nx=case["nx"], dz=case["dx"], dy=case["dx"], dx=case["dx"],
                    dt=case["dt"], nt=case["nt"], fd_order=case["order"], npml=case["npml"], f0=case["f0"], vp=vp,
                    rho=rho, wavelet=_ricker(case), band_precision=BANDS[case["bands"]], recon_mode=recon,
                    free_surface=case["fs"], **geom)


def _image_handle(case):
    """The handle of a program that works on images alone: a one-shot geometry on the image's grid."""
    v = torch.full((case["nz"], case["nx"]), 2000.0, device="cuda")
    return gb.Lsrtm(ndim=2, nz=case["nz"], nx=case["nx"], dz=10.0, dx=10.0, dt=1e-3, nt=2, fd_order=8, npml=8, f0=20.0,
                    vp=v, rho=v, wavelet=np.ones(2, np.float32), src_idx=[case["nx"]], rec_ptr=[0, 1], rec_idx=[case["nx"]])


def _mute(case):
    return dict(v_mute=case["vmin"], t0=1.0 / case["f0"], t_taper=0.25 / case["f0"], o_max=0.75 * case["nx"] * case["dx"],
                o_taper=0.1 * case["nx"] * case["dx"])


def _inputs(case, seed):
    if case["kind"] not in TIME_KINDS:
        m, b = _image_inputs(case, seed)
        return dict(m=m, b=b, psf=_psf_inputs(case, seed) if case["kind"] == "psf_cg" else None)
    vp, rho, dm = _earth(case, seed)
    geom = _geometry(case, seed)
    d = None
    if case["kind"] not in ("born", "psf"):
        # the records' amplitude: that of a pressure wave of this source
        d = _records(case, geom, seed, case["dt"] / case["dx"] ** (3 if case["ny"] > 1 else 2))
    return dict(vp=vp, rho=rho, dm=dm, geom=geom, d=d)


def prepare(case, seed):
    s = _inputs(case, seed)
    s["case"] = case
    s["h"] = _handle(case, s["vp"], s["rho"], s["geom"]) if case["kind"] in TIME_KINDS else _image_handle(case)
    if case["kind"] == "autograd":
        s["op"] = gb.born_op()
        s["dm"].requires_grad_(True)
    return s


def run(s):
    case, h = s["case"], s["h"]
    kind = case["kind"]
    if kind == "born":
        return h.born(s["dm"])
    if kind == "adjoint":
        return h.adjoint(s["d"])
    if kind == "autograd":
        d = s["op"].apply(s["dm"], h)
        (g,) = torch.autograd.grad((d * s["d"]).sum(), s["dm"])
        return d.detach(), g
    if kind == "psf":
        return h.psf(1, case["spacing"])
    if kind == "cg":
        return h.cg_solve(s["d"], case["iters"])
    if kind == "model":
        d = h.model()
        return d, h.mute_residual(s["d"], d, **_mute(case))
    if kind == "psf_cg":
        return h.psf_cg(s["m"], s["psf"][0], s["psf"][1], case["iters"], spacing=case["spacing"], param_mask=case["mask"])
    if kind == "wiener":
        return h.deblur_wiener(s["m"], s["b"], spacing=case["spacing"], eps=case["eps"])
    return h.deblur(s["m"], s["b"], spacing=case["spacing"], flen=case["flen"], eps=case["eps"], return_filters=True)


# --------------------------------------------------------------------------
# Work
# --------------------------------------------------------------------------

def _cell_updates(case):
    p = 2 * case["npml"]
    nz, ny = case["nz"] + p, (case["ny"] + p if case["ny"] > 1 else 1)
    if not case["window"]:
        return case["shots"] * nz * ny * (case["nx"] + p) * case["nt"]
    g = _geometry(case, 0)
    return int((g["win_nx"] + p).sum()) * nz * case["nt"]


def work(case):
    """A time step reads and writes the pressure and the velocities (of both fields in L and L^T) once and reads the
    model once; records and images move once."""
    kind = case["kind"]
    if kind in TIME_KINDS:
        nd, taps = (3 if case["ny"] > 1 else 2), case["order"]
        n = _cell_updates(case)
        state = 4 * (1 + nd) * 2
        # a stencil of 2M taps: M differences and M multiply-adds; one per direction and stage
        st = 2 * nd * 1.5 * taps
        born = (2 * state + 16, 2 * st + 8 * nd)
        adj = (2 * state + 8 + 16, 3 * st + 10 * nd)
        model = (state + 8, st + 4 * nd)
        per = {"born": [born], "adjoint": [adj], "autograd": [born, adj], "psf": [born, adj], "model": [model],
               "cg": [born, adj] * case.get("iters", 0) + [born, adj]}[kind]
        rec = int(_geometry(case, 0)["rec_ptr"][-1]) * case["nt"] * 4
        img = 2 * case["nz"] * case["ny"] * case["nx"] * 4
        extra = {"model": 4 * rec, "cg": (2 + 4 * case.get("iters", 0)) * (rec + img)}.get(kind, len(per) * (rec + img))
        return {"bytes": float(n * sum(b for b, _ in per) + extra), "flops": float(n * sum(f for _, f in per))}
    px, s = case["nz"] * case["nx"], case["spacing"]
    nk = ((case["nz"] - 1 - s // 2) // s + 1) * ((case["nx"] - 1 - s // 2) // s + 1)
    if kind == "psf_cg":
        blocks, L = (4 if case["mask"] == 3 else 1), 2 * ((s - 1) // 2) + 1
        return {"bytes": float(px * 4 * 8), "flops": float((2 * case["iters"] + 1) * px * L * L * blocks * 10)}
    N = 2 * s
    if kind == "wiener":   # three transforms of N x N a block, 5 N^2 log2 N^2 each
        return {"bytes": float(px * 4 * 6), "flops": float(2 * nk * (3 * 5 * N * N * 2 * math.log2(N) + 20 * N * N))}
    n = case["flen"] ** 2   # lag sums, Cholesky factor, the two solves, the filter itself
    return {"bytes": float(px * 4 * 6 + 2 * nk * n * 4),
            "flops": float(2 * nk * (2 * n * (N + 1) * (N + 1) + n ** 3 / 3 + 2 * n * n) + 2 * px * 4 * 2 * n)}


# --------------------------------------------------------------------------
# The same in 64 bits
# --------------------------------------------------------------------------

def _taps(f, dim, c, first):
    """sum_l c_l (f[i + l - 1 + first] - f[i - l + first]), zero outside."""
    M = len(c)
    shape = list(f.shape)
    n = shape[dim]
    shape[dim] = n + 2 * M
    p = f.new_zeros(shape)
    p.narrow(dim, M, n).copy_(f)
    acc = None
    for l in range(1, M + 1):
        a = p.narrow(dim, M + l - 1 + first, n) - p.narrow(dim, M - l + first, n)
        acc = a.mul_(c[l - 1]) if acc is None else acc.add_(a, alpha=c[l - 1])
    return acc


class _Dplus(torch.autograd.Function):
    @staticmethod
    def forward(ctx, f, dim, c):
        ctx.a = (dim, c)
        return _taps(f, dim, c, 1)

    @staticmethod
    def backward(ctx, g):
        return -_taps(g, ctx.a[0], ctx.a[1], 0), None, None


class _Dminus(torch.autograd.Function):
    @staticmethod
    def forward(ctx, f, dim, c):
        ctx.a = (dim, c)
        return _taps(f, dim, c, 0)

    @staticmethod
    def backward(ctx, g):
        return -_taps(g, ctx.a[0], ctx.a[1], 1), None, None


def _profile(N, o, n, case, vmax, half, top_open):
    L = case["npml"]
    i = np.arange(N) + (0.5 if half else 0.0)
    dist = np.maximum(0.0, np.maximum(o - 0.5 - i, i - (o + n - 0.5)))
    if top_open:
        dist[:o] = 0.0
    r = dist / L
    d = -3.0 * vmax * math.log(1e-4) / (2 * L * case["dx"]) * r * r
    al = np.maximum(math.pi * case["f0"] * (1 - r), 0.0)
    b = np.where(dist > 0, np.exp(-(d + al) * case["dt"]), 0.0)
    a = np.where(dist > 0, d * (b - 1) / np.where(dist > 0, d + al, 1.0), 0.0)
    return torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda()


class _Wave64:
    """The discrete operators in 64 bits: staggered leapfrog of order 2M, CPML strips, optional free surface and
    aperture windows; L by the linearised recursion, L^T by reverse-mode differentiation of it."""

    def __init__(self, case, inp):
        self.c, self.geom = case, inp["geom"]
        self.vp, self.rho = inp["vp"].double(), inp["rho"].double()
        self.nd = 3 if case["ny"] > 1 else 2
        self.taps = [x / case["dx"] for x in ((9 / 8, -1 / 24) if case["order"] == 4 else
                                              (1225 / 1024, -245 / 3072, 49 / 5120, -5 / 7168))]
        self.wav = torch.from_numpy(_ricker(case)).double()
        self.vmax = float(inp["vp"].max())
        cells = (case["nz"] + 2 * case["npml"]) * (case["nx"] + 2 * case["npml"])
        cells *= case["ny"] + 2 * case["npml"] if self.nd == 3 else 1
        self.chunk = max(1, min(case["shots"], int(6e10 / (cells * 8 * 5 * case["nt"]))))

    def _setup(self, shots):
        """Padded model, profiles, sources and receivers of some shots, [S, Nz, (Ny,) Nx]."""
        c, geom, P = self.c, self.geom, self.c["npml"]
        nz, ny, nx = c["nz"], c["ny"], c["nx"]
        win = "win_x0" in geom
        wx = geom["win_x0"][shots] if win else np.zeros(1, np.int64)
        wn = geom["win_nx"][shots] if win else np.full(1, nx)
        Nx = int(wn.max()) + 2 * P
        z = np.arange(nz + 2 * P) - P
        iz = np.clip(np.abs(z) if c["fs"] else z, 0, nz - 1)
        zin = (z < nz) & ((z >= 0) | c["fs"])
        xr = np.arange(Nx)[None, :] - P
        ix = np.clip(xr, 0, wn[:, None] - 1) + wx[:, None]
        xin = (xr >= 0) & (xr < wn[:, None])
        ok = xr < wn[:, None] + P
        t = lambda v: torch.from_numpy(np.ascontiguousarray(v)).cuda()  # noqa: E731
        if self.nd == 2:
            at = (t(iz)[None, :, None], t(ix)[:, None, :])
            inner = (t(zin)[None, :, None] & t(xin)[:, None, :]).double()
            self.valid = None if not win else t(ok)[:, None, :].double()
        else:
            yr = np.arange(ny + 2 * P) - P
            at = (t(iz)[None, :, None, None], t(np.clip(yr, 0, ny - 1))[None, None, :, None], t(ix)[:, None, None, :])
            inner = (t(zin)[None, :, None, None] & t((yr >= 0) & (yr < ny))[None, None, :, None]
                     & t(xin)[:, None, None, :]).double()
            self.valid = None
        self.at, self.inner = at, inner
        vp, rho = self.vp[at], self.rho[at]
        self.kdt, self.binv = c["dt"] * rho * vp * vp, 1.0 / rho
        self.dims = list(range(1, self.nd + 1))
        last = torch.from_numpy((wn + 2 * P - 1)).cuda()
        self.bu = []
        for d in self.dims:
            n = self.binv.shape[d]
            nxt = torch.cat([self.binv.narrow(d, 1, n - 1), self.binv.narrow(d, n - 1, 1)], d)
            if win and d == self.nd:
                e = torch.arange(n, device="cuda")[None, None, :] == last[:, None, None]
                nxt = torch.where(e, self.binv, nxt)
            self.bu.append(0.5 * c["dt"] * (self.binv + nxt))
        self.pml = []
        for d in self.dims:
            lead = [1] * (self.nd + 1)
            if win and d == self.nd:
                both = []
                for half in (False, True):
                    ab = [_profile(Nx, P, int(n), c, self.vmax, half, False) for n in wn]
                    both += [torch.stack([q[k] for q in ab])[:, None, :] for k in range(2)]
            else:
                n = {1: nz, self.nd: int(wn[0])}.get(d, ny)
                lead[d] = n + 2 * P
                both = [q.view(lead) for half in (False, True)
                        for q in _profile(n + 2 * P, P, n, c, self.vmax, half, c["fs"] and d == 1)]
            self.pml.append(both)
        S = len(shots)
        self.shape = (S,) + tuple(self.binv.shape[1:])
        off = (lambda k, s: ((k // (nx * ny) + P) * (ny + 2 * P if self.nd == 3 else 1)  # noqa: E731
                             + (((k // nx) % ny) + P if self.nd == 3 else 0)) * Nx
               + (k % nx) - (geom["win_x0"][s] if win else 0) + P)
        self.src = t(np.array([off(int(geom["src_idx"][s]), s) for s in shots], np.int64))
        rs, rc = [], []
        for i, s in enumerate(shots):
            k = geom["rec_idx"][geom["rec_ptr"][s]:geom["rec_ptr"][s + 1]].astype(np.int64)
            rc.append(off(k, s))
            rs.append(np.full(k.size, i))
        self.rs, self.rc = t(np.concatenate(rs)), t(np.concatenate(rc))
        self.vol = c["dx"] ** self.nd

    def _mirror(self, f, even):
        """Rows above the surface row from their mirror rows (p odd with p = 0 on it, v_z even)."""
        P = self.c["npml"]
        if even:
            return torch.cat([f[:, P:2 * P].flip(1), f[:, P:]], 1)
        return torch.cat([-f[:, P + 1:2 * P + 1].flip(1), torch.zeros_like(f[:, :1]), f[:, P + 1:]], 1)

    def _v_stage(self, p, v, psi, src):
        G = []
        for k, d in enumerate(self.dims):
            g = _Dplus.apply(p, d, self.taps)
            psi[k] = self.pml[k][3] * psi[k] + self.pml[k][2] * g
            g = g + psi[k]
            G.append(g)
            v[k] = v[k] - self.bu[k] * g
            if src is not None:
                v[k] = v[k] - src[k]
            if self.valid is not None:
                v[k] = v[k] * self.valid
        if self.c["fs"]:
            v[0] = self._mirror(v[0], True)
        return G

    def _p_stage(self, v, psi):
        Q = 0
        for k, d in enumerate(self.dims):
            q = _Dminus.apply(v[k], d, self.taps)
            psi[k] = self.pml[k][1] * psi[k] + self.pml[k][0] * q
            Q = Q + q + psi[k]
        return Q

    def _end(self, p):
        if self.valid is not None:
            p = p * self.valid
        return self._mirror(p, False) if self.c["fs"] else p

    def _loop(self, shots, dm):
        """Records of the scattered field (dm given) or of the background field."""
        self._setup(shots)
        zero = torch.zeros(self.shape, device="cuda", dtype=torch.float64)
        p, v, a, b = zero, [zero] * self.nd, [zero] * self.nd, [zero] * self.nd
        if dm is not None:
            m = dm[(slice(None),) + self.at] * self.inner
            kd, r = self.kdt * (m[0] + m[1]), (m[1] - m[0]) * self.binv
            db = []
            for d in self.dims:
                n = r.shape[d]
                db.append(-0.5 * self.c["dt"] * (r + torch.cat([r.narrow(d, 1, n - 1), torch.zeros_like(r.narrow(d, 0, 1))], d)))
            dp, dv, da, dbb = zero, [zero] * self.nd, [zero] * self.nd, [zero] * self.nd
        out = []
        rows = torch.arange(len(shots), device="cuda")
        for n in range(self.c["nt"]):
            with torch.no_grad():
                G = self._v_stage(p, v, a, None)
                Q = self._p_stage(v, b)
                p = p - self.kdt * Q
                p.view(len(shots), -1)[rows, self.src] += self.c["dt"] / self.vol * float(self.wav[n])
                p = self._end(p)
            f = p
            if dm is not None:
                self._v_stage(dp, dv, da, [x * g for x, g in zip(db, G)])
                dp = self._end(dp - self.kdt * self._p_stage(dv, dbb) - kd * Q)
                f = dp
            out.append(f.reshape(len(shots), -1)[self.rs, self.rc])
        return torch.stack(out, 1)

    def _chunks(self):
        return [np.arange(i, min(i + self.chunk, self.c["shots"])) for i in range(0, self.c["shots"], self.chunk)]

    def born(self, dm):
        with torch.no_grad():
            return torch.cat([self._loop(s, dm.double()) for s in self._chunks()])

    def model(self):
        with torch.no_grad():
            return torch.cat([self._loop(s, None) for s in self._chunks()])

    def adjoint(self, d):
        shape = (2, self.c["nz"], self.c["nx"]) if self.nd == 2 else (2, self.c["nz"], self.c["ny"], self.c["nx"])
        g = torch.zeros(shape, device="cuda", dtype=torch.float64)
        ptr = self.geom["rec_ptr"]
        for s in self._chunks():
            dm = torch.zeros(shape, device="cuda", dtype=torch.float64, requires_grad=True)
            with torch.enable_grad():
                rec = self._loop(s, dm)
            g += torch.autograd.grad(rec, dm, d[int(ptr[s[0]]):int(ptr[s[-1] + 1])].double())[0]
            del rec
        return g


def _mute64(case, geom, d_obs, d_syn):
    m, nx = _mute(case), case["nx"]
    rec, cnt = torch.from_numpy(geom["rec_idx"].astype(np.int64)), torch.from_numpy(np.diff(geom["rec_ptr"]).astype(np.int64))
    src = torch.repeat_interleave(torch.from_numpy(geom["src_idx"].astype(np.int64)), cnt)
    o = ((rec % nx) - (src % nx)).abs().double().cuda() * case["dx"]
    t = (torch.arange(case["nt"], device="cuda", dtype=torch.float64) + 1) * case["dt"]
    ramp = lambda u, w: torch.where(u <= 0, 0.0, torch.where(u >= w, 1.0, (1 - torch.cos(math.pi * u / w)) / 2))  # noqa: E731
    mask = ramp(t[None, :] - (o / m["v_mute"] + m["t0"])[:, None], m["t_taper"]) * ramp(m["o_max"] - o, m["o_taper"])[:, None]
    return mask * (d_obs.double() - d_syn)


def _nodes(n, s):
    return torch.arange(s // 2, n, s, device="cuda")


class _PsfHessian64:
    """Interpolated PSF Hessian: column of pixel c = bilinear mix of the windows of its four nodes."""

    def __init__(self, case, psf):
        self.c, s = case, case["spacing"]
        self.h = (s - 1) // 2
        nz, nx = case["nz"], case["nx"]
        self.ax = []
        for n in (nz, nx):
            nk = len(_nodes(n, s))
            u = (torch.arange(n, device="cuda", dtype=torch.float64) - s // 2) / s
            u = u.clamp(0, nk - 1)
            k0 = u.floor().clamp(0, max(nk - 2, 0)).long()
            self.ax.append((k0, (k0 + 1).clamp(max=nk - 1), u - k0))
        self.Q = torch.stack([q.double() for q in psf])   # [input plane][output plane]
        self.Q = torch.nn.functional.pad(self.Q, (self.h,) * 4)
        self.zk, self.xk = _nodes(nz, s), _nodes(nx, s)
        self.keep = [bool(case["mask"] >> q & 1) for q in range(2)]

    def _blocks(self, az, ax):
        P = self.Q[:, :, (self.zk + self.h + az)][:, :, :, (self.xk + self.h + ax)]
        (z0, z1, wz), (x0, x1, wx) = self.ax
        R = P[:, :, z0] * (1 - wz)[:, None] + P[:, :, z1] * wz[:, None]
        return R[..., x0] * (1 - wx) + R[..., x1] * wx

    def apply(self, x, transpose):
        nz, nx, h = self.c["nz"], self.c["nx"], self.h
        y = torch.zeros_like(x)
        for az in range(-h, h + 1):
            cz = slice(max(0, -az), min(nz, nz - az))
            rz = slice(max(0, az), min(nz, nz + az))
            for a in range(-h, h + 1):
                cx = slice(max(0, -a), min(nx, nx - a))
                rx = slice(max(0, a), min(nx, nx + a))
                B = self._blocks(az, a)
                for i in range(2):
                    for j in range(2):
                        if not (self.keep[i] and self.keep[j]):
                            continue
                        if transpose:
                            y[j, cz, cx] += B[j, i, cz, cx] * x[i, rz, rx]
                        else:
                            y[i, rz, rx] += B[j, i, cz, cx] * x[j, cz, cx]
        return y

    def solve(self, m, iters):
        m = m.double() * torch.tensor(self.keep, device="cuda").double()[:, None, None]
        x, r = torch.zeros_like(m), m.clone()
        p = s = self.apply(r, True)
        gam = (s * s).sum()
        mis = [1.0]
        for _ in range(iters):
            q = self.apply(p, False)
            al = gam / (q * q).sum()
            x, r = x + al * p, r - al * q
            s = self.apply(r, True)
            new = (s * s).sum()
            p, gam = s + new / gam * p, new
            mis.append(float((r * r).sum() / (m * m).sum()) ** 0.5)
        return x, np.array(mis)


def _hat(n, s):
    """Valence of every node at every pixel of an axis."""
    i = torch.arange(n, device="cuda", dtype=torch.float64)
    return (1 - (i[None, :] - _nodes(n, s).double()[:, None]).abs() / s).clamp(min=0)


def _blend(case, add):
    """sum_k w_k block_k / sum_k w_k; add(kz, kx, z range, x range) gives a node's [2] image there."""
    nz, nx, s = case["nz"], case["nx"], case["spacing"]
    wz, wx = _hat(nz, s), _hat(nx, s)
    num = torch.zeros((2, nz, nx), device="cuda", dtype=torch.float64)
    for i, z in enumerate(_nodes(nz, s).tolist()):
        a, b = max(0, z - s), min(nz, z + s)
        num[:, a:b] += wz[i, a:b, None] * add(i, a, b)
    return num / (wz.sum(0)[:, None] * wx.sum(0)[None, :])


def _row_of_nodes(case, g, z, lo, hi):
    """Pixels z + lo .. z + hi - 1 and x_k + lo .. x_k + hi - 1 of every node of a node row, zero outside: [2, nkx, n, n]."""
    n = hi - lo
    p = torch.nn.functional.pad(g, (n, n, n, n))
    xk = _nodes(case["nx"], case["spacing"]) + n + lo
    rows = p[:, z + n + lo:z + n + hi]
    at = xk[:, None] + torch.arange(n, device="cuda")[None, :]
    return rows[:, :, at].permute(0, 2, 1, 3)


def _wiener64(case, m, b):
    s, nx = case["spacing"], case["nx"]
    zs = _nodes(case["nz"], s).tolist()
    wx = _hat(nx, s)
    m, b = m.double(), b.double()

    def add(i, lo, hi):
        F = [torch.fft.fft2(_row_of_nodes(case, g, zs[i], -s, s)) for g in (m, b)]
        p2 = F[1].abs() ** 2
        eps = case["eps"] * p2.mean(dim=(2, 3), keepdim=True)
        r = torch.fft.ifft2(F[1].conj() * F[0] * F[0] / (p2 + eps)).real
        out = torch.zeros((2, hi - lo, nx), device="cuda", dtype=torch.float64)
        for k, x in enumerate(_nodes(nx, s).tolist()):
            a, e = max(0, x - s), min(nx, x + s)
            out[:, :, a:e] += wx[k, a:e] * r[:, k, lo - zs[i] + s:hi - zs[i] + s, a - x + s:e - x + s]
        return out

    return _blend(case, add)


def _deblur64(case, m, b):
    s, nz, nx, L = case["spacing"], case["nz"], case["nx"], case["flen"]
    h, zs, xs = L // 2, _nodes(case["nz"], s).tolist(), _nodes(case["nx"], s)
    wx = _hat(nx, s)
    m, b = m.double(), b.double()
    inside = torch.ones((2, nz, nx), device="cuda", dtype=torch.float64)
    filt = []
    for z in zs:
        W = 2 * s + 1
        patch = _row_of_nodes(case, b, z, -s - h, s + h + 1)             # [2, nkx, W + 2h, W + 2h]
        ok = _row_of_nodes(case, inside, z, -s, s + 1).reshape(2, len(xs), -1, 1)
        cols = [patch[:, :, h - a:h - a + W, h - e:h - e + W].reshape(2, len(xs), -1)
                for a in range(-h, h + 1) for e in range(-h, h + 1)]
        A = torch.stack(cols, -1) * ok
        rhs = A.transpose(-1, -2) @ _row_of_nodes(case, m, z, -s, s + 1).reshape(2, len(xs), -1, 1)
        N = A.transpose(-1, -2) @ A
        tr = N.diagonal(dim1=-2, dim2=-1).sum(-1)[..., None, None] / (L * L)
        eye = torch.eye(L * L, device="cuda", dtype=torch.float64)
        f = torch.linalg.solve(N + (case["eps"] * tr + (tr == 0)) * eye, rhs * (tr != 0))
        filt.append(f.reshape(2, len(xs), L, L))
    F = torch.stack(filt, 1)
    pad = torch.nn.functional.pad(m, (h, h, h, h))
    k = torch.arange(nx, device="cuda")
    k0 = torch.div(k - s // 2, s, rounding_mode="floor")

    def add(i, lo, hi):
        out = torch.zeros((2, hi - lo, nx), device="cuda", dtype=torch.float64)
        for q in range(2):
            kk = k0 + q
            good = (kk >= 0) & (kk < len(xs))
            kk = kk.clamp(0, len(xs) - 1)
            w = torch.where(good, wx[kk, k], 0.0)
            acc = torch.zeros_like(out)
            for a in range(-h, h + 1):
                for e in range(-h, h + 1):
                    acc += F[:, i, :, a + h, e + h][:, kk][:, None, :] * pad[:, lo + h - a:hi + h - a, h - e:h - e + nx]
            out += w * acc
        return out

    return _blend(case, add), F


def exact(case, seed):
    inp = _inputs(case, seed)
    kind = case["kind"]
    if kind == "psf_cg":
        return _PsfHessian64(case, inp["psf"]).solve(inp["m"], case["iters"])
    if kind == "wiener":
        return _wiener64(case, inp["m"], inp["b"])
    if kind == "deblur":
        return _deblur64(case, inp["m"], inp["b"])
    w = _Wave64(case, inp)
    if kind == "born":
        return w.born(inp["dm"])
    if kind == "adjoint":
        return w.adjoint(inp["d"])
    if kind == "autograd":
        return w.born(inp["dm"]), w.adjoint(inp["d"])
    if kind == "psf":
        comb = torch.zeros_like(inp["dm"])
        comb[1, case["spacing"] // 2::case["spacing"], case["spacing"] // 2::case["spacing"]] = 1
        return w.adjoint(w.born(comb))
    if kind == "model":
        d = w.model()
        return d, _mute64(case, inp["geom"], inp["d"], d)
    # CGNR from zero
    d = inp["d"].double()
    x, r = torch.zeros_like(inp["dm"]).double(), d
    p = s = w.adjoint(r)
    gam, mis = (s * s).sum(), [1.0]
    for _ in range(case["iters"]):
        q = w.born(p)
        al = gam / (q * q).sum()
        x, r = x + al * p, r - al * q
        s = w.adjoint(r)
        new = (s * s).sum()
        p, gam = s + new / gam * p, new
        mis.append(float((r * r).sum() / (d * d).sum()) ** 0.5)
    return x, np.array(mis)
