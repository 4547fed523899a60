"""The work a program gives this engine, as cases that can be timed and checked.

A case is a dict of plain values; ``kind`` says which entry point it goes through:

``grad``      ``Engine.loss_grad`` (or ``loss_grad_ext`` where it asks for slice-gap, Fresnel-number
              or per-angle offset gradients): one minibatch of a reconstruction's inner loop, into
              gradient buffers that the program clears first
``autograd``  ``multislice_loss(...)`` and ``backward()``: the same inside a torch program
``forward``   ``Engine.forward``: simulated data, or the forecast of a finished reconstruction
``reg``       ``Engine.l1_weights`` and ``Engine.regularize`` on the whole object
``serve``     ``Engine.submit`` / ``Engine.poll``: a burst of mixed requests at the serving loop

Inputs are drawn on the GPU from the seed alone: ellipsoid or smooth objects, focused probes with a
phase screen, jittered rasters, and measured intensities that are the FP64 forward model of a second
object with Poisson noise.  ``eps`` is the background (in photons) that a reconstruction adds to both
intensities: 3/8 for the least-squares loss (the variance-stabilising offset of a Poisson count) and
0.1 for the Poisson loss.  The loss is an FP64 sum of FP32 intensities; the programs here keep its
history in FP32.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_2012_12686_gb300.adorym import Engine
from paper_2012_12686_gb300.autograd import engine_for, multislice_loss

KDZ = 2.0 * math.pi * 10.0 / 0.248            # k dz: 10 nm slices at 0.248 nm (5 keV)
STEP = 0.248 * 10.0 / 10.0 ** 2               # lambda dz / dx^2 for 10 nm voxels
NF = (1e-3, 2e-3, 4e-3, 8e-3)                 # Fresnel numbers of the holography distances
LARGEST = 128 * 32 * 256 * 256                # pixel-slices of the largest listed minibatch


def _far(name, N, L, B, Ly, Lx, cols, step, origin, **more):
    c = dict(name=name, kind="grad", farfield=1, N=N, L=L, M=1, B=B, Lz=L, Ly=Ly, Lx=Lx, loss="poisson", tomo=0,
             theta=0.0, cols=cols, step=step, origin=origin, phase=1.5, photons=1e6,
             want="object probe positions")
    c.update(more)
    return c


def _near(name, N, L, B, n_dist, **more):
    c = dict(name=name, kind="grad", farfield=0, N=N, L=L, M=1, B=B, Lz=B * L, Ly=N, Lx=N, loss="lsq", tomo=0,
             theta=0.0, n_dist=n_dist, photons=1e4, want="object positions")
    c.update(more)
    return c


def listed():
    return [
        # the smallest call: 2-D ptychography of a small field, one batch of the whole scan
        _far("ptycho2d_32", 32, 1, 49, 64, 64, 7, 4, 4, loss="lsq", phase=0.25, photons=1e4, want="object probe"),
        # mixed-state 2-D ptychography: five incoherent modes, more positions than the chip has SMs
        _far("mixed_state_64", 64, 1, 256, 401, 390, 16, 21, 8, M=5, photons=1e5),
        # thick samples on a sparse set of slices, with the slice positions and the scan offset refined
        _far("sparse_slices_128", 128, 8, 100, 360, 360, 10, 24, 6, loss="lsq", gaps=1,
             want="object probe positions gaps offset"),
        # 3-D multislice ptychography, the ordinary minibatch
        _far("multislice_128", 128, 32, 128, 512, 512, 32, 12, 6),
        # ptychographic tomography: the positions of one tilt angle, as a torch training step
        _far("tomography_64", 64, 128, 64, 128, 128, 8, 16, -24, kind="autograd", loss="lsq", tomo=1,
             theta=math.pi / 6),
        # a probe beyond the shared-memory tile: ordinary and large batches
        _far("farfield_256", 256, 8, 64, 1024, 1024, 8, 96, 8),
        _far("farfield_256_large", 256, 32, 128, 1024, 1024, 16, 48, 6),
        # simulated data: intensities only, a whole scan row block at once
        _far("forward_128", 128, 32, 256, 512, 512, 32, 12, 6, kind="forward", want=""),
        # near-field holography, full field, four distances with unknown hologram shifts
        _near("holography_1024", 1024, 1, 8, 4),
        # thicker holography samples with the illumination and the distances refined
        _near("holography_512_distances", 512, 3, 2, 3, loss="poisson", want="object probe positions distances"),
        # the regularizer on the ordinary object: reweighted l1 from a snapshot, and total variation
        dict(name="regularizer_512", kind="reg", Lz=32, Ly=512, Lx=512),
        # a burst at the serving loop: 64..256 px tiles, 1..32 slices, 8..64 positions
        dict(name="serving_burst", kind="serve", requests=12, mix=7),
    ]


def draw(rng):
    """One more case of the listed ranges: every size drawn by its logarithm, object sides odd or even alike."""
    def log(lo, hi):
        return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))
    kind = rng.choice(["grad", "grad", "grad", "grad", "autograd", "forward", "near", "near", "reg", "serve"])
    if kind == "reg":
        return dict(kind="reg", Lz=log(1, 64), Ly=log(96, 700), Lx=log(96, 700))
    if kind == "serve":
        return dict(kind="serve", requests=log(4, 16), mix=rng.randrange(1 << 20))
    if kind == "near":
        N = rng.choice([128, 256, 512, 1024])
        n_dist = rng.randint(1, 4)
        L = log(1, 4)
        B = log(1, max(1, min(16, LARGEST // (8 * n_dist * L * N * N))))
        c = _near("", N, L, B, n_dist, loss=rng.choice(["lsq", "poisson"]),
                  want=rng.choice(["object positions", "object probe positions distances"]))
    else:
        N = rng.choice([32, 64, 128, 256])
        M = rng.choice([1, 1, 1, 2, 3, 5])
        tomo = 1 if kind == "autograd" and N < 256 and rng.random() < 0.7 else 0
        L = log(1, 32 if N == 256 else 128 if tomo else 64)
        B = log(4, max(4, min(300, LARGEST // (2 * M * L * N * N))))
        cols = rng.randint(max(2, math.isqrt(B) // 2), 2 * math.isqrt(B) + 2)
        step = log(max(2, N // 16), N // 2)
        span = N + step * (cols - 1), N + step * (-(-B // cols) - 1)
        # most scans lie inside the object, some reach past its edge
        side = min(1024, max(N, int(max(span) * rng.uniform(0.9, 1.3))))
        c = _far("", N, L, B, side + rng.randint(0, 9), side + rng.randint(0, 9), cols, step, 0, M=M, kind=kind,
                 loss=rng.choice(["lsq", "poisson"]), phase=rng.uniform(0.25, 3.0),
                 want=rng.choice(["object probe positions", "object probe", "object"]))
        c["origin"] = (min(c["Ly"], c["Lx"]) - max(span)) // 2
        if tomo:
            c.update(tomo=1, theta=math.pi * rng.randrange(180) / 180)
        elif kind == "grad" and L > 1 and N < 256 and rng.random() < 0.2:
            c.update(gaps=1, want="object probe positions gaps offset")
        if kind == "forward":
            c["want"] = ""
    del c["name"]
    return c


# ------------------------------------------------------------------------------------------ inputs
def _problem(c):
    p = {k: c[k] for k in ("N", "L", "M", "B", "Lz", "Ly", "Lx", "loss", "farfield", "tomo", "theta")}
    p.update(kdz=KDZ, lambda_dz_over_px2=STEP if c["farfield"] else 0.3, eps=0.375 if c["loss"] == "lsq" else 0.1,
             nf=[] if c["farfield"] else list(NF[:c["n_dist"]]), checkpoint_every=0)
    if c.get("gaps"):   # a sparse set of slices: one to three voxels between them
        p["gaps"] = [STEP * (1.0 + 0.25 * (5 * j % 9)) for j in range(c["L"] - 1)]
    return p


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _smooth(shape, sigma, g):
    """White noise through a periodic Gaussian of `sigma` px in the last two axes."""
    f = [torch.fft.fftfreq(n, device="cuda", dtype=torch.float64) for n in shape[-2:]]
    low = torch.exp(-2.0 * (math.pi * sigma) ** 2 * (f[0][:, None] ** 2 + f[1][None, :] ** 2))
    return torch.fft.ifft2(torch.fft.fft2(torch.randn(shape, generator=g, device="cuda", dtype=torch.float64)) * low).real


def _ellipsoids(shape, vmax, seed):
    """Sum of random axis-aligned ellipsoids, clipped to [0, vmax]."""
    Lz, Ly, Lx = shape
    r, vol = random.Random(int(seed)), torch.zeros(shape, device="cuda")
    for _ in range(64):
        at, semi = [], []
        for n, lo, hi in ((Lz, max(1.0, Lz / 16), max(2.0, Lz / 2)), (Ly, Ly / 64, Ly / 8), (Lx, Lx / 64, Lx / 8)):
            at.append(r.uniform(0, n))
            semi.append(r.uniform(lo, hi))
        a = r.uniform(0.2, 0.6) * vmax
        box = [(max(0, int(m - s)), min(n, int(m + s) + 1)) for m, s, n in zip(at, semi, shape)]
        d = [((torch.arange(lo, hi, device="cuda") - m) / s) ** 2 for (lo, hi), m, s in zip(box, at, semi)]
        vol[tuple(slice(lo, hi) for lo, hi in box)] += a * (d[0][:, None, None] + d[1][:, None] + d[2] <= 1.0)
    return vol.clamp_(0.0, vmax)


def _object(c, seed):
    """delta, beta, FP32 [Lz][Ly][Lx]."""
    shape = (c["Lz"], c["Ly"], c["Lx"])
    if not c["farfield"]:   # phase in [0, 2] rad through the sample, absorption of at most 5 %
        out = []
        for k, top in enumerate((2.0, 0.0513)):
            f = _smooth(shape, c["N"] / 64.0, _generator(seed + 17 * k))
            lo, hi = f.amin((1, 2), keepdim=True), f.amax((1, 2), keepdim=True)
            out.append(((f - lo) / (hi - lo) * (top / KDZ / c["L"])).float())
        return out
    top = c["phase"] / (KDZ * c["L"])   # up to `phase` rad through the sample
    if c["L"] == 1:
        g = _generator(seed)
        return [torch.rand(shape, generator=g, device="cuda") * top for _ in range(2)]
    d = _ellipsoids(shape, top, seed)
    return [d, d / 10.0]


def _probe(c, seed):
    """complex64 [M][N][N]: a focus with a phase screen, or the (uneven) illumination of a hologram."""
    N, M, g = c["N"], c["M"], _generator(seed)
    s = _smooth((M, N, N), N / 32.0, g)
    s = s / s.std(dim=(1, 2), keepdim=True)
    if not c["farfield"]:
        return torch.exp(0.05 * torch.complex(s, s.flip(-1))).to(torch.complex64)
    y = torch.arange(N, device="cuda", dtype=torch.float64) - (N - 1) / 2.0
    amp = torch.exp(-(y[:, None] ** 2 + y ** 2) / (2.0 * (N / 7.0) ** 2))
    p = amp * torch.exp(1j * s)
    p = p / p.abs().square().sum((1, 2), keepdim=True).sqrt()
    m = torch.arange(1, M + 1, device="cuda", dtype=torch.float64)
    return (p * (c["photons"] / m).sqrt()[:, None, None]).to(torch.complex64)


def _positions(c, seed):
    """FP32 [B][2] (y, x): a stretch of a jittered raster; near field [B][n_dist][2]: hologram shifts."""
    g, B = np.random.default_rng(int(seed)), c["B"]
    if not c["farfield"]:
        pos = g.integers(-5, 6, (B, c["n_dist"], 2)) + g.uniform(-0.45, 0.45, (B, c["n_dist"], 2))
    else:
        i = np.arange(B)
        pos = c["origin"] + c["step"] * np.stack([i // c["cols"], i % c["cols"]], 1) + g.uniform(-0.45, 0.45, (B, 2))
    return torch.from_numpy(pos.astype(np.float32)).cuda()


def _inputs(c, seed):
    """Everything a user has in hand: problem, object, probe, positions and measured intensities."""
    s = 1000003 * (int(seed) % 1000003)
    p = _problem(c)
    d, b = _object(c, s + 1)
    probe, pos = _probe(c, s + 2), _positions(c, s + 3)
    measured = None
    if c["kind"] != "forward":
        with torch.no_grad():
            I = torch.cat([i for i, _ in _chunks(p, *_object(c, s + 4), probe, pos)])
        scale = 1.0 if c["farfield"] else c["photons"]
        measured = (torch.poisson(I * scale, generator=_generator(s + 5)) / scale).float()
    return p, d, b, probe, pos, measured


class _Held:
    """The program's side of one minibatch: its arrays, and the object registered at the engine."""

    def __init__(self, **k):
        self.__dict__.update(k)

    def __del__(self):
        for eng, oid in getattr(self, "registered", ()):
            try:
                eng.unregister_object(oid)
            except Exception:
                pass


def _buffers(p, c):
    """Output arrays of a loss_grad call; `add` holds those that the call adds into."""
    want, f32 = c["want"].split(), dict(device="cuda", dtype=torch.float32)
    out = {"loss_out": torch.zeros((), device="cuda", dtype=torch.float64)}
    add = []
    if "object" in want:
        out["g_delta"], out["g_beta"] = (torch.zeros((p["Lz"], p["Ly"], p["Lx"]), **f32) for _ in range(2))
        add += [out["g_delta"], out["g_beta"]]
    if "probe" in want:
        out["g_probe"] = torch.zeros((p["M"], p["N"], p["N"]), device="cuda", dtype=torch.complex64)
        add.append(out["g_probe"])
    nd = (len(p["nf"]),) if not p["farfield"] else ()
    if "positions" in want:
        out["g_pos"] = torch.zeros((p["B"], *nd, 2), **f32)
    if "distances" in want:
        out["g_nf"] = torch.zeros((p["B"], *nd), **f32)
    if "gaps" in want:
        out["g_gaps"] = torch.zeros(p["L"] - 1, **f32)
    if "offset" in want:
        out["g_offset"] = torch.zeros(2, **f32)
    return out, add


def _mix(case):
    """The requests of a burst: tile, slices and batch drawn as the serving loop's clients send them."""
    r, got = random.Random(case["mix"]), []
    for _ in range(case["requests"]):
        N, L = r.choice([64, 128, 256]), r.choice([1, 8, 32])
        B = r.choice([8, 16, 32, 64])
        while 2 * B * L * N * N > LARGEST // 8:
            B //= 2
        got.append(_far("", N, L, B, 640, 640, 8, 40, 3, loss=r.choice(["lsq", "poisson"])))
    return got


def prepare(case, seed):
    dev = torch.device("cuda", torch.cuda.current_device())
    if case["kind"] == "serve":
        eng = Engine(dev.index)   # the server's own context: its slots and graphs live with it
        eng.serve_config(8)
        st = _Held(kind="serve", eng=eng, requests=[], registered=[])
        volumes = {}
        for k, c in enumerate(_mix(case)):
            p = _problem(c)
            s = 1000003 * (int(seed) % 1000003) + 7919 * k
            if p["L"] not in volumes:   # resident volumes, one per slice count
                d, b = _object(c, 1000003 * (int(seed) % 1000003) + p["L"])
                volumes[p["L"]] = (d, b, eng.register_object(d, b))
            d, b, oid = volumes[p["L"]]
            probe, pos = _probe(c, s + 2), _positions(c, s + 3)
            with torch.no_grad():
                I = torch.cat([i for i, _ in _chunks(p, *_object(c, s + 4), probe, pos)])
            measured = torch.poisson(I, generator=_generator(s + 5)).float()
            out, add = _buffers(p, c)
            st.requests.append((p, oid, probe, pos, measured, out, add))
        st.volumes = volumes
        st.history = torch.zeros(len(st.requests), device="cuda")
        torch.cuda.synchronize()
        return st
    eng = engine_for(dev)
    if case["kind"] == "reg":
        g = _generator(seed)
        shape = (case["Lz"], case["Ly"], case["Lx"])
        d = _ellipsoids(shape, 5e-6, seed) + 2e-8 * torch.randn(shape, generator=g, device="cuda")
        b = 0.1 * d.roll(1, -1) + 2e-9 * torch.randn(shape, generator=g, device="cuda")
        st = _Held(kind="reg", eng=eng, d=d, b=b, registered=[(eng, eng.register_object(d, b))])
        st.w, st.g = [torch.empty_like(d) for _ in range(2)], [torch.empty_like(d) for _ in range(2)]
        st.value = torch.zeros((), device="cuda", dtype=torch.float64)
        st.history = torch.zeros((), device="cuda")
        return st
    p, d, b, probe, pos, measured = _inputs(case, seed)
    st = _Held(kind=case["kind"], eng=eng, p=p, d=d, b=b, probe=probe, pos=pos, measured=measured, registered=[],
               ext=any(w in case["want"] for w in ("gaps", "offset", "distances")))
    st.history = torch.zeros((), device="cuda")
    if case["kind"] == "autograd":
        want = case["want"].split()
        st.d.requires_grad_(), st.b.requires_grad_()
        st.probe.requires_grad_("probe" in want)
        st.pos.requires_grad_("positions" in want)
        return st
    st.registered.append((eng, eng.register_object(d, b)))
    if case["kind"] == "forward":
        nd = () if p["farfield"] else (len(p["nf"]),)
        st.I = torch.empty((p["B"], *nd, p["N"], p["N"]), device="cuda")
    else:
        st.out, st.add = _buffers(p, case)
    return st


# -------------------------------------------------------------------------------------------- pass
def run(st):
    if st.kind == "grad":
        for t in st.add:
            t.zero_()
        call = st.eng.loss_grad_ext if st.ext else st.eng.loss_grad
        call(st.p, st.registered[0][1], st.probe, st.pos, st.measured, **st.out)
        st.history.copy_(st.out["loss_out"])
        return {"loss": st.history, **{k: v for k, v in st.out.items() if k != "loss_out"}}
    if st.kind == "autograd":
        leaves = {"delta": st.d, "beta": st.b, "probe": st.probe, "pos": st.pos}
        for t in leaves.values():
            t.grad = None
        loss = multislice_loss(st.d, st.b, st.probe, st.pos, st.measured, st.p)
        loss.backward()
        st.history.copy_(loss.detach())
        return {"loss": st.history, **{"g_" + k: t.grad for k, t in leaves.items() if t.grad is not None}}
    if st.kind == "forward":
        st.eng.forward(st.p, st.registered[0][1], st.probe, st.pos, st.I)
        return {"I": st.I}
    if st.kind == "reg":
        oid = st.registered[0][1]
        st.eng.l1_weights(oid, 1e-8, *st.w)
        for t in st.g:
            t.zero_()
        st.eng.regularize(oid, alpha_delta=1e-3, alpha_beta=1e-3, gamma_tv=1e-2, w_delta=st.w[0], w_beta=st.w[1],
                          loss_out=st.value, g_delta=st.g[0], g_beta=st.g[1])
        st.history.copy_(st.value)
        return {"value": st.history, "w_delta": st.w[0], "w_beta": st.w[1], "g_delta": st.g[0], "g_beta": st.g[1]}
    for *_, add in st.requests:
        for t in add:
            t.zero_()
    torch.cuda.current_stream().synchronize()   # the slots run on streams of their own
    tickets = [st.eng.submit(p, oid, probe, pos, measured, **out) for p, oid, probe, pos, measured, out, _ in st.requests]
    for t in tickets:
        st.eng.poll(t)
    st.history.copy_(torch.stack([r[5]["loss_out"] for r in st.requests]))
    return [{"loss": st.history}, *({k: v for k, v in r[5].items() if k != "loss_out"} for r in st.requests)]


# -------------------------------------------------------------------------------------------- work
def work(case):
    if case["kind"] == "reg":   # delta, beta in; weights out; gradients read and written
        n = case["Lz"] * case["Ly"] * case["Lx"]
        return {"bytes": 32.0 * n, "flops": 60.0 * n}
    if case["kind"] == "serve":
        w = [work(c) for c in _mix(case)]
        return {k: sum(x[k] for x in w) for k in ("bytes", "flops")}
    N, L, M, B, NN = case["N"], case["L"], case["M"], case["B"], case["N"] ** 2
    fft = 5.0 * NN * math.log2(NN)
    back = case["kind"] != "forward"
    if case["farfield"]:
        rows, cols = min(-(-B // case["cols"]), B), min(case["cols"], B)
        h = max(0, min(case["Ly"], case["origin"] + case["step"] * (rows - 1) + N) - max(0, case["origin"]))
        w = case["Lx"] if case["tomo"] else max(
            0, min(case["Lx"], case["origin"] + case["step"] * (cols - 1) + N) - max(0, case["origin"]))
        voxels, pixels, ffts = case["Lz"] * h * w, B * NN, B * M * L * (4 if back else 2)
    else:
        voxels, pixels = B * L * NN, B * case["n_dist"] * NN
        ffts = B * M * (2 * (L - 1) + 1 + case["n_dist"]) * (2 if back else 1)
    want = case["want"].split()
    moved = 8.0 * voxels + 4.0 * pixels + 8.0 * M * NN
    moved += 16.0 * voxels * ("object" in want) + 16.0 * M * NN * ("probe" in want)
    return {"bytes": moved, "flops": fft * ffts + (40.0 if back else 20.0) * B * M * L * NN}


# ------------------------------------------------------------------------------------------- exact
def _freq(N):
    return torch.fft.fftfreq(N, device="cuda", dtype=torch.float64)


def _ramp(d, N):
    """exp(-2 pi i d.nu) for shifts d [..., 2]."""
    f = _freq(N)
    return torch.exp(-2j * math.pi * (d[..., 0, None, None] * f[:, None] + d[..., 1, None, None] * f))


def _taps(p):
    """Bilinear taps of the rotation about y in the (z, x) plane: (rotated node, node, weight) lists."""
    Lz, Lx = p["Lz"], p["Lx"]
    z, x = torch.meshgrid(*(torch.arange(n, device="cuda", dtype=torch.float64) for n in (Lz, Lx)), indexing="ij")
    cz, cx, c, s = (Lz - 1) / 2.0, (Lx - 1) / 2.0, math.cos(p["theta"]), math.sin(p["theta"])
    x0, z0 = c * (x - cx) - s * (z - cz) + cx, s * (x - cx) + c * (z - cz) + cz
    node, got = torch.arange(Lz * Lx, device="cuda"), []
    for dz in (0, 1):
        for dx in (0, 1):
            zi, xi = z0.floor().long() + dz, x0.floor().long() + dx
            w = (1 - (z0 - zi).abs()) * (1 - (x0 - xi).abs())
            ok = ((zi >= 0) & (zi < Lz) & (xi >= 0) & (xi < Lx)).reshape(-1)
            got.append((node[ok], (zi * Lx + xi).reshape(-1)[ok], w.reshape(-1)[ok]))
    return [torch.cat(t) for t in zip(*got)]


def _rotate(p, vol, taps, back=False):
    dst, src, w = (taps[1], taps[0], taps[2]) if back else taps
    v = vol.double().permute(0, 2, 1).reshape(-1, p["Ly"])
    out = torch.zeros_like(v).index_add_(0, dst, w[:, None] * v[src])
    return out.reshape(p["Lz"], p["Lx"], p["Ly"]).permute(0, 2, 1)


def _model(p, d, b, probe, pos, corner, gaps, nf):
    """FP64 intensities of a few positions (or problems): d, b are their patches [n][L][N][N]."""
    N, L = p["N"], p["L"]
    f2 = _freq(N)[:, None] ** 2 + _freq(N) ** 2
    psi = probe[None]
    if p["farfield"]:
        psi = torch.fft.ifft2(torch.fft.fft2(psi) * _ramp(pos - corner, N)[:, None])
    for j in range(L):
        phi = psi * torch.exp(torch.complex(-p["kdz"] * b[:, j], p["kdz"] * d[:, j]))[:, None]
        if j < L - 1:
            step = p["lambda_dz_over_px2"] if gaps is None else gaps[j]
            psi = torch.fft.ifft2(torch.fft.fft2(phi) * torch.exp(1j * math.pi * step * f2))
    if p["farfield"]:
        out = torch.fft.ifft2(phi) * N
        return (out.real ** 2 + out.imag ** 2).sum(1)
    G = torch.exp(1j * math.pi * f2 / nf[..., None, None]) * _ramp(pos, N)          # [n][n_dist][N][N]
    out = torch.fft.ifft2(torch.fft.fft2(phi)[:, None] * G[:, :, None])
    return (out.real ** 2 + out.imag ** 2).sum(2)


def _chunks(p, d, b, probe, pos, measured=None, want=None):
    """The FP64 model a few positions at a time: yields (intensities, summed loss terms) with the
    gradients, where `want` is given, added into its tensors."""
    N, L, B, far = p["N"], p["L"], p["B"], p["farfield"]
    probe, pos = probe.detach().to(torch.complex128), pos.detach().double()
    d, b = d.detach(), b.detach()
    taps = _taps(p) if p["tomo"] else None
    if taps is not None:
        d, b = (_rotate(p, v, taps) for v in (d, b))
    span = max(1, int(6e9 // (16 * 8 * p["M"] * (L + 3 * len(p["nf"])) * N * N)))
    gaps = None if p.get("gaps") is None else torch.tensor(p["gaps"], device="cuda", dtype=torch.float64)
    for lo in range(0, B, span):
        at = pos[lo:lo + span]
        n = len(at)
        corner = torch.floor(at + 0.5) if far else None
        nf = None if far else torch.tensor(p["nf"], device="cuda", dtype=torch.float64).repeat(n, 1)
        if far:
            k = torch.arange(N, device="cuda")
            y, x = corner[:, 0, None].long() + k, corner[:, 1, None].long() + k
            inside = ((y >= 0) & (y < p["Ly"]))[:, :, None] & ((x >= 0) & (x < p["Lx"]))[:, None, :]
            flat = y.clamp(0, p["Ly"] - 1)[:, :, None] * p["Lx"] + x.clamp(0, p["Lx"] - 1)[:, None, :]
            cut = [(v.reshape(L, -1)[:, flat].double() * inside).transpose(0, 1).contiguous() for v in (d, b)]
        else:
            cut = [v[lo * L:(lo + n) * L].reshape(n, L, N, N).double() for v in (d, b)]
        leaves = [*cut, probe.clone(), at.clone(), *([gaps.clone()] if gaps is not None else []),
                  *([nf] if nf is not None else [])]
        if want is not None:
            for t in leaves:
                t.requires_grad_()
        g = leaves[4] if gaps is not None else None
        I = _model(p, leaves[0], leaves[1], leaves[2], leaves[3], corner, g, nf)
        if measured is None:
            yield I, None
            continue
        m, e = measured[lo:lo + n].double(), p["eps"]
        terms = ((I + e).sqrt() - (m + e).sqrt()) ** 2 if p["loss"] == "lsq" else I - m * torch.log(I + e)
        loss = terms.sum() / (measured.numel())
        got = torch.autograd.grad(loss, leaves)
        for key, v in zip(("g_delta", "g_beta"), got[:2]):
            if key not in want:
                continue
            if far:
                v = (v * inside[:, None]).transpose(0, 1).reshape(L, -1)
                want[key].reshape(L, -1).index_add_(1, flat.reshape(-1), v)
            else:
                want[key][lo * L:(lo + n) * L] += v.reshape(n * L, N, N)
        if "g_probe" in want:
            want["g_probe"] += got[2]
        if "g_pos" in want:
            want["g_pos"][lo:lo + n] = got[3]
        if "g_offset" in want:
            want["g_offset"] += got[3].sum(0)
        if "g_gaps" in want:
            want["g_gaps"] += got[4]
        if "g_nf" in want:
            want["g_nf"][lo:lo + n] = got[-1]
        yield I.detach(), loss.detach()
    if taps is not None and want is not None:
        for key in ("g_delta", "g_beta"):
            want[key] = _rotate(p, want[key], taps, back=True)


def _exact_grad(p, c, d, b, probe, pos, measured):
    out = {k: torch.zeros(v.shape, device="cuda", dtype=torch.complex128 if v.is_complex() else torch.float64)
           for k, v in _buffers(p, c)[0].items() if k != "loss_out"}
    loss = sum(v for _, v in _chunks(p, d, b, probe, pos, measured, out))
    return loss, {k: v.contiguous() for k, v in out.items()}


def exact(case, seed):
    if case["kind"] == "reg":
        st = prepare(case, seed)
        o = [st.d.double(), st.b.double()]
        for t in o:
            t.requires_grad_()
        w = [(t.abs().max() / (t.abs() + 1e-8)).detach() for t in o]
        value = sum(1e-3 * (u * t.abs()).sum() + 1e-2 * sum(t.diff(dim=a).abs().sum() for a in range(3))
                    for u, t in zip(w, o)) / o[0].numel()
        g = torch.autograd.grad(value, o)
        return {"value": value.detach(), "w_delta": w[0], "w_beta": w[1], "g_delta": g[0], "g_beta": g[1]}
    if case["kind"] == "serve":
        st = prepare(case, seed)
        losses, out = [], []
        for (p, _, probe, pos, measured, _, _), c in zip(st.requests, _mix(case)):
            d, b, _ = st.volumes[p["L"]]
            loss, g = _exact_grad(p, c, d, b, probe, pos, measured)
            losses.append(loss)
            out.append(g)
        return [{"loss": torch.stack(losses)}, *out]
    p, d, b, probe, pos, measured = _inputs(case, seed)
    if case["kind"] == "forward":
        with torch.no_grad():
            return {"I": torch.cat([i for i, _ in _chunks(p, d, b, probe, pos)])}
    loss, g = _exact_grad(p, case, d, b, probe, pos, measured)
    if case["kind"] == "autograd":
        g = {"g_" + k: g[n] for k, n in (("delta", "g_delta"), ("beta", "g_beta"), ("probe", "g_probe"), ("pos", "g_pos"))
             if n in g}
    return {"loss": loss, **g}
