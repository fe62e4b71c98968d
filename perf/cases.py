"""The workloads whose time is watched: what a program that uses libsdmd asks
of it, through the public entry points of the binding, from a 64 x 64 field to
HD video and 4-million-point windows.

Every case is one call sequence of a user's loop on a full window: a state
holds the handle(s), a pool of further snapshots on the device and the output
buffers, and run() takes the next snapshots of the pool. Sizes are those of
the synthetic configurations, the tests and the benchmark, plus the video
sizes of the paper's own timings (2560 x 1440 at m = 90, 1920 x 1080 grey at
m = 120).
"""
import math
import random

import numpy as np
import torch

from paper_1612_07875_gb300 import sdmd

ELEM = {"u8": 1, "f32": 4, "c64": 8}
SDMD_DTYPE = {"u8": sdmd.SDMD_U8, "f32": sdmd.SDMD_F32, "c64": sdmd.SDMD_C64}
TORCH_DTYPE = {"u8": torch.uint8, "f32": torch.float32, "c64": torch.complex64}
HD = 1920 * 1080 * 3


def listed():
    return [
        # the smallest call: one snapshot of a 64 x 64 FP32 field into a window of 32
        {"name": "push_f32_field", "kind": "push", "dtype": "f32", "n": 4096, "m": 32},
        # streaming DMD of that field: push, then the modes of the new window
        {"name": "dmd_f32_field", "kind": "dmd", "dtype": "f32", "n": 4096, "m": 32, "r": 10},
        # one HD video frame into its exact integer Gram
        {"name": "push_u8_hd", "kind": "push", "dtype": "u8", "n": HD, "m": 100},
        # a second of HD video through the pipelined DMD
        {"name": "step_u8_hd", "kind": "step", "n": HD, "m": 100, "r": 10, "depth": 6, "frames": 24, "host": False},
        # background subtraction of one 2560 x 1440 frame
        {"name": "separate_u8_2k", "kind": "separate", "n": 2560 * 1440, "m": 90, "r": 10},
        # streaming SVD of a 1920 x 1080 grey FP32 stream: singular values, V and the POD modes
        {"name": "svd_f32_grey", "kind": "svd", "dtype": "f32", "n": 1920 * 1080, "m": 120, "r": 10},
        # a whole window at once (the first step of the stream), longer than one tensor-core tile, odd n
        {"name": "load_u8_odd", "kind": "batch", "dtype": "u8", "n": 1000003, "m": 200, "k": 200},
        # a video stream that fell 8 frames behind
        {"name": "catchup_u8_hd", "kind": "batch", "dtype": "u8", "n": HD, "m": 100, "k": 8},
        # the same for a long FP32 window with the split-precision option on
        {"name": "catchup_f32_long", "kind": "batch", "dtype": "f32", "n": 1 << 22, "m": 256, "k": 8},
        # DMD of a dense complex 1024 x 1024 field
        {"name": "dmd_c64_field", "kind": "dmd", "dtype": "c64", "n": 1 << 20, "m": 64, "r": 10},
        # the same field by its 1 % of Fourier coefficients: push, modes, compressed modes
        {"name": "fourier_modes", "kind": "fourier", "side": 1024, "m": 64, "r": 10},
        # 64 served streams of mixed size and type: one frame each, then every stream's eigenvalues
        {"name": "serve_64", "kind": "serve", "streams": 64, "mix": 5, "lo": 16.0, "hi": 22.0, "r": 10},
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    kind = rng.choice(["push", "push", "dmd", "step", "separate", "svd", "batch", "batch", "fourier", "serve"])
    m = _logint(rng, 8, 256)
    if kind == "push":
        dtype = rng.choice(["u8", "f32", "c64"])
        n = _logint(rng, 1 << 12, min(6 << 20, int(4.2e9) // (m * ELEM[dtype])))
        return {"kind": kind, "dtype": dtype, "n": n, "m": m}
    if kind == "dmd":
        dtype = rng.choice(["u8", "f32", "c64"])
        m = _logint(rng, 12, 64 if dtype == "c64" else 128)
        n = _logint(rng, 1 << 12, 1 << 21)
        return {"kind": kind, "dtype": dtype, "n": n, "m": m, "r": rng.randint(2, min(16, m - 2))}
    if kind == "step":
        m = _logint(rng, 16, 120)
        host = rng.random() < 0.3
        return {"kind": kind, "n": _logint(rng, 1 << 14, (1 << 20) if host else (5 << 20)), "m": m,
                "r": rng.randint(4, 12), "depth": rng.randint(2, 8), "frames": 24, "host": host}
    if kind == "separate":
        return {"kind": kind, "n": _logint(rng, 1 << 14, 6 << 20), "m": _logint(rng, 20, 120), "r": rng.randint(4, 16)}
    if kind == "svd":
        dtype = rng.choice(["u8", "f32"])
        return {"kind": kind, "dtype": dtype, "n": _logint(rng, 1 << 14, 2 << 20), "m": _logint(rng, 20, 128),
                "r": rng.randint(4, 16)}
    if kind == "batch":
        dtype = rng.choice(["u8", "f32"])
        n = _logint(rng, 1 << 14, min(6 << 20, int(4.2e9) // (m * ELEM[dtype])))
        return {"kind": kind, "dtype": dtype, "n": n, "m": m, "k": min(m, _logint(rng, 2, 64))}
    if kind == "fourier":
        return {"kind": kind, "side": rng.randint(96, 1024), "m": _logint(rng, 16, 64), "r": rng.randint(4, 10)}
    return {"kind": "serve", "streams": rng.randint(4, 64), "mix": rng.randint(0, 1 << 20), "lo": 16.0,
            "hi": round(rng.uniform(17.0, 21.5), 2), "r": rng.randint(4, 10)}


# ------------------------------------------------------------------ inputs --

def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _smooth(n, g, width):
    """Noise with about `width` neighbours alike, zero mean and unit RMS."""
    coarse = torch.randn((1, 1, max(4, n // width)), generator=g, device="cuda", dtype=torch.float64)
    f = torch.nn.functional.interpolate(coarse, size=n, mode="linear")[0, 0]
    f = f - f.mean()
    return (f / f.square().mean().sqrt()).float()


def _pool(count, n, dtype, contiguous):
    """`count` rows of n elements: back to back, or each on a 256-byte boundary as separate allocations are."""
    ld = n if contiguous else -(-n // 256) * 256
    return torch.zeros((count, ld), dtype=TORCH_DTYPE[dtype], device="cuda")[:, :n]


def _video(out, seed):
    """Frames of whole numbers (uint8, or FP32 as grey video is kept): textured background in 0..200, three moving
    rectangles, +-4 pixel noise, clamped to 0..255."""
    count, n = out.shape
    g = _generator(seed)
    host = random.Random(seed)
    bg = _smooth(n, g, 97)
    bg = ((bg - bg.min()) / (bg.max() - bg.min()) * 200).round()
    w = max(1, math.isqrt(n))
    h = -(-n // w)
    i = torch.arange(n, device="cuda", dtype=torch.int32)
    ix, iy = i % w, i // w
    rects = []
    for _ in range(3):
        rw, rh = host.randint(max(1, w // 24), max(1, w // 6)), host.randint(max(1, h // 24), max(1, h // 6))
        rects.append((rw, rh, host.randrange(w), host.randrange(h), host.choice([-7, -5, -3, 2, 4, 6]),
                      host.randint(-5, 5), float(host.randint(0, 255))))
    for t in range(count):
        f = bg
        for rw, rh, x0, y0, vx, vy, colour in rects:
            inside = ((ix - (x0 + vx * t)) % w < rw) & ((iy - (y0 + vy * t)) % h < rh)
            f = torch.where(inside, colour, f)
        f = f + torch.randint(-4, 5, (n,), generator=g, device="cuda")
        out[t] = f.clamp_(0, 255).to(out.dtype)


def _planted(out, seed, restart):
    """FP32 or complex64 snapshots: planted modes with |lambda| in [0.95, 1] and noise of variance 1e-3. The
    dynamics start again every `restart` snapshots, so a long pool does not fade."""
    count, n = out.shape
    g = _generator(seed)
    host = np.random.default_rng(int(seed))
    t = np.arange(count) % max(2, restart)
    if out.dtype == torch.complex64:
        lam = np.linspace(0.955, 0.999, 18) * np.exp(1j * host.permutation(np.linspace(-3.0, 3.0, 18)))
        a = host.uniform(0.5, 1.5, 18) * lam[None, :] ** t[:, None]
        a = torch.from_numpy(a.astype(np.complex64)).cuda()
        f = torch.stack([torch.complex(_smooth(n, g, 33), _smooth(n, g, 33)) for _ in range(18)])
    else:
        lam = host.uniform(0.95, 1.0, 2) * np.exp(1j * host.uniform(0.15, np.pi - 0.15, 2))
        z = host.uniform(0.5, 1.5, 2) * lam[None, :] ** t[:, None]
        real = host.uniform(0.5, 1.5) * host.uniform(0.95, 1.0) ** t
        a = np.stack([z[:, 0].real, z[:, 0].imag, z[:, 1].real, z[:, 1].imag, real], axis=1)
        a = torch.from_numpy(a.astype(np.float32)).cuda()
        f = torch.stack([_smooth(n, g, 33) for _ in range(5)])
    for j in range(count):
        x = (a[j][:, None] * f).sum(0)
        noise = torch.randn(n, generator=g, device="cuda") if x.dtype == torch.float32 else torch.complex(
            torch.randn(n, generator=g, device="cuda"), torch.randn(n, generator=g, device="cuda"))
        out[j] = x + math.sqrt(1e-3) * noise


def _snapshots(case, seed, count, contiguous=False):
    dtype = case.get("dtype", "u8")
    out = _pool(count, case["n"], dtype, contiguous)
    if dtype == "u8" or case["kind"] == "svd":
        _video(out, seed)
    else:
        _planted(out, seed, 2 * case["m"])
    return out


def _fourier(case, seed, count):
    """`count` snapshots of sorted coefficient indices and values: ~1 % of side^2 drawn with P(k) ~ |k|^-5/3, a
    tenth of the support exchanged per snapshot, every coefficient rotating at its own frequency with slow decay."""
    side = case["side"]
    n, nnz = side * side, _nnz(case)
    g = _generator(seed)
    kf = torch.fft.fftfreq(side, 1.0 / side, device="cuda", dtype=torch.float64)
    w = (kf[None, :].square() + kf[:, None].square()).reshape(-1).clamp(min=0.25).pow(-5.0 / 6.0)
    churn = nnz // 10
    pool = torch.multinomial(w, min(n, nnz + 4 * churn + 16), generator=g)
    amp = torch.complex(torch.randn(n, generator=g, device="cuda", dtype=torch.float64),
                        torch.randn(n, generator=g, device="cuda", dtype=torch.float64)) * w.sqrt()
    omega = (torch.rand(n, generator=g, device="cuda", dtype=torch.float64) * 2 - 1) * math.pi
    rho = 0.995 + 0.005 * torch.rand(n, generator=g, device="cuda", dtype=torch.float64)
    idx, val = [], []
    for t in range(count):
        keep = torch.randperm(nnz, generator=g, device="cuda")[: nnz - churn]
        add = nnz + torch.randperm(pool.numel() - nnz, generator=g, device="cuda")[:churn]
        k = torch.sort(pool[torch.cat([keep, add])])[0]
        idx.append(k.to(torch.int32))
        val.append((amp[k] * rho[k] ** t * torch.polar(torch.ones_like(omega[k]), omega[k] * t)).to(torch.complex64))
    return idx, val


def _nnz(case):
    return max(32, case["side"] * case["side"] // 100)


def _mix(case):
    """Sizes of the served streams: element type, n log-uniform, window."""
    host = random.Random(case["mix"])
    specs = []
    for _ in range(case["streams"]):
        specs.append((host.choice(["u8", "f32"]), int(round(2 ** host.uniform(case["lo"], case["hi"]))),
                      host.choice([16, 32, 64, 128, 256])))
    return specs


def _mix_pools(case, seed):
    """One long signal per element type (travelling waves and noise); a stream's frames are shifted windows of it."""
    length = (1 << 22) + 1024 * 4096
    g = _generator(seed)
    host = random.Random(seed)
    i = torch.arange(length, device="cuda", dtype=torch.float64)
    s = torch.zeros(length, device="cuda", dtype=torch.float64)
    for _ in range(4):
        s += host.uniform(0.5, 1.5) * torch.sin(i * (2 * math.pi / host.uniform(9e3, 9e4)) + host.uniform(0, 6.28))
    noise = torch.randn(length, generator=g, device="cuda")
    f32 = (s + 0.05 * noise).float()
    u8 = (128 + 16 * s + 2 * noise).round().clamp(0, 255).to(torch.uint8)
    return {"f32": f32, "u8": u8}


# ------------------------------------------------------------------- state --

class Handle:
    """A libsdmd handle that is destroyed with the state that holds it."""

    def __init__(self, h):
        self.h = h

    def __del__(self):
        if self.h is not None:
            sdmd.sdmd_destroy(self.h)
            self.h = None


def prepare(case, seed):
    kind = case["kind"]
    s = {"case": dict(case), "next": 0}
    if kind == "serve":
        return _prepare_serve(case, seed, s)
    if kind == "fourier":
        return _prepare_fourier(case, seed, s)
    n, m, dtype = case["n"], case["m"], case.get("dtype", "u8")
    if kind == "batch":
        blocks = 2 if case["k"] > 32 else 4
        frames = _snapshots(case, seed, blocks * case["k"], contiguous=True)
        s["blocks"] = [frames[b * case["k"]:(b + 1) * case["k"]] for b in range(blocks)]
        s["frames"] = frames
        fill = [frames[j % frames.shape[0]] for j in range(m)]
    else:
        # a window that is decomposed never holds a snapshot twice
        spare = {"push": 32, "step": case.get("frames", 0) + m}.get(kind, m + 32)
        if kind == "push":
            frames = _snapshots(case, seed, spare)
            fill = [frames[j % spare] for j in range(m)]
            rows = [frames[j] for j in range(spare)]
        else:
            frames = _snapshots(case, seed, m + spare)
            rows = [frames[j] for j in range(m + spare)]
            fill = rows[:m]
            rows = rows[m:] + fill
        s["rows"] = rows
        if case.get("host"):
            s["rows"] = [x.cpu().pin_memory() for x in rows]
    h = sdmd.sdmd_create_ex(n, m, SDMD_DTYPE[dtype], case.get("depth", 1))
    s["handle"], s["h"] = Handle(h), h
    if kind == "batch" and dtype == "f32":
        sdmd.sdmd_set_option(h, sdmd.SDMD_OPT_F32_BF16X3, 1)
    if case.get("host"):
        sdmd.sdmd_set_option(h, sdmd.SDMD_OPT_HOST_EARLY_READ, 1)
    for x in fill:
        sdmd.sdmd_push(h, x)
    dev = dict(device="cuda")
    r = case.get("r", 1)
    if kind in ("push", "batch"):
        gdt = {"u8": torch.int64, "f32": torch.float64, "c64": torch.complex128}[dtype]
        s["G"] = torch.zeros((m, m), dtype=gdt, **dev)
    if kind == "dmd":
        s["phi"] = torch.zeros((r, n), dtype=torch.complex64, **dev)
        s["lam"] = torch.zeros(r, dtype=torch.complex128, **dev)
    if kind == "step":
        s["phi"] = torch.zeros((case["depth"], r, n), dtype=torch.complex64, **dev)
        s["lam"] = torch.zeros((case["frames"], r), dtype=torch.complex128, **dev)
        s["rank"] = torch.zeros(case["frames"], dtype=torch.int32, **dev)
    if kind == "separate":
        s["fg"] = torch.zeros(-(-n // 4) * 4, dtype=torch.float32, **dev)[:n]
    if kind == "svd":
        s["sigma"] = torch.zeros(r, dtype=torch.float64, **dev)
        s["V"] = torch.zeros((r, m - 1), dtype=torch.float64, **dev)
        s["U"] = torch.zeros((r, n), dtype=torch.float32, **dev)
    if kind in ("dmd", "separate", "svd"):
        s["rank"] = torch.zeros(1, dtype=torch.int32, **dev)
    torch.cuda.synchronize()
    return s


def _prepare_fourier(case, seed, s):
    side, m, r = case["side"], case["m"], case["r"]
    idx, val = _fourier(case, seed, m + 64)
    h = sdmd.sdmd_create_sparse(side * side, m, _nnz(case))
    s["handle"], s["h"] = Handle(h), h
    for t in range(m):
        sdmd.sdmd_push_sparse(h, idx[t].numel(), idx[t], val[t])
    s["rows"] = list(zip(idx[m:] + idx[:m], val[m:] + val[:m]))
    s["cap"] = min(side * side, 4 * _nnz(case))
    s["lam"] = torch.zeros(r, dtype=torch.complex128, device="cuda")
    s["rank"] = torch.zeros(1, dtype=torch.int32, device="cuda")
    s["idx"] = torch.zeros(s["cap"], dtype=torch.int32, device="cuda")
    s["phi"] = torch.zeros((r, s["cap"]), dtype=torch.complex64, device="cuda")
    torch.cuda.synchronize()
    return s


def _prepare_serve(case, seed, s):
    specs, pools = _mix(case), _mix_pools(case, seed)
    s["pools"], s["specs"] = pools, specs
    s["handles"] = [Handle(sdmd.sdmd_create(n, m, SDMD_DTYPE[d])) for d, n, m in specs]
    s["hs"] = [x.h for x in s["handles"]]
    for j in range(max(m for _, _, m in specs)):
        due = [i for i, (_, _, m) in enumerate(specs) if j < m]
        sdmd.sdmd_push_many([s["hs"][i] for i in due], [_served_frame(s, i, j) for i in due])
    s["next"] = max(m for _, _, m in specs)
    s["rs"] = [min(case["r"], m - 1) for _, _, m in specs]
    s["lam"] = torch.zeros((case["streams"], case["r"]), dtype=torch.complex128, device="cuda")
    s["lams"] = [s["lam"][i] for i in range(case["streams"])]
    s["rank"] = torch.zeros(case["streams"], dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    return s


def _served_frame(s, i, j):
    d, n, _ = s["specs"][i]
    at = ((j * 4096 + i * 128) % (s["pools"][d].numel() - n)) // 16 * 16
    return s["pools"][d][at:at + n]


# --------------------------------------------------------------------- run --

def run(s):
    case, st = s["case"], torch.cuda.current_stream()
    kind, at = case["kind"], s["next"]
    if kind == "serve":
        frames = [_served_frame(s, i, at) for i in range(case["streams"])]
        sdmd.sdmd_push_many(s["hs"], frames, st)
        sdmd.sdmd_modes_many(s["hs"], s["rs"], s["lams"], s["rank"], st)
        s["next"] = at + 1
        return {"lam": s["lam"], "rank": s["rank"]}
    h = s["h"]
    if kind == "batch":
        x = s["blocks"][at]
        s["next"] = (at + 1) % len(s["blocks"])
        sdmd.sdmd_push_batch(h, case["k"], x, case["n"], st)
        sdmd.sdmd_gram(h, s["G"], st)
        return {"G": s["G"]}
    rows = s["rows"]
    if kind == "step":
        depth = case["depth"]
        for j in range(case["frames"]):
            sdmd.sdmd_step(h, rows[at], case["r"], s["phi"][j % depth], s["lam"][j], s["rank"][j:], st)
            at = (at + 1) % len(rows)
        sdmd.sdmd_sync(h, st)
        s["next"] = at
        return {"phi": s["phi"], "lam": s["lam"], "rank": s["rank"]}
    x = rows[at]
    s["next"] = (at + 1) % len(rows)
    if kind == "fourier":
        sdmd.sdmd_push_sparse(h, x[0].numel(), x[0], x[1], st)
        sdmd.sdmd_modes(h, case["r"], None, s["lam"], s["rank"], st)
        count = sdmd.sdmd_fourier_modes(h, case["r"], s["idx"], s["phi"], s["cap"], st)
        return {"lam": s["lam"], "rank": s["rank"], "count": count, "idx": s["idx"], "phi": s["phi"]}
    sdmd.sdmd_push(h, x, st)
    if kind == "push":
        sdmd.sdmd_gram(h, s["G"], st)
        return {"G": s["G"]}
    if kind == "dmd":
        sdmd.sdmd_modes(h, case["r"], s["phi"], s["lam"], s["rank"], st)
        return {"phi": s["phi"], "lam": s["lam"], "rank": s["rank"]}
    sdmd.sdmd_modes(h, case["r"], None, None, s["rank"], st)
    if kind == "separate":
        sdmd.sdmd_reconstruct(h, case["m"] - 1, sdmd.SDMD_RECON_FOREGROUND, s["fg"], st)
        return {"foreground": s["fg"], "rank": s["rank"]}
    sdmd.sdmd_svd(h, case["r"], s["sigma"], s["V"], st)
    sdmd.sdmd_pod_modes(h, case["r"], s["U"], st)
    return {"sigma": s["sigma"], "V": s["V"], "U": s["U"], "rank": s["rank"]}


def work(case):
    """Snapshots of the window and new ones read once, new ones kept, results written; multiply-adds of the
    inner products and of the modes as two operations (eight for complex ones)."""
    kind = case["kind"]
    if kind == "serve":
        specs = _mix(case)
        return {"bytes": sum((m + 1) * n * ELEM[d] for d, n, m in specs), "flops": sum(2 * m * n for _, n, m in specs)}
    m, r = case["m"], case.get("r", 0)
    if kind == "fourier":
        nnz = _nnz(case)
        return {"bytes": (m + 1) * nnz * 12 + 2 * nnz * (4 + 8 * r), "flops": 8 * m * nnz * (1 + r)}
    n, e = case["n"], ELEM[case.get("dtype", "u8")]
    mul = 8 if e == 8 else 2
    if kind == "batch":
        k = case["k"]
        return {"bytes": (m + k) * n * e + 8 * m * m, "flops": 2 * n * (m * k - k * (k - 1) // 2)}
    if kind == "push":
        return {"bytes": (m + 1) * n * e + m * m * (16 if e == 8 else 8), "flops": mul * m * n}
    modes = {"dmd": 8 * r, "step": 8 * r, "separate": 4, "svd": 4 * r}[kind]
    columns = {"dmd": 4 * r if e < 8 else 8 * r, "step": 4 * r, "separate": 4, "svd": 2 * r}[kind]
    passes = case.get("frames", 1)
    return {"bytes": passes * ((m + 1) * n * e + n * modes), "flops": passes * n * (mul * m + columns * (m - 1))}


# ------------------------------------------------------------------- exact --

def _window(case, seed):
    """The snapshots that the first run() leaves in the window, oldest first (rows)."""
    m = case["m"]
    if case["kind"] == "batch":
        k = case["k"]
        blocks = 2 if k > 32 else 4
        frames = _snapshots(case, seed, blocks * k, contiguous=True)
        order = [j % (blocks * k) for j in range(m)] + list(range(k))
    elif case["kind"] == "push":
        frames = _snapshots(case, seed, 32)
        order = [j % 32 for j in range(m)] + [0]
    else:
        frames = _snapshots(case, seed, 2 * m + 32)
        order = list(range(m + 1))
    return frames[torch.tensor(order[-m:], device="cuda")]


def _gram64(x):
    """x x^H (rows are snapshots) in 64 bits, conj of the first factor."""
    wide = torch.complex128 if x.is_complex() else torch.float64
    g = torch.zeros((x.shape[0], x.shape[0]), dtype=wide, device="cuda")
    step = 1 << 19
    for p in range(0, x.shape[1], step):
        b = x[:, p:p + step].to(wide)
        g += b.conj() @ b.T
    return g


def _dmd64(g, r):
    """Exact DMD of a window from its Gram: sigma, V, V Sigma^-1, eigenvalues, W, the kept rank."""
    p = g.shape[0] - 1
    lam, v = np.linalg.eigh(g[:p, :p])
    lam, v = lam[::-1], v[:, ::-1]
    keep = min(r, int((lam > lam[0] * 64.0 * p * 2.0 ** -52).sum()))
    sigma = np.sqrt(lam[:keep])
    vsi = v[:, :keep] / sigma
    ev, w = np.linalg.eig(vsi.conj().T @ g[:p, 1:] @ vsi)
    order = np.argsort(-np.abs(ev), kind="stable")
    return sigma, v[:, :keep], vsi, ev[order], w[:, order], keep


def exact(case, seed):
    kind = case["kind"]
    if kind in ("serve", "step") or case.get("dtype") == "u8" and kind in ("push", "batch"):
        return None                  # whole numbers, or eigenvalues and modes of real windows (below)
    if kind == "fourier":
        m, n = case["m"], case["side"] ** 2
        idx, val = _fourier(case, seed, m + 64)
        x = torch.zeros((m, n), dtype=torch.complex64, device="cuda")
        for j in range(m):
            x[j, idx[j + 1].long()] = val[j + 1]
        lam = _dmd64(_gram64(x).cpu().numpy(), case["r"])[3]
        out = np.zeros(case["r"], np.complex128)
        out[:lam.size] = lam
        return {"lam": out, "rank": None, "count": None, "idx": None, "phi": None}    # a mode's phase is free
    if kind == "dmd" and case["dtype"] != "c64":
        return None                  # a mode's phase is free, and so is the order within a conjugate pair
    x = _window(case, seed)
    if kind in ("push", "batch"):
        return {"G": _gram64(x)}
    g = _gram64(x).cpu().numpy()
    sigma, v, vsi, lam, w, keep = _dmd64(g, case["r"])
    if kind == "dmd":
        out = np.zeros(case["r"], np.complex128)
        out[:keep] = lam
        return {"lam": out, "phi": None, "rank": None}
    if kind == "svd":
        out = np.zeros(case["r"])
        out[:keep] = sigma
        return {"sigma": out, "V": None, "U": None, "rank": None}      # the sign of a vector is free
    b = np.linalg.solve(w * lam, sigma * v[0].conj())
    i = int(np.argmin(np.abs(np.log(lam.astype(complex)))))
    u = (vsi @ w[:, i] * (b[i] * lam[i] ** (case["m"] - 1))).real
    u = torch.from_numpy(np.ascontiguousarray(u)).cuda()
    back = torch.zeros(case["n"], dtype=torch.float64, device="cuda")
    for j in range(case["m"] - 1):
        back += u[j] * x[j + 1].double()
    return {"foreground": x[-1].double() - back, "rank": None}
