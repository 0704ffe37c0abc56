"""Performance cases of the imaging library: what a user's program calls, over the sizes it meets.

A case describes one station (layout, channels, polarisations, grid, gridding function), one
block of voltages (samples, sample format) and the entry point that images it:

  "image"  Plan.image on device voltages, launches issued call by call
  "graph"  the same as one recorded CUDA graph (EPIC_GRAPH), as a loop over fixed buffers does
  "two"    one integration of two blocks: Plan.image, then Plan.image(accumulate=True)
  "host"   Plan.image_host_ptr from pinned host buffers (copies included)
  "server" a streaming Server that images blocks of three station types submitted together

Voltages are receiver noise plus three random sources, quantised to 4 + 4 or 8 + 8 bits.
"""
import math

import numpy as np
import torch

import paper_2609_03027_gb300 as epic

C0 = 299_792_458.0

#: One station type of the streaming mix: the other fields come from its case.
MIX = ("mix64", "mix256", "mix1024")

BASE = {"layout": "disc", "n_ant": 256, "size": 38.0, "size_y": 38.0, "pols": 2, "chans": 64, "f0": 50e6, "df": 25e3,
        "grid": 128, "K": 5, "sigma": 1.0, "f_ref": 0.0, "table": 0, "T": 64, "bits": 4, "sub": 0, "mix": False,
        "path": "auto", "call": "image", "blocks": 1}


def _case(**kw):
    return dict(BASE, **kw)


def _lwa(**kw):
    """LWA-like station: 256 dual-pol dipoles in a 100 m x 110 m ellipse, 25 kHz channels around 56 MHz."""
    return _case(**dict({"size": 100.0, "size_y": 110.0, "chans": 128, "f0": 54.4125e6, "K": 5, "T": 1000}, **kw))


def _skalow(**kw):
    """SKA-Low-like station: 256 elements in 38 m, 781.25 kHz channels over 50-350 MHz, kernel width scaled with frequency."""
    return _case(**dict({"chans": 384, "f0": 50.390625e6, "df": 781.25e3, "K": 7, "sigma": 1.5, "f_ref": 350e6, "T": 512}, **kw))


def _dense(side, **kw):
    """A side x side lattice at half a wavelength of 150 MHz, elements displaced by up to 5 %."""
    pitch = 0.5 * C0 / 150e6
    return _case(**dict({"layout": "lattice", "n_ant": side * side, "size": pitch, "size_y": pitch, "chans": 64,
                         "f0": 150.390625e6, "df": 781.25e3, "K": 3, "sigma": 0.5, "T": 256}, **kw))


def listed():
    return [
        # the smallest station: 64 single-pol elements, four channels, 32 x 32 images
        _case(name="tiny_station", n_ant=64, size=20.0, size_y=20.0, pols=1, chans=4, f0=C0 / 2.0, df=0.0, grid=32, K=3,
              sigma=0.5, T=256),
        # real-time imaging: a short block replayed as a graph, where launches and latency count
        _lwa(name="lwa_burst_graph", T=32, call="graph"),
        # an LWA station's 40 ms accumulation
        _lwa(name="lwa_station"),
        # an SKA-Low station's whole band, the largest everyday block
        _skalow(name="skalow_station"),
        # the same block from pinned host memory to host images
        _skalow(name="skalow_host", call="host"),
        # calibration inside the imager: 2 x 2 mixing per element, an integration of two blocks
        _skalow(name="skalow_mixed_two", T=96, mix=True, call="two"),
        # a dense large-N array
        _dense(64, name="dense_lattice", grid=256),
        # transient search: 8 + 8-bit samples, an image set every four samples
        _lwa(name="lwa_cadence", T=128, bits=8, sub=4),
        # odd sizes: a station with dead elements, one polarisation, a tabulated complex kernel
        _case(name="ragged_table", n_ant=253, size=70.0, size_y=61.0, pols=1, chans=109, f0=38.0e6, df=97e3, grid=64, K=4, table=8,
              T=333),
        # images in full FP32 precision
        _lwa(name="lwa_fp32", path="plain"),
        # a 20,000-element station on a 512 x 512 grid, one coarse channel
        _case(name="large_grid", n_ant=20000, size=240.0, size_y=240.0, chans=1, f0=159.390625e6, grid=512, K=2, sigma=0.5,
              T=1000),
        # several stations served at once
        _case(name="served_mix", call="server", blocks=9, chans=64, T=256),
    ]


def _pick(rng, lo, hi):
    """A whole number of lo..hi, spread over its logarithm."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


#: Pixel updates of the largest drawn cases by path (below the largest listed ones).
MOST_TENSOR, MOST_PLAIN, MOST_SETS = 4.0e9, 2.5e9, 1.0e9


def draw(rng):
    kind = rng.choice(["station", "station", "band", "lattice", "fp32", "cadence", "short"])
    grid = rng.choice([32, 64, 128, 128, 256] if kind != "fp32" else [32, 64, 128, 256, 512])
    c = _case(grid=grid, pols=rng.choice([1, 2, 2, 2]), K=rng.choice([2, 3, 4, 5, 7]), sigma=round(rng.uniform(0.5, 1.5), 3),
              chans=_pick(rng, 4, 400), T=_pick(rng, 24, 1200), bits=rng.choice([4, 4, 4, 8]))
    if kind == "lattice":
        side = rng.randint(8, min(64, grid // 4))
        c.update(_dense(side, grid=grid, pols=c["pols"], K=rng.choice([2, 3, 4]), chans=_pick(rng, 4, 96), T=c["T"], bits=c["bits"]))
        fill = 0.0
    else:
        f = rng.uniform(40e6, 300e6)
        # longest axis in grid cells at the highest frequency; the largest stations span a third of a 256-wide grid
        fill = rng.uniform(0.2, 0.45 if grid <= 128 else 0.3)
        c.update(n_ant=_pick(rng, 24, 600), f0=f, df=rng.choice([25e3, 97e3, 195e3]))
        if kind == "band":
            c.update(f0=50e6, df=300e6 / c["chans"], K=7, sigma=1.5, f_ref=350e6)
        top = c["f0"] + c["df"] * (c["chans"] - 1)
        cells = fill * grid * C0 / top / 2.0
        c.update(size=round(cells, 3), size_y=round(cells * rng.uniform(0.8, 1.0), 3))
    if kind == "fp32":
        c["path"] = "plain"
    if kind == "station" and rng.random() < 0.3:
        c.update(table=rng.choice([4, 8, 16]), K=min(c["K"], 5))
    elif c["pols"] == 2 and rng.random() < 0.25:
        c["mix"] = True
    if kind == "cadence":
        c.update(sub=rng.choice([4, 5, 8, 16, 50]))
    if kind == "short":
        c.update(T=_pick(rng, 16, 64), call="graph")
    else:
        c["call"] = rng.choice(["image", "image", "graph", "host" if kind != "cadence" else "image", "two" if kind != "cadence" else "graph"])
    most = MOST_PLAIN if kind == "fp32" or c["table"] else MOST_SETS if kind == "cadence" else MOST_TENSOR
    per = grid * grid * c["pols"] * (2 if c["call"] == "two" else 1)
    while c["chans"] * c["T"] * per > most and (c["chans"] > 4 or c["T"] > 16):
        if c["chans"] > 4 and rng.random() < 0.5:
            c["chans"] = max(4, c["chans"] * 3 // 4)
        else:
            c["T"] = max(16, c["T"] * 3 // 4)
    if c["sub"]:  # whole image sets, 2 GB of them at most
        c["T"] = max(c["sub"], c["T"] - c["T"] % c["sub"])
        set_bytes = 4 * grid * grid * c["chans"] * (4 if c["pols"] == 2 else 1)
        c["T"] = min(c["T"], max(1, int(2e9 // set_bytes)) * c["sub"])
    return c


# ------------------------------------------------------------------------------- a case's station

def _freq(c):
    return c["f0"] + c["df"] * np.arange(c["chans"])


def _positions(c, seed):
    r = np.random.default_rng([seed, 1])
    if c["layout"] == "lattice":
        side = int(round(math.sqrt(c["n_ant"])))
        g = (np.arange(side) - 0.5 * (side - 1)) * c["size"]
        x, y = np.meshgrid(g, g)
        p = np.stack([x.ravel(), y.ravel()], axis=1)
        return p + r.uniform(-0.05, 0.05, p.shape) * c["size"]
    rad, th = np.sqrt(r.random(c["n_ant"])), 2.0 * math.pi * r.random(c["n_ant"])
    return np.stack([0.5 * c["size"] * rad * np.cos(th), 0.5 * c["size_y"] * rad * np.sin(th)], axis=1)


def _table(c):
    """A complex kernel sampled `table` times per cell: a Gaussian with a phase gradient."""
    if not c["table"]:
        return None
    d = np.arange(c["K"] * c["table"] + 1) / c["table"] - 0.5 * c["K"]
    x, y = np.meshgrid(d, d)
    w = np.exp(-(x * x + y * y) / (2.0 * c["sigma"] ** 2)) * np.exp(1j * (0.3 * x - 0.2 * y))
    return np.ascontiguousarray(w.astype(np.complex64)).view(np.float32)


def _jones(c, seed):
    """Gains around one with random phases, a few per cent of leakage."""
    if not c["mix"]:
        return None
    r = np.random.default_rng([seed, 2])
    n = (c["chans"], c["n_ant"])
    j = 0.035 * (r.standard_normal(n + (2, 2)) + 1j * r.standard_normal(n + (2, 2)))
    for p in range(2):
        j[..., p, p] = (1.0 + 0.1 * r.standard_normal(n)) * np.exp(1j * r.uniform(-math.pi, math.pi, n))
    return j.astype(np.complex64)


def _voltages(c, seed, pos):
    """Quantised noise and three sources on the GPU: uint8 [T][C][A][P] (8 + 8 bits: [...][2])."""
    g = torch.Generator(device="cuda").manual_seed(seed * 1000003 + 17)
    r = np.random.default_rng([seed, 3])
    lm = r.uniform(-0.5, 0.5, (3, 2))
    lam = C0 / _freq(c)
    ph = torch.from_numpy(np.exp(-2j * math.pi * (pos @ lm.T)[None] / lam[:, None, None]).astype(np.complex64)).cuda()  # C A S
    amp = torch.tensor([0.5, 0.35, 0.25], device="cuda") / math.sqrt(2.0)
    T, C, A, P = c["T"], c["chans"], c["n_ant"], c["pols"]
    out = torch.empty((T, C, A, P) + ((2,) if c["bits"] == 8 else ()), dtype=torch.uint8, device="cuda")
    step = max(1, int(3e7 // (C * A * P)))
    for t in range(0, T, step):
        n = min(step, T - t)
        s = torch.randn((C, 3, n * P, 2), generator=g, device="cuda") * amp[None, :, None, None]
        e = torch.matmul(ph, torch.view_as_complex(s)).reshape(C, A, n, P).permute(2, 0, 1, 3)
        v = torch.view_as_real(e) + 2.0 * torch.randn((n, C, A, P, 2), generator=g, device="cuda")
        if c["bits"] == 8:
            out[t:t + n] = torch.clamp(torch.round(16.0 * v), -127, 127).to(torch.int8).view(torch.uint8)
        else:
            q = torch.clamp(torch.round(v), -7, 7).to(torch.int32)
            out[t:t + n] = ((q[..., 0] & 15) * 16 + (q[..., 1] & 15)).to(torch.uint8)
    return out


def _plan(c, seed):
    f, tab = _freq(c), _table(c)
    return epic.Plan(_positions(c, seed), f, c["pols"], c["grid"], c["K"], c["sigma"], c["f_ref"] or float(f.max()),
                     bool(c["f_ref"]), None, c["path"], c["T"], gcf_table=tab, oversample=max(1, c["table"]),
                     input_bits=c["bits"], sub_int=c["sub"], jones=_jones(c, seed))


def _stations(c):
    """The station types of the streaming mix: 64, 256 and 1024 elements."""
    f = {"chans": c["chans"], "T": c["T"]}
    return [_case(n_ant=64, size=20.0, size_y=20.0, f0=C0 / 2.0, grid=32, K=3, sigma=0.5, **f), _lwa(**f),
            _dense(32, **f)]


# ------------------------------------------------------------------------------- one pass

def prepare(case, seed):
    c = dict(BASE, **case)
    if c["call"] == "server":
        s = {"server": epic.Server(2 << 30, 4), "jobs": [], "plans": []}
        for k, st in enumerate(_stations(c)):
            plan, pos = _plan(st, seed + 100 * k), _positions(st, seed + 100 * k)
            s["plans"].append(plan)
            for b in range(c["blocks"] // len(MIX)):
                volt = _voltages(st, seed + 100 * k + b, pos).cpu().pin_memory()
                s["jobs"].append((plan, volt, torch.zeros(plan.image_shape(st["T"]), device="cuda")))
        s["jobs"] = s["jobs"][::len(MIX)] + s["jobs"][1::len(MIX)] + s["jobs"][2::len(MIX)]
        s["call"] = c["call"]
        torch.cuda.synchronize()
        # a server's slots take their memory with the first block that they run: before it goes live, a
        # program has every slot run each station type
        for job in reversed(s["jobs"][:len(MIX)]):
            spare = [torch.empty_like(job[2]) for _ in range(8)]
            for _ in range(3):
                for t in [s["server"].submit_ptr(job[0], job[1].data_ptr(), job[1].shape[0], o) for o in spare]:
                    s["server"].wait(t)
                torch.cuda.synchronize()
        run(s)
        torch.cuda.synchronize()
        return s
    pos = _positions(c, seed)
    plan = _plan(c, seed)
    s = {"plan": plan, "call": c["call"], "volt": _voltages(c, seed, pos)}
    if c["call"] == "two":
        s["more"] = _voltages(c, seed + 1, pos)
    if c["call"] == "host":
        s["volt"] = s["volt"].cpu().pin_memory()
        s["out"] = torch.empty(plan.image_shape(c["T"])).pin_memory()
    else:
        s["out"] = torch.empty(plan.image_shape(c["T"]), device="cuda")
    torch.cuda.synchronize()
    return s


def run(s):
    call = s["call"]
    if call == "server":
        tickets = [s["server"].submit_ptr(p, v.data_ptr(), v.shape[0], o) for p, v, o in s["jobs"]]
        for t in tickets:
            s["server"].wait(t)
        return [o for _, _, o in s["jobs"]]
    plan = s["plan"]
    if call == "host":
        plan.image_host_ptr(s["volt"].data_ptr(), s["volt"].shape[0], s["out"].data_ptr())
        return s["out"]
    if call == "two":
        plan.image(s["volt"], out=s["out"])
        return plan.image(s["more"], out=s["out"], accumulate=True)
    return plan.image(s["volt"], out=s["out"], graph=call == "graph")


def work(case):
    """Voltages in, images out; gridding (a complex multiply-add per tap, real weights), one 2-D FFT per
    sample, channel and polarisation (5 M log2 M) and the products."""
    c = dict(BASE, **case)
    if c["call"] == "server":
        w = [work(dict(s, call="image")) for s in _stations(c)]
        return {k: sum(x[k] for x in w) * (c["blocks"] // len(MIX)) for k in ("bytes", "flops")}
    n = 2 if c["call"] == "two" else 1
    M, P, C, T = c["grid"] ** 2, c["pols"], c["chans"], c["T"] * n
    volt = T * C * c["n_ant"] * P * (2 if c["bits"] == 8 else 1)
    images = 4 * M * C * (4 if P == 2 else 1) * (c["T"] // c["sub"] if c["sub"] else 1)
    taps = (8 if c["table"] else 4) * c["n_ant"] * c["K"] ** 2
    mix = 28 * c["n_ant"] if c["mix"] else 0
    frame = P * (taps + 5 * M * math.log2(M)) + mix + (16 if P == 2 else 4) * M
    return {"bytes": float(volt + images), "flops": float(T * C * frame)}


# ------------------------------------------------------------------------------- the same in 64 bits

def _exact_block(c, seed, pos, volt, out):
    """Adds the images of one block to out (float64 [sets][C][n_prod][N][N])."""
    N, K, P, T, A = c["grid"], c["K"], c["pols"], c["T"], c["n_ant"]
    dev, f64, c128 = "cuda", torch.float64, torch.complex128
    jones = _jones(c, seed)
    tab = _table(c)
    cen = np.array([sum(pos[:, 0].tolist()) / A, sum(pos[:, 1].tolist()) / A])
    sign = torch.ones((N, N), dtype=f64, device=dev)
    sign[1::2] *= -1
    sign[:, 1::2] *= -1
    for i, f in enumerate(_freq(c)):
        u = (pos - cen) / (0.5 * C0 / f) + 0.5 * N
        first = np.floor(u + 0.5) - (K - 1) // 2 if K % 2 else np.floor(u) - K // 2 + 1
        v = volt[:, i].to(torch.int32)
        if c["bits"] == 8:
            v = torch.where(v > 127, v - 256, v).to(f64)
            e = torch.complex(v[..., 0], v[..., 1])
        else:
            hi, lo = v >> 4, v & 15
            e = torch.complex(torch.where(hi > 7, hi - 16, hi).to(f64), torch.where(lo > 7, lo - 16, lo).to(f64))
        if jones is not None:  # J is E's kernel: its conjugate multiplies the samples
            e = torch.einsum("aqp,tap->taq", torch.from_numpy(jones[i]).to(dev, c128).conj(), e)
        step = max(1, int(1.2e9 // (N * N * P * 16)))  # samples at a time; whole image sets where there are several
        if c["sub"]:
            step = max(1, step // c["sub"]) * c["sub"]
        for t in range(0, T, step):
            n = min(step, T - t)
            sub = c["sub"] or n
            cols = torch.view_as_real(e[t:t + n].permute(1, 0, 2).reshape(A, n * P).contiguous()).reshape(A, -1)
            g = torch.zeros((N * N, n * P * 2), dtype=f64, device=dev)
            for ty in range(K):
                for tx in range(K):
                    jx, jy = first[:, 0] + tx, first[:, 1] + ty
                    at = torch.from_numpy((jy * N + jx).astype(np.int64)).to(dev)
                    dx, dy = jx - u[:, 0], jy - u[:, 1]
                    if tab is None:
                        sg = c["sigma"] * (f / c["f_ref"] if c["f_ref"] else 1.0)
                        w = torch.from_numpy(np.exp(-(dx * dx + dy * dy) / (2.0 * sg * sg))).to(dev)
                        g.index_add_(0, at, w[:, None] * cols)
                    else:
                        side = K * c["table"] + 1
                        ix = np.clip(np.floor((dx + 0.5 * K) * c["table"] + 0.5), 0, side - 1).astype(np.int64)
                        iy = np.clip(np.floor((dy + 0.5 * K) * c["table"] + 0.5), 0, side - 1).astype(np.int64)
                        w = torch.from_numpy(np.conj(tab.view(np.complex64).reshape(side, side)[iy, ix]).astype(np.complex128)).to(dev)
                        z = w[:, None] * torch.view_as_complex(cols.reshape(A, -1, 2))
                        g.index_add_(0, at, torch.view_as_real(z).reshape(A, -1))
            z = torch.view_as_complex(g.reshape(N, N, n * P, 2)).permute(2, 0, 1) * sign
            z = torch.fft.ifft2(z, norm="forward").reshape(n // sub, sub, P, N, N)
            x = z[:, :, 0]
            k = t // c["sub"] if c["sub"] else 0
            s = out[k:k + n // sub, i]
            s[:, 0] += (x.real ** 2 + x.imag ** 2).sum(1)
            if P == 2:
                y = z[:, :, 1]
                xy = (x * y.conj()).sum(1)
                s[:, 1] += (y.real ** 2 + y.imag ** 2).sum(1)
                s[:, 2] += xy.real
                s[:, 3] += xy.imag


def exact(case, seed):
    c = dict(BASE, **case)
    if c["call"] == "server":
        outs = []
        for k, st in enumerate(_stations(c)):
            for b in range(c["blocks"] // len(MIX)):
                outs.append(_exact(st, seed + 100 * k, [seed + 100 * k + b]))
        return outs[::len(MIX)] + outs[1::len(MIX)] + outs[2::len(MIX)]
    return _exact(c, seed, [seed, seed + 1] if c["call"] == "two" else [seed])


def _exact(c, seed, seeds):
    pos = _positions(c, seed)
    sets = c["T"] // c["sub"] if c["sub"] else 1
    out = torch.zeros((sets, c["chans"], 4 if c["pols"] == 2 else 1, c["grid"], c["grid"]), dtype=torch.float64, device="cuda")
    for s in seeds:
        _exact_block(c, seed, pos, _voltages(c, s, pos), out)
    if not c["sub"]:
        out = out[0]
    return out.cpu() if c["call"] == "host" else out
