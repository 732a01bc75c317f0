"""Performance cases of the library: the calls a beamforming program makes, over the range of
lattices, sizes and arithmetic forms it makes them with.

A case is a dict of plain values; ``kind`` names the entry point:

  beams     fftbf_execute: voltages -> integrated FFT-beam intensities
  batch     fftbf_batch_execute: several uneven arrays in one launch
  tied      fftbf_tied_beams: tied-array beams regridded from FFT beams
  products  fftbf_stacked_visibilities and fftbf_localise on the same FFT beams
  serve     fftbf_server_*: a burst of host frames of several lattices, submitted and awaited

Voltages are the synthetic workload of the tests and the benchmark: complex Gaussian noise of
sigma 2.5 per part plus plane-wave sources of amplitude 1.5, rounded and clipped to [-7, 7],
drawn on the device. ``exact`` recomputes the results in FP64 with torch.
"""
import math

import numpy as np
import torch

import paper_1710_08591_gb300 as fb

SIGMA, AMPLITUDE = 2.5, 1.5
PRECISIONS = {"fp32": fb.PREC_FP32, "fp16": fb.PREC_TC_FP16, "bf16": fb.PREC_TC_BF16,
              "fp16x3": fb.PREC_TC_FP16X3}
# lattices of the batched and the serving workload (E-W x N-S feeds)
BATCH_LATTICES = [(4, 256), (8, 64), (16, 16), (2, 512), (1, 1024), (3, 128)]
SERVE_LATTICES = [(4, 256), (8, 64), (16, 16)]


def next_pow2(n):
    return 1 << max(0, n - 1).bit_length()


def beams_case(name, nx, ny, pad_x, pad_y, npol, nfreq, n_int, windows, weights, precision="fp32"):
    return dict(name=name, kind="beams", nx=nx, ny=ny, pad_x=pad_x, pad_y=pad_y, npol=npol,
                nfreq=nfreq, n_int=n_int, windows=windows, weights=weights, precision=precision)


def listed():
    return [
        # a small test array; the smallest call a program makes, so launch and latency count
        beams_case("tiny_2x16", 2, 16, 2, 32, 1, 8, 16, 64, "uniform"),
        # one frame of 16 channels of the CHIME-like lattice: the live, latency-bound call
        beams_case("frame_4x256", 4, 256, 4, 512, 2, 16, 384, 1, "half_sine"),
        # the CHIME-like workload, the ordinary throughput call, in each arithmetic form
        beams_case("chime_fp32", 4, 256, 4, 512, 2, 1024, 384, 4, "half_sine"),
        beams_case("chime_fp16", 4, 256, 4, 512, 2, 1024, 384, 4, "half_sine", "fp16"),
        beams_case("chime_bf16", 4, 256, 4, 512, 2, 1024, 384, 4, "half_sine", "bf16"),
        beams_case("band_fp16x3", 4, 256, 4, 512, 2, 256, 384, 4, "half_sine", "fp16x3"),
        # another lattice with per-feed complex gains (calibration folded into the weights)
        beams_case("gains_8x64", 8, 64, 8, 128, 2, 512, 256, 4, "random"),
        # an odd lattice at the minimum padding 2n - 1, one polarisation, ragged window count
        beams_case("ragged_3x37", 3, 37, 5, 73, 1, 60, 100, 6, "random"),
        # twelve uneven arrays in one launch
        dict(name="batch_12", kind="batch", arrays=12, nfreq_min=64, nfreq_max=512, n_int=256,
             windows=4, npol=2, pick=4),
        # 2048 pointings per channel, the tied-array step behind the CHIME-like workload
        dict(name="tied_2048", kind="tied", nx=4, ny=256, pad_x=4, pad_y=512, nfreq=256,
             windows=64, n_tied=2048),
        # monitoring products of the CHIME-like beams
        dict(name="products_4x256", kind="products", nx=4, ny=256, pad_x=4, pad_y=512,
             nfreq=1024, windows=32, n_iter=5, n_taps=10),
        # frames of the serving workload from 48 streams at once
        dict(name="serve_burst", kind="serve", frames=48, nfreq=16, n_int=384, npol=2, pick=5),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["beams", "beams", "beams", "tensor", "batch", "tied", "products", "serve"])
    if kind == "tensor":                       # the tensor-core forms: 4 x 512 beams
        nx, ny = (4, 256) if rng.random() < 0.5 else (rng.randint(1, 4), rng.randint(100, 256))
        c = beams_case("", nx, ny, 4, 512, rng.choice([1, 2]), _log_int(rng, 4, 512),
                       _log_int(rng, 16, 512), 1, rng.choice(["half_sine", "random"]),
                       rng.choice(["fp16", "bf16", "fp16x3"]))
        budget = 2e8 if c["precision"] == "fp16x3" or (nx, ny) != (4, 256) else 1e9
    elif kind == "beams":
        style = rng.choice(["double", "double", "minimum", "folded"])
        if style == "double":                  # N-S padded to 2x the next power of two
            nx = rng.choice([1, 2, 3, 4, 8, 16])
            ny = rng.randint(max(2, 12 // nx), 1024 // nx)
            px, py = nx, 2 * next_pow2(ny)
            budget = 5e8
        elif style == "minimum":               # 2n - 1 on both axes
            nx, ny = rng.randint(1, 6), _log_int(rng, 6, 64)
            px, py = 2 * nx - 1, 2 * ny - 1
            budget = 4e6
        else:                                  # fewer beams than feeds: cyclic co-adding
            nx, ny = rng.randint(2, 8), rng.randint(8, 100)
            px, py = nx, max(4, next_pow2(ny) // 2)
            budget = 2e7
        c = beams_case("", nx, ny, px, py, rng.choice([1, 2]), _log_int(rng, 4, 512),
                       _log_int(rng, 8, 512), 1, rng.choice(["uniform", "half_sine", "random"]))
    elif kind == "batch":
        c = dict(kind="batch", arrays=rng.randint(2, 10), nfreq_min=32,
                 nfreq_max=rng.randint(64, 400), n_int=rng.choice([64, 100, 128, 256]),
                 windows=rng.randint(1, 4), npol=rng.choice([1, 2]), pick=rng.randint(0, 10 ** 6))
        return c
    elif kind == "tied":
        nx, ny = rng.choice([(4, 256), (2, 300), (4, 100)])
        return dict(kind="tied", nx=nx, ny=ny, pad_x=nx, pad_y=2 * next_pow2(ny),
                    nfreq=_log_int(rng, 4, 256), windows=_log_int(rng, 2, 64),
                    n_tied=_log_int(rng, 64, 2048))
    elif kind == "products":
        nx, ny = rng.choice([(4, 256), (4, 200), (8, 64), (2, 500)])
        return dict(kind="products", nx=nx, ny=ny, pad_x=nx, pad_y=2 * next_pow2(ny),
                    nfreq=_log_int(rng, 8, 512), windows=rng.randint(1, 32), n_iter=5, n_taps=10)
    else:
        return dict(kind="serve", frames=rng.randint(4, 48), nfreq=rng.choice([8, 16, 24]),
                    n_int=rng.choice([128, 384, 500]), npol=2, pick=rng.randint(0, 10 ** 6))
    del c["name"]
    most = max(1, int(budget / (c["nx"] * c["ny"] * c["npol"] * c["nfreq"] * c["n_int"])))
    c["windows"] = _log_int(rng, 1, min(most, 64))
    while c["nx"] * c["ny"] * c["npol"] * c["nfreq"] * c["n_int"] * c["windows"] > budget and c["nfreq"] > 1:
        c["nfreq"] //= 2
    return c


# ------------------------------------------------------------------------------- inputs --
def _generator(seed, salt=0):
    g = torch.Generator(device="cuda")
    g.manual_seed(1000003 * int(seed) + salt)
    return g


def _voltages(nt, nfreq, npol, nx, ny, seed, salt=0, n_src=3):
    """uint8 [nt][nfreq][npol][nx][ny]: noise plus plane waves, rounded and clipped."""
    g = _generator(seed, salt)
    dev = torch.device("cuda")
    uv = torch.rand((n_src, 2), generator=g, device=dev)
    wave = [torch.polar(torch.full((nx, ny), AMPLITUDE, device=dev),
                        2 * math.pi * (uv[s, 0] * torch.arange(nx, device=dev)[:, None] +
                                       uv[s, 1] * torch.arange(ny, device=dev)[None, :]))
            for s in range(n_src)]
    out = torch.empty((nt, nfreq, npol, nx, ny), dtype=torch.uint8, device=dev)
    step = max(1, (1 << 26) // (nfreq * npol * nx * ny))
    for t in range(0, nt, step):
        m = min(step, nt - t)
        x = torch.randn((m, nfreq, npol, nx, ny, 2), generator=g, device=dev).mul_(SIGMA)
        z = torch.view_as_complex(x)
        for s in range(n_src):
            ph = torch.rand((m, nfreq, npol, 1, 1), generator=g, device=dev) * (2 * math.pi)
            z += torch.polar(torch.ones_like(ph), ph) * wave[s]
        q = x.round_().clamp_(-7, 7).to(torch.int8)
        out[t:t + m] = ((q[..., 0] & 15) << 4 | (q[..., 1] & 15)).view(torch.uint8)
    return out


def _weights(kind, nx, ny, seed):
    if kind == "uniform":
        return None
    if kind == "half_sine":                    # the apodisation of the CHIME-like workload
        h = lambda n: np.sin(np.pi * (np.arange(n) + 0.5) / n)  # noqa: E731
        return np.outer(h(nx), h(ny)).astype(np.complex64)
    rng = np.random.default_rng(seed)          # per-feed complex gains
    amp = 0.5 + rng.random((nx, ny))
    return (amp * np.exp(1j * rng.uniform(-np.pi, np.pi, (nx, ny)))).astype(np.complex64)


def _array(c, seed):
    """One array's device voltages, host weights and output buffer."""
    T = c["windows"] * c["n_int"]
    v = _voltages(T, c["nfreq"], c["npol"], c["nx"], c["ny"], seed, c.get("salt", 0))
    return v, _weights(c["weights"], c["nx"], c["ny"], seed)


def _plan(c, w):
    return fb.plan_create(c["nx"], c["ny"], c["pad_x"], c["pad_y"], c["npol"], c["nfreq"],
                          c["n_int"], weights=w)


def _batch_arrays(case):
    """The arrays of a batch: lattices and channel counts from the case alone."""
    rng = np.random.default_rng(case["pick"])
    arrays = []
    for i in range(case["arrays"]):
        nx, ny = BATCH_LATTICES[int(rng.integers(len(BATCH_LATTICES)))]
        nf = int(rng.integers(case["nfreq_min"], case["nfreq_max"] + 1))
        arrays.append(dict(nx=nx, ny=ny, pad_x=nx, pad_y=2 * next_pow2(ny), npol=case["npol"],
                           nfreq=nf, n_int=case["n_int"], windows=case["windows"],
                           weights="half_sine", salt=100 + i))
    return arrays


def _intensities(case, seed):
    """FFT-beam intensities of noise plus one point source per (window, channel)."""
    g = _generator(seed, 7)
    dev, f8 = torch.device("cuda"), torch.float64
    nw, nf = case["windows"], case["nfreq"]

    def response(n, m, y):                     # |sum_a exp(2 pi i a (y - A / m))|^2
        d = y[..., None] - torch.arange(m, device=dev, dtype=f8) / m
        s = torch.sin(math.pi * d)
        near = s.abs() < 1e-9
        return torch.where(near, float(n * n), (torch.sin(n * math.pi * d) /
                                                torch.where(near, 1.0, s)) ** 2)

    y = torch.rand((2, nw, nf), generator=g, device=dev, dtype=f8)
    n_ant, snap = case["nx"] * case["ny"], 768
    out = torch.empty((nw, nf, case["pad_x"], case["pad_y"]), device=dev)
    for w in range(nw):
        src = (response(case["nx"], case["pad_x"], y[0, w])[..., :, None] *
               response(case["ny"], case["pad_y"], y[1, w])[..., None, :]) * (0.25 * snap)
        noise = 1.0 + torch.randn(src.shape, generator=g, device=dev) / math.sqrt(snap)
        out[w] = (src + noise.clamp_min(0.5) * (n_ant * snap * 2 * SIGMA ** 2)).float()
    return out


def _pointings(case, seed):
    """u on the FFT-beam grid (pad_x < 2 nx - 1), v anywhere; the same at every channel."""
    rng = np.random.default_rng(seed)
    nx, px, n = case["nx"], case["pad_x"], case["n_tied"]
    u = rng.random(n) if px >= 2 * nx - 1 else rng.integers(0, px, n) / px
    v = rng.random(n)
    full = (case["nfreq"], n)
    return (np.ascontiguousarray(np.broadcast_to(u, full)),
            np.ascontiguousarray(np.broadcast_to(v, full)))


def _serve_setup(case):
    """Lattices of the frames: the server's three, and which one each frame is of."""
    rng = np.random.default_rng(case["pick"])
    lat = [dict(nx=nx, ny=ny, pad_x=nx, pad_y=2 * next_pow2(ny), npol=case["npol"],
                nfreq=case["nfreq"], n_int=case["n_int"], windows=1, weights="half_sine")
           for nx, ny in SERVE_LATTICES]
    return lat, [int(i) for i in rng.integers(len(lat), size=case["frames"])]


def _serve_frames(case, seed):
    lat, which = _serve_setup(case)
    frames = [None] * len(which)
    for k, c in enumerate(lat):
        mine = [i for i, w in enumerate(which) if w == k]
        if mine:
            v = _voltages(case["n_int"] * len(mine), c["nfreq"], c["npol"], c["nx"], c["ny"],
                          seed, 200 + k)
            for j, i in enumerate(mine):
                frames[i] = v[j * case["n_int"]:(j + 1) * case["n_int"]]
    return lat, which, frames


# ------------------------------------------------------------------------------ the calls --
def prepare(case, seed):
    kind = case["kind"]
    state = dict(case=case)
    if kind == "beams":
        v, w = _array(case, seed)
        plan = _plan(case, w)
        if case["precision"] != "fp32":
            fb.plan_set_precision(plan, PRECISIONS[case["precision"]])
        state.update(v=v, plan=plan, out=torch.empty(
            (case["windows"], case["nfreq"], case["pad_x"], case["pad_y"]), device="cuda"))
    elif kind == "batch":
        arrays = _batch_arrays(case)
        made = [_array(c, seed) for c in arrays]
        plans = [_plan(c, w) for c, (_, w) in zip(arrays, made)]
        state.update(v=[v for v, _ in made], batch=fb.batch_create(plans),
                     stream=torch.cuda.Stream(),
                     out=[torch.empty((c["windows"], c["nfreq"], c["pad_x"], c["pad_y"]),
                                      device="cuda") for c in arrays])
    elif kind == "tied":
        u, v = _pointings(case, seed)
        plan = fb.plan_create(case["nx"], case["ny"], case["pad_x"], case["pad_y"], 2,
                              case["nfreq"], 384)
        state.update(P=_intensities(case, seed), plan=plan, u=u, v=v, out=torch.empty(
            (case["windows"], case["nfreq"], case["n_tied"]), device="cuda"))
    elif kind == "products":
        plan = fb.plan_create(case["nx"], case["ny"], case["pad_x"], case["pad_y"], 2,
                              case["nfreq"], 384)
        full = (case["windows"], case["nfreq"])
        state.update(P=_intensities(case, seed), plan=plan,
                     vis=torch.empty(full + fb.stacked_shape(plan), dtype=torch.complex64,
                                     device="cuda"),
                     pos=torch.empty(full + (3,), device="cuda"))
    else:
        lat, which, frames = _serve_frames(case, seed)
        plans = [_plan(c, _weights(c["weights"], c["nx"], c["ny"], seed)) for c in lat]
        pinned = [torch.empty(f.shape, dtype=torch.uint8, pin_memory=True).copy_(f) for f in frames]
        sizes = [lat[k]["nfreq"] * lat[k]["pad_x"] * lat[k]["pad_y"] for k in which]
        out = torch.zeros(sum(sizes), pin_memory=True).numpy()
        at = np.cumsum([0] + sizes)
        state.update(plans=plans, server=fb.server_create(plans, 4 << 30), which=which,
                     keep=pinned, frames=[p.numpy() for p in pinned], out=out,
                     beams=[out[at[i]:at[i + 1]] for i in range(len(which))])
    return state


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "beams":
        fb.execute(state["plan"], state["v"], case["windows"] * case["n_int"], state["out"])
        return state["out"]
    if kind == "batch":
        st = state["stream"]                   # a batch replays its graph on a stream of its own
        st.wait_stream(torch.cuda.current_stream())
        fb.batch_execute(state["batch"], state["v"], case["windows"] * case["n_int"],
                         state["out"], stream=st)
        torch.cuda.current_stream().wait_stream(st)
        return state["out"]
    if kind == "tied":
        fb.tied_beams(state["plan"], state["P"], case["windows"], case["n_tied"], state["u"],
                      state["v"], state["out"])
        return state["out"]
    if kind == "products":
        fb.stacked_visibilities(state["plan"], state["P"], case["windows"], state["vis"])
        fb.localise(state["plan"], state["P"], case["windows"], state["pos"],
                    n_iter=case["n_iter"], n_taps=case["n_taps"])
        return {"vis": state["vis"], "pos": state["pos"]}
    for k, f, b in zip(state["which"], state["frames"], state["beams"]):
        fb.server_submit(state["server"], k, f, b)
    fb.server_wait(state["server"])            # the results are on the host once this returns
    return state["out"]


def _beam_work(c):
    """Bytes and operations of one array's transform: an FFT of each padded snapshot."""
    snaps = c["windows"] * c["n_int"] * c["npol"] * c["nfreq"]
    nant, nout = c["nx"] * c["ny"], c["pad_x"] * c["pad_y"]
    lx, ly = math.log2(max(2, c["pad_x"])), math.log2(max(2, c["pad_y"]))
    ops = 6 * nant + 5 * c["pad_x"] * lx * min(c["ny"], c["pad_y"]) + 5 * nout * ly + 4 * nout
    return snaps * nant + 4 * c["windows"] * c["nfreq"] * nout, snaps * ops


def work(case):
    kind = case["kind"]
    if kind == "beams":
        b, f = _beam_work(case)
    elif kind == "batch":
        parts = [_beam_work(c) for c in _batch_arrays(case)]
        b, f = (sum(p[i] for p in parts) for i in (0, 1))
    elif kind == "serve":
        lat, which = _serve_setup(case)
        parts = [_beam_work(lat[k]) for k in which]
        b, f = (sum(p[i] for p in parts) for i in (0, 1))
    else:
        rows = case["windows"] * case["nfreq"]
        nout = case["pad_x"] * case["pad_y"]
        if kind == "tied":
            b = 4 * rows * (nout + case["n_tied"]) + 8 * case["nfreq"] * case["n_tied"] * 2
            f = 2.0 * rows * case["n_tied"] * case["pad_y"]
        else:
            dx = 2 * case["nx"] - 1 if case["pad_x"] >= 2 * case["nx"] - 1 else case["pad_x"]
            b = rows * (4 * nout + 8 * dx * (2 * case["ny"] - 1) + 12)
            f = rows * 5.0 * nout * math.log2(case["pad_y"]) / 2
    return {"bytes": float(b), "flops": float(f)}


# ------------------------------------------------------------------- results in 64 bits --
def _unpack64(v):
    q = v.to(torch.int16)
    re, im = q >> 4, q & 15
    re, im = torch.where(re > 7, re - 16, re), torch.where(im > 7, im - 16, im)
    return torch.complex(re.double(), im.double())


def _beams64(c, v, w):
    """The integrated beams of voltages v: fold or pad to the beam grid, FFT, |.|^2, sum."""
    nw, nf, px, py = c["windows"], c["nfreq"], c["pad_x"], c["pad_y"]
    nx, ny, n_int, npol = c["nx"], c["ny"], c["n_int"], c["npol"]
    w64 = torch.ones((nx, ny), dtype=torch.complex128) if w is None else torch.from_numpy(w).to(torch.complex128)
    w64 = w64.cuda()
    out = torch.zeros((nw, nf, px, py), dtype=torch.float64, device="cuda")
    gx, gy = px * math.ceil(nx / px), py * math.ceil(ny / py)
    fstep = max(1, min(nf, (1 << 24) // (npol * max(gx * gy, px * py))))
    tstep = max(1, (1 << 24) // (fstep * npol * max(gx * gy, px * py)))
    for j in range(nw):
        for f in range(0, nf, fstep):
            for t in range(j * n_int, (j + 1) * n_int, tstep):
                x = _unpack64(v[t:min(t + tstep, (j + 1) * n_int), f:f + fstep].contiguous()) * w64
                x = torch.nn.functional.pad(x, (0, gy - ny, 0, gx - nx))
                x = x.reshape(x.shape[:3] + (gx // px, px, gy // py, py)).sum(dim=(3, 5))
                y = torch.fft.fft2(x)
                out[j, f:f + fstep] += (y.real ** 2 + y.imag ** 2).sum(dim=(0, 2))
    return out


def _dirichlet64(n, m, y):
    """Regridding weights of pointings y onto m FFT beams, [.., m]."""
    d = y[..., None] - torch.arange(m, device="cuda", dtype=torch.float64) / m
    s = torch.sin(math.pi * d)
    near = s.abs() < 1e-12
    return torch.where(near, (2 * n - 1.0) / m, torch.sin((2 * n - 1) * math.pi * d) /
                       (m * torch.where(near, 1.0, s)))


def exact(case, seed):
    kind = case["kind"]
    if kind == "beams":
        v, w = _array(case, seed)
        return _beams64(case, v, w)
    if kind == "batch":
        return [_beams64(c, *_array(c, seed)) for c in _batch_arrays(case)]
    if kind == "serve":
        lat, which, frames = _serve_frames(case, seed)
        return torch.cat([_beams64(lat[k], f, _weights(lat[k]["weights"], lat[k]["nx"],
                                                       lat[k]["ny"], seed)).reshape(-1)
                          for k, f in zip(which, frames)])
    P = _intensities(case, seed).double()
    nx, ny, px, py = case["nx"], case["ny"], case["pad_x"], case["pad_y"]
    if kind == "tied":
        u, v = (torch.from_numpy(a[0].copy()).cuda() for a in _pointings(case, seed))
        if px >= 2 * nx - 1:
            wx = _dirichlet64(nx, px, u)
        else:
            wx = torch.nn.functional.one_hot((u * px).round().long() % px, px).double()
        wy = _dirichlet64(ny, py, v)
        return torch.cat([torch.einsum("jfab,sa,sb->jfs", P[j:j + 4], wx, wy)
                          if px > 4 else
                          sum(torch.einsum("jfb,sb->jfs", P[j:j + 4, :, a], wx[:, a, None] * wy)
                              for a in range(px))
                          for j in range(0, case["windows"], 4)])

    def inverse(x, n, m, dim):                 # lags -(n-1) .. n-1 of an axis
        if m < 2 * n - 1:
            return x
        z = torch.fft.ifft(x, dim=dim)
        lags = torch.arange(-(n - 1), n, device="cuda") % m
        return z.index_select(dim, lags)

    V = inverse(inverse(P.to(torch.complex128), ny, py, 3), nx, px, 2)
    return {"vis": V, "pos": None}
