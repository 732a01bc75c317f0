"""The covariance form of the FP32 path (beam_corr.cu), forced at the sizes where its tiles,
runs and stages can go wrong, against the oracle and the FFT kernels."""
import numpy as np
import pytest

import synth
from helpers import TOL_BEAM, make_case, oracle_beams, rel_err_per_beam

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1710_08591_gb300 as fb  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    fb.build()
    fb.lib()


def run(v, w, nx, ny, mx, my, npol, nfreq, n_int, offset=0):
    T = v.shape[0]
    flat = torch.from_numpy(np.ascontiguousarray(v).reshape(-1))
    base = torch.zeros(flat.numel() + 16, dtype=torch.uint8, device="cuda")
    dv = base[offset:offset + flat.numel()]
    dv.copy_(flat)
    out = torch.full((T // n_int, nfreq, mx, my), float("nan"), device="cuda")
    with fb.plan_create(nx, ny, mx, my, npol, nfreq, n_int, weights=w) as plan:
        fb.execute(plan, dv, T, out)
        fb.plan_sync(plan)
    return out.cpu().numpy()


CASES = [
    # nx, ny, mx, my, npol, nfreq, n_int, windows, weights
    (1, 16, 1, 32, 1, 1, 31, 1, "uniform"),      # one tile, 32 columns, part of one K step
    (2, 16, 2, 32, 1, 200, 33, 2, "random"),     # several items per CTA pair, second K step begun
    (16, 16, 16, 32, 2, 2, 48, 1, "half_sine"),  # 16-slot rows, one full tile
    (17, 16, 17, 32, 1, 2, 64, 1, "random"),     # 272 slots: a second tile column of 32
    (4, 32, 4, 64, 2, 2, 40, 1, "half_sine"),    # 32-slot rows
    (9, 32, 9, 63, 1, 2, 65, 1, "random"),       # 288 slots, odd beam counts
    (8, 64, 8, 128, 2, 2, 50, 2, "half_sine"),   # 64-slot rows
    (5, 64, 4, 128, 1, 2, 70, 1, "random"),      # 320 slots, E-W folded
    (3, 128, 3, 256, 2, 2, 36, 1, "half_sine"),  # 128-slot rows, a half-wide tile column
    (3, 128, 4, 256, 4, 1, 20, 1, "random"),     # four polarisations, E-W padded
    (4, 256, 4, 512, 2, 2, 96, 2, "half_sine"),  # 256-slot rows: one pair of rows per tile
    (2, 512, 2, 1024, 1, 1, 40, 1, "half_sine"), # rows longer than a tile
    (1, 1024, 1, 2048, 1, 1, 33, 1, "random"),
    (4, 80, 7, 159, 1, 2, 45, 1, "half_sine"),   # rows of 80: runs of 16, 320 slots
    (3, 96, 3, 192, 2, 2, 40, 1, "half_sine"),   # rows of 96: runs of 32
    (3, 37, 5, 73, 1, 3, 100, 2, "random"),      # not a multiple of 16: direct loads, minimum padding
    (2, 100, 2, 256, 3, 2, 25, 1, "half_sine"),  # direct loads, three polarisations, rows padded to 128
    (2, 200, 2, 512, 1, 2, 64, 1, "random"),     # rows padded to 256
    (6, 20, 4, 8, 1, 2, 96, 1, "random"),        # cyclic co-adding on both axes
    (1, 1, 1, 1, 1, 2, 64, 1, "random"),         # one feed, one beam
]


@pytest.mark.parametrize("case", CASES, ids=lambda c: "x".join(map(str, c[:4])) + f"_p{c[4]}_n{c[6]}_{c[8]}")
def test_covariance_matches_oracle(case, monkeypatch):
    """TOL_BEAM is the FP32 bound of every beam; the sums here are exact integers, weighted in
    FP32 and summed and transformed in two-float arithmetic, so what is left is the rounding
    of the weighted products (about 2^-24 each, random)."""
    monkeypatch.setenv("FFTBF_FP32_PATH", "cov")
    nx, ny, mx, my, npol, nfreq, n_int, nwin, wk = case
    v, w = make_case(nx, ny, mx, my, npol, nfreq, n_int * nwin, n_int, weights=wk, seed=17)
    got = run(v, w, nx, ny, mx, my, npol, nfreq, n_int)
    ref = oracle_beams(v, w, nx, ny, mx, my, npol, nfreq, n_int)
    assert np.all(np.isfinite(got))
    err = rel_err_per_beam(got, ref)
    assert err.max() <= TOL_BEAM, f"max rel err {err.max():.3g}"


def test_misaligned_voltages_give_identical_beams(monkeypatch):
    """Off a 16-byte boundary the voltages are loaded directly instead of by TMA."""
    monkeypatch.setenv("FFTBF_FP32_PATH", "cov")
    shape = (4, 64, 4, 128, 2, 3, 40)
    nx, ny, mx, my, npol, nfreq, n_int = shape
    v, w = make_case(nx, ny, mx, my, npol, nfreq, 2 * n_int, n_int, weights="random", seed=5)
    assert np.array_equal(run(v, w, *shape), run(v, w, *shape, offset=3))


def test_saturated_source_no_worse_than_the_transform(monkeypatch):
    """A full-scale coherent source over quantised noise: the covariance's weak beams are
    small differences of large sums. Its error against the oracle stays within the FFT
    kernels' bound of 1e-5 of every beam."""
    shape = (4, 256, 4, 512, 2, 1, 192)
    nx, ny, mx, my, npol, nfreq, n_int = shape
    v = synth.volts(n_int, nfreq, npol, nx, ny, seed=8, sigma=1.0, sources=[(0.137, 0.291, 5.0)])
    w = synth.separable_weights(synth.half_sine(nx), synth.half_sine(ny))
    ref = oracle_beams(v, w, nx, ny, mx, my, npol, nfreq, n_int)
    monkeypatch.setenv("FFTBF_FP32_PATH", "cov")
    assert rel_err_per_beam(run(v, w, *shape), ref).max() <= TOL_BEAM


def test_constant_input_is_exact(monkeypatch):
    """Every voltage at -8 - 8i, the largest product: uniform weights put all power in beam
    (0, 0) and exactly none elsewhere; nothing is negative."""
    monkeypatch.setenv("FFTBF_FP32_PATH", "cov")
    nx, ny, n_int = 4, 16, 300
    v = np.full((n_int, 1, 1, nx, ny), 0x88, np.uint8)
    got = run(v, None, nx, ny, nx, ny, 1, 1, n_int)[0, 0]
    assert got[0, 0] == n_int * 128 * (nx * ny) ** 2
    rest = got.copy()
    rest[0, 0] = 0
    assert rest.min() >= 0 and rest.max() <= 1e-12 * got[0, 0]


def _batch(arrays, n_int, nwin, stream=None):
    plans = [fb.plan_create(*s, 2, v.shape[1], n_int, weights=w)
             for s, v, w in arrays]
    dvs = [torch.from_numpy(np.ascontiguousarray(v).reshape(-1)).cuda() for _, v, _ in arrays]
    outs = [torch.full((nwin, v.shape[1], s[2], s[3]), float("nan"), device="cuda") for s, v, _ in arrays]
    with fb.batch_create(plans) as b:
        for _ in range(2):
            fb.batch_execute(b, dvs, nwin * n_int, outs, stream)
        torch.cuda.synchronize()
    for p in plans:
        fb.plan_sync(p)
        p.close()
    return [o.cpu().numpy() for o in outs]


@pytest.mark.parametrize("n_int", [50, 320])
def test_batch_of_covariance_and_fft_arrays(n_int):
    """100 snapshots per window: only the 8x64 arrays take the covariance; 640: all do, real
    and complex weights in one launch. Every array matches the oracle and is bit-identical
    alone and in the mix, captured or not."""
    nwin = 2
    shapes = [(4, 256, 4, 512), (8, 64, 8, 128), (16, 16, 16, 32), (2, 512, 2, 1024), (1, 1024, 1, 2048),
              (3, 128, 3, 256)]
    arrays = []
    for k, s in enumerate(shapes):
        v, w = make_case(*s, 2, 1 + k % 3, n_int * nwin, n_int, weights="random" if k % 2 else "half_sine",
                         seed=60 + k)
        arrays.append((s, v, w))
    mix = _batch(arrays, n_int, nwin, torch.cuda.Stream())
    plain = _batch(arrays, n_int, nwin)
    for k, ((s, v, w), g) in enumerate(zip(arrays, mix)):
        ref = oracle_beams(v, w, *s, 2, v.shape[1], n_int)
        assert rel_err_per_beam(g, ref).max() <= TOL_BEAM, s
        assert np.array_equal(g, plain[k]), s
        assert np.array_equal(g, _batch([arrays[k]], n_int, nwin)[0]), s


def test_server_frames_through_the_covariance():
    """Frames of 320 samples x 2 polarisations on two lattices: the server's beams are those of
    a batch of the frame alone and match the oracle."""
    n_int, nf = 320, 2
    shapes = [(8, 64, 8, 128), (4, 256, 4, 512)]
    frames, outs = [], []
    plans = [fb.plan_create(*s, 2, nf, n_int) for s in shapes]
    with fb.server_create(plans, 64 << 20) as sv:
        for k in range(6):
            s = shapes[k % 2]
            v, _ = make_case(*s, 2, nf, n_int, n_int, seed=200 + k)
            frames.append(v)
            outs.append(np.full((nf, s[2], s[3]), np.nan, np.float32))
            fb.server_submit(sv, k % 2, v.reshape(-1), outs[-1])
        fb.server_wait(sv)
    for k, (v, o) in enumerate(zip(frames, outs)):
        s = shapes[k % 2]
        ref = oracle_beams(v, None, *s, 2, nf, n_int)
        assert rel_err_per_beam(o[None], ref).max() <= TOL_BEAM
        assert np.array_equal(o[None], _batch([(s, v, None)], n_int, 1)[0])
    for p in plans:
        p.close()


def test_batch_on_alternating_buffers():
    """One batch on two sets of buffers of different contents in turn: each call rewrites the job
    table and its tensor maps in place, and every array's beams are its own buffers'."""
    n_int, nwin = 320, 2
    shapes = [(4, 256, 4, 512), (8, 64, 8, 128), (16, 16, 16, 32)]
    T = nwin * n_int
    plans = [fb.plan_create(*s, 2, 2, n_int) for s in shapes]
    sets = []
    for k in range(2):
        g = torch.Generator(device="cuda")
        g.manual_seed(40 + k)
        vs = [torch.randint(0, 256, (T * 2 * 2 * s[0] * s[1],), dtype=torch.uint8, device="cuda", generator=g)
              for s in shapes]
        want = [torch.empty((nwin, 2, s[2], s[3]), device="cuda") for s in shapes]
        for p, v, o in zip(plans, vs, want):
            fb.execute(p, v, T, o)
        sets.append((vs, want, [torch.empty_like(o) for o in want]))
    st = torch.cuda.Stream()
    torch.cuda.synchronize()
    with fb.batch_create(plans) as b:
        for turn in range(24):
            vs, want, outs = sets[turn % 2]
            for o in outs:
                o.fill_(float("nan"))
            torch.cuda.synchronize()
            fb.batch_execute(b, vs, T, outs, st if turn % 3 else None)
            torch.cuda.synchronize()
            for o, w in zip(outs, want):
                assert torch.equal(o, w), turn
    for p in plans:
        fb.plan_sync(p)
        p.close()


def test_server_ticks_reuse_slots_for_other_lattices():
    """Rounds of frames through few slots: every tick rewrites its table with other slots, lattices
    and contents, and each frame's beams are those of its own voltages."""
    n_int, nf = 320, 2
    shapes = [(8, 64, 8, 128), (4, 256, 4, 512), (16, 16, 16, 32)]
    plans = [fb.plan_create(*s, 2, nf, n_int) for s in shapes]
    rng = np.random.default_rng(9)
    with fb.server_create(plans, 16 << 20) as sv:
        for _ in range(6):
            frames, outs, which = [], [], rng.integers(3, size=8)
            for k in which:
                s = shapes[k]
                frames.append(rng.integers(0, 256, n_int * nf * 2 * s[0] * s[1], dtype=np.uint8))
                outs.append(np.full((nf, s[2], s[3]), np.nan, np.float32))
                fb.server_submit(sv, int(k), frames[-1], outs[-1])
            fb.server_wait(sv)
            for k, v, o in zip(which, frames, outs):
                want = torch.empty((1,) + o.shape, device="cuda")
                fb.execute(plans[k], torch.from_numpy(v).cuda(), n_int, want)
                assert np.array_equal(o, want.cpu().numpy()[0])
    for p in plans:
        p.close()


STRONG = [(1.5, 2.5), (5.0, 1.0), (6.0, 1.0), (6.5, 0.5), (7.0, 0.3)]    # source amplitude, noise sigma


@pytest.mark.parametrize("weights", ["half_sine", "random"])
@pytest.mark.parametrize("shape", [(4, 256, 4, 512, 2, 384), (8, 64, 8, 128, 2, 256), (4, 32, 4, 64, 2, 256),
                                   (16, 16, 16, 32, 2, 256), (3, 37, 5, 73, 1, 200)],
                         ids=lambda s: "x".join(map(str, s[:4])))
def test_weak_beams_beside_a_strong_source(shape, weights, monkeypatch):
    """Every beam within 1e-6, tighter than TOL_BEAM and than what the transform of every snapshot
    reaches on the larger lattices: the sums keep 2^-37 of a source's power or better and the beams
    here are down to 2^-19 of it, so little more than the last rounding (2^-24) is left."""
    nx, ny, mx, my, npol, n_int = shape
    for amp, sigma in STRONG:
        v = synth.volts(n_int, 1, npol, nx, ny, seed=8, sigma=sigma, sources=[(0.137, 0.291, amp)])
        w = synth.separable_weights(synth.half_sine(nx), synth.half_sine(ny)) if weights == "half_sine" \
            else synth.random_weights(nx, ny, 5)
        ref = oracle_beams(v, w, nx, ny, mx, my, npol, 1, n_int)
        monkeypatch.setenv("FFTBF_FP32_PATH", "cov")
        cov = rel_err_per_beam(run(v, w, nx, ny, mx, my, npol, 1, n_int), ref).max()
        monkeypatch.setenv("FFTBF_FP32_PATH", "fft")
        fft = rel_err_per_beam(run(v, w, nx, ny, mx, my, npol, 1, n_int), ref).max()
        assert fft <= TOL_BEAM, (amp, sigma, fft)
        assert cov <= 1e-6, (amp, sigma, cov, fft)


@pytest.mark.parametrize("kind", ["half_sine", "random"])
def test_weight_scale_and_range(kind, monkeypatch):
    """Weights times a power of two give beams times its square, bit for bit, and what overflows is
    infinite; a weight that is not finite takes the transform."""
    monkeypatch.setenv("FFTBF_FP32_PATH", "cov")
    shape = (4, 32, 4, 64, 2, 1, 64)
    nx, ny, mx, my, npol, nfreq, n_int = shape
    v, w = make_case(nx, ny, mx, my, npol, nfreq, n_int, n_int, weights=kind, seed=6)
    one = run(v, w, *shape)
    for e in (-40, 13, 40):
        assert np.array_equal(run(v, w * np.float32(2.0 ** e), *shape), one * np.float32(2.0 ** (2 * e)))
    assert np.all(np.isposinf(run(v, w * np.float32(2.0 ** 63), *shape)))
    bad = w.copy()
    bad[1, 3] = np.nan
    got = run(v, bad, *shape)
    monkeypatch.setenv("FFTBF_FP32_PATH", "fft")
    assert np.array_equal(got, run(v, bad, *shape), equal_nan=True)


def test_batch_mix_of_both_routes():
    """220 snapshots per window: some arrays take the covariance and others the transform, real and
    complex weights in both; each matches the oracle and is bit-identical alone."""
    n_int, nwin = 110, 2
    shapes = [(4, 256, 4, 512), (8, 64, 8, 128), (16, 16, 16, 32), (2, 512, 2, 1024), (1, 1024, 1, 2048),
              (3, 128, 3, 256), (8, 64, 8, 128), (3, 128, 3, 256)]
    arrays = []
    for k, s in enumerate(shapes):
        v, w = make_case(*s, 2, 1 + k % 3, n_int * nwin, n_int, weights="random" if k % 2 else "half_sine",
                         seed=80 + k)
        arrays.append((s, v, w))
    plans = [fb.plan_create(*s, 2, v.shape[1], n_int, weights=w) for s, v, w in arrays]
    with fb.batch_create(plans) as b:
        steps = [fb.batch_tuned_steps(b, i) for i in range(len(plans))]
    for p in plans:
        p.close()
    assert 64 in steps and any(t != 64 for t in steps), steps
    mix = _batch(arrays, n_int, nwin, torch.cuda.Stream())
    for (s, v, w), g in zip(arrays, mix):
        ref = oracle_beams(v, w, *s, 2, v.shape[1], n_int)
        assert rel_err_per_beam(g, ref).max() <= TOL_BEAM, s
        assert np.array_equal(g, _batch([(s, v, w)], n_int, nwin)[0]), s


@pytest.mark.parametrize("shape", [(4, 512, 4, 1024), (16, 64, 4, 128), (64, 32, 8, 64), (32, 16, 2, 32)],
                         ids=lambda s: "x".join(map(str, s)))
@pytest.mark.parametrize("weight", [0.7, 0.7 + 0.3j])
def test_many_pairs_of_one_separation(shape, weight, monkeypatch):
    """More than 1024 feed pairs of one separation, up to 16384 with co-added E-W rows: equal weights
    that are no short binary fractions and a strong source make every product's part below a unit
    of V alike, so that they add up. The bounds are those of the strong-source test; FP64 route."""
    monkeypatch.setenv("FFTBF_FP32_PATH", "cov")
    nx, ny, mx, my = shape
    n_int = 64
    v = synth.volts(n_int, 1, 1, nx, ny, seed=4, sigma=0.3, sources=[(0.0, 0.0, 7.0)])
    w = np.full((nx, ny), weight, np.complex64)
    got = run(v, w, nx, ny, mx, my, 1, 1, n_int)
    ref = oracle_beams(v, w, nx, ny, mx, my, 1, 1, n_int)
    assert rel_err_per_beam(got, ref).max() <= 1e-6


def test_first_call_of_a_thread():
    """A host thread whose first CUDA call is the covariance route: the tensor map needs a context,
    which the runtime has not bound to the thread yet."""
    import threading
    shape = (8, 64, 8, 128)
    plan = fb.plan_create(*shape, 2, 1, 320)
    v = torch.randint(0, 256, (320 * 2 * 512,), dtype=torch.uint8, device="cuda")
    want, got = (torch.empty((1, 1, 8, 128), device="cuda") for _ in range(2))
    errors = []
    fb.execute(plan, v, 320, want)
    stream = torch.cuda.current_stream()
    torch.cuda.synchronize()

    def work():
        try:
            fb.execute(plan, v, 320, got, stream=stream)
        except Exception as e:  # noqa: BLE001 - reported below
            errors.append(e)

    t = threading.Thread(target=work)
    t.start()
    t.join()
    assert not errors, errors[0]
    fb.plan_sync(plan)
    plan.close()
    assert torch.equal(got, want)


def test_launches_of_different_sizes_from_several_threads(monkeypatch):
    """Threads that launch lattices of different shared-memory sizes at once: the kernel's limit is
    the same for all, so no launch is refused."""
    import threading
    monkeypatch.setenv("FFTBF_FP32_PATH", "cov")
    shapes = [(4, 256, 4, 512), (1, 16, 1, 32), (8, 64, 8, 128), (2, 32, 2, 64)]
    jobs, errors = [], []
    for k, s in enumerate(shapes):
        v, _ = make_case(*s, 1, 1, 32, 32, seed=k)
        dv = torch.from_numpy(np.ascontiguousarray(v).reshape(-1)).cuda()
        jobs.append((fb.plan_create(*s, 1, 1, 32), dv, torch.empty((1, 1, s[2], s[3]), device="cuda"),
                     torch.cuda.Stream()))
    torch.cuda.synchronize()

    def work(plan, dv, out, st):
        try:
            for _ in range(1500):
                fb.execute(plan, dv, 32, out, stream=st)
        except Exception as e:  # noqa: BLE001 - reported below
            errors.append(e)

    threads = [threading.Thread(target=work, args=j) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    for j in jobs:
        fb.plan_sync(j[0])
        j[0].close()
    assert not errors, errors[0]


def test_batch_of_staged_and_direct_voltages(monkeypatch):
    """Aligned arrays beside one of 60-feed rows and one off a 16-byte boundary, several items of each
    per CTA pair: every array's beams are the bits of its own call, and match the oracle."""
    monkeypatch.setenv("FFTBF_FP32_PATH", "cov")
    n_int, nwin = 160, 3
    shapes = [(4, 256, 4, 512, 40), (8, 60, 8, 128, 33), (8, 64, 8, 128, 50), (4, 256, 4, 512, 3), (3, 100, 3, 256, 20)]
    rng = np.random.default_rng(12)
    plans, dvs, outs, vs = [], [], [], []
    for k, (nx, ny, mx, my, nf) in enumerate(shapes):
        w = synth.random_weights(nx, ny, k) if k in (2, 4) else None
        plans.append(fb.plan_create(nx, ny, mx, my, 2, nf, n_int, weights=w))
        v = rng.integers(0, 256, (nwin * n_int, nf, 2, nx, ny), dtype=np.uint8)
        base = torch.empty(v.size + 16, dtype=torch.uint8, device="cuda")
        dvs.append(base[5 * (k == 3):][:v.size])
        dvs[-1].copy_(torch.from_numpy(v.reshape(-1)))
        outs.append(torch.full((nwin, nf, mx, my), float("nan"), device="cuda"))
        vs.append((v, w))
    with fb.batch_create(plans) as b:
        assert {fb.batch_tuned_steps(b, i) for i in range(len(plans))} == {64}
        fb.batch_execute(b, dvs, nwin * n_int, outs, torch.cuda.Stream())
        torch.cuda.synchronize()
    for p, d, o, (v, w), s in zip(plans, dvs, outs, vs, shapes):
        own = torch.empty_like(o)
        fb.execute(p, d, nwin * n_int, own)
        fb.plan_sync(p)
        p.close()
        assert torch.equal(o, own), s
        ref = oracle_beams(np.ascontiguousarray(v[:n_int, :1]), w, *s[:4], 2, 1, n_int)
        assert rel_err_per_beam(o[:1, :1].cpu().numpy(), ref).max() <= TOL_BEAM, s


@pytest.mark.parametrize("npol,n_int", [(1, 65536), (1, 65535), (2, 32768), (64, 1024)])
def test_sums_of_65536_snapshots_are_exact(npol, n_int, monkeypatch):
    """The tensor cores' sums of up to 65536 snapshots, near 2^23 and odd, to the last bit: one feed,
    and two feeds whose beams are |x_0 +- x_1|^2, each as the rounding of the whole number to FP32."""
    monkeypatch.setenv("FFTBF_FP32_PATH", "cov")
    rng = np.random.default_rng(npol + n_int)
    for spread in (0, 1, 4):                                           # all -8, mixed with -7, all signs
        x = np.where(rng.random((n_int, npol, 2, 2)) < 0.9, -8, rng.integers(-8, -7 + spread * 2, (n_int, npol, 2, 2)))
        x[n_int // 2, 0, 0, 0] = -7                                    # one odd term
        for nf in (1, 2):
            y = x[:, :, :nf]
            v = ((y[..., 0] & 15) << 4 | (y[..., 1] & 15)).astype(np.uint8).reshape(n_int, 1, npol, 1, nf)
            got = run(v, None, 1, nf, 1, nf, npol, 1, n_int)[0, 0, 0]
            z = y.astype(np.int64)
            for B in range(nf):
                s = z.sum(axis=2) if B == 0 else z[:, :, 0] - z[:, :, 1]
                assert got[B] == np.float32(int((s ** 2).sum())), (spread, nf, B)
