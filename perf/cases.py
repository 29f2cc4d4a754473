"""The work that users of the SAR compression library have it do, as cases to measure.

A case is a dict of plain values; its "kind" says which public entry point one pass goes through:

  scene   sar_rda_process_oop: an echo [n_az][n_range] to its image (FP32 or split precision, image range-major or azimuth-major)
  host    sar_rda_process_host_n: echoes and images in pinned host memory
  full    sar_rda_full: the processor with range cell migration correction
  lines   sar_range_compress_oop: the compression of every line, alone
  fft     sar_fft_lines: the plain transform of every line, forward or inverse
  batch   sar_batch_run: strips of mixed sizes in one launch
  serve   sar_server_run: a closed loop of requests of mixed scene sizes

Echoes are point targets (linear FM chirps along both axes) in white Gaussian noise, the model of the paper's Sec. V-A, made on the
device from the seed; filters are the conjugate chirp spectra, evaluated in 64 bits.
"""
import math
import random

import torch

import paper_2604_03585_gb300 as sar

DEV = "cuda"
C64, C128 = torch.complex64, torch.complex128
GEOMETRY = dict(kappa=10.0, v_s=0.3, r_near=4000.0)   # migration of up to ~115 bins at the band edge of 4096 bins
MOST_SAMPLES = 1 << 27                                # of a drawn case: no more than the largest listed scene


def listed():
    return [
        # the smallest scene of the workload list: two launches, latency counts
        dict(name="scene_256", kind="scene", n_az=256, n_range=256, precision=0, az_major=False),
        # the benchmark scene of the paper, FP32
        dict(name="scene_4096", kind="scene", n_az=4096, n_range=4096, precision=0, az_major=False),
        # the same scene by split-precision products on the tensor cores
        dict(name="scene_4096_fp16x2", kind="scene", n_az=4096, n_range=4096, precision=1, az_major=False),
        # the longest lines of one block in both directions: the largest scene of the serving mix, half of it
        dict(name="scene_8192x16384", kind="scene", n_az=8192, n_range=16384, precision=0, az_major=False),
        # a recording of a length that nobody rounded to a power of two, prime factors 2, 3 and 5
        dict(name="scene_3000x5000", kind="scene", n_az=3000, n_range=5000, precision=0, az_major=False),
        # odd sizes with large prime factors, the image in the echo's own orientation
        dict(name="scene_1021x3001_az", kind="scene", n_az=1021, n_range=3001, precision=0, az_major=True),
        # the full processor: azimuth transform, migration correction, range-dependent azimuth filter
        dict(name="full_4096", kind="full", n_az=4096, n_range=4096),
        # host to host: two scenes of the benchmark's size in one call, copies in and out included
        dict(name="host_4096_x2", kind="host", n_az=4096, n_range=4096, scenes=2),
        # range lines longer than one block holds
        dict(name="lines_512x65536", kind="lines", n_az=512, n_range=65536),
        # the transform alone, as used for filter design and spectra
        dict(name="fft_inv_4099x8192", kind="fft", n=8192, lines=4099, inverse=True),
        # a ragged batch: range lengths 1024 ... 16384, 256 ... 4096 azimuth lines each, one launch
        dict(name="batch_16", kind="batch", strips=16, sizes=4, least_range=1024, most_range=16384, most_az=4096, flags=0),
        # saturated serving: scenes of 2048, 4096 and 8192 squared, 70 / 25 / 5 %, each image delivered
        dict(name="serve_16", kind="serve", requests=16, largest=8192, size_priority=False),
    ]


# --- more cases of the same ranges -------------------------------------------------------------------------------------------------

def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _pow2(rng, lo, hi):
    return 1 << rng.randint(lo.bit_length() - 1, hi.bit_length() - 1)


def _smooth(n):
    for p in (2, 3, 5, 7):
        while n % p == 0:
            n //= p
    return n == 1


def _length(rng, lo=64, hi=8192):
    """A line length as scenes have it: mostly a power of two, a length with small prime factors, or any."""
    what = rng.random()
    if what < 0.5:
        return _pow2(rng, 256, 16384)
    n = _log(rng, lo, hi)
    if what < 0.8:
        while not _smooth(n):
            n -= 1
    return n


def draw(rng):
    kind = rng.choices(["scene", "full", "lines", "fft", "batch", "serve", "host"], [8, 2, 3, 2, 3, 2, 1])[0]
    if kind == "scene":
        if rng.random() < 0.15:
            return dict(kind=kind, n_az=rng.choice([256, 4096]), n_range=rng.choice([256, 4096]), precision=rng.randint(1, 3),
                        az_major=rng.random() < 0.25)
        n_az, n_range = _length(rng), _length(rng)
        if n_az * n_range > MOST_SAMPLES:
            n_az = 8192
        return dict(kind=kind, n_az=n_az, n_range=n_range, precision=0, az_major=rng.random() < 0.25)
    if kind == "full":
        return dict(kind=kind, n_az=_pow2(rng, 256, 8192), n_range=min(_length(rng, 256), 8192))
    if kind == "lines":
        n = _pow2(rng, 32768, 131072) if rng.random() < 0.5 else _length(rng)
        return dict(kind=kind, n_az=_log(rng, 2, max(2, min(8192, MOST_SAMPLES // n))), n_range=n)
    if kind == "fft":
        n = _pow2(rng, 32768, 131072) if rng.random() < 0.2 else _length(rng)
        return dict(kind=kind, n=n, lines=_log(rng, 1, MOST_SAMPLES // (2 * n)), inverse=rng.random() < 0.5)
    if kind == "batch":
        return dict(kind=kind, strips=rng.randint(2, 16), sizes=rng.randint(0, 1 << 20), least_range=rng.choice([256, 1024]),
                    most_range=rng.choice([4096, 8192, 16384]), most_az=_log(rng, 512, 4096), flags=rng.choice([0, 0, 0, 2]))
    if kind == "serve":
        return dict(kind=kind, requests=rng.randint(6, 16), largest=_pow2(rng, 1024, 8192), size_priority=rng.random() < 0.5)
    return dict(kind=kind, n_az=_pow2(rng, 512, 4096), n_range=_pow2(rng, 512, 4096), scenes=rng.randint(1, 3))


# --- inputs ------------------------------------------------------------------------------------------------------------------------

def _pow2_at_least(n):
    return max(256, 1 << (n - 1).bit_length())


def _strip_sizes(case):
    """[(n_range, n_az), ...]: range lengths powers of two, azimuth counts uniform from 256 (fewer where the batch is small)."""
    r = random.Random(case["sizes"])
    return [(_pow2(r, case["least_range"], case["most_range"]), r.randint(256, case["most_az"])) for _ in range(case["strips"])]


def _serve_classes(case):
    """[(size, requests), ...]: 70 / 25 / 5 % of the smallest, the middle and the largest scenes, at least one of each."""
    n, top = case["requests"], case["largest"]
    big = max(1, round(0.05 * n))
    mid = max(1, round(0.25 * n))
    return [(top // 4, n - mid - big), (top // 2, mid), (top, big)]


def _chirps(n_range, l_az):
    """((samples, time-bandwidth), ...) of the range and the azimuth chirp, scaled to the lines."""
    nr, na = max(2, n_range // 8), max(2, l_az // 4)
    return (nr, max(1.0, nr / 2)), (na, max(1.0, na / 8))


def _chirp(n_c, tbp, dtype=C128):
    m = torch.arange(n_c, dtype=torch.float64, device=DEV) - n_c // 2
    half = torch.remainder(tbp * m * m / float(n_c * n_c), 2.0) * math.pi
    return torch.polar(torch.ones_like(half), half).to(dtype)


def _spectrum(n, n_c, tbp):
    """conj(FFT_n(chirp centred on index 0)), evaluated in 64 bits and rounded once."""
    line = torch.zeros(n, dtype=C128, device=DEV)
    line[:n_c] = _chirp(n_c, tbp)
    return torch.fft.fft(torch.roll(line, -(n_c // 2))).conj().resolve_conj().to(C64)


def _noise(shape, snr_db, gen):
    return torch.randn(shape, dtype=C64, device=DEV, generator=gen) * 10.0 ** (-snr_db / 20.0)


def _generator(seed):
    return torch.Generator(device=DEV).manual_seed(seed % (1 << 62))


def _targets(seed, n_az, n_range):
    r = random.Random(seed)
    return [(r.randrange(n_az), r.randrange(n_range)) for _ in range(1 if n_az * n_range <= 1 << 17 else 5)]


def _echo(n_az, n_range, l_az, seed):
    """Point targets, chirps along both axes (wrapping), noise at 10 dB: complex64 [n_az][n_range] on the device."""
    (ncr, tr), (nca, ta) = _chirps(n_range, l_az)
    nca = min(nca, n_az)
    rows = torch.zeros((0, n_az), dtype=C64, device=DEV)
    cols = torch.zeros((0, n_range), dtype=C64, device=DEV)
    for a0, r0 in _targets(seed, n_az, n_range):
        a, r = torch.zeros((1, n_az), dtype=C64, device=DEV), torch.zeros((1, n_range), dtype=C64, device=DEV)
        a[0, :nca], r[0, :ncr] = _chirp(nca, ta, C64), _chirp(ncr, tr, C64)
        rows = torch.cat([rows, torch.roll(a, a0 - nca // 2, 1)])
        cols = torch.cat([cols, torch.roll(r, r0 - ncr // 2, 1)])
    return torch.addmm(_noise((n_az, n_range), 10.0, _generator(seed)), rows.t(), cols)


def _echo_migrating(n_az, n_range, seed):
    """Targets that follow the hyperbolic range history over an aperture of a quarter of the lines, noise at 10 dB."""
    (n_c, tbp), _ = _chirps(n_range, n_az)
    g = GEOMETRY
    out = _noise((n_az, n_range), 10.0, _generator(seed))
    for a0, n0 in _targets(seed, n_az, n_range):
        m = torch.arange(max(0, a0 - n_az // 8), min(n_az, a0 + n_az // 8), device=DEV)
        r = torch.sqrt((g["r_near"] + n0) ** 2 + (g["v_s"] * (m - a0).double()) ** 2)
        late = r - g["r_near"]
        col = torch.floor(late).long()[:, None] + torch.arange(-(n_c // 2), n_c - n_c // 2 + 1, device=DEV)[None, :]
        t = col.double() - late[:, None]
        phase = math.pi * tbp / (n_c * n_c) * t * t - 2 * math.pi * torch.remainder(g["kappa"] * r, 1.0)[:, None]
        on = (t >= -(n_c // 2)) & (t < n_c - n_c // 2) & (col >= 0) & (col < n_range)
        value = torch.polar(on.double(), phase).to(C64)
        out[m] = out[m].scatter_add(1, col.clamp(0, n_range - 1), value)
    return out


def _filters(n_range, l_az):
    (ncr, tr), (nca, ta) = _chirps(n_range, l_az)
    return _spectrum(n_range, ncr, tr), _spectrum(l_az, nca, ta)


def _inputs(case, seed):
    """Everything of a case that the seed decides, on the device."""
    kind = case["kind"]
    if kind == "fft":
        return torch.randn((case["lines"], case["n"]), dtype=C64, device=DEV, generator=_generator(seed))
    if kind == "batch":
        return [_echo(a, r, _pow2_at_least(a), seed + 7919 * i) for i, (r, a) in enumerate(_strip_sizes(case))]
    if kind == "serve":
        return [_echo(n, n, n, seed + 7919 * i) for i, (n, _) in enumerate(_serve_classes(case))]
    if kind == "full":
        return _echo_migrating(case["n_az"], case["n_range"], seed)
    if kind == "host":
        return [_echo(case["n_az"], case["n_range"], case["n_az"], seed + 7919 * i) for i in range(case["scenes"])]
    return _echo(case["n_az"], case["n_range"], case["n_az"], seed)


def _serve_order(case, seed):
    order = [k for k, (_, count) in enumerate(_serve_classes(case)) for _ in range(count)]
    random.Random(seed).shuffle(order)
    return order


def _like(n_range, n_az, az_major=False):
    return torch.empty((n_az, n_range) if az_major else (n_range, n_az), dtype=C64, device=DEV)


def prepare(case, seed):
    kind, x = case["kind"], _inputs(case, seed)
    s = dict(case=case, kind=kind, x=x)
    if kind == "fft":
        s["out"] = torch.empty_like(x)
    elif kind == "batch":
        spectra, strips = {}, []
        for (r, a), raw in zip(_strip_sizes(case), x):
            L = _pow2_at_least(a)
            for axis, n in (("range", r), ("az", L)):
                if (axis, n) not in spectra:
                    spectra[axis, n] = _filters(n, n)[axis == "az"]
            strips.append(dict(n_range=r, n_az=a, raw=raw, image=_like(r, a), range_spectrum=spectra["range", r],
                               az_spectrum=spectra["az", L]))
        s["out"], s["keep"] = [st["image"] for st in strips], spectra
        s["batch"] = sar.sar_batch_create(strips, flags=case["flags"])
    elif kind == "serve":
        classes, s["requests"] = [], []
        for (n, _), raw in zip(_serve_classes(case), x):
            hr, ha = _filters(n, n)
            classes.append(dict(n_range=n, n_az=n, pool=raw, range_spectrum=hr, az_spectrum=ha))
        for k in _serve_order(case, seed):
            image = _like(classes[k]["n_range"], classes[k]["n_az"])
            s["requests"].append((0.0, k, image))
        s["out"] = [r[2] for r in sorted(s["requests"], key=lambda r: r[1])]   # by class: the order of arrival is the seed's
        s["server"] = sar.sar_server_create(classes, hbm_budget_bytes=16 << 30, max_inflight=8, size_priority=case["size_priority"])
    else:
        n_az, n_range = case["n_az"], case["n_range"]
        hr, ha = _filters(n_range, n_az)
        flags = sar.SAR_PLAN_OUT_AZ_MAJOR if case.get("az_major") else 0
        s["plan"] = sar.sar_plan_create(n_range, n_az, hr, ha, precision=case.get("precision", 0), flags=flags)
        if kind == "host":
            s["x"] = [raw.cpu().pin_memory() for raw in x]
            s["out"] = [torch.empty((n_range, n_az), dtype=C64, pin_memory=True) for _ in x]
        elif kind == "lines":
            s["out"] = _like(n_range, n_az, True)
        else:
            s["out"], s["work"] = _like(n_range, n_az, case.get("az_major", False)), _like(n_range, n_az)
            if kind == "full":
                sar.sar_plan_set_geometry(s["plan"], GEOMETRY["kappa"], GEOMETRY["v_s"], GEOMETRY["r_near"], 16)
    return s


def run(s):
    kind = s["kind"]
    if kind == "scene":
        sar.sar_rda_process_oop(s["plan"], s["x"], s["work"], s["out"])
    elif kind == "full":
        sar.sar_rda_full(s["plan"], s["x"], s["work"], s["out"])
    elif kind == "lines":
        sar.sar_range_compress_oop(s["plan"], s["x"], s["out"])
    elif kind == "fft":
        sar.sar_fft_lines(s["case"]["n"], s["case"]["lines"], s["x"], s["out"], inverse=s["case"]["inverse"])
    elif kind == "batch":
        sar.sar_batch_run(s["batch"])
    elif kind == "serve":
        sar.sar_server_run(s["server"], s["requests"], mode=sar.SAR_SERVE_CLOSED_LOOP)
    else:
        sar.sar_rda_process_host_n(s["plan"], s["x"], s["out"])
    return s["out"]


# --- what the work is --------------------------------------------------------------------------------------------------------------

def work(case):
    """Each input read once and each output written once (8 bytes per sample each); 5 n log2 n per transform of n, 6 per multiply."""
    def fft(n, lines):
        return 5.0 * n * math.log2(n) * lines

    def scene(n_az, n_range, l_az=None):
        l_az = l_az or n_az
        return 2 * fft(n_range, n_az) + 2 * fft(l_az, n_range) + 6.0 * (n_range * n_az + l_az * n_range)

    kind = case["kind"]
    if kind == "fft":
        return dict(bytes=16 * case["n"] * case["lines"], flops=fft(case["n"], case["lines"]))
    if kind == "batch":
        sizes = _strip_sizes(case)
        return dict(bytes=sum(16 * r * a for r, a in sizes), flops=sum(scene(a, r, _pow2_at_least(a)) for r, a in sizes))
    if kind == "serve":
        classes = _serve_classes(case)
        return dict(bytes=sum(16 * n * n * k for n, k in classes), flops=sum(scene(n, n) * k for n, k in classes))
    n_az, n_range = case["n_az"], case["n_range"]
    scenes = case.get("scenes", 1)
    if kind == "lines":
        return dict(bytes=16 * n_az * n_range, flops=(2 * fft(n_range, n_az) + 6.0 * n_az * n_range))
    # the migration correction: 16 complex-by-real taps and about 40 operations for a weight set, per sample
    extra = 104.0 * n_az * n_range if kind == "full" else 0.0
    return dict(bytes=16 * n_az * n_range * scenes, flops=(scene(n_az, n_range) + extra) * scenes)


def tolerance(case):
    # measured against exact(): FP32 1.3e-7 ... 3.8e-7 (the longest lines); split products 2.8e-6 (FP16 in two parts), 8.2e-6 (BF16 in
    # two), 3.2e-6 (BF16 in three); single values at most 1.3e-4 and 1e-4 (FP16) of the image's root mean square; four times that
    split = {1: 1.2e-5, 2: 3.3e-5, 3: 1.3e-5}.get(case.get("precision", 0))
    return {"rel": split, "max": 1e-3} if split else {"rel": 1.5e-6, "max": 5e-4}


# --- the same in 64 bits -----------------------------------------------------------------------------------------------------------

def _compress(x, spectrum, length=None):
    n = x.shape[-1]
    y = torch.fft.fft(x, n=length)
    y *= spectrum.to(C128)
    return torch.fft.ifft(y)[..., :n]


def _image(raw, hr, ha, az_major=False):
    y = _compress(raw.to(C128), hr).t().contiguous()
    y = _compress(y, ha, ha.numel())
    return (y.t() if az_major else y).contiguous()


def _image_full(raw, hr):
    n_az, n_range = raw.shape
    g = GEOMETRY
    y = torch.fft.fft(_compress(raw.to(C128), hr).t().contiguous())
    j = torch.arange(n_az, device=DEV, dtype=torch.float64)
    f = torch.where(j < n_az / 2, j, j - n_az) / n_az
    d = torch.sqrt(1.0 - (f / (g["kappa"] * g["v_s"])) ** 2)
    n = torch.arange(n_range, device=DEV, dtype=torch.float64)[:, None]
    src = n + (g["r_near"] + n) * (1.0 / d - 1.0)[None, :]
    k0 = torch.floor(src)
    z = torch.zeros_like(y)
    for t in range(-7, 9):
        k = k0 + t
        x = src - k
        h = torch.sinc(x) * 0.5 * (1.0 + torch.cos(2 * math.pi * x / 16))
        h = torch.where((k >= 0) & (k < n_range), h, torch.zeros_like(h))
        z += h * torch.gather(y, 0, k.clamp(0, n_range - 1).long())
    cycles = torch.remainder(g["kappa"] * (g["r_near"] + n) * d[None, :], 1.0)
    return torch.fft.ifft(z * torch.polar(torch.ones_like(cycles), 2 * math.pi * cycles))


def exact(case, seed):
    kind, x = case["kind"], _inputs(case, seed)
    if kind == "fft":
        x = x.to(C128)
        return torch.fft.ifft(x, norm="forward") if case["inverse"] else torch.fft.fft(x)
    if kind == "batch":
        out = []
        for (r, a), raw in zip(_strip_sizes(case), x):
            L = _pow2_at_least(a)
            out.append(_image(raw, _filters(r, r)[0], _filters(L, L)[1]))
        return out
    if kind == "serve":
        images = [_image(raw, *_filters(raw.shape[0], raw.shape[0])) for raw in x]
        return [images[k] for k in sorted(_serve_order(case, seed))]
    hr, ha = _filters(case["n_range"], case["n_az"])
    if kind == "lines":
        return _compress(x.to(C128), hr)
    if kind == "full":
        return _image_full(x, hr)
    if kind == "host":
        return [_image(raw, hr, ha).cpu() for raw in x]
    return _image(x, hr, ha, case["az_major"])
