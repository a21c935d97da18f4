"""The direct forms on the tensor cores (direct_mma.cu) where they can go wrong: tile edges and remainders on both
sides, groups of 32 points and accumulation chains with a remainder, one CTA and many per tile, wide and extreme
amplitudes, both planes of the wave.

Tolerance: an entry is good to 1.2e-7 RMS and a term has two (1.7e-7); a chain's truncation leaves up to 3e-7 of its
value, the split's dropped lo lo product 6e-8, and the FP32 additions of n chains sqrt(n / 2) 2^-25 (3.4e-7 at 10^4
points): under 6e-7 together, 1e-6 with the spread of a few hundred sampled pixels.
"""
import numpy as np
import pytest

import oracle
from paper_1309_2734_gb300 import Hologram, _lib, workloads

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

TOL = 1e-6


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1309_2734_gb300.build import build
    build()
    torch.cuda.set_device(0)


def _field(c, form="direct_sfu", wave=False, options=()):
    xyz, amp = torch.from_numpy(c.xyz).cuda(), torch.from_numpy(c.amp).cuda()
    with Hologram(c.width, c.height, c.pitch_m, c.lambda_m, form=form) as h:
        for k, v in options:
            h.set_option(k, v)
        f = h.wave(xyz, amp) if wave else h.point_cloud(xyz, amp)
        h.sync()
        return f.cpu().numpy()


def _sampled(c, n=400):
    rng = np.random.default_rng(c.width + c.n_points)
    cols, rows = rng.integers(0, c.width, n), rng.integers(0, c.height, n)
    cols[:4], rows[:4] = [0, c.width - 1, 0, c.width - 1], [0, 0, c.height - 1, c.height - 1]
    return cols, rows, oracle.field_at(c.pitch_m, c.lambda_m, c.xyz, c.amp, cols, rows)


@pytest.mark.parametrize("w,h", [(1, 1), (127, 65), (128, 64), (129, 257), (260, 130), (2000, 130), (130, 2000),
                                 (1920, 224), (1027, 1025)])
@pytest.mark.parametrize("n", [1, 31, 33, 97, 2050])
def test_tile_and_group_edges(w, h, n):
    c = workloads.random_cloud(9000 + w + n, w, h, n)
    cols, rows, ref = _sampled(c)
    got = _field(c)
    assert oracle.nrms(got[rows, cols], ref) <= TOL
    both = _field(c, wave=True)
    assert oracle.nrms(both[0][rows, cols], ref) <= TOL


@pytest.mark.parametrize("split,ctas", [(1, 0), (3, 0), (0, 1), (0, 5), (0, 700)])
def test_cta_counts(split, ctas):
    c = workloads.random_cloud(9100, 300, 200, 1500)
    cols, rows, ref = _sampled(c)
    got = _field(c, options=[(_lib.CGH_OPT_POINT_SPLIT, split), (_lib.CGH_OPT_DIRECT_CTAS, ctas)])
    assert oracle.nrms(got[rows, cols], ref) <= TOL


@pytest.mark.parametrize("lo,hi", [(-6.0, 0.0), (29.0, 30.0), (-30.0, -29.0), (-12.0, 3.0)])
def test_amplitude_ranges(lo, hi):
    """Amplitudes over many decades, and near the ends of single precision; either sign."""
    c = workloads.random_cloud(9200, 200, 150, 3000)
    rng = np.random.default_rng(1)
    c.amp = (10.0 ** rng.uniform(lo, hi, c.n_points) * rng.choice([-1.0, 1.0], c.n_points)).astype(np.float32)
    cols, rows, ref = _sampled(c)
    for form in ("direct_sfu", "direct_accurate"):
        assert oracle.nrms(_field(c, form)[rows, cols] * 10.0 ** -hi, ref * 10.0 ** -hi) <= TOL


def test_zero_amplitudes():
    c = workloads.random_cloud(9300, 200, 150, 100)
    c.amp[:] = 0.0
    assert not _field(c).any()


@pytest.mark.parametrize("extra", [False, True])
@pytest.mark.parametrize("w,h,n", [(256, 256, 9), (256, 256, 20), (256, 256, 32), (256, 256, 300), (256, 256, 2048), (640, 64, 1024),
                                   (128, 128, 1000), (1283, 717, 33)])
def test_accurate_form_is_no_coarser_than_the_simt_kernel(w, h, n, extra):
    # the same cloud by the SIMT kernel with the cosine polynomial (a pinned thread block): its error is the bound, and
    # 5 % for the draw of clouds and pixels
    mma = simt = 0.0
    for seed in range(3):
        c = workloads.random_cloud(9700 + 10 * n + seed, w, h, n)
        rng = np.random.default_rng(seed)
        cols, rows = rng.integers(0, w, 20000), rng.integers(0, h, 20000)
        tilt = (0.011, -0.007, 0.6) if extra else (0.0, 0.0, 0.0)
        ref = oracle.model_wave_at(1 if extra else 0, c.pitch_m, c.lambda_m, c.xyz, c.amp, cols, rows, reference=tilt).real
        xyz, amp = torch.from_numpy(c.xyz).cuda(), torch.from_numpy(c.amp).cuda()
        err = []
        for shape in (0, 5):
            with Hologram(w, h, c.pitch_m, c.lambda_m, form="direct_accurate") as hg:
                hg.set_option(_lib.CGH_OPT_DIRECT_SHAPE, shape)
                if extra:
                    hg.set_phase_model("fresnel_piston")
                    hg.set_reference(*tilt)
                f = hg.point_cloud(xyz, amp)
                hg.sync()
                err.append(oracle.nrms(f.cpu().numpy()[rows, cols], ref))
        mma, simt = mma + err[0] ** 2, simt + err[1] ** 2
    assert mma <= simt * 1.05 ** 2, (mma ** 0.5, simt ** 0.5)


MMA, SIMT = 1.5e-6, 1e-5   # the SIMT kernel's tolerance is that of its own tests


@pytest.mark.parametrize("w,h,n,z,tol", [
    (129, 257, 15, (0.3, 0.5), MMA), (300, 200, 17, (0.2, 0.3), MMA), (1920, 224, 130, (0.4, 1.0), MMA), (130, 2000, 33, (0.5, 0.9), MMA),
    (1920, 1080, 65, (0.3, 1.0), MMA),      # the widest tile
    (1920, 1080, 65, (0.2, 0.25), MMA),     # corner points beyond the tiles' range of the remainder: the SIMT kernel
    (1920, 1080, 65, (0.05, 0.1), SIMT),     # beyond its bound: the SIMT kernel
    (1920, 1080, 65, (0.005, 1.0), SIMT),    # a close point among far ones: the SIMT kernel
    (1000, 600, 2050, (0.25, 0.6), MMA),
])
@pytest.mark.parametrize("ref", [(0.0, 0.0, 0.0), (0.01, -0.02, 0.4)])
def test_spherical(w, h, n, z, tol, ref):
    """The spherical model on either side of the bounds that pick its kernel.  The tensor-core form adds to the errors
    above at most 4e-7 of a term for the third order and 5e-7 for the FP16 products at the largest cross phase."""
    c = workloads.random_cloud(9400 + w + n, w, h, n, z)
    rng = np.random.default_rng(3)
    cols, rows = rng.integers(0, w, 300), rng.integers(0, h, 300)
    cols[:4], rows[:4] = [0, w - 1, 0, w - 1], [0, 0, h - 1, h - 1]
    want = oracle.model_wave_at(2, c.pitch_m, c.lambda_m, c.xyz, c.amp, cols, rows, reference=ref).real
    xyz, amp = torch.from_numpy(c.xyz).cuda(), torch.from_numpy(c.amp).cuda()
    with Hologram(w, h, c.pitch_m, c.lambda_m, form="direct_sfu") as hg:
        hg.set_phase_model("spherical")
        hg.set_reference(*ref)
        f = hg.point_cloud(xyz, amp)
        hg.sync()
        got = f.cpu().numpy()
    assert oracle.nrms(got[rows, cols], want) <= tol


def _sph_bound(c):
    # the point preparation's bounds: the largest cross phase over tiles of 128 x 256 pixels (rad; a tile of 128 x bn takes
    # up to 0.05 x 256 / bn) and the range of the remainder along a side (turns; up to 0.45)
    x, y, z = c.xyz.astype(np.float64).T
    q, Z = (c.pitch_m / z) ** 2, z / c.lambda_m
    cx = np.maximum(abs(x), abs(c.width - 1 - x)) + 128
    cy = np.maximum(abs(y), abs(c.height - 1 - y)) + 128
    x64, x128, y64, y128 = (q * (2 * s * v + s * s) for v in (cx, cy) for s in (64, 128))
    w = np.maximum(x128, y128)
    return ((np.pi / 2 * Z * np.maximum(x64 * y128, x128 * y64)).max(),
            (0.25 * Z * ((cx ** 2 + cy ** 2) * q + w) * w).max())


@pytest.mark.parametrize("w,h,n,z,lo,hi", [
    (1920, 1080, 600, (0.28, 0.281), 0.045, 0.05),   # the widest tile at nearly the largest cross phase it takes
    (1920, 1080, 600, (0.25, 0.251), 0.05, 0.1),     # the narrowest, after the widest has declined
    (1000, 600, 2050, (0.145, 0.146), 0.1, 0.2),     # only the narrowest takes it
    (640, 360, 700, (0.0985, 0.099), 0.16, 0.2),     # nearly its largest cross phase
    (300, 260, 65, (0.08, 0.081), 0.16, 0.2),
])
def test_spherical_tiles_near_their_bounds(w, h, n, z, lo, hi):
    # Tolerance: the SIMT kernel's measured 9.5e-7 at most on such clouds, and the draw of pixels; the third order left out
    # is 4e-7 of a term at the largest cross phase
    c = workloads.random_cloud(9450 + w, w, h, n, z)
    c.xyz[0] = (0.0, 0.0, z[0])
    phase, spread = _sph_bound(c)
    assert lo < phase <= hi and spread <= 0.45
    rng = np.random.default_rng(4)
    cols, rows = rng.integers(0, w, 3000), rng.integers(0, h, 3000)
    want = oracle.model_wave_at(2, c.pitch_m, c.lambda_m, c.xyz, c.amp, cols, rows).real
    xyz, amp = torch.from_numpy(c.xyz).cuda(), torch.from_numpy(c.amp).cuda()
    with Hologram(w, h, c.pitch_m, c.lambda_m, form="direct_sfu") as hg:
        hg.set_phase_model("spherical")
        f = hg.point_cloud(xyz, amp)
        hg.sync()
    assert oracle.nrms(f.cpu().numpy()[rows, cols], want) <= 1e-6


@pytest.mark.parametrize("n", [1, 63, 64, 65, 256, 257, 1500])
def test_largest_amplitude_in_any_block(n):
    # max |A| comes from one value per 64 points: wherever the largest stands, the scaled entries stay in FP16's range
    c = workloads.random_cloud(77 + n, 200, 150, n)
    cols, rows, _ = _sampled(c)
    for at in sorted({0, n // 2, min(n, 64) - 1, n - 1}):
        amp = c.amp.copy()
        amp[at] = -3e8
        ref = oracle.field_at(c.pitch_m, c.lambda_m, c.xyz, amp, cols, rows)
        for wave in (False, True):
            with Hologram(200, 150, c.pitch_m, c.lambda_m, form="direct_sfu") as h:
                x, a = torch.from_numpy(c.xyz).cuda(), torch.from_numpy(amp).cuda()
                f = h.wave(x, a)[0] if wave else h.point_cloud(x, a)
                h.sync()
                assert oracle.nrms(f.cpu().numpy()[rows, cols], ref) <= TOL


@pytest.mark.parametrize("w,h", [(130, 67), (67, 132)])
@pytest.mark.parametrize("n", [20480, 20481, 41000])
def test_points_beyond_one_launch(w, h, n):
    # one CTA takes every point of a tile: beyond 20480 points a second launch adds to the first one's output
    c = workloads.random_cloud(500 + n + w, w, h, n)
    cols, rows, ref = _sampled(c)
    for wave in (False, True):
        f = _field(c, wave=wave, options=((_lib.CGH_OPT_POINT_SPLIT, 1),))
        assert oracle.nrms((f[0] if wave else f)[rows, cols], ref) <= TOL


def test_point_split_beyond_the_point_tiles():
    # chunks of 256 points at least, however many are asked for: 30 tiles x 391 slots of 2 x 131,072 bytes (3.1 GB), a
    # quarter more reserved, and not 3125 for each of them
    c = workloads.random_cloud(9110, 1280, 720, 100000)
    cols, rows, ref = _sampled(c, 100)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    xyz, amp = torch.from_numpy(c.xyz).cuda(), torch.from_numpy(c.amp).cuda()
    with Hologram(c.width, c.height, c.pitch_m, c.lambda_m, form="direct_sfu") as h:
        h.set_option(_lib.CGH_OPT_POINT_SPLIT, 4096)
        f = h.point_cloud(xyz, amp)
        h.sync()
        assert free - torch.cuda.mem_get_info()[0] < 6 << 30
    assert oracle.nrms(f.cpu().numpy()[rows, cols], ref) <= TOL


def test_launches_share_the_points_evenly():
    # 12 tiles of 480,943 groups on 13 CTAs: 694 launches of 693 groups would leave the last one a single group.  To the tolerance
    # above come the launches' additions to the output, sqrt(694 / 2) 2^-25 = 5.6e-7
    c = workloads.random_cloud(611, 384, 896, 15390145)
    cols, rows, ref = _sampled(c, 24)
    got = _field(c, options=[(_lib.CGH_OPT_DIRECT_CTAS, 13)])
    assert oracle.nrms(got[rows, cols], ref) <= TOL + 6e-7


@pytest.mark.parametrize("what", ["cloud", "accurate", "wave", "spherical", "spherical_close", "gemm_wave", "launches", "gemm", "gemm_pair",
                                  "gemm_chunks"])
def test_captured_and_replayed(what):
    # dependent launches and the kernels' own clears inside a CUDA graph: a replay on new amplitudes gives the bits of
    # a plain call
    # (spherical_close: every tensor-core launch declines, the SIMT kernel after them takes the cloud)
    c = workloads.random_cloud(811, 300, 200, 21000 if what == "launches" else 900,
                               (0.005, 0.01) if what == "spherical_close" else (0.3, 1.0))
    xyz, amp = torch.from_numpy(c.xyz).cuda(), torch.from_numpy(c.amp).cuda()
    form = {"accurate": "direct_accurate", "gemm_wave": "gemm_split16", "gemm": "gemm_f16", "gemm_pair": "gemm_split16",
            "gemm_chunks": "gemm_bf16"}.get(what, "direct_sfu")
    s = torch.cuda.Stream()
    with Hologram(300, 200, c.pitch_m, c.lambda_m, form=form, stream=s) as h:
        if "spherical" in what:
            h.set_phase_model("spherical")
        if what == "gemm_pair":
            h.set_option(_lib.CGH_OPT_GEMM_PAIR, 1)
        if what == "gemm_chunks":
            h.set_option(_lib.CGH_OPT_FACTOR_BUDGET_MB, 1)
        if what == "launches":
            h.set_option(_lib.CGH_OPT_POINT_SPLIT, 1)

        def call():
            if "wave" in what:
                w = h.wave(xyz, amp)
                return w, h.kinoform8(w)
            f = h.point_cloud(xyz, amp)
            return f, h.quantize8(f)
        s.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(s):
            call()
        h.sync()
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            f, q = call()
        amp.mul_(-3.0)
        torch.cuda.synchronize()
        g.replay()
        torch.cuda.synchronize()
        got = f.clone(), q.clone()
        with torch.cuda.stream(s):
            want = call()
        h.sync()
        torch.cuda.synchronize()
        assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])
