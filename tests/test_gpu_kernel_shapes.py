"""Launch shapes that depend on sizes, at the sizes where they can go wrong,
against the FP64 oracle."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_0908_3252_gb300 import synth
from tests.helpers import c64, empty_c64, from_dev, rel, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sp():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0908_3252_gb300 import build, spirec
    build.build()
    spirec.load()
    yield spirec


def _stream():
    import torch
    return torch.cuda.current_stream().cuda_stream


# The sum of the contraction's partials: CTA counts that give every shape of
# the sum (76, 25, 9 and 2 owners a tile and more than there are units), one
# and two column tiles, ragged rows and columns.  The operand split and the
# FP32 partial sums are below 1e-5 of the result (4e-7 a phase, at most 384
# accumulation steps between FP32 sums).
@pytest.mark.parametrize("prec", [1, 2])
@pytest.mark.parametrize("ctas", [2, 4, 18, 50, 152])
@pytest.mark.parametrize("N,L", [(5, 40), (37, 2500), (130, 2600)])
def test_partial_sum_shapes(sp, N, L, ctas, prec):
    g = synth.rng(N + ctas)
    kx, ky = synth.uniform_k(L, g)
    y = c64(synth.complex_normal(L, g))
    sp.spirec_tune_clear()
    p = sp.Plan(N, L, 0, prec, _stream())
    try:
        for knob in (sp.SPIREC_KNOB_GRAM_SPLIT, sp.SPIREC_KNOB_ADJOINT_SPLIT):
            sp.spirec_tune_set(knob, N, p.M, prec, L, ctas)
        sp.spirec_set_trajectory(p.h, kx, ky)
        G, x = empty_c64((N, 2 * N - 1)), empty_c64((N, N))
        sp.spirec_gram_dev(p.h, G)
        sp.spirec_adjoint_dev(p.h, to_dev(y), x)
        sp.spirec_sync(p.h)
        assert rel(from_dev(G), O.gram(kx, ky, N)[:, N - 1:].T) < 1e-5
        assert rel(from_dev(x), O.adjoint(kx, ky, y, N)) < 1e-5
    finally:
        p.close()
        sp.spirec_tune_clear()


# The forward contraction: odd and even image sides (the centre row alone or
# paired), one and several chunks of folded rows with one or two 16-deep
# slices in the last, one and two column tiles of uneven width, sample counts
# around the 256 samples of a pair tile and around the pairs of the device.
# Bound as above.
@pytest.mark.parametrize("prec", [1, 2])
@pytest.mark.parametrize("N,L", [(2, 1), (31, 255), (33, 257), (64, 256), (65, 130), (97, 3000), (130, 20000), (257, 513),
                                 (300, 700)])
def test_forward_shapes(sp, N, L, prec):
    g = synth.rng(N + L)
    kx, ky = synth.uniform_k(L, g)
    f = c64(synth.complex_normal((N, N), g))
    with sp.Plan(N, L, 0, prec, _stream(), kx, ky) as p:
        y = empty_c64((L,))
        sp.spirec_forward_dev(p.h, to_dev(f), y)
        sp.spirec_sync(p.h)
        assert rel(from_dev(y), O.forward(kx, ky, f)) < 1e-5


# The FP32 contractions: blocks of 64 and of 128 rows, one to three row and
# column blocks, ragged chunks of 32 samples, one slice, a few, and more than
# there are chunks.  FP32 sums of at most 2500 terms: below 1e-5.
@pytest.mark.parametrize("slices", [0, 1, 3, 100])
@pytest.mark.parametrize("N,L", [(2, 1), (33, 31), (64, 33), (65, 2500), (129, 64), (130, 1000), (200, 500)])
def test_fp32_contraction_shapes(sp, N, L, slices):
    g = synth.rng(N + L)
    kx, ky = synth.uniform_k(L, g)
    y = c64(synth.complex_normal(L, g))
    sp.spirec_tune_clear()
    p = sp.Plan(N, L, 0, 0, _stream())
    try:
        for knob in (sp.SPIREC_KNOB_GRAM_SPLIT, sp.SPIREC_KNOB_ADJOINT_SPLIT):
            sp.spirec_tune_set(knob, N, p.M, 0, L, slices)
        sp.spirec_set_trajectory(p.h, kx, ky)
        G, x = empty_c64((N, 2 * N - 1)), empty_c64((N, N))
        sp.spirec_gram_dev(p.h, G)
        sp.spirec_adjoint_dev(p.h, to_dev(y), x)
        sp.spirec_sync(p.h)
        assert rel(from_dev(G), O.gram(kx, ky, N)[:, N - 1:].T) < 1e-5
        assert rel(from_dev(x), O.adjoint(kx, ky, y, N)) < 1e-5
    finally:
        p.close()
        sp.spirec_tune_clear()


# The kernel spectrum in the caller's layout and T, on grids that are a power
# of two (the transforms' own) and that are not (the spectrum then comes from
# G on the caller's grid, the transforms run on a power of two, smaller than M
# in the last case).  G and FP32 transforms of at most 4096 points: below 1e-5.
@pytest.mark.parametrize("N,M", [(2, 0), (5, 0), (5, 16), (8, 0), (20, 0), (33, 0), (33, 128), (64, 160), (100, 0), (150, 512),
                                 (150, 0), (260, 0), (513, 0), (520, 2048)])
def test_spectrum_and_toeplitz_grids(sp, N, M):
    import torch
    from oracle import toeplitz_cpu as TC
    L = 300
    g = synth.rng(N + M)
    kx, ky = synth.uniform_k(L, g)
    x = c64(synth.complex_normal((N, N), g))
    with sp.Plan(N, L, M, 0, _stream(), kx, ky) as p:
        C = torch.zeros((p.M, p.M), dtype=torch.float32, device="cuda")
        Tx = empty_c64((N, N))
        sp.spirec_kernel_spectrum_dev(p.h, C)
        sp.spirec_toeplitz_dev(p.h, to_dev(x), Tx)
        sp.spirec_sync(p.h)
        G = O.gram(kx, ky, N)
        # spirec_kernel_spectrum_dev divides by M^2
        want = TC.kernel_spectrum(G, N, p.M)
        assert rel(from_dev(C) * float(p.M) ** 2, want) < 1e-5
        Mp = 1 << (2 * N - 1).bit_length()
        assert rel(from_dev(Tx), TC.toeplitz_apply(TC.kernel_spectrum(G, N, Mp), x)) < 1e-5
        if N <= 512 and p.M <= 1024:
            sp.spirec_toeplitz_noalloc(to_dev(x), C, Tx, N, p.M, _stream())
            assert rel(from_dev(Tx), TC.toeplitz_apply(want, x)) < 1e-5


# T on the grids of 2048 and 4096 points (rows and columns split into warp-sized
# transforms, two rows and two columns a sector): odd and even sides, the last
# rows of a block missing, rows that do not start on 16 bytes, sides up to the
# grid's largest.  G by matrix products in 64 bits.
@pytest.mark.parametrize("N,M", [(3, 2048), (6, 4096), (515, 0), (1023, 0), (1024, 0), (1025, 0), (1030, 0), (2047, 0)])
def test_toeplitz_large_grids(sp, N, M):
    import torch
    from oracle import factored as F
    from oracle import toeplitz_cpu as TC
    g = synth.rng(N)
    kx, ky = synth.uniform_k(40, g)
    x = c64(synth.complex_normal((N, N), g))
    with sp.Plan(N, 40, M, 0, _stream(), kx, ky) as p:
        buf = torch.zeros(N * N + 1, dtype=torch.complex64, device="cuda")
        Mp = max(1 << (2 * N - 1).bit_length(), M)
        want = TC.toeplitz_apply(TC.kernel_spectrum(F.gram(kx, ky, N), N, Mp), x)
        for shift in (0, 1):  # the second input starts 8 bytes past a 16-byte boundary
            xd = buf[shift:shift + N * N].view(N, N)
            xd.copy_(to_dev(x))
            Tx = empty_c64((N, N))
            sp.spirec_toeplitz_dev(p.h, xd, Tx)
            sp.spirec_sync(p.h)
            assert rel(from_dev(Tx), want) < 1e-5


# The persistent loop with blocks beyond the rows (fewer row blocks than column
# groups), with one row a block and with a last block of fewer rows, against
# the kernel graph of the same plan's penalty and data (three iterations: the
# FP32 rounding model's distance is below 1e-6, G and D are the same).
@pytest.mark.parametrize("N,M", [(33, 0), (40, 128), (66, 0), (100, 256), (130, 0), (150, 1024), (200, 0), (260, 0), (303, 0),
                                 (400, 0)])
def test_loop_grids(sp, monkeypatch, N, M):
    g = synth.rng(N)
    kx, ky = synth.spiral(N, 4, 700, "variable")
    s = synth.complex_normal(kx.shape[0], g).astype(np.complex64)
    x0 = synth.complex_normal((N, N), g).astype(np.complex64)
    with sp.Plan(N, kx.shape[0], M, 1, _stream(), kx, ky) as p:
        sp.spirec_set_data(p.h, s)
        sp.spirec_set_reg(p.h, 0.05, 0.05, 0.02, 0.1, 0)
        x, J = sp.spirec_solve(p.h, x0, 3, N)
        monkeypatch.setenv("SPIREC_NO_LOOP", "1")
        y, Jy = sp.spirec_solve(p.h, x0, 3, N)
    assert rel(x, y) < 1e-5 and rel(J, Jy) < 1e-5


# The loop's half-warp FFTs (M = 256, 512) at the edges of their ranges: the
# smallest image of each grid, one short of the largest and the largest.
# Distance as above.
@pytest.mark.parametrize("N,M", [(65, 0), (72, 512), (127, 0), (128, 0), (129, 0), (255, 0), (256, 0)])
def test_loop_half_warp_ffts(sp, monkeypatch, N, M):
    g = synth.rng(N)
    kx, ky = synth.spiral(N, 4, 1100, "variable")
    s = synth.complex_normal(kx.shape[0], g).astype(np.complex64)
    with sp.Plan(N, kx.shape[0], M, 1, _stream(), kx, ky) as p:
        sp.spirec_set_data(p.h, s)
        sp.spirec_set_reg(p.h, 0.05, 0.05, 0.02, 0.1, 0)
        x, J = sp.spirec_solve(p.h, None, 3, N)
        monkeypatch.setenv("SPIREC_NO_LOOP", "1")
        y, Jy = sp.spirec_solve(p.h, None, 3, N)
    assert rel(x, y) < 1e-5 and rel(J, Jy) < 1e-5


# T on grids of 256 and 512 points (256-point transforms of half a warp each): the
# smallest and largest sides, odd ones (the last block with fewer rows), sides
# far below the grid's, through a plan and without one.
@pytest.mark.parametrize("N,M", [(2, 256), (9, 512), (65, 0), (127, 0), (128, 0), (129, 0), (255, 0), (256, 0)])
def test_toeplitz_half_warp_grids(sp, N, M):
    import torch
    from oracle import factored as F
    from oracle import toeplitz_cpu as TC
    g = synth.rng(N)
    kx, ky = synth.uniform_k(40, g)
    x = c64(synth.complex_normal((N, N), g))
    with sp.Plan(N, 40, M, 0, _stream(), kx, ky) as p:
        Mp = max(1 << (2 * N - 2).bit_length(), M)
        spec = TC.kernel_spectrum(F.gram(kx, ky, N), N, Mp)
        want = TC.toeplitz_apply(spec, x)
        Tx = empty_c64((N, N))
        sp.spirec_toeplitz_dev(p.h, to_dev(x), Tx)
        sp.spirec_sync(p.h)
        assert rel(from_dev(Tx), want) < 1e-5
        C = torch.from_numpy((spec.real / Mp**2).astype(np.float32)).cuda()  # the library scales its spectrum by 1 / M^2
        sp.spirec_toeplitz_noalloc(to_dev(x), C, Tx, N, Mp, _stream())
        assert rel(from_dev(Tx), want) < 1e-5
