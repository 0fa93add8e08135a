"""Synthesis over every transform length, ragged point counts and pulse groupings, against the
discrete Fourier sum of Eq. (inverseFourier) in FP64 (numpy).

Tolerances: a transform of n samples makes log2 n additions and rotations of relative error a few eps
each, so its relative 2-norm error is below 4 eps log2 n: 12 x 4 x 2^-24 = 2.9e-6 in FP32 and
12 x 4 x 2^-53 = 5.4e-15 in FP64, plus eps of the result (and 2 eps of the reference)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _reference(T, midx, S, Nt):
    H = np.zeros((S.shape[0], T.shape[1], Nt // 2 + 1), complex)
    H[:, :, midx] = S[:, None, midx] * T.T[None]
    return np.fft.irfft(np.conj(H), n=Nt, axis=2)


def _case(Nt, M, P, seed, picked):
    rng = np.random.default_rng(seed)
    nm = Nt // 2 + 1
    midx = np.sort(rng.choice(nm, max(1, nm // 3), replace=False)) if picked else np.arange(nm)
    T = rng.standard_normal((len(midx), M)) + 1j * rng.standard_normal((len(midx), M))
    S = rng.standard_normal((P, nm)) + 1j * rng.standard_normal((P, nm))
    return T, midx.astype(np.int64), S


@pytest.mark.parametrize("f32", [False, True])
@pytest.mark.parametrize("Nt", [2 ** i for i in range(1, 13)])
def test_synthesis_over_lengths(Nt, f32):
    import torch
    from paper_1706_07919_gb300 import Solver
    from paper_1706_07919_gb300 import binding as B

    sol = Solver(0)
    dt = torch.float32 if f32 else torch.float64
    eps = 2.0 ** -24 if f32 else 2.0 ** -53
    # one point; ragged groups of points; enough points that a CTA keeps them for all pulses
    for M, P, picked in ((1, 1, False), (3, 2, True), (41, 5, False), (4 * 152 * max(1, 8192 // Nt) + 1, 2, True)):
        T, midx, S = _case(Nt, M, P, Nt + M, picked)
        Td, Sd = torch.tensor(T, device="cuda:0"), torch.tensor(S, device="cuda:0")
        ref = _reference(T, midx, S, Nt)
        tol = (4 * np.log2(Nt) + 3) * eps
        got = sol.synthesize(Td, midx, Sd, Nt, dt).cpu().numpy()
        assert np.linalg.norm(got - ref) <= tol * np.linalg.norm(ref), (M, P)
        out = torch.empty((P, M, Nt), dtype=dt, device="cuda:0")
        B.bie_synthesize_noalloc(Td, midx, Sd, Nt, out, 1 if f32 else 0)
        assert np.linalg.norm(out.cpu().numpy() - ref) <= tol * np.linalg.norm(ref), (M, P)
    sol.close()


def test_fp32_synthesis_takes_values_outside_fp32():
    """Field spectra below and above FP32's range with pulses that bring the product back into it."""
    import torch
    from paper_1706_07919_gb300 import Solver

    sol = Solver(0)
    T, midx, S = _case(64, 5, 3, 1, False)
    for scale in (1e-60, 1e-33, 1e33, 1e60):
        got = sol.synthesize(torch.tensor(T * scale, device="cuda:0"), midx, torch.tensor(S / scale, device="cuda:0"), 64,
                             torch.float32).cpu().numpy()
        ref = _reference(T, midx, S, 64)
        assert np.linalg.norm(got - ref) <= 27 * 2.0 ** -24 * np.linalg.norm(ref)
    sol.close()


def test_many_pulses_take_bounded_scratch():
    """FP32 output of 6000 pulses of 4096 samples: the device memory a context takes for their split spectra
    stays below 64 MB (197 MB for all of them at once), and a pulse's signal is its own."""
    import torch
    from paper_1706_07919_gb300 import Solver

    Nt, P = 4096, 6000
    g = torch.Generator("cuda:0").manual_seed(3)
    midx = np.arange(1, 40, dtype=np.int64)
    T = torch.randn((len(midx), 1), dtype=torch.complex128, device="cuda:0", generator=g)
    S = torch.randn((P, Nt // 2 + 1), dtype=torch.complex128, device="cuda:0", generator=g)
    out = torch.empty((P, 1, Nt), dtype=torch.float32, device="cuda:0")
    sol = Solver(0)
    sol.synthesize(T, midx, S[:2], Nt, torch.float32, out=out[:2])  # (module and tables loaded)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    sol.synthesize(T, midx, S, Nt, torch.float32, out=out)
    torch.cuda.synchronize()
    assert free - torch.cuda.mem_get_info()[0] < 64 << 20
    for p in (0, 1022, 1023, 1024, 2046, P - 1):
        assert torch.equal(sol.synthesize(T, midx, S[p:p + 1], Nt, torch.float32)[0], out[p])
    sol.close()


def _radix2_fp32(c):
    """Re FFT(c) over the last axis by a radix-2 Stockham transform in FP32 (fused products, factors rounded
    from FP64): a plain transform's rounding, to hold another one against."""
    f32 = np.float32

    def fma(a, b, d):
        return (a.astype(np.float64) * b + d).astype(f32)

    n = c.shape[-1]
    xr, xi = c.real.astype(f32), c.imag.astype(f32)
    m, j = 1, np.arange(n // 2)
    while m < n:
        k = j & (m - 1)
        wr, wi = np.cos(np.pi * k / m).astype(f32), (-np.sin(np.pi * k / m)).astype(f32)
        ar, ai, br, bi = xr[..., : n // 2], xi[..., : n // 2], xr[..., n // 2:], xi[..., n // 2:]
        tr, ti = fma(br, wr, -(bi * wi)), fma(br, wi, bi * wr)
        yr, yi = np.empty_like(xr), np.empty_like(xi)
        at = 2 * (j - k) + k
        yr[..., at], yi[..., at], yr[..., at + m], yi[..., at + m] = ar + tr, ai + ti, ar - tr, ai - ti
        xr, xi, m = yr, yi, 2 * m
    return xr


@pytest.mark.parametrize("share", [2, 4])
@pytest.mark.parametrize("Nt", [64, 256, 1024, 4096])
def test_fp32_rounding_is_no_larger_than_a_radix_2_transforms(Nt, share):
    """Spectra that fill a half or a quarter of the samples, products rounded once: over 256 signals (a few
    tenths of a percent of scatter) the error against 64 bits is at most that of a radix-2 FP32 transform."""
    import torch
    from paper_1706_07919_gb300 import Solver

    rng = np.random.default_rng(Nt)
    nk, P, M = Nt // share - 1, 4, 64
    midx = np.arange(1, nk + 1, dtype=np.int64)
    T = rng.standard_normal((nk, M)) + 1j * rng.standard_normal((nk, M))
    S = rng.standard_normal((P, Nt // 2 + 1)) + 1j * rng.standard_normal((P, Nt // 2 + 1))
    c = np.zeros((P, M, Nt), complex)
    c[:, :, midx] = 2 * S[:, None, midx] * T.T[None]
    ref = np.fft.fft(c, axis=2).real / Nt
    plain = _radix2_fp32(c) / np.float32(Nt)
    sol = Solver(0)
    got = sol.synthesize(torch.tensor(T, device="cuda:0"), midx, torch.tensor(S, device="cuda:0"), Nt, torch.float32)
    assert np.linalg.norm(got.cpu().numpy() - ref) <= np.linalg.norm(plain - ref)
    sol.close()


@pytest.mark.parametrize("f32", [False, True])
@pytest.mark.parametrize("Nt", [32, 64, 512, 1024])
def test_few_and_many_signals(Nt, f32):
    """Counts of signals at which short ones change from the radix-2 kernel to the other (four to an SM)."""
    import torch
    from paper_1706_07919_gb300 import Solver
    from paper_1706_07919_gb300 import binding as B

    sm = torch.cuda.get_device_properties(0).multi_processor_count
    dt, eps = (torch.float32, 2.0 ** -24) if f32 else (torch.float64, 2.0 ** -53)
    sol = Solver(0)
    for M, P in ((4 * sm, 1), (4 * sm + 1, 1), (2 * sm, 2), (sm, 5)):
        T, midx, S = _case(Nt, M, P, Nt + M, True)
        Td, Sd = torch.tensor(T, device="cuda:0"), torch.tensor(S, device="cuda:0")
        ref = _reference(T, midx, S, Nt)
        out = torch.empty((P, M, Nt), dtype=dt, device="cuda:0")
        B.bie_synthesize_noalloc(Td, midx, Sd, Nt, out, 1 if f32 else 0)
        for got in (sol.synthesize(Td, midx, Sd, Nt, dt), out):
            assert np.linalg.norm(got.cpu().numpy() - ref) <= (4 * np.log2(Nt) + 3) * eps * np.linalg.norm(ref), (M, P)
    sol.close()


def test_fp32_synthesis_keeps_products_of_values_that_vanish_in_fp32():
    """Field spectra that round to zero in FP32 with pulses near the upper end of its safe range."""
    import torch
    from paper_1706_07919_gb300 import Solver

    sol = Solver(0)
    T, midx, S = _case(1024, 700, 3, 2, False)
    for a, b in ((1e-47, 1e24), (1e24, 1e-47)):
        got = sol.synthesize(torch.tensor(T * a, device="cuda:0"), midx, torch.tensor(S * b, device="cuda:0"), 1024,
                             torch.float32).cpu().numpy()
        ref = _reference(T * a, midx, S * b, 1024)
        assert np.linalg.norm(got - ref) <= 43 * 2.0 ** -24 * np.linalg.norm(ref)
    sol.close()
