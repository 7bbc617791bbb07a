"""The grid step on grids beyond the plane passes, FP32, over the lengths the two-pass transforms take:
every radix of the x and y passes, z in registers (Pz a radix) and as two passes (nz > 16), rows that
are no multiple of eight, equal and unlike x and y, one to five components where the entry allows
four. Against NumPy's FFT in 64 bits; 2e-6, the tolerance of the other FP32 convolution tests."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import operators as op  # noqa: E402
from paper_2108_03991_gb300 import api, synth  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2108_03991_gb300 import build
    build.build()


@pytest.mark.parametrize("n", [(128, 125, 8), (150, 90, 21), (113, 101, 9), (135, 144, 7), (203, 48, 33),
                               (321, 37, 12), (76, 200, 40), (512, 61, 6), (97, 97, 16), (240, 162, 25),
                               (313, 365, 8), (405, 75, 10)])
def test_conv(n):
    grid = synth.Grid(np.array([-1.1, -1.1, -1.1]), np.array([0.5, 0.4, 0.5]), np.array(n))
    freq = 3e13  # kR up to a hundred: the phase of the grid kernel matters
    ctx = api.Context(synth.bar_mesh(1.0, 1.0, 1.0, 0.5), grid, freq)
    k0 = op.k0_of(freq)
    P = [2 * v for v in n]
    ax = [np.minimum(np.arange(p), p - np.arange(p)) * h for p, h in zip(P, grid.h)]
    R = np.sqrt(ax[2][:, None, None] ** 2 + ax[1][None, :, None] ** 2 + ax[0][None, None, :] ** 2)
    R[0, 0, 0] = 1.0
    G = np.exp(-1j * k0 * R) / (4 * np.pi * R)
    G[0, 0, 0] = 0
    G = np.fft.fftn(G)
    for ncomp in (1, 4) if n[2] < 20 else (3,):
        s = synth.rand_cvec(ncomp * ctx.ng, 9).reshape(ncomp, n[2], n[1], n[0])
        f = np.fft.ifftn(np.fft.fftn(s, s=(P[2], P[1], P[0]), axes=(1, 2, 3)) * G, axes=(1, 2, 3))
        ref = f[:, :n[2], :n[1], :n[0]]
        d = torch.from_numpy(s.astype(np.complex64).ravel()).cuda()
        out = ctx.conv(d, ncomp=ncomp).cpu().numpy().reshape(s.shape)
        inplace = ctx.conv(d, d, ncomp=ncomp).cpu().numpy().reshape(s.shape)
        for c in range(ncomp):
            assert np.linalg.norm(out[c] - ref[c]) <= 2e-6 * np.linalg.norm(ref[c])
        assert np.array_equal(out, inplace)
    ctx.close()


def _reference(ctx, grid, freq, n, s):
    k0 = op.k0_of(freq)
    P = [2 * v for v in n]
    ax = [np.minimum(np.arange(p), p - np.arange(p)) * h for p, h in zip(P, grid.h)]
    R = np.sqrt(ax[2][:, None, None] ** 2 + ax[1][None, :, None] ** 2 + ax[0][None, None, :] ** 2)
    R[0, 0, 0] = 1.0
    G = np.exp(-1j * k0 * R) / (4 * np.pi * R)
    G[0, 0, 0] = 0
    f = np.fft.ifftn(np.fft.fftn(s, s=(P[2], P[1], P[0]), axes=(1, 2, 3)) * np.fft.fftn(G), axes=(1, 2, 3))
    return f[:, :n[2], :n[1], :n[0]]


@pytest.mark.parametrize("prec,n", [(api.BEM_C32, n) for n in ((7, 7, 43), (12, 11, 8), (20, 20, 9), (10, 9, 13),
                                                                (8, 16, 16), (18, 18, 14), (23, 41, 8))] +
                         [(api.BEM_C64, n) for n in ((7, 7, 43), (20, 20, 8), (24, 21, 9), (40, 33, 8))])
def test_small_planes(prec, n):
    """Small planes with a z line per thread (Pz a radix) or the shared-memory z pass, the first sizes of
    the two-pass form, and FP64 planes as lines; C32 2e-6, C64 1e-12 as the other convolution tests."""
    grid = synth.Grid(np.array([-1.1, -1.1, -1.1]), np.array([0.5, 0.4, 0.5]), np.array(n))
    freq = 3e13
    ctx = api.Context(synth.bar_mesh(1.0, 1.0, 1.0, 0.5), grid, freq)
    s = synth.rand_cvec(3 * ctx.ng, 11).reshape(3, n[2], n[1], n[0])
    ref = _reference(ctx, grid, freq, n, s)
    out = ctx.conv(torch.from_numpy(s.ravel()).to(api.cdtype(prec)).cuda(), ncomp=3, prec=prec)
    out = out.cpu().numpy().reshape(s.shape)
    for c in range(3):
        assert np.linalg.norm(out[c] - ref[c]) <= (2e-6 if prec == api.BEM_C32 else 1e-12) * np.linalg.norm(ref[c])
    ctx.close()


RADICES = [1, 2, 3, 4, 5, 6, 8, 9, 10, 12, 15, 16, 18, 20, 24, 25, 27, 30, 32]


@pytest.mark.parametrize("n,slab", [((500, 60, 8), True), ((540, 61, 12), True), ((486, 500, 8), True),
                                    ((520, 90, 16), True), ((61, 540, 12), False), ((520, 90, 17), False),
                                    ((400, 401, 20), False)])
def test_lengths_without_two_passes(n, slab):
    """FP32 grids that the two-pass form does not take: an x or y length that is no product of two radices
    (the slab passes where nz <= 16 and their slab fits shared memory, else the line passes), or a y-z
    slab beyond shared memory (line passes). 2e-6 and 1e-5 of the largest value, as the other convolution tests; one component and two."""
    grid = synth.Grid(np.array([-1.1, -1.1, -1.1]), np.array([0.5, 0.4, 0.5]), np.array(n))
    freq = 3e13
    ctx = api.Context(synth.bar_mesh(1.0, 1.0, 1.0, 0.5), grid, freq)
    P = ctx.padded
    two = [any(P[a] % r == 0 and P[a] // r in RADICES for r in RADICES) for a in (0, 1)]
    assert not all(two) or 8 * P[1] * P[2] > 200 * 1024  # else the two-pass form takes it
    floats2 = P[1] + P[2] + (P[2] // 2 + 1) * (P[1] // 2 + 1) + 2 * n[2] * (P[1] + P[1] // 16 + 1)
    assert slab == (n[2] <= 16 and 8 * floats2 <= 200 * 1024)
    s = synth.rand_cvec(2 * ctx.ng, 13).reshape(2, n[2], n[1], n[0])
    ref = _reference(ctx, grid, freq, n, s)
    for ncomp in (1, 2):
        d = torch.from_numpy(s[:ncomp].astype(np.complex64).ravel()).cuda()
        out = ctx.conv(d, ncomp=ncomp).cpu().numpy().reshape(s[:ncomp].shape)
        for c in range(ncomp):
            assert np.linalg.norm(out[c] - ref[c]) <= 2e-6 * np.linalg.norm(ref[c])
            assert np.abs(out[c] - ref[c]).max() <= 1e-5 * np.abs(ref[c]).max()
    ctx.close()
