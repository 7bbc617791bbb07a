"""More than four right-hand sides through the FP32 block products (eight at a time, pairs of eights
per CTA, 4 rows per warp): counts around 4, 8 and 16, blocks whose size is odd, below a task of 16
rows and no multiple of it, both outputs or one. internal_apply against the FP64 product of the same
context, bem_blockdiag_gemv against NumPy; C32 1e-5 as the other GEMV tests."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2108_03991_gb300 import api, synth  # noqa: E402

COUNTS = [5, 8, 9, 16, 17, 31, 33]


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2108_03991_gb300 import build
    build.build()
    mesh = synth.small_bars(3, 3.0)
    c = api.Context(mesh, synth.grid_box(mesh, 0.5), 10e9)
    yield c
    c.close()


@pytest.mark.parametrize("nrhs", COUNTS)
def test_internal(ctx, nrhs):
    h = torch.from_numpy(synth.rand_cvec(nrhs * ctx.ne, 80 + nrhs).astype(np.complex64)).cuda()
    e, q = ctx.internal(h, nrhs=nrhs)
    e1, _ = ctx.internal(h, nrhs=nrhs, want_heq=False)
    _, q1 = ctx.internal(h, nrhs=nrhs, want_e=False)
    er, qr = ctx.internal(h.to(torch.complex128), nrhs=nrhs, prec=api.BEM_C64)
    assert torch.equal(e, e1) and torch.equal(q, q1)
    for out, ref in ((e, er), (q, qr)):
        d = (out - ref).view(nrhs, -1).norm(dim=1)
        assert bool((d <= 1e-5 * ref.view(nrhs, -1).norm(dim=1)).all())


@pytest.mark.parametrize("nrhs", COUNTS)
def test_blocks(ctx, nrhs):
    sizes = [1, 2, 15, 16, 17, 63, 65, 130, 257]
    blocks = synth.rand_blocks(sizes, 7)
    N = sum(sizes)
    x = synth.rand_cvec(nrhs * N, 90 + nrhs).reshape(nrhs, N)
    ref = np.concatenate([x[:, o:o + B.shape[0]] @ B.T
                          for o, B in zip(np.cumsum([0] + sizes), blocks)], axis=1)
    A = torch.from_numpy(api.pack_blocks(blocks, np.complex64)).cuda()
    xd = torch.from_numpy(x.astype(np.complex64).ravel()).cuda()
    y = api.blockdiag_gemv(sizes, A, xd, torch.empty_like(xd), nrhs).cpu().numpy().reshape(nrhs, N)
    assert np.all(np.linalg.norm(y - ref, axis=1) <= 1e-5 * np.linalg.norm(ref, axis=1))


def test_pinned_form(ctx):
    """A launch form that the caller chose holds for every count: each group of four gives the bits
    of a call with that group alone; select(0) gives the eights back."""
    h = torch.from_numpy(synth.rand_cvec(9 * ctx.ne, 70).astype(np.complex64)).cuda()
    free = ctx.internal(h, nrhs=9)
    ctx.gemv_plan(0, 6, 2, 4)
    try:
        e, q = ctx.internal(h, nrhs=9)
        for r, n in ((0, 4), (4, 4), (8, 1)):
            sl = slice(r * ctx.ne, (r + n) * ctx.ne)
            e1, q1 = ctx.internal(h[sl].contiguous(), nrhs=n)
            assert torch.equal(e[sl], e1) and torch.equal(q[sl], q1)
    finally:
        ctx.gemv_select(0)
    for out, ref in zip(ctx.internal(h, nrhs=9), free):
        assert torch.equal(out, ref)


def test_blocks_beyond_one_grid(ctx):
    """More right-hand sides than the pairs of eights of one launch (65,535 along the grid's y): the
    vectors on both sides of the cut and the last ones, against NumPy."""
    sizes, nrhs = [1, 2], 16 * 65535 + 5
    blocks = synth.rand_blocks(sizes, 8)
    x = torch.randn(nrhs * 3, dtype=torch.complex64, device="cuda")
    A = torch.from_numpy(api.pack_blocks(blocks, np.complex64)).cuda()
    y = api.blockdiag_gemv(sizes, A, x, torch.full_like(x, float("nan")), nrhs).view(nrhs, 3)
    x = x.view(nrhs, 3).to(torch.complex128)
    ref = torch.empty_like(x)
    for o, B in zip((0, 1), blocks):
        k = B.shape[0]
        ref[:, o:o + k] = x[:, o:o + k] @ torch.from_numpy(B).to(x).T
    # per vector: |y - ref| <= 1e-5 |A| |x|
    d = (y - ref).norm(dim=1)
    assert bool((d <= 1e-5 * max(np.linalg.norm(B) for B in blocks) * x.norm(dim=1)).all())


@pytest.fixture(scope="module")
def rings():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    c = api.Context(*synth.srr_array_config(2, 2))
    assert c.sparse_internal["on"]
    yield c
    c.close()


@pytest.mark.parametrize("prec", [api.BEM_C32, api.BEM_C64])
@pytest.mark.parametrize("nrhs", [4, 5, 8, 9, 16])
def test_internal_sparse(rings, nrhs, prec):
    """More vectors than the sparse internal operator takes at once, e and h_eq, either and both: e has
    the bits of a call with that vector alone, h_eq is the FP64 product's (C32 1e-5, C64 1e-12)."""
    h = torch.from_numpy(synth.rand_cvec(nrhs * rings.ne, 60 + nrhs)).to(api.cdtype(prec)).cuda()
    e, q = rings.internal(h, nrhs=nrhs, prec=prec)
    e1, _ = rings.internal(h, nrhs=nrhs, prec=prec, want_heq=False)
    _, q1 = rings.internal(h, nrhs=nrhs, prec=prec, want_e=False)
    assert torch.equal(e, e1) and torch.equal(q, q1)
    for r in range(nrhs):
        sl = slice(r * rings.ne, (r + 1) * rings.ne)
        hr = h[sl].contiguous()
        assert torch.equal(e[sl], rings.internal(hr, prec=prec, want_heq=False)[0])
        ref = rings.internal(hr.to(torch.complex128), prec=api.BEM_C64, want_e=False)[1]
        assert float((q[sl] - ref).norm()) <= (1e-5 if prec == api.BEM_C32 else 1e-12) * float(ref.norm())
    assert not rings.internal_sparse(True)["wait_timed_out"]
