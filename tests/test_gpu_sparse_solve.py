"""Block substitutions of the sparse internal operator at the sizes where they can go wrong: edge
counts that are no multiple of a block, a half-bandwidth next to a block's width (32 columns, whose
triangle has to fit the stored band) and one above the 128 rows an update pass takes.
e = Z_s h against the dense Z h of the same context in the same precision, one to four right-hand
sides. Tolerances: the dropped pairs are below e^-23 = 1e-10 of the kept ones (C64 1e-9, ten times
that); FP32 products of these lengths round to about 1e-6 (C32 1e-5, the tolerance of the matvec)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2108_03991_gb300 import api, synth  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2108_03991_gb300 import build
    build.build()


def thin_bar():  # 486 edges, half-bandwidth 33 at 20 THz
    mesh = synth.bar_mesh(0.5, 0.5, 20.0, 0.5)
    return mesh, synth.grid_box(mesh, 0.5), 2e13


def rings(n_theta, n_r):  # two rings at 1 THz
    return synth.srr_array(2, 2, 1, n_theta=n_theta, n_r=n_r, n_z=1), synth.srr_grid(2), 1e12


@pytest.mark.parametrize("make,lo,hi", [(thin_bar, 31, 40), (lambda: rings(61, 2), 97, 128),
                                        (lambda: rings(80, 3), 160, 192)])
def test_sparse_against_dense(make, lo, hi):
    mesh, grid, freq = make()
    ctx = api.Context(mesh, grid, freq)
    info = ctx.sparse_internal
    assert info["objects"] == mesh.nobj and info["on"] and lo <= info["band"] <= hi
    for prec, tol in ((api.BEM_C64, 1e-9), (api.BEM_C32, 1e-5)):
        for nrhs in range(1, 5):
            h = torch.from_numpy(synth.rand_cvec(nrhs * ctx.ne, 31 + nrhs)).to(api.cdtype(prec)).cuda()
            e = {}
            for on in (True, False):
                ctx.internal_sparse(on)
                e[on] = ctx.internal(h, nrhs=nrhs, prec=prec, want_heq=False)[0].cpu().numpy()
            for s, d in zip(np.split(e[True], mesh.nobj * nrhs), np.split(e[False], mesh.nobj * nrhs)):
                assert np.linalg.norm(s - d) <= tol * np.linalg.norm(d)
    assert not ctx.internal_sparse(True)["wait_timed_out"]
    ctx.close()


def test_explicit_choice_holds():
    """FP64 system products of one to four vectors on two rings: dense after set-up (two rings are
    bound by two SMs' FP64 rate otherwise), sparse once a caller chose the sparse form, which the
    status reports and the bits show (both forms agree to 1e-12, not to the last bit)."""
    ctx = api.Context(*rings(60, 2))
    n0 = ctx.sparse_internal["fp64_dense"]
    assert ctx.sparse_internal["on"] and 1 in n0

    def products():
        out = []
        for r in range(1, 5):
            x = torch.from_numpy(synth.rand_cvec(r * ctx.n, 40 + r)).cuda()
            y = ctx.matvec(x, prec=api.BEM_C64) if r == 1 else ctx.matvec_batch(x, prec=api.BEM_C64)
            out.append(y.view(r, ctx.n)[:, :ctx.ne].clone())
        return out
    auto = products()
    assert ctx.internal_sparse(True)["fp64_dense"] == []
    sparse = products()
    assert ctx.internal_sparse(False)["fp64_dense"] == []
    dense = products()
    for r, (a, s, d) in enumerate(zip(auto, sparse, dense), 1):
        assert torch.equal(a, d if r in n0 else s)
        assert not torch.equal(s, d) and float((s - d).norm()) <= 1e-12 * float(d.norm())
    assert not ctx.internal_sparse(True)["wait_timed_out"]
    ctx.close()


def _probe(n):
    """The set-up check's probe vector: a hash of the index, 24 bits a part."""
    v = np.arange(n, dtype=np.uint64) * np.uint64(0x9E3779B97F4A7C15) + np.uint64(0xD1B54A32D192ED03)
    v ^= v >> np.uint64(31)
    v *= np.uint64(0xBF58476D1CE4E5B9)
    v ^= v >> np.uint64(29)
    part = lambda b: b.astype(np.float64) / 2.0 ** 23 - 1.0  # noqa: E731
    return part(v >> np.uint64(40)) + 1j * part((v >> np.uint64(8)) & np.uint64(0xFFFFFF))


@pytest.mark.parametrize("make", [thin_bar, lambda: rings(80, 3)])
def test_fp32_form_is_checked(make):
    """The set-up check covers the FP32 tables: the status reports their error against the FP64 dense
    Z h, below 1e-5, and it is the one measured here (to a percent: it is rounded to 1e-12)."""
    mesh, grid, freq = make()
    ctx = api.Context(mesh, grid, freq)
    check = ctx.sparse_internal["check_c32"]
    assert ctx.sparse_internal["on"] and check is not None and 0 < check < 1e-5
    h = torch.from_numpy(_probe(ctx.ne)).cuda()
    e = ctx.internal(h.to(torch.complex64), want_heq=False)[0].cpu().numpy()
    ctx.internal_sparse(False)
    d = ctx.internal(h, prec=api.BEM_C64, want_heq=False)[0].cpu().numpy()
    worst = max(np.linalg.norm(a - b) / np.linalg.norm(b)
                for a, b in zip(np.split(e, mesh.nobj), np.split(d, mesh.nobj)))
    assert abs(worst - check) <= 0.01 * worst
    ctx.close()
