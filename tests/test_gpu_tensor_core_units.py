"""aim_internal_tc where its units and scales can go wrong: one block whose tiles are cut along K
(2,016 rows), blocks of unlike sizes in one launch, every width of the packed right-hand sides and
its edges, either output alone, and slices of unlike magnitude (every object's slice of every
right-hand side has its own scale, from 1e-25 to 1e25, and one is zero). Against the FP64 product
of the context, per object and right-hand side. The accumulator truncates about 2 n / 16 sums of
2^-24 each: 1e-5, the matvec's tolerance, holds to n of 2,500 if every truncation went one way."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2108_03991_gb300 import api, synth  # noqa: E402


@pytest.fixture(scope="module", params=["one_block", "unlike_blocks"])
def ctx(request):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2108_03991_gb300 import build
    build.build()
    if request.param == "one_block":
        c = api.Context(*synth.copper_bar())
    else:
        parts = [synth.box((4.0 * i, 0.0, 0.0), (1.0, 1.0, L), (2, 2, int(2 * L)))
                 for i, L in enumerate((0.5, 9.0, 2.5, 20.0))]
        mesh = synth.merge(parts, [synth.SIGMA_CU] * len(parts))
        c = api.Context(mesh, synth.grid_box(mesh, 0.5), 10e9)
        c.sizes = [t.shape[0] * 3 // 2 for _, t in parts]
    if request.param == "one_block":
        c.sizes = [c.ne]
    yield c
    c.close()


@pytest.mark.parametrize("nrhs", [1, 16, 17, 32, 33, 64, 65, 128, 129])
def test_units_and_scales(ctx, nrhs):
    rng = np.random.default_rng(nrhs)
    h = synth.rand_cvec(nrhs * ctx.ne, 70 + nrhs).reshape(nrhs, ctx.ne)
    cut = np.cumsum([0] + ctx.sizes)
    assert cut[-1] == ctx.ne
    for r in range(nrhs):
        for a, b in zip(cut[:-1], cut[1:]):
            h[r, a:b] *= 10.0 ** rng.uniform(-25, 25)
    h[nrhs // 2, :cut[1]] = 0.0
    h32 = torch.from_numpy(h.astype(np.complex64).ravel()).cuda()
    e, q = ctx.internal_tc(h32, nrhs=nrhs)
    e1, _ = ctx.internal_tc(h32, nrhs=nrhs, want_heq=False)
    _, q1 = ctx.internal_tc(h32, nrhs=nrhs, want_e=False)
    er, qr = ctx.internal(h32.to(torch.complex128), nrhs=nrhs, prec=api.BEM_C64)
    for out, ref in ((e, er), (q, qr), (e1, er), (q1, qr)):
        out, ref = out.cpu().numpy().reshape(nrhs, -1), ref.cpu().numpy().reshape(nrhs, -1)
        for a, b in zip(cut[:-1], cut[1:]):
            d = np.linalg.norm(out[:, a:b] - ref[:, a:b], axis=1)
            assert np.all(d <= 1e-5 * np.linalg.norm(ref[:, a:b], axis=1))
    assert ctx.tensor_core_status()["wait_timed_out"] is False


def test_unit_vectors(ctx):
    """A unit vector (one edge, one port) gives back a column of Z and of C, whose entries fall by tens of
    binades along a bar: each real and imaginary part within 2^-22 of the FP32 entry (three parts hold its
    24 bits; two accumulators and their sum round once each). Entries and products below 2^-100 are left
    out: the third part of one below 2^-110 leaves the normal range of BF16 (and FP32) numbers."""
    ks = [0, 1, ctx.ne // 3, ctx.ne // 2 + 1, ctx.ne - 1] * 4
    h = torch.zeros(len(ks), ctx.ne, dtype=torch.complex64, device="cuda")
    for r, k in enumerate(ks):
        h[r, k] = 2.0 ** (7 * r - 60)
    for out, ref in zip(ctx.internal_tc(h.view(-1), nrhs=len(ks)), ctx.internal(h.view(-1), nrhs=len(ks))):
        out = torch.view_as_real(out).double().view(len(ks), -1)
        ref = torch.view_as_real(ref).double().view(len(ks), -1)
        entry = ref / h.abs().amax(dim=1, keepdim=True).double()
        live = (entry.abs() >= 2.0 ** -100) & (ref.abs() >= 2.0 ** -100)
        assert bool(((out - ref).abs() <= 2.0 ** -22 * ref.abs())[live].all())
        assert float(entry.abs()[entry != 0].min() / entry.abs().max()) < 2.0 ** -18
    assert ctx.tensor_core_status()["wait_timed_out"] is False
