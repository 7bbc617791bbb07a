"""bem_blockdiag_gemv where its table of blocks can go wrong: one block, blocks smaller than a task
of 4 (one right-hand side) or 16 rows, sizes in any order (the launch takes them largest first),
one block more than the small argument table holds (64) and more than one launch takes (1,984), in a
captured graph, against NumPy in 64 bits. Tolerances as the other GEMV tests: C32 1e-5, C64 1e-13."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2108_03991_gb300 import api, synth  # noqa: E402

LAYOUTS = {"one": [1], "small": [3, 1, 17, 4, 16, 5], "ragged": [33, 260, 7, 128, 129, 1, 64],
           "over_small": [5 + (i * 7) % 23 for i in range(65)],
           "over_large": [1 + (i * 5) % 9 for i in range(1984 * 2 + 3)]}


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2108_03991_gb300 import build
    build.build()


@pytest.mark.parametrize("name", list(LAYOUTS))
@pytest.mark.parametrize("nrhs", [1, 2, 5])
@pytest.mark.parametrize("prec,tol", [(api.BEM_C32, 1e-5), (api.BEM_C64, 1e-13)])
def test_layout(name, nrhs, prec, tol):
    sizes = LAYOUTS[name]
    blocks = synth.rand_blocks(sizes, 3)
    N = sum(sizes)
    x = synth.rand_cvec(nrhs * N, 4)
    ref = np.empty((nrhs, N), dtype=np.complex128)
    o = 0
    for B in blocks:
        ref[:, o:o + B.shape[0]] = x.reshape(nrhs, N)[:, o:o + B.shape[0]] @ B.T
        o += B.shape[0]
    dt = api.cdtype(prec)
    A = torch.from_numpy(api.pack_blocks(blocks, np.complex128)).to(dt).cuda()
    xd = torch.from_numpy(x).to(dt).cuda()
    y = api.blockdiag_gemv(sizes, A, xd, torch.empty_like(xd), nrhs, prec).cpu().numpy()
    assert np.linalg.norm(y - ref.ravel()) <= tol * np.linalg.norm(ref)


def test_captured():
    sizes = LAYOUTS["ragged"]
    A = torch.from_numpy(api.pack_blocks(synth.rand_blocks(sizes, 5), np.complex64)).cuda()
    x = torch.from_numpy(synth.rand_cvec(sum(sizes), 6)).to(torch.complex64).cuda()
    y, yg = torch.empty_like(x), torch.zeros_like(x)
    api.blockdiag_gemv(sizes, A, x, y)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        api.blockdiag_gemv(sizes, A, x, yg)
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(y, yg)
