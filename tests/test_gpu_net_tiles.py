"""The correction network's passes at the grids where their tiles can go wrong: smaller than a
tile, one point over a tile or a quad of points, one long axis, more tiles than the weight gradient
has CTAs (456). The forward reference forms each output as the network does, FP32 sums in the order
input channel, tap (every fused multiply-add emulated in FP64 and rounded to FP32), activations
stored in BF16, so that no activation rounds the other way; the gradients are plain torch
convolutions in FP64 over those activations. FP32 sums of at most 432 terms (and one term per grid
point for the weights): 1e-4 relative."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2108_03991_gb300 import api  # noqa: E402

CH = [(8, 16), (16, 16), (16, 16), (16, 8)]


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2108_03991_gb300 import build
    build.build()


def bf(t):
    return t.to(torch.bfloat16).to(torch.float64)


def conv_fma(x, k):
    """x [ci, nz, ny, nx], k [co, ci, 3, 3, 3] (FP64 holding FP32 values): the sum in FP32."""
    p = torch.nn.functional.pad(x, (1,) * 6)
    nz, ny, nx = x.shape[1:]
    acc = torch.zeros((k.shape[0], nz, ny, nx), dtype=torch.float32, device=x.device)
    for ci in range(x.shape[0]):
        for t in range(27):
            dz, dy, dx = t // 9, t // 3 % 3, t % 3
            v = p[ci, dz:dz + nz, dy:dy + ny, dx:dx + nx]
            acc = (acc.to(torch.float64) + k[:, ci, dz, dy, dx].view(-1, 1, 1, 1) * v).to(torch.float32)
    return acc


@pytest.mark.parametrize("n", [(1, 1, 1), (3, 2, 5), (4, 8, 2), (13, 5, 7), (1, 1, 70), (97, 1, 3),
                               (70, 66, 31)])  # (nz, ny, nx)
def test_tiles(n):
    rng = np.random.default_rng(sum(n))
    w = np.concatenate([np.sqrt(2 / (27 * a)) * rng.standard_normal(a * b * 27) for a, b in CH])
    w = w.astype(np.float32)
    x = torch.from_numpy(rng.standard_normal((8, *n)).astype(np.float32)).cuda()
    go = torch.from_numpy(rng.standard_normal((8, *n)).astype(np.float32)).cuda()
    out, gw, gx = api.convnet_run(w, x, go)
    ks, o = [], 0
    for a, b in CH:
        ks.append(bf(torch.from_numpy(w[o:o + a * b * 27]).cuda().view(b, a, 3, 3, 3)))
        o += a * b * 27
    acts = [bf(x)[None]]
    for k in ks[:-1]:
        acts.append(bf(torch.relu(conv_fma(acts[-1][0], k)))[None])
    ref = conv_fma(acts[-1][0], ks[-1])
    assert (out - ref).norm() <= 1e-4 * ref.norm()
    g, grads = go.to(torch.float64)[None], []
    for l in range(3, -1, -1):
        grads.insert(0, torch.nn.grad.conv3d_weight(acts[l], ks[l].shape, g, padding=1).reshape(-1))
        g = torch.nn.grad.conv3d_input(acts[l].shape, ks[l], g, padding=1)
        if l:
            g = g * (acts[l] > 0)
    gwr = torch.cat(grads).cpu().numpy()
    assert np.linalg.norm(gw - gwr) <= 1e-4 * np.linalg.norm(gwr)
    assert (gx - g[0]).norm() <= 1e-4 * g[0].norm()
