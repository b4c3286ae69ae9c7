"""The training step's fused epilogues at the edges of their tiles: batches that end inside a 32-row
block, a 64-row transpose and a 128-row tile, the smallest and the widest inputs. Every stage in
FP64 from the GPU's own inputs, with the bounds of tests/test_mlp_gpu.py."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from oracle import mlp as ref  # noqa: E402
from tests.test_mlp_gpu import acc_bound, check, f32, run_backward, setup  # noqa: E402


@pytest.mark.parametrize("n_in,B", [(16, 16), (16, 144), (80, 48), (368, 1040), (496, 272)])
def test_training_stages_at_tile_edges(n_in, B):
    net, q, X, t = setup(n_in, B, seed=n_in + B)
    L, g, tp = run_backward(net, X, t)
    h1, dz2, dz1 = (ref.from_bf16_bits(tp[k]) for k in ("h1", "dz2", "dz1"))
    dz1 = dz1.T
    check("z1", tp["z1"], X @ q["W1"].T, acc_bound(np.abs(X) @ np.abs(q["W1"]).T, n_in))
    assert np.array_equal(h1, ref.bf16(np.maximum(f32(tp["z1"]) + f32(q["b1"]), np.float32(0))))
    check("z2", tp["z2"], h1 @ q["W2"].T, acc_bound(np.abs(h1) @ np.abs(q["W2"]).T, 256))
    h2 = np.maximum(f32(tp["z2"]) + f32(q["b2"]), np.float32(0)).astype(np.float64)
    y = h2 @ q["w3"] + q["b3"][0]
    e_y = acc_bound(np.abs(h2) @ np.abs(q["w3"]) + abs(q["b3"][0]), 257)
    dy = tp["dy"].astype(np.float64)
    check("dy", dy, 2 * (y - t) / B, 2 / B * (e_y + 4 * 2.0 ** -24 * (np.abs(y) + np.abs(t))))
    check("loss", L, ((B * dy / 2) ** 2).sum() / B, acc_bound(((B * dy / 2) ** 2).sum() / B, B + 8))
    e2 = np.where(f32(tp["z2"]) + f32(q["b2"]) > 0, f32(tp["dy"])[:, None] * f32(q["w3"])[None, :], np.float32(0))
    assert np.array_equal(dz2, ref.bf16(e2))
    e1 = np.where(f32(tp["z1"]) + f32(q["b1"]) > 0, f32(tp["dh1"]), np.float32(0))
    assert np.array_equal(dz1, ref.bf16(e1))
    e1, e2 = e1.astype(np.float64), e2.astype(np.float64)
    check("gw3", g["w3"], h2.T @ dy, acc_bound(np.abs(h2).T @ np.abs(dy), B + 8))
    check("gb2", g["b2"], e2.sum(axis=0), acc_bound(np.abs(e2).sum(axis=0), B + 8))
    check("gb3", g["b3"], [dy.sum()], acc_bound([np.abs(dy).sum()], B + 8))
    check("gb1", g["b1"], e1.sum(axis=0), acc_bound(np.abs(e1).sum(axis=0), B + 8))
    check("dW2", g["W2"], dz2.T @ h1, acc_bound(np.abs(dz2).T @ np.abs(h1), B + 16))
    check("dh1", tp["dh1"], dz2 @ q["W2"], acc_bound(np.abs(dz2) @ np.abs(q["W2"]), 256))
    check("dW1", g["W1"], dz1.T @ X, acc_bound(np.abs(dz1).T @ np.abs(X), B + 16))
    got = net.predict(torch.as_tensor(X, device="cuda").to(torch.bfloat16)).double().cpu().numpy()
    check("y", got, y, e_y)
