"""The fused network kernel at the edges of its 128-row clusters, and a training
step against its parts: the rows that the documented Philox draw picks, the
gradient of those rows, and one Adam update in float64."""
import numpy as np
import pytest

from oracle import mlp_oracle as mo
from paper_2407_11349_gb300.hawkes import MLP

pytestmark = pytest.mark.gpu

BLOCKS = [(0, 1792), (1792, 2048), (2048, 67584), (67584, 67840), (67840, 69632), (69632, 69639)]


# half a cluster is empty (64), exactly one (128), one and a half (320 = 2.5),
# the most (4096)
@pytest.mark.parametrize("B", [64, 128, 320, 4096])
def test_gradient_at_cluster_edges(B):
    """A row's outputs do not depend on its place in the batch: equal, to the
    last bit, to those of a batch of 64 (which test_gpu_mlp.py holds to the
    reference).  Loss and gradient blocks: tolerances as there (2e-4, 2e-3 of
    the block's largest entry)."""
    rng = np.random.default_rng(B + 1)
    theta = (mo.init_params(6) + rng.normal(0, 0.02, mo.N_PARAMS)).astype(np.float32)
    x = rng.normal(size=(B, 7)).astype(np.float32)
    t = rng.normal(size=(B, 7)).astype(np.float32)
    net = MLP(0, seed=1)
    try:
        net.set_params(theta)
        L, g, Y = net.loss_grad(x, t)
        L2, g2, Y2 = net.loss_grad(x, t)
        parts = np.concatenate([net.loss_grad(x[k:k + 64], t[k:k + 64])[2] for k in range(0, B, 64)])
    finally:
        net.close()
    assert np.array_equal(g, g2) and np.array_equal(Y, Y2)  # fixed order of every sum
    th64, x64, t64 = theta.astype(np.float64), x.astype(np.float64), t.astype(np.float64)
    Lref, gref = mo.loss_and_grad(th64, x64, t64, bf16=True)
    assert np.array_equal(Y, parts)
    assert abs(L - Lref) <= 2e-4 * Lref
    for a, b in BLOCKS:
        assert np.max(np.abs(g[a:b] - gref[a:b])) <= 2e-3 * np.max(np.abs(gref[a:b])), (a, b)


def _philox4x32(c0, c1, c2, c3, k0, k1):
    c = [np.asarray(v, dtype=np.uint64) for v in (c0, c1, c2, c3)]
    m = np.uint64(0xFFFFFFFF)
    for r in range(10):
        p0, p1 = c[0] * np.uint64(0xD2511F53), c[2] * np.uint64(0xCD9E8D57)
        s = np.uint64(32)
        ka, kb = np.uint64((k0 + r * 0x9E3779B9) & 0xFFFFFFFF), np.uint64((k1 + r * 0xBB67AE85) & 0xFFFFFFFF)
        c = [((p1 >> s) ^ c[1] ^ ka) & m, p1 & m, ((p0 >> s) ^ c[3] ^ kb) & m, p0 & m]
    return c


@pytest.mark.parametrize("n", [2, 3, 1000, 65537])
def test_training_step_is_its_parts(n):
    rng = np.random.default_rng(n)
    X, Yt = rng.normal(size=(n, 6)), rng.normal(size=(n, 7))
    B, seed, lr = 192, 0x123456789ABC, 1e-3
    net = MLP(0, seed=2)
    try:
        net.set_data(X, Yt)
        st = net.stats()
        theta = net.get_params()
        loss = net.train(1, batch=B, lr=lr, seed=seed)
        after = net.get_params().astype(np.float64)
        r = _philox4x32(np.arange(B), np.zeros(B), np.zeros(B), np.full(B, 0x4D4C50), seed & 0xFFFFFFFF, seed >> 32)
        u = [(int(a) << 32) | int(b) for a, b in zip(r[0], r[1])]
        rows = np.array([v % n for v in u])
        xs = np.column_stack([(X - st[:6]) / st[6:12], np.ones(n)]).astype(np.float32)[rows]
        ts = ((Yt - st[12:19]) / st[19:26]).astype(np.float32)[rows]
        net.set_params(theta)
        L, g, _ = net.loss_grad(xs, ts)
    finally:
        net.close()
    assert abs(loss - L) <= 1e-6 * L
    g = g.astype(np.float64)
    want = theta.astype(np.float64) - lr * g / (np.abs(g) + 1e-8)  # Adam's first step
    # FP32 roundings of the moments and the update: 1e-5 of the step, and one
    # rounding of the weight; gradients too small for their sign to be certain
    # (the rows' FP32 standardisation may differ in the last bit) are left out
    sure = np.abs(g) > 1e-3 * np.abs(g).max()
    assert sure.sum() > 1000
    assert np.all(np.abs(after - want)[sure] <= 1e-5 * lr + 2.0 ** -23 * np.abs(want[sure]))


@pytest.mark.parametrize("count", [1, 127, 128, 129, 4096])
def test_predictions_at_cluster_edges(count):
    """Equal, to the last bit, to predictions in batches of 77 (the size that
    test_gpu_mlp.py holds to the reference), and nothing written past the end."""
    torch = pytest.importorskip("torch")
    rng = np.random.default_rng(count)
    X, Yt = rng.normal(size=(400, 6)), rng.normal(size=(400, 7)) * 50.0 - 1e5
    net = MLP(0, seed=3)
    try:
        net.set_data(X, Yt)
        net.train(30, batch=64, lr=1e-3, seed=2)
        q = rng.normal(size=(count, 6))
        dq = torch.tensor(q, dtype=torch.float64, device="cuda")
        out = torch.full((count + 1, 7), -7.0, dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        net.predict(dq.data_ptr(), count, out.data_ptr())
        net.wait()
        got = out.cpu().numpy()
        for k in range(0, count, 77):
            m = min(77, count - k)
            net.predict(dq[k:].data_ptr(), m, out[k:].data_ptr())
        net.wait()
        parts = out.cpu().numpy()
    finally:
        net.close()
    assert np.all(got[count] == -7.0) and np.array_equal(got, parts)
