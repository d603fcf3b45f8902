"""fp32 products in each of their tile plans (32 x 32, 32 x 64, 64 x 64 or
128 x 64 by the launch's size), with ragged rows, columns and depths and a batch
below the capacity.  Values against fp64 on the activations the GPU itself
stored, so that a ReLU on the edge does not matter: a sum of n products in any
order differs from fp64 by at most n 2^-24 of the sum of their magnitudes; 3e-5
= 503 2^-24 is the mean case of the largest n here, 528, and of two chained
sums."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from test_gpu_parity import DEV, make_data, pair, to_dev, tp  # noqa: E402,F401
from workloads import random_pack  # noqa: E402


# (members, width, d_in, batch): tiles of 128 x 64 in the hidden layer's forward launch, and its plan
@pytest.mark.parametrize("m,w,d_in,B", [
    (3, 112, 9, 200),     # 12: 32 x 32
    (12, 144, 40, 77),    # 72: 32 x 32, the second of two row tiles empty; backward 72 + 72: 32 x 64
    (13, 144, 24, 129),   # 78: 32 x 64
    (10, 528, 61, 256),   # 180: 64 x 64; backward 180 + 450, 128 x 64
    (20, 528, 200, 250),  # 360 at depth 528: 64 x 64
    (20, 240, 8, 193),    # 160: 64 x 64; backward 160 + 160 at depth 248: 128 x 64
    (34, 528, 24, 100),   # 612: 128 x 64
])
def test_products(tp, m, w, d_in, B):  # noqa: F811
    hp = random_pack(m, d_in, 1, seed=3, depth=(2, 2), dropout=(0.0, 0.0))
    hp["width"], hp["depth"] = np.full(m, w, dtype=np.int32), np.full(m, 2, dtype=np.int32)
    pk, _ = pair(tp, "regression", d_in, 1, hp, "fp32", 256)
    X, y = make_data("regression", 400, d_in, 1, 5)
    idx = np.random.default_rng(6).choice(400, B, replace=False).astype(np.int32)
    Xd, yd, idxd = to_dev(X, y, idx)
    pk.forward_backward(Xd, idxd, yd, 0)
    out = pk.predict(Xd[torch.from_numpy(idx).long().to(DEV)].contiguous()).cpu().numpy().reshape(m, B)
    x, t = X[idx].astype(np.float64), y[idx].astype(np.float64)

    def close(got, ref, mag, what):
        bad = np.abs(got - ref) > 3e-5 * mag + 1e-12
        assert not bad.any(), (what, int(bad.sum()), np.abs(got - ref).max())

    for i in range(m):
        (W1, b1), (W2, b2), (W3, b3) = [[a.astype(np.float64) for a in pk.get_params(i, l)] for l in range(3)]
        H1, H2 = (pk.debug_activations(i, l).astype(np.float64)[:B] for l in range(2))
        close(H1, np.maximum(x @ W1.T + b1, 0), np.abs(x) @ np.abs(W1).T + np.abs(b1), (i, "forward 0"))
        close(H2, np.maximum(H1 @ W2.T + b2, 0), H1 @ np.abs(W2).T + np.abs(b2), (i, "forward 1"))
        z = (H2 @ W3.T + b3)[:, 0]
        close(out[i], z, H2 @ np.abs(W3[0]) + np.abs(b3[0]) + 1, (i, "prediction"))
        d = 2 * (z - t) / B
        da = 2 * (H2 @ np.abs(W3[0]) + np.abs(b3[0]) + np.abs(t)) / B
        dz2, az2 = d[:, None] * W3 * (H2 > 0), da[:, None] * np.abs(W3) * (H2 > 0)
        dz1, az1 = (dz2 @ W2) * (H1 > 0), (az2 @ np.abs(W2)) * (H1 > 0)
        for l, dz, az, h in ((1, dz2, az2, H1), (0, dz1, az1, x)):
            gW, gb = pk.get_grads(i, l)
            close(gW, dz.T @ h, az.T @ np.abs(h), (i, "weights", l))
            close(gb, dz.sum(0), az.sum(0), (i, "bias", l))
    pk.close()
