"""The tensor-core multiclass head (bf16): widths around its 64-column chunks
and 128-column steps, class counts around its 16- and 32-class layouts, batches
around its 128-row blocks.  Logits, losses, head gradients and probabilities
against fp64 on the activations the GPU itself stored, within fp32
accumulation: a sum of n products differs from fp64 by at most n 2^-24 of the
sum of their magnitudes; 1e-5 = 168 2^-24 is the mean case of n up to 2048.
dZ reaches the hidden layers' gradients, which are compared with the oracle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from parity import compare_step  # noqa: E402
from test_gpu_parity import DEV, make_data, pair, to_dev, tp  # noqa: E402,F401
from workloads import random_pack  # noqa: E402

WIDTHS = np.array([16, 64, 80, 128, 144, 208, 1040, 2048], dtype=np.int32)


def _step(tp, d_out, B, widths, depth, dropout):  # noqa: F811
    m = len(widths)
    hp = random_pack(m, 24, d_out, seed=7, depth=(1, 2), dropout=dropout)
    hp["width"], hp["depth"] = widths, np.resize(np.array(depth, dtype=np.int32), m)
    pk, orc = pair(tp, "multiclass", 24, d_out, hp, "bf16", 256)
    X, y = make_data("multiclass", 400, 24, d_out, 3)
    idx = np.random.default_rng(5).choice(400, B, replace=False).astype(np.int32)
    Xd, yd, idxd = to_dev(X, y, idx)
    loss = torch.zeros(m, dtype=torch.float32, device=DEV)
    pk.forward_backward(Xd, idxd, yd, 3, loss)
    return pk, orc, hp, X, y, idx, Xd, loss.cpu().numpy()


@pytest.mark.parametrize("d_out", [2, 10, 16, 17, 32])
@pytest.mark.parametrize("B", [1, 128, 129, 256])
def test_head_against_stored_activations(tp, d_out, B):  # noqa: F811
    pk, _, hp, X, y, idx, Xd, loss = _step(tp, d_out, B, WIDTHS, [1], (0.0, 0.0))
    probs = pk.predict(Xd[torch.from_numpy(idx).long().to(DEV)].contiguous()).cpu().numpy().astype(np.float64)
    for i in range(len(WIDTHS)):
        H = pk.debug_activations(i, 0).astype(np.float64)
        W, b = (a.astype(np.float64) for a in pk.get_params(i, 1))
        z = H @ W.T + b
        assert np.all(np.abs(pk.logits(i) - z) <= 1e-5 * (np.abs(H) @ np.abs(W).T + np.abs(b))), i
        zmx = z - z.max(1, keepdims=True)
        p = np.exp(zmx) / np.exp(zmx).sum(1, keepdims=True)
        t = np.eye(d_out)[y[idx]]
        ref = -np.mean(np.sum(t * (zmx - np.log(np.exp(zmx).sum(1, keepdims=True))), 1))
        assert abs(loss[i] - ref) <= 2e-5 * max(1.0, abs(ref)), i
        d = (p - t) / B
        gW, gb = pk.get_grads(i, 1)
        assert np.all(np.abs(gW - d.T @ H) <= 2e-5 * ((p + t).T / B @ np.abs(H)) + 1e-12), i
        assert np.all(np.abs(gb - d.sum(0)) <= 2e-5 * (p + t).sum(0) / B + 1e-12), i
        assert np.all(np.abs(probs[i] - p) <= 3e-5), i


@pytest.mark.parametrize("d_out,B", [(2, 200), (16, 256), (19, 129), (32, 256)])
@pytest.mark.parametrize("colsum", [0, 1])
def test_head_step_against_oracle(tp, d_out, B, colsum):  # noqa: F811
    """dZ through the hidden layers; colsum: the last hidden layer's bias
    gradient from the head's column sums of dZ (widths 256 and 512)."""
    widths = np.array([256, 512, 256, 512] if colsum else [16, 80, 144, 336], dtype=np.int32)
    m = len(widths)
    hp = random_pack(m, 24, d_out, seed=9, depth=(2, 2), dropout=(0.0, 0.3))
    hp["width"], hp["depth"] = widths, np.full(m, 2, dtype=np.int32)
    pk, orc = pair(tp, "multiclass", 24, d_out, hp, "bf16", 256)
    pk.debug_bias_path(colsum)
    X, y = make_data("multiclass", 400, 24, d_out, 3)
    idx = np.random.default_rng(5).choice(400, B, replace=False).astype(np.int32)
    Xd, yd, idxd = to_dev(X, y, idx)
    loss = torch.zeros(m, dtype=torch.float32, device=DEV)
    pk.forward_backward(Xd, idxd, yd, 3, loss)
    orc.train_step(X, idx, y, 3, update=False)
    problems = compare_step(pk, orc, hp, "bf16", loss.cpu().numpy())
    assert not problems, problems


@pytest.mark.parametrize("d_out", [10, 20])
def test_head_sums_keep_fp32_precision(tp, d_out):  # noqa: F811
    """Sums over 1024 and 2048 columns and 2048 rows are as close to fp64 as
    fp32 additions are: k roundings to nearest of partial sums no larger than
    the result leave 0.58 sqrt(k) 2^-24 of it (norm-wise); 4 2^-24 covers 48 of
    them.  (Accumulators that cut off instead lose 10^-8 per instruction of a
    chain: over 2048 columns 1.4e-6.)"""
    widths, B = [1024, 2048], 2048
    rng = np.random.default_rng(1)
    pk = tp.Pack(64, d_out, "multiclass", [1, 1], widths, [0.0] * 2, [1e-3] * 2, [0.0] * 2, B, seed=3)
    for i, w in enumerate(widths):
        pk.set_params(i, 0, rng.standard_normal((w, 64)) * np.sqrt(2 / 64), 0.1 * rng.standard_normal(w))
        pk.set_params(i, 1, rng.standard_normal((d_out, w)) * np.sqrt(2 / w), 0.1 * rng.standard_normal(d_out))
    X, y = make_data("multiclass", B, 64, d_out, 3)
    Xd, yd = to_dev(X, y)
    loss = torch.zeros(2, dtype=torch.float32, device=DEV)
    pk.forward_backward(Xd, torch.arange(B, dtype=torch.int32, device=DEV), yd, 0, loss)
    probs = pk.predict(Xd).cpu().numpy().astype(np.float64)

    def off(got, ref):
        return np.linalg.norm(got - ref) / np.linalg.norm(ref)

    for i in range(2):
        H = pk.debug_activations(i, 0).astype(np.float64)
        W, b = (a.astype(np.float64) for a in pk.get_params(i, 1))
        z = H @ W.T + b
        e = np.exp(z - z.max(1, keepdims=True))
        p = e / e.sum(1, keepdims=True)
        d = (p - np.eye(d_out)[y]) / B
        gW, gb = pk.get_grads(i, 1)
        errs = [off(a, r) for a, r in ((pk.logits(i), z), (probs[i], p), (gW, d.T @ H), (gb, d.sum(0)))]
        assert max(errs) <= 4 * 2.0 ** -24, (i, errs)


@pytest.mark.parametrize("d_out", [3, 20])
@pytest.mark.parametrize("value", [-np.inf, -3.4e38, -3.38e38, 3.4e38])
def test_head_weights_at_the_ends_of_the_range(tp, d_out, value):  # noqa: F811
    """A head weight past bf16's largest number (3.39e38) or infinite acts on
    its own class as in fp32 arithmetic: the class gets probability 0 (or 1)
    and the others share the rest."""
    pk = tp.Pack(8, d_out, "multiclass", [1], [80], [0.0], [0.0], [0.0], 128)
    pk.set_params(0, 0, np.zeros((80, 8)), np.full(80, 1.0))
    rng = np.random.default_rng(0)
    W, b = 0.1 * rng.standard_normal((d_out, 80)), 0.1 * rng.standard_normal(d_out)
    W[1, 7] = value
    pk.set_params(0, 1, W, b)
    z = W.astype(np.float32).astype(np.float64).sum(1) + b.astype(np.float32)     # every activation is 1
    p = np.exp(z - z.max()) / np.exp(z - z.max()).sum()
    X, idx = torch.zeros(5, 8, device=DEV), torch.arange(5, dtype=torch.int32, device=DEV)
    probs = pk.predict(X).cpu().numpy()[0]
    assert np.all(np.abs(probs - p) <= 1e-6)
    loss = torch.zeros(1, dtype=torch.float32, device=DEV)
    pk.forward_backward(X, idx, torch.full((5,), 1 if value > 0 else 2, dtype=torch.int32, device=DEV), 0, loss)
    assert abs(loss.item() + np.log(p[1 if value > 0 else 2])) <= 1e-5
    fin = np.isfinite(z)
    assert np.all(pk.logits(0)[:, ~fin] == z[~fin])
    assert np.all(np.abs(pk.logits(0)[:, fin] - z[fin]) <= 1e-5 * np.abs(z[fin]))
