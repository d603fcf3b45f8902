"""Greedy selection on inputs where a fast path of the kernels could go wrong:
ROC-AUC with ties, constant, saturated, skewed and non-finite predictions and
sizes around the bucket path's limits; accuracy with exact ties; squared
errors that overflow an fp32 sum; cross-entropy with and without the compact
label values.  The reference is the definition in numpy: ensemble values in
fp64, rounded to fp32, ranked or scored; integer counts make the AUC and
accuracy scores equal bit for bit."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle  # noqa: E402


@pytest.fixture(scope="module")
def tp():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2607_05380_gb300 import build
    build.build()
    import paper_2607_05380_gb300 as tpm
    tpm.load_library()
    return tpm


def _select(tp, preds, y, *a, **kw):
    return tp.select_greedy(torch.from_numpy(preds).cuda(), torch.from_numpy(y).cuda(), *a, **kw)


def _neg_auc(v, y):
    """-AUC of fp64 values rounded to fp32, ordered by their bit patterns (a
    NaN below all numbers)."""
    u = v.astype(np.float32).view(np.uint32)
    k = np.where(u >> 31, ~u, u | np.uint32(0x80000000)).astype(np.int64)
    k[np.isnan(v)] = 0
    neg = np.sort(k[y != 1])
    pos = k[y == 1]
    if not len(neg) or not len(pos):
        return np.nan
    u2 = int(np.searchsorted(neg, pos, "left").sum()) + int(np.searchsorted(neg, pos, "right").sum())
    return -(0.5 * u2 / (float(len(pos)) * float(len(neg))))


def _neg_acc(v, y):
    pred = np.argmax(v, 1) if v.shape[1] > 1 else (v[:, 0] > 0.5).astype(np.int64)
    return -(float(np.sum(pred == y)) / len(y))


def _greedy(preds, y, m_ens, score):
    S, sel, best = np.zeros(preds.shape[1:]), [], np.inf
    while len(sel) < m_ens:
        inv = 1.0 / (len(sel) + 1)
        sc = [np.nan if c in sel else score((S + preds[c].astype(np.float64)) * inv, y) for c in range(len(preds))]
        k = min((c for c in range(len(sc)) if sc[c] == sc[c]), key=lambda c: (sc[c], c), default=None)
        if k is None or not sc[k] < best:
            break
        best = sc[k]
        sel.append(k)
        S = S + preds[k].astype(np.float64)
    return sel, best


def _auc_preds(kind, P, N, rng, y):
    z = rng.standard_normal((P, N)) + 0.7 * (y == 1)
    p = 1 / (1 + np.exp(-z))
    if kind == "ties":
        p = np.round(p * 16) / 16
    elif kind == "const":
        p[:] = 0.25
    elif kind == "saturated":
        p = np.where(z > 1.0, 1.0, np.where(z < -0.5, 0.0, p))
    elif kind == "skew":
        p = np.exp(-30 * rng.uniform(0, 1, (P, N))) * (1 + 0.1 * (y == 1))
    elif kind == "signed":      # values around zero, of very different sizes
        p = z * 10.0 ** rng.integers(-6, 6, (P, 1))
    p = p.astype(np.float32)
    if kind == "nonfinite":
        p[1, :: max(1, N // 3)] = np.inf
        p[2, 0] = np.nan
        p[3, -1] = -np.inf
    return p


@pytest.mark.parametrize("kind", ["plain", "ties", "const", "saturated", "skew", "signed", "nonfinite", "rare"])
@pytest.mark.parametrize("N", [1, 2, 15, 16, 17, 1025, 30001])
def test_auc(tp, kind, N):
    rng = np.random.default_rng(N)
    y = (rng.uniform(size=N) < (0.01 if kind == "rare" else 0.4)).astype(np.int32)
    preds = _auc_preds(kind, 5, N, rng, y)
    with np.errstate(invalid="ignore"):
        ref, best = _greedy(preds[:, :, None], y, 4, lambda v, yy: _neg_auc(v[:, 0], yy))
    for static in (False, True):
        sel, fin = _select(tp, preds[:, :, None].copy(), y, "binary", "auc", m_ens=4, static_scratch=static)
        assert list(sel) == ref and (fin == best or not ref), (list(sel), ref, fin, best)


@pytest.mark.parametrize("size", [1e-25, 1e-30, 1e-35, 1e-38, 1e-40, 1e-43])
@pytest.mark.parametrize("N", [15, 4001, 90001])
def test_auc_of_tiny_values(tp, size, N):
    """Scores near the bottom of the fp32 range (a confident sigmoid's), a few
    units in the last place apart: averaged in fp64 and rounded once, their
    order and ties decide the AUC to the last pair."""
    rng = np.random.default_rng(1)
    y = (rng.uniform(size=N) < 0.4).astype(np.int32)
    y[:2] = [0, 1]
    step = 3e-6 if size > 1e-39 else 1.0
    preds = (size * (1 + step * (rng.integers(0, 8, (5, N)) + (y == 1)))).astype(np.float32)
    preds[:, ::7] = 0.0
    ref, best = _greedy(preds[:, :, None], y, 4, lambda v, yy: _neg_auc(v[:, 0], yy))
    sel, fin = _select(tp, preds[:, :, None].copy(), y, "binary", "auc", m_ens=4)
    assert list(sel) == ref and fin == best, (list(sel), ref, fin, best)


# the smaller class valued once up to 79873 rows, beside the buckets in shared memory, or not
@pytest.mark.parametrize("N", [79873, 79874, 200003])
@pytest.mark.parametrize("kind", ["plain", "ties"])
def test_auc_large(tp, kind, N):
    rng = np.random.default_rng(N)
    y = rng.integers(0, 2, N).astype(np.int32)
    preds = _auc_preds(kind, 4, N, rng, y)
    ref, best = _greedy(preds[:, :, None], y, 3, lambda v, yy: _neg_auc(v[:, 0], yy))
    sel, fin = _select(tp, preds[:, :, None].copy(), y, "binary", "auc", m_ens=3)
    assert list(sel) == ref and fin == best


@pytest.mark.parametrize("P", [1, 7, 8, 9, 19])
@pytest.mark.parametrize("d_out,N", [(1, 1), (1, 1024), (1, 3001), (2, 255), (10, 1025), (32, 2049)])
def test_accuracy_with_exact_ties(tp, P, d_out, N):
    """Multiples of 1/8: averages land on 1/2 and classes tie exactly."""
    rng = np.random.default_rng(P + N)
    preds = (rng.integers(0, 9, (P, N, d_out)) / 8).astype(np.float32)
    preds[P // 2, :, 0] += np.float32(2.0 ** -24)     # nearly tied
    preds[-1] = preds[0]                              # a duplicate: the lower index wins
    y = rng.integers(0, max(2, d_out), N).astype(np.int32)
    ref, best = _greedy(preds, y, 5, _neg_acc)
    sel, fin = _select(tp, preds, y, "binary" if d_out == 1 else "multiclass", "accuracy", m_ens=5)
    assert list(sel) == ref and fin == best, (list(sel), ref, fin, best)


@pytest.mark.parametrize("P,N,m_ens", [(1, 1, 1), (9, 1023, 5), (17, 3001, 1), (17, 3001, 6)])
def test_cross_entropy_label_values(tp, P, N, m_ens):
    """m_ens = 1 and the static variant read the predictions, more iterations
    the compact label values: the same selection; an invalid label leaves no
    score."""
    rng = np.random.default_rng(P)
    lg = rng.standard_normal((P, N, 7)) * 2
    preds = (np.exp(lg) / np.exp(lg).sum(-1, keepdims=True)).astype(np.float32)
    y = rng.integers(0, 7, N).astype(np.int32)
    preds[-1] = preds[P // 2]
    a = _select(tp, preds, y, "multiclass", "loss", m_ens=m_ens)
    b = _select(tp, preds, y, "multiclass", "loss", m_ens=m_ens, static_scratch=True)
    osel, ofin, obest, ogap = oracle.greedy(preds, y, "multiclass", "loss", m_ens=m_ens, fp32_terms=True)
    assert list(a[0]) == list(b[0]) and a[1] == b[1]
    k = next((j for j, (s, o) in enumerate(zip(a[0], osel)) if s != o), None)
    assert k is None and len(osel) == len(a[0]) or ogap[k or 0] <= 1e-6
    assert k is not None or abs(a[1] - ofin) <= 1e-6 * max(1.0, abs(ofin))
    y[N // 2] = 7
    assert len(_select(tp, preds, y, "multiclass", "loss", m_ens=m_ens)[0]) == 0


@pytest.mark.parametrize("size", [1.0, 3e18, 1e-20])
def test_squared_error_range(tp, size):
    """Squares near the ends of the fp32 range: 3e18 squared is 9e36, whose
    sum over 1024 rows overflows fp32; the score is an fp64 sum of fp32 terms."""
    rng = np.random.default_rng(5)
    N = 2500
    y = (size * rng.standard_normal(N)).astype(np.float32)
    preds = (y[None, :, None] + (size * rng.standard_normal((6, N, 1))).astype(np.float32)).astype(np.float32)

    def mse(v, yy):
        d = v[:, 0].astype(np.float32) - yy
        return float(np.mean((d * d).astype(np.float64)))

    ref, best = _greedy(preds, y, 4, mse)
    sel, fin = _select(tp, preds, y, "regression", "loss", m_ens=4)
    assert list(sel) == ref and abs(fin - best) <= 1e-12 * best   # sums of 2500 terms in fp64 and in two fp32 numbers
