"""Deactivating members across the sizes at which the work lists change shape
(AdamW's chunks shrink from 4096 to 1024 elements, fp32 products take smaller
tiles, tensor-core products narrower ones): every active set is accepted, and
the members that stay train exactly as in a pack that keeps them all -- a
member's arithmetic does not depend on the others -- while the others stand
still and report NaN."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from test_gpu_parity import DEV, make_data, tp  # noqa: E402,F401


# many head chunks beside just under 4096 x 1216 other elements: the longest chunk lists
PACKS = {
    "wide_table": (300, 20, [1] * 64, [256] * 64),
    "wide_members": (64, 10, [1] * 38, [2048] * 38),
    "two_layers": (96, 20, [2] * 64, [240] * 64),
    "ragged": (64, 14, [1 + i % 2 for i in range(16)], [512 + 16 * (i * 13 % 30) for i in range(16)]),
    "small_tiles": (16, 3, [2] * 40, [16] * 30 + [1040] * 10),
}


@pytest.mark.parametrize("prec", ["bf16", "fp32"])
@pytest.mark.parametrize("name,muon", [(n, False) for n in PACKS] + [("two_layers", True)])
def test_deactivation_one_by_one(tp, name, prec, muon):  # noqa: F811
    d_in, d_out, depth, width = PACKS[name]
    m, B = len(depth), 128
    rng = np.random.default_rng(3)
    hp = (rng.uniform(0.0, 0.3, m).astype(np.float32), np.full(m, 1e-3, np.float32), np.full(m, 1e-3, np.float32))
    full, part = (tp.Pack(d_in, d_out, "multiclass", depth, width, *hp, B, seed=5, precision=prec) for _ in range(2))
    if muon:
        for pk in (full, part):
            pk.set_muon(np.full(m, 1e-2, np.float32))
    X, y = make_data("multiclass", 300, d_in, d_out, 4)
    Xd, yd = torch.from_numpy(X).to(DEV), torch.from_numpy(y).to(DEV)
    on = np.ones(m, dtype=np.uint8)
    order = list(range(m - 1, 1, -1))
    if name == "small_tiles":
        order = list(range(0, 30)) + order[:8]     # the small members first
    loss, ref = (torch.zeros(m, dtype=torch.float32, device=DEV) for _ in range(2))
    stopped = {}
    for step, i in enumerate(order):
        stopped[i] = part.snapshot(i)
        on[i] = 0
        part.set_active(on)
        idx = torch.from_numpy(rng.choice(300, B - step % 3, replace=False).astype(np.int32)).to(DEV)
        part.train_step(Xd, idx, yd, step, loss)
        full.train_step(Xd, idx, yd, step, ref)
        act = torch.from_numpy(on.astype(bool)).to(DEV)
        assert torch.equal(loss[act], ref[act]) and bool(torch.isnan(loss[~act]).all()), (step, i)
    for j in range(m):
        want = stopped[j] if j in stopped else full.snapshot(j)
        assert torch.equal(part.snapshot(j), want), j
    # and back: all members step again
    part.set_active(np.ones(m, dtype=np.uint8))
    part.train_step(Xd, idx, yd, len(order), loss)
    assert bool(torch.isfinite(loss).all())
    assert all(not torch.equal(part.snapshot(j), stopped[j]) for j in list(stopped)[:3])
    full.close()
    part.close()
