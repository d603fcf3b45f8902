"""A member's snapshot in recycled device memory: the alignment gaps between
its blocks are zero, as documented, whatever the memory held before."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from test_gpu_parity import tp  # noqa: E402,F401


@pytest.mark.parametrize("precision", ["bf16", "fp32"])
def test_gaps_are_zero(tp, precision):  # noqa: F811
    for _ in range(3):
        junk = [torch.full((n,), float("nan"), device="cuda") for n in (1 << 12, 1 << 16, 1 << 20, 1 << 24)]
        torch.cuda.synchronize()
        del junk
        torch.cuda.empty_cache()
        pk = tp.Pack(19, 1, "regression", [2, 3], [16, 48], [0.1, 0.0], [1e-3] * 2, [1e-3] * 2, 64, precision=precision)
        for i, (L, w) in enumerate(((2, 16), (3, 48))):
            run = pk.snapshot(i).cpu().numpy()
            off, used = 0, np.zeros(len(run), dtype=bool)
            for l in range(L + 1):
                for n in ((1 if l == L else w) * (24 if l == 0 else w), 1 if l == L else w):
                    off = -(-off // 32) * 32
                    used[off:off + n] = True
                    off += n
            assert off == len(run) and np.all(run[~used] == 0.0) and np.all(np.isfinite(run))
        pk.close()
