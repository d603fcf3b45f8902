"""A member's snapshot in recycled device memory: the alignment gaps between
its blocks are zero, as documented, whatever the memory held before.  And into
every kind of destination: at any byte of device memory, in managed and pinned
memory; a destination that is too short is refused."""
import ctypes

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


@pytest.fixture()
def runtime():
    name = "libcudart.so.%s" % torch.version.cuda.split(".")[0]
    return ctypes.CDLL(name)


def _pack(tp):  # noqa: F811
    return tp.Pack(19, 1, "regression", [2], [48], [0.0], [1e-3], [1e-3], 64)


@pytest.mark.parametrize("shift", [0, 1, 2, 3, 4, 8, 12, 16])
def test_any_byte_address(tp, shift):  # noqa: F811
    pk = _pack(tp)
    n, L = pk.member_size(0), tp.load_library()
    want = pk.snapshot(0).cpu().numpy().tobytes()
    buf = torch.full((4 * n + 64,), 0xAB, dtype=torch.uint8, device="cuda")
    assert L.pack_snapshot(pk._h, 0, ctypes.c_void_p(buf.data_ptr() + shift)) == 0
    got = buf.cpu().numpy().tobytes()
    assert got[shift:shift + 4 * n] == want
    assert set(got[:shift] + got[shift + 4 * n:]) == {0xAB}
    pk.close()


def test_other_kinds_of_memory(tp, runtime):  # noqa: F811
    pk = _pack(tp)
    n, L = pk.member_size(0), tp.load_library()
    want = pk.snapshot(0).cpu().numpy()
    pinned = torch.zeros(n, dtype=torch.float32, pin_memory=True)
    assert L.pack_snapshot(pk._h, 0, ctypes.c_void_p(pinned.data_ptr())) == 0
    torch.cuda.synchronize()
    assert np.array_equal(pinned.numpy(), want)
    p = ctypes.c_void_p()
    assert runtime.cudaMallocManaged(ctypes.byref(p), ctypes.c_size_t(4 * n), 1) == 0
    assert L.pack_snapshot(pk._h, 0, p) == 0
    torch.cuda.synchronize()
    assert np.array_equal(np.ctypeslib.as_array(ctypes.cast(p, ctypes.POINTER(ctypes.c_float)), (n,)), want)
    runtime.cudaFree(p)
    pk.close()


def test_short_destination_is_refused(tp, runtime):  # noqa: F811
    pk = _pack(tp)
    L = tp.load_library()
    p = ctypes.c_void_p()
    assert pk.member_size(0) * 4 > 4096
    assert runtime.cudaMalloc(ctypes.byref(p), ctypes.c_size_t(4096)) == 0
    assert L.pack_snapshot(pk._h, 0, p) != 0
    runtime.cudaFree(p)
    # and the refusal is over: the next launches do not report it again
    out = pk.snapshot(0)
    assert torch.equal(out, pk.snapshot(0))
    y = torch.zeros(8, device="cuda")
    assert len(tp.select_greedy(torch.zeros(2, 8, 1, device="cuda"), y, "regression", "loss", m_ens=1)[0]) == 1
    pk.close()
