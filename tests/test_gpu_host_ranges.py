"""Which host arrays lj_step_host lets its kernels read and write in place:
those that lie in one pinned allocation or registration as a whole.  Only the
decision is taken here; no kernel touches the arrays."""
import ctypes
import mmap

import pytest

pytestmark = pytest.mark.gpu

PAGE = 65536   # a multiple of the host's pages


@pytest.fixture()
def decide():
    from paper_0709_3225_gb300 import lj
    fn = lj.load().lj_mapped_host
    fn.argtypes, fn.restype = [ctypes.c_void_p, ctypes.c_size_t], ctypes.c_int
    return lambda p, n: bool(fn(p, n))


@pytest.fixture()
def memory():
    m = mmap.mmap(-1, 6 * PAGE)
    m[:] = bytes(6 * PAGE)
    c = (ctypes.c_char * (6 * PAGE)).from_buffer(m)
    yield -(-ctypes.addressof(c) // PAGE) * PAGE   # five whole pages from here on
    del c
    m.close()


def _register(rt, p, n):
    assert int(rt.cudaHostRegister(p, n, 0)) == 0


def test_registrations_with_a_gap(decide, memory):
    import torch
    torch.zeros(1, device="cuda")
    rt = torch.cuda.cudart()
    assert not decide(memory, 5 * PAGE)
    _register(rt, memory, PAGE)
    _register(rt, memory + 2 * PAGE, 2 * PAGE)
    try:
        assert decide(memory, PAGE) and decide(memory + 16, PAGE - 16) and decide(memory + 2 * PAGE, 2 * PAGE)
        assert decide(memory + 3 * PAGE, PAGE)
        assert not decide(memory, PAGE + 1)              # ends in the gap
        assert not decide(memory, 3 * PAGE)              # both ends pinned, the middle not
        assert not decide(memory + PAGE, PAGE)
        assert not decide(memory + 2 * PAGE, 2 * PAGE + 1)
        assert not decide(memory + 8, 64)                # not aligned
    finally:
        for p in (memory, memory + 2 * PAGE):
            assert int(rt.cudaHostUnregister(p)) == 0
    _register(rt, memory, 5 * PAGE)
    try:
        assert decide(memory, 5 * PAGE) and decide(memory + PAGE, 3 * PAGE)
    finally:
        assert int(rt.cudaHostUnregister(memory)) == 0
    assert not decide(memory, PAGE)


@pytest.mark.parametrize("n", [1, 4096, 500009])
def test_pinned_tensors(decide, n):
    import torch
    torch.zeros(1, device="cuda")
    a = torch.empty((n, 3), dtype=torch.float64, pin_memory=True)
    assert decide(a.data_ptr(), 24 * n)
    assert not decide(torch.empty((n, 3), dtype=torch.float64).data_ptr(), 24 * n)
    assert not decide(torch.empty((n, 3), dtype=torch.float64, device="cuda").data_ptr(), 24 * n)
