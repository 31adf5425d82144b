"""pc_streams_serialize into host memory of every kind a caller may pass."""
import ctypes as C
import mmap
import time

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _fresh(n):  # memory without a page behind it yet
    m = mmap.mmap(-1, n)
    return m, C.addressof(C.c_char.from_buffer(m))


def test_into_fresh_memory():
    # The bytes are those of Streams.serialize whatever the buffer's alignment,
    # and a buffer whose pages are not there yet takes no longer than filling one
    # with zeros, serializing into that and copying the bytes out (43 MB: 1.9 ms
    # against 5.7; with the device copies faulting the pages in 20 ms).
    import paper_2308_11759_gb300 as P

    g = torch.Generator(device="cuda")
    g.manual_seed(3)
    x = torch.randn((256, 256, 256), generator=g, device="cuda")
    st = P.compress(x, [1e-1, 1e-3])
    want = st.serialize()
    n = C.c_size_t(len(want))

    def call(at):
        t = time.perf_counter()
        assert P.lib().pc_streams_serialize(st._h, C.c_void_p(at), C.byref(n), None) == 0
        return time.perf_counter() - t

    fresh, filled, keep = [], [], []
    for i in range(7):
        m, at = _fresh(len(want) + 4096)
        fresh.append(call(at))
        assert m[:len(want)] == want
        keep.append(m)
        t = time.perf_counter()
        b = C.create_string_buffer(len(want))
        raw = (call(C.addressof(b)), b.raw)[1]
        filled.append(time.perf_counter() - t)
        assert raw == want
    for off in (8, 24, 4088):
        m, at = _fresh(len(want) + 4096)
        call(at + off)
        assert m[off:off + len(want)] == want and m[off + len(want):] == bytes(4096 - off) and m[:off] == bytes(off)
    assert min(fresh) <= np.median(filled), (fresh, filled)
