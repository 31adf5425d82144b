"""Retrieval units of one to four sets of 32 bricks, with plane words that fit in
shared memory and with ones that spill: the same values as small boxes, whose
units are one set, and at a corner as the oracle.  A child process repeats it
with the debug library, whose bounds checks must stay clean."""
import os
import subprocess
import sys

import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CTAS = {np.float32: 7, np.float64: 5}  # of the retrieval kernel per SM
POOL = 1792                            # plane words that fit in shared memory

# tolerances relative to the field's scale; the first number is the sets of a unit
# where there are bricks enough.  The wide ones have more plane words than fit.
SCHEDULES = {
    np.float32: {"one": (4, [2.0 ** -6]), "two": (3, [2.0 ** -4, 2.0 ** -8]), "three": (2, [2.0 ** -3, 2.0 ** -6, 2.0 ** -9]),
                 "wide": (4, [2.0 ** -20]), "two wide": (3, [2.0 ** -14, 2.0 ** -21])},
    np.float64: {"one": (4, [2.0 ** -6]), "two": (3, [2.0 ** -4, 2.0 ** -8]), "three": (2, [2.0 ** -3, 2.0 ** -6, 2.0 ** -9]),
                 "wide": (4, [2.0 ** -40]), "two wide": (3, [2.0 ** -20, 2.0 ** -40]),
                 "three wide": (2, [2.0 ** -14, 2.0 ** -28, 2.0 ** -42]),
                 "seven wide": (1, [2.0 ** (-7 * i) for i in range(1, 8)])},
}


def _shape(bricks):  # odd extents of at least (at most a layer more than) `bricks` bricks
    n = int(bricks ** (1 / 3))
    return (4 * -(-bricks // (n * n)) - 1, 4 * n - 2, 4 * n - 3)


def _same(a, b):
    return np.array_equal(a.cpu().numpy().view(np.uint8), b.cpu().numpy().view(np.uint8))


@pytest.mark.parametrize("dtype,schedule", [(t, s) for t in SCHEDULES for s in SCHEDULES[t]])
def test_units_of_several_sets(dtype, schedule):
    import paper_2308_11759_gb300 as P

    most, tau = SCHEDULES[dtype][schedule]
    n = len(tau)
    wave = 32 * CTAS[dtype] * torch.cuda.get_device_properties(0).multi_processor_count
    g = torch.Generator(device="cuda")
    g.manual_seed(41)
    for sets in range(1, most + 1):
        for bricks in ((sets + 1) * wave - 2000, sets * wave + 10):  # the same units' upper and lower end
            shape = _shape(bricks if sets < most else sets * wave + 10)
            x = torch.randn(shape, generator=g, device="cuda", dtype=torch.float32 if dtype == np.float32 else torch.float64)
            x[:, :5] *= 2.0 ** -12  # blocks of other lengths beside the first ones
            st = P.compress(x, tau)
            if "wide" in schedule and sets == most:
                # a block of length l has at least (l - 200) / 65 planes
                planes = sum((st.info(i)[1] / (-(-shape[0] // 4) * -(-shape[1] // 4) * -(-shape[2] // 4)) - 200) / 65
                             for i in range(n))
                assert 32 * most * planes > POOL or n > 6
            corner = O.Streams(np.ascontiguousarray(x[:12, :16, :20].cpu().numpy()), tau)
            for k in sorted({1, n}):
                full = st.retrieve(k=k)
                for z in range(0, shape[0], 16):  # slabs: one set per unit
                    hi = min(z + 16, shape[0])
                    assert _same(full[z:hi], st.retrieve(k=k, box=([z, 0, 0], [hi, shape[1], shape[2]]))), (shape, k, z)
                assert np.array_equal(full[:12, :16, :20].cpu().numpy(), corner.retrieve(k))
                if k > 1:
                    assert _same(st.refine(1, k, st.retrieve(k=1)), full)
            both = P.retrieve_batch([st, st], [1, n], [None, ([1, 2, 3], [shape[0] - 1, shape[1], shape[2] - 2])])
            assert _same(both[0], st.retrieve(k=1))
            assert _same(both[1], st.retrieve(k=n)[1:shape[0] - 1, 2:, 3:shape[2] - 2].contiguous())
            st.close()
            if sets == most:
                break
    word, debug = P.debug_status()
    assert not debug or word == 0, hex(word)


def test_units_with_bounds_checks():
    from paper_2308_11759_gb300 import build as B

    B.build(debug=True)
    env = dict(os.environ, PCZ_LIBRARY=B.LIB_DEBUG)
    r = subprocess.run([sys.executable, "-m", "pytest", "-q", "-x", "-p", "no:cacheprovider", os.path.abspath(__file__), "-k",
                        "several_sets and wide"], capture_output=True, text=True, env=env, cwd=ROOT, timeout=900)
    assert r.returncode == 0 and "6 passed" in r.stdout, r.stdout[-3000:] + r.stderr[-3000:]
