"""Kernel variants and dispatch rules at the sizes where they change: against
the oracle, numpy or the general path, bit for bit."""
import numpy as np
import pytest

import oracle as O
import synth_fields as S
from oracle import derivatives as D
from tests.gpu_helpers import parse_serialized

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def P():
    import paper_2308_11759_gb300 as pcz

    pcz.lib()
    return pcz


def _bits(a):
    a = np.ascontiguousarray(a)
    return a.view(np.uint32 if a.dtype == np.float32 else np.uint64)


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("n", [1, 2, 3, 5, 17, 1023, 4097, 100003])
@pytest.mark.parametrize("off", [0, 1, 3])
def test_range_of_any_length_and_alignment(P, dtype, n, off):
    rng = np.random.default_rng(1000 * n + off)
    x = (rng.standard_normal(n) * 2.0 ** rng.integers(-60, 60, n)).astype(dtype)
    buf = torch.empty(n + off, dtype=torch.float32 if dtype == np.float32 else torch.float64, device="cuda")
    view = buf[off:]
    for at in (0, n // 2, n - 1):  # an extreme at the head, in the middle and at the tail
        for sign in (1, -1):
            y = x.copy()
            y[at] = sign * dtype(3e30)
            view.copy_(torch.from_numpy(y))
            assert P.field_range(view) == (float(y.min()), float(y.max()))
        for bad in (np.inf, -np.inf, np.nan, -np.nan):
            y = x.copy()
            y[at] = bad
            view.copy_(torch.from_numpy(y))
            with pytest.raises(P.PczError) as e:
                P.field_range(view)
            assert e.value.name == "PC_ERR_NONFINITE"


@pytest.mark.parametrize("n", [1, 3, 8])
def test_units_of_every_size_give_the_same(P, n):
    # 128 x 130 x 127: enough bricks for units of several pairs per warp; the
    # sub-boxes below it take smaller ones
    x = torch.from_numpy(S.powerlaw((127, 130, 128), seed=77, dtype=np.float32)).cuda()
    st = P.compress(x, P.field_tau_schedule(x, "decade", n))
    for k in {1, n}:
        full = st.retrieve(k=k)
        for lo, hi in (([0, 0, 0], [64, 130, 128]), ([64, 0, 0], [127, 130, 128]), ([3, 5, 7], [4, 6, 8]),
                       ([1, 2, 3], [40, 39, 41])):
            part = st.retrieve(k=k, box=(lo, hi))
            sl = tuple(slice(a, b) for a, b in zip(lo, hi))
            assert torch.equal(part, full[sl])
        boxes = [([0, 0, 0], [127, 130, 128]), ([100, 100, 100], [101, 102, 103]), ([8, 8, 8], [72, 72, 72])]
        outs = P.retrieve_batch([st] * 3, [k] * 3, boxes)
        for (lo, hi), o in zip(boxes, outs):
            assert torch.equal(o, full[tuple(slice(a, b) for a, b in zip(lo, hi))])


@pytest.mark.parametrize("h", [0.5, 1.0, 2.0 ** -500, 2.0 ** 400, 0.3])
def test_derivatives_outside_the_normal_range(P, h):
    # zeros, subnormals, values near the largest and infinities beside ordinary
    # ones: the float64 kernels scale exponent fields and redo such values
    shape = (9, 11, 70)
    rng = np.random.default_rng(5)
    def field():
        f = rng.standard_normal(shape)
        pick = rng.integers(0, 12, shape)
        f[pick == 0] = 0.0
        f[pick == 1] = -0.0
        f[pick == 2] *= 2.0 ** -1060
        f[pick == 3] *= 2.0 ** 1020
        f[(pick == 4) & (rng.random(shape) < 0.1)] = np.inf
        f[:, 4:6] = 1.25  # equal neighbours: exact zeros
        return f
    u, v = field(), field()
    with np.errstate(all="ignore"):
        want = [D.vorticity_z(u, v, h)] + [D.second(u, a, h) for a in range(3)]
    ud, vd = torch.from_numpy(u).cuda(), torch.from_numpy(v).cuda()
    got = [P.fd_vorticity_z(ud, vd, h)] + [P.fd_second(ud, a, h) for a in range(3)]
    for w, g in zip(want, got):
        g = g.cpu().numpy()
        nan = np.isnan(w)
        assert np.array_equal(nan, np.isnan(g))
        assert np.array_equal(_bits(w)[~nan], _bits(g)[~nan])


# components whose coded planes span at most 8, 16 and 32 planes and more, at
# block scales on both sides of the common range (float32 s in [-96, 126],
# float64 [-960, 1000]; s = 24 or 56 minus the block exponent) and of the
# 32-bit decode-back of float64
@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("exp", ["low", "low+", "mid", "high-", "high"])
@pytest.mark.parametrize("rel", [[0.25, 2.0 ** -4], [2.0 ** -9, 2.0 ** -14], [2.0 ** -20], [2.0 ** -45]])
@pytest.mark.parametrize("shape", [(9, 10, 37), (21, 37), (203,)])
def test_construction_by_span_and_scale(P, dtype, exp, rel, shape):
    e = {np.float32: {"low": -103, "low+": -99, "mid": 3, "high-": 117, "high": 121},
         np.float64: {"low": -946, "low+": -940, "mid": 3, "high-": 1012, "high": 1017}}[dtype][exp]
    x = np.ldexp(S.powerlaw(shape, seed=61, dtype=np.float64) / 4.0, e).astype(dtype)
    tau = [float(np.ldexp(r, e)) for r in rel]
    st, ref = P.compress(torch.from_numpy(x).cuda(), tau), O.Streams(x, tau, nthreads=4)
    d = parse_serialized(st.serialize())
    for i in range(len(tau)):
        c = d["comps"][i]
        assert np.array_equal(c["brick_len"], ref.brick_len(i))
        assert np.array_equal(c["payload"], ref.payload(i))
        assert c["counts"] == [int(v) for v in ref.stats(i)]
        assert c["measured"] == ref.measured(i)
    got = st.retrieve(k=len(tau)).cpu().numpy()
    assert np.array_equal(_bits(got), _bits(ref.retrieve(len(tau))))


# results of a server batch written into the callers' buffers: buffers that
# start at any byte of an allocation, 140 of them (more than one list of
# copies holds), some without a buffer; buffers shared by two queries
# (the later one's result stays: the boxes all hold the field's centre, so
# batches wait for one another)
@pytest.mark.parametrize("where", ["apart", "shared"])
def test_server_results(P, where):
    x = torch.from_numpy(S.powerlaw((40, 44, 52), seed=67, dtype=np.float32)).cuda()
    st = P.compress(x, [0.1, 0.01, 0.001])
    rng = np.random.default_rng(68)
    qs, off, at = [], [], 0
    for i in range(140):
        lo = [int(rng.integers(0, s // 2)) for s in x.shape]
        hi = [int(rng.integers(s // 2 + 1, s + 1)) for s in x.shape]
        qs.append((0, (lo, hi), 0.0, int(rng.integers(1, 4))))
        at += int(rng.integers(0, 9)) * 4 if i % 3 else int(rng.integers(0, 300))
        off.append(at)
        at += 4 * int(np.prod([h - l for l, h in zip(lo, hi)]))
    memory = torch.full((at + 64,), 7, dtype=torch.uint8, device="cuda")
    if where == "shared":
        off = [off[i - 1] if i and i % 4 == 0 else o for i, o in enumerate(off)]

    class Out:  # a buffer at any byte address (a tensor's must be a multiple of its type)
        def __init__(self, p):
            self.p = p

        def data_ptr(self):
            return self.p

    outs = [None if i % 11 == 10 else Out(memory.data_ptr() + o) for i, o in enumerate(off)]
    want = memory.cpu().numpy().copy()
    for q, o, out in zip(qs, off, outs):
        if out is not None:
            b = st.retrieve(k=q[3], box=q[1]).cpu().numpy().view(np.uint8).reshape(-1)
            want[o:o + b.size] = b
    srv = P.Server(1 << 30)
    srv.add_field(st)
    srv.replay(qs[:1], [0.0], None)  # (starts the dispatcher)
    srv.replay(qs, [0.0] * len(qs), outs)
    torch.cuda.synchronize()
    srv.close()
    assert np.array_equal(memory.cpu().numpy(), want)
