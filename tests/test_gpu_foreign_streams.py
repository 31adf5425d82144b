"""Streams that the format allows and the encoder does not write, made by hand:
pc_streams_deserialize accepts them, and retrieval gives the oracle's values."""
import struct

import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

PLANES = {np.float32: 32, np.float64: 64}
EXP_BITS, EXP_BIAS = {np.float32: 8, np.float64: 11}, {np.float32: 126, np.float64: 1022}
EXP_MIN, EXP_MAX = {np.float32: -125, np.float64: -1021}, {np.float32: 128, np.float64: 1024}


def _lowest(dtype, log_tau, emax, esc):
    """Scale exponent and lowest coded plane of a 3D block (R6, R10)."""
    s = PLANES[dtype] - 8 - emax
    return s, min(max(log_tau + s - 4 - esc, 0), PLANES[dtype])


def _block(dtype, log_tau, emax, esc, u=None):
    """Bits of a CODED 3D block, as '0'/'1' characters; u: its coefficients in
    negabinary and coded order, None for a block without a non-empty plane."""
    p = _lowest(dtype, log_tau, emax, esc)[1]
    w = EXP_BITS[dtype]
    head = "10" + format(esc, "03b")[::-1] + format(emax + EXP_BIAS[dtype], f"0{w}b")[::-1]
    if u is None:
        return head + "0" * (PLANES[dtype] - p)
    words, n = O.encode_planes(u, 64, PLANES[dtype], p)
    return head + O.bits_to_str(words, n)


def _serialized(head, tau, comps):
    """The byte form of a 3D stream (header `head`) whose component i has the
    blocks comps[i]."""
    nb = len(comps[0])
    records, data = b"", b""
    for t, blocks in zip(tau, comps):
        words, first = [], []
        for c in range(0, nb, 32):
            first.append(sum(len(w) for w in words))
            bits = "".join(blocks[c:c + 32])
            words.append(O.str_to_bits(bits + "0" * (-len(bits) % 64))[0])
        records += struct.pack("<dQ5Qd", t, sum(len(w) for w in words), 0, nb, 0, 0, 0, 0.0)
        data += np.array(first, dtype=np.uint64).tobytes()
        data += np.array([len(b) for b in blocks], dtype=np.uint16).tobytes() + b"\0" * (-2 * nb % 8)
        data += np.concatenate(words).tobytes()
    return head + records + data


@pytest.mark.parametrize("dtype,log_tau", [(np.float32, -116), (np.float32, -112), (np.float32, 0), (np.float32, 90),
                                           (np.float64, -1000), (np.float64, 0), (np.float64, 900)])
def test_coded_blocks_without_planes(dtype, log_tau):
    # beside one ordinary block of few planes (the short decodings) in each 8:
    # blocks of every exponent whose coded planes are all empty decode to 0
    # whatever their scale
    import paper_2308_11759_gb300 as P

    rng = np.random.default_rng(31)
    ordinary = PLANES[dtype] - 8 - (10 - log_tau)  # the exponent whose lowest plane is 6
    _, p = _lowest(dtype, log_tau, ordinary, 0)
    assert p == 6
    tau = [2.0 ** (log_tau + 1), 2.0 ** log_tau]

    def some(lt):  # digits in planes p .. p + 6
        low = _lowest(dtype, lt, ordinary, 0)[1]
        return [int(v) << low for v in rng.integers(0, 128, 64)]

    exps = range(EXP_MIN[dtype], EXP_MAX[dtype] + 1, 1 if dtype == np.float32 else 9)
    empty = [(e, esc) for e in exps for esc in (0, 1, 4, 7)]
    empty += empty[:-len(empty) % 7]
    blocks = []
    for i, (e, esc) in enumerate(empty):
        if i % 7 == 0:
            blocks.append(_block(dtype, log_tau, ordinary, 0, some(log_tau)))
        blocks.append(_block(dtype, log_tau, e, esc))
    first = [_block(dtype, log_tau + 1, ordinary, 0, some(log_tau + 1)) for _ in blocks]
    shape = (4, 4, 4 * len(blocks))
    x = torch.zeros(shape, dtype=torch.float32 if dtype == np.float32 else torch.float64, device="cuda")
    st = P.Streams.deserialize(_serialized(P.compress(x, tau).serialize()[:64], tau, [first, blocks]))
    want = {1: np.empty(shape, dtype), 2: np.empty(shape, dtype)}
    for b, (f, s) in enumerate(zip(first, blocks)):
        words = np.zeros((2, 80), dtype=np.uint64)
        for i, bits in enumerate((f, s)):
            w = O.str_to_bits(bits)[0]
            words[i, :len(w)] = w
        for k in (1, 2):
            v = O.decode_brick(dtype, 3, tau, k, words, np.array([len(f), len(s)]))
            want[k][:, :, 4 * b:4 * b + 4] = v.reshape(4, 4, 4)
    assert not np.isnan(want[2]).any()
    for k in (1, 2):
        got = st.retrieve(k=k).cpu().numpy()
        assert np.array_equal(got.view(np.uint8), want[k].view(np.uint8))
    st.close()


# Every decoding of the 3D retrieval -- 8, 16, 20 and 32 planes aligned to the
# highest, and any -- with digits up to the largest, whose values wrap as the
# oracle's do, at scales on both sides of the common range: 8 blocks of one kind
# together, then the same blocks in any order
@pytest.mark.parametrize("dtype,log_tau", [(np.float32, 0), (np.float32, -112), (np.float32, 100), (np.float64, 0),
                                           (np.float64, -1000), (np.float64, 968)])
def test_blocks_of_any_planes(dtype, log_tau):
    import paper_2308_11759_gb300 as P

    rng = np.random.default_rng(37)
    width = PLANES[dtype]
    blocks = []
    for p in range(width):
        emax = width - 8 - (p + 4 - log_tau)
        if not EXP_MIN[dtype] <= emax <= EXP_MAX[dtype]:
            continue
        assert _lowest(dtype, log_tau, emax, 0)[1] == p
        for planes in (1, 7, 8, 9, 15, 16, 17, 19, 20, 21, 31, 32, 33, 47, 64):
            if p + planes > width:
                continue
            for i in range(8):
                few = 64 if i % 2 else 3  # (a few coefficients only: blocks that do not wrap)
                u = [(int(rng.integers(0, 1 << 63)) * 2 + int(rng.integers(0, 2))) % (1 << planes) << p
                     if r < few else 0 for r in range(64)]
                u[int(rng.integers(0, few))] |= 1 << (p + planes - 1)
                blocks.append(_block(dtype, log_tau, emax, 0, u))
    assert len(blocks) > 300
    blocks += [blocks[i] for i in rng.permutation(len(blocks))]
    shape, tau = (4, 4, 4 * len(blocks)), [2.0 ** log_tau]
    x = torch.zeros(shape, dtype=torch.float32 if dtype == np.float32 else torch.float64, device="cuda")
    st = P.Streams.deserialize(_serialized(P.compress(x, tau).serialize()[:64], tau, [blocks]))
    want = np.empty(shape, dtype)
    for b, bits in enumerate(blocks):
        words = np.zeros((1, 160), dtype=np.uint64)
        w = O.str_to_bits(bits)[0]
        words[0, :len(w)] = w
        want[:, :, 4 * b:4 * b + 4] = O.decode_brick(dtype, 3, tau, 1, words, np.array([len(bits)])).reshape(4, 4, 4)
    got = st.retrieve(k=1).cpu().numpy()
    assert np.array_equal(got.view(np.uint8), want.view(np.uint8))
    st.close()
