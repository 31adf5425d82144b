"""3D RAW blocks beside ZERO and CODED ones, at every place of a stream word that
occurs, through retrieval, refinement and sub-boxes, against the oracle."""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("dtype,tau", [(np.float32, [2.0 ** -2, 2.0 ** -40]), (np.float64, [2.0 ** -2, 2.0 ** -80])])
@pytest.mark.parametrize("shape", [(8, 12, 520), (7, 10, 333), (4, 4, 4)])
def test_raw_blocks_at_any_bit(dtype, tau, shape):
    import paper_2308_11759_gb300 as P

    rng = np.random.default_rng(43)
    x = rng.standard_normal(shape)
    kind = rng.integers(0, 4, tuple(-(-s // 4) for s in shape))
    kind = np.kron(kind, np.ones((4, 4, 4), int))[tuple(slice(0, s) for s in shape)]
    x[kind == 1] = 0.0
    x[kind == 2] = np.round(x[kind == 2] * 8.0) / 8.0
    if shape == (4, 4, 4):
        x = rng.standard_normal(shape)
    x = x.astype(dtype)
    st, ref = P.compress(torch.from_numpy(x).cuda(), tau), O.Streams(x, tau)
    assert st.counts(1)[2] > 0 or shape == (4, 4, 4)  # (one brick: RAW in float32, CODED in float64)
    for k in (1, 2):
        got = st.retrieve(k=k).cpu().numpy()
        assert np.array_equal(got.view(np.uint8), ref.retrieve(k).view(np.uint8))
    assert np.array_equal(st.refine(1, 2, st.retrieve(k=1)).cpu().numpy(), ref.retrieve(2))
    lo, hi = [s // 3 for s in shape], [s - s // 4 for s in shape]
    assert np.array_equal(st.retrieve(k=2, box=(lo, hi)).cpu().numpy(),
                          ref.retrieve(2)[tuple(slice(a, b) for a, b in zip(lo, hi))])
