"""1D and 2D retrieval around whole CTAs of 128 bricks: threads past the last brick,
single and batched, from zero and refined, against the oracle."""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("bricks", [1, 2, 127, 128, 129, 257])
def test_around_whole_ctas(dtype, bricks):
    import paper_2308_11759_gb300 as P

    rng = np.random.default_rng(bricks)
    tau = [2.0 ** -3, 2.0 ** -9, 2.0 ** -14]
    sts, refs = [], []
    for shape in ((4 * bricks - 1,), (3, 4 * bricks - 2), (4 * bricks - 3, 4)):
        x = rng.standard_normal(shape).astype(dtype)
        x.reshape(-1)[::7] *= 2.0 ** -12
        st, ref = P.compress(torch.from_numpy(x).cuda(), tau), O.Streams(x, tau)
        for k in (1, 2, 3):
            assert np.array_equal(st.retrieve(k=k).cpu().numpy(), ref.retrieve(k))
        assert np.array_equal(st.refine(1, 3, st.retrieve(k=1)).cpu().numpy(), ref.retrieve(3))
        sts.append(st)
        refs.append(ref)
    order = [0, 1, 2, 1, 0, 0]
    ks = [3, 2, 1, 3, 1, 2]
    for q, k, out in zip(order, ks, P.retrieve_batch([sts[q] for q in order], ks)):
        assert np.array_equal(out.cpu().numpy(), refs[q].retrieve(k))
