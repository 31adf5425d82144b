"""The derivative kernels where a thread's planes do not divide into the steps they
are handled in: few planes of many tiles, slices of every length, odd rows,
both kinds of spacing, against the oracle bit for bit."""
import numpy as np
import pytest

from oracle import derivatives as D

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("h", [1.0, 0.3])
@pytest.mark.parametrize("shape", [(611, 1003), (1, 90, 1001), (2, 300, 301), (3, 611, 603), (4, 600, 601), (5, 610, 603),
                                   (6, 601, 602), (7, 257, 601), (9, 600, 601), (18, 300, 601), (37, 256, 257),
                                   (70, 65, 129)])
def test_slices_of_any_length(dtype, h, shape):
    import paper_2308_11759_gb300 as P

    rng = np.random.default_rng(71)
    u, v = (rng.standard_normal(shape).astype(dtype) for _ in range(2))
    ud, vd = torch.from_numpy(u).cuda(), torch.from_numpy(v).cuda()
    assert np.array_equal(P.fd_vorticity_z(ud, vd, h).cpu().numpy(), D.vorticity_z(u, v, h))
    for axis in range(len(shape)):
        if shape[len(shape) - 1 - axis] >= 4:
            assert np.array_equal(P.fd_second(ud, axis, h).cpu().numpy(), D.second(u, axis, h)), axis
