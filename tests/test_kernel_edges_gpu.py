"""Kernels and dispatch branches at the sizes where they can go wrong (tile and stage edges,
remainders, the ends of their ranges), bit for bit against the oracle."""

import numpy as np
import pytest

import oracle
from paper_1401_8288_gb300 import synth, xcorr

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    t = pytest.importorskip("torch")
    if not t.cuda.is_available():
        pytest.skip("needs a CUDA device")
    return t


@pytest.mark.parametrize("variant", [4, 5, 6, 10])
@pytest.mark.parametrize("n_sta,n_chan,n_time", [(8, 3, 129), (32, 9, 300), (72, 2, 65), (136, 2, 257)])
def test_adding_launch_of_the_fused_kernel(torch, variant, n_sta, n_chan, n_time):
    """A second and third execute add into sums that are there: full and ragged tiles, odd row
    alignments, packed channels, and (variant 10) the time-split form."""
    x = synth.uniform_ci4(3 * n_time, n_chan, n_sta, seed=n_sta + n_time, lo=-8, hi=7)
    xd = torch.from_numpy(x).cuda()
    with xcorr.Plan(n_sta, n_chan, n_time, fmt="ci4", engine="tensor") as plan:
        plan.set_tuning(variant, 0, 2, 0)
        for k in range(3):
            plan.execute(xd[k * n_time:(k + 1) * n_time].clone())
        got = plan.dump().cpu().numpy()
        plan.sync()
    assert np.array_equal(got.astype(np.int64), oracle.correlate(oracle.FMT_CI4, x))
