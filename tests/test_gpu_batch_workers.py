"""A batch's workers share the GPU: their k x k inversions take smaller launch shapes (a fourth
or half of the SMs where the steps' latency allows) and run at the same time.  The shapes do
the same operations, so the results do not depend on the number of workers, bit for bit."""
import numpy as np
import pytest
import torch

from paper_1604_08057_gb300 import binding, inputs

pytestmark = pytest.mark.gpu


# below one block's three rows; a fourth of the SMs; half of them; too many rows for either
@pytest.mark.parametrize("k", [2, 33, 160, 260, 420])
def test_results_do_not_depend_on_the_number_of_workers(k):
    wl = inputs.WORKLOADS["4x4^3"]
    u, b, xbar = inputs.make_inputs(wl)
    dev = torch.device("cuda:0")
    ut, bt, xt = (torch.tensor(a, device=dev) for a in (u, b, xbar))
    probs = [dict(u=ut, mu=0.1 * (i + 1), m_w=-1.0, b=bt[0], k=k, xbar=xt[0]) for i in range(4)]
    out = [binding.tsl_batch(probs, nworkers=n, precision="fp64", rebiorth=20, passes=1) for n in (1, 2, 4)]
    for other in out[1:]:
        for a, c in zip(out[0], other):
            assert torch.equal(a["x"], c["x"]) and torch.equal(a["dU"], c["dU"]) and a["dmu"] == c["dmu"]
            assert np.isfinite(a["dmu"])
