"""The fitting step at 16 student lobes with teachers of more than four (directions read from L1 whatever
their number), against the step over the same directions given twice: the same mean. FP32 sums over up to
600 terms: under sqrt(600) 2^-24 = 1.5e-6 relative each; 1e-5 relative L2 per plane of the first moments, and
of the loss."""
import numpy as np
import pytest

from tests._parity import rel_l2

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lt,n,count", [(8, 301, 7), (16, 77, 64), (8, 40, 300)])
def test_directions_given_twice(lib, lt, n, count):
    import torch
    from paper_2606_09794_gb300 import inputs
    t = inputs.device_point_cloud(n, lt, 61, "cuda")
    dirs = torch.from_numpy(inputs.fit_directions(1, 62, count)).cuda()
    out = []
    for d in (dirs, torch.cat([dirs, dirs])):
        s = inputs.device_point_cloud(n, 16, 63, "cuda")
        st = lib.TrainState(s["params"], s["c0"])
        loss = lib.nasgabor_fit_step(st, t["params"], t["c0"], lt, d.contiguous(), 16, 1)
        lib.nasg_device_status()
        out.append((float(loss), st.m.cpu().numpy(), st.c0_m.cpu().numpy()))
    (la, ma, ca), (lb, mb, cb) = out
    assert la > 0 and abs(la - lb) <= 1e-5 * la
    assert rel_l2(ca, cb) <= 1e-5
    for p in range(10):
        assert np.abs(ma[p]).max() > 0 and rel_l2(ma[p], mb[p]) <= 1e-5, p
