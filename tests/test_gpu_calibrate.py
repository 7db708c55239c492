"""Column maxima of the calibration rows and the weight rows taken by one launch: the split of the blocks between the two matrices
and the last, partly filled pass of a block."""
import numpy as np
import pytest
import torch

import oracle
import paper_2509_21302_b200 as q
import workload
from _util import dev_bf16

pytestmark = pytest.mark.gpu


# a pass of a block is 16 rows (K = 1024) or 4 rows (K = 4096); 296 blocks on 148 SMs
@pytest.mark.parametrize("K,N,rows", [(1024, 15, 16), (1024, 17, 1), (1024, 1, 20011), (1024, 9000, 3), (4096, 3, 4), (4096, 5, 1), (4096, 1, 5003), (4096, 2999, 2)])
def test_column_maxima_at_the_edges_of_the_split(K, N, rows):
    spec = workload.LinearSpec("c", K, N, workload.DIST_NORMAL, 11, 0)
    Xc, W = spec.x_calib(rows), spec.weight()
    x, w = dev_bf16(Xc), dev_bf16(W)
    scratch = torch.full((2 * K,), 7.0, dtype=torch.float32, device="cuda")
    c = torch.empty(K, dtype=torch.float32, device="cuda")
    st = q.lib().qvggt_calibrate_smooth(x.data_ptr(), rows, w.data_ptr(), N, K, 0.5, 0.01, 100.0, scratch.data_ptr(), c.data_ptr(),
                                        torch.cuda.current_stream().cuda_stream)
    assert st == 0
    got = scratch.cpu().numpy().reshape(2, K)
    # the fp32 butterflies in the stated order and a power-of-two factor: the maxima are exact
    for g, m in zip(got, (Xc, W)):
        want = np.zeros(K, np.float32)
        for r in m:
            want = np.maximum(want, np.abs(oracle.fwht_f32(oracle.bf16_to_f32(r))))
        assert np.array_equal(g, want * np.float32(K ** -0.5))
