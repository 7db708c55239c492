"""How the TMA-fed GEMM deals its tiles: shapes whose tiles fill no round, one, or several rounds of the chip's CTA pairs, whose
remainder is cut into pieces of 1 to 4 units of 64 channels, and whose row tiles are not a whole number of 256-channel tiles.
The whole result is compared with the packed GEMM's (another kernel, another tiling), sampled rows with the oracle, bit for bit."""
import numpy as np
import pytest
import torch

import oracle
import paper_2509_21302_b200 as q
import workload
from _util import dev_bf16, host_bits

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K,N,M", [
    (1024, 1152, 256 * 90 + 5),      # five tiles of a row tile, 4 or 3 units: runs that end inside a row tile
    (1024, 128, 256 * 80 + 1),       # one tile of two units per row tile
    (1024, 384, 256 * 37),           # a whole number of rounds: no piece behind them
    (1024, 4096, 2600),              # two rounds, then pieces
    (1024, 3072, 256 * 5 + 3),       # less than a round: 72 tiles of four units
    (1024, 1024, 2748),              # less than a round: 66 pieces of three units
    (1024, 4096, 4122),              # three tiles per worker, none of which share token rows, then pieces of three units
    (1024, 1152, 256 * 120 + 5),     # two runs of four tiles, the second begins inside a row tile; no single tile behind them
    (1024, 640, 700), (4096, 640, 700),
    (4096, 384, 20000),              # tiles of three units, then pieces of one
    (4096, 1024, 256 * 37 + 1),      # two full rounds and one row tile
    (4096, 1024, 2748), (4096, 896, 4700), (4096, 128, 256 * 74 + 9),
    (4096, 640, 6500), (1024, 1152, 3867),     # two rounds of 128 channels where 256 are just more than one
    (1024, 1024, 513), (1024, 1024, 400),      # nothing but pieces: of 128 channels (48 of 64 would not leave half of the chip), of 64
])
def test_tiles(K, N, M):
    rng = np.random.default_rng(K + 7 * N + M)
    spec = workload.LinearSpec("tiles", K, N, workload.DIST_NORMAL, 95, 0)
    W, b = spec.weight(), spec.bias()
    c = oracle.smooth_factors(spec.x_calib(16), W)
    prep = oracle.prepare_weights(W, c)
    h = q.prepare_weights(dev_bf16(W), dev_bf16(b), torch.from_numpy(c).cuda(), None, c8=True)
    xq = rng.integers(-7, 8, (M, K)).astype(np.int8)
    a = (rng.random((M,)) + 0.5).astype(np.float32) * 1e-2
    A, X8 = torch.from_numpy(a).cuda(), torch.from_numpy(xq).cuda()
    Y = torch.full((M + 2, N + 8), 7.0, dtype=torch.bfloat16, device="cuda")
    q.w4a4_linear_c8(h, X8, A, Y[1:M + 1, :N])
    assert torch.all(Y[0] == 7) and torch.all(Y[M + 1] == 7) and torch.all(Y[:, N:] == 7)
    P = q.w4a4_linear(h, torch.from_numpy(oracle.pack_int4(xq)).cuda(), A, 0)
    assert torch.equal(Y[1:M + 1, :N].view(torch.int16), P.view(torch.int16))
    rows = np.unique(np.concatenate([[0, M - 1], rng.integers(0, M, 40)]))
    want = oracle.epilogue(oracle.gemm_i32(xq[rows], prep["wq"]), a[rows], prep["w_scale"], b)
    assert np.array_equal(host_bits(P[torch.from_numpy(rows).cuda()]), want)
    assert h.device_status() == 0
    h.free()
