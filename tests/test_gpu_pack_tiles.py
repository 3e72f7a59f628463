"""The calibrated packing at the row counts where its kernel changes shape (one to five rows per warp, several waves of
warps, ragged last rows) and the tied packing on an unaligned matrix, against the oracle, bit for bit."""
import numpy as np
import pytest
import torch

from paper_2504_15299_b200 import synth
from tests.helpers import np_f32

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    from paper_2504_15299_b200 import binding, build
    build.build_library()
    binding.lib()
    return binding


@pytest.mark.parametrize("bits,g,rows,cols", [((2, 4, 8), 64, 1100, 192), ((2, 3, 4, 8), 128, 2000, 384), ((3, 5), 32, 4700, 96),
                                              ((2, 3, 4, 8), 128, 14301, 256), ((4, 8), 256, 4701, 512)])
def test_pack_calibrated_rows_per_warp(B, bits, g, rows, cols):
    from oracle import mwq
    cfg = B.Config(cols, cols, 2, 1, g, bits, scale_mode=1)
    W = synth.normal(17, 5, (rows, cols), 0.02, "cuda")
    X = synth.normal(17, 6, (cols, 2 * cols), 1.0, "cpu").double()
    X = (X + 0.6 * torch.roll(X, 1, 0)) * (0.5 + synth.normal(17, 7, (cols, 1), 1.0, "cpu").abs().double())
    H = 2.0 * X @ X.T / X.shape[1] + 1e-2 * torch.eye(cols, dtype=torch.float64)
    hc = torch.linalg.cholesky(torch.linalg.inv(H), upper=True).float().contiguous()
    energy = (X * X).mean(dim=1).float().contiguous()
    blob = B.pack_mwq_calibrated(cfg, W, hc.cuda(), energy.cuda())
    q = mwq.quantize_calibrated(np_f32(W), bits, g, hc.numpy(), energy.numpy())
    codes, s1, lo = B.unpack_codes(cfg, blob, rows, cols, bits[-1])
    assert np.array_equal(codes.cpu().numpy(), q.code)
    assert np.array_equal(np_f32(s1), q.s1) and np.array_equal(np_f32(lo), q.lo)
    assert np.array_equal(np_f32(B.unpack_scales(cfg, blob, rows, cols)), q.s_extra)


@pytest.mark.parametrize("g", [32, 64, 128, 256])
def test_pack_unaligned_matrix_and_large_offsets(B, g):
    from oracle import mwq
    bits, rows, cols = (2, 3, 4, 8), 70, 512
    cfg = B.Config(cols, cols, 2, 1, g, bits)
    W = torch.empty(rows * cols + 1, device="cuda")[1:].view(rows, cols)       # four bytes off a 16-byte boundary
    W.copy_(synth.normal(18, 5, (rows, cols), 0.02, "cuda"))
    W[3] += 50.0                                                              # an offset far above the group's range
    W[5] *= 1e4
    W[7, ::2] = -0.0
    blob = B.pack_mwq(cfg, W)
    q = mwq.quantize(np_f32(W), bits, g)
    codes, s1, lo = B.unpack_codes(cfg, blob, rows, cols, 8)
    assert np.array_equal(codes.cpu().numpy(), q.code)
    assert np.array_equal(np_f32(s1), q.s1) and np.array_equal(np_f32(lo), q.lo)


@pytest.mark.parametrize("scale_mode", [0, 1])
@pytest.mark.parametrize("g", [32, 64, 128, 256])
@pytest.mark.parametrize("bits", [(1, 8), (1, 2, 3), (1,)])
def test_pack_range_beyond_the_scale_format(B, bits, g, scale_mode):
    # a base of one bit takes the whole range of a group as its scale, which fp16 does not hold from 65520 on: no residual is
    # a number then and every bit is 0
    from oracle import mwq
    rows, cols = 67, 512
    cfg = B.Config(cols, cols, 2, 1, g, bits, scale_mode=scale_mode)
    W = synth.normal(19, 5, (rows, cols), 0.02, "cuda")
    W[3, 0], W[3, 1], W[66, 300], W[66, 301], W[8, 7] = 65000.0, -65000.0, 40000.0, -30000.0, 65503.0
    blob = B.pack_mwq(cfg, W)
    with np.errstate(all="ignore"):
        q = mwq.quantize(np_f32(W), bits, g, scale_mode)
    assert np.isinf(q.s1).sum() == 2
    codes, s1, lo = B.unpack_codes(cfg, blob, rows, cols, bits[-1])
    assert np.array_equal(codes.cpu().numpy(), q.code)
    assert np.array_equal(np_f32(s1), q.s1) and np.array_equal(np_f32(lo), q.lo)
    if scale_mode and bits[-1] > bits[0]:
        assert np.array_equal(np_f32(B.unpack_scales(cfg, blob, rows, cols)), q.s_extra, equal_nan=True)


@pytest.mark.parametrize("g", [32, 64, 128, 256])
@pytest.mark.parametrize("bits", [(2, 3, 4, 8), (1, 8), (3, 5), (7, 8)])
def test_pack_groups_without_energy(B, bits, g):
    # columns the calibration activations never excite: where a whole group has none, the weighted mean of Eq. 5 is 0 / 0, the
    # first residual bit stands and every later one is 0
    from oracle import mwq
    rows, cols = 130, 1024
    cfg = B.Config(cols, cols, 2, 1, g, bits, scale_mode=1)
    W = synth.normal(20, 5, (rows, cols), 0.02, "cuda")
    energy = synth.normal(20, 6, (1, cols), 1.0, "cuda")[0].abs() + 0.1
    energy[:256], energy[512:768], energy[900] = 0.0, 0.0, 0.0
    blob = B.pack_mwq_calibrated(cfg, W, None, energy)
    with np.errstate(all="ignore"):
        q = mwq.quantize(np_f32(W), bits, g, 1, col_energy=np_f32(energy))
    assert np.isnan(q.s_extra).any() and not np.isnan(q.s_extra).all()
    codes, s1, lo = B.unpack_codes(cfg, blob, rows, cols, bits[-1])
    assert np.array_equal(codes.cpu().numpy(), q.code)
    assert np.array_equal(np_f32(s1), q.s1) and np.array_equal(np_f32(lo), q.lo)
    assert np.array_equal(np_f32(B.unpack_scales(cfg, blob, rows, cols)), q.s_extra, equal_nan=True)
