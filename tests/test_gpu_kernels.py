"""GPU parity of kernel variants at the sizes where their dispatch or tiling changes, against the oracle."""
import numpy as np
import pytest
import torch

import oracle as vo
import paper_2504_18547_b200 as vt
import synth_inputs as si
from gpu_util import GELU_TOL_REL, dev, from_codes, padding_is_zero, rand_codes, to_codes

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _device_status_clean():
    yield
    assert vt.vitint_device_status() == 0


def byte_codes(q, bits, signed):
    return to_codes(q, bits, signed) if bits == 8 else vt.vitint_widen(to_codes(q, bits, signed))


# ---- byte-stored operands, whole column blocks: single rows, row remainders of a 16-row unit and of a tile, one and
# ---- several column blocks, a last tile narrower than the others, K remainders of a block and of an MMA step
@pytest.mark.parametrize("M,K,N", [(1, 64, 64), (17, 48, 128), (127, 144, 320), (129, 768, 192), (145, 1000, 576), (1576, 320, 1088),
                                   (2600, 768, 2304)])
@pytest.mark.parametrize("bits", [2, 3, 4, 8])
def test_linear_direct_epilogues(M, K, N, bits):
    qx, qw = rand_codes(101 + M, (M, K), bits, True), rand_codes(102 + N, (N, K), bits, True)
    x, w = byte_codes(qx, bits, True), byte_codes(qw, bits, True)
    acc = vo.matmul_i32(qx, qw)
    spread = max(float(np.abs(acc).mean()), 1.0)
    s_w = ((np.abs(si.normal(103, (N,), 0.0, 0.2)) + 0.5) / spread).astype(np.float32)
    bias, res = si.normal(104, (N,), 0.0, 0.3), si.normal(105, (M, N))
    alpha, beta = s_w * np.float32(2 ** (bits - 1)), bias
    for cont, pitch in ((8, None), (0, None), (8, N + 48)):
        out = vt.Codes.empty(M, N, bits, True, container=cont, pitch=pitch)
        out.data.fill_(0xA5)
        vt.vitint_linear(x, 1.0, w, None, None, vt.Epilogue(mode=vt.EPI_REQUANT, alpha=dev(alpha), beta=dev(beta), out_bits=bits,
                                                            out_signed=True, out_container=cont), out=out)
        assert np.array_equal(from_codes(out), vo.epilogue_requant(acc, alpha, beta, bits, True)) and padding_is_zero(out)
    for r in (None, res):
        y = vt.vitint_linear(x, 0.75, w, dev(s_w), dev(bias), vt.Epilogue(mode=vt.EPI_DEQUANT_F32, residual=dev(r)))
        want = vo.epilogue_dequant(acc, np.float32(0.75), s_w, bias, r)
        assert np.array_equal(y.cpu().numpy().view(np.uint32), want.view(np.uint32))
    inv = np.full(N, (2 ** bits - 1) / 1.5, np.float32)
    g = vt.vitint_linear(x, 1.0, w, dev(s_w), dev(bias), vt.Epilogue(mode=vt.EPI_REQUANT, act=1, inv_out_step=dev(inv), out_bits=bits,
                                                                    out_signed=False, out_container=8))
    _, lo, hi = vo.epilogue_gelu_requant(acc, 1.0, s_w, bias, inv, bits, False, GELU_TOL_REL)
    q = from_codes(g)
    assert ((q >= lo) & (q <= hi)).all() and padding_is_zero(g)


@pytest.mark.parametrize("M,N", [(16300, 768), (16250, 768)])
def test_linear_fp32_dispatch_boundary(M, N):
    """Around the size from which a short contraction with a residual takes the staged fp32 epilogue."""
    K = 96
    qx, qw = rand_codes(111, (M, K), 4, True), rand_codes(112, (N, K), 4, True)
    s_w = (np.abs(si.normal(113, (N,), 0.0, 0.01)) + 1e-3).astype(np.float32)
    bias, res = si.normal(114, (N,), 0.0, 0.05), si.normal(115, (M, N))
    y = vt.vitint_linear(byte_codes(qx, 4, True), 0.37, byte_codes(qw, 4, True), dev(s_w), dev(bias),
                         vt.Epilogue(mode=vt.EPI_DEQUANT_F32, residual=dev(res)))
    want = vo.epilogue_dequant(vo.matmul_i32(qx, qw), np.float32(0.37), s_w, bias, res)
    assert np.array_equal(y.cpu().numpy().view(np.uint32), want.view(np.uint32))
