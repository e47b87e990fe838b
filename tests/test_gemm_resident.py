"""The rule by which packed linears keep their expanded weights in shared memory (gemm_resident.cuh), compiled for the host."""
import ctypes
import subprocess
from pathlib import Path

import pytest

CSRC = Path(__file__).resolve().parent.parent / "paper_2504_18547_b200" / "csrc"
SHARED_MEMORY = 227 * 1024
REQUANT, GELU, FP32 = 0, 1, 2


@pytest.fixture(scope="module")
def tile_columns(tmp_path_factory):
    d = tmp_path_factory.mktemp("resident")
    (d / "rule.cpp").write_text('#include "gemm_resident.cuh"\nextern "C" int rule(int sms, int m, int k, int n, int bits, int block, int bn0, int epi)\n'
                                '{ return vitint::resident_tile_columns(sms, m, k, n, bits, block, bn0, (vitint::PackedEpilogue)epi); }\n')
    subprocess.run(["g++", "-O1", "-std=c++17", "-fPIC", "-shared", f"-I{CSRC}", str(d / "rule.cpp"), "-o", str(d / "rule.so")], check=True)
    return ctypes.CDLL(str(d / "rule.so")).rule


@pytest.mark.parametrize("M,K,N,bits,bn0,epi,taken", [
    (12608, 768, 3072, 4, 192, REQUANT, True), (25216, 768, 3072, 4, 256, GELU, True), (12608, 512, 2048, 4, 256, FP32, True),
    (197, 768, 3072, 4, 128, REQUANT, False),                                                   # one tile a CTA
    # slower with kept weights (time without / with them, us): more epilogues than expansions saved
    (50432, 1024, 1024, 4, 256, REQUANT, False), (25216, 192, 768, 4, 256, REQUANT, False),     # 77.0 / 79.5, 15.8 / 17.5
    (25216, 640, 640, 2, 256, REQUANT, False), (25216, 192, 768, 4, 256, GELU, False),          # 18.4 / 21.2, 21.6 / 25.1
    (25216, 640, 640, 2, 256, GELU, False), (3000, 768, 3072, 2, 256, GELU, False),             # 23.6 / 28.5, 15.2 / 16.9
    (25216, 768, 2304, 2, 256, FP32, False), (12608, 768, 3072, 4, 192, FP32, False),           # 61.2 / 75.4, 49.9 / 58.2
    (50432, 768, 768, 2, 256, FP32, False), (9000, 768, 2304, 4, 192, FP32, False)])            # 42.6 / 54.3, 29.1 / 33.2
def test_sizes_on_both_sides_of_the_rule(tile_columns, M, K, N, bits, bn0, epi, taken):
    assert (tile_columns(148, -(-M // 128), -(-K // 128), N, bits, 32 if epi == FP32 else 64, bn0, epi) > 0) == taken


@pytest.mark.parametrize("bits,max_k", [(2, 2 ** 31 // 9), (4, 2 ** 31 // 225)])      # unsigned codes: the int32 bound allows this much
def test_what_is_kept_fits_at_every_length(tile_columns, bits, max_k):
    """Sizes that exceed 32 bits must not come out small: K = 2^24 with 256 columns is 2^32 bytes of expanded weights."""
    lengths = sorted({k for e in range(27) for k in (2 ** e - 1, 2 ** e, 2 ** e + 1, 3 * 2 ** e // 2) if 0 < k * 128 <= max_k})
    for epi in (REQUANT, GELU, FP32):
        for m_tiles in (18, 99, 2000):
            for n in (192, 1000, 2304, 3072):
                for k_blocks in lengths:
                    bn = tile_columns(148, m_tiles, k_blocks, n, bits, 32 if epi == FP32 else 64, 256, epi)
                    assert bn == 0 or 2 * 128 * 128 + 2 * (128 + bn) * 16 * bits + k_blocks * 128 * bn <= SHARED_MEMORY, (m_tiles, n, k_blocks, bn)
