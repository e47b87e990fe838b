"""The rule by which packed linears keep their expanded weights in shared memory (gemm_resident.cuh), compiled for the host."""
import ctypes
import subprocess
from pathlib import Path

import pytest

CSRC = Path(__file__).resolve().parent.parent / "paper_2504_18547_b200" / "csrc"
SHARED_MEMORY = 227 * 1024


@pytest.fixture(scope="module")
def tile_columns(tmp_path_factory):
    d = tmp_path_factory.mktemp("resident")
    (d / "rule.cpp").write_text('#include "gemm_resident.cuh"\nextern "C" int rule(int sms, int m, int k, int n, int bits, int block, int bn0, int f32)\n'
                                '{ return vitint::resident_tile_columns(sms, m, k, n, bits, block, bn0, f32 != 0); }\n')
    subprocess.run(["g++", "-O1", "-std=c++17", "-fPIC", "-shared", f"-I{CSRC}", str(d / "rule.cpp"), "-o", str(d / "rule.so")], check=True)
    return ctypes.CDLL(str(d / "rule.so")).rule


def test_a_usual_packed_linear_keeps_its_weights(tile_columns):
    assert tile_columns(148, 99, 6, 3072, 4, 64, 256, 0) > 0              # 12,608 x 768 -> 3072
    assert tile_columns(148, 2, 6, 3072, 4, 64, 128, 0) == 0              # one tile a CTA


@pytest.mark.parametrize("bits,max_k", [(2, 2 ** 31 // 9), (4, 2 ** 31 // 225)])      # unsigned codes: the int32 bound allows this much
def test_what_is_kept_fits_at_every_length(tile_columns, bits, max_k):
    """Sizes that exceed 32 bits must not come out small: K = 2^24 with 256 columns is 2^32 bytes of expanded weights."""
    lengths = sorted({k for e in range(27) for k in (2 ** e - 1, 2 ** e, 2 ** e + 1, 3 * 2 ** e // 2) if 0 < k * 128 <= max_k})
    for block, f32 in ((64, 0), (32, 1)):
        for m_tiles in (18, 99, 2000):
            for n in (192, 1000, 2304, 3072):
                for k_blocks in lengths:
                    bn = tile_columns(148, m_tiles, k_blocks, n, bits, block, 256, f32)
                    assert bn == 0 or 2 * 128 * 128 + 2 * (128 + bn) * 16 * bits + k_blocks * 128 * bn <= SHARED_MEMORY, (m_tiles, n, k_blocks, bn)
