"""Packed codes with rows of at most 512 codes, several of which share a CTA."""
import numpy as np
import pytest
import torch

from paper_2309_01885_gb300 import qe

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    qe.load()


@pytest.mark.parametrize("p", [1, 7, 15, 16, 17, 31, 33, 65, 127, 129, 255, 257, 511, 512, 513])
@pytest.mark.parametrize("q,bits,extra", [(1, 3, 0), (255, 5, 3), (257, 8, 1), (1031, 2, 0), (70001, 3, 7)])
def test_narrow_rows(q, p, bits, extra):
    """Against numpy's bit packing, and back; bytes around the rows stay."""
    if q * p > 1 << 23:
        q = (1 << 23) // p
    g = torch.Generator(device="cuda").manual_seed(q + p)
    full = torch.randint(0, 256, (q, p + extra), generator=g, device="cuda", dtype=torch.uint8)
    codes = full[:, :p] & ((1 << bits) - 1) if extra == 0 else full[:, :p]
    codes = codes.contiguous() if extra == 0 else codes.bitwise_and_((1 << bits) - 1)
    packed = qe.qe_pack_codes(codes, bits)
    c = codes.cpu().numpy()
    ref = np.packbits(((c[:, :, None] >> np.arange(bits)) & 1).reshape(q, -1), axis=1, bitorder="little")
    assert np.array_equal(packed.cpu().numpy(), ref)
    assert torch.equal(qe.qe_unpack_codes(packed, p, bits), codes)
