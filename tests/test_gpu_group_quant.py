"""Fused group quantiser of an fp32 matrix (shape-agnostic forward): group widths at the edges of its variants."""
import numpy as np
import pytest

import cafeq_synth as syn
from oracle import cafeq_oracle as orc
from parity_utils import f32_dev, to_dev, w64

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cq():
    import paper_2511_19705_b200 as m
    m.lib()
    return m


# (d_out, d_in, group): a lane more or less than each variant holds, one group per row, widths that are no multiple of 4
@pytest.mark.parametrize("d_out,d_in,group", [(3, 96, 32), (37, 72, 36), (5, 128, 64), (9, 340, 68), (33, 256, 128), (7, 264, 132),
                                              (5, 512, 256), (5, 1040, 260), (2, 1024, 512), (3, 1032, 516), (3, 1024, 1024),
                                              (2, 1028, 1028), (11, 99, 33)])
@pytest.mark.parametrize("bits", [2, 4, 8])
def test_codes_and_scales_bit_exact(cq, d_out, d_in, group, bits):
    """The identity through the transform path: U is exact, so codes and scales are those of the oracle."""
    Wb = syn.weight_student_t(d_out, d_in, 3 + group, 2, 10.0)
    Wb[0, :group] = 0
    Wb[1, :2] = Wb[1, group - 2:group]      # equal maxima are possible; exact halves of the maximum are
    k = 1
    codes, scales = cq.cafeq_rtn(to_dev(Wb), f32_dev(syn.identity_blocks(d_in, k)), bits=bits, group=group, tblock=k)
    Q = orc.quant_sym(w64(Wb), bits, group)
    assert np.array_equal(codes.cpu().numpy().astype(np.int32), Q["q"])
    assert np.array_equal(scales.cpu().numpy(), Q["s"])


# the same from 2^20 entries on, where a lane takes more of a group
@pytest.mark.parametrize("d_out,d_in,group", [(1031, 1024, 32), (1000, 1080, 36), (1025, 1024, 64), (820, 1360, 68), (1024, 1024, 128),
                                              (1000, 1056, 132), (1027, 1024, 256), (1010, 1040, 260)])
def test_codes_and_scales_bit_exact_large(cq, d_out, d_in, group):
    test_codes_and_scales_bit_exact(cq, d_out, d_in, group, 3)
