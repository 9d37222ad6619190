"""Sizes, alignments, non-finite values and workspaces at the limits of what the calls accept."""
import ctypes

import numpy as np
import pytest

import cafeq_synth as syn
from oracle import cafeq_oracle as orc
from parity_utils import f32_dev, rel_err, to_dev, w64

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cq():
    import paper_2511_19705_b200 as m
    m.lib()
    return m


def test_second_factor_of_more_rows_than_a_grid_has_slices(cq):
    """65 600 rows (gridDim.y ends at 65 535): the product, its quantised error, its straight-through gradient, Algorithm 1."""
    h, d1, d3, k = 64, 64, 65600, 64
    W1 = to_dev(syn.weight_student_t(h, d1, 3))
    W2 = to_dev(np.tile(syn.weight_student_t(64, h, 4), (d3 // 64, 1)))
    M = f32_dev(syn.perturbed_blocks(1, k, 5, 0.02))
    P = cq.cafeq_pair_product(W1, W2, k=k)
    P64 = W1.double().T @ W2.double().T
    assert float((P - P64).norm() / P64.norm()) <= 1e-6
    kw = dict(bits=4, group1=64, group2=64)
    # the rows repeat 64 rows 1025 times, so the squared error and its gradient are 1025 times theirs
    small = cq.cafeq_pair_loss_fwd_bwd(W1, W2[:64], M, P=cq.cafeq_pair_product(W1, W2[:64], k=k), loss_kind=cq.LOSS_PQE_STE, **kw)
    out = cq.cafeq_pair_loss_fwd_bwd(W1, W2, M, P=P, loss_kind=cq.LOSS_PQE_STE, **kw)
    assert int(out["status"].item()) == 0
    assert abs(float(out["losses"][3]) / (1025 * float(small["losses"][3])) - 1) <= 1e-5
    # one chain of d3 / 16 = 4100 fp32 additions in the tensor core, 2^-23 each: 5e-4 in each of the two factors' parts
    assert rel_err(out["gradM"].cpu().numpy(), 1025 * small["gradM"].cpu().numpy()) <= 2e-3
    r = cq.cafeq_adaptive_round(W1, W2, M, iters=1, **kw)
    assert int(r["status"].item()) == 0
    U = r["codes1"].double() * r["scales1"].double()  # one group per row
    V = r["codes2"].double() * r["scales2"].double()
    Mc = M.bfloat16().double()[0]
    Minv = torch.from_numpy(orc.round_bf16(orc.block_inverse(Mc.cpu().numpy()[None]))).cuda().double()[0]
    target = (Mc.T @ W1.double()).T @ (W2.double() @ Minv.T).T
    assert abs(float((U.T @ V.T - target).norm()) / float(r["pqe"][2]) - 1) <= 1e-3


def test_more_operator_blocks_than_a_grid_has_slices(cq):
    """65 600 blocks of 64: row and operators repeat every 64 blocks, and so must the codes and scales."""
    W = to_dev(syn.weight_student_t(1, 4096, 3))
    T = f32_dev(syn.perturbed_blocks(64, 64, 5, 0.1))
    codes, scales = cq.cafeq_rtn(W.repeat(1, 1025), T.repeat(1025, 1, 1), bits=4, group=128, tblock=64)
    c0, s0 = cq.cafeq_rtn(W, T, bits=4, group=128, tblock=64)
    assert torch.equal(codes.view(1025, -1), c0.repeat(1025, 1)) and torch.equal(scales.view(1025, -1), s0.repeat(1025, 1))
