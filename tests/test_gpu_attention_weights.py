"""How exactly the attention applies its softmax weights.  The bf16 output hides
their rounding unless it is near zero, so here it is: half of the tokens have the
weight 1 and the value 1, the other half a weight p and the value -v with v = 1 / p
in one column, which then holds (1 - p v) / (1 + p): the weight's error and little else."""
import numpy as np
import pytest

from oracle import attention as oattn
from oracle.sampling import bf16_bits_to_f32
from paper_2607_20791_gb300 import workloads
from paper_2607_20791_gb300.workloads import f32_to_bf16_bits
from test_gpu_attention import _run

pytestmark = pytest.mark.gpu


def _case(D, rpg, heads, tokens):
    case = workloads.make_attn_case("weights", 1, rpg, heads, 1, D, [tokens], [0] * rpg, seed=D + rpg)
    case.softmax_scale = 1.0
    col = np.arange(rpg * heads) % D
    v = bf16_bits_to_f32(f32_to_bf16_bits((1.06 * 18.0 ** (np.arange(D) / D)).astype(np.float32)))
    # q k = -ln(v) of the query's column for the tokens of weight p, in two parts of 8 bits
    s = np.log(v[col].astype(np.float64))
    q = np.zeros((rpg * heads, D), np.float32)
    q[:, 0] = bf16_bits_to_f32(f32_to_bf16_bits(s.astype(np.float32)))
    q[:, 1] = (s - q[:, 0]) * 256.0
    case.q = f32_to_bf16_bits(q).reshape(rpg, heads, D)
    k = np.zeros(case.k_pages.shape, np.float32)
    k[:, 0, 1::2, 0], k[:, 0, 1::2, 1] = -1.0, -1.0 / 256.0
    vals = np.ones(case.v_pages.shape, np.float32)
    vals[:, 0, 1::2] = -v
    case.k_pages, case.v_pages = f32_to_bf16_bits(k), f32_to_bf16_bits(vals)
    return case, col, 1.0 / v[col]


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("rpg,heads", [(2, 4), (5, 4), (9, 4), (9, 8), (16, 8)])
def test_weights_are_unbiased_to_2_17(gpu_lib, D, rpg, heads):
    case, col, p = _case(D, rpg, heads, 256)
    out = _run(case, num_ctas=1).out.float().cpu().numpy().reshape(rpg * heads, D).astype(np.float64)
    ref, _ = oattn.decode_attention_case(case)
    at = np.arange(rpg * heads), col
    err = (out[at] - np.asarray(ref).reshape(rpg * heads, D)[at]) * (1.0 + p)
    # p = hi + lo, both rounded to bf16: |p - hi| <= 2^-8 of p's power of two, so
    # |p - hi - lo| <= 2^-17 p.  1.5e-6 for p itself (a score of up to 4 units in
    # fp32, 2^x to 2 ulp) and the fp32 sums of 256 terms
    assert np.abs(err).max() <= 2.0 ** -17 + 1.5e-6
    # without a bias the mean of n errors of at most 2^-17 (rms 2^-17 / sqrt(3) at most)
    # is within 4 standard errors of 0
    assert abs(err.mean()) <= 4 * 2.0 ** -17 / np.sqrt(3 * err.size) + 5e-7
