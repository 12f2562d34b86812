"""The sample head's splits at their edges: CTAs per row (1, 8, 16), ring slots
that a row's share just fills or just overruns, rows off 16-byte boundaries up to
the end of the buffer, and clusters that walk many rows (several rounds, more
than one block of 32 rounds, inactive rows between).  Against the fp64 oracle:
greedy tokens and kept counts exact, sampled tokens exact but for flagged
boundary draws."""
import numpy as np
import pytest

from paper_2607_20791_gb300 import workloads
from test_gpu_sample_head import _check, _run

pytestmark = pytest.mark.gpu


def _case(rows, vocab, dtype, seed, inactive=False):
    rng = np.random.default_rng([seed, rows, vocab])
    logits = rng.standard_normal((rows, vocab), dtype=np.float32) * 2.0
    temps = np.array([0.0, 1.0, 1.5, 3.0], np.float32)[np.arange(rows) % 4]
    minp = np.array([0.05, 0.1, 0.0], np.float32)[np.arange(rows) % 3]
    active = (rng.random(rows) > 0.4).astype(np.uint8) if inactive else None
    return workloads.make_head_case("splits", logits, dtype, (np.arange(rows) % 5 == 0).astype(np.uint8), temps, minp,
                                    seed, step=3, row_active=active)


@pytest.mark.parametrize("rows,vocab,dtype", [
    (3, 4096, "f32"), (3, 4100, "f32"), (3, 8192, "bf16"), (2, 8200, "bf16"),   # one slot, and one vector more
    (3, 32768, "f32"), (3, 32772, "f32"), (3, 65544, "bf16"),                   # one slot at 8 CTAs per row
    (3, 196608, "f32"), (3, 196612, "f32"),                                     # 6 slots at 8 CTAs; 16 CTAs per row
    (2, 524288, "f32"), (2, 524287, "f32"), (2, 1048576, "bf16"), (2, 1048573, "bf16"),  # the largest rows
    (5, 2047, "bf16"), (7, 4093, "f32"), (9, 12291, "bf16"),                    # off 16-byte boundaries
])
def test_edges(gpu_lib, rows, vocab, dtype):
    case = _case(rows, vocab, dtype, seed=vocab)
    _check(case, _run(case))  # (a draw that differs must be a flagged boundary draw)


@pytest.mark.parametrize("rows,vocab,dtype", [(1000, 40, "f32"), (1400, 4099, "bf16"), (700, 33000, "bf16"),
                                              (15000, 8, "bf16")])
def test_rounds(gpu_lib, rows, vocab, dtype):
    # rows in several rounds per cluster, a part of them inactive; 15000 rows of one
    # CTA each are more than 32 rounds
    case = _case(rows, vocab, dtype, seed=rows, inactive=True)
    step = max(1, rows // 400)
    _check(case, _run(case, with_mask=False), rows=list(range(0, rows, step)), check_mask=False)
