"""The soft gate at the edges of its splits: every number of CTAs per group (6, 4
or 2 by the number of groups), shares that stay in shared memory for the search
and shares that do not, rows off 16 bytes, and searches over every count of
candidates around the probes of a pass.  Against the fp64 oracle as in the
other soft-gate tests (appended token, decision and mass)."""
import numpy as np
import pytest

from paper_2607_20791_gb300 import binding, workloads
from test_gpu_soft_gate import _run_loop

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("groups", [16, 25, 39, 77, 160])
@pytest.mark.parametrize("vocab", [1003, 4096])
def test_ctas_per_group(gpu_lib, dtype, groups, vocab):
    P = workloads.make_refusal_set(60, 2, 5, vocab, groups, avoid=[vocab - 1])
    _, soft, _ = _run_loop(P, vocab - 1, groups, vocab, 2, 3, 200, 0.01, 16, seed=groups + vocab, dtype=dtype)
    assert soft > 0


@pytest.mark.parametrize("groups,vocab,k", [(2, 140000, 3000), (2, 300000, 3000), (30, 90000, 800), (60, 60001, 500)])
def test_search_in_and_out_of_shared_memory(gpu_lib, groups, vocab, k):
    # 96 KB of a row's share is staged: 6 CTAs hold 147456 fp32 logits, 4 98304, 2 49152
    P = workloads.make_refusal_set(300, 2, 4, vocab, 5, avoid=[vocab - 1])
    _, soft, deep = _run_loop(P, vocab - 1, groups, vocab, 1, 3, k, 0.001, 16, seed=vocab, boost=1.0)
    assert soft > 0 and deep > 0


@pytest.mark.parametrize("children", [1, 3, 4, 5, 6, 7, 8, 9, 10, 13, 24, 33, 64, 100])
@pytest.mark.parametrize("k", [1, 4, 5, 9, 40, 700, 2000])
def test_search_over_candidates(gpu_lib, children, k):
    vocab = 2000
    P = [[7 * i + 1, 3] for i in range(children)]
    _run_loop(P, vocab - 1, 6, vocab, 2, 3, k, 0.0, 16, seed=children * 10 + k, boost=0.9)


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("vocab", [262143, 262144])
def test_mass_error_does_not_grow_with_the_share(gpu_lib, dtype, vocab):
    # one candidate's mass on rows on and off 16 bytes, with 6, 4 and 2 CTAs a group (a
    # thread of 2 CTAs sums 256 elements of a row off 16 bytes): 2^x is good to 2 ulp
    # (2.4e-7) and its exponent to a last place where the weights carry mass, and the
    # sums add their last place only
    import torch
    n, cand, greedy = 64, 1234, 7
    logits = torch.from_numpy(workloads.zipf_logits(n, vocab, seed=3)).cuda()
    logits[:, cand] = 0.5
    logits[:, greedy] = logits.max(1).values + 1.0  # leaves the set
    if dtype == "bf16":
        logits = logits.bfloat16()
    exact = torch.softmax(logits.double(), 1)[:, cand].cpu().numpy()
    trie = binding.Trie([[cand, 5]], 2)
    for groups in (16, 32, 64):
        mass = []
        for a in range(0, n, groups):
            st = binding.new_gate_state(groups)
            binding.rgd_gate_state_init(st, groups)
            tok = torch.empty(groups, dtype=torch.int32, device="cuda")
            m = torch.empty(groups, dtype=torch.float32, device="cuda")
            binding.rgd_soft_gate(trie, groups, 1, logits[a:a + groups], vocab, vocab, 0.0, 4, -1, 16, st, tok, mass_out=m)
            mass.append(m.cpu().numpy())
        err = np.concatenate(mass).astype(np.float64) / exact - 1.0
        assert np.sqrt((err * err).mean()) <= 2.4e-7, groups
    trie.close()
