"""The gated head where a cluster of several CTAs walks more than 32 rows, so that
its warps take the rows' flags in several blocks while the gate clears flags of
rows that the cluster has finished: one row per group, greedy probes that end at
this step (they are masked as soon as one CTA has finished them) between sampled
ones (whose draw keeps another CTA's warp busy), and inactive rows.  Against the
separate head and gate calls bit for bit, the greedy tokens against the planted
ones and a part of the sampled ones against the oracle."""
import numpy as np
import pytest

from oracle import gate as ogate
from oracle import sampling as osamp
from paper_2607_20791_gb300 import binding, workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows,vocab", [(9000, 49408), (9001, 49411), (4200, 98816), (1300, 400000)])
def test_probes_that_end_in_many_rounds(gpu_lib, rows, vocab):
    import torch
    eos, rng = vocab - 1, np.random.default_rng(rows)
    seqs = workloads.make_refusal_set(40, 2, 5, vocab - 1, seed=1)
    trie = binding.Trie(seqs, 2)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(rows)
    logits = torch.randn((rows, vocab), generator=gen, device="cuda", dtype=torch.bfloat16)
    # a greedy row's token ends its probe: the stop token, or a token that starts no refusal;
    # a few rows go on with a refusal's first token
    greedy = rng.random(rows) < 0.6
    token = np.where(rng.random(rows) < 0.5, eos, rng.integers(0, vocab - 1, rows)).astype(np.int64)
    first = rng.random(rows) < 0.05
    token[first] = [int(seqs[i][0]) for i in rng.integers(0, len(seqs), int(first.sum()))]
    at = np.nonzero(greedy)[0]
    logits[torch.from_numpy(at).cuda(), torch.from_numpy(token[at]).cuda()] = 32.0
    active = (rng.random(rows) > 0.15).astype(np.uint8)
    temp = torch.from_numpy(np.where(greedy, 0.0, 1.5).astype(np.float32)).cuda()
    minp = torch.full((rows,), 0.02, dtype=torch.float32, device="cuda")
    seeds = rng.integers(0, 2 ** 62, rows)
    seed = torch.from_numpy(seeds).cuda()
    res = []
    for fused in (False, True):
        state = binding.new_gate_state(rows)
        binding.rgd_gate_state_init(state, rows)
        ra = torch.from_numpy(active).cuda()
        tok = torch.full((rows,), -7, dtype=torch.int32, device="cuda")
        cnt = torch.full((rows,), -7, dtype=torch.int32, device="cuda")
        status = torch.zeros(1, dtype=torch.int32, device="cuda")
        if fused:
            binding.rgd_sample_head_gated(logits, None, temp, minp, seed, 2, ra, tok, cnt, trie, 1, eos, 16, state, status)
        else:
            binding.rgd_sample_head(logits, None, temp, minp, seed, 2, ra, tok, cnt, None, status)
            binding.rgd_probe_gate(trie, rows, 1, tok, 1, 1, eos, 16, state, ra, status)
        torch.cuda.synchronize()
        res.append([x.cpu().numpy() for x in (tok, cnt, state, ra, status)])
    trie.close()
    for a, b in zip(*res):
        assert np.array_equal(a, b)
    tok, cnt, _, ra, status = res[1]
    assert int(status[0]) == binding.RGD_DEV_BAD_TOKEN  # (the inactive rows' probes give no token)
    live = active != 0
    assert np.array_equal(tok[live & greedy], token[live & greedy]) and np.all(tok[~live] == -1)
    states = ogate.run_gate(tok[live].reshape(-1, 1), seqs, eos, 16, 2)
    want = active.copy()
    want[live] = ogate.row_mask_update(states, 1, active[live])
    assert np.array_equal(ra, want) and ra.sum() > 0 and (live & (ra == 0)).sum() > rows // 4
    some = np.nonzero(live & ~greedy)[0][::97]
    host = logits[torch.from_numpy(some).cuda()].view(torch.int16).cpu().numpy().view(np.uint16)
    n = len(some)
    ref = osamp.sample_head(host, "bf16", np.zeros(n, np.uint8), np.full(n, 1.5, np.float32),
                            np.full(n, 0.02, np.float32), seeds[some].astype(np.uint64), 2, np.ones(n, np.uint8))
    for i, r in enumerate(some):
        assert cnt[r] == ref.kept_count[i] and (tok[r] == ref.tokens[i] or ref.boundary[i]), r
