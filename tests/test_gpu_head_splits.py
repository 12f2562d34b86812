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
    # CTA each are 33 rounds: a second block of 32, with an active row in it
    case = _case(rows, vocab, dtype, seed=rows, inactive=True)
    step = max(1, rows // 400)
    _check(case, _run(case, with_mask=False), rows=list(range(0, rows, step)), check_mask=False)


@pytest.mark.parametrize("rows,vocab", [(150000, 8), (30000, 49408), (30000, 49413)])
@pytest.mark.parametrize("gated", [False, True])
def test_blocks_of_rounds_without_an_active_row(gpu_lib, rows, vocab, gated):
    # hundreds of rounds per cluster (one CTA, or two), of which whole blocks of 32 have
    # no active row, between and before blocks that do: the warps count the parameter
    # buffers by the others
    import torch

    from oracle import sampling as osamp
    from paper_2607_20791_gb300 import binding
    rng = np.random.default_rng(rows)
    live = np.zeros(rows, bool)
    live[:60] = live[rows * 3 // 5:rows * 3 // 5 + 90] = live[rows - 200:] = True
    live &= rng.random(rows) > 0.2
    gen = torch.Generator(device="cuda")
    gen.manual_seed(vocab)
    logits = torch.randn((rows, vocab), generator=gen, device="cuda", dtype=torch.bfloat16)
    temps = np.array([0.0, 1.0, 2.0], np.float32)[np.arange(rows) % 3]
    seeds = rng.integers(0, 2 ** 62, rows)
    temp, seed = torch.from_numpy(temps).cuda(), torch.from_numpy(seeds).cuda()
    minp = torch.full((rows,), 0.05, dtype=torch.float32, device="cuda")
    active = torch.from_numpy(live.astype(np.uint8)).cuda()
    tok = torch.full((rows,), -7, dtype=torch.int32, device="cuda")
    cnt = torch.full((rows,), -7, dtype=torch.int32, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    if gated:
        trie = binding.Trie([[3, 4], [5, 2, 1]], 2)
        state = binding.new_gate_state(rows // 3)
        binding.rgd_gate_state_init(state, rows // 3)
        binding.rgd_sample_head_gated(logits, None, temp, minp, seed, 1, active, tok, cnt, trie, 3, -1, 8, state, status)
    else:
        binding.rgd_sample_head(logits, None, temp, minp, seed, 1, active, tok, cnt, None, status)
    torch.cuda.synchronize()
    # (a group whose probe row is inactive and has not ended gives the gate no token)
    assert int(status.item()) == (binding.RGD_DEV_BAD_TOKEN if gated else 0)
    tok, cnt = tok.cpu().numpy(), cnt.cpu().numpy()
    assert np.all(tok[~live] == -1) and np.all(cnt[~live] == 0)
    at = np.nonzero(live)[0]
    n = len(at)
    host = logits[torch.from_numpy(at).cuda()].view(torch.int16).cpu().numpy().view(np.uint16)
    ref = osamp.sample_head(host, "bf16", np.zeros(n, np.uint8), temps[at], np.full(n, 0.05, np.float32),
                            seeds[at].astype(np.uint64), 1, np.ones(n, np.uint8))
    for i, r in enumerate(at):
        assert cnt[r] == ref.kept_count[i] and (tok[r] == ref.tokens[i] or ref.boundary[i]), r
    if gated:
        trie.close()
