"""The probe gate and the precheck at the edges of their splits: nodes with one
child to more than two steps of 32-way search, tokens on both sides of the
32-token chunks of a confirmed probe, activation rows on and off 16 bytes.  Gate
outcomes bit for bit against the oracle's naive scan; prechecks with the other
precheck tests' bound (the vector path sums d products in fp32 as well)."""
import numpy as np
import pytest

from oracle import gate as ogate
from oracle import precheck as opre
from paper_2607_20791_gb300 import binding, workloads
from test_gpu_gate import _compare, _gpu_gate

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("children", [1, 2, 31, 32, 33, 63, 64, 65, 1023, 1024, 1025, 2100])
def test_nodes_of_many_children(gpu_lib, children):
    # every child (even tokens), its neighbours and the ends, out of the root and
    # out of an inner node
    kids = [2 * i + 2 for i in range(children)]
    P = [[k, 1, 1] for k in kids] + [[3, k, 4] for k in kids]
    edge = sorted({0, 1, kids[-1] + 1, kids[-1] + 2, *kids[:40], *kids[-40:], *(k + 1 for k in kids[::7])})
    toks = np.array([[a, 1, 1, 0] for a in edge] + [[3, a, 4, 0] for a in edge], np.int32)
    _compare(P, toks, -1, 16, rpg=3)


@pytest.mark.parametrize("n", [1, 31, 32, 33, 64, 100])
@pytest.mark.parametrize("max_len", [2, 3, 31, 32, 33, 34, 64, 65, 200])
def test_confirmed_probe_over_token_chunks(gpu_lib, n, max_len):
    # confirmed after two tokens; a stop token at every kind of position
    rows = []
    for stop in (2, 3, 30, 31, 32, 33, 63, 64, 65, 99, 1000):
        t = np.full(n, 5, np.int32)
        t[:2] = [7, 8][:len(t[:2])]
        if stop < n:
            t[stop] = 0
        rows.append(t)
    toks = np.stack(rows)
    _compare([[7, 8], [7, 9, 9]], toks, 0, max_len, rpg=2)
    _compare([[7, 8], [7, 9, 9]], toks, 0, max_len, rpg=2, per_token=n <= 33)


@pytest.mark.parametrize("at", [2, 31, 32, 40, 70])
def test_negative_tokens_of_a_confirmed_probe(gpu_lib, at):
    # reported and skipped before the probe's end, not looked at after it
    toks = np.full((2, 80), 5, np.int32)
    toks[:, :2] = [7, 8]
    toks[0, at] = -9
    for max_len, seen in ((at + 1, True), (at, False)):
        got, _, status = _gpu_gate([[7, 8]], toks, -1, max_len)
        ref = ogate.run_gate(np.delete(toks[:1], at, axis=1), [[7, 8]], -1, max_len)
        assert (status == binding.RGD_DEV_BAD_TOKEN) == seen
        assert got["length"][0] == len(ref[0].q) and got["steps"][0] == ref[0].steps and got["done"][0]
        assert got["length"][1] == max_len and got["done"][1]


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("d", [4, 8, 12, 1024, 2048, 2056, 8192, 8196])
@pytest.mark.parametrize("shift", [0, 1])
def test_precheck_vectors_and_elements(gpu_lib, dtype, d, shift):
    import torch
    G = 9
    case = workloads.make_precheck_case("vec", G, d, dtype, 0.5, seed=d + shift, weight_scale=4.0)
    raw = torch.from_numpy(case.h if dtype == "f32" else case.h.view(np.int16))
    buf = torch.zeros(G * d + shift, dtype=raw.dtype, device="cuda")
    buf[shift:] = raw.flatten().cuda()
    h = buf[shift:].view(G, d)
    h = h if dtype == "f32" else h.view(torch.bfloat16)
    prob = torch.full((G,), -1.0, dtype=torch.float32, device="cuda")
    st = binding.new_gate_state(G)
    binding.rgd_gate_state_init(st, G)
    binding.rgd_residual_precheck(h, torch.from_numpy(case.w).cuda(), case.b, case.theta, 1, st, None, prob)
    h64 = (case.h.astype(np.float64) if dtype == "f32"
           else (case.h.astype(np.uint32) << 16).view(np.float32).astype(np.float64))
    z, p, _ = opre.precheck(h64, case.w, case.b, case.theta)
    got = prob.cpu().numpy()
    assert np.all(np.abs(got - p) <= 1e-6 + 1e-5 * p), float(np.abs(got - p).max())
