"""Host requests with several streaming width classes, rows written by queued work, and Pauli types
that follow one another in one call, against device batches, shots alone and types alone."""
import numpy as np
import pytest

import paper_2603_05381_gb300 as pkg
from gpu_util import gpu_sample, torch_cuda
from test_gpu_lists import _pair, _syndromes

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    return torch_cuda()


# sizes by case: one class that fills the device and few shots in others (beside it, with scratch of
# their own); one class alone; the general kernel's class (above 512 defects in FP64, 1024 in FP32)
# beside others
CASES = {
    "full_and_few": [200] * 340 + [170] * 20 + [300] * 15 + [400] * 5 + [50] * 20,
    "few_of_each": [170] * 40 + [200] * 70 + [300] * 30 + [400] * 15 + [9] * 5,
    "one_class": [170] * 400,
    "general_fp64": [130] * 10 + [220] * 10 + [400] * 4 + [520, 600],
    "general_fp32": [1030, 1100] + [200] * 30 + [300] * 3,
}


@pytest.mark.parametrize("case,prec,decoder,forced,early", [
    ("full_and_few", "fp32", "bp4m", "greedy", True), ("full_and_few", "bf16", "bp4m", "static", True),
    ("full_and_few", "fp32", "bp4m", "greedy", False), ("full_and_few", "fp16", "bp4mf", "static", True),
    ("full_and_few", "fp32", "bp4mf", "greedy", True), ("few_of_each", "fp32", "bp4m", "greedy", True),
    ("few_of_each", "fp32", "bp4mf", "static", True), ("few_of_each", "fp16", "bp4m", "static", False),
    ("one_class", "fp32", "bp4m", "greedy", True), ("one_class", "bf16", "bp4mf", "greedy", True),
    ("general_fp64", "fp64", "bp4m", "greedy", True), ("general_fp32", "fp32", "bp4m", "greedy", True)])
def test_width_classes_of_a_host_request(torch, case, prec, decoder, forced, early):
    g, og, _ = _pair(13)
    rng = np.random.default_rng(41)
    sizes = rng.permutation(CASES[case])
    n, T = len(sizes), 4
    _, packed, synd = _syndromes(torch, og, sizes, seed=42)
    opts = pkg.make_opts(precision=prec, decoder=decoder, forced=forced, early_exit=early)
    types = (np.uint8, np.uint8, np.int16)
    host = [np.full(n, 77, dtype=t) for t in types]
    g.decode_batch(packed, T, opts, *host)
    dev = [torch.full((n,), 77, dtype=t, device="cuda") for t in (torch.uint8, torch.uint8, torch.int16)]
    g.decode_batch(synd, T, opts, *dev)
    torch.cuda.synchronize()
    for a, b in zip(dev, host):
        assert np.array_equal(a.cpu().numpy(), b)
    # one shot of each size alone
    for s in sorted(set(sizes.tolist())):
        for k in np.flatnonzero(sizes == s)[[0, -1]]:
            one = [np.full(1, 77, dtype=t) for t in types]
            g.decode_batch(packed[k:k + 1], T, opts, *one)
            assert [int(x[0]) for x in one] == [int(x[k]) for x in host], (case, s, k)


@pytest.mark.parametrize("prec,sizes", [("fp32", (161, 192)), ("fp32", (256,)), ("fp32", (257, 320)), ("fp32", (384,)),
                                        ("fp32", (448,)), ("fp32", (449, 512)), ("fp16", (193, 256)), ("fp16", (321, 384)),
                                        ("bf16", (192,)), ("bf16", (384,))])
@pytest.mark.parametrize("decoder,forced", [("bp4m", "greedy"), ("bp4mf", "greedy"), ("bp4mf", "static")])
def test_one_block_per_sm_matches_two(torch, prec, sizes, decoder, forced):
    # a launch of no more shots than SMs has blocks of twice the warps: one shot more, and one alone
    g, og, _ = _pair(13)
    n = torch.cuda.get_device_properties(0).multi_processor_count + 1
    T = 3
    _, _, synd = _syndromes(torch, og, [sizes[k % len(sizes)] for k in range(n)], seed=45)
    opts = pkg.make_opts(precision=prec, decoder=decoder, forced=forced, early_exit=False, stream_cluster=1)
    got = []
    for k in (n, n - 1, len(sizes)):
        out = [torch.full((k,), 77, dtype=t, device="cuda") for t in (torch.uint8, torch.uint8, torch.int16)]
        g.decode_batch(synd[:k], T, opts, *out)
        torch.cuda.synchronize()
        got.append([x.cpu().numpy() for x in out])
    for few in got[1:]:
        for a, b in zip(got[0], few):
            assert np.array_equal(a[:len(b)], b)


@pytest.mark.parametrize("prio", [None, 0, -1])  # the default stream, side streams of two priorities
def test_host_rows_written_by_queued_work(torch, prio):
    # a copy into pinned rows, behind gigabytes of other copies in the caller's stream
    g, og, _ = _pair(9)
    n, T = 64, 10
    _, packed, synd = _syndromes(torch, og, [1 + k % 40 for k in range(n)], seed=43)
    opts = pkg.make_opts()
    want = [torch.zeros(n, dtype=t, device="cuda") for t in (torch.uint8, torch.uint8, torch.int16)]
    g.decode_batch(synd, T, opts, *want)
    rows = torch.zeros(synd.shape, dtype=torch.int32).pin_memory()
    a = torch.zeros(1 << 28, dtype=torch.float32, device="cuda")
    b = torch.empty_like(a)
    torch.cuda.synchronize()
    st = torch.cuda.default_stream() if prio is None else torch.cuda.Stream(priority=prio)
    got = [np.full(n, 77, dtype=t) for t in (np.uint8, np.uint8, np.int16)]
    with torch.cuda.stream(st):
        for _ in range(20):
            b.copy_(a)
        rows.copy_(synd, non_blocking=True)
        g.decode_batch(rows, T, opts, *got, stream=st.cuda_stream)
    for x, y in zip(want, got):
        assert np.array_equal(x.cpu().numpy(), y)


@pytest.mark.parametrize("prec,d,p", [("fp32", 7, 0.1), ("fp16", 9, 0.15), ("fp64", 5, 0.1)])
def test_types_that_follow_one_another_match_types_alone(torch, prec, d, p):
    # both types of a call go through the same lists, counters and scratch with no wait of the caller's
    # between them
    n, T = 5000, 12
    g = pkg.Graph(d, "code_capacity", p, family="unrotated")
    synds, obs = gpu_sample(g, 0, n, seed=44)
    counts = g.sample_and_decode(n, seed=44, iters=T, opts=pkg.make_opts(precision=prec))
    iters = 0
    for ty in range(2):
        out = [torch.zeros(n, dtype=t, device="cuda") for t in (torch.uint8, torch.uint8, torch.int16)]
        g.decode_batch(synds[ty], T, pkg.make_opts(precision=prec, type=ty), *out)
        torch.cuda.synchronize()
        assert counts["fail"][ty] == int((out[0] != obs[ty]).sum())
        assert counts["unconverged"][ty] == int((out[1] == 0).sum())
        iters += int(out[2].to(torch.int64).sum())
    assert counts["iterations"] == iters and counts["shots"] == n
