"""Decode lists by defect count and the host-request path on the GPU: the forms of 8 to 96 rows
(several shots per warp up to 32) at the edges of their row counts, the streaming tier at the
edges of its widest classes, and small host batches against device batches of the same shots."""
import numpy as np
import pytest

import paper_2603_05381_gb300 as pkg
from gpu_util import compare_shots, gpu_decode, torch_cuda
from oracle.bp import run_bp
from oracle.circuit import Noise, circuit_graph
from oracle.graph import circuit_tables
from oracle.sampler import pack_syndromes

pytestmark = pytest.mark.gpu

# the repository's bounds per message format: posteriors relative to |l| + 1, decision margins
RTOL = {"fp32": 1e-4, "fp16": 5e-3, "bf16": 4e-2}
TAU = {"fp32": 1e-2, "fp16": 0.2, "bf16": 1.5}
EDGES = sorted({1, 2, 3, 5} | {b + k for b in (8, 16, 24, 32, 48, 64, 80, 96) for k in (-1, 0, 1)})


@pytest.fixture(scope="module")
def torch():
    return torch_cuda()


_cache = {}


def _pair(d):
    if d not in _cache:
        og, _, _ = circuit_graph(d, Noise(0.005))
        _cache[d] = (pkg.Graph(d, "circuit", 0.005), og, circuit_tables(og))
    return _cache[d]


def _syndromes(torch, og, sizes, seed):
    rng = np.random.default_rng(seed)
    sb = np.zeros((len(sizes), og.n_det), dtype=bool)
    for r, s in enumerate(sizes):
        sb[r, rng.choice(og.n_det, size=s, replace=False)] = True
    packed = pack_syndromes(sb)
    return sb, packed, torch.as_tensor(packed.view(np.int32), device="cuda")


def _check_posteriors(ot, sb, sizes, got, T, rtol):
    worst = 0.0
    for k, s in enumerate(sizes):
        if s < 2:
            continue
        dets = np.flatnonzero(sb[k])
        L = ot.L[np.ix_(dets, dets)]
        lam = run_bp(L, T)[-1][1]
        worst = max(worst, float(np.max(np.abs(got[k][:s, :s].astype(np.float64) - lam) / (np.abs(L) + 1.0))))
    assert worst < rtol, worst


@pytest.mark.parametrize("prec", ["fp32", "fp16", "bf16"])
def test_list_edges_posteriors(torch, prec):
    g, og, ot = _pair(9)
    sizes = EDGES * 2  # two of each: the shots of a warp differ in size and content
    sb, _, synd = _syndromes(torch, og, sizes, seed=31)
    T = 4
    res = gpu_decode(g, synd, T, pkg.make_opts(precision=prec, early_exit=False), s_cap=100)
    assert list(res["s"]) == sizes
    _check_posteriors(ot, sb, sizes, res["lam"], T, RTOL[prec])


@pytest.mark.parametrize("prec,decoder,early,alpha,forced", [
    ("fp32", "bp4m", True, 1.0, "greedy"), ("fp32", "bp4m", False, 0.9, "static"), ("fp32", "bp4mf", False, 0.85, "greedy"),
    ("fp32", "bp4mf", False, 1.0, "static"), ("fp16", "bp4m", True, 1.0, "greedy"), ("fp16", "bp4mf", False, 1.0, "greedy")])
def test_list_edges_decisions(torch, prec, decoder, early, alpha, forced):
    g, og, ot = _pair(9)
    sizes = EDGES * 2
    sb, _, synd = _syndromes(torch, og, sizes, seed=32)
    T = 6
    opts = pkg.make_opts(precision=prec, early_exit=early, decoder=decoder, alpha=alpha, forced=forced)
    res = gpu_decode(g, synd, T, opts, s_cap=100)
    cnt, bad = compare_shots(ot, sb, res, T, range(len(sizes)), TAU[prec], decoder=decoder, early_exit=early, alpha=alpha,
                             forced=forced)
    assert all(m < TAU[prec] for _, m in bad), bad
    assert np.array_equal(res["obs"], res["obs2"]) and np.array_equal(res["flags"] & 1, res["conv"])


@pytest.mark.parametrize("prec,sizes", [("fp32", [641, 768]), ("fp32", [897, 1023, 1024]), ("fp16", [641, 1024])])
def test_widest_streaming_classes(torch, prec, sizes):
    g, og, ot = _pair(13)
    sb, _, synd = _syndromes(torch, og, sizes, seed=33)
    T = 2
    res = gpu_decode(g, synd, T, pkg.make_opts(precision=prec, early_exit=False), s_cap=1024)
    _check_posteriors(ot, sb, sizes, res["lam"], T, RTOL[prec])


@pytest.mark.parametrize("prec,decoder", [("fp64", "bp4m"), ("fp32", "bp4m"), ("fp32", "bp4mf"), ("fp16", "bp4m")])
@pytest.mark.parametrize("n", [1, 45, 2048, 2049])
def test_host_requests_match_device_batches(torch, prec, decoder, n):
    # small host batches are counted and listed on the host, larger and device batches on the
    # device; sizes from none to three streaming width classes
    g, og, _ = _pair(13)
    base = [0, 1, 2, 7, 16, 33, 64, 81, 113, 129, 145, 160, 161, 200, 257, 330] if n < 100 else [0, 1, 3, 9, 20, 40, 70]
    sizes = [170] if n == 1 else [base[k % len(base)] for k in range(n)]
    _, packed, synd = _syndromes(torch, og, sizes, seed=34)
    T = 5
    opts = pkg.make_opts(precision=prec, decoder=decoder)
    dev = [torch.zeros(n, dtype=t, device="cuda") for t in (torch.uint8, torch.uint8, torch.int16)]
    g.decode_batch(synd, T, opts, *dev)
    torch.cuda.synchronize()
    host = [np.full(n, 77, dtype=t) for t in (np.uint8, np.uint8, np.int16)]
    g.decode_batch(packed, T, opts, *host)
    for a, b in zip(dev, host):
        assert np.array_equal(a.cpu().numpy(), b)
    # outputs may be left out
    only = np.full(n, 77, dtype=np.uint8)
    g.decode_batch(packed, T, opts, None, only, None)
    assert np.array_equal(only, host[1])


@pytest.mark.parametrize("prec,decoder,forced", [("fp32", "bp4m", "greedy"), ("fp16", "bp4m", "static"), ("fp32", "bp4mf", "greedy"),
                                                 ("fp64", "bp4m", "greedy")])
@pytest.mark.parametrize("sizes", [[1, 9], [7, 15, 23, 31, 47, 63, 79, 95, 111, 127, 143, 159], [30, 161, 200, 257, 330],
                                   [2, 40, 100, 130, 190, 300, 700]])
def test_lists_beside_one_another_match_shots_alone(torch, prec, decoder, forced, sizes):
    # the lists of a batch run on several streams and its few large shots at one width; a shot
    # alone runs on one stream at its own width.  Two batches follow one another on the caller's
    # stream, the second over the first's lists, without a wait between them.
    g, og, _ = _pair(13)
    T = 6
    opts = pkg.make_opts(precision=prec, decoder=decoder, forced=forced)
    n = len(sizes)
    st = torch.cuda.Stream()
    runs = []
    for seed in (35, 36):
        _, _, synd = _syndromes(torch, og, sizes if seed == 35 else sizes[::-1], seed=seed)
        runs.append((synd, [torch.full((n,), 77, dtype=t, device="cuda") for t in (torch.uint8, torch.uint8, torch.int16)]))
    torch.cuda.synchronize()
    for synd, out in runs:
        g.decode_batch(synd, T, opts, *out, stream=st.cuda_stream)
    with torch.cuda.stream(st):
        got = [[x.clone() for x in out] for _, out in runs]
    st.synchronize()
    for (synd, _), out in zip(runs, got):
        for k in range(n):
            one = [torch.zeros(1, dtype=t, device="cuda") for t in (torch.uint8, torch.uint8, torch.int16)]
            g.decode_batch(synd[k:k + 1], T, opts, *one)
            torch.cuda.synchronize()
            assert [int(x[k]) for x in out] == [int(x[0]) for x in one], (prec, sizes, k)
