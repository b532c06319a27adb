"""CPU tests of the host side of decoding calls (streams, lists, workspaces) on a stand-in CUDA runtime
whose streams run as late as allowed (fake_cuda.cpp)."""
import ctypes

import numpy as np
import pytest

from fake_cuda import CLASSIFY, GLOBAL, Fake, build_fake
from paper_2603_05381_gb300 import _capi

# defect counts: none, every list, and four streaming width classes
SIZES = [0, 1, 5, 9, 20, 30, 40, 60, 70, 90, 100, 120, 140, 150, 161, 200, 257, 330, 64, 8]


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    return Fake(build_fake(tmp_path_factory.mktemp("fake")))


def _out(fake, n, where):
    return [fake.buffer(n, t, where) for t in (np.uint8, np.uint8, np.int16)]


def _same(fake, synd, out):
    return all(np.array_equal(a, b) for a, b in zip(out, fake.expected(synd)))


@pytest.mark.parametrize("where", ["pageable", "pinned", "device"])
@pytest.mark.parametrize("n", [1, 20, 300, 2048, 2049])
def test_batches_reach_their_lists(fake, where, n):
    fake.lib.fake_reset()
    g = fake.graph()
    rows = fake.syndromes(g, [SIZES[(7 * k) % len(SIZES)] for k in range(n)], seed=n)
    synd = fake.buffer(rows.size, np.uint32, where).reshape(rows.shape)
    synd[:] = rows
    out = _out(fake, n, where)
    assert fake.decode(g, synd, out) == 0
    assert _same(fake, rows, out) and fake.lib.fake_list_errors() == 0


@pytest.mark.parametrize("n", [3, 2048, 2049])
@pytest.mark.parametrize("where", ["pageable", "pinned"])
@pytest.mark.parametrize("writer,caller", [("nonblocking",) * 2, ("blocking",) * 2, ("legacy",) * 2, ("blocking", "legacy"), ("legacy", "blocking")])
def test_host_rows_are_read_after_the_work_queued_before_the_call(fake, writer, caller, where, n):
    # rows written by work queued in the caller's stream, or in one that the legacy stream's rules
    # order before it
    fake.lib.fake_reset()
    g = fake.graph()
    streams = {"legacy": None, "nonblocking": fake.stream(), "blocking": fake.stream(nonblocking=False)}
    rows = fake.syndromes(g, [SIZES[(3 * k) % len(SIZES)] for k in range(n)], seed=9)
    synd = fake.buffer(rows.size, np.uint32, where).reshape(rows.shape)
    out = _out(fake, n, where)
    fake.lib.fake_enqueue_write(streams[writer], synd.ctypes.data, rows.ctypes.data, rows.nbytes)
    assert fake.decode(g, synd, out, stream=streams[caller]) == 0
    assert _same(fake, rows, out)
    for s in streams.values():
        if s:
            fake.lib.cudaStreamDestroy(s)


def test_an_error_of_one_call_does_not_fail_the_next(fake):
    # the runtime keeps the last error until it is asked for: the next call's launches ask
    fake.lib.fake_reset()
    g = fake.graph()
    rows = fake.syndromes(g, SIZES, seed=4)
    synd = fake.buffer(rows.size, np.uint32, "device").reshape(rows.shape)
    synd[:] = rows
    out = _out(fake, len(SIZES), "device")
    for k in range(1, 4):
        fake.lib.fake_fail_launch(k)
        assert fake.decode(g, synd, out) != 0
        fake.lib.fake_fail_launch(0)
        fake.lib.cudaDeviceSynchronize()
        assert fake.decode(g, synd, out) == 0 and _same(fake, rows, out)


@pytest.mark.parametrize("call", ["pageable", "pinned", "device", "sample", "bbp4mf", "fused", "service"])
def test_a_failed_launch_leaves_no_work_behind(fake, call):
    # every launch of a call in turn is made to fail: the call returns an error with nothing queued
    # (its buffers and staging may be used again), and the next call is right
    lib = fake.lib
    lib.fake_reset()
    opts = _capi.Opts(_capi.FP32, 1, 0, 1.0, 0, 0, 0, 0)
    bbp = call == "bbp4mf"
    g = fake.graph(5, _capi.CODE_CAPACITY, 0.1) if bbp else fake.graph()
    n = 60
    sizes = [k % 9 for k in range(n)] if bbp else [SIZES[(3 * k) % len(SIZES)] for k in range(n)]
    rows = fake.syndromes(g, sizes, seed=9)
    where = call if call in ("pageable", "pinned", "device") else "pageable"
    synd = fake.buffer(rows.size, np.uint32, where).reshape(rows.shape)
    synd[:] = rows
    out = _out(fake, n, where)
    server = multi = None
    if call == "service":
        server = lib.bp4m_server_create(1, 64, 0)
        gid = lib.bp4m_server_add_graph(server, g)
    if call == "fused":
        hs, ns = (ctypes.c_void_p * 1)(g.value), (ctypes.c_int64 * 1)(n)
        multi = lib.bp4m_multi_create(1, hs, None, ns, 5, ctypes.byref(opts), 448, 0)
        assert multi

    def run():
        if call == "sample":
            return lib.bp4m_sample_and_decode_range(g, 0, n, 1, 0, 5, ctypes.byref(opts), ctypes.byref(_capi.Counts()), None)
        if bbp:
            two = np.concatenate([rows.ravel(), rows.ravel()])
            return lib.bp4m_decode_bbp4mf(g, two.ctypes.data, n, 5, ctypes.byref(opts), np.zeros(2 * n, np.uint8).ctypes.data, None, None)
        if server:
            r = lib.bp4m_server_submit(server, gid, rows.ctypes.data, n, 5, ctypes.byref(opts), out[0].ctypes.data, out[1].ctypes.data)
            return lib.bp4m_server_wait(server, r, -1.0, None)
        if multi:
            ptr = [(ctypes.c_void_p * 1)(x.ctypes.data) for x in (synd, out[0], out[1])]
            return lib.bp4m_multi_run(multi, ptr[0], ns, ptr[1], ptr[2])
        return fake.decode(g, synd, out)

    for k in range(1, 200):
        lib.fake_fail_launch(k)
        rc = run()
        pending = lib.fake_pending()
        lib.fake_fail_launch(0)
        if rc == 0:
            break
        assert pending == 0, k
        assert run() == 0 and lib.fake_pending() == 0
        if call in ("pageable", "pinned", "device"):
            assert _same(fake, rows, out)
    assert rc == 0 and k >= (4 if multi else 5)
    if server:
        lib.bp4m_server_destroy(server)
    if multi:
        lib.bp4m_multi_destroy(multi)


@pytest.mark.parametrize("left", [0, 1, 4, 7])
@pytest.mark.parametrize("where", ["pageable", "device"])
def test_a_batch_is_decoded_on_the_streams_there_are(fake, where, left):
    # no more than `left` further streams can be made: the lists share them, or run on the caller's
    lib = fake.lib
    lib.fake_reset()
    g = fake.new_graph(13)
    rows = fake.syndromes(g, SIZES, seed=6)
    synd = fake.buffer(rows.size, np.uint32, where).reshape(rows.shape)
    synd[:] = rows
    out = _out(fake, len(SIZES), where)
    for k in range(2):
        lib.fake_fail_stream_create(left if k == 0 else -1)
        assert fake.decode(g, synd, out) == 0, lib.bp4m_last_error()
        assert _same(fake, rows, out) and lib.fake_list_errors() == 0
    lib.bp4m_free_graph(g)


@pytest.mark.parametrize("where", ["pageable", "device"])
def test_every_list_has_the_callers_priority(fake, where):
    lib = fake.lib
    lib.fake_reset()
    g = fake.graph()
    rows = fake.syndromes(g, SIZES, seed=7)
    synd = fake.buffer(rows.size, np.uint32, where).reshape(rows.shape)
    synd[:] = rows
    out = _out(fake, len(SIZES), where)
    used = set()
    for prio in (0, -2, -5, 0):
        st = fake.stream(prio=prio)
        lib.fake_reset()
        assert fake.decode(g, synd, out, stream=st) == 0 and _same(fake, rows, out)
        got = fake.launches()
        assert np.all(got[:, 3] == prio) and len(set(got[:, 2])) > 5
        # a priority's streams are made once
        used |= {(p, s) for p, s in got[:, [3, 2]].tolist() if s != got[0, 2]}
        lib.cudaStreamDestroy(st)
    assert len(used) == 3 * 8


def test_streams_of_a_service_belong_to_its_slots(fake):
    # a slot decodes one batch at a time: its streams serve every graph it meets
    lib = fake.lib
    lib.fake_reset()
    opts = _capi.Opts(_capi.FP32, 1, 0, 1.0, 0, 0, 0, 0)
    graphs = [fake.graph(13), fake.graph(11), fake.graph(9), fake.graph(7)]
    sizes = [1, 9, 20, 30, 40, 60, 70, 90]
    rows = [fake.syndromes(g, sizes, seed=8) for g in graphs]
    before, slots = lib.fake_streams(), 2
    server = lib.bp4m_server_create(slots, 64, 0)
    ids = [lib.bp4m_server_add_graph(server, g) for g in graphs]
    for _ in range(6):
        reqs = []
        for gid, r in zip(ids, rows):
            out = [np.zeros(len(sizes), np.uint8) for _ in range(2)]
            reqs.append((lib.bp4m_server_submit(server, gid, r.ctypes.data, len(sizes), 5, ctypes.byref(opts), out[0].ctypes.data,
                                                out[1].ctypes.data), r, out))
        for rid, r, out in reqs:
            assert lib.bp4m_server_wait(server, rid, -1.0, None) == 0
            assert all(np.array_equal(a, b) for a, b in zip(out, Fake.expected(r)[:2]))
    assert lib.fake_max_streams() <= before + slots * (1 + 8)
    lib.bp4m_server_destroy(server)
    assert lib.fake_streams() == before


def test_a_graphs_streams_outlive_its_workspace(fake):
    # larger batches and other error rates reuse the streams
    lib = fake.lib
    lib.fake_reset()
    g = fake.new_graph(5)
    before = lib.fake_streams()
    opts = _capi.Opts(_capi.FP32, 1, 0, 1.0, 0, 0, 0, 0)
    for n in (30, 300, 3000):
        rows = fake.syndromes(g, [(5 * k) % 60 for k in range(n)], seed=n)
        synd = fake.buffer(rows.size, np.uint32, "device").reshape(rows.shape)
        synd[:] = rows
        out = _out(fake, n, "device")
        assert fake.decode(g, synd, out) == 0 and _same(fake, rows, out)
    for p in (0.004, 0.006):
        assert lib.bp4m_sample_and_decode(g, p, 300, 1, 5, ctypes.byref(opts), ctypes.byref(_capi.Counts()), None) == 0
    used = set(fake.launches()[:, 2].tolist())
    assert lib.fake_streams() - before <= 8 and len(used) <= 9
    lib.bp4m_free_graph(g)
    assert lib.fake_streams() == before
    # a graph of which only another error rate's was used
    g = fake.new_graph(5)
    assert lib.bp4m_sample_and_decode(g, 0.004, 300, 1, 5, ctypes.byref(opts), ctypes.byref(_capi.Counts()), None) == 0
    lib.bp4m_free_graph(g)
    assert lib.fake_streams() == before


@pytest.mark.parametrize("d,n,on_host", [(3, 2048, True), (3, 2049, False), (13, 1700, True), (13, 1800, False)])
def test_host_counts_small_batches_only(fake, d, n, on_host):
    # at most 2048 shots and 65,536 words of rows (37 a row at d = 13): beyond that the host's count
    # takes longer than the launches it saves
    lib = fake.lib
    lib.fake_reset()
    g = fake.graph(d)
    rows = fake.syndromes(g, [k % 9 for k in range(n)], seed=n)
    out = _out(fake, n, "pageable")
    assert fake.decode(g, rows, out) == 0 and _same(fake, rows, out)
    assert (CLASSIFY not in fake.launches()[:, 0]) == on_host


@pytest.mark.parametrize("where", ["pageable", "device"])
def test_small_width_classes_run_beside_the_largest(fake, where):
    # two shots of one class and one of each of two others, all classes of few shots: the first stays
    # on the caller's stream, the others share the second
    lib = fake.lib
    lib.fake_reset()
    g = fake.graph()
    rows = fake.syndromes(g, [300, 170, 250, 310, 410], seed=11)
    synd = fake.buffer(rows.size, np.uint32, where).reshape(rows.shape)
    synd[:] = rows
    out = _out(fake, len(rows), where)
    st = fake.stream()
    assert fake.decode(g, synd, out, stream=st) == 0 and _same(fake, rows, out) and lib.fake_list_errors() == 0
    got = {int(w): int(s) for k, w, s, _ in fake.launches() if k == GLOBAL}
    assert len(got) == 4 and got[192] == got[256] == got[448] and got[320] != got[192]
    lib.cudaStreamDestroy(st)
