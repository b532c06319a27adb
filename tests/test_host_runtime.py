"""CPU tests of the host side of decoding calls (streams, lists, workspaces) on a stand-in CUDA runtime
whose streams run as late as allowed (fake_cuda.cpp)."""
import ctypes

import numpy as np
import pytest

from fake_cuda import Fake, build_fake

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
