"""What the host entry points leave to their streams and events: the host side of the library linked against
stand-ins that keep track of which memory every stream's work touches and of what nothing orders (host_fakes.cpp)."""
import ctypes as C
import os
import subprocess

import pytest

from paper_2512_04939_b200.binding import Config

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2512_04939_b200", "csrc")


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("host") / "libhost.so")
    sources = [os.path.join(CSRC, f) for f in ("api.cu", "attn_static.cu", "host_pipeline.cu")] + [os.path.join(HERE, "host_fakes.cpp")]
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-w", "-Wl,-Bsymbolic", "-I/usr/local/cuda/include", "-x", "c++",
                    *sources, "-o", so], check=True)
    return C.CDLL(so)


class Layer:
    """A context of three 37 x 37 frames, a plan and page-locked buffers, every call on another pair of them."""

    def __init__(self, lib, ratio=0.0, frames=3):
        cfg = Config()
        assert lib.litevggt_default_config(frames, 37, 37, C.c_float(ratio), C.byref(cfg)) == 0
        self.lib, self.h, self.plan = lib, C.c_void_p(), C.c_void_p()
        assert lib.litevggt_create(C.byref(cfg), 0, C.byref(self.h)) == 0
        n = C.c_int64()
        lib.litevggt_sizes(self.h, C.byref(n), None, None, None, None)
        self.n, self.kept = n.value, []
        self.p = self.buffer(1 << 12)
        lib.fake_forget_accesses()
        assert lib.litevggt_merge_plan(self.h, self.buffer(2048 * self.n), self.p, C.byref(self.plan), None) == 0

    def buffer(self, size):
        self.kept.append(C.create_string_buffer(size + 256))
        return C.c_void_p((C.addressof(self.kept[-1]) + 255) & ~255)

    def call(self, entry, grad=False, out=None):
        p, x, out = self.p, self.buffer(2048 * self.n), out or self.buffer(2048 * self.n)
        return getattr(self.lib, entry)(self.h, C.byref(self.plan), p if grad else None, x, p, p, p, p, out, None)

    def drain(self):
        assert self.lib.litevggt_host_drain(self.h, None) == 0

    def close(self):
        self.lib.litevggt_plan_destroy(self.plan)
        self.lib.litevggt_destroy(self.h)


PIPED, ORDERED = "litevggt_global_layer_host_pipelined", "litevggt_global_layer_host"


@pytest.mark.parametrize("ratio", [0.0, 0.4])  # 4,122 merged rows leave in slabs, 2,474 behind the layer
@pytest.mark.parametrize("calls", [(PIPED, ORDERED), (ORDERED, PIPED), (PIPED, PIPED, PIPED, PIPED), (PIPED, PIPED, ORDERED, PIPED, ORDERED, PIPED)])
def test_nothing_unordered_between_host_entries(host, calls, ratio):
    """The pipelined entry's copies and writers run on streams of their own; whatever the next call does, of either entry,
    on a plan that it rebuilds in place, must not meet them in memory."""
    layer = Layer(host, ratio)
    for entry in calls:
        assert layer.call(entry, grad=True) == 0
    assert host.fake_races() == 0
    layer.close()


@pytest.mark.parametrize("locked,direct", [
    ([(0, 1)], True), ([(-4096, 2)], True),                             # one range, from the buffer's start or before
    ([(0, 0.999)], False), ([(4096, 1)], False),                        # its end or its beginning is not in it
    ([(0, 0.25), (0.75, 0.25)], False), ([(0, 0.5), (0.5, 0.5)], False),  # both ends are, in two ranges
    ([(0, -1)], False)])                                                # nothing is page-locked
def test_only_a_buffer_in_one_page_locked_range_is_written_by_kernels(host, locked, direct):
    """Kernels write the output only where one page-locked range holds all of it; any other buffer gets a copy."""
    layer = Layer(host)
    size = 2048 * layer.n
    out = layer.buffer(size)
    for at, length in locked:
        begin = out.value + int(at if abs(at) > 1 else at * size)
        host.fake_page_lock(C.c_void_p(begin), C.c_longlong(int(length * size)))
    before = host.fake_rows_written()
    assert layer.call(PIPED, out=out) == 0
    assert (host.fake_rows_written() > before) == direct
    host.fake_page_lock_all()
    layer.close()


@pytest.mark.parametrize("sms", [1, 7, 8, 15, 16, 20, 36, 74, 132, 148])
@pytest.mark.parametrize("rows", [1, 4096, 4097, 22000, 40000, 65535, 65536, 65537, 4000000])
def test_slabs_cover_a_sequence_on_any_number_of_sms(host, rows, sms):
    """In order, in whole query blocks, no more of them than there are job counters - or the sequence as a whole."""
    end = lambda row0: host.fake_slab_end(C.c_longlong(rows), C.c_longlong(row0), sms)
    host.fake_slab_end.restype = C.c_longlong
    row0, slabs = 0, 0
    while row0 < rows:
        row1 = end(row0)
        assert row0 < row1 <= rows and slabs < 64
        if rows > row1 or row0 > 0:
            assert host.fake_slab_index(C.c_longlong(row0), sms) == slabs and row0 % 256 == 0
        row0, slabs = row1, slabs + 1
    if rows <= 4096 or rows > 65536 or sms < 16:
        assert slabs == 1
    if sms == 148 and 4096 < rows <= 65536:
        assert slabs > 1


@pytest.mark.parametrize("sms", [12, 20])
def test_a_layer_of_a_partitioned_gpu_leaves_for_host_memory(host, sms):
    host.fake_sms(sms)
    layer = Layer(host)
    before = host.fake_rows_written()
    assert layer.call(PIPED) == 0 and layer.call(PIPED, grad=True) == 0
    assert (host.fake_rows_written() > before) == (sms >= 16) and host.fake_races() == 0
    layer.close()
    host.fake_sms(148)


def test_in_a_stream_of_calls_copies_take_the_output(host):
    """Kernels write the output of a call that follows a drain (or nothing); without one in between, the copy of a call is
    hidden behind the next one's kernels and takes no SM from them."""
    layer = Layer(host)
    direct = []
    for drain in (False, False, True, False, True, True, False):
        before = host.fake_rows_written()
        assert layer.call(PIPED) == 0
        direct.append(host.fake_rows_written() > before)
        if drain:
            layer.drain()
    assert direct == [True, False, False, True, False, True, True]
    assert host.fake_races() == 0
    layer.close()


def test_one_stopwatch_record_per_layer_and_step(host):
    """4,122 rows in two slabs: attention, output projection and unmerge are launched once for each, 500 ns by the stand-ins'
    clock, and leave one record of both, also when the ring has come round and where whole layers' records come between."""
    layer = Layer(host)

    def samples(which):
        one, count = (C.c_float * 64)(), C.c_int32()
        assert host.litevggt_timer_samples(layer.h, which, one, 64, C.byref(count)) == 0
        return [round(v * 1e6) for v in one[:count.value]]

    for call in range(3):
        assert layer.call(PIPED) == 0  # in slabs
        if call == 1:
            assert layer.call(ORDERED) == 0
        layer.drain()
    for which in (7, 8, 9):
        assert samples(which) == [1000, 1000, 500, 1000]
    x, out = layer.buffer(2048 * layer.n), layer.buffer(2048 * layer.n)
    for _ in range(70):
        assert host.litevggt_global_layer_host_pipelined(layer.h, C.byref(layer.plan), None, x, *[layer.p] * 4, out, None) == 0
        layer.drain()
    for which in (7, 8, 9):
        assert samples(which) == [1000] * 64
    host.fake_fail_linear(1)
    assert layer.call(PIPED) != 0
    assert samples(7) == [1000] * 63 + [0] and samples(8) == [1000] * 63 + [0] and samples(9) == [1000] * 64
    layer.close()


def test_a_poll_sees_what_the_writers_of_an_output_have_flagged(host):
    """The kernels that write an output check their indices on a stream of the context's own; a poll comes after them
    without a drain.  (An unordered read of the status word would count as a race.)"""
    layer = Layer(host)
    for _ in range(2):
        assert layer.call(PIPED) == 0
        assert host.litevggt_poll_device_status(layer.h, None) == 0
    assert host.fake_races() == 0
    layer.close()


@pytest.mark.parametrize("frames,ratio,direct", [(3, 0.0, True), (5, 0.3, True), (7, 0.55, False), (6, 0.47, False), (3, 0.01, False)])
def test_short_sequences_of_many_tokens_leave_by_a_copy(host, frames, ratio, direct):
    """4,122 rows of as many tokens, 4,809 of 6,870 | 4,386 of 9,618, 4,370 of 8,244, 4,081 of 4,122."""
    layer = Layer(host, ratio, frames)
    before = host.fake_rows_written()
    assert layer.call(PIPED) == 0
    assert (host.fake_rows_written() > before) == direct
    layer.close()
