"""The host side of the library (api.cu, attn_static.cu) linked against stand-ins for the CUDA runtime and
the kernel launchers (host_fakes.cpp): what it hands from call to call, without a GPU."""
import ctypes as C
import os
import subprocess

import pytest

from paper_2512_04939_b200.binding import AttnExt, Config

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2512_04939_b200", "csrc")


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("host") / "libhost.so")
    # (-Bsymbolic: its own stand-ins, not the runtime that torch has loaded into the process)
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-w", "-Wl,-Bsymbolic", "-I/usr/local/cuda/include", "-x", "c++",
                    os.path.join(CSRC, "api.cu"), os.path.join(CSRC, "attn_static.cu"), os.path.join(HERE, "host_fakes.cpp"),
                    "-o", so], check=True)
    lib = C.CDLL(so)
    lib.fake_norm_seen.restype = lib.fake_norm_last_seen.restype = C.c_float
    return lib


class Ctx:
    def __init__(self, lib, qkv_dtype=0):
        cfg = Config()
        assert lib.litevggt_default_config(3, 4, 5, C.c_float(0.5), C.byref(cfg)) == 0
        cfg.qkv_dtype = qkv_dtype
        self.lib, self.h = lib, C.c_void_p()
        assert lib.litevggt_create(C.byref(cfg), 0, C.byref(self.h)) == 0
        n, m = C.c_int64(), C.c_int64()
        lib.litevggt_sizes(self.h, C.byref(n), C.byref(m), None, None, None)
        self.n, self.m = n.value, m.value
        self.buf = C.create_string_buffer(1 << 12)
        self.p = C.c_void_p((C.addressof(self.buf) + 255) & ~255)  # the stand-ins read none of it

    def layernorm(self, rows):
        return self.lib.litevggt_layernorm(self.h, self.p, C.c_int64(rows), self.p, self.p, C.c_float(1e-6), self.p, None)

    def mlp(self, rows):
        p = self.p
        return self.lib.litevggt_mlp(self.h, p, C.c_int64(rows), p, p, p, p, None, p, None)

    def global_attn(self):
        p = self.p
        return self.lib.litevggt_global_attn(self.h, p, C.c_int64(self.m), p, p, p, p, p, None)

    def global_attn_ext(self, normed):
        p, ext = self.p, AttnExt()
        if normed:
            ext.q_norm_gamma = ext.q_norm_beta = ext.k_norm_gamma = ext.k_norm_beta = p
        ext.norm_eps = 1e-5
        return self.lib.litevggt_global_attn_ext(self.h, None, p, C.c_int64(self.m), p, p, p, p, C.byref(ext), p, None)

    def frame_attn(self):
        p = self.p
        return self.lib.litevggt_frame_attn(self.h, p, p, p, p, p, None, p, None)

    def merge_plan(self):
        plan = C.c_void_p()
        assert self.lib.litevggt_merge_plan(self.h, self.p, self.p, C.byref(plan), None) == 0
        return plan

    def timer(self, which):
        ms, count, one = C.c_float(), C.c_int32(), (C.c_float * 64)()
        assert self.lib.litevggt_timer_samples(self.h, which, one, 64, C.byref(count)) == 0
        samples = [round(v * 1e6) for v in one[:count.value]]
        assert self.lib.litevggt_timer_read(self.h, which, C.byref(ms), C.byref(count)) == 0
        assert count.value == len(samples) and round(ms.value * 1e6) == sum(samples)
        return samples  # nanoseconds


@pytest.mark.parametrize("which", [10, 12, 13, 8])
def test_a_step_that_launched_nothing_took_no_time(host, which):
    """LayerNorm and MLP of no rows, the Q/K pass with neither option, an output projection that is refused:
    their records are zero, also where the ring slot held an earlier step's times."""
    c = Ctx(host)
    busy = {10: lambda: c.layernorm(7), 12: lambda: c.mlp(7), 13: lambda: c.global_attn_ext(True), 8: c.global_attn}[which]
    each = 1000 if which == 12 else 500  # the stand-in kernels take 500 ns, the MLP has two
    for _ in range(64):
        assert busy() == 0
    assert c.timer(which) == [each] * 64
    if which == 8:
        host.fake_fail_linear(1)
        assert c.global_attn() != 0
    else:
        assert {10: lambda: c.layernorm(0), 12: lambda: c.mlp(0), 13: lambda: c.global_attn_ext(False)}[which]() == 0
    assert c.timer(which) == [each] * 63 + [0]
    host.litevggt_timers_reset(c.h)
    assert busy() == 0
    assert c.timer(which) == [each]
    host.litevggt_destroy(c.h)


@pytest.mark.parametrize("entry", ["global_attn", "frame_attn", "static"])
def test_key_norms_are_zero_after_a_call_that_failed_half_way(host, entry):
    """The projection raises the key norms, the output projection zeroes them; where that one is refused, the
    next call - also of the other layer, with more or fewer sequences - must not start from what is left."""
    c = Ctx(host)
    buf = C.create_string_buffer(1 << 12)
    p = C.c_void_p((C.addressof(buf) + 255) & ~255)

    def static():
        return host.litevggt_global_attn_static(p, C.c_int64(100), p, p, p, p, p, p, None)

    call = static if entry == "static" else getattr(c, entry)
    for follow in (call, c.frame_attn if entry != "static" else call):
        assert call() == 0 and call() == 0
        assert host.fake_norm_seen() == 0.0 and host.fake_norm_last_seen() == 0.0
        host.fake_fail_linear(1)
        assert call() != 0
        assert follow() == 0
        assert host.fake_norm_seen() == 0.0 and host.fake_norm_last_seen() == 0.0
    host.litevggt_destroy(c.h)


def test_a_new_context_has_nothing_pending_on_the_default_stream(host):
    """The key norms and stopwatch stamps start at zero.  A caller's stream that does not wait for the default
    stream may use the context at once: a late clearing would wipe norms between projection and attention."""
    for _ in range(2):
        c = Ctx(host)
        assert host.fake_default_stream_pending() == 0
        host.litevggt_destroy(c.h)


def test_a_new_plan_is_cleared_on_the_stream_that_fills_it(host):
    c = Ctx(host)
    plan = c.merge_plan()
    assert host.fake_default_stream_pending() == 0
    assert host.litevggt_plan_destroy(plan) == 0
    host.litevggt_destroy(c.h)
