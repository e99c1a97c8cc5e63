"""What the library's host code asks of the CUDA runtime, on the CPU: the sources are built against a stand-in runtime
(fake_cudart.cpp) that keeps shared-memory limits, can refuse a launch and writes down which kernels were launched."""
import ctypes as C
import glob
import os
import subprocess

import pytest

from paper_2608_07964_b200 import binding as B, build

HERE = os.path.dirname(os.path.abspath(__file__))
EB_ERR_CUDA = 4


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("host") / "libeb_host.so")
    # the device code is of no interest here: kept as PTX, which spares the assembler's time
    cmd = [build._nvcc(), "-gencode", "arch=compute_100a,code=compute_100a", "-O0", "-std=c++17", "--shared", "-cudart", "none", "-t", "8",
           "-Xcompiler", "-fPIC", "-Xlinker", "-Bsymbolic", "-I", os.path.join(build.ROOT, "include"),
           "-I", os.path.join(build.PKG, "csrc"), "-o", so, os.path.join(HERE, "fake_cudart.cpp")] + build.SOURCES
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    l = B.load_library(so)
    l.fake_name.restype = C.c_char_p
    l.fake_host_memory.restype = C.c_void_p
    return l


class Context:
    """A context whose buffers are addresses that nothing ever reads."""

    def __init__(self, lib, E, K, S, D, max_tokens, H=64, I=64, L=4):
        self.lib, self.D = lib, D
        self.ctx = C.c_void_p()
        e2d = (C.c_int32 * E)(*[e % D for e in range(E)])
        cfg = B.EbConfig(L, E, K, S, H, I, D, 1, max_tokens, e2d)
        assert lib.eb_create(C.byref(cfg), C.byref(self.ctx)) == 0
        assert lib.eb_set_workspace(self.ctx, 1 << 20, lib.eb_workspace_bytes(self.ctx)) == 0
        assert lib.eb_bind_weights(self.ctx, 1 << 30, 1 << 30, 1 << 30) == 0
        self.p = 1 << 30
        self.bufs = B.EbStepBuffers(*([self.p] * 15), None)

    def batch(self, n_mb, tokens):
        return B.Batch([j * tokens for j in range(n_mb + 1)], [j % 4 for j in range(n_mb)])

    def step(self, n_mb, tokens, m=1, policy=B.POLICY_MAXUTIL):
        b = self.batch(n_mb, tokens)
        return self.lib.eb_step(self.ctx, None, C.byref(b.c), b.pool_mask, m, policy, C.byref(self.bufs))

    def names(self):
        return [self.lib.fake_name(i).decode() for i in range(self.lib.fake_launched())]


SHAPES = [dict(E=256, K=8, S=8, D=16), dict(E=64, K=6, S=2, D=8), dict(E=60, K=4, S=4, D=8), dict(E=8, K=2, S=0, D=4)]


def test_a_context_keeps_its_shared_memory_whatever_others_do(lib):
    """The shared-memory limit belongs to the kernel, not to the context that sets it: contexts of other shapes, smaller
    and larger ones, may make their first step at any time between the steps of one."""
    lib.fake_reset(-1)
    ctxs = [Context(lib, max_tokens=16 * 96, **s) for s in SHAPES]
    for order in ((0, 1, 2, 3), (3, 2, 1, 0), (1, 3, 0, 2)):
        for i in order:
            assert ctxs[i].step(16, 96) == 0 and ctxs[i].step(4, 3) == 0, SHAPES[i]
    late = Context(lib, max_tokens=64, E=2, K=1, S=0, D=1)
    assert late.step(4, 3) == 0
    for c, s in zip(ctxs, SHAPES):
        assert c.step(16, 96) == 0, s


def _calls(c, n_mb, tokens):
    """Every call that enqueues kernels, by name."""
    l, b, p = c.lib, c.batch(n_mb, tokens), c.p
    ref = C.byref(b.c)
    bad, gave_up = C.c_int32(), C.c_int32()
    e2d = (C.c_int32 * 8)(*[e % 4 for e in range(8)])
    cfg = B.EbConfig(4, 8, 2, 1, 64, 64, 4, 1, 4096, e2d)
    err = C.create_string_buffer(256)
    return dict(
        route=lambda: l.eb_route(c.ctx, None, ref, b.pool_mask, p, p, p, p, p),
        schedule=lambda: l.eb_schedule(c.ctx, None, ref, 1, 0, p, p, None),
        permute=lambda: l.eb_permute(c.ctx, None, ref, p, p, p, p, p, p, p, p, p),
        permute_noalloc=lambda: l.eb_permute_noalloc(C.byref(cfg), None, ref, p, p, p, p, p, p, p, p, p, err, 256),
        expert_ffn=lambda: l.eb_expert_ffn_grouped(c.ctx, None, p, p, p, p, p),
        expert_ffn_device=lambda: l.eb_expert_ffn_device(c.ctx, None, p, p, p, p, p, 1),
        copy_16=lambda: l.eb_copy(c.ctx, None, p, p + 4096, 48),
        copy_4=lambda: l.eb_copy(c.ctx, None, p + 4, p + 4096, 48),
        copy_1=lambda: l.eb_copy(c.ctx, None, p, p + 4096, 47),
        combine=lambda: l.eb_combine(c.ctx, None, ref, p, p, p, p, p),
        step=lambda: c.step(n_mb, tokens),
        step_host=lambda: l.eb_step_host(c.ctx, None, ref, b.pool_mask, 1, 0, C.byref(c.bufs), p, p, p, None),
        check_permutation=lambda: l.eb_check_permutation(c.ctx, None, ref, p, p, p, p, p, p, p, C.byref(bad)),
        check_guards=lambda: l.eb_check_workspace_guards(c.ctx, None, C.byref(bad)),
        selftest=lambda: l.eb_selftest_bounded_wait(c.ctx, None, 1000, C.byref(gave_up)))


@pytest.mark.parametrize("timing", [0, 1])
@pytest.mark.parametrize("n_mb,tokens", [(3, 5), (8, 400), (1, 4096)])   # the fused permute kernel, the four it stands for, sums of histograms
def test_nothing_is_launched_behind_a_refused_kernel(lib, n_mb, tokens, timing):
    """Each kernel of a call works from what the one before it wrote: when the runtime refuses one, the call says so and
    launches no further kernel, and the next call starts clean."""
    lib.fake_reset(-1)
    c = Context(lib, E=8, K=2, S=1, D=4, max_tokens=4096)
    assert lib.eb_set_timing(c.ctx, timing) == 0
    for name, call in _calls(c, n_mb, tokens).items():
        lib.fake_reset(-1)
        assert call() == 0, name
        chain = c.names()
        assert chain, name
        for i in range(len(chain)):
            lib.fake_reset(i)
            assert call() == EB_ERR_CUDA, (name, chain[i])
            assert c.names() == chain[:i], (name, chain[i])
            lib.fake_reset(-1)
            assert call() == 0 and c.names() == chain, (name, chain[i], "afterwards")


def test_the_library_finds_every_runtime_function_in_the_stand_in(lib):
    """Nothing of the real runtime, which torch may have put in reach, is called in its place."""
    r = subprocess.run(["nm", "-D", "--undefined-only", lib._name], capture_output=True, text=True)
    assert r.returncode == 0
    assert [n for n in r.stdout.split() if n.startswith(("cuda", "__cuda", "cu"))] == []


def test_copies_look_at_their_arguments(lib):
    lib.fake_reset(-1)
    c = Context(lib, E=8, K=2, S=1, D=4, max_tokens=64)
    assert lib.eb_copy(None, None, 16, 32, 4) == 1
    assert lib.eb_copy(c.ctx, None, None, 32, 4) == 1 and lib.eb_copy(c.ctx, None, 16, None, 4) == 1
    assert lib.eb_copy(c.ctx, None, None, None, 0) == 0 and c.names() == []


def _wait(c, ticket, n_mb=4, res=1 << 30, load=1 << 30):
    h, ld = B.EbSchedResult(), (C.c_int32 * (16 * c.D))()
    code = c.lib.eb_schedule_wait(c.ctx, None, ticket, n_mb, res, load, C.addressof(h), C.addressof(ld))
    return code, h, ld


def test_watched_schedules_keep_their_contract(lib):
    """Which tickets can be waited for, and when the device's buffers are fallen back on (the stand-in's copies leave the result
    as it was: zeros), when the record is read."""
    lib.fake_reset(-1)
    c = Context(lib, E=8, K=2, S=1, D=4, max_tokens=4096)
    INVALID, UNSUPPORTED = 1, 2
    assert lib.eb_watch_schedule(None, 1) == INVALID
    assert _wait(c, 5)[0] == INVALID                     # nothing was ever watched
    assert lib.eb_watch_schedule(c.ctx, 0) == 0 and _wait(c, 5)[0] == INVALID
    assert lib.eb_watch_schedule(c.ctx, 5) == 0
    assert _wait(c, 0)[0] == INVALID and _wait(c, 6)[0] == INVALID
    assert _wait(c, 5, res=None)[0] == INVALID and _wait(c, 5, load=None)[0] == INVALID
    assert _wait(c, 5, n_mb=17)[0] == UNSUPPORTED and _wait(c, 5, n_mb=-1)[0] == UNSUPPORTED
    assert _wait(c, 5)[0] == 0                           # nothing was launched: the stream is idle
    assert lib.eb_watch_schedule(c.ctx, 6) == 0
    assert _wait(c, 5)[0] == INVALID                     # its record may be written over
    # captured, refused: no mark is on its way
    lib.fake_capturing(1)
    assert c.step(4, 3) == 0 and _wait(c, 6)[0] == 0
    lib.fake_capturing(0)
    lib.fake_reset(-1)
    assert c.step(4, 3) == 0
    chain = c.names()
    scatter = [i for i, n in enumerate(chain) if "scatter" in n][0]
    assert lib.eb_watch_schedule(c.ctx, 7) == 0
    lib.fake_reset(scatter)
    assert c.step(4, 3) == EB_ERR_CUDA and _wait(c, 7)[0] == 0
    # launched: the mark is waited for, and the record is what comes back
    lib.fake_reset(-1)
    for call in (lambda: c.step(4, 3), _calls(c, 4, 3)["schedule"]):
        assert lib.eb_watch_schedule(c.ctx, 8) == 0
        assert call() == 0
        words = (C.c_uint32 * (24 + 256 + 1)).from_address(lib.fake_host_memory())
        assert words[280] == 0
        words[0], words[24], words[39], words[280] = 0xb, 41, 43, 8
        code, h, ld = _wait(c, 8)
        assert code == 0 and h.run_mask == 0xb and ld[0] == 41 and ld[15] == 43 and ld[16] == 0
    assert lib.eb_watch_schedule(c.ctx, 0) == 0 and _wait(c, 8)[0] == 0      # the mark stays
    assert lib.eb_watch_schedule(c.ctx, 8) == 0 and words[280] == 0          # and is cleared with the next ticket
    assert lib.eb_destroy(c.ctx) == 0 and lib.fake_host_memory() is None
