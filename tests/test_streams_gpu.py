"""The library under several streams, in CUDA graphs and with a host that is out of memory: what include/bigbird.h says
about overlap, capture and error codes."""
import ctypes
import os
import subprocess
import sys
import textwrap

import pytest
import torch

import paper_2007_14062_b200 as bb
from paper_2007_14062_b200 import synth

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


class Problem:
    """Inputs of one call on the GPU, and its results on the default stream."""

    def __init__(self, dtype, B, H, nb, seed, lengths=None, mode=0, g=2, r=3):
        wl = self.wl = synth.Workload("streams", dtype, B, H, nb * 64, 64, 64, 3, g, r, mode, seed=seed)
        dev = torch.device("cuda:0")
        gen = torch.Generator(dev).manual_seed(seed)
        self.q, self.k, self.v, self.dout = (torch.randn((B, H, wl.N, 64), generator=gen, device=dev).to(synth.torch_dtype(dtype)) for _ in range(4))
        self.mask = None
        if lengths is not None:
            self.mask = (torch.arange(wl.N)[None, :] < torch.tensor(lengths)[:, None]).to(torch.uint8).to(dev)
        self.layout = bb.bigbird_build_layout(wl.N, 64, 3, g, r, seed, H, mode)

    def outputs(self, bwd=False):
        nan = [torch.full_like(self.q, float("nan")), torch.full(self.q.shape[:3], float("nan"), device=self.q.device)]
        return nan + [torch.full_like(self.q, float("nan")) for _ in range(3 if bwd else 0)]

    def run(self, o, stream=None, fwd=bb.bigbird_attn_fwd):
        fwd(self.q, self.k, self.v, self.layout, self.mask, o[0], o[1], self.wl.scale, stream)
        if len(o) > 2:
            bb.bigbird_attn_bwd(self.q, self.k, self.v, o[0], o[1], self.dout, self.layout, self.mask, *o[2:], self.wl.scale, stream)

    def expected(self, bwd=False):
        o = self.outputs(bwd)
        self.run(o)
        torch.cuda.synchronize()
        return o


def same(a, b):
    return all(torch.equal(x, y) for x, y in zip(a, b))


# More tiles than the GPU has tile streams, so that a call draws work from its counter.
BUSY = [dict(dtype="bf16", B=3, H=12, nb=32, seed=5), dict(dtype="bf16", B=3, H=12, nb=32, seed=6, lengths=[2048, 1999, 777])]


@pytest.mark.parametrize("kw", BUSY, ids=["full", "padded"])
def test_many_calls_queued_on_two_streams(kw):
    """More calls in flight on each of two streams than the library has counters of its own, the second stream's queued behind
    all of the first's; the same bits as one call at a time."""
    p = Problem(**kw)
    want = p.expected()
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in range(2)]
    outs = [[p.outputs() for _ in range(80)] for _ in streams]
    torch.cuda.synchronize()
    for s, os_ in zip(streams, outs):
        for o in os_:
            p.run(o, s.cuda_stream)
    torch.cuda.synchronize()
    assert bb.bigbird_last_status() == (0, 0)
    assert all(same(want, o) for os_ in outs for o in os_)


def test_training_steps_queued_on_two_streams():
    ps = [Problem(**kw) for kw in BUSY]
    want = [p.expected(bwd=True) for p in ps]
    streams = [torch.cuda.Stream() for _ in ps]
    outs = [[p.outputs(bwd=True) for _ in range(20)] for p in ps]
    torch.cuda.synchronize()
    for i in range(20):
        for p, s, os_ in zip(ps, streams, outs):
            p.run(os_[i], s.cuda_stream)
    torch.cuda.synchronize()
    assert bb.bigbird_last_status() == (0, 0)
    assert all(same(w, o) for w, os_ in zip(want, outs) for o in os_)


def test_more_streams_than_the_library_has_counters():
    p = Problem(**BUSY[0])
    want = p.expected()
    rt = torch.cuda.cudart()
    handles = []
    for _ in range(70):
        h = ctypes.c_uint64(0)
        assert int(rt.cudaStreamCreate(ctypes.addressof(h))) == 0
        handles.append(h.value)
    outs = [p.outputs() for _ in handles]
    torch.cuda.synchronize()
    for _ in range(2):
        for h, o in zip(handles, outs):
            p.run(o, h)
    torch.cuda.synchronize()
    for h in handles:
        assert int(rt.cudaStreamDestroy(h)) == 0
    assert bb.bigbird_last_status() == (0, 0)
    assert all(same(want, o) for o in outs)


# Calls with and without a mask, with and without scratch for the parts of global tiles; the gradients of each; CUDA cores.
CAPTURED = [dict(dtype="bf16", B=3, H=12, nb=32, seed=5), dict(dtype="bf16", B=2, H=2, nb=12, seed=8, lengths=[768, 197]),
            dict(dtype="bf16", B=1, H=2, nb=100, seed=9, lengths=[4000]), dict(dtype="bf16", B=1, H=4, nb=64, seed=10),
            dict(dtype="fp32", B=1, H=2, nb=10, seed=11, lengths=[600])]


@pytest.mark.parametrize("kw", CAPTURED, ids=lambda kw: f"{kw['dtype']}_{kw['B']}_{kw['H']}_{kw['nb']}")
def test_captured_forward_and_backward_replay_on_new_inputs(kw):
    """A training step in a CUDA graph, replayed on other inputs while the same layout is used outside the graph."""
    p = Problem(**kw)
    other = Problem(**dict(kw, seed=kw["seed"] + 50))
    p.expected(bwd=True)                                          # the layout goes to the device outside capture
    o = p.outputs(bwd=True)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        p.run(o)
    side = torch.cuda.Stream()
    for data in (p, other, p):
        q = [t.clone() for t in (p.q, p.k, p.v, p.dout)]
        for dst, src in zip((p.q, p.k, p.v, p.dout), (data.q, data.k, data.v, data.dout)):
            dst.copy_(src)
        want = p.expected(bwd=True)
        for t in o:
            t.fill_(float("nan"))
        torch.cuda.synchronize()
        eager = p.outputs(bwd=True)
        torch.cuda.synchronize()
        graph.replay()
        p.run(eager, side.cuda_stream)
        graph.replay()
        torch.cuda.synchronize()
        assert same(want, o) and same(want, eager)
        for dst, src in zip((p.q, p.k, p.v, p.dout), q):
            dst.copy_(src)
    assert bb.bigbird_last_status() == (0, 0)


def test_first_calls_of_layouts_on_a_side_stream():
    """The device copy of a layout is complete before any stream can reach it."""
    side = torch.cuda.Stream()
    for seed in range(30):
        p = Problem("bf16", 1, 2, 40, seed=100 + seed)
        o = p.outputs()
        torch.cuda.synchronize()
        p.run(o, side.cuda_stream)
        torch.cuda.synchronize()
        assert same(o, p.expected())
        p.layout.close()


def test_running_out_of_host_memory_is_an_error_code(tmp_path):
    """A call that cannot get the host memory for the device copy of its layout returns BIGBIRD_ENOMEM: nothing is thrown
    through the C entry point, and the next call is fine."""
    src = tmp_path / "no_memory.cpp"
    src.write_text(textwrap.dedent("""
        #include <cstdlib>
        #include <new>
        static thread_local bool armed = false;
        extern "C" void arm(int on) { armed = on != 0; }
        void* operator new(std::size_t n) {
            void* p = armed && n >= 65536 ? nullptr : std::malloc(n ? n : 1);
            if (!p) throw std::bad_alloc();
            return p;
        }
        void* operator new[](std::size_t n) { return operator new(n); }
        void* operator new(std::size_t n, const std::nothrow_t&) noexcept { return armed && n >= 65536 ? nullptr : std::malloc(n ? n : 1); }
        void* operator new[](std::size_t n, const std::nothrow_t& t) noexcept { return operator new(n, t); }
        void operator delete(void* p) noexcept { std::free(p); }
        void operator delete[](void* p) noexcept { std::free(p); }
        void operator delete(void* p, std::size_t) noexcept { std::free(p); }
        void operator delete[](void* p, std::size_t) noexcept { std::free(p); }
    """))
    so = tmp_path / "no_memory.so"
    subprocess.run(["g++", "-O1", "-shared", "-fPIC", "-o", str(so), str(src)], check=True)
    code = textwrap.dedent(f"""
        import ctypes, torch
        import paper_2007_14062_b200 as bb
        arm = ctypes.CDLL({str(so)!r}).arm
        q = torch.randn(1, 12, 4096, 64, device="cuda", dtype=torch.bfloat16)
        out = torch.empty_like(q)
        L = bb.bigbird_build_layout(4096, 64, 3, 2, 3, 0, 12)
        L2 = bb.bigbird_build_layout(4096, 64, 3, 2, 3, 0, 12)
        bb.bigbird_attn_fwd(q, q, q, L, None, out, None, 0.125)
        torch.cuda.synchronize()
        arm(1)
        try:
            bb.bigbird_attn_fwd(q, q, q, L2, None, torch.empty_like(q), None, 0.125)
            code = 0
        except bb.BigBirdError as e:
            code = e.code
        arm(0)
        assert code in (0, -5), code
        again = torch.empty_like(q)
        bb.bigbird_attn_fwd(q, q, q, L2, None, again, None, 0.125)
        assert torch.equal(out, again)
        print("fine", code)
    """)
    r = subprocess.run([sys.executable, "-c", code], cwd=ROOT, env=dict(os.environ, LD_PRELOAD=str(so)), capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "fine -5" in r.stdout, r.stdout[-2000:] + r.stderr[-2000:]
