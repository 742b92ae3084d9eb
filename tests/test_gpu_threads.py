"""Two host threads call the same form at once, each on a stream of its own,
with batches or trees whose launches take different amounts of shared memory:
every call is accepted and gives, bit for bit, what it gives alone. The threads
are C++ threads (Python's would take turns at the interpreter's lock and seldom
meet inside the library).
"""
import ctypes as C
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")
wt = pytest.importorskip("paper_1909_03956_gb300")

pytestmark = pytest.mark.gpu

CALLER = r"""
#include <atomic>
#include <cstdint>
#include <thread>
using Tree = int (*)(void*, void*, int64_t, void*, int, int, int, void*);
using Direct = int (*)(void*, void*, void*, int64_t, void*, int64_t, void*, int, int, void*);
static void* p(int64_t x) { return reinterpret_cast<void*>(x); }
static int call(int direct, void* fn, const int64_t* a)
{
    if (direct)
        return reinterpret_cast<Direct>(fn)(p(a[0]), p(a[1]), p(a[2]), a[3], p(a[4]), a[5], p(a[6]), (int)a[7],
                                            (int)a[8], p(a[9]));
    return reinterpret_cast<Tree>(fn)(p(a[0]), p(a[1]), a[2], p(a[3]), (int)a[4], (int)a[5], (int)a[6], p(a[7]));
}
// Each argument list `repeats` times in a thread of its own; calls that failed.
extern "C" int together(int direct, void* fn, const int64_t* a, const int64_t* b, int repeats)
{
    std::atomic<int> ready{0}, failed{0};
    auto work = [&](const int64_t* x) {
        ++ready;
        while (ready.load() < 2) std::this_thread::yield();
        for (int i = 0; i < repeats; ++i)
            if (call(direct, fn, x) != 0) ++failed;
    };
    std::thread t(work, a), u(work, b);
    t.join();
    u.join();
    return failed.load();
}
"""

dev = lambda a: torch.as_tensor(np.ascontiguousarray(a), device="cuda")


@pytest.fixture(scope="module")
def together(tmp_path_factory):
    d = tmp_path_factory.mktemp("caller")
    (d / "caller.cpp").write_text(CALLER)
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-pthread", str(d / "caller.cpp"), "-o",
                    str(d / "caller.so")], check=True)
    f = C.CDLL(str(d / "caller.so")).together
    f.argtypes = [C.c_int, C.c_void_p, C.c_void_p, C.c_void_p, C.c_int]
    return f


def _tree_calls(trees, uvw, mode, which, streams):
    dt = torch.complex128 if mode == wt.WT_FP64 else torch.complex64
    out = [torch.empty(u.shape[0], dtype=dt, device="cuda") for u in uvw]
    args = [[t.h.value, u.data_ptr(), u.shape[0], o.data_ptr(), mode, 1, which, s.cuda_stream]
            for t, u, o, s in zip(trees, uvw, out, streams)]
    return args, out


def _batches(g, streams):
    # float64 tiles of 64: 100 of them take an SM's shared memory each, 600 a quarter of it
    l, m = g.uniform(-0.02, 0.02, (2, 50))
    t = wt.wt_build_tree(dev(l), dev(m), dev(np.ones(50)), np.pi, np.pi / 4, 12)
    uvw = [dev(g.uniform(-2e4, 2e4, (64 * n, 3))) for n in (100, 600)]
    return (0, *_tree_calls([t, t], uvw, wt.WT_FP64, wt.WT_SUM_EQ17, streams), (t, uvw))


def _depths(g, streams):
    l, m = g.uniform(-0.02, 0.02, (2, 50))
    trees = [wt.wt_build_tree(dev(l), dev(m), dev(np.ones(50)), np.pi, np.pi / 4, J) for J in (6, 13)]
    uvw = [dev(g.uniform(-2e4, 2e4, (2000, 3)))] * 2
    return (0, *_tree_calls(trees, uvw, wt.WT_MIXED, wt.WT_SUM_EQ17, streams), (trees, uvw))


def _tensor_cores(g, streams):
    l, m = g.uniform(-0.02, 0.02, (2, 60))
    c = dev(l), dev(m), dev(np.ones(60))
    uvw = [dev(g.uniform(-2e4, 2e4, (n, 3))) for n in (100000, 100300)]   # many enough not to be cut
    out = [torch.empty(u.shape[0], dtype=torch.complex64, device="cuda") for u in uvw]
    args = [[c[0].data_ptr(), c[1].data_ptr(), c[2].data_ptr(), 60, u.data_ptr(), u.shape[0], o.data_ptr(),
             wt.WT_MIXED_TC, 1, s.cuda_stream] for u, o, s in zip(uvw, out, streams)]
    return 1, args, out, (c, uvw)


@pytest.mark.parametrize("make", [_batches, _depths, _tensor_cores])
def test_two_threads(make, together):
    streams = [torch.cuda.Stream() for _ in range(2)]
    direct, args, out, keep = make(np.random.default_rng(5), streams)
    torch.cuda.synchronize()
    fn = wt.load().dft_predict_vis if direct else wt.load().wt_predict_vis
    alone = []
    for a, o in zip(args, out):
        assert fn(*a) == 0               # launch shapes are chosen here
        torch.cuda.synchronize()
        alone.append(o.clone())
        o.zero_()
    torch.cuda.synchronize()
    a, b = (np.array(x, dtype=np.int64) for x in args)
    failed = together(direct, C.cast(fn, C.c_void_p), a.ctypes.data, b.ctypes.data, 2000)
    assert failed == 0
    torch.cuda.synchronize()
    assert all(torch.equal(x, y) for x, y in zip(alone, out))
    wt.wt_device_status()
    del keep
