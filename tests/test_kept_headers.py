"""The pool of pinned headers (csrc/kept.h), on the CPU: what is taken was kept
by the same context, every block is either handed out again or left to its owner
to free, whichever devices the work moves between, and threads may share it.
"""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include "kept.h"
#include <atomic>
#include <cstdio>
#include <set>
#include <thread>
using wt::Kept;
#define CHECK(x) if (!(x)) { std::printf("line %d: %s\n", __LINE__, #x); return 1; }
static char mem[1 << 16];
int main()
{
    static Kept k;
    // two devices, both alive: none of either's blocks is lost, 32 each are kept
    std::set<void*> kept;
    int refused = 0;
    for (int i = 0; i < 100; ++i) {
        const int dev = i & 1;
        if (k.keep(dev, 11 + dev, mem + i)) kept.insert(mem + i);
        else ++refused;
    }
    CHECK(kept.size() == 64 && refused == 36);
    for (int r = 0; r < 3; ++r)
        for (int dev = 0; dev < 2; ++dev)
            for (int i = 0; i < 32; ++i) {
                void* p = k.take(dev, 11 + dev);
                CHECK(p && kept.count(p) && ((static_cast<char*>(p) - mem) & 1) == dev);
                CHECK(k.keep(dev, 11 + dev, p));
            }
    // another context on a device: the old one's blocks are not handed out
    CHECK(k.take(0, 20) == nullptr);
    CHECK(k.keep(0, 20, mem + 200));
    CHECK(k.take(0, 20) == mem + 200 && k.take(0, 20) == nullptr && k.take(0, 11) == nullptr);
    CHECK(k.take(1, 12) != nullptr);
    // no context, no such device
    CHECK(!k.keep(0, 0, mem) && !k.keep(-1, 5, mem) && !k.keep(64, 5, mem));
    CHECK(k.take(-1, 5) == nullptr && k.take(64, 5) == nullptr && k.take(3, 5) == nullptr);
    // threads: a block is never handed out twice
    static Kept t;
    static std::atomic<int> owner[1 << 16];
    std::atomic<bool> twice{false};
    auto work = [&](int me) {
        for (int i = 0; i < 20000; ++i) {
            char* p = static_cast<char*>(t.take(0, 1));
            if (!p) p = mem + 20000 * me + i;                   // a new block
            if (owner[p - mem].exchange(me) != 0) twice = true;
            owner[p - mem] = 0;
            t.keep(0, 1, p);
        }
    };
    std::thread a(work, 1), b(work, 2);
    a.join();
    b.join();
    CHECK(!twice);
    std::puts("ok");
    return 0;
}
"""


def test_pool(tmp_path):
    (tmp_path / "pool.cpp").write_text(PROGRAM)
    exe = tmp_path / "pool"
    subprocess.run(["g++", "-O1", "-std=c++17", "-pthread", "-I",
                    os.path.join(ROOT, "paper_1909_03956_gb300", "csrc"), str(tmp_path / "pool.cpp"), "-o", str(exe)],
                   check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout
