"""The host memory of the serving scheduler (csrc/ept_host.h), compiled alone: which memory a request gets,
how much is kept, when it is given back, and which copies take the worker threads."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _run(d, body):
    src = d / "host.cpp"
    src.write_text("#include <cstdio>\n#include <cstdlib>\n"
                   '#include "ept_host.h"\nusing namespace ept;\n'
                   '#define CHECK(x) do { if (!(x)) { printf("%d: %s\\n", __LINE__, #x); return 1; } } while (0)\n' + body)
    exe = d / "host"
    inc = os.path.join(ROOT, "paper_2406_06488_gb300", "csrc")
    try:
        subprocess.run([os.environ.get("CXX", "g++"), "-O1", "-std=c++17", "-pthread", "-I" + inc, "-o", str(exe),
                        str(src)], check=True, capture_output=True)
    except OSError as e:
        pytest.skip("no C++ compiler here: %s" % e)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout


def test_kept_memory_follows_the_request_sizes(tmp_path):
    _run(tmp_path, r"""
int main() {
    constexpr size_t MB = (1 << 20) / sizeof(float);
    HostPool pool;
    for (int k = 0; k < 2; ++k) {          // a burst of 40 MB requests, then it is what a second one gets
        HostBuffer b[8];
        for (HostBuffer &x : b) { x = pool.take(40 * MB); CHECK(x.data); }
        CHECK(pool.bytes() == 0);
        for (HostBuffer &x : b) pool.give(std::move(x));
        CHECK(pool.bytes() == 6 * (size_t)40 << 20);   // as many as the limit holds
    }
    // sizes change: the new size is kept too, in the place of the oldest of the other
    for (int k = 0; k < 3; ++k) {
        HostBuffer x = pool.take(90 * MB);
        CHECK(x.cap == 90 * MB);
        const float *p = x.data.get();
        pool.give(std::move(x));
        CHECK(pool.bytes() <= HostPool::LIMIT);
        HostBuffer y = pool.take(90 * MB);
        CHECK(y.data.get() == p);
        pool.give(std::move(y));
    }
    // half to all of a buffer, the smallest that will do; small and huge ones are not kept
    HostBuffer z = pool.take(21 * MB);
    CHECK(z.cap == 40 * MB);
    const size_t held = pool.bytes();
    pool.give(pool.take(100));
    pool.give(pool.take(300 * MB));
    CHECK(pool.bytes() == held);
    return 0;
}
""")


def test_kept_memory_is_given_back(tmp_path):
    _run(tmp_path, r"""
int main() {
    HostPool pool;
    CHECK(!pool.idle(HostPool::Clock::now() + HostPool::IDLE));   // nothing to give back
    pool.give(pool.take(1 << 20));
    CHECK(pool.bytes() == 4 << 20);
    CHECK(!pool.idle(HostPool::Clock::now()));
    CHECK(pool.idle(HostPool::Clock::now() + HostPool::IDLE));
    pool.release();
    CHECK(pool.bytes() == 0 && !pool.idle(HostPool::Clock::now() + HostPool::IDLE));
    HostBuffer b = pool.take(1 << 20);
    CHECK(b.data && b.cap == 1 << 20);
    return 0;
}
""")


def test_small_copies_leave_the_workers_alone(tmp_path):
    _run(tmp_path, r"""
struct CountedMutex {   // how often it is asked for; refused while `taken`
    static int asked;
    static bool taken;
    void lock() {}
    void unlock() {}
    bool try_lock() { ++asked; return !taken; }
};
int CountedMutex::asked = 0;
bool CountedMutex::taken = false;
int main() {
    using Copier = SharedCopier<CountedMutex>;
    Copier copier;
    for (size_t bytes : {(size_t)0, (size_t)1, (size_t)4097, Copier::PARALLEL - 2, Copier::PARALLEL, (size_t)50000001})
        for (bool taken : {false, true}) {
            std::vector<uint8_t> x(bytes), y(bytes + 1);
            for (size_t k = 0; k < bytes; ++k) x[k] = (uint8_t)(k * 131 + (k >> 9) + 1);
            const size_t h = bytes / 3;   // two jobs
            const HostCopier::Job jobs[2] = {{y.data(), x.data(), h}, {y.data() + h, x.data() + h, bytes - h}};
            CountedMutex::taken = taken;
            CountedMutex::asked = 0;
            copier.copy(jobs, 2);
            CHECK(CountedMutex::asked == (bytes >= Copier::PARALLEL ? 1 : 0));
            CHECK(std::equal(x.begin(), x.end(), y.begin()) && y[bytes] == 0);
        }
    return 0;
}
""")
