"""Kernel attributes are kept per CUDA context (csrc/tv_once.h): set in every context that a call
meets, again after a failure or where the context cannot be told, and by threads at once. The
contexts are numbers here; the network's launchers set shared-memory limits no other way."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1502_07770_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <thread>
#include <vector>
#include "tv_once.h"
enum Status { OK = 0, FAILED = 2 };
static thread_local long long current = 0;
static bool id(unsigned long long *out) { *out = (unsigned long long)current; return current >= 0; }
int main()
{
    tvh::OncePerContext once;
    int sets = 0;
    auto call = [&](long long ctx, Status result) {
        current = ctx;
        const int before = sets;
        const Status st = once.run(id, [&] { ++sets; return result; });
        std::printf("%d%d ", sets - before, (int)st);
    };
    call(0, OK), call(0, OK);            // the first context, whose id may be 0
    call(9, OK), call(9, OK);            // a second device
    call(0, OK), call(9, OK);            // back and forth
    call(-1, OK), call(-1, OK);          // no id
    call(11, FAILED), call(11, OK), call(11, OK);
    // threads, each on its own context: whoever launches has set its own
    std::atomic<int> bad{0};
    std::atomic<int> limit[4] = {};
    std::vector<std::thread> ts;
    tvh::OncePerContext shared;
    for (int t = 0; t < 4; ++t)
        ts.emplace_back([&, t] {
            current = t;
            for (int k = 0; k < 20000; ++k) {
                shared.run(id, [&] { limit[t] = 1; return OK; });
                if (!limit[t]) ++bad;
            }
        });
    for (auto &t : ts) t.join();
    std::printf("%d\n", bad.load());
}
"""


def test_contexts_failures_and_threads(tmp_path):
    src, exe = tmp_path / "once.cpp", str(tmp_path / "once")
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-pthread", "-I", CSRC, str(src), "-o", exe], check=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True, timeout=60).stdout.split()
    assert out == ["10", "00", "10", "00", "10", "10", "10", "10", "12", "10", "00", "0"]


def test_the_networks_launchers_use_it():
    text = open(os.path.join(CSRC, "tv_net.cu")).read()
    helper = text[text.index("tv_status smem_opt_in("):]
    helper = helper[:helper.index("\n}\n")]
    assert text.count("cudaFuncSetAttribute(") == helper.count("cudaFuncSetAttribute(") == 2
    assert text.count("smem_opt_in(") == 1 + 5
