"""The queue that sends the passes of a step together (csrc/pass_queue.hpp): every pass goes out
once and in order, together or one by one, whichever launch of a step is the first that cannot be
made -- also the launch of a full queue, with the pass that found it full still to come."""
import os
import shutil
import subprocess

import pytest

SOURCE = r"""
#include <cstdio>
#include <vector>
#include "pass_queue.hpp"
struct Chain {
    static constexpr int capacity = 4;
    int n, pass[capacity];
};
int main() {
    int bad = 0;
    for (int npass = 0; npass <= 13; ++npass)
        for (int fail_at = -1; fail_at <= 3; ++fail_at)
            for (int together = 0; together < 2; ++together) {
                ewv::PassQueue<Chain> q;
                int launches = 0;
                for (int step = 0; step < 2; ++step) {
                    std::vector<int> sent;
                    int singles = 0;
                    auto all = [&](const Chain& c) {
                        if (launches++ == fail_at) return false;
                        for (int k = 0; k < c.n; ++k) sent.push_back(c.pass[k]);
                        return true;
                    };
                    auto one = [&](int p) {
                        sent.push_back(p);
                        ++singles;
                    };
                    q.begin(together != 0);
                    for (int p = 0; p < npass; ++p) q.add(p, all, one);
                    q.end(all, one);
                    bool ok = (int)sent.size() == npass;
                    for (int p = 0; ok && p < npass; ++p) ok = sent[p] == p;
                    const int want = (npass + Chain::capacity - 1) / Chain::capacity;    // launches of a whole step
                    if (!together) ok = ok && launches == 0 && singles == npass;
                    else if (fail_at < 0 || fail_at >= want * (step + 1))
                        ok = ok && launches == want * (step + 1) && singles == 0 && !q.broken();
                    else
                        ok = ok && launches == fail_at + 1 && q.broken() && (step == 0 || fail_at >= want || singles == npass);
                    if (!ok) {
                        std::printf("npass %d fail_at %d together %d step %d: %zu sent, %d singly, %d launches\n", npass,
                                    fail_at, together, step, sent.size(), singles, launches);
                        ++bad;
                    }
                }
            }
    return bad != 0;
}
"""


def test_every_pass_is_sent_once_and_in_order(repo_root, tmp_path):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no host compiler")
    src, exe = tmp_path / "q.cpp", tmp_path / "q"
    src.write_text(SOURCE)
    include = os.path.join(repo_root, "paper_2401_16322_gb300", "csrc")
    subprocess.run([cxx, "-std=c++17", "-O1", "-Wall", "-Werror", "-I", include, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
