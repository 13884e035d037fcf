"""The end of the copy rings of the prefill attention and of the CTA-pair GEMMs
(csrc/copy_ring.cuh, the code the kernels run), compiled for the host with
waits that give up at every point: no copy may be in flight when the filling
thread is done."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SRC = r"""
#include "copy_ring.cuh"
#include <cstdio>
#include <vector>
constexpr int ST = 2;
// copies of a run whose `fail`-th wait for a free stage gives up (fail < 0: none), and whose drain waits
// give up too when `lost`
static int run(int nt, int fail, bool lost) {
    std::vector<int> state[2];  // per copy: 1 in flight, 2 arrived (its stage's next user waited, or the drain)
    int calls = 0, bad = 0;
    pipo::ring_fill_pair<ST>(
        nt,
        [&](int v, int st, uint32_t ph, int t) {
            if (calls++ == fail) return false;
            const int prev = t - ST;  // the tile that leaves the stage had arrived
            if (prev < 0 || prev % ST != st || ph != (uint32_t)((prev / ST) & 1)) ++bad;
            else state[v][prev] = 2;
            return true;
        },
        [&](int v, int st, int t) {
            if (t != (int)state[v].size() || st != t % ST) ++bad;
            state[v].push_back(1);
        },
        [&](int v, int st, uint32_t ph, int t) {
            if (t < 0 || t >= (int)state[v].size() || st != t % ST || ph != (uint32_t)((t / ST) & 1)) ++bad;
            else state[v][t] = 2;
            return !lost;
        });
    if (fail < 0 && ((int)state[0].size() != nt || (int)state[1].size() != nt)) ++bad;
    for (auto& c : state)
        for (int x : c) bad += x != 2;
    return bad;
}
// a pair's leader after n stages, the commits from stage `gone` on never made: copies not waited for,
// waits for commits after one that gave up
template <int S>
static int pair(int n, int gone, bool leader) {
    std::vector<int> state(n, 1);
    int bad = 0, last = -1;
    bool over = false;
    pipo::pair_drain<S>(
        n, leader,
        [&](int st, uint32_t ph, int i) {
            if (i < 0 || i >= n || st != i % S || ph != (uint32_t)((i / S) & 1)) ++bad;
            else state[i] = 2;
            return false;  // a full barrier that gives up does not end the waiting
        },
        [&](int st, uint32_t ph, int i) {
            if (over || i < n - S || i <= last || st != i % S || ph != (uint32_t)((i / S) & 1)) ++bad;
            last = i;
            over = i >= gone;
            return !over;
        });
    for (int i = n > S ? n - S : 0; i < n; ++i) bad += leader && state[i] != 2;
    if (n > 0 && gone >= n) bad += last != n - 1;
    return bad;
}
int main() {
    int bad = 0, runs = 0;
    for (int n = 0; n <= 20; ++n)
        for (int gone = 0; gone <= n; ++gone)
            for (int leader = 0; leader < 2; ++leader) {
                const int b = pair<4>(n, gone, leader) + pair<6>(n, gone, leader) + pair<8>(n, gone, leader);
                if (b) std::printf("pair n=%d gone=%d leader=%d: %d\n", n, gone, leader, b);
                bad += b;
            }
    for (int nt = 0; nt <= 9; ++nt)
        for (int fail = -1; fail < 2 * nt; ++fail)
            for (int lost = 0; lost < 2; ++lost) {
                const int b = run(nt, fail, lost);
                if (b) std::printf("nt=%d fail=%d lost=%d: %d\n", nt, fail, lost, b);
                bad += b;
                ++runs;
            }
    std::printf("%d runs\n", runs);
    return bad != 0;
}
"""


def test_no_copy_in_flight_whatever_wait_gives_up(tmp_path):
    src, exe = tmp_path / "ring.cpp", tmp_path / "ring"
    src.write_text(SRC)
    subprocess.check_call(["g++", "-std=c++17", "-Wall", "-Werror", "-I",
                           os.path.join(ROOT, "paper_2605_27255_gb300", "csrc"), str(src), "-o", str(exe)])
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
    assert r.stdout.strip() == "200 runs", r.stdout
