"""How a kernel reports to the host (csrc/report.cuh), on the CPU: its blocks one after the other in every order."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SOURCE = r"""
#include <algorithm>
#include <cstdio>
#include <cstring>
#include <numeric>
#include <vector>

#define __device__
#define __forceinline__ inline
#define CKV_REPORT_ON_HOST
struct Dim { unsigned x, y; };
static Dim blockIdx, threadIdx;
static bool __syncthreads_or(bool b) { return b; }
static void __threadfence() {}
static int told, left_behind;  // reports to the host, and those at which the counter was not zero by additions alone

namespace ckv { struct Report; unsigned count_block(unsigned*, unsigned); void tell_host(const Report&, bool); }
#include "report.cuh"

static unsigned last;  // what the last addition left
static bool news;
unsigned ckv::count_block(unsigned* count, unsigned add)
{
    const unsigned before = *count;
    last = *count = before + add;
    return before;
}
void ckv::tell_host(const Report& r, bool bad)
{
    ++told;
    news = bad;
    if (*r.count != 0 || (!bad && last != 0)) ++left_behind;
}

// the blocks of a grid of `rows` rows in the given order; those with a bit in `bad` have bad news
static bool launch(unsigned* count, int* words, const std::vector<int>& order, int rows, unsigned bad)
{
    const unsigned n = (unsigned)order.size();
    told = left_behind = 0;
    last = 0;
    for (unsigned i = 0; i < n; ++i) {
        if (told) return false;  // not before the last block
        blockIdx = Dim{(unsigned)order[i] / rows, (unsigned)order[i] % rows};
        ckv::report_done(ckv::Report{words, words + 1, count}, bad >> order[i] & 1, n);
    }
    return told == 1 && left_behind == 0 && news == (bad != 0) && *count == 0;
}

int main()
{
    alignas(8) int words[2] = {};
    unsigned count = 0;  // one for all launches
    for (int n = 1; n <= 6; ++n)
        for (int rows = 1; rows <= 2; ++rows) {
            if (n % rows) continue;
            std::vector<int> order(n);
            std::iota(order.begin(), order.end(), 0);
            do
                for (unsigned bad = 0; bad < 1u << n; ++bad)
                    if (!launch(&count, words, order, rows, bad)) return std::printf("n %d rows %d bad %x\n", n, rows, bad), 1;
            while (std::next_permutation(order.begin(), order.end()));
        }
    // as many blocks as may take part, block (0, 0) first or last, none or all of them with bad news
    for (int n : {65534, 65535})
        for (int first = 0; first < 2; ++first)
            for (int all = 0; all < 2; ++all) {
                told = left_behind = 0;
                for (int i = 0; i < n; ++i) {
                    if (told) return std::printf("early\n"), 1;
                    blockIdx = Dim{(unsigned)(first ? i : n - 1 - i), 0};
                    ckv::report_done(ckv::Report{words, words + 1, &count}, all, n);
                }
                if (told != 1 || left_behind || news != all || count) return std::printf("n %d\n", n), 1;
            }
    // other threads than the first say nothing; without a word `done` only bad news are told, by the thread that has them
    threadIdx.x = 1;
    told = 0;
    ckv::report_done(ckv::Report{words, words + 1, &count}, true, 2);
    if (told || count) return std::printf("thread 1\n"), 1;
    ckv::report_done(ckv::Report{words}, false, 2);
    if (words[0]) return std::printf("no news\n"), 1;
    ckv::report_done(ckv::Report{words}, true, 2);
    if (words[0] != 1 || words[1]) return std::printf("bad news\n"), 1;
    return 0;
}
"""


def test_a_report_in_every_order_of_its_blocks(tmp_path):
    """The host hears once, from the last block, in one word with the outcome; the last addition itself leaves the counter at zero
    (nothing is left to be written behind the report), whichever blocks have bad news."""
    src, exe = tmp_path / "report.cpp", tmp_path / "report"
    src.write_text(SOURCE)
    subprocess.run(["g++", "-O1", "-std=c++17", "-Wall", "-I", os.path.join(ROOT, "paper_2601_19178_b200", "csrc"), str(src), "-o", str(exe)],
                   check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
