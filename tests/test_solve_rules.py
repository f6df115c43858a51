"""The host's rules of the solve path (csrc/solve_rules.h, compiled here with the host's compiler).

What the host makes of a whole-solve launch's report, for a wait that runs out at any barrier of
any block: the model follows the kernel's protocol (a block that gave up arrives at no later barrier,
block 0 writes a column's status before the column's last barrier and leaves behind it if it gave
up, and whoever gives up sets the barrier's status word)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

MODEL = r"""
#include <cstdio>
#include "solve_rules.h"
using namespace asss;

constexpr int BLOCKS = 4, COLS = 3, BARS = 5;   // barriers of a column; the last one closes it

// one launch in which block q gives up at barrier `at` (counted over the launch; -1: none), though all
// arrive there (it was late): what it leaves in r
static void launch(ClReport& r, unsigned phase0, int q, int at) {
    bool dead[BLOCKS] = {}, left[BLOCKS] = {};
    for (int c = 0; c < COLS; ++c)
        for (int b = 0; b < BARS; ++b) {
            const int bar = c * BARS + b;
            if (b == BARS - 1 && !left[0]) {   // block 0 reports the column
                ClStat s = {};
                s.status = dead[0] ? ASSS_ERR_TIMEOUT : ASSS_OK;
                s.phase = phase0 + bar + 1;
                r.st[c] = s;
            }
            bool all = true;
            for (int t = 0; t < BLOCKS; ++t) all = all && !dead[t] && !left[t];
            for (int t = 0; t < BLOCKS; ++t)
                if (!left[t] && !dead[t] && (!all || (bar == at && t == q))) {
                    dead[t] = true;
                    r.wait = ASSS_ERR_TIMEOUT;
                }
            if (b == BARS - 1)
                for (int t = 0; t < BLOCKS; ++t) left[t] = left[t] || dead[t];
        }
}

int main() {
    ClReport r;
    int bad = 0;
    unsigned phase = 0;
    cl_expect(r, COLS);
    launch(r, 40, 0, -1);
    if (cl_outcome(r, COLS, &phase) != ASSS_OK || phase != 40 + COLS * BARS) bad += 1;
    for (int q = 0; q < BLOCKS; ++q)
        for (int at = 0; at < COLS * BARS; ++at) {
            cl_expect(r, COLS);
            launch(r, 100, 0, -1);   // an earlier call's results stay in the report
            cl_outcome(r, COLS, &phase);
            cl_expect(r, COLS);
            launch(r, phase, q, at);
            if (cl_outcome(r, COLS, &phase) != ASSS_ERR_TIMEOUT || phase != 0) {
                std::printf("block %d barrier %d\n", q, at);
                bad += 1;
            }
        }
    // nothing was reported at all; other ends of a column are not this rule's; a column without a report
    cl_expect(r, COLS);
    if (cl_outcome(r, COLS, &phase) != ASSS_ERR_TIMEOUT || phase != 0) bad += 1;
    cl_expect(r, 1);
    r.st[0].status = ASSS_ERR_STAGNATION;
    if (cl_outcome(r, 1, &phase) != ASSS_OK) bad += 1;
    cl_expect(r, COLS);
    r.st[0].status = r.st[2].status = ASSS_OK;
    if (cl_outcome(r, COLS, &phase) != ASSS_ERR_TIMEOUT) bad += 1;
    return bad != 0;
}
"""


STREAM = r"""
#include "solve_rules.h"
using namespace asss;

int main() {
    int bad = 0;
    for (int tb = 4; tb <= 8; tb += 4) {
        const int most = 192000 / tb;
        bad += !stream_fits(1000, 64000, tb) + stream_fits(1000, 63999, tb);
        bad += !stream_fits(most, 64LL * most, tb) + stream_fits(most + 1, 64LL * (most + 1), tb);
        // padded by up to 3 entries a row the offsets stay below 2^31; SELL takes what may not
        const long long full = (1LL << 31) - 1024 - 3LL * most;
        if ((long long)most * (most - 1) >= full) bad += !stream_fits(most, full - 1, tb) + stream_fits(most, full, tb);
    }
    return bad;
}
"""


WAVES = r"""
#include "solve_rules.h"
using namespace asss;

int main() {
    int bad = 0;
    // the benchmark's 100^3 is in grid scope at every width, the largest systems go launch by launch
    bad += !grid_scope_pays(1000000, 0) + !grid_scope_pays(2500000, 4) + grid_scope_pays(2500001, 32) +
           grid_scope_pays(1600001, 0);
    for (int side = 1; side <= 20; ++side)
        for (int nrhs = 1; nrhs <= 70; ++nrhs) {
            int rounds = 0;
            for (int left = nrhs; left > 0; left -= CL_CHUNK)   // a launch each
                for (int c = left < CL_CHUNK ? left : CL_CHUNK; c > 0; c -= side) ++rounds;
            bad += cl_waves(nrhs, side) != rounds;
        }
    return bad != 0;
}
"""


def _run(tmp_path, source):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no host C++ compiler")
    src, exe = tmp_path / "model.cpp", tmp_path / "model"
    src.write_text(source)
    inc = [f"-I{os.path.join(ROOT, 'include')}", f"-I{os.path.join(ROOT, 'paper_2009_06954_gb300', 'csrc')}"]
    subprocess.run([cxx, "-std=c++17", "-O1", "-Wall", "-Werror", *inc, str(src), "-o", str(exe)], check=True)
    p = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert p.returncode == 0, p.stdout


def test_a_wait_that_runs_out_is_never_a_success(tmp_path):
    _run(tmp_path, MODEL)


def test_row_stream_leaves_to_sell_what_its_offsets_cannot_hold(tmp_path):
    _run(tmp_path, STREAM)


def test_waves_are_counted_by_launch_and_scopes_by_rows(tmp_path):
    _run(tmp_path, WAVES)
