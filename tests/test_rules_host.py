"""The dispatch rules over sizes and times (csrc/sgtv_rules.h), compiled for the host."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1601_08201_gb300", "csrc")


def run(tmp_path, body):
    src, exe = tmp_path / "rules.cpp", tmp_path / "rules"
    src.write_text('#include <stdio.h>\n#include <vector>\n#include "sgtv_rules.h"\nusing namespace sgtv;\n'
                   "int main()\n{\n%s\n}\n" % body)
    subprocess.run(["g++", "-std=c++17", "-Wall", "-Werror", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout
    return [line.split() for line in out.splitlines()]


def test_loss_head_fills_the_chip_whatever_the_planes(tmp_path):
    sizes = [(1, 1), (1, 1024), (1, 1025), (1, 262144), (3, 5000), (2560, 4096), (7, 1 << 24), (1 << 20, 16), (5, 999)]
    body = "".join('printf("%%lld\\n", (long long)mse_pieces(%dLL, %dLL, 1216));\n' % s for s in sizes)
    for (planes, n), (pieces,) in zip(sizes, run(tmp_path, body)):
        pieces = int(pieces)
        length = -(-n // pieces)
        assert pieces >= 1 and pieces * length >= n
        # all blocks have work, or no piece is longer than one round of a block's loads
        assert planes * pieces >= 1216 or length <= 1024, (planes, n, pieces)
        # no more pieces than that takes
        assert pieces == 1 or (planes * (pieces - 1) < 1216 and length > 512), (planes, n, pieces)


AUTOTUNE = """
    // times of single launches in turn, in ms; every one after the list's end takes the last
    auto time = [](std::vector<float> t, int reps, float so_far) {
        size_t at = 0;
        auto timed = [&](int n, float *ms) {
            *ms = 0.f;
            for (int k = 0; k < n; k++, at++) *ms += t[at < t.size() ? at : t.size() - 1];
            return 0;
        };
        float ms = -1.f;
        const int e = tuned_time(timed, reps, so_far, &ms);
        printf("%d %d %.4f\\n", e, int(at), ms);
    };
"""


def test_autotuner_drops_a_form_on_two_slow_launches_only(tmp_path):
    cases = [("{3.f, 0.5f}", 10, 1.0, (11, 0.5)),    # one disturbed launch, then twice as fast as the best: kept
             ("{3.f, 0.5f}", 10, 0.2, (2, 0.5)),     # both slow, the lower counted
             ("{1.2f}", 10, 1.0, (11, 1.2)),         # not far off: timed in full
             ("{3.f}", 10, 1.0, (2, 3.0)),           # slow
             ("{3.f}", 10, 0.04, (10, 3.0)),         # against a short best: timed in full
             ("{0.01f}", 10, 3.4e38, (11, 0.01))]    # the first form
    body = AUTOTUNE + "".join("    time(%s, %d, %ef);\n" % c[:3] for c in cases)
    for c, (e, n, ms) in zip(cases, run(tmp_path, body)):
        assert int(e) == 0
        if c[0] == "{3.f, 0.5f}" and c[3][0] == 11:
            assert int(n) == 12 and float(ms) == pytest.approx(0.5), c  # two single launches, then ten
        else:
            assert int(n) == c[3][0] and float(ms) == pytest.approx(c[3][1], rel=1e-4), c


def test_autotuner_passes_errors_on(tmp_path):
    body = """
    for (int bad = 0; bad < 3; bad++) {
        int call = 0;
        float ms = 0.f;
        const int e = tuned_time([&](int, float *t) { *t = 9.f; return call++ == bad ? 7 : 0; }, 10, bad == 2 ? 8.f : 1.f, &ms);
        printf("%d\\n", e);
    }
"""
    # in the first single launch, in the second, and (a form not dropped) not at all in a third that does not happen
    assert [r[0] for r in run(tmp_path, body)] == ["7", "7", "0"]


def test_deviance_form(tmp_path):
    sms, rows = 152, (1, 64, 1216, 1217, 2432, 2433, 20000, 1 << 20)
    cases = [(r, mean, tiled) for r in rows for mean in (0, 64, 256, 257, 512, 513, 5000) for tiled in (0, 1)]
    body = "".join('printf("%%d\\n", dev_rows_per_warp(%d, %d, %d, %d));\n' % (r, m, sms, t) for r, m, t in cases)
    for (r, mean, tiled), (form,) in zip(cases, run(tmp_path, body)):
        form = int(form)
        assert form in (0, 1, 8) and (form != 0 or tiled)
        if r <= 16 * sms:  # a warp for each row: none has two
            assert form == 1, (r, mean, tiled)
        if r > 16 * sms and tiled:
            assert form == 0, (r, mean)


def test_shrink_is_spread_beside_kernels_without_staging_only(tmp_path):
    cases = [(e, st, s) for e in (4, 8) for st in (0, 1) for s in (1, 369, 1215, 1216, 1 << 20)]
    body = "".join('printf("%%d\\n", int(shrink_spread(%d, %d, %d, 152)));\n' % c for c in cases)
    for (elem, staged, sites), (spread,) in zip(cases, run(tmp_path, body)):
        assert int(spread) == (elem == 8 and not staged and sites < 1216)
