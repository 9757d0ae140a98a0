"""The dispatch rules over sizes and times (csrc/sgtv_rules.h), compiled for the host."""
import os
import subprocess

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
