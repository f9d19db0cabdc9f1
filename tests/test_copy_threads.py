"""How many host threads copy a call's results out (host only): none besides the
caller's where starting them costs more than they save, few for results of some MB,
never more than the machine has cores.  The rule is compiled from its header."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = r'''
#include "sbg_host.h"
#include <cstdio>
#include <cstdlib>
int main(int argc, char** argv) {
  for (int i = 1; i + 1 < argc; i += 2)
    printf("%d ", sbg::copy_threads((size_t)strtoull(argv[i], nullptr, 10), (unsigned)atoi(argv[i + 1])));
  printf("%d\n", sbg::copy_threads(1000));
}
'''
KB, MB = 1 << 10, 1 << 20


@pytest.mark.parametrize("size,cores,threads", [
    (0, 16, 1), (256 * KB, 16, 1), (1152 * KB, 16, 1), (1638 * KB, 16, 1),  # a second thread loses 10 to 30 us
    (1850 * KB, 16, 3), (2 * MB, 16, 4), (4352 * KB, 16, 4), (15 * MB, 16, 4),  # eight lose 140 to 320 us against four
    (54 * MB, 16, 8), (512 * MB, 64, 8), (54 * MB, 1, 1), (54 * MB, 0, 1), (54 * MB, 6, 6), (4 * MB, 2, 2)])
def test_threads_by_size(tmp_path, size, cores, threads):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(SRC)
    subprocess.run(["g++", "-std=c++17", "-I", os.path.join(ROOT, "paper_2210_10206_gb300", "csrc"), str(src), "-o", str(exe),
                    "-lpthread"], check=True)
    out = subprocess.run([str(exe), str(size), str(cores)], check=True, capture_output=True, text=True).stdout.split()
    assert [int(x) for x in out] == [threads, 1]
