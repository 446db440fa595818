"""Capacity answers kept for a problem (csrc/at_fit.h): known ones are not asked
again, failed ones are."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2204_01133_gb300", "csrc")
MAIN = """
#include "at_fit.h"
#include <cassert>
int main()
{
    atk::FitCache c;
    const int64_t zero[8] = {0}, a[8] = {1, 2, 3, 4, 5, 6, 7, 8}, b[8] = {1, 2, 3, 4, 5, 6, 7, 9};
    assert(!c.knows(zero) && !c.knows(a));
    c.ask(a);
    assert(c.take(456) == 456 && c.take(0) == 0);
    assert(c.knows(a) && !c.knows(b));
    c.ask(b);
    assert(c.take(16) == 16 && c.take(-1) == 0 && c.take(3) == 3);
    assert(!c.knows(b) && !c.knows(a));  // one query failed: all are asked again
    c.ask(b);
    assert(c.take(16) == 16 && c.take(304) == 304);
    assert(c.knows(b));
    return 0;
}
"""


def test_failed_queries_are_asked_again(tmp_path):
    src, exe = tmp_path / "m.cpp", tmp_path / "m"
    src.write_text(MAIN)
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    subprocess.run([str(exe)], check=True)
