"""Rules of the host code, compiled on their own."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2010_10272_gb300", "csrc")


def run_cpp(tmp_path, body):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text('#include <stdio.h>\n#include "hgp_rules.h"\nint main() {\n' + body + "\nreturn 0;\n}\n")
    subprocess.check_call(["g++", "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)])
    return subprocess.check_output([str(exe)], text=True).split()


def test_range_inside(tmp_path):
    """A caller's array is read where it is only if it lies in one allocation, whole."""
    cases = [(1000, 100, 1000, 100, 1), (1000, 101, 1000, 100, 0), (1050, 50, 1000, 100, 1), (1050, 51, 1000, 100, 0),
             (999, 1, 1000, 100, 0), (1100, 0, 1000, 100, 1), (1100, 4, 1000, 100, 0), (1101, 0, 1000, 100, 0),
             (2000, 4, 1000, 100, 0), (1050, 2**64 - 1, 1000, 100, 0), (2**64 - 8, 16, 2**64 - 16, 16, 0)]
    got = run_cpp(tmp_path, "".join(f'printf("%d ", hgp::range_inside({p}ull, {b}ull, {base}ull, {size}ull));'
                                    for p, b, base, size, _ in cases))
    assert [int(x) for x in got] == [c[-1] for c in cases]


def test_chunks_of_a_list_that_ends_at_the_largest_index(tmp_path):
    """The chunks of a pin array of up to 2^31 - 1 entries cover it once, the last one included."""
    chunk = 8192
    for end in (1, 8191, 8192, 8193, 2**31 - 1, 2**31 - 8192, 2**31 - 8193, 2**31 - 8191):
        first = max(0, (end - 1) // chunk - 2)
        got = run_cpp(tmp_path, "".join(f'printf("%d ", hgp::chunk_length({c * chunk}, {end}, {chunk}));'
                                        for c in range(first, (end + chunk - 1) // chunk)))
        assert [int(x) for x in got] == [min(chunk, end - c * chunk) for c in range(first, (end + chunk - 1) // chunk)]
