"""The host rules of csrc/hp_host.h, compiled with the system compiler (no GPU)."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2605_20497_gb300", "csrc")


def run(tmp_path, body):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text('#include <cstdio>\n#include "hp_host.h"\n' + body)
    subprocess.run(["g++", "-std=c++17", "-O1", "-Wall", "-Werror", "-pthread", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    return subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split()


# a batch of few instances, of few workers, or at its end leaves the side streams to its instances
def test_batch_streams(tmp_path):
    cases = [(1, 24), (4, 24), (16, 1), (16, 5), (64, 3), (8, 24), (16, 24), (16, 8), (64, 64)]
    out = run(tmp_path, "int main() { long c[][2] = {" + ",".join("{%d,%d}" % c for c in cases) + "};\n"
              'for (auto &x : c) std::printf("%d ", (int)hp::batch_one_stream(hp::batch_in_flight(x[0], x[1]))); }\n')
    assert out == [str(int(min(c) >= 6)) for c in cases]
    assert out == ["0"] * 5 + ["1"] * 4


# the table of occupancies stays small however many sizes a process asks for
def test_occupancy_table_is_bounded(tmp_path):
    out = run(tmp_path, """
int main() {
    hp::OccTable t;
    const char k[3] = {};
    for (size_t bytes = 0; bytes <= 227 * 1024; bytes++)
        for (int x = 0; x < 3; x++) {
            const hp::OccTable::Key key{&k[x], 0, 256, hp::smem_steps(bytes)};
            if (!t.find(key)) t.put(key, 1 + (int)(key.steps % 31) + x);
            if (t.find(key) != 1 + (int)(key.steps % 31) + x) return 1;
        }
    std::printf("%zu ", t.size());
    for (size_t b : {0, 1, 1023, 1024, 1025, 227 * 1024}) std::printf("%zu ", hp::smem_steps(b));
    std::printf("%d %d", t.find({&k[0], 1, 256, 5}), t.find({&k[0], 0, 512, 5}));
}
""")
    assert out == ["684", "0", "1", "1", "1", "2", "227", "0", "0"]
