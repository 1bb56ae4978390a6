"""Scratch that one part of the library reserves and another fills
(csrc/size_rules.h), compiled with the host C++ compiler: whatever batches a
call is cut into, every batch fits what was reserved for the first."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2009_12663_gb300", "csrc")


def run(tmp_path, body):
    src = tmp_path / "rules.cpp"
    src.write_text("#include <cstdio>\n#include <initializer_list>\n#include \"size_rules.h\"\nusing namespace sizes;\n"
                   "int main() {\n  int bad = 0;\n" + body + "  return bad != 0;\n}\n")
    exe = str(tmp_path / "rules")
    subprocess.check_call(["g++", "-std=c++17", "-Wall", "-Werror", "-I", CSRC, str(src), "-o", exe])
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


def test_strain_sums_of_every_batch_fit_the_buffer_of_the_first(tmp_path):
    run(tmp_path, r"""
  for (int nex : {1, 5, 12, 57, 81, 126, 160, 253, 340})
    for (int nez : {1, 3, 6, 21, 46, 60, 70})
      for (int nt : {2, 15, 16, 40, 500, 800, 1333, 3000})
        for (int nshot = 1; nshot <= 24; ++nshot)
          for (int most = 1; most <= nshot; ++most) {
            const int last = last_batch(nshot, most);
            const long long ne = (long long)nex * nez;
            if (last < 1 || last > most || (nshot - last) % most || integral_bytes(ne, nt, last) > integral_bytes(ne, nt, most)) {
              std::printf("%d x %d, nt %d: %d shots by %d\n", nex, nez, nt, nshot, most);
              ++bad;
            }
          }
""")
