"""What mars_energy returns for each status word its kernels can leave: bad spins
are the caller's fault, a bounded wait that gave up is not."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_status_words(tmp_path):
    src = tmp_path / "status.cpp"
    src.write_text('#include "device_status.h"\n#include <cstdio>\nint main() {\n'
                   "  using namespace mars;\n"
                   "  const int got[4] = {energy_status_rc(kDevOk), energy_status_rc(kDevBadIndex),\n"
                   "                      energy_status_rc(kDevTimeout), energy_status_rc(77)};\n"
                   "  const int want[4] = {MARS_OK, MARS_EINVAL, MARS_ETIMEOUT, MARS_EDEVICE};\n"
                   "  for (int k = 0; k < 4; ++k)\n"
                   '    if (got[k] != want[k]) return std::printf("status %d: %d\\n", k, got[k]), 1;\n'
                   "  return 0;\n}\n")
    exe = tmp_path / "status"
    csrc = os.path.join(ROOT, "paper_1907_05124_gb300", "csrc")
    subprocess.run(["g++", "-std=c++17", "-I", csrc, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
