"""The host's rules that choose a kernel, a tile or a schedule, on the CPU."""
import subprocess

from paper_2402_08725_gb300 import build


def _run_cpp(tmp_path, body):
    """Integers printed by the statements `body`, compiled against the library's internal headers."""
    src, exe = tmp_path / "rule.cu", str(tmp_path / "rule")
    src.write_text('#include <cstdio>\n#include "kernels.cuh"\nint main() {\n' + body + "\n}\n")
    subprocess.run([build.nvcc(), "-std=c++17", "-I", build.INCLUDE, "-I", build.CSRC, str(src), "-o", exe], check=True)
    return [int(v) for v in subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split()]


def test_an_epoch_without_a_second_pairs_its_phases(tmp_path):
    """Transforms of the kernel spectra: one per phase of two epochs, half as many for a single one."""
    calls = "".join(f'  printf("%d\\n", sr::fft_kappa_items({E}, {f}));\n' for E in (1, 2, 3, 8) for f in (1, 2, 3))
    assert _run_cpp(tmp_path, calls) == [1, 2, 5, 1, 4, 9, 2, 6, 14, 4, 16, 36]
