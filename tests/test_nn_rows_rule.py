"""Which images the row-marching convolution takes: at the sizes measured on either side
of each line the rule takes the kernel that was faster (host code, compiled and run here)."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2605_02185_gb300", "csrc")

# channels, 128-pixel tiles per SM, us of the tile (or mma.sync) kernel, us of the row kernel
MEASURED = [
    (8, 32, 0.05, 4.88, 3.99), (8, 32, 1, 6.92, 4.97), (8, 32, 4, 9.60, 6.63), (8, 32, 32, 64.5, 18.2),
    (32, 8, 0.33, 6.41, 4.97), (32, 8, 2, 7.11, 6.80), (32, 8, 3, 7.54, 7.76), (32, 8, 4, 8.15, 9.13),
    (32, 8, 6, 15.6, 9.31), (32, 8, 32, 52.5, 22.2),
    (32, 32, 0.33, 4.43, 5.59), (32, 32, 4, 7.96, 9.07), (32, 32, 6, 12.8, 10.6), (32, 32, 32, 45.4, 26.0),
    (32, 64, 0.33, 5.02, 6.98), (32, 64, 3, 8.46, 9.80), (32, 64, 4, 12.0, 11.2), (32, 64, 32, 86.1, 48.5),
    (32, 96, 0.33, 5.25, 8.16), (32, 96, 3, 10.4, 11.4), (32, 96, 4, 13.2, 12.7), (32, 96, 32, 98.9, 58.2),
    (64, 32, 0.33, 5.65, 7.29), (64, 32, 8, 15.6, 16.1), (64, 32, 12, 21.3, 20.2), (64, 32, 32, 53.0, 42.3),
    (64, 64, 0.33, 6.02, 9.50), (64, 64, 6, 15.8, 17.6), (64, 64, 8, 20.1, 20.0), (64, 64, 32, 69.9, 51.0),
    (96, 32, 0.33, 6.50, 9.22), (96, 32, 8, 25.5, 26.3), (96, 32, 16, 47.2, 45.2), (96, 32, 32, 90.4, 84.6),
]


def test_rule_takes_the_faster_kernel(tmp_path):
    sms = 152
    args = "".join(f"p({ci}, {co}, {int(r * sms)});" for ci, co, r, _, _ in MEASURED)
    src, exe = tmp_path / "p.cc", tmp_path / "p"
    src.write_text('#include <cstdio>\n#include "nn_rows_rule.h"\n'
                   f'int main() {{ auto p = [](int a, int b, long long u) {{ '
                   f'std::putchar(gbnn_tc::rows_pay(a, b, u, {sms}) ? 49 : 48); }}; {args} }}')
    subprocess.run(["g++", "-std=c++17", f"-I{CSRC}", str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout
    for (ci, co, r, tile, row), took in zip(MEASURED, out, strict=True):
        assert (took == "1") == (row < tile), (ci, co, r)
