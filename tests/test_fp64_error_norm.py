"""The FP64 step control's position error with infinite or NaN components, on
the host: max(|e_r|, r |e_theta|, r sin(theta) |e_phi|), NaN ignored and the last
term taken with its sign, the value the finite case has."""
import subprocess

import numpy as np

from paper_2506_18579_gb300 import build as rtbuild

CODE = """#include <cstdio>
#include "rtgd_fp64.cuh"
int main() {
    double r, sth, a, b, c;
    while (std::scanf("%lf %lf %lf %lf %lf", &r, &sth, &a, &b, &c) == 5)
        std::printf("%.17g\\n", rtgd::max3_rare(a, r, b, r * sth, c));
}
"""


def test_rare_position_error(tmp_path):
    src, exe = tmp_path / "norm.cu", tmp_path / "norm"
    src.write_text(CODE)
    subprocess.run([rtbuild.NVCC, *rtbuild.ARCH, *rtbuild.FLAGS, str(src), "-o", str(exe)], check=True)
    inf, nan = float("inf"), float("nan")
    rows = [(6400.0, s, *e) for s in (0.5, -0.25) for e in
            ((nan, 2e-9, 3.0), (nan, -2e-9, inf), (1e-7, nan, -4.0), (inf, 1.0, 1.0), (nan, nan, -1e-3), (-3e-6, inf, nan))]
    got = subprocess.run([str(exe)], input="\n".join(" ".join(map(repr, r)) for r in rows), text=True,
                         capture_output=True, check=True).stdout.split()
    for (r, s, a, b, c), g in zip(rows, got):
        want = np.fmax(abs(a), np.fmax(r * abs(b), r * s * abs(c)))
        assert float(g) == want or (np.isnan(want) and np.isnan(float(g))), (r, s, a, b, c)
