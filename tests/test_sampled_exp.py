"""The acceptance kernel's exponential (csrc/exp_le0.cuh: a table of 2^(i/64) and five terms of the series), the
kernel's own source compiled for the host: within two units in the last place of e^t over the range of softmax
arguments, 0 below -700."""
import os
import subprocess

import numpy as np

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2601_12212_b200", "csrc")
DRIVER = """
#include <cstdio>
#include "exp_le0.cuh"
int main() {
    double table[resps::kExpTable], t;
    for (int i = 0; i < resps::kExpTable; ++i) table[i] = std::exp2(static_cast<double>(i) / resps::kExpTable);
    while (std::fread(&t, 8, 1, stdin) == 1) {
        const double v = resps::exp_le0(t, table);
        std::fwrite(&v, 8, 1, stdout);
    }
}
"""


def test_table_driven_exponential(tmp_path):
    src, exe = tmp_path / "driver.cpp", tmp_path / "driver"
    src.write_text(DRIVER)
    # (no contraction: the device code's only fused operations are those written as fma)
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    rng = np.random.default_rng(0)
    edges = np.arange(-64000, 1) * np.log(2) / 128          # ends and middles of the table's intervals
    t = np.concatenate([-rng.exponential(8.0, 200000), -rng.uniform(0, 699.9, 200000), edges[edges > -699.9],
                        [0.0, -0.0, -1e-15, -1e-300, -5e-324, -699.9999]])
    below = np.array([-700.0, -700.5, -745.0, -1e4, -1e300, -np.inf])
    out = subprocess.run([str(exe)], input=np.concatenate([t, below]).tobytes(), capture_output=True, check=True).stdout
    got = np.frombuffer(out, np.float64)
    want = np.exp(t.astype(np.longdouble))
    assert np.max(np.abs(got[:len(t)] / want - 1)) < 2 * 2.3e-16
    assert np.all(got[len(t):] == 0.0)


def test_the_kernel_has_no_other_exponential():
    text = open(os.path.join(CSRC, "sampled.cu")).read()
    assert '#include "exp_le0.cuh"' in text and "double exp_le0(" not in text
    assert text.count("exp_le0(") == 3                      # target side, draft side, the CTAs' common scale
