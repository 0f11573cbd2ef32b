"""Coefficients of the sixth-order kernels (fch_coef, csrc/molt_internal.h): sums of constants are formed in 64 bits and
rounded once to the field's precision."""
import numpy as np

from _host_unit import run_host_unit

PROGRAM = r"""
#include <cuda_runtime.h>
#include <cstdio>
#include "molt_internal.h"
int main() {
    molt::FchConsts c;
    for (int i = 0; i < 4000; ++i) {
        c.c_eta = -8.0 + 16.0 * ((i * 2654435761u) % 4001u) / 4001.0;
        const molt::FchCoef<float> f = molt::fch_coef<float>(c);
        const molt::FchCoef<double> d = molt::fch_coef<double>(c);
        std::printf("%.17g %.9g %.9g %.17g %.17g\n", c.c_eta, f.c3, f.c32, d.c3, d.c32);
    }
    return 0;
}
"""


def test_sums_are_rounded_once(tmp_path):
    rows = np.array([[float(x) for x in line.split()] for line in run_host_unit(tmp_path, PROGRAM).splitlines()])
    c = rows[:, 0]
    for k, exact in ((1, 3 + c), (2, 3 + 2 * c)):
        assert np.array_equal(rows[:, k].astype(np.float32), exact.astype(np.float32))
        assert np.array_equal(rows[:, k + 2], exact)
    # (summed in the field's precision they would differ here)
    assert (np.float32(3) + c.astype(np.float32) != (3 + c).astype(np.float32)).any()
