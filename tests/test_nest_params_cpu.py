"""The FP32 line parameters of the nested passes (nest_line_params, csrc/line_params.cpp): their nu belongs to the rounded
decay, and stays the line's own where the decay is subnormal or underflows (nu above 87)."""
import math

import numpy as np
import pytest

from _host_unit import run_host_unit

PROGRAM = r"""
#include <cuda_runtime.h>
#include <cmath>
#include <cstdio>
#include "molt_internal.h"
int main() {
    const double nus[] = {0.05, 0.7, 5.0, 60.0, 87.0, 88.0, 96.0, 102.5, 103.0, 103.5, 110.0};
    for (double nu : nus)
        for (int M = 2; M <= 6; M += 2) {
            molt::LineParams<double> p;
            const char* err = nullptr;
            if (!molt::build_line_params(1.0, nu, 64, M, molt::BC_NEUMANN, &p, &err)) return 1;
            const molt::LineParams<float> own = molt::cast_line_params<float>(p), q = molt::nest_line_params(own);
            double sum = 0.0;
            for (int o = 0; o <= M; ++o) sum += q.wl[o];
            std::printf("%.17g %d %.9g %.9g %.9g %.17g\n", nu, M, q.nu, q.d, own.d, sum);
        }
    return 0;
}
"""


@pytest.fixture(scope="module")
def rows(tmp_path_factory):
    out = run_host_unit(tmp_path_factory.mktemp("params"), PROGRAM, ["line_params.cpp"])
    return [tuple(float(x) for x in line.split()) for line in out.splitlines()]


def test_nu_is_that_of_the_line(rows):
    for nu, M, q_nu, q_d, own_d, _ in rows:
        assert q_d == own_d                                        # (the recurrence keeps its decay)
        # a normal decay is half an ulp off: nu' within 2^-24 (1 + 1/nu) of nu, as FP32 stores it
        assert abs(q_nu / nu - 1) <= 2.0 ** -24 * (2 + 1 / nu), (nu, M, q_nu)


def test_weights_sum_to_the_mass_of_the_kernel(rows):
    # H 1 = 1: the local weights add up to (1 - d) / 2 for the d in use, each rounded to FP32
    for nu, M, _, d, _, total in rows:
        assert abs(total - (1 - d) / 2) <= (M + 1) * 2.0 ** -24, (nu, M)
        assert math.isfinite(total) and np.float32(d) == np.float32(math.exp(-nu))
