"""A kernel's attributes are set once on every device that a process uses (csrc/per_device.h), and no launch keeps
them once per process.  The device is a fake one."""
import os
import re

from _host_unit import CSRC, run_host_unit

PROGRAM = r"""
#include <cstdio>
#include "per_device.h"
static int device = 0;
extern "C" cudaError_t cudaGetDevice(int* d) { *d = device; return cudaSuccess; }
int main() {
    static molt::PerDevice kept;
    int runs = 0;
    auto launch = [&](int dev, int value) {
        device = dev;
        const int got = kept.get([&] { ++runs; return value; });
        std::printf("%d %d\n", got, runs);
    };
    launch(0, 100);    // set up on device 0
    launch(0, 7);      // kept
    launch(1, 200);    // device 1 has its own
    launch(0, 7);
    launch(2, -1);     // an error is not kept
    launch(2, 300);
    launch(1000, 5);   // beyond the table: every time
    launch(1000, 6);
    return 0;
}
"""


def test_attributes_are_set_up_on_every_device(tmp_path):
    got = [tuple(map(int, line.split())) for line in run_host_unit(tmp_path, PROGRAM).splitlines()]
    assert got == [(100, 1), (100, 1), (200, 2), (100, 2), (-1, 3), (300, 4), (5, 5), (6, 6)]


def test_no_launch_sets_attributes_once_per_process():
    for name in os.listdir(CSRC):
        with open(os.path.join(CSRC, name)) as fh:
            text = fh.read()
        once = re.findall(r"static (?:const )?\w+ \w+ =[^;]*(?:smem_optin|cudaFuncSetAttribute)", text)
        assert not once, (name, once)
