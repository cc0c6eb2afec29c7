"""Radix plans on the host: an element count that no kernel is compiled for is
refused for every length, zero and negative counts included (the table of stage
twiddles asks for each count up to 16)."""
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CODE = """
import ctypes, sys
from paper_1003_4322_gb300 import _native
lib = ctypes.CDLL(_native.LIB_PATH)
make = lib._ZN3nsk11make_plan_eEiiPNS_4PlanE   # nsk::make_plan_e(int, int, Plan *)
make.restype = ctypes.c_bool
buf = ctypes.create_string_buffer(256)
for n in range(0, 1025):
    print(n, *(E for E in range(-2, 33) if make(n, E, buf)))
"""


def test_element_counts_that_a_length_takes():
    from paper_1003_4322_gb300 import _native, build
    if not os.path.exists(_native.LIB_PATH):
        build.build()
    r = subprocess.run([sys.executable, "-c", CODE], cwd=ROOT, capture_output=True, text=True)
    assert r.returncode == 0, r.returncode   # a division by zero ends the process here
    for line in r.stdout.splitlines():
        n, *taken = map(int, line.split())
        want = []
        for E in (4, 6, 8, 9, 12, 16):
            m = n
            for p in (2, 3):   # the factors of n that radices dividing E can take
                while n >= 4 and n % E == 0 and E % p == 0 and m % p == 0:
                    m //= p
            if n >= 4 and n % E == 0 and m == 1:
                want.append(E)
        assert taken == want, n
