"""The library's sample-size bound (host code, compiled on its own) against the
oracle's scan of every grid point."""
import ctypes
import os
import random
import subprocess

import pytest

import oracle

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2509_11454_gb300", "csrc")


@pytest.fixture(scope="module")
def bound(tmp_path_factory):
    d = tmp_path_factory.mktemp("bounds")
    src, lib = d / "b.cpp", d / "b.so"
    src.write_text(f'#include "{CSRC}/bounds.cpp"\n'
                   'extern "C" long long sup(double e, double d, double dh, double r, double xh)'
                   '{ return (long long)std::ceil(percis::sup_objective(e, d, dh, r, xh)); }\n')
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-ffp-contract=off", "-I/usr/local/cuda/include",
                    "-o", str(lib), str(src)], check=True)
    f = ctypes.CDLL(str(lib)).sup
    f.restype, f.argtypes = ctypes.c_longlong, [ctypes.c_double] * 5
    return f


def test_sample_size_equals_the_full_scan(bound):
    rng = random.Random(0)
    for _ in range(400):
        eps, delta = 10 ** rng.uniform(-3.5, -0.3), 10 ** rng.uniform(-4, -0.05)
        dhat = 1.0 + 10 ** rng.uniform(-6, 4)
        rho = rng.choice([10 ** rng.uniform(-3, 4), 10 ** rng.uniform(4, 9)])
        xh = dhat / 2 * 10 ** rng.choice([0.0, rng.uniform(-8, 0)])
        try:
            ref, val = oracle.ell_sup(eps, delta, dhat, rho, xh)
        except (ValueError, ZeroDivisionError, OverflowError):  # a logarithm of 0 or a y of 0
            continue
        if val != val or abs(val) > 2.0 ** 62:
            continue
        assert bound(eps, delta, dhat, rho, xh) == ref, (eps, delta, dhat, rho, xh)
