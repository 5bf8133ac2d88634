"""The polynomial that replaces some of the attention kernels' exponentials where only the E2M1 code of the value counts: its coefficients,
evaluated as the kernel does (fp32 fused multiply-adds), round to the code of the exact 2^x at every argument that ex2.approx itself
is sure of (2^x at least its error, 2^-22, away from where the code changes).  On the GPU both are compared at every argument."""
import os
import re

import numpy as np
import pytest
import torch

from oracle import mxfp4

SRC = os.path.join(os.path.dirname(__file__), "..", "paper_2607_24377_b200", "csrc", "tc_helpers.cuh")
EDGES = (0.25, 0.75, 1.25, 1.75, 2.5, 3.5, 5.0)


def coefficients():
    text = re.search(r"kExp2Poly\[8\] = \{([^}]*)\}", open(SRC).read()).group(1)
    return np.array([float(v.strip().rstrip("f")) for v in text.split(",")], dtype=np.float32)


def poly(x):
    y = np.full(x.shape, coefficients()[7], dtype=np.float32)
    with np.errstate(over="ignore", invalid="ignore"):
        for c in coefficients()[6::-1]:            # the product of two fp32 values and the sum in 64 bits of significand, rounded once
            y = (y.astype(np.longdouble) * x.astype(np.longdouble) + np.longdouble(c)).astype(np.float32)
    return y


def code(y):                                       # the conversion with .relu: what is not positive is 0, ties to even, 6 is the largest
    return sum((y >= e) if e in (0.75, 1.75, 3.5) else (y > e) for e in EDGES)


def check(x):
    exact = np.exp2(x.astype(np.float64))
    sure = np.all([np.abs(exact / e - 1.0) > 2.0 ** -22 for e in EDGES], axis=0)
    assert sure.mean() > 0.9
    assert np.array_equal(code(poly(x))[sure], code(exact)[sure])


def test_codes_are_those_of_the_format():
    v = np.concatenate([np.linspace(0.0, 8.0, 4097), np.array(EDGES)])
    assert np.array_equal(code(v), mxfp4.e2m1_index(v))


@pytest.mark.parametrize("edge", EDGES)
def test_beside_a_change_of_code(edge):
    at = np.float32(np.log2(edge)).view(np.int32).astype(np.int64)
    check((at + np.arange(-40000, 40001)).astype(np.int32).view(np.float32))


def test_from_minus_infinity_to_the_largest_probability():
    check(np.linspace(-30.0, 3.01, 400001).astype(np.float32))
    far = -np.logspace(0.7, 38, 2000).astype(np.float32)
    assert (code(poly(np.append(far, -np.float32(np.inf)))) == 0).all()
    assert (code(poly(np.linspace(2.33, 128.0, 20001).astype(np.float32))) == 7).all()


def test_error_in_between_is_as_stated():
    err = lambda lo, hi: np.abs(poly(x := np.linspace(lo, hi, 100001).astype(np.float32)).astype(np.float64) - np.exp2(x.astype(np.float64))).max()
    assert 0.006 < err(-4.0, -2.0) <= 0.0065 and err(-2.0, np.log2(5.0)) < 3e-4


@pytest.mark.gpu
def test_codes_of_every_argument_are_those_of_the_exponential():
    import paper_2607_24377_b200 as mx
    status = torch.zeros(4, dtype=torch.int32, device="cuda")
    mx.selftest_exp2_codes(status)
    assert status.tolist()[:2] == [0, 0], hex(int(status[2]) & 0xFFFFFFFF)
