"""The arithmetic the transforms run (residues in [0, 2r), products by a constant with
its quotient) as exact integers: every operation of field.cuh against its definition
and the bounds stated there, on operands at the ends of its range and with limbs whose
carries run the length of a chain.  Two moduli without a shortcut for their lowest limb
take the products' general rows, which none of the three fields does."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from oracle import field as fld
from workloads import ints_to_limbs, limbs_to_ints, splitmix64

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
R = 1 << 256
MODULI = {"bls12_381_fr": fld.BLS12_381.r, "bn254_fr": fld.BN254.r, "bls12_377_fr": fld.BLS12_377.r,
          "general_252": (1 << 252) + 27742317777372353535851937790883648493,
          "general_255": (1 << 255) - 19}
OPS = ["mul", "add_loose", "sub_loose", "diff_loose", "mul_factor", "mul_high", "mul_low",
       "mul_low_fold", "make_factor", "reduce_once"]
N = 1 << 13


@pytest.fixture(scope="module")
def check(tmp_path_factory):
    from paper_2509_22684_gb300 import build
    so = str(tmp_path_factory.mktemp("arith") / "arith_check.so")
    subprocess.run([build._nvcc(), *build.ARCH, "-O3", "-std=c++17", "-Xcompiler", "-fPIC", "-shared",
                    f"-I{build.CSRC}", os.path.join(ROOT, "tests", "cuda", "arith_check.cu"), "-o", so],
                   check=True)
    fn = ctypes.CDLL(so).arith_check
    fn.argtypes = [ctypes.c_int, ctypes.c_int] + [ctypes.c_void_p] * 5 + [ctypes.c_size_t]

    def call(modulus, op, a, b, c):
        import torch
        torch.cuda.init()
        v = [np.ascontiguousarray(ints_to_limbs(u), dtype=np.uint32) for u in (a, b, c)]
        out = [np.zeros_like(v[0]) for _ in range(2)]
        st = fn(list(MODULI).index(modulus), OPS.index(op), *(x.ctypes.data for x in v + out), len(a))
        assert st == 0, f"CUDA error {st}"
        return [limbs_to_ints(x) for x in out]
    return call


def _operands(r, top, seed):
    """N integers in [0, top]: the ends of the range and of the residues', limbs of 0,
    1, 2^31, 2^32 - 1 and the modulus's own, and uniform ones."""
    words = splitmix64(seed, 0, 24 * N).reshape(N, 24)
    edge = [v for m in range(5) for v in (m * r - 1, m * r, m * r + 1)]
    edge += [0, 1, top, top - 1, r >> 1, (1 << 255) - 1, 1 << 255, (1 << 224) - 1, R - (1 << 228)]
    edge = [v for v in edge if 0 <= v <= top]
    out = []
    for i in range(N):
        w = [int(x) for x in words[i]]
        if i % 3 == 0:
            v = edge[w[0] % len(edge)]
        elif i % 3 == 1:
            limb = [0, 1, 1 << 31, 0xFFFFFFFF]
            v = sum((limb + [(r >> (32 * k)) & 0xFFFFFFFF])[w[k] % 5] << (32 * k) for k in range(8))
        else:
            v = w[0] | w[1] << 64 | w[2] << 128 | w[3] << 192
        out.append(v if v <= top else v % (top + 1))
    return out


@pytest.mark.parametrize("modulus", list(MODULI))
@pytest.mark.parametrize("op", OPS)
def test_operation(check, modulus, op):
    r = MODULI[modulus]
    a, b, c = (_operands(r, R - 1, 70 + k) for k in range(3))
    canonical = _operands(r, r - 1, 80)
    loose = [_operands(r, 2 * r - 1, 90 + k) for k in range(2)]
    if op == "mul":         # canonical by anything below 2^256, canonical
        got, _ = check(modulus, op, canonical, b, c)
        inv = pow(R, -1, r)
        bad = [i for i in range(N) if got[i] != canonical[i] * b[i] * inv % r]
    elif op in ("add_loose", "sub_loose"):      # in [0, 2r) from [0, 2r)
        x, y = loose
        got, _ = check(modulus, op, x, y, c)
        bad = [i for i in range(N) if got[i] >= 2 * r or
               (got[i] - (x[i] + y[i] if op == "add_loose" else x[i] - y[i])) % r]
    elif op == "diff_loose":    # where 4r < 2^256 the exact x + 2r - y, else in [0, 2r)
        x, y = loose
        got, _ = check(modulus, op, x, y, c)
        if 4 * r < R:
            bad = [i for i in range(N) if got[i] != x[i] + 2 * r - y[i]]
        else:
            bad = [i for i in range(N) if got[i] >= 2 * r or (got[i] - x[i] + y[i]) % r]
    elif op == "mul_factor":    # in [0, 2r) for x up to 2^256 - 2^228
        x = _operands(r, R - (1 << 228), 100)
        got, _ = check(modulus, op, x, canonical, [w * R // r for w in canonical])
        bad = [i for i in range(N) if got[i] >= 2 * r or (got[i] - x[i] * canonical[i]) % r]
    elif op == "mul_high":      # the quotient, short by at most 1
        got, _ = check(modulus, op, a, b, c)
        bad = [i for i in range(N) if not 0 <= a[i] * b[i] // R - got[i] <= 1]
    elif op == "mul_low":
        got, _ = check(modulus, op, a, b, c)
        bad = [i for i in range(N) if got[i] != a[i] * b[i] % R]
    elif op == "mul_low_fold":
        got, _ = check(modulus, op, a, b, c)
        bad = [i for i in range(N) if got[i] != (a[i] * b[i] + c[i] * (R - r)) % R]
    elif op == "make_factor":   # w without its Montgomery factor, and floor(w 2^256 / r)
        ninv = -pow(r, -1, R) % R
        got, quo = check(modulus, op, canonical, [ninv] * N, c)
        inv = pow(R, -1, r)
        w = [m * inv % r for m in canonical]
        bad = [i for i in range(N) if (got[i], quo[i]) != (w[i], w[i] * R // r)]
    else:
        x = loose[0]
        got, _ = check(modulus, op, x, b, c)
        bad = [i for i in range(N) if got[i] != x[i] % r]
    assert not bad, f"{len(bad)} of {N} wrong, first at {bad[0]}: {got[bad[0]]:x}"
