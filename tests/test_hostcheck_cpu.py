"""Host-compiled checks of device logic (no GPU): the production headers are
compiled as host code with nvcc.

* The band kernel's triangle items: the compact enumeration (cumulative
  table, binary search, column range) equals the skipping raster, tile for
  tile, over every small geometry (tests/hostcheck/tri_enum.cu).
* The CRT reconstruction's rounding of the exact integer Z 2^s to dd
  (bigfloat.cuh): against exact rationals, hi is the nearest binary64 of the
  value when Z has at most 128 significant bits, and |hi + lo - Z 2^s| stays
  within (2^-106 + 2^-126) |Z 2^s| (plus the subnormal spacing), with
  overflow to a correctly signed infinity.
* The digit form's rounding of the recombined integer V 2^s: hi and lo are the
  nearest binary64 numbers of the value and of what hi leaves, both signs
  (hostcheck/bands_dd.cu).
* two_sum (dd_arith.cuh), which orders its operands by their leading words:
  equal to Knuth's TwoSum over the whole binary64 range (hostcheck/two_sum.cu).
* A device wait that gives up takes its call's certificate back, so that the
  plain kernel computes C (hostcheck/give_up.cu).
"""
from __future__ import annotations

import ctypes
import math
import os
import random
import shutil
import subprocess
from fractions import Fraction

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(ROOT, "paper_2109_13406_gb300", "csrc")
INCLUDE = os.path.join(ROOT, "include")


def _nvcc():
    path = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(path):
        pytest.skip("nvcc not available")
    return path


def _build(src, out, shared):
    cmd = [_nvcc(), "-O2", "-std=c++17", "-x", "cu", "-I", CSRC, "-I", INCLUDE, src, "-o", out]
    if shared:
        cmd[1:1] = ["-shared", "-Xcompiler", "-fPIC"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]


def test_triangle_items_match_the_skipping_raster(tmp_path):
    exe = str(tmp_path / "tri_enum")
    _build(os.path.join(HERE, "hostcheck", "tri_enum.cu"), exe, shared=False)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    cases, bad = (int(x) for x in r.stdout.split()[1::2])
    assert cases > 3000 and bad == 0


def test_two_sum_equals_knuths(tmp_path):
    exe = str(tmp_path / "two_sum")
    _build(os.path.join(HERE, "hostcheck", "two_sum.cu"), exe, shared=False)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    pairs, bad = (int(x) for x in r.stdout.split()[1::2])
    assert pairs == 8000000 and bad == 0


def test_prod_error_equals_the_fma(tmp_path):
    exe = str(tmp_path / "prod_error")
    _build(os.path.join(HERE, "hostcheck", "prod_error.cu"), exe, shared=False)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    pairs, bad = (int(x) for x in r.stdout.split()[1::2])
    assert pairs == 6000000 and bad == 0


def test_a_wait_that_gave_up_leaves_c_to_the_plain_kernel(tmp_path):
    exe = str(tmp_path / "give_up")
    _build(os.path.join(HERE, "hostcheck", "give_up.cu"), exe, shared=False)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    cases, bad = (int(x) for x in r.stdout.split()[1::2])
    assert cases == 21 and bad == 0


def test_words_to_dd_rounding(tmp_path):
    so = str(tmp_path / "words_dd.so")
    _build(os.path.join(HERE, "hostcheck", "words_dd.cu"), so, shared=True)
    lib = ctypes.CDLL(so)
    U8 = ctypes.c_uint32 * 8
    D2 = ctypes.c_double * 2
    lib.words_to_dd.argtypes = [U8, ctypes.c_uint32, ctypes.c_int, D2]
    g = random.Random(11)
    for it in range(20000):
        nbits = g.choice([1, 31, 32, 33, 53, 54, 64, 105, 106, 107, 127, 128, 129, 200, 256])
        Z = g.getrandbits(nbits) | (1 << (nbits - 1))
        if g.random() < 0.1:
            Z = (1 << nbits) - 1                       # all ones: the rounding carries
        s = g.choice([g.randint(-300, 50), g.randint(-1300, -1000), g.randint(800, 1100)])
        neg = g.random() < 0.5
        out = D2()
        lib.words_to_dd(U8(*[(Z >> (32 * t)) & 0xFFFFFFFF for t in range(8)]), int(neg), s, out)
        x = Fraction(Z) * Fraction(2) ** s * (-1 if neg else 1)
        if abs(x) >= Fraction(2) ** 1024 * (1 - Fraction(2) ** -54):
            assert math.isinf(out[0]) and (out[0] < 0) == neg
            continue
        err = abs(Fraction(out[0]) + Fraction(out[1]) - x)
        assert err <= abs(x) * (Fraction(2) ** -106 + Fraction(2) ** -126) + Fraction(2) ** -1074
        if Z.bit_length() <= 128 and abs(x) > Fraction(2) ** -900:
            assert out[0] == float(x)


def test_signed_words_to_dd_is_the_general_rounding(tmp_path):
    """The reconstruction kernel's rounding of a two's complement Z equals
    from_words and to_dd on its magnitude bit for bit: leading bits in every
    word, zero and all-one words below, exponents past the normal range."""
    so = str(tmp_path / "words_dd.so")
    _build(os.path.join(HERE, "hostcheck", "words_dd.cu"), so, shared=True)
    lib = ctypes.CDLL(so)
    U8 = ctypes.c_uint32 * 8
    D2 = ctypes.c_double * 2
    for f in (lib.words_to_dd, lib.signed_words_to_dd):
        f.argtypes = [U8, ctypes.c_uint32, ctypes.c_int, D2]
    g = random.Random(12)
    fill = [0, 0xFFFFFFFF, 0x80000000, 1, 0x7FF, 0x400, 0x800]
    for it in range(60000):
        nbits = g.choice([0, 1, 53, 54, 96, 107, 127, 128, 160, 192, 193, 223, 224, 225, 230, 240, 254, 255])
        z = [g.choice(fill) if g.random() < 0.3 else g.getrandbits(32) for _ in range(8)]
        Z = sum(w << (32 * t) for t, w in enumerate(z)) & ((1 << nbits) - 1)
        if nbits:
            Z |= 1 << (nbits - 1)
        if g.random() < 0.2:
            Z = (Z >> (nbits // 2)) << (nbits // 2)
        s = g.choice([g.randint(-300, 50), g.randint(-1300, -1000), g.randint(700, 1100)])
        neg = int(Z != 0 and g.random() < 0.5)
        words = U8(*[(Z >> (32 * t)) & 0xFFFFFFFF for t in range(8)])
        a, b = D2(), D2()
        lib.words_to_dd(words, neg, s, a)
        lib.signed_words_to_dd(words, neg, s, b)
        assert bytes(a) == bytes(b), (hex(Z), neg, s, list(a), list(b))


def test_bands_to_dd_is_the_nearest_dd(tmp_path):
    """V of up to 159 bits, as 14 or 15 bands of digit products give it: hi is
    V 2^s rounded to nearest and lo the rest rounded to nearest, whatever lies
    below the leading 128 bits.  Ties of both roundings that only the tail
    decides, all-one and zero words, both signs; exponents past the normal
    range within two subnormal units, or an infinity of V's sign."""
    so = str(tmp_path / "bands_dd.so")
    _build(os.path.join(HERE, "hostcheck", "bands_dd.cu"), so, shared=True)
    lib = ctypes.CDLL(so)
    U6 = ctypes.c_uint32 * 6
    D2 = ctypes.c_double * 2
    lib.bands_to_dd.argtypes = [U6, ctypes.c_int, D2]
    g = random.Random(13)
    fill = [0, 0xFFFFFFFF, 0x80000000, 1, 0x7FF, 0x400, 0x800]
    for it in range(60000):
        nbits = g.choice([0, 1, 53, 54, 96, 107, 127, 128, 129, 140, 145, 150, 157, 158, 159])
        Z = sum((g.choice(fill) if g.random() < 0.3 else g.getrandbits(32)) << (32 * t)
                for t in range(5)) & ((1 << nbits) - 1)
        if nbits:
            Z |= 1 << (nbits - 1)
        if nbits > 128 and g.random() < 0.5:
            # a tie of hi (or one of lo) in the leading 128 bits, 0 or 1 below
            low = nbits - 53 if g.random() < 0.5 else nbits - 53 - g.randint(53, 75)
            Z = (Z >> low << low) + (1 << (low - 1)) + g.choice([-1, 0, 1])
        s = g.choice([g.randint(-300, 50), g.randint(-1200, -1000), g.randint(700, 1100)])
        V = -Z if g.random() < 0.5 else Z
        out = D2()
        lib.bands_to_dd(U6(*[(V >> (32 * t)) & 0xFFFFFFFF for t in range(6)]), s, out)
        x = Fraction(V) * Fraction(2) ** s
        if abs(x) >= Fraction(2) ** 1024 * (1 - Fraction(2) ** -54):
            assert math.isinf(out[0]) and (out[0] < 0) == (V < 0)
            continue
        hi, lo = Fraction(out[0]), Fraction(out[1])
        if x == 0 or abs(x) > Fraction(2) ** -860:
            assert out[0] == float(x) and out[1] == float(x - hi), (hex(V), s, list(out))
        else:
            assert abs(x - hi - lo) <= abs(x) * Fraction(2) ** -106 + Fraction(2) ** -1073
