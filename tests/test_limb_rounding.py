"""Host check of the rounding that the finite differences end with (csrc/stage_int.cuh, limb_bits).

The function is compiled for the host and run on sums x + y 2^21 + z 2^42 of every size (random, ties and their
neighbours, the edges between its one-word and its shortened form, zero) and on reference exponents
inside and outside the range of normal results; the exact value is an integer times a power of two, so
Python's integers give the correctly rounded FP64 result (round to nearest even) to the last bit.
"""
import random
import struct
import subprocess

from paper_2606_02053_gb300 import build as libbuild

SRC = r"""
#include <cstdio>
#include "stage_split.cuh"
template <bool ODD>
static unsigned long long both(cosmos::Limb S, int e) {
  const unsigned long long any = cosmos::limb_bits<ODD, true>(S, e);
  // sums that fit one word take the shorter form in a warp without large ones: the same bits
  return cosmos::limb_big(S) || cosmos::limb_bits<ODD, false>(S, e) == any ? any : ~0ull;
}
static unsigned long long form(cosmos::Limb S, int e) { return cosmos::limb_odd(e) ? both<true>(S, e) : both<false>(S, e); }
int main() {
  int x, y, z, e;
  while (scanf("%d %d %d %d", &x, &y, &z, &e) == 4)
    printf("%llu\n", form({(unsigned long long)x + ((unsigned long long)y << 21) + ((unsigned long long)z << 42), z}, e));
  return 0;
}
"""
TOP = 679_000_000  # 324 x 2^21: the largest sum of upper parts


def rounded(v, e):
    """FP64 bits of v 2^(e - 1085), round to nearest even; results below the normal range are zero."""
    if e >= 2047:
        return 0x7FF8000000000000
    if v == 0:
        return 0
    sign, u = (1 << 63 if v < 0 else 0), abs(v)
    n = u.bit_length() - 1
    if n > 52:
        q, r = u >> (n - 52), u & ((1 << (n - 52)) - 1)
        half = 1 << (n - 53)
        q += r > half or (r == half and q & 1)
    else:
        q = u << (52 - n)
    if q >> 53:
        q, n = q >> 1, n + 1
    ex = n + e - 1085 + 1023
    if ex <= 0:
        return sign
    if ex >= 2047:
        return sign | 0x7FF0000000000000
    return sign | ex << 52 | (q & ((1 << 52) - 1))


def digit_sums():
    r = random.Random(7)
    out = [(0, 0, 0)]
    for _ in range(20000):
        bits = [r.randint(0, 29) for _ in range(3)]
        out.append(tuple(r.randint(-min(TOP, 1 << b), min(TOP, 1 << b)) for b in bits))
    for _ in range(20000):  # a chosen value, ties among them, split into digits that may carry
        n = r.randint(50, 70)
        v = (r.getrandbits(53) | 1 << 52) << (n - 52) if n >= 52 else r.getrandbits(n)
        v += r.choice([0, 0, 1, -1, r.randint(-9, 9)]) + (1 << (n - 53) if n > 53 else 0) * r.choice([0, 1])
        v *= r.choice([1, -1])
        z = v >> 42
        y = (v >> 21) & ((1 << 21) - 1)
        x = v & ((1 << 21) - 1)
        c = r.randint(-200, 200)  # move a carry between the digits: the value stays
        out.append((x + (c << 21), y - c, z))
    edge = (1 << 21) - (1 << 11)
    for z in (edge, 1 << 28, 1 << 20, 1 << 21):
        for dz in range(-2, 3):
            for y in (0, 1, -1, TOP, -TOP):
                for x in (0, 1, -1, 255, 256, 511, 512, -256, -512, TOP, -TOP):
                    out += [(x, y, z + dz), (x, y, -z - dz)]
    return out


def test_limb_bits_is_round_to_nearest_even(tmp_path):
    cu, exe = tmp_path / "limbs.cu", tmp_path / "limbs"
    cu.write_text(SRC)
    subprocess.check_call([libbuild.nvcc(), "-std=c++17", "-O1", *libbuild.ARCH, "-I", libbuild.CSRC, "-o", str(exe), str(cu)])
    r = random.Random(8)
    cases = [(s, r.choice([1023, 1030, 900, 1085, 80, 79, 60, 1, 1960, 1961, 2030, 2046, 2047])) for s in digit_sums()]
    text = "".join("%d %d %d %d\n" % (*s, e) for s, e in cases)
    got = [int(v) for v in subprocess.run([str(exe)], input=text, capture_output=True, text=True, check=True).stdout.split()]
    assert len(got) == len(cases)
    for (s, e), g in zip(cases, got):
        want = rounded(s[0] + (s[1] << 21) + (s[2] << 42), e)
        assert g == want, (s, e, struct.pack(">Q", g).hex(), struct.pack(">Q", want).hex())
