"""The FP64 path's far field (double-float arithmetic, df_field.cuh) on the CPU.

The header compiles for the host as well; df_field_check.cpp evaluates it pair by
pair, and the nodal force parts of small loop ensembles in the kernel's groups of
60 sources, against 80-bit numbers.  The reciprocal seeds are perturbed by the error
of the hardware's.

The bars, derived from the arithmetic (u = 2^-24, the FP32 rounding):
  * a split value: each part to nearest, so within u^2 of the value, and unbiased: the
    mean over 10^6 values within 2^-56 (truncation: 2^-46 at most, 2^-48 on average);
  * a pair: an operation rounds a low part of up to 2^-23 of the value, 2^-47; some 40
    lie on the longest path, so 40 x 2^-47 = 2.8e-13 if all pull the same way and the
    square root of that count, 4.5e-14, at random.  The point-to-line geometry loses up to a
    factor of 16 (the near limit is 1/16 of a length).  Median 1e-13, 99 % 1e-12, all 1e-11;
  * force parts: neighbouring sources of a loop pull against each other by up to ten times what
    is left: 4.5e-13, bar 1e-12.

Mistakes planted in copies of the header (a sign, a coefficient, a dropped low part,
a truncated split) must break a bar.
"""

import concurrent.futures
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2005_02498_gb300", "csrc")
KINDS = ["near_limit", "middle", "ends", "screw", "almost_screw", "long_source", "range_limit"]

MUTANTS = [
    ("aw_sign", "df_add_big(ssum, df_neg(df_mul(G.d2, i12)))", "df_add_big(ssum, df_mul(G.d2, i12))"),
    ("kn_dropped", "df_fma(df_all(K.nra2), K3, df_mul(df_all(K.kn), J1))", "df_fma(df_all(K.nra2), K3, J1)"),
    ("cb_sign", "cb = df_mul(df_neg(ga), B0);", "cb = df_mul(ga, B0);"),
    ("b_part_from_a0", "cb = df_mul(df_neg(ga), B0);", "cb = df_mul(df_neg(ga), A0);"),
    ("straddling_sum", "df_mul(df_sub(p, m), rr)", "df_mul(df_add(p, m), rr)"),
    ("product_low_part", "return DF2{p, p_fma(a.l, b.h, p_fma(a.h, b.l, p_fma(a.h, b.h, p_neg(p))))};",
     "return DF2{p, p_fma(a.l, b.h, p_fma(a.h, b.h, p_neg(p)))};"),
    ("sum_low_parts", "return DF2{s, p_add(e, p_add(a.l, b.l))};\n}\nDF_FN DF2 df_sub",
     "return DF2{s, p_add(a.l, b.l)};\n}\nDF_FN DF2 df_sub"),
    ("root_second_order", "p_fma(e, p_all(0.375f), p_all(0.5f))", "p_all(0.25f)"),
    ("split_truncates", " + ((lo >> 28) & 1u);", ";"),
    ("shape_functions_swapped", "F[e] = ch ? df_fma(f, ws, F[e]) : df_mul(f, ws);",
     "F[e] = ch ? df_fma(f, we, F[e]) : df_mul(f, we);"),
    ("group_b_part", "s[e] = df_fma(b, bt[e], s[e]);", "s[e] = df_add(b, s[e]);"),
]


def results(workdir, mutant=None):
    """The program's lines for the header, or for a copy of it with a mistake: {(word, kind): numbers}."""
    inc = CSRC
    if mutant:
        inc = str(workdir)
        text = open(os.path.join(CSRC, "df_field.cuh")).read()
        assert text.count(mutant[1]) == 1, "%s: the text to mutate occurs %d times" % (mutant[0], text.count(mutant[1]))
        open(os.path.join(inc, "df_field.cuh"), "w").write(text.replace(mutant[1], mutant[2]))
    exe = os.path.join(str(workdir), "check")
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-Wno-attributes", "-I" + cuda, "-I" + inc,
                    os.path.join(HERE, "df_field_check.cpp"), "-o", exe], check=True, capture_output=True, text=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True, timeout=300).stdout
    found = {}
    for line in out.splitlines():
        w = line.split()
        key = (w[0], w[1]) if w[0] in ("pair", "forces") else (w[0], "")
        found[key] = [float(x) for x in w[2 if key[1] else 1:]]
    return found


def broken(r):
    """The bars that the results break ("not <=", so that NaN breaks them)."""
    bars = [(("split", ""), [2.0 ** -48, 2.0 ** -56]), (("round", ""), [0.0])]
    bars += [(("pair", k), [1e-13, 1e-12, 1e-11]) for k in KINDS]
    bars += [(("forces", k), [1e-12]) for k in ("2", "16")]
    return [(key, x, b) for key, most in bars for x, b in zip(r[key], most) if not x <= b]


def test_far_field_against_80_bits(tmp_path):
    assert not broken(results(tmp_path))


def test_planted_mistakes_break_a_bar(tmp_path):
    def run(m):
        d = tmp_path / m[0]
        d.mkdir()
        return broken(results(d, m))

    with concurrent.futures.ThreadPoolExecutor(max_workers=4) as ex:
        found = list(ex.map(run, MUTANTS))
    survivors = [m[0] for m, b in zip(MUTANTS, found) if not b]
    assert not survivors, "mistakes that no bar catches: %s" % survivors
