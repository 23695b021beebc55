"""The 16-bit stores' rounding code, compiled for the host from ld_common.cuh
with the device intrinsics it names defined as the C operations they round
like. Stochastic rounding against the checker over every exponent, with the
infinities, NaN, the largest finite values and the subnormals; the initial
state's encode_r against the FP64 form it stands for."""

import os
import shutil
import subprocess

import numpy as np
import pytest

from oracle import rounding as R

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <math.h>
#include <stdio.h>
#include <string.h>
#include <algorithm>
#include <vector>
#include <cuda_runtime.h>
#define __noinline__
using std::max;
using std::min;
template <class T, class U> static T bits(U u) { T t; memcpy(&t, &u, sizeof t); return t; }
static inline double __fma_rn(double a, double b, double c) { return fma(a, b, c); }
static inline float __fmaf_rn(float a, float b, float c) { return fmaf(a, b, c); }
static inline double __dmul_rn(double a, double b) { return a * b; }
static inline double __dadd_rn(double a, double b) { return a + b; }
static inline double __dsub_rn(double a, double b) { return a - b; }
static inline double __ddiv_rn(double a, double b) { return a / b; }
static inline double __drcp_rn(double a) { return 1.0 / a; }
static inline float __fmul_rn(float a, float b) { return a * b; }
static inline float __fadd_rn(float a, float b) { return a + b; }
static inline float __fsub_rn(float a, float b) { return a - b; }
static inline float __fdiv_rn(float a, float b) { return a / b; }
static inline float __frcp_rn(float a) { return 1.0f / a; }
static inline int __float_as_int(float a) { return bits<int>(a); }
static inline unsigned __float_as_uint(float a) { return bits<unsigned>(a); }
static inline float __int_as_float(int a) { return bits<float>(a); }
static inline float __uint_as_float(unsigned a) { return bits<float>(a); }
static inline int __double2hiint(double a) { return (int)(bits<long long>(a) >> 32); }
static inline int atomicOr(int* p, int v) { int o = *p; *p |= v; return o; }
#include "ld_common.cuh"
using namespace ld;
struct In { float x, ref; unsigned k; };
template <int P> void run(const std::vector<In>& in, std::vector<unsigned short>& out) {
    using S = typename Prec<P>::store_t;
    for (const In& v : in) {
        out.push_back(bits<unsigned short, S>(Prec<P>::encode_sr(v.x, v.ref, v.k)));
        out.push_back(bits<unsigned short, S>(Prec<P>::encode_r(v.x, v.ref)));
        out.push_back(bits<unsigned short, S>(Prec<P>::encode_d((double)v.x, v.ref)));
    }
}
int main(int, char** v) {
    std::vector<In> in;
    In one;
    FILE* f = fopen(v[2], "rb");
    while (fread(&one, sizeof one, 1, f) == 1) in.push_back(one);
    fclose(f);
    std::vector<unsigned short> out;
    if (!strcmp(v[1], "fp16")) run<LD_FP16DEV>(in, out); else run<LD_BF16DEV>(in, out);
    f = fopen(v[3], "wb");
    fwrite(out.data(), 2, out.size(), f);
    fclose(f);
}
"""


@pytest.fixture(scope="module")
def encode(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("no CUDA headers")
    out = tmp_path_factory.mktemp("encode")
    (out / "encode.cpp").write_text(PROGRAM)
    inc = [os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include"), os.path.join(ROOT, "include"),
           os.path.join(ROOT, "paper_1609_01479_gb300", "csrc")]
    subprocess.run(["g++", "-std=c++17", "-O1", "-w", "-ffp-contract=off", *(a for i in inc for a in ("-I", i)),
                    str(out / "encode.cpp"), "-o", str(out / "encode")], check=True, capture_output=True, text=True)

    def call(fmt, x, ref, k):
        rec = np.empty(x.size, dtype=[("x", "f4"), ("ref", "f4"), ("k", "u4")])
        rec["x"], rec["ref"], rec["k"] = x.ravel(), np.broadcast_to(ref, x.shape).ravel(), np.broadcast_to(k, x.shape).ravel()
        rec.tofile(out / "in")
        subprocess.run([str(out / "encode"), fmt, str(out / "in"), str(out / "out")], check=True)
        return np.fromfile(out / "out", np.uint16).reshape(-1, 3).T  # encode_sr, encode_r, encode_d

    return call


def every_exponent():
    """Both signs of every exponent (subnormals, infinities and NaN are the first and last) with the mantissas around
    the ends of the formats' cells and some in between."""
    rng = np.random.default_rng(31)
    edge = [0, 1, 0x1FFF, 0x2000, 0x2001, 0x7FFF, 0x8000, 0x8001, 0xFFFF, 0x10000, 0x10001, 0x3FFFFF, 0x400000, 0x7F0000,
            0x7FE000, 0x7FEFFF, 0x7FF000, 0x7FFFFE, 0x7FFFFF]
    m = np.concatenate([np.array(edge), rng.integers(0, 1 << 23, 24)]).astype(np.uint32)
    e = np.arange(256, dtype=np.uint32) << np.uint32(23)
    b = (e[:, None] | m[None, :]).ravel()
    return np.concatenate([b, b | np.uint32(0x80000000)]).view(np.float32)


@pytest.mark.parametrize("fmt", ["fp16", "bf16"])
def test_stochastic_rounding_of_every_exponent(encode, fmt):
    h = every_exponent()
    for k in (0, 1, 0x7FFF, 0x8000, 0xFFFF, None):
        k = np.random.default_rng(32).integers(0, 1 << 16, h.size) if k is None else np.full(h.size, k)
        k = k.astype(np.uint32)
        got, want = encode(fmt, h, np.float32(0), k)[0], R.stochastic_round(h, k, fmt)
        nan = np.isnan(h)
        assert np.array_equal(got[~nan], want[~nan])
        assert np.isnan(R.decode(got[nan], fmt)).all()


@pytest.mark.parametrize("fmt", ["fp16", "bf16"])
def test_initial_rounding_is_the_fp64_one(encode, fmt):
    rng = np.random.default_rng(33)
    x = every_exponent()
    for ref in (np.float32(0), np.float32(-0.0), np.float32(1 / 3), np.float32(1 / 36), np.float32(-0.01)):
        _, r, d = encode(fmt, x, ref, np.uint32(0))
        nan = np.isnan(x)
        assert np.array_equal(r[~nan], d[~nan]) and np.isnan(R.decode(r[nan], fmt)).all()
    # differences that FP32 rounds, many of them next to the middle of a cell
    ref = (rng.choice([1 / 3, 1 / 18, 1 / 36], 400000) * (1 + 0.1 * rng.random(400000))).astype(np.float32)
    x = (ref + rng.integers(-4096, 4096, ref.size) * np.float64(2.0 ** -14) * (1 + 2.0 ** -12 * rng.random(ref.size)))
    _, r, d = encode(fmt, x.astype(np.float32), ref, np.uint32(0))
    assert np.array_equal(r, d)
