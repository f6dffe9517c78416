"""The two-float transcendental functions (canon_math.cuh) against their
double-precision definitions, bit for bit: softplus and sigmoid for every
float, standardisation for every float under each transform with the
constants of a predictor, and for counts and other constants (random ones among
them) on a sample around the values where the evaluation changes its way; and
the bound on the quotient's error where it is tightest."""
import importlib
import os
import subprocess

import pytest

B = importlib.import_module("paper_2608_14575_gb300.build")

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))

SRC = r"""
#include <cstdio>
#include <cstdlib>
#include <cuda_runtime.h>
#include "canon_math.cuh"
using namespace hwr;

__device__ bool same(float a, float b) {
    return __float_as_int(a) == __float_as_int(b) || (a != a && b != b);
}

// op 0 softplus, 1 sigmoid, 2..4 standardise code 0..2: all 2^32 floats
__global__ void all(int op, float mu, float sd, unsigned long long *bad) {
    const unsigned long long n = (unsigned long long)gridDim.x * blockDim.x;
    unsigned long long b = 0;
    for (unsigned long long i = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x;
         i < (1ull << 32); i += n) {
        const float x = __int_as_float((int)(unsigned)i);
        bool ok;
        if (op == 0) ok = same(softplus_c(x), softplus_dp(x));
        else if (op == 1) ok = same(sigmoid_c(x), sigmoid_dp(x));
        else ok = same(standardise((uint8_t)(op - 2), x, mu, sd),
                       standardise_dp((uint8_t)(op - 2), x, 0.f, mu, sd));
        b += !ok;
    }
    if (b) atomicAdd(bad, b);
}

// counts 0 .. 2^31 - 1 (all below 2^22, then strided), every transform
__global__ void counts(int code, float mu, float sd, unsigned long long *bad) {
    const long long n = (long long)gridDim.x * blockDim.x;
    unsigned long long b = 0;
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < (1 << 23); k += n) {
        const int i = k < (1 << 22) ? (int)k : (int)((k - (1 << 22)) * 511 + 1);
        const ff c = ff_count(i);
        const double raw = (double)i;
        double t = raw;
        if (code == 1) t = log1p(raw);
        else if (code == 2) t = log(raw);
        const float want = (float)((t - (double)mu) / (double)sd);
        b += !same(standardise((uint8_t)code, c, mu, sd), want);
    }
    if (b) atomicAdd(bad, b);
}

__device__ unsigned long long next(unsigned long long &s) {
    s ^= s << 13;
    s ^= s >> 7;
    s ^= s << 17;
    return s;
}

// random constants of any size and sign, arguments near and far from the mean,
// counts among them
__global__ void random_constants(int code, unsigned long long *bad) {
    unsigned long long s = 88172645463325252ull + 2 * (blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x), b = 0;
    for (int k = 0; k < 20; ++k) next(s);
    for (int k = 0; k < 512; ++k) {
        const unsigned long long u = next(s), v = next(s), w = next(s);
        const float sd = __int_as_float((int)((unsigned)(v & 0x807fffffu) | (unsigned)(97 + (v >> 32) % 60) << 23));
        const float m = __int_as_float((int)((unsigned)(w & 0x007fffffu) | (unsigned)(87 + (w >> 32) % 60) << 23));
        const int i = (int)((u >> 8) & 0x7fffffffu) >> (u & 31);
        const ff c = u & 128 ? ff_count(i) : ff{m * (1.f + (float)((int)(u >> 40) - (1 << 23)) * 0x1p-30f), 0.f};
        const double raw = (double)c.h + (double)c.l;
        double t = raw;
        if (code == 1) t = log1p(raw);
        else if (code == 2) t = log(raw);
        const float mu = u & 64 ? (float)t * (w & (1u << 30) ? 1.f : 1.0001f) : m * (w & (1u << 30) ? 1.f : -1.f);
        b += !same(standardise((uint8_t)code, c, mu, sd), (float)((t - (double)mu) / (double)sd));
    }
    if (b) atomicAdd(bad, b);
}

// what the rounding test needs of the quotient: the two sums it compares lie on
// either side of the value, here for counts past 2^24 whose distance from the
// mean lets the low part reach its limit
__global__ void brackets(unsigned long long *bad) {
    unsigned long long s = 88172645463325252ull + 2 * (blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x), b = 0;
    for (int k = 0; k < 20; ++k) next(s);
    for (int k = 0; k < 4096; ++k) {
        const unsigned long long u = next(s), v = next(s);
        const int i = (1 << 24) + (int)(v % (u & 1 ? 1u << 28 : 0x7effffffu));
        const ff c = ff_count(i);
        if (c.l == 0.f) continue;
        const float d = fabsf(c.l) * 0x1p20f * (1.f + (float)(u >> 54) * 0x1p-12f);
        const float mu = u & 2 ? c.h - d : c.h + d;
        const float sd = __int_as_float(0x3f800000 | (int)((u >> 8) & 0x7fffff));
        float err;
        const ff x = ff_standard(c, 0.f, mu, sd, &err);
        if (fabsf(x.l) > 0x1p-20f * fabsf(x.h)) continue;
        const double want = ((double)i - (double)mu) / (double)sd;
        const float up = x.l + err, dn = x.l - err;
        b += !((double)x.h + (double)up >= want && (double)x.h + (double)dn <= want);
    }
    if (b) atomicAdd(bad, b);
}

int main(int argc, char **argv) {
    const int op = atoi(argv[1]);
    const float mu = argc > 2 ? (float)atof(argv[2]) : 0.f, sd = argc > 3 ? (float)atof(argv[3]) : 1.f;
    unsigned long long *d, h = 0;
    cudaMalloc(&d, 8);
    cudaMemcpy(d, &h, 8, cudaMemcpyHostToDevice);
    if (op < 10) all<<<152 * 8, 256>>>(op, mu, sd, d);
    else if (op < 20) counts<<<152 * 8, 256>>>(op - 10, mu, sd, d);
    else if (op < 30) random_constants<<<152 * 8, 256>>>(op - 20, d);
    else brackets<<<152 * 8, 256>>>(d);
    cudaMemcpy(&h, d, 8, cudaMemcpyDeviceToHost);
    printf("%s %llu\n", cudaGetErrorString(cudaGetLastError()), h);
    return 0;
}
"""


@pytest.fixture(scope="module")
def prog():
    out = os.path.join(HERE, "_build")
    os.makedirs(out, exist_ok=True)
    src, exe = os.path.join(out, "canon_math.cu"), os.path.join(out, "canon_math")
    with open(src, "w") as f:
        f.write(SRC)
    subprocess.run([B._nvcc(), "-O3", "-std=c++17", "--fmad=false", *B.ARCH, "-I", B.CSRC,
                    src, "-o", exe], check=True)
    return exe


def _run(exe, *a):
    r = subprocess.run([exe, *map(str, a)], check=True, capture_output=True, text=True, timeout=120)
    assert r.stdout.strip() == "no error 0", r.stdout


@pytest.mark.parametrize("op", [0, 1])
def test_softplus_and_sigmoid_for_every_float(prog, op):
    _run(prog, op)


# the constants of a length, a time, a count, a utilisation; a large mean, a
# negative and a tiny deviation, no shift at all
CONSTANTS = [(5.5099, 0.99718), (-2.0006, 0.49971), (2.0738, 0.39), (0.4, 0.2), (0.0, 1.0),
             (1000.5, -3.7), (1.0, 1e-7)]


@pytest.mark.parametrize("mu,sd", CONSTANTS)
@pytest.mark.parametrize("code", [0, 1, 2])
def test_standardise_for_every_float_and_count(prog, code, mu, sd):
    _run(prog, 2 + code, mu, sd)
    _run(prog, 10 + code, mu, sd)


@pytest.mark.parametrize("code", [0, 1, 2])
def test_standardise_for_random_constants(prog, code):
    _run(prog, 20 + code)


def test_the_quotient_stays_within_its_bound(prog):
    _run(prog, 30)
