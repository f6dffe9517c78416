"""The two-float transcendental functions (canon_math.cuh) against their
double-precision definitions, bit for bit: softplus and sigmoid for every
float, standardisation for every float under each transform with the
constants of a predictor, and for counts and other constants on a sample
around the values where the evaluation changes its way."""
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

int main(int argc, char **argv) {
    const int op = atoi(argv[1]);
    const float mu = argc > 2 ? (float)atof(argv[2]) : 0.f, sd = argc > 3 ? (float)atof(argv[3]) : 1.f;
    unsigned long long *d, h = 0;
    cudaMalloc(&d, 8);
    cudaMemcpy(d, &h, 8, cudaMemcpyHostToDevice);
    if (op < 10) all<<<152 * 8, 256>>>(op, mu, sd, d);
    else counts<<<152 * 8, 256>>>(op - 10, mu, sd, d);
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
