"""The node values of a particle are formed at several places of the streaming kernels: unrolled
(recon_all), rolled (recon_all_rolled: the particles counted again, the screen taken in FP64) and one
node at a time (recon_at; recon_stored: the FP64 nodes near a cell edge).  A cell or a screen may be decided by any of them, so they are the same
operations in the same order: bit for bit equal, for every kind of shape in both precisions, over
ordinary coefficients and over ones of which the sums cancel.  The functions are compiled from the
library's header into a program of their own."""
import ctypes
import subprocess

import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

SRC = r"""
#include <random>
#include "pgc_kernels.cuh"
using namespace pgc;

template <int P, int Q, typename R>
__global__ void k_forms(const __grid_constant__ Nodes<P, Q, R> nd, const R *c, R *out, int n)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    R cx[P], cy[P];
#pragma unroll
    for (int h = 0; h < P; ++h) { cx[h] = c[(size_t)h * n + i]; cy[h] = c[(size_t)(P + h) * n + i]; }
    R *o = out + (size_t)i * 8 * Q;
    recon_all(nd, cx, cy, [&](int q, R kx, R ky) { o[q] = kx; o[Q + q] = ky; });
    recon_all_rolled(nd, cx, cy, [&](int q, R kx, R ky) { o[2 * Q + q] = kx; o[3 * Q + q] = ky; });
#pragma unroll 1
    for (int q = 0; q < Q; ++q) {
        recon_at(nd, q, cx, cy, o[4 * Q + q], o[5 * Q + q]);
        if constexpr (sizeof(R) == 8) recon_stored(nd, q, c + i, (int64_t)n, o[6 * Q + q], o[7 * Q + q]);
    }
}

template <int P, int Q, typename R>
static long differ(int n, double spread)
{
    std::mt19937_64 g(P * 100 + Q + sizeof(R));
    std::normal_distribution<double> z;
    Nodes<P, Q, R> nd;
    memset(&nd, 0, sizeof(nd));
    auto pair = [](float f) { uint32_t u; memcpy(&u, &f, 4); return ((unsigned long long)u << 32) | u; };
    for (int j = 0; j < Q * P; ++j) nd.psi[j] = (R)z(g);
    if constexpr (TensorShape<P, Q>::value)
        for (int j = 0; j < 36; ++j) {
            nd.a1[j] = j % 6 ? (R)z(g) : (R)1;
            nd.b2[j] = j % 6 ? (R)z(g) : (R)1;
            nd.a1_2[j] = pair((float)nd.a1[j]);
            nd.b2_2[j] = pair((float)nd.b2[j]);
        }
    if constexpr (TensorShape<P, Q>::value)
        for (int q = 0; q < Q; ++q)
            for (int h2 = 0; h2 < 6; ++h2)
                for (int h1 = 0; h1 + h2 <= 5; ++h1) nd.psi[q * P + hidx2(h1, h2)] = nd.a1[q / 6 * 6 + h1] * nd.b2[q % 6 * 6 + h2];
    if (!TensorShape<P, Q>::value && sizeof(R) == 4)
        for (int j = 0; j < Q * P; ++j) nd.psi2[j] = pair((float)nd.psi[j]);
    std::vector<R> c((size_t)2 * P * n);
    for (R &v : c) v = (R)(z(g) * std::pow(10.0, spread * z(g)));
    std::vector<R> out((size_t)8 * Q * n);
    R *dc = nullptr, *dout = nullptr;
    if (cudaMalloc(&dc, c.size() * sizeof(R)) || cudaMalloc(&dout, out.size() * sizeof(R)) ||
        cudaMemcpy(dc, c.data(), c.size() * sizeof(R), cudaMemcpyHostToDevice)) return -1;
    k_forms<P, Q, R><<<(n + 127) / 128, 128>>>(nd, dc, dout, n);
    if (cudaGetLastError() || cudaMemcpy(out.data(), dout, out.size() * sizeof(R), cudaMemcpyDeviceToHost)) return -1;
    cudaFree(dc);
    cudaFree(dout);
    long bad = 0;
    for (int i = 0; i < n; ++i)
        for (int j = 0; j < 2 * Q; ++j) {
            const R *o = &out[(size_t)i * 8 * Q];
            bad += !(o[j] == o[2 * Q + j]);
            bad += !(o[j] == o[4 * Q + j]);
            if (sizeof(R) == 8) bad += !(o[j] == o[6 * Q + j]);
        }
    return bad;
}

extern "C" long recon_differ(int shape, int fp64, int n, double spread)
{
    switch (shape * 2 + fp64) {
        case 0: return differ<1, 1, float>(n, spread);
        case 1: return differ<1, 1, double>(n, spread);
        case 2: return differ<6, 6, float>(n, spread);
        case 3: return differ<6, 6, double>(n, spread);
        case 4: return differ<13, 13, float>(n, spread);
        case 5: return differ<13, 13, double>(n, spread);
        case 6: return differ<21, 36, float>(n, spread);
        case 7: return differ<21, 36, double>(n, spread);
    }
    return -2;
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    from paper_2404_19602_gb300 import build

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    d = tmp_path_factory.mktemp("recon")
    src, lib = str(d / "recon.cu"), str(d / "recon.so")
    open(src, "w").write(SRC)
    subprocess.run([build._nvcc()] + build.ARCH + build.FLAGS + ["-shared", "-cudart", "shared", "-o", lib, src], check=True)
    so = ctypes.CDLL(lib)
    so.recon_differ.restype = ctypes.c_long
    so.recon_differ.argtypes = [ctypes.c_int, ctypes.c_int, ctypes.c_int, ctypes.c_double]
    return so


@pytest.mark.parametrize("spread", [0.0, 3.0])
@pytest.mark.parametrize("fp64", [0, 1])
@pytest.mark.parametrize("shape", range(4), ids=["1x1", "6x6", "13x13", "21x36"])
def test_node_values_are_the_same_bits(program, shape, fp64, spread):
    assert program.recon_differ(shape, fp64, 1001, spread) == 0
