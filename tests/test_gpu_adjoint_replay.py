"""The adjoint's replay of a step's collision chains against the step itself: for every queued particle
the coefficients after the replayed chain equal the state that the collider kernel left, bit for bit, in
FP64.  In FP32 the replay rounds eps^2 of the selecting rates with its other product fused, so that a
target within a rounding of a mechanism's boundary may replay the neighbour's chain: per event at most
nodes x 6 boundaries x 2^-24 (a rounding of the total rate), and one for chance.  The replay function is
compiled from the library's headers into a program that drives the library's own step."""
import ctypes
import subprocess

import pytest

from paper_2404_19602_gb300 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

SRC = r"""
#include "pgc_adjoint.cuh"
#include "pgc_ctx.h"
using namespace pgc;

template <int P, int Q, typename R>
__global__ void __launch_bounds__(kPhase2Threads)
k_check(const __grid_constant__ AdjArgs<P, Q, R> a, const R *khat, unsigned long long *n)
{
    constexpr int G = GroupOf<Q>::G, NPL = GroupOf<Q>::NPL;
    __shared__ __align__(16) uint32_t sph[(sizeof(Phys<R>) + 3) / 4];
    __shared__ __align__(16) uint32_t snd[(sizeof(Nodes<P, Q, R>) + 3) / 4];
    __shared__ R sred[ProjRed<P, Q, R>::value ? (kPhase2Threads / 32) * ProjRed<P, Q, R>::warp_elems : 1];
    stage(sph, a.ph);
    stage(snd, a.nd);
    __syncthreads();
    const Phys<R> &ph = *reinterpret_cast<const Phys<R> *>(sph);
    const Nodes<P, Q, R> &nd = *reinterpret_cast<const Nodes<P, Q, R> *>(snd);
    const uint32_t count = *a.qcount;
    const int lane = threadIdx.x & 31, r = lane % G;
    const unsigned gmask = (G == 32) ? 0xffffffffu : (((1u << G) - 1u) << (lane - r));
    const QueueShare qs = queue_share<G>(count, blockIdx.x, gridDim.x);
    for (uint32_t j = qs.first; j < count; j += qs.stride) {
        const int64_t i = a.queue[j];
        R cx[P], cy[P], kx[NPL], ky[NPL];
        int nev = 0, lsel[NPL];
        U4 rr{0u, 0u, 0u, 0u};
        replay_events(ph, nd, a, i, j, r, gmask, 1 << 30, cx, cy, kx, ky, &nev, lsel, &rr, sred,
                      [](int, int, R, R, int, const U4 &) {});
        if (r == 0) {
            bool same = true;
#pragma unroll
            for (int h = 0; h < P; ++h)
                same = same && cx[h] == khat[(int64_t)h * a.ld + i] && cy[h] == khat[(int64_t)(P + h) * a.ld + i];
            if (!same) atomicAdd(&n[0], 1ull);
            atomicAdd(&n[1], (unsigned long long)nev);
        }
    }
}

template <int P, int Q, typename R>
static int run_steps(pgc_ctx *ctx, int steps, unsigned long long out[2])
{
    const DevBuffers &b = ctx->b;
    const cudaStream_t s = ctx->stream;
    const size_t hist = (size_t)b.hist_stride * 4, marks = (size_t)b.mark_words * 4, save = (size_t)2 * P * b.ld * sizeof(R);
    char *buf = nullptr;
    auto up = [](size_t v) { return (v + 255) & ~(size_t)255; };
    const size_t total = 2 * up(hist) + up(marks) + up(save) + up((size_t)b.N * 4) + 512;
    if (cudaMalloc(&buf, total) || cudaMemsetAsync(buf, 0, total, s)) return 1;
    uint32_t *H[2] = {(uint32_t *)buf, (uint32_t *)(buf + up(hist))};
    uint32_t *mark = (uint32_t *)(buf + 2 * up(hist));
    R *sv = (R *)((char *)mark + up(marks));
    uint32_t *queue = (uint32_t *)((char *)sv + up(save)), *cnt = (uint32_t *)((char *)queue + up((size_t)b.N * 4));
    unsigned long long *n = (unsigned long long *)(cnt + 64);
    AdjArgs<P, Q, R> a{};
    const auto &fa = static_cast<RunnerT<P, Q, R> *>(ctx->run)->args();
    a.ph = fa.ph;
    a.nd = fa.nd;
    a.khat_n = sv;
    a.compact = 1;
    a.queue = queue;
    a.qcount = cnt;
    a.nmax = b.nmax;
    a.N = b.N;
    a.ld = b.ld;
    a.key0 = b.key0;
    a.key1 = b.key1;
    a.stream_id = b.stream_id;
    cudaError_t e = cudaMemcpyAsync(H[0], b.hist, hist, cudaMemcpyDeviceToDevice, s);   // f^0
    for (int k = 0; k < steps && e == cudaSuccess; ++k) {
        if ((e = cudaMemsetAsync(H[(k + 1) & 1], 0, hist, s)) || (e = cudaMemsetAsync(mark, 0, marks, s))) break;
        if ((e = ctx->run->step_replay(k, H[k & 1], H[(k + 1) & 1], mark, sv, queue, cnt, s))) break;
        a.Hn = H[k & 1];
        a.step = (uint32_t)k;
        k_check<P, Q, R><<<kGrid2, kPhase2Threads, 0, s>>>(a, (const R *)b.state, n);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpyAsync(out, n, 16, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    cudaFree(buf);
    return (int)e;
}

extern "C" int replay_check(pgc_ctx *ctx, int steps, unsigned long long *out)
{
    if (ctx->cfg.precision == PGC_FP32) {
        if (ctx->t.Q == 6) return run_steps<6, 6, float>(ctx, steps, out);
        if (ctx->t.Q == 36) return run_steps<21, 36, float>(ctx, steps, out);
    } else if (ctx->t.Q == 1) return run_steps<1, 1, double>(ctx, steps, out);
    return -1;
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    from paper_2404_19602_gb300 import build

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    lib = build.build()
    d = tmp_path_factory.mktemp("replay")
    src, so = str(d / "replay.cu"), str(d / "replay.so")
    open(src, "w").write(SRC)
    subprocess.run([build._nvcc()] + build.ARCH + build.FLAGS + ["-shared", "-cudart", "shared", "-o", so, src, lib], check=True)
    ctypes.CDLL(lib, mode=ctypes.RTLD_GLOBAL)
    f = ctypes.CDLL(so).replay_check
    f.argtypes = [ctypes.c_void_p, ctypes.c_int, ctypes.POINTER(ctypes.c_ulonglong)]
    return f


@pytest.mark.parametrize("base,N,steps,seed", [(W.GAP_UQ_1E6, 1_000_000, 1500, 3), (W.GAP_FIELD_UQ_4E6, 200_000, 200, 8),
                                               (W.DET_FP64_1E4, 10_000, 200, 1)], ids=["6x6", "21x36", "1x1-fp64"])
def test_replayed_chains_end_in_the_forward_state(program, base, N, steps, seed):
    from paper_2404_19602_gb300 import pgc

    p = W.scaled(base, N=N, seed=seed)
    sim = pgc.Simulation(p, max_outputs=4)
    out = (ctypes.c_ulonglong * 2)()
    assert program(sim.ctx, steps, out) == 0
    print(list(out))
    assert out[1] > N * steps // 1000   # events replayed
    assert out[0] <= (1 + out[1] * sim.Q * 6 * 2.0 ** -24 if p["precision"] == "fp32" else 0)
    sim.close()
