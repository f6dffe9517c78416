// fp32 SIMT kernels of the route-scoring path, in "canonical order".
//
// Canonical order (the fp32 evaluation order this library guarantees, so
// that the same scores come out bit for bit on every run and agree with any
// other implementation that follows the same written order):
//   * feature slot k:  x = (float)((t(raw) - mu[k]) / sd[k]) with the slot
//     transform t (identity, log1p, log) and the arithmetic in double (here
//     and below: canon_math.cuh computes the same rounded values without it);
//   * every dot product starts from its bias (0 for the quality score) and
//     accumulates acc = fma(w[k], x[k], acc) for k ascending, one rounding per
//     step; the two query slots are the last two features, so the
//     deployment-only part of layer 1 is a prefix of the same chain and is
//     computed once per snapshot;
//   * ReLU is (acc > 0 ? acc : 0);
//   * softplus(z) = max(z, 0) + log1p(exp(-|z|)) and sigmoid(s) =
//     1 / (1 + exp(-s)) in double, rounded to float once;
//   * C = fma(N_out, TPOT, TTFT);  U = fma(-lambda, C, w * Qual).
// This file is compiled with --fmad=false so no other contraction happens.
//
// Method (HW-Router Sec. 3.2): feature assembly and the latency predictor
// (Eq. 1), cost (Eq. 2), hardware-independent quality, and the decision maker
// with its SLO constraint (Eq. 3).
#include <cuda_bf16.h>
#include <math.h>

#include "canon_math.cuh"
#include "hwr_internal.cuh"
#include "select.cuh"
#include "umma.cuh"
#include "warp_tile.cuh"

namespace hwr {

// ---------------------------------------------------------------------------
// scalar pieces

// Raw value of deployment feature slot k < F - 2 (layout in hwr.h).
__device__ ff deployment_raw(const Model &m, int d, int k, int32_t running) {
    const int M = m.M, P = m.P;
    if (k < M) return ff{m.dep_model[d] == k ? 1.f : 0.f, 0.f};
    if (k < P) return ff{m.dep_gpu[d] == k - M ? 1.f : 0.f, 0.f};
    if (k == P) return ff{m.log10p[m.dep_model[d]], 0.f};
    if (k == P + 1) return ff_count(running);
    if (k == P + 2) return ff_count(m.waiting[d]);
    if (k == P + 3) return ff{m.kv[d], 0.f};
    if (k == P + 4) return ff{m.gpu_util[d], 0.f};
    if (k == P + 5) return ff{m.ttft[d], 0.f};
    if (k == P + 6) return ff{m.tpot[d], 0.f};
    return ff{0.f, 0.f};
}

__device__ __forceinline__ float emb_at(const void *emb, int bf16, size_t i) {
    if (bf16) {
        uint32_t u = (uint32_t)((const uint16_t *)emb)[i] << 16;
        return __uint_as_float(u);
    }
    return ((const float *)emb)[i];
}

// Quality score (Sec. 3.2, hardware-independent term) of queries
// [q0, q0 + nq): one serial chain per (query, model) from 0 with k ascending,
// then the sigmoid.  The embedding rows (as stored, fp32 or bf16) and the
// model columns are staged through `stage` (at least (nq + M) * 8 + 64
// floats) in chunks of the embedding dimension by 16-byte asynchronous copies
// when the embeddings are 16-byte aligned (plain loads otherwise); the
// chains read shared memory only.  Every thread of the block calls this;
// thread t < nq * M returns the score of query t / M, model t % M (rows at or
// past q.Q give sigmoid(0)), the others return 0.  Ends with the stage free
// for reuse after a barrier.  NT threads take part: the whole block
// (NT = SIMT_THREADS, block barriers, thread index t = threadIdx.x) or one
// warp (NT = 32, warp barriers, t = lane), which then runs the chains
// t, t + 32 (CH = 2: at most 64 (query, model) pairs) and returns the score of
// chain t + 32 j in res[j].
template <int NT>
__device__ __forceinline__ void group_sync() {
    if constexpr (NT == 32) __syncwarp();
    else __syncthreads();
}

template <int NT, int CH>
__device__ void quality_group(const Model &m, const Queries &q, int q0, int nq, float *stage,
                              int stage_floats, int t, float (&res)[CH]) {
    const int tid = t, M = m.M, E = m.E;
    const int es = q.emb_bf16 ? 2 : 4;
    const bool async = !q.inputs_host && ((uintptr_t)q.emb & 15) == 0;
    // row stride ld (elements): 16-byte rows whose 4-byte word stride is 4
    // mod 32, so the chains of one warp (up to 8 rows) read distinct banks
    auto stride = [&](int ek) {
        return es == 4 ? ((ek - 4 + 31) / 32) * 32 + 4 : ((ek - 8 + 63) / 64) * 64 + 8;
    };
    int ek = E;
    while (ek > 8 && ((size_t)nq * stride(ek) * es + 16 + (size_t)ek * M * 4) > 4 * (size_t)stage_floats)
        ek -= 8;
    const int ld = stride(ek);
    char *er = reinterpret_cast<char *>(stage);
    float *mb = reinterpret_cast<float *>(er + (((size_t)nq * ld * es + 15) & ~(size_t)15));
    float s[CH];
#pragma unroll
    for (int j = 0; j < CH; ++j) s[j] = 0.f;
    for (int k0 = 0; k0 < E; k0 += ek) {
        const int kc = min(ek, E - k0);
        group_sync<NT>();
        if (async) {
            const int gpr = kc * es / 16;     // granules per row (kc is a multiple of 8)
            const uint32_t eb = (uint32_t)__cvta_generic_to_shared(er);
            for (int g = tid; g < nq * gpr; g += NT) {
                const int i = g / gpr, c = g - i * gpr, qq = q0 + i;
                const char *src = (const char *)q.emb + ((size_t)(qq < q.Q ? qq : 0) * E + k0) * es + 16 * c;
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(
                                 eb + (uint32_t)(i * ld * es + 16 * c)),
                             "l"(__cvta_generic_to_global(src)), "r"(qq < q.Q ? 16 : 0)
                             : "memory");
            }
            const uint32_t mbs = (uint32_t)__cvta_generic_to_shared(mb);
            for (int g = tid; g < kc * M / 4; g += NT)
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(mbs + 16u * g),
                             "l"(__cvta_generic_to_global(m.memb + (size_t)k0 * M + 4 * g))
                             : "memory");
            asm volatile("cp.async.commit_group;" ::: "memory");
            asm volatile("cp.async.wait_group 0;" ::: "memory");
        } else {
            for (int t = tid; t < nq * kc; t += NT) {
                const int i = t / kc, k = t - i * kc, qq = q0 + i;
                const size_t src = (size_t)(qq < q.Q ? qq : 0) * E + k0 + k;
                if (es == 4) reinterpret_cast<float *>(er)[i * ld + k] = qq < q.Q ? ((const float *)q.emb)[src] : 0.f;
                else reinterpret_cast<uint16_t *>(er)[i * ld + k] = qq < q.Q ? ((const uint16_t *)q.emb)[src] : 0;
            }
            for (int t = tid; t < kc * M; t += NT) mb[t] = m.memb[(size_t)k0 * M + t];
        }
        group_sync<NT>();
#pragma unroll
        for (int j = 0; j < CH; ++j) {
            const int e = tid + NT * j, qi = e / M, mi = e - qi * M;
            if (e < nq * M) {
                const float *b = mb + mi;
                float acc = s[j];
                if (es == 4) {
                    const float *a = reinterpret_cast<const float *>(er) + qi * ld;
#pragma unroll 8
                    for (int k = 0; k < kc; ++k) acc = __fmaf_rn(a[k], b[k * M], acc);
                } else {
                    const uint16_t *a = reinterpret_cast<const uint16_t *>(er) + qi * ld;
#pragma unroll 8
                    for (int k = 0; k < kc; ++k)
                        acc = __fmaf_rn(__uint_as_float((uint32_t)a[k] << 16), b[k * M], acc);
                }
                s[j] = acc;
            }
        }
    }
#pragma unroll
    for (int j = 0; j < CH; ++j) res[j] = tid + NT * j < nq * M ? sigmoid_c(s[j]) : 0.f;
}

__device__ __forceinline__ float quality_staged(const Model &m, const Queries &q, int q0, int nq,
                                                float *stage, int stage_floats) {
    float r[1];
    quality_group<SIMT_THREADS, 1>(m, q, q0, nq, stage, stage_floats, threadIdx.x, r);
    return r[0];
}

// ---------------------------------------------------------------------------
// K_snap: standardised deployment features and the deployment prefix of
// layer 1 (the part of W1 x + b1 that does not depend on the query).

__global__ void __launch_bounds__(SIMT_THREADS) k_snapshot(Model m, const uint32_t *stage) {
    extern __shared__ float xs[];
    const int d = blockIdx.x;
    // this deployment's six signals, from the host's staging ([6][D], mapped)
    // into the context's device arrays (running, waiting, kv, gpu_util, ttft, tpot)
    if (threadIdx.x < 6)
        reinterpret_cast<uint32_t *>(m.running)[(size_t)threadIdx.x * m.D + d] =
            stage[(size_t)threadIdx.x * m.D + d];
    __syncthreads();
    for (int k = threadIdx.x; k < m.F - 2; k += blockDim.x) {
        float x = standardise(m.xform[k], deployment_raw(m, d, k, m.running[d]),
                              m.mu[k], m.sd[k]);
        xs[k] = x;
        m.X[(size_t)d * m.F + k] = x;
    }
    __syncthreads();
    for (int j = threadIdx.x; j < m.H1; j += blockDim.x) {
        const float *w = m.W1T + j;   // slot k at w[k * H1]
        float acc = m.b1[j];
        // slots k0 .. k1 - 1 in order, their weights loaded eight at a time
        // ahead of the FMAs (the loads would otherwise wait one by one)
        auto chain = [&](int k0, int k1) {
            int k = k0;
            for (; k + 8 <= k1; k += 8) {
                float wv[8];
#pragma unroll
                for (int t = 0; t < 8; ++t) wv[t] = w[(size_t)(k + t) * m.H1];
#pragma unroll
                for (int t = 0; t < 8; ++t) acc = __fmaf_rn(wv[t], xs[k + t], acc);
            }
            for (; k < k1; ++k) acc = __fmaf_rn(w[(size_t)k * m.H1], xs[k], acc);
        };
        chain(0, m.P + 1);
        m.Spre[(size_t)d * m.H1 + j] = acc;
        chain(m.P + 1, m.F - 2);
        m.A[(size_t)d * m.H1 + j] = acc;
        m.Abf[(size_t)d * m.H1 + j] = __bfloat16_as_ushort(__float2bfloat16_rn(acc));
    }
}

// ---------------------------------------------------------------------------
// The shared SIMT tile: up to TILE_ROWS rows, each a (query, deployment) pair
// or a sequential-table entry.  For every row it completes layer 1 from a
// deployment prefix and the two query features, runs layer 2 (register-tiled,
// K ascending in chunks of SIMT_KC), layer 3 and the softplus heads.  Output:
// sp[NH r + 0] = TTFT, sp[NH r + 1] = TPOT and, with three heads,
// sp[NH r + 2] = N_out.
//
// Thread map: warp w owns rows 8w .. 8w + 7 and lane l owns columns
// 128 j + VW l + v (v < VW = min(CPT, 4), j < CPT / VW): a lane reads its
// rows' layer-1 values as two 16-byte broadcasts and its W2 columns as
// vectors that are contiguous across the warp.  Shared memory: the layer-1
// chunk [KC][TILE_ROWS] (k-major) and two W2 chunks [KC][32 CPT] (rows of W2
// transposed; the next chunk's cp.async copies run while this one is used),
// then h2 [TILE_ROWS][H2 + 1] in the same space; W3 [NH][H2] in w3s.

constexpr int TILE_ROWS = 64;

// Barrier of the tile's SIMT_THREADS threads only (named barrier 1), so a
// block may run other warps beside the tile.
__device__ __forceinline__ void tile_sync() {
    asm volatile("bar.sync 1, %0;" ::"n"(SIMT_THREADS) : "memory");
}

// n rounded up to a multiple of 4, then to an odd multiple of 4: rows of
// this stride, read by a warp as 16-byte vectors (one row per lane), fall in
// distinct banks across each wavefront's 8 lanes.
__host__ __device__ constexpr int odd_units(int n) {
    return (((n + 3) & ~3) >> 2) & 1 ? (n + 3) & ~3 : ((n + 3) & ~3) + 4;
}

__host__ __device__ constexpr int tile_width(int H2) {
    return H2 <= 32 ? 32 : H2 <= 64 ? 64 : H2 <= 128 ? 128 : 256;
}

__host__ __device__ constexpr size_t tile_floats_for(int H2) {
    return (size_t)SIMT_KC * TILE_ROWS + 2 * (size_t)SIMT_KC * tile_width(H2) >
                   (size_t)TILE_ROWS * odd_units(H2)
               ? (size_t)SIMT_KC * TILE_ROWS + 2 * (size_t)SIMT_KC * tile_width(H2)
               : (size_t)TILE_ROWS * odd_units(H2);
}

// Rows k0 .. k0 + kc - 1 of W2 transposed into dst [kc][W] by 16-byte
// asynchronous copies (W2T rows are H2p floats, 16-byte aligned); one group.
__device__ __forceinline__ void w2_chunk_async(const Model &m, int k0, int kc, float *dst, int W) {
    const int gpr = m.H2p >> 2;
    const uint32_t base = (uint32_t)__cvta_generic_to_shared(dst);
    for (int g = threadIdx.x; g < kc * gpr; g += SIMT_THREADS) {
        const int kk = g / gpr, c4 = g - kk * gpr;
        const float *src = m.W2T + (size_t)(k0 + kk) * m.H2p + 4 * c4;
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                         base + (uint32_t)(4 * (kk * W + 4 * c4))),
                     "l"(__cvta_generic_to_global(src))
                     : "memory");
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
}

// The tile's weights that no row depends on: W3 for the head chains, the two
// query columns of W1 (both visible after the first barrier of the K loop)
// and the first W2 chunk (one cp.async group).  pair_mlp runs this itself
// unless the caller did, e.g. before waiting for a preceding kernel.
template <int CPT>
__device__ void pair_mlp_stage(const Model &m, float *tile, float *w3s, float *w1q) {
    const int tid = threadIdx.x, H1 = m.H1, H2 = m.H2, F = m.F;
    for (int i = tid; i < m.NH * H2; i += SIMT_THREADS) w3s[i] = m.W3[i];
    for (int k = tid; k < H1; k += SIMT_THREADS) {
        w1q[k] = m.W1[(size_t)k * F + F - 2];
        w1q[H1 + k] = m.W1[(size_t)k * F + F - 1];
    }
    w2_chunk_async(m, 0, min(SIMT_KC, H1), tile + SIMT_KC * TILE_ROWS, 32 * CPT);
}

template <int CPT, class Rows>
__device__ void pair_mlp(const Model &m, int R, const Rows &rows, const float *us,
                         const float *vs, float *tile, float *w3s, float *w1q, float *sp,
                         bool staged = false) {
    constexpr int VW = CPT < 4 ? CPT : 4, W = 32 * CPT;
    static_assert(SIMT_THREADS == 4 * TILE_ROWS, "layer-1 map: 4 threads per row");
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int H1 = m.H1, H2 = m.H2;
    float *h1T = tile;
    float *w2b = tile + SIMT_KC * TILE_ROWS;

    if (!staged) pair_mlp_stage<CPT>(m, tile, w3s, w1q);
    // layer-1 map: thread t fills row t % 64 at k offsets t / 64 + 4 j of a chunk
    const int r1 = tid % TILE_ROWS, kq = tid / TILE_ROWS;
    const bool rv = r1 < R;
    const float *pr = rv ? rows.prefix(r1) : m.W1;
    const float uq = rv ? us[rows.query(r1)] : 0.f, vq = rv ? vs[rows.query(r1)] : 0.f;
    tile_sync();
    float acc[8][CPT];
#pragma unroll
    for (int j = 0; j < CPT; ++j) {
        const int n = 128 * (j / VW) + VW * lane + j % VW;
        const float b = n < H2 ? m.b2[n] : 0.f;
#pragma unroll
        for (int i = 0; i < 8; ++i) acc[i][j] = b;
    }
    const bool active = 8 * warp < R;

    for (int k0 = 0, it = 0; k0 < H1; k0 += SIMT_KC, ++it) {
        const int kc = min(SIMT_KC, H1 - k0);
        // layer 1, query suffix: h1 = relu(fma(w_out, v, fma(w_in, u, prefix)));
        // rows at or past R hold 0; a thread's prefix loads are issued together
        float pv[SIMT_KC / 4];
#pragma unroll
        for (int j = 0; j < SIMT_KC / 4; ++j) {
            const int kk = kq + 4 * j;
            pv[j] = rv && kk < kc ? pr[k0 + kk] : 0.f;
        }
#pragma unroll
        for (int j = 0; j < SIMT_KC / 4; ++j) {
            const int kk = kq + 4 * j;
            float a = 0.f;
            if (rv && kk < kc) {
                a = __fmaf_rn(w1q[k0 + kk], uq, pv[j]);
                a = __fmaf_rn(w1q[H1 + k0 + kk], vq, a);
                a = a > 0.f ? a : 0.f;
            }
            h1T[kk * TILE_ROWS + r1] = a;
        }
        // the next W2 chunk goes into the other buffer; this one must be complete
        if (k0 + SIMT_KC < H1) {
            w2_chunk_async(m, k0 + SIMT_KC, min(SIMT_KC, H1 - k0 - SIMT_KC),
                           w2b + ((it + 1) & 1) * SIMT_KC * W, W);
            asm volatile("cp.async.wait_group 1;" ::: "memory");
        } else {
            asm volatile("cp.async.wait_group 0;" ::: "memory");
        }
        tile_sync();
        if (active) {
            const float *wb = w2b + (it & 1) * SIMT_KC * W;
#pragma unroll 4
            for (int kk = 0; kk < kc; ++kk) {
                const float4 a0 = *reinterpret_cast<const float4 *>(h1T + kk * TILE_ROWS + 8 * warp);
                const float4 a1 =
                    *reinterpret_cast<const float4 *>(h1T + kk * TILE_ROWS + 8 * warp + 4);
                const float a[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
                float b[CPT];
                const float *wr = wb + kk * W + VW * lane;
#pragma unroll
                for (int v = 0; v < CPT / VW; ++v) {
                    if constexpr (VW == 4) {
                        const float4 t = *reinterpret_cast<const float4 *>(wr + 128 * v);
                        b[4 * v] = t.x;
                        b[4 * v + 1] = t.y;
                        b[4 * v + 2] = t.z;
                        b[4 * v + 3] = t.w;
                    } else if constexpr (VW == 2) {
                        const float2 t = *reinterpret_cast<const float2 *>(wr);
                        b[0] = t.x;
                        b[1] = t.y;
                    } else {
                        b[0] = wr[0];
                    }
                }
                // rows 2ip and 2ip + 1 in one packed fp32 FMA (fma.rn.f32x2:
                // each lane the same single rounding as __fmaf_rn)
#pragma unroll
                for (int ip = 0; ip < 4; ++ip) {
                    const float2 a2 = make_float2(a[2 * ip], a[2 * ip + 1]);
#pragma unroll
                    for (int j = 0; j < CPT; ++j) {
                        const float2 r = __ffma2_rn(make_float2(b[j], b[j]), a2,
                                                    make_float2(acc[2 * ip][j], acc[2 * ip + 1][j]));
                        acc[2 * ip][j] = r.x;
                        acc[2 * ip + 1][j] = r.y;
                    }
                }
            }
        }
        tile_sync();
    }

    float *h2s = tile;
    const int ld = odd_units(H2);
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int r = 8 * warp + i;
#pragma unroll
        for (int j = 0; j < CPT; ++j) {
            const int n = 128 * (j / VW) + VW * lane + j % VW;
            if (r < R && n < H2) {
                const float v = acc[i][j];
                h2s[r * ld + n] = v > 0.f ? v : 0.f;
            }
        }
    }
    tile_sync();
    for (int e = tid; e < m.NH * R; e += SIMT_THREADS) {
        // head chain o of row r, n ascending: eight n of operands as 16-byte
        // vectors before their FMAs (a chain step waiting on its own shared
        // loads costs several times its FMA)
        const int r = e / m.NH, o = e - r * m.NH;
        const float *w3 = w3s + (size_t)o * H2, *hr = h2s + (size_t)r * ld;
        float z = m.b3[o];
        int n = 0;
        if ((H2 & 3) == 0) {
            for (; n + 8 <= H2; n += 8) {
                const float4 h0 = *reinterpret_cast<const float4 *>(hr + n);
                const float4 h1 = *reinterpret_cast<const float4 *>(hr + n + 4);
                const float4 v0 = *reinterpret_cast<const float4 *>(w3 + n);
                const float4 v1 = *reinterpret_cast<const float4 *>(w3 + n + 4);
                z = __fmaf_rn(v0.x, h0.x, z);
                z = __fmaf_rn(v0.y, h0.y, z);
                z = __fmaf_rn(v0.z, h0.z, z);
                z = __fmaf_rn(v0.w, h0.w, z);
                z = __fmaf_rn(v1.x, h1.x, z);
                z = __fmaf_rn(v1.y, h1.y, z);
                z = __fmaf_rn(v1.z, h1.z, z);
                z = __fmaf_rn(v1.w, h1.w, z);
            }
        }
        for (; n < H2; ++n) z = __fmaf_rn(w3[n], hr[n], z);
        sp[e] = softplus_c(z);
    }
    tile_sync();
}

// ---------------------------------------------------------------------------
// K_route_simt: one block routes QB = 64 / D queries end to end.

struct RouteRows {
    const float *A;
    int D, H1;
    __device__ const float *prefix(int r) const { return A + (size_t)(r % D) * H1; }
    __device__ int query(int r) const { return r / D; }
};

__host__ __device__ inline int route_qb(int D) { return D >= 64 ? 1 : 64 / D; }

constexpr int ROUTE_QSTAGE = 4096;   // floats of the quality warp's staging space

struct RouteLayout {
    int QB, R;
    size_t us, vs, ol, qual, sp, C, U, w3, w1q, qstage, tile, total;  // float offsets
};

__host__ __device__ inline RouteLayout route_layout(int D, int M, int H2) {
    RouteLayout L;
    L.QB = route_qb(D);
    L.R = L.QB * D;
    size_t o = 0;
    L.us = o; o += 64;
    L.vs = o; o += 64;
    L.ol = o; o += 64;
    L.qual = o; o += (size_t)L.QB * M;
    L.sp = o; o += 3 * 64;
    L.C = o; o += 64;
    L.U = o; o += 64;
    o = (o + 3) & ~(size_t)3;   // W3 rows read as 16-byte vectors
    L.w3 = o; o += 3 * (size_t)H2;
    L.w1q = o; o += 2 * (size_t)MAX_H;
    o = (o + 3) & ~(size_t)3;
    L.qstage = o; o += ROUTE_QSTAGE;
    L.tile = o;
    o += tile_floats_for(H2);
    L.total = o;
    return L;
}

// K_route_simt runs the tile on warps 0-7 and the quality chains on warp 8,
// side by side.
constexpr int ROUTE_THREADS = SIMT_THREADS + 32;

template <int CPT>
__global__ void __launch_bounds__(ROUTE_THREADS, CPT <= 4 ? 3 : 2)
k_route_simt(Model m, Queries q, HostFlag flag) {
    extern __shared__ float4 sm4[];
    float *sm = reinterpret_cast<float *>(sm4);
    const RouteLayout L = route_layout(m.D, m.M, m.H2);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int D = m.D, M = m.M, F = m.F, QB = L.QB, R = L.R;
    const int q0 = blockIdx.x * QB;
    float *us = sm + L.us, *vs = sm + L.vs, *ol = sm + L.ol, *qual = sm + L.qual;
    float *sp = sm + L.sp, *Cs = sm + L.C, *Us = sm + L.U;

    if (warp < SIMT_THREADS / 32) {
        // the two query slots on two warps, side by side
        if (tid < QB) {
            const int qq = q0 + tid;
            us[tid] = qq < q.Q ? standardise(m.xform[F - 2], q.in_len[qq], m.mu[F - 2],
                                             m.sd[F - 2])
                               : 0.f;
        } else if (tid >= 64 && tid < 64 + QB) {
            const int qi = tid - 64, qq = q0 + qi;
            const float o = qq < q.Q ? q.out_len[qq] : 0.f;
            vs[qi] = qq < q.Q ? standardise(m.xform[F - 1], o, m.mu[F - 1], m.sd[F - 1])
                              : 0.f;
            ol[qi] = o;
        }
        tile_sync();
        RouteRows rows{m.A, D, m.H1};
        pair_mlp<CPT>(m, R, rows, us, vs, sm + L.tile, sm + L.w3, sm + L.w1q, sp);
    } else {
        // quality (QB M <= 64 chains) on the last warp, while the tile runs
        float qv[2];
        quality_group<32, 2>(m, q, q0, QB, sm + L.qstage, ROUTE_QSTAGE, lane, qv);
        if (lane < QB * M) qual[lane] = qv[0];
        if (lane + 32 < QB * M) qual[lane + 32] = qv[1];
    }
    __syncthreads();

    for (int r = tid; r < R; r += ROUTE_THREADS) {
        const int qi = r / D, d = r - qi * D;
        const float *h = sp + m.NH * r;   // TTFT, TPOT (, N_out)
        const float C = __fmaf_rn(m.NH == 3 ? h[2] : ol[qi], h[1], h[0]);
        const float Ql = qual[qi * M + m.dep_model[d]];
        Cs[r] = C;
        Us[r] = __fmaf_rn(-q.lam, C, __fmul_rn(q.wq, Ql));
        if (q.pair_C && q0 + qi < q.Q) q.pair_C[(size_t)(q0 + qi) * D + d] = C;
    }
    if (q.qual_out)
        for (int e = tid; e < QB * M; e += ROUTE_THREADS)
            if (q0 + e / M < q.Q) q.qual_out[(size_t)q0 * M + e] = qual[e];
    __syncthreads();

    for (int qi = warp; qi < QB; qi += ROUTE_THREADS / 32) {
        const int qq = q0 + qi;
        if (qq >= q.Q) continue;
        Cand best = no_cand();
        const float slo = query_budget(q, qq);
        for (int d = lane; d < D; d += 32) {
            Cand c = make_cand(Cs[qi * D + d], Us[qi * D + d], d, slo);
            if (better(c, best)) best = c;
        }
        best = warp_best(best);
        if (lane == 0) {
            const bool ok = best.cls > 0;
            q.chosen[qq] = ok ? best.d : -1;
            q.lat[qq] = ok ? best.C : __int_as_float(0x7fc00000);
            q.util[qq] = ok ? best.U : __int_as_float(0x7fc00000);
        }
    }
    if (flag.word) {
        __syncthreads();
        if (tid == 0) flag_block_done(flag);
    }
}

// ---------------------------------------------------------------------------
// K_route_rows: the fp32 kernel of large batches.  A block (one an SM) takes
// an equal run of the batch's queries, in blocks of QBK (32, or 16 for more
// than 32 deployments).  NW warps score their pairs in groups of RG rows with
// the warp tile; NQ warps hold one query per lane and, a block of queries
// ahead of the tile, run its quality chains, then wait for the block's costs
// and decide.  The costs pass through a ring of NB blocks in shared memory
// (done, an mbarrier: the groups' arrivals; freed, a count: the decisions), so
// the two sides meet only when one is a whole ring ahead.
// Bound: the FMA pipe; measured 43.1 TFLOP/s at 100,000 queries, D = 12,
// H = 128 (54 % of 80.5; k_route_simt 31), where a k step's 64 packed FMAs
// come with about 50 other instructions (the pairs of a W2 value with itself,
// loads) and fill the issue slots.

constexpr int QUAL_KC = 32;      // embedding elements per staged chunk
constexpr int QUAL_MC = 16;      // model columns per staged chunk

// Shape of the batch kernel by the width W of the layer-2 tile: rows per
// group (lane tiles of 8 x 8, 8 x 4, 8 x 2 values), and 16 warps in all, so
// that each thread can hold 128 registers.  Groups of 8 rows at W <= 128 read
// more shared memory per FMA (1,048 against 969 us for 100,000 queries at
// D = 12, H = 128), 16 at W = 256 need 16 x 8 lane tiles.
template <int W>
struct RouteShape {
    static constexpr int RG = W == 256 ? 8 : 16;                 // rows per group
    static constexpr int NQ = W <= 64 ? 4 : 2;                   // deciding warps
    static constexpr int NW = 16 - NQ;                           // scoring warps
    static constexpr int NB = NQ + 2;                            // query blocks in flight
    static constexpr int NS = W <= 64 ? 8 : W == 128 ? 4 : 3;    // W2 stages at most
    static constexpr int QST = 3;                                // embedding stages per deciding warp
    static constexpr int THREADS = 32 * (NW + NQ);
};

constexpr size_t ROWS_SMEM = 227 * 1024;

struct RowsLayout {
    int qbk, cld, rowb, ns, nch;                     // query block, cost stride, embedding row bytes
    size_t w2, bufs, ri, w1q, b2, w3, b3, cost, qst, qual, dms, bars, pre, total;   // bytes
    bool pre_sm;                                     // the deployment prefixes in shared memory too
    size_t qst_bytes;                                // one embedding stage
};

template <int W>
__host__ __device__ inline RowsLayout rows_layout(int D, int M, int NH, int H1, int H2p, int es) {
    using S = RouteShape<W>;
    constexpr int RG = S::RG;
    RowsLayout L;
    L.qbk = D > 32 ? 16 : 32;
    L.cld = D | 1;
    L.rowb = QUAL_KC * es + 16;                      // an odd number of 16-byte units
    L.nch = (H1 + TILE_KC - 1) / TILE_KC;
    L.ns = L.nch < S::NS ? L.nch : S::NS;
    L.qst_bytes = (size_t)L.qbk * L.rowb + (QUAL_KC + 1) * QUAL_MC * 4;
    size_t o = 0;
    auto take = [&o](size_t bytes) {
        const size_t at = o;
        o += (bytes + 15) & ~(size_t)15;
        return at;
    };
    L.bufs = take((size_t)S::NW * Tile<W, RG>::BUF * 4);
    L.ri = take((size_t)S::NW * RG * sizeof(RowInfo));
    L.w1q = take(2 * (size_t)H1 * 4);
    L.b2 = take(W * 4);
    L.w3 = take((size_t)NH * H2p * 4);
    L.b3 = take(16);
    L.cost = take((size_t)S::NB * L.qbk * L.cld * 4);
    L.qst = take((size_t)S::NQ * S::QST * L.qst_bytes);
    L.qual = take((size_t)S::NQ * L.qbk * (M | 1) * 4);
    L.dms = take((size_t)D * 4);
    L.bars = take((S::NS + S::NB) * 8 + (S::NB + S::NS + 2) * 4);
    // W2 stages: as many as fit, all of it if possible (and slack: the widest
    // lane reads past a row that ends before W)
    const size_t stage = (size_t)TILE_KC * H2p * 4;
    while (L.ns > 2 && o + L.ns * stage + W * 4 > ROWS_SMEM) --L.ns;
    L.w2 = take(L.ns * stage + W * 4);
    // the deployment prefixes where they fit: they are read once per row and
    // 32 k (from global memory, a third of a group's time outside layer 2)
    L.pre = o;
    L.pre_sm = o + (size_t)D * H1 * 4 <= ROWS_SMEM;
    if (L.pre_sm) take((size_t)D * H1 * 4);
    L.total = o;
    return L;
}

// One staged chunk of the quality chains of a query (row: its embedding,
// mb: 4 NG of the staged model columns, rows of ms floats): KS elements'
// operands at a time ahead of their FMAs.
template <int NG>
__device__ __forceinline__ void qual_chunk(const char *row, const float *mb, int ms, int kc, bool bf,
                                           float (&acc)[QUAL_MC]) {
    constexpr int KS = NG == 1 ? 8 : 4;
#pragma unroll 1
    for (int k = 0; k < kc; k += KS) {      // kc is a multiple of 8
        float e[KS];
        float4 b[KS][NG];
        if (bf) {
#pragma unroll
            for (int i = 0; i < KS; i += 4) {
                const uint2 t = *reinterpret_cast<const uint2 *>(row + 2 * (k + i));
                e[i] = __uint_as_float(t.x << 16);
                e[i + 1] = __uint_as_float(t.x & 0xffff0000u);
                e[i + 2] = __uint_as_float(t.y << 16);
                e[i + 3] = __uint_as_float(t.y & 0xffff0000u);
            }
        } else {
#pragma unroll
            for (int i = 0; i < KS; i += 4) {
                const float4 t = *reinterpret_cast<const float4 *>(row + 4 * (k + i));
                e[i] = t.x;
                e[i + 1] = t.y;
                e[i + 2] = t.z;
                e[i + 3] = t.w;
            }
        }
#pragma unroll
        for (int i = 0; i < KS; ++i)
#pragma unroll
            for (int g = 0; g < NG; ++g)
                b[i][g] = *reinterpret_cast<const float4 *>(mb + (k + i) * ms + 4 * g);
#pragma unroll
        for (int i = 0; i < KS; ++i)
#pragma unroll
            for (int g = 0; g < NG; ++g) {
                acc[4 * g] = __fmaf_rn(e[i], b[i][g].x, acc[4 * g]);
                acc[4 * g + 1] = __fmaf_rn(e[i], b[i][g].y, acc[4 * g + 1]);
                acc[4 * g + 2] = __fmaf_rn(e[i], b[i][g].z, acc[4 * g + 2]);
                acc[4 * g + 3] = __fmaf_rn(e[i], b[i][g].w, acc[4 * g + 3]);
            }
    }
}

// A cost slot's count of decisions: its deciding warps say that the n-th use is
// over; the others wait for it.  A count and not an mbarrier's phase: with few
// deployments a pass of the scoring warps spans more blocks than the ring has,
// a warp then comes to a slot that it has not seen for two uses, and the
// parity of the phase before last reads like that of the last one.
__device__ __forceinline__ void slot_free(uint32_t *freed, uint32_t n) {
    asm volatile("st.release.cta.shared.u32 [%0], %1;" ::"r"(umma::smem_u32(freed)), "r"(n) : "memory");
}

__device__ __forceinline__ bool slot_wait(const uint32_t *freed, uint32_t n, volatile int *abort_f,
                                          int32_t *status) {
    const uint32_t a = umma::smem_u32(freed);
    const long long t0 = clock64();
    while (true) {
        uint32_t v;
        asm volatile("ld.acquire.cta.shared.u32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
        if (v >= n) return true;
        if (*abort_f) return false;
        if (clock64() - t0 > umma::WAIT_CYCLES) {
            *abort_f = 1;
            *(volatile int32_t *)status = ST_TIMEOUT;
            __threadfence_system();
            return false;
        }
        __nanosleep(64);
    }
}

template <int W>
__global__ void __launch_bounds__(RouteShape<W>::THREADS, 1)
k_route_rows(Model m, Queries q, int32_t *status) {
    using S = RouteShape<W>;
    constexpr int RG = S::RG, NW = S::NW, NQ = S::NQ, NB = S::NB, QST = S::QST;
    extern __shared__ float4 sm4[];
    char *sm = reinterpret_cast<char *>(sm4);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int D = m.D, M = m.M, F = m.F, H1 = m.H1, E = m.E;
    const int es = q.emb_bf16 ? 2 : 4;
    const RowsLayout L = rows_layout<W>(D, M, m.NH, H1, m.H2p, es);
    const int QBK = L.qbk;
    // this block's queries, their blocks, and the groups of a whole block
    const int qa = (int)((long long)blockIdx.x * q.Q / gridDim.x);
    const int qb = (int)((long long)(blockIdx.x + 1) * q.Q / gridDim.x);
    const int nblk = (qb - qa + QBK - 1) / QBK;
    const int G = (QBK * D + RG - 1) / RG;
    const int last_groups = nblk ? ((qb - qa - (nblk - 1) * QBK) * D + RG - 1) / RG : 0;
    const int ngroups = nblk ? (nblk - 1) * G + last_groups : 0;
    const int passes = (ngroups + NW - 1) / NW;

    uint64_t *full = reinterpret_cast<uint64_t *>(sm + L.bars), *done = full + S::NS;
    uint32_t *freed = reinterpret_cast<uint32_t *>(done + NB), *used = freed + NB;
    volatile int *abort_f = reinterpret_cast<volatile int *>(used + S::NS);
    W2Feed f;
    f.w2t = m.W2T;
    f.sm = reinterpret_cast<float *>(sm + L.w2);
    f.full = full;
    f.used = used;
    f.issued = used + S::NS + 1;
    f.abort_f = abort_f;
    f.status = status;
    f.H1 = H1;
    f.ldw = m.H2p;
    f.ns = L.ns;
    f.nch = L.nch;
    f.warps = NW;
    f.total = (uint32_t)passes * L.nch;
    if (tid == 0) {
        for (int s = 0; s < S::NS; ++s) {
            umma::mbar_init(&full[s], 1);
            used[s] = 0;
        }
        for (int b = 0; b < NB; ++b) {
            umma::mbar_init(&done[b], G);
            freed[b] = 0;
        }
        *abort_f = 0;
        umma::fence_mbar_init();
        w2_start(f);
    }
    TileWeights w;
    uint32_t prefix_s = 0;
    {
        float *w1q = reinterpret_cast<float *>(sm + L.w1q), *b2 = reinterpret_cast<float *>(sm + L.b2);
        float *w3 = reinterpret_cast<float *>(sm + L.w3), *b3 = reinterpret_cast<float *>(sm + L.b3);
        int *dms = reinterpret_cast<int *>(sm + L.dms);
        for (int k = tid; k < 2 * H1; k += S::THREADS) w1q[k] = m.W1T[(size_t)(F - 2) * H1 + k];
        for (int n = tid; n < W; n += S::THREADS) b2[n] = n < m.H2 ? m.b2[n] : 0.f;
        for (int i = tid; i < m.NH * m.H2; i += S::THREADS) {
            const int o = i / m.H2;
            w3[o * m.H2p + i - o * m.H2] = m.W3[i];
        }
        if (tid < m.NH) b3[tid] = m.b3[tid];
        for (int d = tid; d < D; d += S::THREADS) dms[d] = m.dep_model[d];
        if (L.pre_sm) {
            float *pre = reinterpret_cast<float *>(sm + L.pre);
            for (int i = tid; i < D * H1; i += S::THREADS) pre[i] = m.A[i];
            prefix_s = umma::smem_u32(pre);
        }
        w.w1q = w1q;
        w.b2 = b2;
        w.w3 = w3;
        w.b3 = b3;
    }
    __syncthreads();
    float *costs = reinterpret_cast<float *>(sm + L.cost);

    if (warp < NW) {
        // ---- scoring warps --------------------------------------------------
        float *buf = reinterpret_cast<float *>(sm + L.bufs) + (size_t)warp * Tile<W, RG>::BUF;
        RowInfo *ri = reinterpret_cast<RowInfo *>(sm + L.ri) + RG * warp;
        // lane l standardises slot l / RG (input, then output length) of row l % RG
        const int r = lane % RG, slot_k = lane / RG == 1 ? F - 1 : F - 2;
        const uint8_t xf = m.xform[slot_k];
        const float mu = m.mu[slot_k], sd = m.sd[slot_k];
        const float *lens = lane / RG == 1 ? q.out_len : q.in_len;
        // row p of group g: its query and deployment (qq = -1 past the end)
        auto row_of = [&](int g, int &qq, int &ql, int &d) {
            const int blk = g / G, p = (g - blk * G) * RG + r;
            ql = p / D;
            d = p - ql * D;
            qq = qa + blk * QBK + ql;
            if (g >= ngroups || ql >= QBK || qq >= qb) qq = -1;
        };
        // the next group's lengths are loaded a group ahead
        int qq, ql, d;
        row_of(warp, qq, ql, d);
        float len = qq < 0 ? 0.f : lens[qq];
        for (int ps = 0, g = warp; ps < passes; ++ps, g += NW) {
            const uint32_t n0 = (uint32_t)ps * (uint32_t)L.nch;
            if (g >= ngroups) {
                if (!w2_skip(f, n0)) break;
                continue;
            }
            {
                const float x = standardise(xf, len, mu, sd);
                const float v = __shfl_down_sync(0xffffffffu, x, RG),
                            ol = __shfl_down_sync(0xffffffffu, len, RG);
                if (lane < RG) ri[lane] = RowInfo{x, v, qq < 0 ? 0 : d * H1, ol};
            }
            const int cq = qq, cql = ql, cd = d;
            row_of(g + NW, qq, ql, d);
            len = qq < 0 ? 0.f : lens[qq];
            __syncwarp();
            float C;
            if (!warp_tile<W, RG>(m, f, w, n0, ri, m.A, prefix_s, buf, C)) break;
            // the block's slot is free once the decisions NB blocks back are out
            const int blk = g / G, slot = blk % NB;
            if (blk >= NB) {
                const bool ok = slot_wait(&freed[slot], (uint32_t)(blk / NB), abort_f, status);
                if (!__all_sync(0xffffffffu, ok)) break;
            }
            if (lane < RG && cq >= 0) {
                costs[(size_t)slot * QBK * L.cld + cql * L.cld + cd] = C;
                if (q.pair_C) q.pair_C[(size_t)cq * D + cd] = C;
            }
            __syncwarp();
            if (lane == 0) umma::mbar_arrive(&done[slot]);
        }
    } else {
        // ---- deciding warps -------------------------------------------------
        const int qw = warp - NW;
        char *stages = sm + L.qst + (size_t)qw * QST * L.qst_bytes;
        float *qs = reinterpret_cast<float *>(sm + L.qual) + (size_t)qw * QBK * (M | 1);
        const int *dms = reinterpret_cast<const int *>(sm + L.dms);
        const bool async = !q.inputs_host && ((uintptr_t)q.emb & 15) == 0;
        const int ql = lane & (QBK - 1), nhalf = 32 / QBK, half = lane / QBK;
        const int nck = (E + QUAL_KC - 1) / QUAL_KC, npass = (M + QUAL_MC - 1) / QUAL_MC;
        const int myblk = nblk > qw ? (nblk - qw + NQ - 1) / NQ : 0;
        const uint32_t stage_s = umma::smem_u32(stages);
        // The next chunk (block nb, model pass np, k chunk nc, in order) into
        // stage t % QST: the block's embedding rows and the pass's model columns;
        // one cp.async group (empty past the last).  A lane copies granule ec of
        // every er_step-th row.  Model columns: whole rows of M floats where M is
        // at most 16 and a multiple of 4 (contiguous), else padded to 16.
        const int gpr = QUAL_KC * es / 16, ec = lane & (gpr - 1), er0 = lane / gpr, er_step = 32 / gpr;
        const bool mrow = M <= QUAL_MC && (M & 3) == 0;
        const int ms = mrow ? M : QUAL_MC;
        int nb = 0, np = 0, nc = 0;
        auto issue = [&](int t) {
            if (nb < myblk) {
                const int k0 = nc * QUAL_KC, kc = min(QUAL_KC, E - k0), bq0 = qa + (qw + nb * NQ) * QBK;
                const int nq = min(QBK, qb - bq0), m0 = np * QUAL_MC, mn = min(QUAL_MC, M - m0);
                const size_t so = (size_t)(t % QST) * L.qst_bytes;
                char *er = stages + so;
                if (async) {
                    if (ec * 16 < kc * es) {
                        const char *src = (const char *)q.emb + ((size_t)(bq0 + er0) * E + k0) * es + 16 * ec;
                        uint32_t dst = stage_s + (uint32_t)(so + (size_t)er0 * L.rowb + 16 * ec);
                        for (int i = er0; i < nq; i += er_step) {
                            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst),
                                         "l"(__cvta_generic_to_global(src)) : "memory");
                            src += (size_t)er_step * E * es;
                            dst += (uint32_t)(er_step * L.rowb);
                        }
                    }
                } else {
                    for (int e = lane; e < nq * kc; e += 32) {
                        const int i = e / kc, k = e - i * kc;
                        const size_t src = (size_t)(bq0 + i) * E + k0 + k;
                        if (es == 4) reinterpret_cast<float *>(er + (size_t)i * L.rowb)[k] = ((const float *)q.emb)[src];
                        else reinterpret_cast<uint16_t *>(er + (size_t)i * L.rowb)[k] = ((const uint16_t *)q.emb)[src];
                    }
                }
                const uint32_t mbs = stage_s + (uint32_t)(so + (size_t)QBK * L.rowb);
                const float *mg = m.memb + (size_t)k0 * M + m0;
                if (mrow) {
                    for (int g = lane; g < kc * M / 4; g += 32)
                        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(mbs + 16u * g),
                                     "l"(__cvta_generic_to_global(mg + 4 * g)) : "memory");
                } else {
                    for (int g = lane; g < kc * QUAL_MC; g += 32) {
                        const int k = g / QUAL_MC, c = g % QUAL_MC;
                        if (c < mn)
                            asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(mbs + 4u * g),
                                         "l"(__cvta_generic_to_global(mg + (size_t)k * M + c)) : "memory");
                    }
                }
                if (++nc == nck) {
                    nc = 0;
                    if (++np == npass) {
                        np = 0;
                        ++nb;
                    }
                }
            }
            asm volatile("cp.async.commit_group;" ::: "memory");
        };
        for (int t = 0; t < QST - 1; ++t) issue(t);
        float acc[QUAL_MC];
        int t = 0;
        bool ok = true;
        for (int bi = 0; ok && bi < myblk; ++bi) {
            const int blk = qw + bi * NQ, slot = blk % NB, bq0 = qa + blk * QBK, nq = min(QBK, qb - bq0);
            const int qq = bq0 + ql;
            const bool valid = ql < nq;
            for (int ps = 0; ps < npass; ++ps) {
                const int m0 = ps * QUAL_MC, mn = min(QUAL_MC, M - m0);
                const int ng = (mn + 4 * nhalf - 1) / (4 * nhalf);      // 4 model columns each
                const int col = half * 4 * ng;
#pragma unroll
                for (int j = 0; j < QUAL_MC; ++j) acc[j] = 0.f;
                for (int c = 0; c < nck; ++c, ++t) {
                    asm volatile("cp.async.wait_group %0;" ::"n"(QST - 2) : "memory");
                    __syncwarp();
                    issue(t + QST - 1);
                    const int kc = min(QUAL_KC, E - c * QUAL_KC);
                    const char *er = stages + (size_t)(t % QST) * L.qst_bytes;
                    const float *mb = reinterpret_cast<const float *>(er + (size_t)QBK * L.rowb) + col;
                    const char *row = er + (size_t)ql * L.rowb;
                    if (ng == 1) qual_chunk<1>(row, mb, ms, kc, es == 2, acc);
                    else if (ng == 2) qual_chunk<2>(row, mb, ms, kc, es == 2, acc);
                    else qual_chunk<4>(row, mb, ms, kc, es == 2, acc);
                }
#pragma unroll
                for (int j = 0; j < QUAL_MC; ++j)
                    if (j < 4 * ng && col + j < mn) {
                        const float s = sigmoid_c(valid ? acc[j] : 0.f);
                        qs[ql * (M | 1) + m0 + col + j] = s;
                        if (q.qual_out && valid) q.qual_out[(size_t)qq * M + m0 + col + j] = s;
                    }
            }
            __syncwarp();
            // The slot is this block's once the block NB before it is decided; that
            // one may be another deciding warp's and still wait for its groups, and
            // `done` would then be a phase behind, whose parity reads as complete.
            if (blk >= NB) {
                ok = slot_wait(&freed[slot], (uint32_t)(blk / NB), abort_f, status);
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) break;
            }
            // the groups that the last block does not have arrive from here
            if (blk == nblk - 1 && last_groups < G) {
                if (lane == 0)
                    for (int g = last_groups; g < G; ++g) umma::mbar_arrive(&done[slot]);
                __syncwarp();
            }
            ok = umma::mbar_wait(&done[slot], (blk / NB) & 1, abort_f, status);
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
            // the decision: each lane its query's deployments in order (with 16
            // queries: half of them), then the better half
            const float slo = valid ? query_budget(q, qq) : 0.f;
            const float *cr = costs + (size_t)slot * QBK * L.cld + ql * L.cld;
            const float *qr = qs + ql * (M | 1);
            Cand best = no_cand();
            if (valid) {
                const int d0 = half * D / nhalf, d1 = (half + 1) * D / nhalf;
                for (int d = d0; d < d1; ++d) {
                    const float C = cr[d], U = __fmaf_rn(-q.lam, C, __fmul_rn(q.wq, qr[dms[d]]));
                    const Cand c = make_cand(C, U, d, slo);
                    if (better(c, best)) best = c;
                }
            }
            if (nhalf == 2) {
                Cand o;
                o.cls = __shfl_xor_sync(0xffffffffu, best.cls, 16);
                o.d = __shfl_xor_sync(0xffffffffu, best.d, 16);
                o.C = __shfl_xor_sync(0xffffffffu, best.C, 16);
                o.U = __shfl_xor_sync(0xffffffffu, best.U, 16);
                if (better(o, best)) best = o;
            }
            __syncwarp();
            if (lane == 0) slot_free(&freed[slot], (uint32_t)(blk / NB) + 1u);
            if (valid && half == 0) {
                const bool sel = best.cls > 0;
                q.chosen[qq] = sel ? best.d : -1;
                q.lat[qq] = sel ? best.C : __int_as_float(0x7fc00000);
                q.util[qq] = sel ? best.U : __int_as_float(0x7fc00000);
            }
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
    }
    __syncthreads();
    if (tid == 0) w2_drain(f);
}

// ---------------------------------------------------------------------------
// Sequential mode.  Query i of a chunk is scored with running count r_d + c_d
// where c_d counts the chunk's earlier picks of d, c_d <= i.  K_seq_table
// scores every (c, d, i) with c <= i in parallel; K_seq_chain then walks the
// chunk in order reading the table entry of the current c_d.
//
// Table layout (triangular): for c in [0, Qs), d in [0, D), i in [c, Qs):
//   index = D * (c * Qs - c (c - 1) / 2) + d * (Qs - c) + (i - c).
// A table block takes an equal run of consecutive entries.

size_t seq_table_floats(int D, int Qs) { return tri_off(D, Qs, Qs); }

// Auxiliary arrays (one scratch buffer, seq_aux_floats floats) of a run of
// chunks, Ns queries in all: a chunk's quality [<= SEQ_MAX_CHUNK][M], the
// queries' standardised slots u [Ns] and v [Ns], and, for every deployment d
// and count c = 0 .. Ns of picks since the run began, the standardised running
// count xr [D][Ns + 1] and the layer-1 prefix through slot F - 3
// pre [D][Ns + 1][H1] (the snapshot kernel's chain with running rbase[d] + c,
// rbase [D] the running counts as the run began).
struct SeqAux {
    float *qual, *us, *vs, *xr;
    int32_t *rbase;
    float *pre;
};

__host__ __device__ inline SeqAux seq_aux(float *aux, int D, int M, int Ns) {
    SeqAux a;
    a.qual = aux;
    a.us = aux + (size_t)SEQ_MAX_CHUNK * M;
    a.vs = a.us + Ns;
    a.xr = a.vs + Ns;
    a.rbase = reinterpret_cast<int32_t *>(a.xr + (size_t)D * (Ns + 1));
    a.pre = aux + (((size_t)SEQ_MAX_CHUNK * M + 2 * (size_t)Ns + (size_t)D * (Ns + 2) + 3) & ~(size_t)3);
    return a;
}

size_t seq_aux_floats(int D, int M, int H1, int Ns) {
    return (((size_t)SEQ_MAX_CHUNK * M + 2 * (size_t)Ns + (size_t)D * (Ns + 2) + 3) & ~(size_t)3) +
           (size_t)D * (Ns + 1) * H1;
}

// K_seq_prep: a run's standardised features and layer-1 prefixes, each
// computed once (every table block would otherwise repeat it).  Blocks [0, nuv): the query slots; then
// one block per deployment d and run of PREP_COUNTS counts c.
constexpr int PREP_THREADS = 128;
constexpr int PREP_COUNTS = 8;   // counts c per preparation block
__host__ __device__ inline int seq_prep_blocks_per_dep(int Qs) {
    return (Qs + PREP_COUNTS) / PREP_COUNTS;   // counts 0 .. Qs
}

__global__ void __launch_bounds__(PREP_THREADS)
k_seq_prep(Model m, Queries q, int Qs, float *aux, uint16_t *pre_bf, int32_t *dmv) {
    // launched as a programmatic dependent of the kernel before (the snapshot
    // kernel, or the chain of the chunk before): only the launch itself overlaps
    // that kernel; nothing is read or written, and this kernel's own dependents
    // don't start, before it has finished.  A 64-request micro-batch through
    // host buffers: 59.8 -> 57.2 us; a backlog's chunks: no change.
    umma::grid_dependency_wait();
    umma::grid_launch_dependents();
    const SeqAux a = seq_aux(aux, m.D, m.M, Qs);
    const int tid = threadIdx.x, F = m.F, P = m.P, H1 = m.H1;
    const int nuv = (2 * Qs + PREP_THREADS - 1) / PREP_THREADS;
    if ((int)blockIdx.x < nuv) {
        const int t = blockIdx.x * PREP_THREADS + tid;
        if (t < Qs) {
            a.us[t] = standardise(m.xform[F - 2], q.in_len[t], m.mu[F - 2], m.sd[F - 2]);
        } else if (t < 2 * Qs) {
            const int i = t - Qs;
            a.vs[i] = standardise(m.xform[F - 1], q.out_len[i], m.mu[F - 1], m.sd[F - 1]);
        }
        return;
    }
    // block: deployment d, counts c0 .. c0 + cn - 1
    const int nc = seq_prep_blocks_per_dep(Qs);
    const int gb = blockIdx.x - nuv, d = gb / nc, c0 = (gb - d * nc) * PREP_COUNTS;
    const int cn = Qs + 1 - c0 < PREP_COUNTS ? Qs + 1 - c0 : PREP_COUNTS;
    const int g0 = d * (Qs + 1) + c0;
    __shared__ float xr[PREP_COUNTS];
    if (tid < cn) {
        const float v = standardise(m.xform[P + 1], ff_count(m.running[d] + c0 + tid), m.mu[P + 1],
                                    m.sd[P + 1]);
        xr[tid] = v;
        a.xr[g0 + tid] = v;
        if (c0 + tid == 0) a.rbase[d] = m.running[d];
        if (dmv) dmv[g0 + tid] = m.dep_model[d];
    } else if (tid < PREP_COUNTS) {
        xr[tid] = 0.f;   // past the last count: computed, never stored
    }
    __syncthreads();
    // continue the chain from slot P + 1 (running) with the deployment's other
    // features, every count of the block at once (W1 read slot-major: a warp's
    // loads of one slot are contiguous)
    const float *x = m.X + (size_t)d * F;
    for (int j = tid; j < H1; j += PREP_THREADS) {
        const float s0 = m.Spre[(size_t)d * H1 + j], w = m.W1T[(size_t)(P + 1) * H1 + j];
        float acc[PREP_COUNTS];
#pragma unroll
        for (int c = 0; c < PREP_COUNTS; ++c) acc[c] = __fmaf_rn(w, xr[c], s0);
        // the remaining slots in order, their weights and features loaded
        // eight at a time ahead of the FMAs
        int k = P + 2;
        for (; k + 8 <= F - 2; k += 8) {
            float wv[8], xv[8];
#pragma unroll
            for (int t = 0; t < 8; ++t) {
                wv[t] = m.W1T[(size_t)(k + t) * H1 + j];
                xv[t] = x[k + t];
            }
#pragma unroll
            for (int t = 0; t < 8; ++t)
#pragma unroll
                for (int c = 0; c < PREP_COUNTS; ++c) acc[c] = __fmaf_rn(wv[t], xv[t], acc[c]);
        }
        for (; k < F - 2; ++k) {
            const float wk = m.W1T[(size_t)k * H1 + j], xk = x[k];
#pragma unroll
            for (int c = 0; c < PREP_COUNTS; ++c) acc[c] = __fmaf_rn(wk, xk, acc[c]);
        }
#pragma unroll
        for (int c = 0; c < PREP_COUNTS; ++c) {
            if (c < cn) {
                a.pre[(size_t)(g0 + c) * H1 + j] = acc[c];
                if (pre_bf)
                    pre_bf[(size_t)(g0 + c) * H1 + j] = __bfloat16_as_ushort(__float2bfloat16_rn(acc[c]));
            }
        }
    }
}

// Table rows of one block: row r is table entry t0 + r, i.e. (c, d, i) with
// prefix pre[d][c] and query slot i (decoded into shared memory).
struct FlatRows {
    const float *pre;
    const int *gi, *qi;
    int H1;
    __device__ const float *prefix(int r) const { return pre + (size_t)gi[r] * H1; }
    __device__ int query(int r) const { return qi[r]; }
};

struct SeqLayout {
    size_t us, vs, gi, qi, di, sp, w3, w1q, tile, total;
};

__host__ __device__ inline SeqLayout seq_layout(int H2) {
    SeqLayout L;
    size_t o = 0;
    L.us = o; o += SEQ_MAX_CHUNK;
    L.vs = o; o += SEQ_MAX_CHUNK;
    L.gi = o; o += TILE_ROWS;
    L.qi = o; o += TILE_ROWS;
    L.di = o; o += TILE_ROWS;
    L.sp = o; o += 3 * TILE_ROWS;
    o = (o + 3) & ~(size_t)3;   // W3 rows read as 16-byte vectors
    L.w3 = o; o += 3 * (size_t)H2;
    L.w1q = o; o += 2 * (size_t)MAX_H;
    o = (o + 3) & ~(size_t)3;
    L.tile = o;
    o += tile_floats_for(H2);
    L.total = o;
    return L;
}

// Queries per quality block of the sequential table (at most 256 chains).
__host__ __device__ inline int seq_qual_rows(int M) {
    const int n = SIMT_THREADS / M;
    return n < 1 ? 1 : (n > 8 ? 8 : n);
}

// K_seq_table: blocks [0, nb_qual) compute the chunk's quality; the others
// take rows_per_block consecutive table entries each (the last block fewer),
// so that every SM gets the same number of rows.
template <int CPT>
__global__ void __launch_bounds__(SIMT_THREADS, CPT <= 4 ? 3 : 2)
k_seq_table(Model m, Queries q, int Qs, int Ns, int off0, int nb_qual, int rows_per_block,
            float *ctab, float *aux) {
    extern __shared__ float4 sm4[];
    float *sm = reinterpret_cast<float *>(sm4);
    const int tid = threadIdx.x;
    const int D = m.D, M = m.M;
    const SeqLayout L = seq_layout(m.H2);
    const SeqAux A = seq_aux(aux, D, M, Ns);
    // launched as a programmatic dependent of the preparation kernel, or of the
    // chain of the chunk before: the chain may be scheduled now; nothing that
    // those kernels write is read, and nothing they read is written, before
    // this grid has waited for them
    umma::grid_launch_dependents();
    if ((int)blockIdx.x < nb_qual) {
        // quality of the chunk's queries [q0, q0 + nq), staged through the whole
        // shared space
        const int nq = seq_qual_rows(M), q0 = (int)blockIdx.x * nq;
        const float v = quality_staged(m, q, q0, nq, sm, (int)L.total);
        umma::grid_dependency_wait();
        if (tid < nq * M && q0 + tid / M < Qs) A.qual[(size_t)q0 * M + tid] = v;
        return;
    }
    const int T = (int)tri_off(D, Qs, Qs);
    const int t0 = ((int)blockIdx.x - nb_qual) * rows_per_block;
    const int R = min(rows_per_block, T - t0);
    float *us = sm + L.us, *vs = sm + L.vs, *sp = sm + L.sp;
    int *gi = reinterpret_cast<int *>(sm + L.gi), *qi = reinterpret_cast<int *>(sm + L.qi);
    int *di = reinterpret_cast<int *>(sm + L.di);
    for (int r = tid; r < R; r += SIMT_THREADS) {
        // entry t: the count c with tri_off(c) <= t < tri_off(c + 1), then d and i
        const int t = t0 + r;
        int lo = 0, hi = Qs - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if ((int)tri_off(D, Qs, mid) <= t) lo = mid;
            else hi = mid - 1;
        }
        const int off = t - (int)tri_off(D, Qs, lo), len = Qs - lo, d = off / len;
        gi[r] = d * (Ns + 1) + lo;
        di[r] = d;
        qi[r] = lo + off - d * len;
    }
    // the weights need nothing from the preparation kernel
    pair_mlp_stage<CPT>(m, sm + L.tile, sm + L.w3, sm + L.w1q);
    umma::grid_dependency_wait();    // the run's features and prefixes, the picks so far
    for (int i = tid; i < Qs; i += SIMT_THREADS) {
        us[i] = A.us[off0 + i];
        vs[i] = A.vs[off0 + i];
    }
    // counts are of the run: the deployment's picks in the chunks before count too
    for (int r = tid; r < R; r += SIMT_THREADS)
        gi[r] += __ldcg(m.running + di[r]) - __ldcg(A.rbase + di[r]);
    __syncthreads();

    FlatRows rows{A.pre, gi, qi, m.H1};
    pair_mlp<CPT>(m, R, rows, us, vs, sm + L.tile, sm + L.w3, sm + L.w1q, sp, true);

    for (int r = tid; r < R; r += SIMT_THREADS) {
        const float *h = sp + m.NH * r;
        ctab[t0 + r] = __fmaf_rn(m.NH == 3 ? h[2] : q.out_len[qi[r]], h[1], h[0]);
    }
}

// Chain shared memory (4-byte words): dep_model and picks per deployment
// [MAX_D] ints each, the walk's picks [SEQ_MAX_CHUNK], the table [T rounded up
// to 4] (16-byte aligned), the chunk's quality [Qs][M] and budgets [Qs].
constexpr int CHAIN_THREADS = 1024;

__host__ __device__ inline size_t chain_tab_floats(int D, int Qs) {
    return (tri_off(D, Qs, Qs) + 3) & ~(size_t)3;
}

// Largest value over a full warp (NaN lanes do not count).
__device__ __forceinline__ float warp_max(float x) {
    float r;
    asm volatile("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(r) : "f"(x));
    return r;
}

// HI: deployments 32 .. 63 exist (D > 32); without them every lane of the
// walk carries one deployment and the second half of the step is compiled out.
// BIG: only the table's first `tsm` entries (the rows of the first counts)
// fit in shared memory; the walk reads the rest from global memory (L2).
template <bool HI, bool BIG>
__global__ void __launch_bounds__(CHAIN_THREADS)
k_seq_chain(Model m, Queries q, int Qs, int Ns, const float *ctab, float *aux, const float *qsrc,
            int qstride, int tsm, int more) {
    extern __shared__ float4 sm4[];
    float *sm = reinterpret_cast<float *>(sm4);
    const int tid = threadIdx.x, lane = tid & 31;
    const int D = m.D, M = m.M, F = m.F, H1 = m.H1, P = m.P;
    const SeqAux A = seq_aux(aux, D, M, Ns);
    const size_t T = tri_off(D, Qs, Qs);
    int *dm = reinterpret_cast<int *>(sm), *cnt = dm + MAX_D, *o_ch = cnt + MAX_D;
    float *tab = sm + 2 * MAX_D + SEQ_MAX_CHUNK;
    float *qs = tab + (BIG ? (size_t)tsm : chain_tab_floats(D, Qs)), *slo = qs + (size_t)Qs * M;
    const size_t Ts = BIG ? (size_t)tsm : T;    // entries staged in shared memory
    // entry e of the table: shared memory, or (BIG, e >= tsm) global memory
    auto at = [&](int e) -> float {
        if constexpr (BIG) {
            return e < tsm ? tab[e] : __ldcg(ctab + (e < (int)T ? e : (int)T - 1));
        } else {
            return tab[e];
        }
    };

    // launched as a programmatic dependent of the table kernel: budgets and
    // the model map first, then wait for the table (and, through it, for the
    // preparation kernel)
    // the call's next chunk may be launched now (its table, or the preparation
    // of a further run of chunks: both wait for this grid before they touch
    // what it uses); after the last chunk anything may follow, the tensor-core
    // route among them, whose predictor reads the prefixes that this kernel
    // persists without waiting for more than the kernel before it
    if (more) umma::grid_launch_dependents();
    for (int i = tid; i < Qs; i += CHAIN_THREADS) slo[i] = query_budget(q, i);
    for (int e = tid; e < D; e += CHAIN_THREADS) dm[e] = m.dep_model[e];
    umma::grid_dependency_wait();
    const uint32_t tab_s = (uint32_t)__cvta_generic_to_shared(tab);
    // the triangular table, by 16-byte asynchronous copies (both sides
    // 16-byte aligned)
    for (size_t e = tid; e < Ts / 4; e += CHAIN_THREADS)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(tab_s + (uint32_t)(16 * e)),
                     "l"(__cvta_generic_to_global(ctab + 4 * e))
                     : "memory");
    for (size_t e = Ts / 4 * 4 + tid; e < Ts; e += CHAIN_THREADS) tab[e] = __ldcg(ctab + e);
    asm volatile("cp.async.commit_group;" ::: "memory");
    for (int e = tid; e < Qs * M; e += CHAIN_THREADS) {
        const int i = e / M;
        qs[e] = __ldcg(qsrc + (size_t)i * qstride + e - i * M);
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();

    if (tid < 32) {
        // The walk.  Lane l holds deployments d0 = l and d1 = l + 32; entry
        // (c, d, i) is tab[tab_row(c, d) + i], c the deployment's picks so far.
        // While step i is decided, step i + 1's entries at the current count
        // and at one more pick are loaded and made candidates, so a step is two
        // float maxima over the warp (the feasible utilities; the costs, for a
        // step without a feasible deployment), one vote, the lowest lane that
        // holds the maximum, and a choice between two ready candidates.  It is
        // one chain of dependent instructions, and each one on it counts: no
        // find-first-set (a lane asks its lane mask), no store, no branch; only
        // the picks are kept (lane i % 32 keeps step i's), the outputs follow
        // from them below.  A step takes ~145 cycles at D = 12 and ~255 at
        // D = 32 with part of the table in L2; with 40-bit integer keys, stores
        // and branches 260 and 411, the walk of a 64-request chunk 8.0 -> 4.5 us.
        // Exact while the costs met and the weights are ordinary numbers: then a
        // utility is finite, and the maximum is -inf only if nothing is
        // feasible.  Otherwise the walk runs again the long way.
        // Lanes without a deployment shadow deployment D - 1 (valid addresses)
        // and are no candidates.  The last step loads a column past the end: the
        // row after, or the value behind the table (both unused).
        const unsigned full = 0xffffffffu, below = (1u << lane) - 1u;
        const float ninf = __int_as_float(0xff800000), pinf = __int_as_float(0x7f800000);
        const int d0 = lane, d1 = lane + 32;
        const bool h0 = d0 < D, h1 = HI && d1 < D;
        const int e0 = h0 ? d0 : D - 1, e1 = h1 ? d1 : D - 1;
        const int m0 = dm[e0], m1 = HI ? dm[e1] : 0;
        const float lam = q.lam, wq = q.wq;
        // a candidate: minus its cost, and its utility if feasible (a NaN there
        // is never the maximum)
        struct Entry {
            float n, v;
        };
        auto entry = [&](float C, float wQ, float b, bool h) -> Entry {
            return Entry{h ? -C : ninf, h && C <= b ? __fmaf_rn(-lam, C, wQ) : ninf};
        };
        // next column's entry at this count and at one more; the latter's row
        // moves on by s = D (Qs - c) - d - 1 with each pick
        int a0, a1, s0, s1, a0p, a1p;
        const float *qn0, *qn1;
        Entry E0, E1;
        auto start = [&]() {
            a0 = tab_row(D, Qs, 0, e0);
            a1 = HI ? tab_row(D, Qs, 0, e1) : 0;
            s0 = D * Qs - e0 - 1;
            s1 = D * Qs - e1 - 1;
            E0 = entry(at(a0), __fmul_rn(wq, qs[m0]), slo[0], h0);
            E1 = E0;
            if (HI) E1 = entry(at(a1), __fmul_rn(wq, qs[m1]), slo[0], h1);
            ++a0;
            ++a1;
            a0p = a0 + s0;
            a1p = a1 + s1;
            qn0 = qs + m0;
            qn1 = qs + m1;
        };
        // one step's state from its decision
        auto advance = [&](bool p, const Entry &es, const Entry &ep, Entry &e, int &ac, int &ap, int &st) {
            e.n = p ? ep.n : es.n;
            e.v = p ? ep.v : es.v;
            st -= p ? D : 0;
            ac = (p ? ap : ac) + 1;
            ap += (p ? st : 0) + 1;
        };
        bool odd = !(fabsf(lam) <= 1e6f && fabsf(wq) <= 1e6f);
        // steps lo .. hi - 1 (at most 32); lane i % 32 keeps step i's votes
        auto steps = [&](int lo, int hi, uint32_t &rec0, uint32_t &rec1) {
#pragma unroll 2
            for (int i = lo; i < hi; ++i) {
                const bool next = i + 1 < Qs;
                const float b = slo[next ? i + 1 : i];
                qn0 += next ? M : 0;
                const float q0 = *qn0, x0s = at(a0), x0p = at(a0p);
                float q1 = 0.f, x1s = 0.f, x1p = 0.f;
                if (HI) {
                    qn1 += next ? M : 0;
                    q1 = *qn1;
                    x1s = at(a1);
                    x1p = at(a1p);
                }
                const float mx = warp_max(HI ? fmaxf(E0.v, E1.v) : E0.v);
                const float mn = warp_max(HI ? fmaxf(E0.n, E1.n) : E0.n);
                const bool feas = mx > ninf;
                const bool k0 = feas ? E0.v == mx : E0.n == mn;
                const bool k1 = HI && (feas ? E1.v == mx : E1.n == mn);
                const unsigned w0 = __ballot_sync(full, k0), w1 = HI ? __ballot_sync(full, k1) : 0u;
                const bool p0 = k0 && (w0 & below) == 0u, p1 = HI && k1 && (w0 | (w1 & below)) == 0u;
                odd = odd || (h0 && !(fabsf(E0.n) <= 1e30f)) || (h1 && !(fabsf(E1.n) <= 1e30f));
                rec0 = lane == (i & 31) ? w0 : rec0;
                if (HI) rec1 = lane == (i & 31) ? w1 : rec1;
                const float wQ0 = __fmul_rn(wq, q0);
                advance(p0, entry(x0s, wQ0, b, h0), entry(x0p, wQ0, b, h0), E0, a0, a0p, s0);
                if (HI) {
                    const float wQ1 = __fmul_rn(wq, q1);
                    advance(p1, entry(x1s, wQ1, b, h1), entry(x1p, wQ1, b, h1), E1, a1, a1p, s1);
                }
            }
        };
        start();
        uint32_t ra0 = 0u, ra1 = 0u, rb0 = 0u, rb1 = 0u;
        steps(0, min(Qs, 32), ra0, ra1);
        steps(32, Qs, rb0, rb1);
        if (lane < Qs) o_ch[lane] = ra0 ? __ffs(ra0) - 1 : 31 + __ffs(ra1);
        if (lane + 32 < Qs) o_ch[lane + 32] = rb0 ? __ffs(rb0) - 1 : 31 + __ffs(rb1);
        if (__any_sync(full, odd)) {
            __syncwarp();
            start();
#pragma unroll 1
            for (int i = 0; i < Qs; ++i) {
                const bool next = i + 1 < Qs;
                const float b = slo[next ? i + 1 : i], bi = slo[i];
                qn0 += next ? M : 0;
                qn1 += HI && next ? M : 0;
                const float x0s = at(a0), x0p = at(a0p), x1s = HI ? at(a1) : 0.f, x1p = HI ? at(a1p) : 0.f;
                // the classes in turn: feasible with a defined utility (-inf among
                // them), any defined cost, none
                const float C0 = -E0.n, C1 = -E1.n;
                const bool f0 = h0 && C0 <= bi && E0.v == E0.v, f1 = h1 && C1 <= bi && E1.v == E1.v;
                const float mx = warp_max(HI ? fmaxf(f0 ? E0.v : ninf, f1 ? E1.v : ninf) : f0 ? E0.v : ninf);
                bool k0 = f0 && E0.v == mx, k1 = f1 && E1.v == mx;
                unsigned w0 = __ballot_sync(full, k0), w1 = __ballot_sync(full, k1);
                if ((w0 | w1) == 0u) {
                    const bool n0 = h0 && C0 == C0, n1 = h1 && C1 == C1;
                    const float mn = warp_max(fmaxf(n0 ? E0.n : ninf, n1 ? E1.n : ninf));
                    k0 = n0 && E0.n == mn;
                    k1 = n1 && E1.n == mn;
                    w0 = __ballot_sync(full, k0);
                    w1 = __ballot_sync(full, k1);
                }
                if (lane == 0) o_ch[i] = w0 ? __ffs(w0) - 1 : w1 ? 31 + __ffs(w1) : -1;
                const bool p0 = k0 && (w0 & below) == 0u, p1 = k1 && (w0 | (w1 & below)) == 0u;
                const float wQ0 = __fmul_rn(wq, *qn0);
                advance(p0, entry(x0s, wQ0, b, h0), entry(x0p, wQ0, b, h0), E0, a0, a0p, s0);
                if (HI) {
                    const float wQ1 = __fmul_rn(wq, *qn1);
                    advance(p1, entry(x1s, wQ1, b, h1), entry(x1p, wQ1, b, h1), E1, a1, a1p, s1);
                }
            }
        }
    }
    __syncthreads();
    // The outputs of step i: its pick's count is the number of earlier steps
    // that picked the same deployment.  Sixteen threads a step (and as many a
    // deployment, for its picks in all) look at four picks each.
    static_assert(CHAIN_THREADS == 16 * SEQ_MAX_CHUNK && MAX_D == SEQ_MAX_CHUNK, "sixteen threads a step");
    {
        const int i = tid / 16, j0 = 4 * (tid % 16);
        const int4 v = *reinterpret_cast<const int4 *>(o_ch + j0);   // (past the picks: never counted)
        const int pick[4] = {v.x, v.y, v.z, v.w};
        const int d = i < Qs ? o_ch[i] : -1;
        int c = 0, all = 0;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            c += pick[k] == d && j0 + k < i ? 1 : 0;
            all += pick[k] == i && j0 + k < Qs ? 1 : 0;      // this group's deployment is i too
        }
#pragma unroll
        for (int s = 8; s; s >>= 1) {
            c += __shfl_xor_sync(0xffffffffu, c, s);
            all += __shfl_xor_sync(0xffffffffu, all, s);
        }
        if (tid % 16 == 0) {
            cnt[i] = all;
            if (i < Qs) {
                float C = __int_as_float(0x7fc00000), U = C;
                if (d >= 0) {
                    C = at(tab_row(D, Qs, c, d) + i);
                    U = __fmaf_rn(-q.lam, C, __fmul_rn(q.wq, qs[i * M + dm[d]]));
                }
                q.lat[i] = C;
                q.util[i] = U;
                if (q.inputs_host) {
                    // outputs in host memory: the host may poll chosen with
                    // acquire loads, so it is stored last, with release
                    // semantics at system scope
                    asm volatile("st.release.sys.global.b32 [%0], %1;" ::"l"(q.chosen + i), "r"(d)
                                 : "memory");
                } else {
                    q.chosen[i] = d;
                }
            }
        }
    }
    __syncthreads();

    // persist the picks and, after the call's last chunk, the state they touch:
    // the standardised running count and the layer-1 prefix are the preparation
    // kernel's values for the final count
    if (tid < D) {
        const int r = m.running[tid] + cnt[tid];
        m.running[tid] = r;
        cnt[tid] = tid * (Ns + 1) + r - A.rbase[tid];
        if (!more) m.X[(size_t)tid * F + P + 1] = A.xr[cnt[tid]];
    }
    if (more) return;
    __syncthreads();
    for (int e = tid; e < D * H1; e += CHAIN_THREADS) {
        const int d = e / H1, j = e - d * H1;
        const float v = A.pre[(size_t)cnt[d] * H1 + j];
        m.A[e] = v;
        m.Abf[e] = __bfloat16_as_ushort(__float2bfloat16_rn(v));
    }
}

// ---------------------------------------------------------------------------
// K_route_pairs: the small-batch (latency) variant.  The (query, deployment)
// pairs p = qq D + d are taken in groups of PAIR_G consecutive pairs, and a
// group's layer 2 is split by columns over ncb column blocks, in one of two
// shapes.  Split (PAIR_COLS columns per block, when groups are many): each
// block stages its W2 columns k-major and the group's layer-1 rows in shared
// memory, runs its columns' serial chains (warp w: columns 4w .. 4w + 3,
// lane: pair, so a W2 load is a broadcast) and stores them to a scratch h2
// [groups][H2][PAIR_G].  Fused (PAIR_FUSED_COLS columns per block, when every
// block of the grid has an SM of its own, e.g. one query): each block stages
// its W2 rows, the pairs' deployment prefixes and W1's query columns, and
// rebuilds every layer-1 unit inside the layer-2 chains (warp w: columns 2w,
// 2w + 1), storing h2 rows [groups][PAIR_G][H2].  The last column block of a
// group (arrival counter, self-resetting) copies the group's h2 back with
// 16-byte async copies and runs the head chains and the cost of Eq. 2.
// Quality blocks run the per-(query, model) chains from shared memory.  A
// query is decided by the block that completes its count of D pairs and
// qblocks quality blocks (self-resetting).  Same canonical order as the
// kernels above in both shapes: every chain is the same sequence of roundings.

struct PairArgs {
    float *pairC;       // [Q][D] scratch
    float *qualS;       // [Q][M] scratch
    float *h2;          // [groups][H2][PAIR_G] scratch
    int32_t *count;     // [Q] arrivals, zero between calls
    int32_t *gcount;    // [groups] column-block arrivals, zero between calls
    int qblocks;        // quality blocks per query
    int ncb;            // column blocks per group
    int cols;           // layer-2 columns per column block: PAIR_FUSED_COLS or PAIR_COLS
};

constexpr int PAIR_MPB = 8;    // models per quality block
constexpr int PAIR_G = 32;     // pairs per group
constexpr int PAIR_COLS = 32;  // layer-2 columns per block, split shape
constexpr int PAIR_FUSED_COLS = 8;   // layer-2 columns per block, fused shape

__device__ void pair_select(const Model &m, const Queries &q, const PairArgs &a, int qq) {
    // one warp: utility, SLO mask, argmax over the query's stored costs
    const int lane = threadIdx.x & 31;
    Cand best = no_cand();
    const float slo = query_budget(q, qq);
    for (int d = lane; d < m.D; d += 32) {
        const float C = __ldcg(&a.pairC[(size_t)qq * m.D + d]);
        const float Ql = __ldcg(&a.qualS[(size_t)qq * m.M + m.dep_model[d]]);
        const float U = __fmaf_rn(-q.lam, C, __fmul_rn(q.wq, Ql));
        Cand c = make_cand(C, U, d, slo);
        if (better(c, best)) best = c;
    }
    best = warp_best(best);
    if (lane == 0) {
        const bool ok = best.cls > 0;
        q.lat[qq] = ok ? best.C : __int_as_float(0x7fc00000);
        q.util[qq] = ok ? best.U : __int_as_float(0x7fc00000);
        a.count[qq] = 0;
        const int32_t v = ok ? best.d : -1;
        if (q.inputs_host) {
            // outputs in mapped host memory: the host polls chosen with
            // acquire loads, so chosen is stored with release semantics at
            // system scope, after latency and utility
            asm volatile("st.release.sys.global.b32 [%0], %1;" ::"l"(q.chosen + qq), "r"(v)
                         : "memory");
        } else {
            q.chosen[qq] = v;
        }
    }
}

__host__ __device__ inline int pair_groups(int npair) { return (npair + PAIR_G - 1) / PAIR_G; }

// Shared-memory layout of a fused-shape column block (floats; every region
// 16-byte aligned), and of the group's last block over the same space.  Rows
// that a warp reads as 16-byte vectors, one row per lane, have a stride of an
// odd number of 16-byte units, so that the 8 lanes of each wavefront fall in
// distinct banks.
struct PairSmem {
    int ldk, lda, ld2;          // W2 / W1-column row stride; prefix and layer-2 row strides
    int w2, as, w1;             // column block: W2 rows, prefix rows, W1's query columns
    int h2, w3;                 // last block: layer-2 rows, W3
    int total;
};

__host__ __device__ inline PairSmem pair_smem(int H1, int H2) {
    PairSmem L;
    L.ldk = (H1 + 3) & ~3;
    L.lda = (H1 & 3) == 0 ? odd_units(H1) : H1;
    L.ld2 = odd_units(H2);
    int o = 3 * PAIR_G;                     // qu, qv, qo
    L.w2 = o;
    o += PAIR_FUSED_COLS * L.ldk;
    L.as = o;
    o += (PAIR_G * L.lda + 3) & ~3;
    L.w1 = o;
    o += 2 * L.ldk;
    L.h2 = 3 * PAIR_G;
    L.w3 = L.h2 + PAIR_G * L.ld2;
    const int fin = L.w3 + 3 * H2;
    L.total = o > fin ? o : fin;
    return L;
}

// Layers 1 and 2 of pair p (deployment prefix row ar, query slots u, v) for
// the block's columns c0, c0 + 1: each layer-1 unit is rebuilt where
// layer 2 consumes it (same two FMAs and ReLU as everywhere), and each
// layer-2 chain is bias, then k ascending.  Shared-memory operands come as
// 16-byte vectors, eight k at a time ahead of their FMAs: on this GPU a
// chain step waiting on its own shared loads costs several times its FMA.
// Stores relu(h2) into the group's scratch rows [PAIR_G][H2].
__device__ __forceinline__ void pair_layers(const Model &m, const PairArgs &a, const PairSmem &L,
                                            const float *w2c, const float *ar, const float *w1s,
                                            float u, float v, int g, int n0, int nb, int c0,
                                            int p) {
    constexpr int NC = 2;
    const int H1 = m.H1, H2 = m.H2;
    float acc[NC];
    const float *wr[NC];
#pragma unroll
    for (int j = 0; j < NC; ++j) {
        const int c = c0 + j;
        acc[j] = c < nb ? m.b2[n0 + c] : 0.f;
        wr[j] = w2c + (size_t)(c < nb ? c : 0) * L.ldk;
    }
    const float *wi = w1s, *wo = w1s + L.ldk;
    int k = 0;
    if ((H1 & 3) == 0) {
        for (; k + 8 <= H1; k += 8) {
            const float4 a0 = *reinterpret_cast<const float4 *>(ar + k);
            const float4 a1 = *reinterpret_cast<const float4 *>(ar + k + 4);
            const float4 i0 = *reinterpret_cast<const float4 *>(wi + k);
            const float4 i1 = *reinterpret_cast<const float4 *>(wi + k + 4);
            const float4 o0 = *reinterpret_cast<const float4 *>(wo + k);
            const float4 o1 = *reinterpret_cast<const float4 *>(wo + k + 4);
            float4 w0[NC], w1[NC];
#pragma unroll
            for (int j = 0; j < NC; ++j) {
                w0[j] = *reinterpret_cast<const float4 *>(wr[j] + k);
                w1[j] = *reinterpret_cast<const float4 *>(wr[j] + k + 4);
            }
            const float av[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
            const float iv[8] = {i0.x, i0.y, i0.z, i0.w, i1.x, i1.y, i1.z, i1.w};
            const float ov[8] = {o0.x, o0.y, o0.z, o0.w, o1.x, o1.y, o1.z, o1.w};
            float h[8];
#pragma unroll
            for (int t = 0; t < 8; ++t) {
                const float x = __fmaf_rn(ov[t], v, __fmaf_rn(iv[t], u, av[t]));
                h[t] = x > 0.f ? x : 0.f;
            }
#pragma unroll
            for (int j = 0; j < NC; ++j) {
                acc[j] = __fmaf_rn(w0[j].x, h[0], acc[j]);
                acc[j] = __fmaf_rn(w0[j].y, h[1], acc[j]);
                acc[j] = __fmaf_rn(w0[j].z, h[2], acc[j]);
                acc[j] = __fmaf_rn(w0[j].w, h[3], acc[j]);
                acc[j] = __fmaf_rn(w1[j].x, h[4], acc[j]);
                acc[j] = __fmaf_rn(w1[j].y, h[5], acc[j]);
                acc[j] = __fmaf_rn(w1[j].z, h[6], acc[j]);
                acc[j] = __fmaf_rn(w1[j].w, h[7], acc[j]);
            }
        }
    }
    for (; k < H1; ++k) {
        const float x = __fmaf_rn(wo[k], v, __fmaf_rn(wi[k], u, ar[k]));
        const float h = x > 0.f ? x : 0.f;
#pragma unroll
        for (int j = 0; j < NC; ++j) acc[j] = __fmaf_rn(wr[j][k], h, acc[j]);
    }
    float *dst = a.h2 + ((size_t)g * PAIR_G + p) * H2 + n0;
#pragma unroll
    for (int j = 0; j < NC; ++j)
        if (c0 + j < nb) dst[c0 + j] = acc[j] > 0.f ? acc[j] : 0.f;
    __threadfence();   // before the group's arrival
}

// The decision for each query of a group: its pairs arrive; the warp that
// completes the query's count (pairs and quality blocks) decides it.
__device__ __forceinline__ void pair_decide(const Model &m, const Queries &q, const PairArgs &a,
                                            int p0, int np, int q0, int nq) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, D = m.D;
    for (int ql = warp; ql < nq; ql += SIMT_THREADS / 32) {
        const int qq = q0 + ql;
        const int cnt = min(p0 + np, (qq + 1) * D) - max(p0, qq * D);
        int done = 0;
        if (lane == 0) done = atomicAdd(&a.count[qq], cnt) + cnt == D + a.qblocks;
        done = __shfl_sync(0xffffffffu, done, 0);
        if (done) {
            __threadfence();
            pair_select(m, q, a, qq);
        }
    }
}

// Column block, split shape (many groups): W2 columns n0 .. n0 + 31 k-major,
// layer 1 written once per (pair, unit), layer-2 chains of 4 columns per warp
// (lane = pair), h2 scratch [groups][H2][PAIR_G]; the group's last column
// block runs the heads.
__device__ __forceinline__ void pair_cols_split(const Model &m, const Queries &q, const PairArgs &a,
                                             float *sm, int *s_last_p) {
    int &s_last = *s_last_p;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int F = m.F, H1 = m.H1, H2 = m.H2, D = m.D;
    const int npair = q.Q * D;
    const int g = blockIdx.x / a.ncb, cb = blockIdx.x - g * a.ncb;
    const int p0 = g * PAIR_G, np = min(PAIR_G, npair - p0);
    const int q0 = p0 / D, nq = (p0 + np - 1) / D - q0 + 1;   // queries touched, <= PAIR_G
    const int n0 = cb * PAIR_COLS, nb = min(PAIR_COLS, H2 - n0);
    float *qu = sm, *qv = sm + PAIR_G, *qo = sm + 2 * PAIR_G;
    float *w2s = sm + 3 * PAIR_G;               // [H1][PAIR_COLS]
    const int ld1 = H1 | 1;                     // odd: rows of 4 pairs in distinct banks
    float *h1s = w2s + (size_t)H1 * PAIR_COLS;  // [PAIR_G][ld1]
    // W2 columns n0 .. n0 + 31 of every k (only within the padded row)
    {
        const int c4n = min(PAIR_COLS, m.H2p - n0) >> 2;
        const uint32_t base = (uint32_t)__cvta_generic_to_shared(w2s);
        for (int e = tid; e < H1 * c4n; e += SIMT_THREADS) {
            const int k = e / c4n, c4 = e - k * c4n;
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                             base + (uint32_t)(4 * (k * PAIR_COLS + 4 * c4))),
                         "l"(__cvta_generic_to_global(m.W2T + (size_t)k * m.H2p + n0 + 4 * c4)) : "memory");
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    }
    // the query slots of the group's queries, side by side
    if (tid < nq) {
        qu[tid] = standardise(m.xform[F - 2], q.in_len[q0 + tid], m.mu[F - 2], m.sd[F - 2]);
    } else if (tid >= 32 && tid < 32 + nq) {
        const float o = q.out_len[q0 + tid - 32];
        qv[tid - 32] = standardise(m.xform[F - 1], o, m.mu[F - 1], m.sd[F - 1]);
        qo[tid - 32] = o;
    }
    // this thread's unit k of layer 1 for every pair of the group: the
    // prefix loads first, all in flight together
    const int k = tid;
    const bool hk = k < H1;
    float av[PAIR_G];
    {
        int qq = q0, d = p0 - q0 * D;
#pragma unroll
        for (int p = 0; p < PAIR_G; ++p) {
            av[p] = hk && p < np ? m.A[(size_t)d * H1 + k] : 0.f;
            if (++d == D) {
                d = 0;
                ++qq;
            }
        }
    }
    const float wi = hk ? m.W1T[(size_t)(F - 2) * H1 + k] : 0.f;
    const float wo = hk ? m.W1T[(size_t)(F - 1) * H1 + k] : 0.f;
    __syncthreads();
    if (hk) {
        int ql = 0, d = p0 - q0 * D;
#pragma unroll
        for (int p = 0; p < PAIR_G; ++p) {
            if (p < np) {
                float x = __fmaf_rn(wi, qu[ql], av[p]);
                x = __fmaf_rn(wo, qv[ql], x);
                h1s[p * ld1 + k] = x > 0.f ? x : 0.f;
            }
            if (++d == D) {
                d = 0;
                ++ql;
            }
        }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    // layer 2: thread (pair p = lane, columns c .. c + 3 of warp w), serial over k
    {
        const int p = lane, c = 4 * warp;
        if (p < np && c < nb) {
            float acc[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) acc[j] = c + j < nb ? m.b2[n0 + c + j] : 0.f;
            const float *hr = h1s + p * ld1;
            const float *wr = w2s + c;
#pragma unroll 8
            for (int kk = 0; kk < H1; ++kk) {
                const float4 w = *reinterpret_cast<const float4 *>(wr + kk * PAIR_COLS);
                const float h = hr[kk];
                acc[0] = __fmaf_rn(w.x, h, acc[0]);
                acc[1] = __fmaf_rn(w.y, h, acc[1]);
                acc[2] = __fmaf_rn(w.z, h, acc[2]);
                acc[3] = __fmaf_rn(w.w, h, acc[3]);
            }
            float *dst = a.h2 + ((size_t)g * H2 + n0 + c) * PAIR_G + p;
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (c + j < nb) dst[j * PAIR_G] = acc[j] > 0.f ? acc[j] : 0.f;
            __threadfence();   // before the group's arrival below
        }
    }
    __syncthreads();
    if (tid == 0) {
        __threadfence();
        s_last = atomicAdd(&a.gcount[g], 1) == a.ncb - 1;
    }
    __syncthreads();
    if (!s_last) return;
    // the group's last column block: heads and cost of every pair
    __threadfence();
    float *h2s = w2s;                            // [H2][PAIR_G]
    float *w3s = h2s + (size_t)H2 * PAIR_G;      // [NH][H2]
    {
        // the group's whole block (rows of pairs past np are not read),
        // L2 to shared memory by 16-byte copies that skip L1
        const uint32_t base = (uint32_t)__cvta_generic_to_shared(h2s);
        const float *src = a.h2 + (size_t)g * H2 * PAIR_G;
        for (int e = tid; e < H2 * PAIR_G / 4; e += SIMT_THREADS)
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(base + 16u * e),
                         "l"(__cvta_generic_to_global(src + 4 * e)) : "memory");
        asm volatile("cp.async.commit_group;" ::: "memory");
    }
    for (int i = tid; i < m.NH * H2; i += SIMT_THREADS) w3s[i] = m.W3[i];
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    __shared__ float hd[PAIR_G * 3];
    if (warp < m.NH) {
        // head o = warp of pair p = lane: W3 reads are broadcasts, h2
        // reads consecutive words
        const int o = warp, p = lane;
        const float *w3 = w3s + (size_t)o * H2;
        float z = m.b3[o];
#pragma unroll 8
        for (int n = 0; n < H2; ++n) z = __fmaf_rn(w3[n], h2s[n * PAIR_G + p], z);
        if (p < np) hd[p * m.NH + o] = softplus_c(z);
    }
    __syncthreads();
    for (int p = tid; p < np; p += SIMT_THREADS) {
        const int qq = (p0 + p) / D, NH = m.NH;
        a.pairC[p0 + p] =
            __fmaf_rn(NH == 3 ? hd[p * NH + 2] : qo[qq - q0], hd[p * NH + 1], hd[p * NH]);
    }
    if (tid == 0) a.gcount[g] = 0;
    __threadfence();
    __syncthreads();
    pair_decide(m, q, a, p0, np, q0, nq);
}

// Column block, fused shape (few groups, so that every block has an SM of
// its own): the block's 8 W2 rows, each pair's deployment prefix row and
// W1's query columns staged by asynchronous copies behind the query slots'
// loads; each layer-1 unit rebuilt where layer 2 consumes it (no layer-1
// pass); h2 scratch [groups][PAIR_G][H2], a row per pair, so that the last
// block's head chains read it as vectors.
__device__ __forceinline__ void pair_cols_fused(const Model &m, const Queries &q, const PairArgs &a,
                                             float *sm, int *s_last_p) {
    int &s_last = *s_last_p;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int F = m.F, H1 = m.H1, H2 = m.H2, D = m.D;
    const int npair = q.Q * D;
    const int g = blockIdx.x / a.ncb, cb = blockIdx.x - g * a.ncb;
    const int p0 = g * PAIR_G, np = min(PAIR_G, npair - p0);
    const int q0 = p0 / D, nq = (p0 + np - 1) / D - q0 + 1;   // queries touched, <= PAIR_G
    const int cols = a.cols, n0 = cb * cols, nb = min(cols, H2 - n0);
    const PairSmem L = pair_smem(H1, H2);
    float *qu = sm, *qv = sm + PAIR_G, *qo = sm + 2 * PAIR_G;
    float *w2c = sm + L.w2;    // [cols][ldk]: W2 rows n0 .. n0 + cols - 1
    float *as = sm + L.as;     // [PAIR_G][lda]: each pair's deployment prefix
    float *w1s = sm + L.w1;    // [2][ldk]: W1's two query columns
    // the query slots' raw lengths first: what follows from them below is this
    // block's longest wait
    float iv = 0.f, ov = 0.f;
    if (tid < nq) iv = q.in_len[q0 + tid];
    else if (tid >= 32 && tid < 32 + nq) ov = q.out_len[q0 + tid - 32];
    {
        // pair p of the group is deployment (p0 + p) mod D; 16-byte copies
        // where the rows allow, else 4-byte ones
        const uint32_t wb = (uint32_t)__cvta_generic_to_shared(w2c);
        const uint32_t ab = (uint32_t)__cvta_generic_to_shared(as);
        const int d0 = p0 - q0 * D;
        if ((H1 & 3) == 0) {
            const int r4 = H1 >> 2;
            for (int e = tid; e < nb * r4; e += SIMT_THREADS) {
                const int c = e / r4, j = e - c * r4;
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                                 wb + (uint32_t)(4 * (c * L.ldk + 4 * j))),
                             "l"(__cvta_generic_to_global(m.W2 + (size_t)(n0 + c) * H1 + 4 * j)) : "memory");
            }
            for (int e = tid; e < np * r4; e += SIMT_THREADS) {
                const int p = e / r4, j = e - p * r4;
                int d = d0 + p;
                d -= (d / D) * D;
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                                 ab + (uint32_t)(4 * (p * L.lda + 4 * j))),
                             "l"(__cvta_generic_to_global(m.A + (size_t)d * H1 + 4 * j)) : "memory");
            }
        } else {
            for (int e = tid; e < nb * H1; e += SIMT_THREADS) {
                const int c = e / H1, j = e - c * H1;
                asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(
                                 wb + (uint32_t)(4 * (c * L.ldk + j))),
                             "l"(__cvta_generic_to_global(m.W2 + (size_t)(n0 + c) * H1 + j)) : "memory");
            }
            for (int e = tid; e < np * H1; e += SIMT_THREADS) {
                const int p = e / H1, j = e - p * H1;
                int d = d0 + p;
                d -= (d / D) * D;
                asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(
                                 ab + (uint32_t)(4 * (p * L.lda + j))),
                             "l"(__cvta_generic_to_global(m.A + (size_t)d * H1 + j)) : "memory");
            }
        }
        const uint32_t w1b = (uint32_t)__cvta_generic_to_shared(w1s);
        for (int e = tid; e < 2 * H1; e += SIMT_THREADS) {
            const int r = e / H1, j = e - r * H1;
            asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(
                             w1b + (uint32_t)(4 * (r * L.ldk + j))),
                         "l"(__cvta_generic_to_global(m.W1T + (size_t)(F - 2 + r) * H1 + j)) : "memory");
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    }
    // the query slots of the group's queries, side by side
    if (tid < nq) {
        qu[tid] = standardise(m.xform[F - 2], iv, m.mu[F - 2], m.sd[F - 2]);
    } else if (tid >= 32 && tid < 32 + nq) {
        qv[tid - 32] = standardise(m.xform[F - 1], ov, m.mu[F - 1], m.sd[F - 1]);
        qo[tid - 32] = ov;
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    // layers 1 and 2: lane = pair p, warp w = columns 2w, 2w + 1
    if (lane < np && 2 * warp < nb) {
        const int p = lane, ql = (p0 + p) / D - q0;
        pair_layers(m, a, L, w2c, as + (size_t)p * L.lda, w1s, qu[ql], qv[ql], g, n0, nb,
                    2 * warp, p);
    }
    __syncthreads();
    if (tid == 0) {
        __threadfence();
        s_last = atomicAdd(&a.gcount[g], 1) == a.ncb - 1;
    }
    __syncthreads();
    if (!s_last) return;
    // the group's last column block: heads and cost of every pair
    __threadfence();
    float *h2s = sm + L.h2;     // [PAIR_G][ld2]: layer 2, a row per pair
    float *w3s = sm + L.w3;     // [NH][H2]
    {
        // the group's rows, L2 to shared memory by copies that skip L1
        const float *src = a.h2 + (size_t)g * PAIR_G * H2;
        if ((H2 & 3) == 0) {
            const uint32_t base = (uint32_t)__cvta_generic_to_shared(h2s);
            const int r4 = H2 >> 2;
            for (int e = tid; e < np * r4; e += SIMT_THREADS) {
                const int p = e / r4, j = e - p * r4;
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                                 base + (uint32_t)(4 * (p * L.ld2 + 4 * j))),
                             "l"(__cvta_generic_to_global(src + (size_t)p * H2 + 4 * j)) : "memory");
            }
            asm volatile("cp.async.commit_group;" ::: "memory");
        } else {
            for (int e = tid; e < np * H2; e += SIMT_THREADS) {
                const int p = e / H2, j = e - p * H2;
                h2s[p * L.ld2 + j] = __ldcg(src + (size_t)p * H2 + j);
            }
        }
    }
    for (int i = tid; i < m.NH * H2; i += SIMT_THREADS) w3s[i] = m.W3[i];
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    __shared__ float hd[PAIR_G * 3];
    if (warp < m.NH && lane < np) {
        // head o = warp, pair p = lane: W3 reads are broadcasts, each lane
        // reads its own row of layer 2, four n per vector
        const int o = warp, p = lane;
        const float *w3 = w3s + (size_t)o * H2, *hr = h2s + (size_t)p * L.ld2;
        float z = m.b3[o];
        int n = 0;
        if ((H2 & 3) == 0) {
            for (; n + 8 <= H2; n += 8) {
                const float4 h0 = *reinterpret_cast<const float4 *>(hr + n);
                const float4 h1 = *reinterpret_cast<const float4 *>(hr + n + 4);
                const float4 v0 = *reinterpret_cast<const float4 *>(w3 + n);
                const float4 v1 = *reinterpret_cast<const float4 *>(w3 + n + 4);
                z = __fmaf_rn(v0.x, h0.x, z);
                z = __fmaf_rn(v0.y, h0.y, z);
                z = __fmaf_rn(v0.z, h0.z, z);
                z = __fmaf_rn(v0.w, h0.w, z);
                z = __fmaf_rn(v1.x, h1.x, z);
                z = __fmaf_rn(v1.y, h1.y, z);
                z = __fmaf_rn(v1.z, h1.z, z);
                z = __fmaf_rn(v1.w, h1.w, z);
            }
        }
        for (; n < H2; ++n) z = __fmaf_rn(w3[n], hr[n], z);
        hd[p * m.NH + o] = softplus_c(z);
    }
    __syncthreads();
    for (int p = tid; p < np; p += SIMT_THREADS) {
        const int qq = (p0 + p) / D, NH = m.NH;
        a.pairC[p0 + p] =
            __fmaf_rn(NH == 3 ? hd[p * NH + 2] : qo[qq - q0], hd[p * NH + 1], hd[p * NH]);
    }
    if (tid == 0) a.gcount[g] = 0;
    __threadfence();
    __syncthreads();
    pair_decide(m, q, a, p0, np, q0, nq);
}

__global__ void __launch_bounds__(SIMT_THREADS) k_route_pairs(Model m, Queries q, PairArgs a) {
    extern __shared__ float4 sm4[];   // 16-byte aligned: operands arrive as 16-byte copies
    float *sm = reinterpret_cast<float *>(sm4);
    __shared__ int s_last;
    const int tid = threadIdx.x;
    const int D = m.D, M = m.M;
    const int npair = q.Q * D, ncolb = pair_groups(npair) * a.ncb;
    if ((int)blockIdx.x < ncolb) {
        if (a.cols == PAIR_COLS) pair_cols_split(m, q, a, sm, &s_last);
        else pair_cols_fused(m, q, a, sm, &s_last);
        return;
    }
    // quality of models [m0, m0 + PAIR_MPB) for one query
    const int b = blockIdx.x - ncolb;
    const int qq = b / a.qblocks;
    const int m0 = (b - qq * a.qblocks) * PAIR_MPB, mn = min(PAIR_MPB, M - m0), E = m.E;
    // emb row [E] and the block's model columns as [E / 4][mn][4] (E is a
    // multiple of 8), so that a chain reads 4 consecutive k of its column as
    // one 16-byte load and the mn chains' loads fall in distinct banks; a
    // thread's staging loads are issued before its stores
    float *er = sm, *mb = sm + E;
    const size_t row = (size_t)qq * E;
    for (int k0 = 0; k0 < E; k0 += SIMT_THREADS) {
        const int k = k0 + tid;
        const bool ok = k < E;
        float v[PAIR_MPB];
        const float ev = ok ? emb_at(q.emb, q.emb_bf16, row + k) : 0.f;
#pragma unroll
        for (int j = 0; j < PAIR_MPB; ++j) v[j] = ok && j < mn ? m.memb[(size_t)k * M + m0 + j] : 0.f;
        if (ok) {
            er[k] = ev;
#pragma unroll
            for (int j = 0; j < PAIR_MPB; ++j)
                if (j < mn) mb[((size_t)(k >> 2) * mn + j) * 4 + (k & 3)] = v[j];
        }
    }
    __syncthreads();
    if (tid < mn) {
        const float4 *c = reinterpret_cast<const float4 *>(mb) + tid;
        const float4 *e4 = reinterpret_cast<const float4 *>(er);
        float s = 0.f;
        // E is a multiple of 8: two 4-term groups' operands, then their FMAs
        for (int k4 = 0; k4 < E / 4; k4 += 2) {
            const float4 x0 = e4[k4], y0 = c[(size_t)k4 * mn];
            const float4 x1 = e4[k4 + 1], y1 = c[(size_t)(k4 + 1) * mn];
            s = __fmaf_rn(x0.x, y0.x, s);
            s = __fmaf_rn(x0.y, y0.y, s);
            s = __fmaf_rn(x0.z, y0.z, s);
            s = __fmaf_rn(x0.w, y0.w, s);
            s = __fmaf_rn(x1.x, y1.x, s);
            s = __fmaf_rn(x1.y, y1.y, s);
            s = __fmaf_rn(x1.z, y1.z, s);
            s = __fmaf_rn(x1.w, y1.w, s);
        }
        a.qualS[(size_t)qq * M + m0 + tid] = sigmoid_c(s);
        __threadfence();
    }
    __syncthreads();
    if (tid == 0) {
        __threadfence();
        s_last = atomicAdd(&a.count[qq], 1) + 1 == D + a.qblocks;
    }
    __syncthreads();
    if (s_last && tid < 32) {
        __threadfence();
        pair_select(m, q, a, qq);
    }
}

// ---------------------------------------------------------------------------
// K_select_multi: the decision maker for several lambdas over stored scores.
// SEL_LANES lanes per query: lane j scans every SEL_LANES-th group of four
// deployments in order and keeps, for each of KT lambdas, the largest feasible
// utility of a group and the group, and the smallest cost for the queries that
// have no feasible deployment; the lanes' results are merged, and one lane per
// lambda looks up the winner inside its group.  Bound: the ALU pipe (half the
// FMA pipe's rate), so a (query, deployment, lambda) costs three FMA-pipe
// instructions (an infeasible utility is pushed to -inf by an addition) and
// one and a half ALU ones: 16 us for 8 lambdas over 65,536 queries
// at D = 64 (a warp per query with two warp reductions per lambda took 53.5, a
// compare and two selects per candidate 21).
// Same order as make_cand / better: a feasible candidate is C <= SLO with a
// defined utility; where a lambda has none, every defined cost is a candidate
// of the other class, so the smallest cost serves all lambdas.
constexpr int SEL_LANES = 4;

template <int KT, bool VEC>
__global__ void __launch_bounds__(SIMT_THREADS)
k_select_multi(Model m, Queries q, const float *C, const float *qual, int qstride, Lambdas L,
               int ostride) {
    __shared__ int dms[MAX_D + 4];
    const int D = m.D;
    for (int d = threadIdx.x; d < D; d += SIMT_THREADS) dms[d] = m.dep_model[d];
    __syncthreads();
    const int t = blockIdx.x * SIMT_THREADS + threadIdx.x, j = t % SEL_LANES;
    const int qq = min(t / SEL_LANES, q.Q - 1);      // the last warp's spare lanes repeat the last query
    const float slo = query_budget(q, qq), nan = __int_as_float(0x7fc00000);
    const float inf = __int_as_float(0x7f800000);
    const float *cr = C + (size_t)qq * D, *qr = qual + (size_t)qq * qstride;
    float bu[KT], bc = nan;       // best utility per lambda, smallest cost
    int bg[KT], bcd = -1;         // the group of bu (its first deployment), bc's deployment
    bool any = false;             // a feasible cost
#pragma unroll
    for (int k = 0; k < KT; ++k) {
        bu[k] = -inf;
        bg[k] = 4 * j;
    }
    for (int d0 = 4 * j; d0 < D; d0 += 4 * SEL_LANES) {
        float c[4], g[4], pen[4];
        if constexpr (VEC) {
            const float4 v = *reinterpret_cast<const float4 *>(cr + d0);
            c[0] = v.x;
            c[1] = v.y;
            c[2] = v.z;
            c[3] = v.w;
        } else {
#pragma unroll
            for (int i = 0; i < 4; ++i) c[i] = d0 + i < D ? cr[d0 + i] : nan;
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            g[i] = VEC || d0 + i < D ? qr[dms[d0 + i]] : 0.f;
            pen[i] = c[i] <= slo ? 0.f : -inf;          // NaN costs too
            any = any || c[i] <= slo;
            // !(c >= bc): also when there is none yet; NaN costs never win
            if (c[i] == c[i] && !(c[i] >= bc)) {
                bc = c[i];
                bcd = d0 + i;
            }
        }
#pragma unroll
        for (int k = 0; k < KT; ++k) {
            float u[4];
#pragma unroll
            for (int i = 0; i < 4; ++i)
                u[i] = __fadd_rn(__fmaf_rn(-L.lam[k], c[i], __fmul_rn(L.wq[k], g[i])), pen[i]);
            // (a NaN utility is no candidate, and fmaxf drops it)
            const float best = fmaxf(fmaxf(u[0], u[1]), fmaxf(u[2], u[3]));
            const bool win = best > bu[k];
            bu[k] = win ? best : bu[k];
            bg[k] = win ? d0 : bg[k];
        }
    }
    const unsigned all = 0xffffffffu;
#pragma unroll
    for (int s = 1; s < SEL_LANES; s *= 2) {
        const float oc = __shfl_xor_sync(all, bc, s);
        const int ocd = __shfl_xor_sync(all, bcd, s);
        if (ocd >= 0 && (bcd < 0 || oc < bc || (oc == bc && ocd < bcd))) {
            bc = oc;
            bcd = ocd;
        }
        any = __shfl_xor_sync(all, (int)any, s) || any;
#pragma unroll
        for (int k = 0; k < KT; ++k) {
            const float ou = __shfl_xor_sync(all, bu[k], s);
            const int og = __shfl_xor_sync(all, bg[k], s);
            const bool win = ou > bu[k] || (ou == bu[k] && og < bg[k]);
            bu[k] = win ? ou : bu[k];
            bg[k] = win ? og : bg[k];
        }
    }
    if (t / SEL_LANES >= q.Q) return;
    // lane j finishes lambdas j, j + SEL_LANES, ...
#pragma unroll
    for (int k0 = 0; k0 < KT; k0 += SEL_LANES) {
        float b = bu[k0];
        int d0 = bg[k0];
#pragma unroll
        for (int i = 1; i < SEL_LANES; ++i) {
            b = j == i ? bu[k0 + i] : b;
            d0 = j == i ? bg[k0 + i] : d0;
        }
        const int k = k0 + j;
        if (k >= L.K) continue;
        const float lam = L.lam[k], wq = L.wq[k];
        int bd = -1;
        float cost = nan, u = nan;
        if (any) {
            // the first of the winning group's candidates with the best utility;
            // a best of -inf may also be no group's: then all of them
            const int d1 = b > -inf ? min(d0 + 4, D) : D;
            for (int d = b > -inf ? d0 : 0; d < d1 && bd < 0; ++d) {
                const float c = cr[d], v = __fmaf_rn(-lam, c, __fmul_rn(wq, qr[dms[d]]));
                if (c <= slo && v == b) {
                    bd = d;
                    cost = c;
                    u = v;
                }
            }
        }
        if (bd < 0 && bcd >= 0) {
            bd = bcd;
            cost = bc;
            u = __fmaf_rn(-lam, bc, __fmul_rn(wq, qr[dms[bcd]]));
        }
        const size_t o = (size_t)k * ostride + qq;
        q.chosen[o] = bd;
        q.lat[o] = cost;
        q.util[o] = u;
    }
}

// ---------------------------------------------------------------------------
// host launchers

static int cpt_for(int H2) { return H2 <= 32 ? 1 : H2 <= 64 ? 2 : H2 <= 128 ? 4 : 8; }

size_t seq_table_smem(const Model &m) {
    return seq_layout(m.H2).total * sizeof(float);
}

static size_t chain_smem(int D, int M, int Qs) {
    return (2 * MAX_D + SEQ_MAX_CHUNK + chain_tab_floats(D, Qs) + (size_t)Qs * M + (size_t)Qs) * sizeof(float);
}


int seq_chunk(const Model &m) {
    int Qs = SEQ_MAX_CHUNK;
    while (Qs > 1 && chain_smem(m.D, m.M, Qs) > (size_t)SEQ_CHAIN_SMEM) --Qs;
    return Qs;
}

// Launch configuration of a programmatic dependent launch: the grid may be
// scheduled before the previous kernel in the stream has finished; it calls
// griddepcontrol.wait before it reads that kernel's results.
static cudaLaunchAttribute g_pdl_attr = [] {
    cudaLaunchAttribute a = {};
    a.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    a.val.programmaticStreamSerializationAllowed = 1;
    return a;
}();

static cudaLaunchConfig_t dependent_launch(int grid, int block, size_t smem, cudaStream_t s) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3((unsigned)block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = &g_pdl_attr;
    cfg.numAttrs = 1;
    return cfg;
}

template <class K>
static cudaError_t opt_in(K kernel, int bytes) {
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
}

cudaError_t simt_prepare() {
    const int big = 200 * 1024, most = 227 * 1024;
    cudaError_t e = cudaSuccess;
    if (e == cudaSuccess) e = opt_in(k_route_rows<32>, most);
    if (e == cudaSuccess) e = opt_in(k_route_rows<64>, most);
    if (e == cudaSuccess) e = opt_in(k_route_rows<128>, most);
    if (e == cudaSuccess) e = opt_in(k_route_rows<256>, most);
    if (e == cudaSuccess) e = opt_in(k_route_simt<1>, big);
    if (e == cudaSuccess) e = opt_in(k_route_simt<2>, big);
    if (e == cudaSuccess) e = opt_in(k_route_simt<4>, big);
    if (e == cudaSuccess) e = opt_in(k_route_simt<8>, big);
    if (e == cudaSuccess) e = opt_in(k_seq_table<1>, big);
    if (e == cudaSuccess) e = opt_in(k_seq_table<2>, big);
    if (e == cudaSuccess) e = opt_in(k_seq_table<4>, big);
    if (e == cudaSuccess) e = opt_in(k_seq_table<8>, big);
    if (e == cudaSuccess) e = opt_in(k_seq_chain<false, false>, SEQ_CHAIN_SMEM + 1024);
    if (e == cudaSuccess) e = opt_in(k_seq_chain<true, false>, SEQ_CHAIN_SMEM + 1024);
    if (e == cudaSuccess) e = opt_in(k_seq_chain<false, true>, SEQ_CHAIN_SMEM + 1024);
    if (e == cudaSuccess) e = opt_in(k_seq_chain<true, true>, SEQ_CHAIN_SMEM + 1024);
    if (e == cudaSuccess) e = opt_in(k_route_pairs, big);
    return e;
}

cudaError_t launch_snapshot(const Model &m, const uint32_t *stage, cudaStream_t s) {
    k_snapshot<<<m.D, SIMT_THREADS, (size_t)m.F * sizeof(float), s>>>(m, stage);
    return cudaGetLastError();
}

template <int W>
static cudaError_t launch_rows(const Model &m, const Queries &q, int nsm, int32_t *status,
                               cudaStream_t s) {
    const RowsLayout L = rows_layout<W>(m.D, m.M, m.NH, m.H1, m.H2p, q.emb_bf16 ? 2 : 4);
    k_route_rows<W><<<q.Q < nsm ? q.Q : nsm, RouteShape<W>::THREADS, L.total, s>>>(m, q, status);
    return cudaGetLastError();
}

// Which of the two batch kernels.  Up to one round of k_route_simt's blocks (64
// rows; 3 an SM, 2 with more than 128 columns) its short critical path wins.
// Above, k_route_rows keeps the FMA pipe busier, unless its deciding warps'
// quality chains (E x M a query, 32 or 16 queries a warp, 16 models a pass) take
// longer than the tiles (D x H1 x H2 a query): k_route_simt has a warp for them
// in every block.  Where the chains stay under 0.6 of the tiles and a query has
// 4 deployments or more, k_route_rows is taken; elsewhere both kernels' times
// are estimated (us, GB300) from those parts and the smaller wins.  The
// constants were chosen on 4,861 measured shapes (D 1 to 64, M 1 to 64, E 8 to
// 8,192, H1 and H2 1 to 256, one round to sixteen, fp32 and bf16 embeddings) so
// that the choice costs least: 0.5 % over the better kernel on average on them,
// 0.9 % on 900 others (the worst: 17 / 27 us at H1 = 1, D = 64, M = 4).
// Measured (us, simt / rows): H = 128, D = 12, E = 768: 1.2 M pairs 1,330 / 954;
// H = 128, D = M = 64, E = 1,024: 30,000 pairs 100 / 191, 146,000 291 / 234;
// H = 64, D = 4, M = 2, E = 4,096: 88,000 310 / 323, 233,000 813 / 511; H = 256,
// D = 12, E = 1,024: 27,000 109 / 102, 97,000 361 / 307.
static bool rows_kernel(const Model &m, int Q, bool bf, int nsm) {
    const int D = m.D, M = m.M, W = tile_width(m.H2), per = W == 256 ? 2 : 3;
    if ((long)Q * D <= 64L * per * nsm) return false;
    const double hk = (m.H1 + 31) / 32, fma = hk * W / 256;     // 32 x 256 multiply-adds a row
    const double three = m.NH == 3 ? 1.0 : 0.0;
    auto up = [](long a, long b) { return (a + b - 1) / b; };
    // k_route_rows: the deciding warps' and the scoring warps' time
    const int nq = W <= 64 ? 4 : 2, nw = 16 - nq, rg = W == 256 ? 8 : 16, qbk = D > 32 ? 16 : 32;
    const long q = up(Q, nsm);
    const int cols = M < QUAL_MC ? M : QUAL_MC, ng = (cols + 4 * (32 / qbk) - 1) / (4 * (32 / qbk));
    const double chunk = 0.57 + (bf ? 0.19 : 0.11) * (ng == 3 ? 4 : ng) +
                         (M <= QUAL_MC && M % 4 == 0 ? 0.0 : 0.51);
    const double dec = up(up(q, qbk), nq) * (up(M, QUAL_MC) * up(m.E, QUAL_KC) * chunk + 3.22);
    const double group = 3.31 + 0.62 * hk + 3.22 * three +
                         (W == 256 ? 7.67 : W == 128 ? 10.59 : 5.88) * fma * nw * rg / 192.0;
    const double score = up(up(q * D, rg), nw) * group;
    if (D >= 4 && dec < 0.6 * score) return true;
    const double rows = 8.95 + (dec > score ? dec + 0.47 * score : score + 0.47 * dec);
    // k_route_simt: waves of `per` blocks an SM, each the longer of its tiles and
    // its quality chains and a part of the other
    const int qb = route_qb(D);
    const double chains = 1e-3 * m.E * (9.36 + (bf ? 0.58 : 0.83) * qb + 0.35 * M + (qb * M > 32 ? 5.5 : 0.0));
    const double block = 1.44 + (W >= 128 ? 3.53 : 5.6) * fma + 1.44 * three;
    auto wave = [&](long n) {
        const double tile = n * block > 3.24 * hk ? n * block : 3.24 * hk;
        return 0.04 * qb + (tile > chains ? tile + 0.59 * chains : chains + 0.59 * tile);
    };
    const long blocks = up(Q, qb), full = blocks / ((long)per * nsm), rest = up(blocks - full * per * nsm, nsm);
    const double simt = 8.1 + full * wave(per) + (rest ? wave(rest) : 0.0);
    return rows < simt;
}

cudaError_t launch_route_simt(const Model &m, const Queries &q, int nsm, int kernel, int32_t *status,
                              HostFlag flag, uint32_t *blocks_done, bool *flagged, cudaStream_t s) {
    *flagged = false;
    if (q.Q <= 0) return cudaSuccess;
    if (kernel < 0 ? rows_kernel(m, q.Q, q.emb_bf16, nsm) : kernel == 1) {
        switch (tile_width(m.H2)) {
            case 32: return launch_rows<32>(m, q, nsm, status, s);
            case 64: return launch_rows<64>(m, q, nsm, status, s);
            case 128: return launch_rows<128>(m, q, nsm, status, s);
            default: return launch_rows<256>(m, q, nsm, status, s);
        }
    }
    const RouteLayout L = route_layout(m.D, m.M, m.H2);
    const int blocks = (q.Q + L.QB - 1) / L.QB;
    const size_t smem = L.total * sizeof(float);
    if (flag.word) flag.target = *blocks_done + (uint32_t)blocks;
    switch (cpt_for(m.H2)) {
        case 1: k_route_simt<1><<<blocks, ROUTE_THREADS, smem, s>>>(m, q, flag); break;
        case 2: k_route_simt<2><<<blocks, ROUTE_THREADS, smem, s>>>(m, q, flag); break;
        case 4: k_route_simt<4><<<blocks, ROUTE_THREADS, smem, s>>>(m, q, flag); break;
        default: k_route_simt<8><<<blocks, ROUTE_THREADS, smem, s>>>(m, q, flag); break;
    }
    const cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess && flag.word) {      // (a launch that failed counts no blocks)
        *blocks_done = flag.target;
        *flagged = true;
    }
    return e;
}

size_t route_pairs_smem(const Model &m) {
    const size_t fused = (size_t)pair_smem(m.H1, m.H2).total;
    const size_t split = 3 * PAIR_G + (size_t)m.H1 * PAIR_COLS + (size_t)PAIR_G * (m.H1 | 1);
    const size_t fin = 3 * PAIR_G + (size_t)m.H2 * PAIR_G + (size_t)m.NH * m.H2;
    size_t blk = fused > split ? fused : split;
    blk = blk > fin ? blk : fin;
    const size_t qual = (size_t)m.E * (1 + PAIR_MPB);
    return (blk > qual ? blk : qual) * sizeof(float);
}

cudaError_t launch_route_pairs(const Model &m, const Queries &q, float *pairC, float *qualS,
                               float *h2, int32_t *count, int nsm, cudaStream_t s) {
    if (q.Q <= 0) return cudaSuccess;
    if ((long)q.Q * m.D > PAIRS_MAX_PAIRS) return cudaErrorInvalidValue;
    PairArgs a;
    a.pairC = pairC;
    a.qualS = qualS;
    a.h2 = h2;
    a.count = count;
    a.gcount = count + PAIRS_MAX_PAIRS;
    a.qblocks = (m.M + PAIR_MPB - 1) / PAIR_MPB;
    // The fused shape, 8 columns per block, when the whole grid still has an
    // SM per block: a layer-2 chain step there waits mostly on its shared
    // loads, so narrower blocks (fewer chains sharing an SM's shared memory)
    // finish sooner; with more groups the split shape's 32 columns per block
    // keep the grid to one wave.
    const int groups = pair_groups(q.Q * m.D);
    a.cols = (long)groups * ((m.H2 + PAIR_FUSED_COLS - 1) / PAIR_FUSED_COLS) +
                         (long)q.Q * a.qblocks <= nsm
                 ? PAIR_FUSED_COLS
                 : PAIR_COLS;
    a.ncb = (m.H2 + a.cols - 1) / a.cols;
    const int blocks = pair_groups(q.Q * m.D) * a.ncb + q.Q * a.qblocks;
    k_route_pairs<<<blocks, SIMT_THREADS, route_pairs_smem(m), s>>>(m, q, a);
    return cudaGetLastError();
}

cudaError_t launch_select_multi(const Model &m, const Queries &q, const float *C,
                                const float *qual, int qstride, const Lambdas &L, int ostride,
                                cudaStream_t s) {
    if (q.Q <= 0 || L.K <= 0 || L.K > MAX_LAMBDAS) return q.Q <= 0 || L.K <= 0 ? cudaSuccess : cudaErrorInvalidValue;
    const long threads = (long)q.Q * SEL_LANES;
    const int blocks = (int)((threads + SIMT_THREADS - 1) / SIMT_THREADS);
    // rows of costs as 16-byte vectors where every row allows it
    const bool vec = m.D % 4 == 0 && ((uintptr_t)C & 15) == 0;
    const int kt = (L.K + 3) / 4;     // lambdas in fours (those past K are not written)
#define HWR_SELECT(KT)                                                                              \
    (vec ? k_select_multi<KT, true><<<blocks, SIMT_THREADS, 0, s>>>(m, q, C, qual, qstride, L, ostride) \
         : k_select_multi<KT, false><<<blocks, SIMT_THREADS, 0, s>>>(m, q, C, qual, qstride, L, ostride))
    if (kt == 1) HWR_SELECT(4);
    else if (kt == 2) HWR_SELECT(8);
    else if (kt == 3) HWR_SELECT(12);
    else HWR_SELECT(16);
#undef HWR_SELECT
    return cudaGetLastError();
}

// Blocks of a chunk's table: quality blocks, and blocks of rpb rows (a multiple
// of 8, whole warps of the tile) that spread the table evenly over the blocks
// resident at once.
struct SeqGrid {
    int nb_qual, rpb, blocks;
};

static SeqGrid seq_grid(const Model &m, int Qs, int slots) {
    SeqGrid g;
    const int T = (int)tri_off(m.D, Qs, Qs);
    g.nb_qual = (Qs + seq_qual_rows(m.M) - 1) / seq_qual_rows(m.M);
    const int want = slots - g.nb_qual > 1 ? slots - g.nb_qual : 1;
    const int rpb = ((T + want - 1) / want + 7) / 8 * 8;
    g.rpb = rpb < 8 ? 8 : (rpb > TILE_ROWS ? TILE_ROWS : rpb);
    g.blocks = g.nb_qual + (T + g.rpb - 1) / g.rpb;
    return g;
}

// Queries per chunk of a sequential call of Q.  A chunk costs a fixed part (its
// launches, the tables' serial parts, the walk and its copy) and its table, which
// grows with the square of a chunk, so wide clusters take shorter chunks.  The
// table's time goes by the blocks that the busiest SM takes, resident or one after
// the other, and by their rows: above 32 a block's warps double up on the SM's
// sub-partitions (H = 256, D = 20, us: 43.0 at 32 rows, 58.0 at 40, 62.5 to 65 at 48
// to 64; a third block on an SM, a fourth: 91, 117).  The constants (us) fit every
// chunk size from 8 on of 110 shapes measured on GB300 (D 2 to 64, H1 and H2 16 to
// 256, apart in half of them), chosen for calls of 64 to 1,000: 0.9 % over the best
// chunk on average, 13 % at most (fitted to half of the shapes only, 1.3 % and
// 14 % on the others).
// 1,000 requests in the largest chunks that the chain takes / in the ones
// chosen here (us): D = 12, H = 128 541 / 511; D = 32, H = 64 479 / 458; D = 32,
// H = 256 2,674 / 1,726; D = 64, H = 256 4,433 / 2,786.
int seq_pick_chunk(const Model &m, int Q, int limit, int slots, int nsm) {
    const int W = tile_width(m.H2);
    const double hk = (m.H1 + 31) / 32, fma = m.H1 * W / 8192.0;
    const double fixed_us = 4.9 + 0.8 * hk + 0.33 * W / 32, block_us = 0.6 + 0.065 * hk + 1.1 * fma;
    int best = limit;
    double best_cost = 1e300;
    for (int n = (Q + limit - 1) / limit;; ++n) {
        const int Qs = (Q + n - 1) / n;
        const SeqGrid g = seq_grid(m, Qs, slots);
        const int blocks = (g.blocks - g.nb_qual + nsm - 1) / nsm;      // on the busiest SM
        const double rows = 0.3 * ((g.rpb + 31) / 32) + 0.7 * (g.rpb < 16 ? 16 : g.rpb) / 32;
        const double cost = ((Q + Qs - 1) / Qs) * (fixed_us + 0.057 * Qs + block_us * blocks * rows);
        if (cost < best_cost) {
            best_cost = cost;
            best = Qs;
        }
        if (Qs <= 8) break;
        // the next chunk size below this one
        n = (Q + Qs - 2) / (Qs - 1) - 1 > n ? (Q + Qs - 2) / (Qs - 1) - 1 : n;
    }
    return best;
}

cudaError_t launch_seq_table(const Model &m, const Queries &q, int Qs, int Ns, int off0, int slots,
                             float *ctab, float *aux, cudaStream_t s) {
    const SeqGrid g = seq_grid(m, Qs, slots);
    const int nb_qual = g.nb_qual, rpb = g.rpb;
    cudaLaunchConfig_t cfg = dependent_launch(g.blocks, SIMT_THREADS, seq_layout(m.H2).total * sizeof(float), s);
    switch (cpt_for(m.H2)) {
        case 1: return cudaLaunchKernelEx(&cfg, k_seq_table<1>, m, q, Qs, Ns, off0, nb_qual, rpb, ctab, aux);
        case 2: return cudaLaunchKernelEx(&cfg, k_seq_table<2>, m, q, Qs, Ns, off0, nb_qual, rpb, ctab, aux);
        case 4: return cudaLaunchKernelEx(&cfg, k_seq_table<4>, m, q, Qs, Ns, off0, nb_qual, rpb, ctab, aux);
        default: return cudaLaunchKernelEx(&cfg, k_seq_table<8>, m, q, Qs, Ns, off0, nb_qual, rpb, ctab, aux);
    }
}

int seq_table_slots(const Model &m) {
    int dev = 0, nsm = 0, per = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return 1;
    const size_t smem = seq_layout(m.H2).total * sizeof(float);
    cudaError_t e;
    switch (cpt_for(m.H2)) {
        case 1: e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_seq_table<1>, SIMT_THREADS, smem); break;
        case 2: e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_seq_table<2>, SIMT_THREADS, smem); break;
        case 4: e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_seq_table<4>, SIMT_THREADS, smem); break;
        default: e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_seq_table<8>, SIMT_THREADS, smem); break;
    }
    if (e != cudaSuccess || per < 1) per = 1;
    return nsm * per;
}

cudaError_t launch_seq_chain(const Model &m, const Queries &q, int Qs, int Ns, const float *ctab,
                             float *aux, bool more, cudaStream_t s) {
    cudaLaunchConfig_t cfg = dependent_launch(1, CHAIN_THREADS, chain_smem(m.D, m.M, Qs), s);
    const SeqAux A = seq_aux(aux, m.D, m.M, Ns);
    if (m.D > 32)
        return cudaLaunchKernelEx(&cfg, k_seq_chain<true, false>, m, q, Qs, Ns, ctab, aux,
                                  (const float *)A.qual, m.M, 0, (int)more);
    return cudaLaunchKernelEx(&cfg, k_seq_chain<false, false>, m, q, Qs, Ns, ctab, aux,
                              (const float *)A.qual, m.M, 0, (int)more);
}

cudaError_t launch_seq_prep(const Model &m, const Queries &q, int Ns, float *aux, uint16_t *pre_bf,
                            int32_t *dmv, cudaStream_t s) {
    const int nuv = (2 * Ns + PREP_THREADS - 1) / PREP_THREADS;
    cudaLaunchConfig_t cfg =
        dependent_launch(nuv + m.D * seq_prep_blocks_per_dep(Ns), PREP_THREADS, 0, s);
    return cudaLaunchKernelEx(&cfg, k_seq_prep, m, q, Ns, aux, pre_bf, dmv);
}

cudaError_t launch_seq_chain_tc(const Model &m, const Queries &q, int Qs, const float *ctab,
                                float *aux, const float *qual, int qstride, bool more,
                                cudaStream_t s) {
    if (chain_smem(m.D, m.M, Qs) <= (size_t)SEQ_CHAIN_SMEM) {
        cudaLaunchConfig_t cfg = dependent_launch(1, CHAIN_THREADS, chain_smem(m.D, m.M, Qs), s);
        if (m.D > 32)
            return cudaLaunchKernelEx(&cfg, k_seq_chain<true, false>, m, q, Qs, Qs, ctab, aux, qual,
                                      qstride, 0, (int)more);
        return cudaLaunchKernelEx(&cfg, k_seq_chain<false, false>, m, q, Qs, Qs, ctab, aux, qual,
                                  qstride, 0, (int)more);
    }
    // the table's first rows in shared memory, the rest read from L2
    const size_t rest = chain_smem(m.D, m.M, Qs) - chain_tab_floats(m.D, Qs) * sizeof(float);
    if (rest + 4 * sizeof(float) > (size_t)SEQ_CHAIN_SMEM) return cudaErrorInvalidValue;
    const int tsm = (int)(((size_t)SEQ_CHAIN_SMEM - rest) / sizeof(float)) & ~3;
    cudaLaunchConfig_t cfg =
        dependent_launch(1, CHAIN_THREADS, rest + (size_t)tsm * sizeof(float), s);
    if (m.D > 32)
        return cudaLaunchKernelEx(&cfg, k_seq_chain<true, true>, m, q, Qs, Qs, ctab, aux, qual,
                                  qstride, tsm, (int)more);
    return cudaLaunchKernelEx(&cfg, k_seq_chain<false, true>, m, q, Qs, Qs, ctab, aux, qual, qstride,
                              tsm, (int)more);
}

}  // namespace hwr

