// The fp32 tile of the large-batch kernel: one warp scores RG rows, each a (query,
// deployment) pair, from a deployment prefix of layer 1 and two query features to
// the cost, in canonical order (every dot product bias first, k ascending, one
// fused rounding per step).
//
// What bounds it is the FMA pipe (128 a cycle and SM), so the layout keeps
// everything else off its way:
//   * A warp is on its own: it builds its rows' layer 1 in its own shared
//     buffer, runs layer 2, the heads and the cost, and never meets a block
//     barrier, so one warp's serial parts (head chains, softplus) run under
//     the other warps' FMAs.
//   * A lane holds LR rows x LC columns of layer 2; the warp's lanes cover the
//     W columns, 32 LC / W times over for as many sets of LR rows.  Every
//     16-byte shared load costs the shared pipe about three cycles, whether its
//     lanes read the same address or not, so a k step's loads per FMA count:
//     8 x 8 takes 4 for 2,048 FMAs, 8 x 4 takes 3 for 1,024.  16 x 8 (6 for
//     4,096) leaves room for 3 warps a sub-partition instead of 4 and measured
//     slower: 1,120 against 969 us for 100,000 queries at D = 12, H = 128.
//   * W2 (transposed, rows of k) is read from chunks of TILE_KC rows that bulk
//     copies bring: all of it where it fits, loaded once per block, else a
//     ring that every warp walks once per group of rows; the warp that uses a
//     stage last asks for its next contents, so no warp waits to produce.
#pragma once

#include "canon_math.cuh"
#include "hwr_internal.cuh"
#include "umma.cuh"

namespace hwr {

constexpr int TILE_KC = 32;

// Lane tile of a group of RG rows with W columns (8 rows at W = 256, else 16): LC
// columns and LR rows a lane, NSET sets of rows.
template <int W, int RG>
struct Tile {
    static constexpr int LC = W >= 128 ? 8 : W == 64 ? 4 : 2;
    static constexpr int NSET = 32 * LC / W, LR = RG / NSET;
    static constexpr int LD = RG + 4;                    // layer-1 chunk [TILE_KC][LD], k-major:
                                                         // a lane's 16-byte stores of its k fall in
                                                         // distinct banks, eight lanes a wavefront
    static constexpr int PIECE = W < 64 ? 32 : 64;       // layer-2 columns the head chains read at a time
    static constexpr int PLD = PIECE + 4;                // their row stride: odd in 16-byte units
    static constexpr int BUF = TILE_KC * LD > RG * PLD ? TILE_KC * LD : RG * PLD;
    static_assert(LR == 8 && NSET >= 1 && RG == (W == 256 ? 8 : 16), "lane tile");
};

// One row as the tile reads it: standardised query slots, offset of the
// deployment prefix, expected output length.
struct __align__(16) RowInfo {
    float u, v;
    int off;
    float ol;
};

// W2 chunk feed of a block.  Chunk c of a pass sits in stage c % ns; with
// ns = nch every stage is loaded once and kept.
struct W2Feed {
    const float *w2t;            // [H1][ldw] in global memory
    float *sm;                   // [ns][TILE_KC][ldw] (and slack for the widest lane)
    uint64_t *full;              // [ns]
    uint32_t *used;              // [ns] warps that have used the stage's contents
    uint32_t *issued;            // chunks asked for so far
    volatile int *abort_f;
    int32_t *status;
    int H1, ldw, ns, nch, warps;
    __device__ __forceinline__ bool resident() const { return ns == nch; }
    uint32_t total;              // chunks that all passes use (ring)
};

// Ask for chunk n (counted over all passes): one thread.
__device__ __forceinline__ void w2_issue(const W2Feed &f, uint32_t n) {
    const int c = (int)(n % (uint32_t)f.nch), s = (int)(n % (uint32_t)f.ns);
    const int k0 = c * TILE_KC, kc = min(TILE_KC, f.H1 - k0);
    const uint32_t bytes = (uint32_t)(kc * f.ldw) * 4u;
    umma::mbar_arrive_expect_tx(&f.full[s], bytes);
    umma::bulk_g2s(f.sm + (size_t)s * TILE_KC * f.ldw, f.w2t + (size_t)k0 * f.ldw, bytes, &f.full[s]);
}

// The first chunks: one thread, after the barriers are initialised.
__device__ __forceinline__ void w2_start(const W2Feed &f) {
    const uint32_t n = f.resident() ? (uint32_t)f.nch : min((uint32_t)f.ns, f.total);
    for (uint32_t i = 0; i < n; ++i) w2_issue(f, i);
    *f.issued = n;
}

// Wait for chunk n; false after a timeout.
__device__ __forceinline__ bool w2_wait(const W2Feed &f, uint32_t n) {
    const uint32_t s = n % (uint32_t)f.ns, ph = f.resident() ? 0u : (n / (uint32_t)f.ns) & 1u;
    return umma::mbar_wait(&f.full[s], ph, f.abort_f, f.status);
}

// This warp is done with chunk n (after a __syncwarp): the last of the
// block's warps asks for the chunk that takes its stage next.
__device__ __forceinline__ void w2_release(const W2Feed &f, uint32_t n) {
    if (f.resident() || (threadIdx.x & 31) != 0) return;
    const uint32_t s = n % (uint32_t)f.ns;
    uint32_t seen;
    asm volatile("atom.acq_rel.cta.shared.add.u32 %0, [%1], 1;"
                 : "=r"(seen) : "r"(umma::smem_u32(&f.used[s])) : "memory");
    if (seen != (uint32_t)f.warps - 1) return;
    *(volatile uint32_t *)&f.used[s] = 0;
    if (n + (uint32_t)f.ns < f.total) {
        w2_issue(f, n + (uint32_t)f.ns);
        atomicAdd(f.issued, 1u);
    }
}

// Before the block ends: every chunk asked for has landed (one thread; bounded).
__device__ __forceinline__ void w2_drain(const W2Feed &f) {
    const uint32_t n = *(volatile uint32_t *)f.issued;
    for (uint32_t i = n > (uint32_t)f.ns ? n - (uint32_t)f.ns : 0; i < n; ++i) {
        const uint32_t s = i % (uint32_t)f.ns, ph = f.resident() ? 0u : (i / (uint32_t)f.ns) & 1u;
        const long long t0 = clock64();
        while (!umma::mbar_try_wait(&f.full[s], ph) && clock64() - t0 < umma::WAIT_CYCLES) {
        }
    }
}

// A pass over the ring by a warp that has no rows in it.
__device__ __forceinline__ bool w2_skip(const W2Feed &f, uint32_t n0) {
    if (f.resident()) return true;
    for (int c = 0; c < f.nch; ++c) {
        const bool ok = w2_wait(f, n0 + c);
        if (!__all_sync(0xffffffffu, ok)) return false;
        w2_release(f, n0 + c);
    }
    return true;
}

// The block's weights that every row uses, in shared memory.
struct TileWeights {
    const float *w1q;   // [2][H1]: W1's query columns
    const float *b2;    // [W], zero past H2
    const float *w3;    // [NH][H2p]
    const float *b3;    // [NH]
};

__device__ __forceinline__ float relu(float x) { return x > 0.f ? x : 0.f; }

// Shared-memory loads by 32-bit address.
__device__ __forceinline__ float4 lds4(uint32_t a) {
    float4 t;
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(t.x), "=f"(t.y), "=f"(t.z), "=f"(t.w) : "r"(a));
    return t;
}
__device__ __forceinline__ float2 lds2(uint32_t a) {
    float2 t;
    asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(t.x), "=f"(t.y) : "r"(a));
    return t;
}
__device__ __forceinline__ float lds1(uint32_t a) {
    float t;
    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(t) : "r"(a));
    return t;
}

// One k of layer 2: this set's layer-1 values ar [LR] times this lane's
// columns of W2 at wr (shared addresses; pieces of 4 columns W / (LC / 4)
// columns apart).
template <int W, int LR, int LC>
__device__ __forceinline__ void tile_step(uint32_t ar, uint32_t wr, float2 (&acc)[LR / 2][LC]) {
    constexpr int VW = LC < 4 ? LC : 4, NP = LR / 2, NV = LC / VW;
    float2 a[NP];
#pragma unroll
    for (int i = 0; i < NP; i += 2) {
        const float4 t = lds4(ar + 8 * i);
        a[i] = make_float2(t.x, t.y);
        a[i + 1] = make_float2(t.z, t.w);
    }
    float b[LC];
#pragma unroll
    for (int v = 0; v < NV; ++v) {
        if constexpr (VW == 4) {
            const float4 t = lds4(wr + 4 * (W / NV) * v);
            b[4 * v] = t.x;
            b[4 * v + 1] = t.y;
            b[4 * v + 2] = t.z;
            b[4 * v + 3] = t.w;
        } else {
            const float2 t = lds2(wr);
            b[0] = t.x;
            b[1] = t.y;
        }
    }
    // each lane of the packed FMA rounds once, as __fmaf_rn
#pragma unroll
    for (int j = 0; j < LC; ++j)
#pragma unroll
        for (int i = 0; i < NP; ++i) acc[i][j] = __ffma2_rn(make_float2(b[j], b[j]), a[i], acc[i][j]);
}

// Scores the RG rows ri[0 .. RG - 1]; lane r < RG returns row r's cost.  Every
// lane of the warp calls it; n0 is the feed's chunk count at this group's
// first chunk; prefix_s: the prefixes' address in shared memory (0: they are
// in global memory, at prefix).  False after a timeout.
template <int W, int RG>
__device__ __forceinline__ bool warp_tile(const Model &m, const W2Feed &f, const TileWeights &w,
                                          uint32_t n0, const RowInfo *ri, const float *prefix,
                                          uint32_t prefix_s, float *buf, float &cost) {
    using T = Tile<W, RG>;
    constexpr int LR = T::LR, LC = T::LC, NP = LR / 2, LD = T::LD, PLD = T::PLD, PIECE = T::PIECE;
    constexpr int VW = LC < 4 ? LC : 4, NV = LC / VW, CL = W / LC;    // CL lanes cover the columns
    const int lane = threadIdx.x & 31, H1 = m.H1, H2 = m.H2, ldw = f.ldw;
    const int cl = lane % CL, set = lane / CL;
    float2 acc[NP][LC];
#pragma unroll
    for (int j = 0; j < LC; ++j) {
        const float b = w.b2[(W / NV) * (j / VW) + VW * cl + j % VW];
#pragma unroll
        for (int i = 0; i < NP; ++i) acc[i][j] = make_float2(b, b);
    }
    const uint32_t ar = umma::smem_u32(buf) + 4u * (uint32_t)(set * LR);
    uint32_t stage = n0 % (uint32_t)f.ns;
    for (int k0 = 0, c = 0; k0 < H1; k0 += TILE_KC, ++c) {
        const int kc = min(TILE_KC, H1 - k0), k = k0 + lane;
        // layer 1 of unit k0 + lane for every row: relu(fma(w_out, v, fma(w_in, u, prefix)))
        if (lane < kc) {
            const float wi = w.w1q[k], wo = w.w1q[H1 + k];
            auto rows4 = [&](auto prefix_at) {
#pragma unroll
                for (int i0 = 0; i0 < RG; i0 += 4) {
                    RowInfo t[4];
                    float x[4];
#pragma unroll
                    for (int i = 0; i < 4; ++i) t[i] = ri[i0 + i];
#pragma unroll
                    for (int i = 0; i < 4; ++i) x[i] = prefix_at(t[i].off + k);
#pragma unroll
                    for (int i = 0; i < 4; ++i) x[i] = relu(__fmaf_rn(wo, t[i].v, __fmaf_rn(wi, t[i].u, x[i])));
                    *reinterpret_cast<float4 *>(buf + lane * LD + i0) = make_float4(x[0], x[1], x[2], x[3]);
                }
            };
            if (prefix_s) rows4([&](int i) { return lds1(prefix_s + 4u * (uint32_t)i); });
            else rows4([&](int i) { return prefix[i]; });
        }
        __syncwarp();
        if (!f.resident() || n0 == 0) {
            const bool ok = w2_wait(f, n0 + c);
            if (!__all_sync(0xffffffffu, ok)) return false;
        }
        const uint32_t wr = umma::smem_u32(f.sm) + 4u * (stage * (uint32_t)(TILE_KC * ldw) + (uint32_t)(VW * cl));
        if (++stage == (uint32_t)f.ns) stage = 0;
        if (kc == TILE_KC) {
#pragma unroll 4
            for (int kk = 0; kk < TILE_KC; ++kk) tile_step<W, LR, LC>(ar + 4 * kk * LD, wr + 4 * kk * ldw, acc);
        } else {
#pragma unroll 1
            for (int kk = 0; kk < kc; ++kk) tile_step<W, LR, LC>(ar + 4 * kk * LD, wr + 4 * kk * ldw, acc);
        }
        __syncwarp();
        w2_release(f, n0 + c);
    }

    // heads: layer 2 through the buffer in pieces of PIECE columns; lane (row,
    // head), and for RG = 16 the lanes of the first head run the third as well
    const int NH = m.NH, H2p = m.H2p;
    const int r = lane % RG, o = min(lane / RG, NH - 1);
    const bool three = RG == 16 && NH == 3;
    float z0 = w.b3[o], z2 = three ? w.b3[2] : 0.f;
    const float *hr = buf + r * PLD;
#pragma unroll
    for (int pc = 0; pc < W / PIECE; ++pc) {
        if (PIECE * pc < H2) {
            if constexpr (VW == 4) {
                // columns PIECE pc ..: in this lane's block v, lanes c0 .. of the set
                constexpr int per = W / NV;                   // columns per block of 4-column lanes
                const int v = PIECE * pc / per, c0 = (PIECE * pc % per) / 4;
                if (cl >= c0 && cl < c0 + PIECE / 4) {
                    const int j = 4 * v;
#pragma unroll
                    for (int i = 0; i < NP; ++i) {
                        float4 t0, t1;
                        t0.x = relu(acc[i][j].x);
                        t0.y = relu(acc[i][j + 1].x);
                        t0.z = relu(acc[i][j + 2].x);
                        t0.w = relu(acc[i][j + 3].x);
                        t1.x = relu(acc[i][j].y);
                        t1.y = relu(acc[i][j + 1].y);
                        t1.z = relu(acc[i][j + 2].y);
                        t1.w = relu(acc[i][j + 3].y);
                        float *d = buf + (set * LR + 2 * i) * PLD + 4 * (cl - c0);
                        *reinterpret_cast<float4 *>(d) = t0;
                        *reinterpret_cast<float4 *>(d + PLD) = t1;
                    }
                }
            } else {
                const int n = VW * cl - PIECE * pc;
                if (n >= 0 && n < PIECE) {
#pragma unroll
                    for (int i = 0; i < NP; ++i)
#pragma unroll
                        for (int j = 0; j < LC; ++j) {
                            float *d = buf + (set * LR + 2 * i) * PLD + n + j;
                            d[0] = relu(acc[i][j].x);
                            d[PLD] = relu(acc[i][j].y);
                        }
                }
            }
            __syncwarp();
            const int n1 = min(PIECE, H2 - PIECE * pc);
            const float *w30 = w.w3 + o * H2p + PIECE * pc,
                        *w32 = w.w3 + 2 * H2p + PIECE * pc;
            int n = 0;
#pragma unroll 4
            for (; n + 4 <= n1; n += 4) {
                const float4 h = *reinterpret_cast<const float4 *>(hr + n);
                const float4 t = *reinterpret_cast<const float4 *>(w30 + n);
                z0 = __fmaf_rn(t.x, h.x, z0);
                z0 = __fmaf_rn(t.y, h.y, z0);
                z0 = __fmaf_rn(t.z, h.z, z0);
                z0 = __fmaf_rn(t.w, h.w, z0);
                if (three) {
                    const float4 s = *reinterpret_cast<const float4 *>(w32 + n);
                    z2 = __fmaf_rn(s.x, h.x, z2);
                    z2 = __fmaf_rn(s.y, h.y, z2);
                    z2 = __fmaf_rn(s.z, h.z, z2);
                    z2 = __fmaf_rn(s.w, h.w, z2);
                }
            }
            for (; n < n1; ++n) {
                z0 = __fmaf_rn(w30[n], hr[n], z0);
                if (three) z2 = __fmaf_rn(w32[n], hr[n], z2);
            }
            __syncwarp();
        }
    }
    const unsigned all = 0xffffffffu;
    const float ttft = softplus_c(z0);
    const float tpot = __shfl_sync(all, ttft, RG + r);
    float nout = ri[r].ol;
    if (NH == 3) nout = RG == 8 ? __shfl_sync(all, ttft, 16 + r) : softplus_c(z2);
    cost = __fmaf_rn(nout, tpot, ttft);       // lanes r < RG: z0 is the first head
    return true;
}

}  // namespace hwr
