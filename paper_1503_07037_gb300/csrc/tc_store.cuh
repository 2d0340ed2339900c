// Epilogue stores of the tcgen05 kernels through a per-warp shared-memory transpose.
//
// tcgen05.ld leaves one output row per lane (TMEM lane = row), so a lane that applies the
// epilogue where it stands writes 16 bytes into each of 32 different rows per instruction,
// and every load of C or E that follows a store has to wait for it (the compiler cannot
// move a load of C above a store to D that may alias it). On short-K tiles, the grouped
// products of a batch, those dependent row-strided accesses cost more than the tile's
// MMAs. Here a 32 x 32 block goes through a 32 x 33 shared-memory buffer instead: lanes
// then take 32 consecutive columns of one row, so each access of C, D, Dhi, Dlo and E is a
// 128-byte row segment, and the loads of a batch of rows are issued before its first store.
// Symmetric results send the values back through the buffer for the mirrored block, whose
// rows are the block's columns: those stores are row segments as well.
//
// A single warp per scheduler runs this code while the tensor pipe works, so it is written
// for few instructions: two warps per scheduler execute straight-line code at about one
// instruction in eight clocks (the stall is instruction fetch), and the element-wise form of a
// block, about a thousand instructions, took 8000 clocks whether or not it stored anything;
// four such blocks were 17 of the 35 us of a 256 x 256 tile at K = 512. Blocks off
// the diagonal and with 16-byte rows therefore move four elements per instruction
// (epi_block32_vec, epi_block32_trans_vec); the other blocks take the masked element-wise form,
// where the symmetric mirror and the TF32 split copies are template parameters chosen once per
// tile, beta C, gamma I and the dot enter through selects, and out-of-range elements are
// masked by predicated stores.
#pragma once

#include <cstdint>

#include "epilogue.cuh"

namespace cdmpt {
namespace tc {

// Words of one warp's transpose buffer: 32 rows of 33 for the element-wise form, the pad word
// keeping both the row-wise and the column-wise passes free of bank conflicts. The
// four-element form takes 32 rows of 32 words whose 16-byte chunk j stands at j ^ (row % 8), so
// that eight lanes cover all banks once along a row and down a column of chunks.
constexpr int kXposeWords = 32 * 33;
__device__ __forceinline__ int xpose_at(int row, int chunk) {
    return row * 32 + 4 * (chunk ^ (row & 7));
}

__device__ __forceinline__ void split_tf32(float v, float& h, float& l) {
    uint32_t hb, lb;
    asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(hb) : "f"(v));
    h = __uint_as_float(hb);
    asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(lb) : "f"(v - h));
    l = __uint_as_float(lb);
}

// The block through the buffer: S[row][col] = a, lane = row on entry.
__device__ __forceinline__ void xpose_in(const float (&a)[32], float* S, int lane) {
#pragma unroll
    for (int j = 0; j < 32; ++j) S[lane * 33 + j] = a[j];
    __syncwarp();
}

template <bool SYM, bool SPLIT>
__device__ __forceinline__ float epi_block32_plain(const EpiParams<float>& p, int m0, int n,
                                                   bool diag, float* S, int lane) {
    constexpr int RB = 8;   // rows whose loads are issued together
    // every field the loops use, read once (p may live in global memory, where the
    // stores below could alias it)
    const int M = p.M, N = p.N;
    const size_t ldd = (size_t)p.ldd, ldc = (size_t)p.ldc, lde = (size_t)p.lde;
    float* const D = p.D;
    float* const Dhi = p.Dhi;
    float* const Dlo = p.Dlo;
    const int c = n + lane;
    const bool col_ok = c < N;
    const float alpha = p.alpha, beta = p.beta, gamma = p.gamma;
    const bool has_c = beta != 0.f, has_g = gamma != 0.f, has_dot = p.dot != nullptr;
    const bool has_e = has_dot && p.E != nullptr;
    const int db = p.diag_block;
    int mm = has_g ? m0 % db : -1;   // (m0 + r) % diag_block, advanced row by row
    const size_t o0 = (size_t)m0 * ldd + c;
    const float* Cp = has_c ? p.C + (size_t)m0 * ldc + c : nullptr;
    const float* Ep = has_e ? p.E + (size_t)m0 * lde + c : nullptr;
    float local = 0.f;
#pragma unroll 1
    for (int r0 = 0; r0 < 32; r0 += RB) {
        float cv[RB], ev[RB];
#pragma unroll
        for (int i = 0; i < RB; ++i) {
            const int m = m0 + r0 + i;
            const bool ok = col_ok && m < M && !(diag && c < m);
            cv[i] = (ok && has_c) ? Cp[(size_t)(r0 + i) * ldc] : 0.f;
            ev[i] = (ok && has_e) ? Ep[(size_t)(r0 + i) * lde] : 0.f;
        }
#pragma unroll
        for (int i = 0; i < RB; ++i) {
            const int m = m0 + r0 + i;
            const bool ok = col_ok && m < M && !(diag && c < m);
            float v = alpha * S[(r0 + i) * 33 + lane];
            v = has_c ? fmaf(beta, cv[i], v) : v;
            v = (has_g && mm == c) ? v + gamma : v;
            mm = (mm + 1 == db) ? 0 : mm + 1;
            if constexpr (SYM) S[(r0 + i) * 33 + lane] = v;
            const size_t o = o0 + (size_t)(r0 + i) * ldd;
            if (ok) D[o] = v;
            if constexpr (SPLIT) {
                float h, l;
                split_tf32(v, h, l);
                if (ok) {
                    Dhi[o] = h;
                    Dlo[o] = l;
                }
            }
            const float d = v * (has_e ? ev[i] : v);
            const float w = (SYM && m != c) ? 2.f * d : d;
            local += (ok && has_dot) ? w : 0.f;
        }
    }
    if constexpr (SYM) {
        // the mirrored block: lane l on row m0 + l again, column n + j goes to row n + j
        __syncwarp();
        const int m = m0 + lane;
        const bool row_ok = m < M;
        const size_t q0 = (size_t)n * ldd + m;
#pragma unroll 8
        for (int j = 0; j < 32; ++j) {
            const int cj = n + j;
            const bool ok = row_ok && cj < N && cj != m && !(diag && cj < m);
            const float w = S[lane * 33 + j];
            const size_t o = q0 + (size_t)j * ldd;
            if (ok) D[o] = w;
            if constexpr (SPLIT) {
                float h, l;
                split_tf32(w, h, l);
                if (ok) {
                    Dhi[o] = h;
                    Dlo[o] = l;
                }
            }
        }
    }
    return local;
}

// Transposed placement (never symmetric): element (m, n) of the product goes to row
// trans_block b + n, column m - trans_block b of its row block b, so that the 32 lanes (rows)
// write consecutive columns. The loads of eight columns are issued before their stores: an
// element-wise loop waits one memory latency per column for C, 32 per block.
template <bool SPLIT>
__device__ __forceinline__ float epi_block32_trans(const EpiParams<float>& p, int m0, int n,
                                                   const float* S, int lane) {
    constexpr int RB = 8;
    const int m = m0 + lane, N = p.N;
    const bool row_ok = m < p.M;
    const int b = m / p.trans_block;
    const size_t r0 = (size_t)b * p.trans_block + n, c = (size_t)(m - b * p.trans_block);
    const size_t ldd = (size_t)p.ldd, ldc = (size_t)p.ldc, lde = (size_t)p.lde;
    float* const D = p.D;
    float* const Dhi = p.Dhi;
    float* const Dlo = p.Dlo;
    const float alpha = p.alpha, beta = p.beta, gamma = p.gamma;
    const bool has_c = beta != 0.f, has_g = gamma != 0.f, has_dot = p.dot != nullptr;
    const bool has_e = has_dot && p.E != nullptr;
    const int md = has_g ? m % p.diag_block : -1;
    float local = 0.f;
#pragma unroll 1
    for (int j0 = 0; j0 < 32; j0 += RB) {
        float cv[RB], ev[RB];
#pragma unroll
        for (int i = 0; i < RB; ++i) {
            const bool ok = row_ok && n + j0 + i < N;
            cv[i] = (ok && has_c) ? p.C[(r0 + j0 + i) * ldc + c] : 0.f;
            ev[i] = (ok && has_e) ? p.E[(r0 + j0 + i) * lde + c] : 0.f;
        }
#pragma unroll
        for (int i = 0; i < RB; ++i) {
            const bool ok = row_ok && n + j0 + i < N;
            float v = alpha * S[lane * 33 + j0 + i];
            v = has_c ? fmaf(beta, cv[i], v) : v;
            v = md == n + j0 + i ? v + gamma : v;
            const size_t o = (r0 + j0 + i) * ldd + c;
            if (ok) D[o] = v;
            if constexpr (SPLIT) {
                float h, l;
                split_tf32(v, h, l);
                if (ok) {
                    Dhi[o] = h;
                    Dlo[o] = l;
                }
            }
            local += (ok && has_dot) ? v * (has_e ? ev[i] : v) : 0.f;
        }
    }
    return local;
}

// Four elements' TF32 split, stored.
__device__ __forceinline__ void split_tf32_x4(const float4& v, float* hi, float* lo) {
    float4 h, l;
    split_tf32(v.x, h.x, l.x);
    split_tf32(v.y, h.y, l.y);
    split_tf32(v.z, h.z, l.z);
    split_tf32(v.w, h.w, l.w);
    *(float4*)hi = h;
    *(float4*)lo = l;
}

// The block, off the diagonal of a symmetric result, arrays and leading dimensions 16-byte and
// its columns inside the matrix a multiple of 4: lane l takes columns 4 (l % 8) of rows
// l / 8 + 4 i, so a warp instruction moves four 128-byte row segments.
template <bool SYM, bool SPLIT>
__device__ __forceinline__ float epi_block32_vec(const EpiParams<float>& p, int m0, int n,
                                                 float* S, int lane) {
    constexpr int RB = 2;   // row groups whose loads are issued together
    const size_t ldd = (size_t)p.ldd;
    const float alpha = p.alpha, beta = p.beta, gamma = p.gamma;
    const bool has_c = beta != 0.f, has_dot = p.dot != nullptr;   // E is null here
    const int r0 = lane >> 3, c0 = (lane & 7) * 4;
    // column of the diagonal of gamma I in row m0 + r0, relative to this lane's first column
    int dg = gamma != 0.f ? (m0 + r0) % p.diag_block - (n + c0) : 1 << 30;
    const int db = p.diag_block;
    const size_t o0 = (size_t)(m0 + r0) * ldd + n + c0;
    float* Dp = p.D + o0;
    float* Hp = SPLIT ? p.Dhi + o0 : nullptr;
    float* Lp = SPLIT ? p.Dlo + o0 : nullptr;
    const float* Cp = has_c ? p.C + (size_t)(m0 + r0) * p.ldc + n + c0 : nullptr;
    const size_t sd = 4 * ldd, sc = 4 * (size_t)p.ldc;
    // rows r0 + 4 i: chunk l % 8 alternates between two places
    const int rows = n + c0 < p.N ? p.M - m0 - r0 : 0;   // this lane's rows 4 i < rows exist
    float* Sp = S + r0 * 32;
    const int s0 = 4 * ((lane & 7) ^ r0), s1 = s0 ^ 16;
    float local = 0.f;
#pragma unroll 1
    for (int i0 = 0; i0 < 8; i0 += RB) {
        float4 v[RB], cv[RB];
#pragma unroll
        for (int i = 0; i < RB; ++i) {
            if (has_c && 4 * (i0 + i) < rows) cv[i] = *(const float4*)(Cp + i * sc);
            v[i] = *(const float4*)(Sp + i * 128 + ((i & 1) ? s1 : s0));
        }
#pragma unroll
        for (int i = 0; i < RB; ++i) {
            float4 w = v[i];
            w.x *= alpha;
            w.y *= alpha;
            w.z *= alpha;
            w.w *= alpha;
            if (has_c) {
                w.x = fmaf(beta, cv[i].x, w.x);
                w.y = fmaf(beta, cv[i].y, w.y);
                w.z = fmaf(beta, cv[i].z, w.z);
                w.w = fmaf(beta, cv[i].w, w.w);
            }
            if ((unsigned)dg < 4u) {
                w.x += dg == 0 ? gamma : 0.f;
                w.y += dg == 1 ? gamma : 0.f;
                w.z += dg == 2 ? gamma : 0.f;
                w.w += dg == 3 ? gamma : 0.f;
            }
            dg += 4;
            if (gamma != 0.f && dg + n + c0 >= db) dg -= db;
            if constexpr (SYM) *(float4*)(Sp + i * 128 + ((i & 1) ? s1 : s0)) = w;
            v[i] = w;
            if (has_dot && 4 * (i0 + i) < rows)
                local += w.x * w.x + w.y * w.y + w.z * w.z + w.w * w.w;
        }
#pragma unroll
        for (int i = 0; i < RB; ++i) {
            if (4 * (i0 + i) < rows) {
                *(float4*)(Dp + i * sd) = v[i];
                if constexpr (SPLIT) split_tf32_x4(v[i], Hp + i * sd, Lp + i * sd);
            }
        }
        Dp += RB * sd;
        if constexpr (SPLIT) {
            Hp += RB * sd;
            Lp += RB * sd;
        }
        Cp += has_c ? RB * sc : 0;
        Sp += RB * 128;
    }
    if constexpr (SYM) {
        // the mirrored block: lane l on row m0 + l, columns n + j to rows n + j
        __syncwarp();
        const size_t q0 = (size_t)n * ldd + m0 + lane;
        float* Mp = p.D + q0;
        float* Mh = SPLIT ? p.Dhi + q0 : nullptr;
        float* Ml = SPLIT ? p.Dlo + q0 : nullptr;
        const int cols = m0 + lane < p.M ? p.N - n : 0;   // rows n + j, j < cols, take this lane's
#pragma unroll 1
        for (int j = 0; j < 32; j += 8) {
            const float4 a = *(const float4*)(S + xpose_at(lane, j >> 2)),
                         b = *(const float4*)(S + xpose_at(lane, (j >> 2) + 1));
            const float w[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                if (j + i >= cols) break;
                Mp[i * ldd] = w[i];
                if constexpr (SPLIT) {
                    float h, l;
                    split_tf32(w[i], h, l);
                    Mh[i * ldd] = h;
                    Ml[i * ldd] = l;
                }
            }
            Mp += 8 * ldd;
            if constexpr (SPLIT) {
                Mh += 8 * ldd;
                Ml += 8 * ldd;
            }
        }
        local *= 2.f;   // the mirror counts too
    }
    return local;
}

// Transposed placement of a block inside one row block: lane l holds row m0 + l, so that the lanes write consecutive columns of each row n + j of the row block.
template <bool SPLIT>
__device__ __forceinline__ float epi_block32_trans_vec(const EpiParams<float>& p, int m0, int n,
                                                       const float* S, int lane) {
    const int b = m0 / p.trans_block;
    const size_t r0 = (size_t)b * p.trans_block + n, c = (size_t)(m0 + lane - b * p.trans_block);
    const size_t ldd = (size_t)p.ldd, ldc = (size_t)p.ldc;
    const float alpha = p.alpha, beta = p.beta, gamma = p.gamma;
    const bool has_c = beta != 0.f, has_dot = p.dot != nullptr;   // E is null here
    const int md = gamma != 0.f ? (m0 + lane) % p.diag_block - n : -1;
    float* Dp = p.D + r0 * ldd + c;
    float* Hp = SPLIT ? p.Dhi + r0 * ldd + c : nullptr;
    float* Lp = SPLIT ? p.Dlo + r0 * ldd + c : nullptr;
    const float* Cp = has_c ? p.C + r0 * ldc + c : nullptr;
    const int cols = m0 + lane < p.M ? p.N - n : 0;
    float local = 0.f;
#pragma unroll 1
    for (int j = 0; j < 32; j += 8) {
        float cv[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            if (has_c && j + i < cols) cv[i] = Cp[i * ldc];
        }
        const float4 x = *(const float4*)(S + xpose_at(lane, j >> 2)),
                     y = *(const float4*)(S + xpose_at(lane, (j >> 2) + 1));
        const float w[8] = {x.x, x.y, x.z, x.w, y.x, y.y, y.z, y.w};
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            if (j + i >= cols) break;
            float v = alpha * w[i];
            if (has_c) v = fmaf(beta, cv[i], v);
            if (md == j + i) v += gamma;
            Dp[i * ldd] = v;
            if constexpr (SPLIT) {
                float h, l;
                split_tf32(v, h, l);
                Hp[i * ldd] = h;
                Lp[i * ldd] = l;
            }
            if (has_dot) local += v * v;
        }
        Dp += 8 * ldd;
        if constexpr (SPLIT) {
            Hp += 8 * ldd;
            Lp += 8 * ldd;
        }
        Cp += has_c ? 8 * ldc : 0;
    }
    return local;
}

// The parked block by the four-element form.
__device__ __forceinline__ float epi_block32_parked(const EpiParams<float>& p, int m0, int n, float* S,
                                                 int lane) {
    const bool split = p.Dhi != nullptr;
    if (p.trans_block > 0)
        return split ? epi_block32_trans_vec<true>(p, m0, n, S, lane)
                     : epi_block32_trans_vec<false>(p, m0, n, S, lane);
    if (p.sym)
        return split ? epi_block32_vec<true, true>(p, m0, n, S, lane)
                     : epi_block32_vec<true, false>(p, m0, n, S, lane);
    return split ? epi_block32_vec<false, true>(p, m0, n, S, lane)
                 : epi_block32_vec<false, false>(p, m0, n, S, lane);
}

// The masked element-wise form of a block in the 33-word layout.
__device__ __forceinline__ float epi_block32_masked(const EpiParams<float>& p, int m0, int n, bool diag,
                                                 float* S, int lane) {
    const bool split = p.Dhi != nullptr;
    if (p.trans_block > 0)
        return split ? epi_block32_trans<true>(p, m0, n, S, lane)
                     : epi_block32_trans<false>(p, m0, n, S, lane);
    if (p.sym)
        return split ? epi_block32_plain<true, true>(p, m0, n, diag, S, lane)
                     : epi_block32_plain<true, false>(p, m0, n, diag, S, lane);
    return split ? epi_block32_plain<false, true>(p, m0, n, diag, S, lane)
                 : epi_block32_plain<false, false>(p, m0, n, diag, S, lane);
}

// Applies the epilogue (alpha, beta C, gamma I, transposed placement, TF32 split copies,
// symmetric mirror, Frobenius dot; the same arithmetic as epi_apply and epi_apply_sym) to
// the block of an output tile with rows m0 .. m0 + 31 and columns n .. n + 31. Lane l holds
// row m0 + l in a[0 .. 31]. diag: a diagonal tile of a symmetric result, whose elements
// below the diagonal are not taken. S: this warp's kXposeWords-word buffer. Returns the
// lane's share of the D * E sum (mirrored elements counted twice). Warp-collective.
__device__ __forceinline__ float epi_block32(const EpiParams<float>& p, int m0, int n,
                                             bool diag, const float (&a)[32], float* S,
                                             int lane) {
    // outside the matrix, or below the diagonal of a symmetric result
    if (m0 >= p.M || n >= p.N || (diag && n + 31 < m0)) return 0.f;
    bool vec = !(diag && n < m0 + 32) && !(p.dot && p.E);
    if (p.trans_block > 0) {
        const int last = m0 + 31 < p.M ? m0 + 31 : p.M - 1;
        vec = vec && m0 / p.trans_block == last / p.trans_block;
    } else {
        vec = vec && (n + 32 <= p.N || (p.N & 3) == 0);
        const uintptr_t al = (uintptr_t)p.D | (uintptr_t)p.Dhi | (uintptr_t)p.Dlo |
                             (p.beta != 0.f ? (uintptr_t)p.C : 0);
        const int lds = p.ldd | (p.beta != 0.f ? p.ldc : 0);
        vec = vec && (al & 15) == 0 && (lds & 3) == 0;
        // the four-element form follows the diagonal of gamma I by one wrap per four rows
        vec = vec && (p.gamma == 0.f || p.diag_block >= 4);
    }
    float local;
    if (vec) {
#pragma unroll
        for (int j = 0; j < 32; j += 4)
            *(float4*)(S + xpose_at(lane, j >> 2)) =
                make_float4(a[j], a[j + 1], a[j + 2], a[j + 3]);
        __syncwarp();
        local = epi_block32_parked(p, m0, n, S, lane);
    } else {
        xpose_in(a, S, lane);
        local = epi_block32_masked(p, m0, n, diag, S, lane);
    }
    __syncwarp();   // the buffer is reused by the next block
    return local;
}

}  // namespace tc
}  // namespace cdmpt
