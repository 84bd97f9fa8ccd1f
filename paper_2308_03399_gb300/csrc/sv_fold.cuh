// Stage folding: the active stages of a complex64 pass composed into one
// matrix, by one warp.  Used by the register pass kernel (per warp and
// branch) and by resident runs (per block).
#pragma once

#include "sv_common.cuh"

namespace sv {

// One entry per active stage, in op order: x one of these, y the byte offset
// of its matrix in shared memory, z its structure (one-qubit shape, mono_info,
// or the packed masks of a Pauli string or projection in group form), w the
// group bits it acts on, 4 bits each.
enum : int32_t { RA_ONE = 0, RA_ONE_SHAPED, RA_TWO, RA_MONO, RA_PAULI, RA_PROJ };

// Folded pass (complex64): the active stages composed on the 16 unit vectors,
// one warp.  Column c of the matrix belongs to lanes c and c + 16, which
// take half of the row pairs (or quads) of a stage each; the arithmetic is
// that of the register stages on one group.
// Work matrix: rows r and r + 1 of column c side by side, so that the dense
// product reads two entries with one 128-bit load.
constexpr int FOLD_LD = 17;  // columns of a row pair, padded (bank spread)
__device__ __forceinline__ int fold_at(int r) { return ((r >> 1) * FOLD_LD << 1) | (r & 1); }

// m0 u + m1 w with every rounding spelled out (the contraction that
// reg_apply1 compiles to: left to itself, the compiler picks another one here)
__device__ __forceinline__ float2 row2(float2 m0, float2 m1, float2 u, float2 w) {
    float2 r;
    r.x = __fmaf_rn(-m1.y, w.y, __fmaf_rn(m1.x, w.x, __fmaf_rn(m0.x, u.x, -__fmul_rn(m0.y, u.y))));
    r.y = __fmaf_rn(m1.y, w.x, __fmaf_rn(m1.x, w.y, __fmaf_rn(m0.x, u.y, __fmul_rn(m0.y, u.x))));
    return r;
}

// cmul as the register stages round it
__device__ __forceinline__ float2 cmul_rn(float2 a, float2 b) {
    return make_float2(__fmaf_rn(a.x, b.x, -__fmul_rn(a.y, b.y)), __fmaf_rn(a.y, b.x, __fmul_rn(a.x, b.y)));
}

static __device__ __noinline__ void res_compose(const int4* act, int cnt, const unsigned char* smem, float2* M) {
    const int lane = threadIdx.x & 31, c = lane & 15, h = lane >> 4;
    float2* const col = M + 2 * c;
#pragma unroll
    for (int r = 0; r < 8; ++r) col[fold_at(8 * h + r)] = make_float2(8 * h + r == c ? 1.f : 0.f, 0.f);
    __syncwarp();
    for (int s = 0; s < cnt; ++s) {
        const int4 a = act[s];
        const int j0 = a.w & 15, j1 = (a.w >> 4) & 15;
        const float2* m = reinterpret_cast<const float2*>(smem + a.y);
        if (a.x == RA_ONE || a.x == RA_ONE_SHAPED) {
            // every load before the first store: the compiler cannot move a
            // load of one pair above the stores of another
            const float2 m0 = m[0], m1 = m[1], m2 = m[2], m3 = m[3];
            float2 u[4], w[4];
            int r0[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int g = 4 * h + i, r = ((g >> j0) << (j0 + 1)) | (g & ((1 << j0) - 1));
                r0[i] = fold_at(r);
                u[i] = col[r0[i]];
                w[i] = col[fold_at(r | (1 << j0))];
            }
            const int step = fold_at(1 << j0);
            const bool diag = (a.z & 3) == 1;
            const float2 p = diag ? m0 : m1, q = diag ? m3 : m2;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                float2 x, y;
                if (a.x == RA_ONE) {
                    x = row2(m0, m1, u[i], w[i]);
                    y = row2(m2, m3, u[i], w[i]);
                } else {
                    const float2 pu = diag ? u[i] : w[i], qu = diag ? w[i] : u[i];
                    if (a.z & 4) {
                        x = make_float2(p.x * pu.x, p.x * pu.y);
                        y = make_float2(q.x * qu.x, q.x * qu.y);
                    } else {
                        x = cmul_rn(p, pu);
                        y = cmul_rn(q, qu);
                    }
                }
                col[r0[i]] = x;
                col[r0[i] + step] = y;
            }
        } else if (a.x == RA_TWO || a.x == RA_MONO) {
            const int lo = j0 < j1 ? j0 : j1, hi = j0 < j1 ? j1 : j0;
            const int s0 = fold_at(1 << j0), s1 = fold_at(1 << j1);
            float2 v[2][4];
            int at[2];
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                int g = 2 * h + i;
                g = ((g >> lo) << (lo + 1)) | (g & ((1 << lo) - 1));
                g = ((g >> hi) << (hi + 1)) | (g & ((1 << hi) - 1));
                at[i] = fold_at(g);
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const int pq = a.x == RA_MONO ? (a.z >> (8 + 2 * q)) & 3 : q;
                    v[i][q] = col[at[i] + (pq & 1 ? s0 : 0) + (pq & 2 ? s1 : 0)];
                }
            }
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                float2 o[4];
                if (a.x == RA_MONO) {
#pragma unroll
                    for (int q = 0; q < 4; ++q) o[q] = a.z & 2 ? v[i][q] : cmul_rn(m[q], v[i][q]);
                } else {
                    const ulonglong2* mx = reinterpret_cast<const ulonglong2*>(m);
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        unsigned long long acc = 0ull;
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            const ulonglong2 mm = mx[q * 4 + e];
                            acc = fma2(mm.x, pk2(v[i][e].x, v[i][e].y), acc);
                            acc = fma2(mm.y, pk2(v[i][e].y, v[i][e].x), acc);
                        }
                        o[q] = upk2(acc);
                    }
                }
#pragma unroll
                for (int q = 0; q < 4; ++q) col[at[i] + (q & 1 ? s0 : 0) + (q & 2 ? s1 : 0)] = o[q];
            }
        } else {  // Pauli string or projection: elementwise on rows, moved by a flip mask
            float2 o[8];
            const int x = a.x == RA_PAULI ? a.z & 15 : (a.z >> 16) & 15;
            const float sc = a.x == RA_PAULI ? 0.f : *reinterpret_cast<const float*>(smem + a.y);
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const int e = 8 * h + i;
                float2 t = col[fold_at(e ^ x)];
                if (a.x == RA_PAULI) {
                    if ((a.z >> 4) & 1) t = make_float2(t.y, -t.x);
                    if ((a.z >> (8 + e)) & 1) t = make_float2(-t.x, -t.y);
                } else if ((a.z >> (e ^ x)) & 1) {
                    t = make_float2(t.x * sc, t.y * sc);
                } else {
                    t = make_float2(0.f, 0.f);
                }
                o[i] = t;
            }
            __syncwarp();
#pragma unroll
            for (int i = 0; i < 8; ++i) col[fold_at(8 * h + i)] = o[i];
        }
        __syncwarp();
    }
}

}  // namespace sv
