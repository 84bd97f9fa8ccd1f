// Philox draws and the final sampling building blocks (Section IV-B-2's
// sampling measure), used by
// the batch path (sv_kernels.cu), resident runs (sv_resident.cuh) and
// sv_final_sample_noalloc (sv_noalloc.cu), so all give the same key for the
// same state and draw.
//
// A state of 2^n amplitudes is cut into `chunks` contiguous chunks of L
// amplitudes (final_chunks).  chunk_sum() / chunk_sum_warp() give one chunk's
// sum of |psi_j|^2 (one CTA or one warp, float-float or float64 per lane, the
// lanes combined to float64 precision in a fixed order); chunk_cum()
// turns a state's chunk sums into a running sum (one warp, fixed order);
// sample_warp() draws one key: the chunk by a two-level warp search over the
// running sums, then the first j with u < C_j by a warp prefix sum over 256
// amplitudes at a time (8 per lane), to float64 precision.
#pragma once
#include <cuda_runtime.h>

#include <cstdint>

namespace svs {

// Philox4x32-10 (Salmon, Moraes, Dror, Shaw, SC'11): ten rounds of two 32x32
// multiplies with the published multipliers and Weyl key increments.
// key = (seed lo, seed hi), counter = (shot lo, shot hi, op, 0); the draw is
// the top 53 bits of words 0 and 1.
__device__ __forceinline__ uint64_t philox_k53(uint64_t seed, uint64_t shot, uint32_t op) {
    uint32_t key0 = (uint32_t)seed, key1 = (uint32_t)(seed >> 32);
    uint32_t w0 = (uint32_t)shot, w1 = (uint32_t)(shot >> 32), w2 = op, w3 = 0u;
#pragma unroll
    for (int round = 0; round < 10; ++round) {
        const uint32_t a_hi = __umulhi(0xD2511F53u, w0), a_lo = 0xD2511F53u * w0;
        const uint32_t b_hi = __umulhi(0xCD9E8D57u, w2), b_lo = 0xCD9E8D57u * w2;
        const uint32_t n0 = b_hi ^ w1 ^ key0;
        const uint32_t n2 = a_hi ^ w3 ^ key1;
        w0 = n0;
        w1 = b_lo;
        w2 = n2;
        w3 = a_lo;
        key0 += 0x9E3779B9u;
        key1 += 0xBB67AE85u;
    }
    return ((((uint64_t)w0) << 32) | (uint64_t)w1) >> 11;
}

// the uniform draw u = k * 2^-53 in [0, 1)
__device__ __forceinline__ double philox_uniform(uint64_t seed, uint64_t shot, uint32_t op) {
    return (double)philox_k53(seed, shot, op) * 0x1.0p-53;
}

// chunks of a state's final sample: 2048 amplitudes each, at most 1024 of them
constexpr int64_t CHUNK_AMPS = 2048;
__host__ __device__ __forceinline__ int final_chunks(int64_t dim) {
    const int64_t c = dim / CHUNK_AMPS;
    return (int)(c < 1 ? 1 : (c > 1024 ? 1024 : c));
}

template <class R> struct Cx;
template <> struct Cx<float> { using T = float2; };
template <> struct Cx<double> { using T = double2; };

// A sum in three float32 words, each TwoSum's error carried on to the next
// word: value() is it rounded to float64 once, so sums kept this way lose no
// more than float64 ones.  complex64 sums of a warp meet in this form: the
// float64 pipe retires two lanes per clock per SM (16 clocks an instruction),
// a merge is 21 float32 instructions on a pipe of 128.
struct Sum3 {
    float hi = 0.f, mid = 0.f, lo = 0.f;
    static __device__ __forceinline__ float two_sum(float& a, float x) {
        const float s = __fadd_rn(a, x), bp = __fsub_rn(s, a);
        const float e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bp)), __fsub_rn(x, bp));
        a = s;
        return e;
    }
    __device__ __forceinline__ void add_mid(float x) { lo = __fadd_rn(lo, two_sum(mid, x)); }
    __device__ __forceinline__ void add_sq(float x) {
        const float p = __fmul_rn(x, x);
        add_mid(two_sum(hi, p));
        add_mid(__fmaf_rn(x, x, -p));
    }
};
__device__ __forceinline__ void merge(Sum3& a, const Sum3& b) {  // the same bits for (b, a)
    const float e = Sum3::two_sum(a.hi, b.hi), f = Sum3::two_sum(a.mid, b.mid), g = Sum3::two_sum(a.mid, e);
    a.lo = __fadd_rn(__fadd_rn(a.lo, b.lo), __fadd_rn(f, g));
}
__device__ __forceinline__ void merge(double& a, double b) { a += b; }
__device__ __forceinline__ Sum3 lane_xor(const Sum3& a, int o) {
    return {__shfl_xor_sync(0xffffffffu, a.hi, o), __shfl_xor_sync(0xffffffffu, a.mid, o),
            __shfl_xor_sync(0xffffffffu, a.lo, o)};
}
__device__ __forceinline__ double lane_xor(double a, int o) { return __shfl_xor_sync(0xffffffffu, a, o); }
__device__ __forceinline__ double value(const Sum3& a) { return (double)a.hi + ((double)a.mid + (double)a.lo); }
__device__ __forceinline__ double value(double a) { return a; }

// the warp's sum (every lane; fixed order)
template <class W> __device__ __forceinline__ double warp_sum(W a) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) merge(a, lane_xor(a, o));
    return value(a);
}

template <class R> struct Sum;
template <> struct Sum<double> {
    double s = 0.0;
    __device__ __forceinline__ void add_sq(double x, double y) { s += x * x + y * y; }
    __device__ __forceinline__ double wide() const { return s; }
};
// float-float pair (Knuth's TwoSum); the squares of float32 values enter
// exactly: x*x rounded plus its error fma(x, x, -x*x) (Dekker's product)
template <> struct Sum<float> {
    float hi = 0.f, lo = 0.f;
    __device__ __forceinline__ void add(float x) {
        float s = __fadd_rn(hi, x);
        float bp = __fsub_rn(s, hi);
        float e = __fadd_rn(__fsub_rn(hi, __fsub_rn(s, bp)), __fsub_rn(x, bp));
        hi = s;
        lo = __fadd_rn(lo, e);
    }
    __device__ __forceinline__ void add_sq(float x, float y) {
        const float px = __fmul_rn(x, x), py = __fmul_rn(y, y);
        const float ex = __fmaf_rn(x, x, -px), ey = __fmaf_rn(y, y, -py);
        add(px);
        add(py);
        lo = __fadd_rn(lo, __fadd_rn(ex, ey));
    }
    __device__ __forceinline__ Sum3 wide() const { return {hi, lo, 0.f}; }
};
// the sum of |psi_j|^2 over a block of 256 amplitudes, one warp, every lane:
// first the lane's amplitudes, pair(j) giving j and j + 1 (j even)
template <class Pair> __device__ __forceinline__ void block_load(float4 (&v)[4], Pair pair) {
#pragma unroll
    for (int k = 0; k < 4; ++k) v[k] = pair(2 * ((threadIdx.x & 31) + 32 * k));
}
__device__ __forceinline__ double block_sum(const float4 (&v)[4]) {
    Sum3 t;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        t.add_sq(v[k].x);
        t.add_sq(v[k].y);
        t.add_sq(v[k].z);
        t.add_sq(v[k].w);
    }
    return warp_sum(t);
}

// amplitudes j and j + 1 (j even): one 128-bit load where the state starts on
// a 16-byte boundary
__device__ __forceinline__ void add_pair(Sum<float>& a, float4 v) {
    a.add_sq(v.x, v.y);
    a.add_sq(v.z, v.w);
}
__device__ __forceinline__ float4 load_pair(const float2* g, bool aligned) {
    if (aligned) return *reinterpret_cast<const float4*>(g);
    const float2 x = g[0], y = g[1];
    return make_float4(x.x, x.y, y.x, y.y);
}

// lanes first, first + step, ... (in units of two amplitudes for complex64,
// one for complex128) of g[0..L): eight loads in flight
template <class R>
__device__ __forceinline__ void sum_strided(Sum<R>& a, const typename Cx<R>::T* g, int64_t L, int first, int step) {
    if constexpr (sizeof(R) == 4) {
        const bool aligned = (reinterpret_cast<uintptr_t>(g) & 15) == 0;
        const int64_t n = L / 2;  // L is a power of two, at least 2
        for (int64_t j0 = first; j0 < n; j0 += 8 * (int64_t)step) {
            float4 v[8];
#pragma unroll
            for (int k = 0; k < 8; ++k)
                if (j0 + k * (int64_t)step < n) v[k] = load_pair(g + 2 * (j0 + k * (int64_t)step), aligned);
#pragma unroll
            for (int k = 0; k < 8; ++k)
                if (j0 + k * (int64_t)step < n) add_pair(a, v[k]);
        }
    } else {
        for (int64_t j0 = first; j0 < L; j0 += 8 * (int64_t)step) {
            double2 v[8];
#pragma unroll
            for (int k = 0; k < 8; ++k)
                if (j0 + k * (int64_t)step < L) v[k] = g[j0 + k * (int64_t)step];
#pragma unroll
            for (int k = 0; k < 8; ++k)
                if (j0 + k * (int64_t)step < L) a.add_sq(v[k].x, v[k].y);
        }
    }
}

// sum of |psi_j|^2 over g[0..L), one warp, every lane
template <class R> __device__ __forceinline__ double chunk_sum_warp(const typename Cx<R>::T* g, int64_t L) {
    Sum<R> a;
    sum_strided<R>(a, g, L, threadIdx.x & 31, 32);
    return warp_sum(a.wide());
}

// chunks of at most this many amplitudes take a warp each (no block barrier,
// several chunks of a CTA in flight), longer ones a CTA
constexpr int64_t WARP_CHUNK = 4096;

// sum of |psi_j|^2 over g[0..L), whole CTA; result valid in thread 0
template <class R>
__device__ __forceinline__ double chunk_sum(const typename Cx<R>::T* g, int64_t L, double* sh32) {
    Sum<R> a;
    sum_strided<R>(a, g, L, threadIdx.x, blockDim.x);
    const double x = warp_sum(a.wide());
    __syncthreads();
    if ((threadIdx.x & 31) == 0) sh32[threadIdx.x >> 5] = x;
    __syncthreads();
    double s = 0.0;
    if (threadIdx.x == 0)
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += sh32[w];
    return s;
}

// every chunk sum of n_states states (item = state x chunk): put(item, sum)
// is called by one thread per item
template <class R, class State, class Put>
__device__ __forceinline__ void chunk_sums(int64_t items, int chunks, int64_t L, double* sh32, State state, Put put) {
    if (L <= WARP_CHUNK) {
        const int64_t nw = (int64_t)gridDim.x * (blockDim.x >> 5);
        for (int64_t it = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); it < items; it += nw) {
            const double s = chunk_sum_warp<R>(state(it / chunks) + (it % chunks) * L, L);
            if ((threadIdx.x & 31) == 0) put(it, s);
        }
    } else {
        for (int64_t it = blockIdx.x; it < items; it += gridDim.x) {
            const double s = chunk_sum<R>(state(it / chunks) + (it % chunks) * L, L, sh32);
            if (threadIdx.x == 0) put(it, s);
        }
    }
}

// running sum of sums[0..chunks) (stride `stride` doubles) into cum (same
// stride), one warp
__device__ __forceinline__ void chunk_cum(const double* sums, double* cum, int chunks, int stride) {
    const int lane = threadIdx.x & 31;
    const int per = (chunks + 31) / 32;
    const int c0 = lane * per, c1 = min(c0 + per, chunks);
    double t = 0.0;
    for (int c = c0; c < c1; ++c) t += sums[(int64_t)c * stride];
    double incl = t;
    for (int o = 1; o < 32; o <<= 1) {
        const double y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    double run = incl - t;
    for (int c = c0; c < c1; ++c) {
        run += sums[(int64_t)c * stride];
        cum[(int64_t)c * stride] = run;
    }
}

// one key for draw u from the state g (whole warp; result in every lane);
// BLOCKS: the caller has the block_sums of the draw's chunk, but for its last
template <class R, bool BLOCKS = false>
__device__ __forceinline__ int64_t sample_warp(const typename Cx<R>::T* g, int64_t dim, int chunks,
                                               const double* cum, int stride, double u, double* lo_out,
                                               double* hi_out, const double* blocks = nullptr) {
    using T = typename Cx<R>::T;
    const int lane = threadIdx.x & 31;
    const int64_t L = dim / chunks;
    // chunk: first c with u < cum[c], coarse blocks of 32 then within; a
    // lone chunk is searched as it is
    int c = chunks > 1 ? chunks : 0;
    if (chunks > 1) {
        const int nb = (chunks + 31) / 32;
        int blk = nb;
        for (int b0 = 0; b0 < nb && blk == nb; b0 += 32) {
            const int bi = b0 + lane;
            const int last = min(bi * 32 + 31, chunks - 1);
            const bool hit = bi < nb && u < cum[(int64_t)last * stride];
            const unsigned m = __ballot_sync(0xffffffffu, hit);
            if (m) blk = b0 + __ffs(m) - 1;
        }
        if (blk < nb) {
            const int ci = blk * 32 + lane;
            const bool hit = ci < chunks && u < cum[(int64_t)ci * stride];
            const unsigned m = __ballot_sync(0xffffffffu, hit);
            if (m) c = blk * 32 + __ffs(m) - 1;
        }
    }
    int64_t key = -1;
    double lo = 0.0, hi = 0.0;
    if (c < chunks) {
        double acc = c ? cum[(int64_t)(c - 1) * stride] : 0.0;
        const int64_t j0 = (int64_t)c * L;
        // (complex64) a block's amplitudes are on their way while the one
        // before it is summed
        float4 v[4];
        auto load = [&](float4 (&w)[4], int64_t blk) {
            if constexpr (sizeof(R) == 4 && !BLOCKS) {
                const typename Cx<R>::T* gb = g + j0 + blk;
                const bool aligned = (reinterpret_cast<uintptr_t>(gb) & 15) == 0;
                block_load(w, [&](int j) { return load_pair(gb + j, aligned); });
            }
        };
        if (L > 256) load(v, 0);
        for (int64_t blk = 0; blk < L && key < 0; blk += 256) {
            if constexpr (sizeof(R) == 4) {
                // the block's total (some 500 float32 instructions, where
                // float64 takes 45 of 16 clocks); the running sums below
                // only for the block that holds the draw
                if (blk + 256 < L) {
                    double tot;
                    float4 next[4];
                    if constexpr (BLOCKS) {
                        tot = blocks[blk / 256];
                    } else {
                        load(next, blk + 256);
                        tot = block_sum(v);
                    }
                    if (!(u < acc + tot)) {
                        acc += tot;
                        if constexpr (!BLOCKS)
#pragma unroll
                            for (int k = 0; k < 4; ++k) v[k] = next[k];
                        continue;
                    }
                }
            }
            double pe[8];
            double tot = 0.0;
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const int64_t j = blk + lane * 8 + e;
                double p = 0.0;
                if (j < L) {
                    const T v = g[j0 + j];
                    p = (double)v.x * (double)v.x + (double)v.y * (double)v.y;
                }
                pe[e] = p;
                tot += p;
            }
            double incl = tot;
            for (int o = 1; o < 32; o <<= 1) {
                const double y = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += y;
            }
            const double base = acc + (incl - tot);
            const unsigned m = __ballot_sync(0xffffffffu, u < acc + incl);
            if (m) {
                const int f = __ffs(m) - 1;
                int64_t k = -1;
                double h = 0.0, l = 0.0;
                if (lane == f) {
                    double run = base;
#pragma unroll
                    for (int e = 0; e < 8; ++e) {
                        const double before = run;
                        run += pe[e];
                        if (k < 0 && u < run && blk + lane * 8 + e < L) {
                            k = j0 + blk + lane * 8 + e;
                            l = before;
                            h = run;
                        }
                    }
                }
                key = __shfl_sync(0xffffffffu, k, f);
                lo = __shfl_sync(0xffffffffu, l, f);
                hi = __shfl_sync(0xffffffffu, h, f);
            }
            acc += __shfl_sync(0xffffffffu, incl, 31);
        }
    }
    if (key < 0) {  // u at or past the rounded total: the last nonzero entry
        const double total = cum[(int64_t)(chunks - 1) * stride];
        for (int64_t top = dim; top > 0 && key < 0; top -= 32) {
            const int64_t j = top - 32 + lane;
            double p = 0.0;
            if (j >= 0) {
                const T v = g[j];
                p = (double)v.x * (double)v.x + (double)v.y * (double)v.y;
            }
            const unsigned m = __ballot_sync(0xffffffffu, j >= 0 && p > 0);
            if (m) {
                const int f = 31 - __clz(m);
                key = top - 32 + f;
                const double pf = __shfl_sync(0xffffffffu, p, f);
                hi = total;
                lo = total - pf;
            }
        }
        if (key < 0) key = dim - 1;
    }
    *lo_out = lo;
    *hi_out = hi;
    return key;
}

}  // namespace svs
