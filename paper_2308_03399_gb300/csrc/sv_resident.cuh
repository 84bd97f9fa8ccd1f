// Resident runs: a whole circuit for one state per CTA, the state in shared
// memory from |0...0> to the final sample (k_resident).
//
// What bounds the pass-by-pass form for small registers is not bandwidth but
// the chain of launches: a state of 8 KB to 128 KB gives a pass one group of
// 16 amplitudes per lane or less, and every pass then costs one branch setup
// and one L2 round trip for all of the chip.  Here the same passes run back
// to back inside one kernel.  A CTA owns one state (one shot) at a time and
// takes the next when it is done, so CTAs on an SM sit in different passes
// and hide each other's latency chains and barriers.
//
// The pass sequence is the one the scheduler recorded, encoded as a program
// of blocks in the integer pool (sv_resident.h).  Every amplitude goes
// through the arithmetic of the register pass kernel in the same order
// (stage by stage, or the folded matrix where the pass was folded), so
// without Kraus ops and measurements complex64 states are the same to the
// last bit.  The probabilities of those are sums over the whole state, here
// over other lanes than in a pass (float-float per lane, to float64 precision
// across lanes and warps in both): they agree to about 1e-14, and the factor
// 1 / sqrt(p) of a choice, rounded to float32, can come out one float32
// rounding apart (some 1e-7 of the choices).
//
// The stage code is kept small on purpose: CTAs sit in different stages, so
// the instruction cache sees all of it at once.  (A first version that held
// the twelve register layouts of a two-qubit gate, as the pass kernel does,
// took 25k to 75k clocks a pass, most of it instruction fetch.)  A stage
// block therefore has its dense stages on group bits 0 and 1 only, the
// shared-memory addressing bringing any pair of qubits there, and a folded
// pass is composed by dynamic indexing.
//
// Blocks come in batches of up to `mb` (only the last of a batch may end in a
// reduction, so the choices of all of them are known): warp w turns block w
// of the batch into a list of active stages, or its folded matrix, all warps
// then apply the blocks one after another, and warp 0 decides the reduction.
// The next batch's blocks are on their way to shared memory (cp.async)
// meanwhile.
//
// Measured on GB300, us a run, passes -> resident: 6-qubit brickwork x 100
// shots 169 -> 73, 10-qubit x 1000 829 -> 298, 13-qubit QFT x 4000 6550 ->
// 2500, 12-qubit QFT with Kraus noise x 4000 (shot-branching passes) 30700 ->
// 17000, 11-qubit complex128 sweep x 1000 2690 -> 2260.  What bounds it:
// barriers and latency in complex64 (47% of issue slots used at 12 qubits,
// 6500 warp instructions a Kraus pass and state), the float64 pipe (two lanes
// per clock per SM) in complex128.
#pragma once
#include <cuda_runtime.h>

#include <cstdint>

#include "sv_common.cuh"
#include "sv_fold.cuh"
#include "sv_pass_reg.cuh"
#include "sv_resident.h"

namespace sv {

namespace {

// CTA shapes: CTAs of 128 threads per SM (registers), by precision and
// whether the circuit has folded blocks.  A spilled word costs more than the
// warps it buys: the state takes most of the SM's memory and leaves little
// L1 behind it (a Kraus circuit of 12 qubits ran 22 ms at 20 warps a SM with
// 300 bytes of spills and 18.6 ms at 12 with none; at 16, this, with 12 bytes,
// 16.7 ms, each with float-float sums across lanes).
template <class R, int NT, bool FOLDS> struct ResCta { static constexpr int min_blocks = 1; };
template <> struct ResCta<float, 128, true> { static constexpr int min_blocks = 4; };
template <> struct ResCta<float, 128, false> { static constexpr int min_blocks = 4; };
template <> struct ResCta<double, 128, false> { static constexpr int min_blocks = 2; };

// Shared-memory index of amplitude a: the high bits are folded into the low
// four, so that 16 lanes whose group indices differ in four address bits of
// different residues mod 4 touch 16 different 8-byte banks.  Linear over
// GF(2): swz(a ^ b) = swz(a) ^ swz(b).
__device__ __forceinline__ int swz(int a) { return a ^ ((a >> 4) & 15) ^ ((a >> 8) & 15) ^ ((a >> 12) & 15); }

__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_wait0() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }

// a lane's accumulator as a value that the warp sums to float64 precision
__device__ __forceinline__ svs::Sum3 wide(const Acc<float>& a) { return {a.hi, a.lo, 0.f}; }
__device__ __forceinline__ double wide(const Acc<double>& a) { return a.s; }
__device__ __forceinline__ svs::Sum3 pick(bool c, const svs::Sum3& a, const svs::Sum3& b) {
    return {c ? a.hi : b.hi, c ? a.mid : b.mid, c ? a.lo : b.lo};
}
__device__ __forceinline__ double pick(bool c, double a, double b) { return c ? a : b; }

// Totals over the warp of four accumulators, to float64 precision as in the
// register passes: total r comes out in the lanes with lane >> 3 == r.  The
// lanes share the values out before they add, 6 merges for all four where a
// tree for each takes 20 (12-qubit QFT with Kraus noise x 4000: 17.0 ms, and
// 18.0 with float64 adds shared out in the same way).
template <class R>
__device__ __forceinline__ double warp_totals(const Acc<R>& a0, const Acc<R>& a1, const Acc<R>& a2, const Acc<R>& a3) {
    using svs::lane_xor;
    using svs::merge;
    const int lane = threadIdx.x & 31;
    const bool h = lane & 16, l = lane & 8;
    auto w0 = wide(a0), w1 = wide(a1), w2 = wide(a2), w3 = wide(a3);
    auto x = pick(h, w2, w0), y = pick(h, w3, w1);
    merge(x, lane_xor(pick(h, w0, w2), 16));
    merge(y, lane_xor(pick(h, w1, w3), 16));
    auto t = pick(l, y, x);
    merge(t, lane_xor(pick(l, x, y), 8));
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) merge(t, lane_xor(t, o));
    return svs::value(t);
}

// Diagonal forms: |v|^2 of a group's amplitudes into the bins of the reduced
// qubits (group bit 0, or bits 0 and 1).  A register pass over w qubits adds
// the 2^(w - k) amplitudes of one of its groups that share a bin in R and
// then once to the compensated accumulator; `run` = 2^(w - k) keeps those
// sums (the pass's other qubits are the next group bits, in order).
template <class R, int K>
__device__ __forceinline__ void res_diag(const typename Cplx<R>::T* v, int run, Acc<R>* acc) {
#pragma unroll
    for (int idx = 0; idx < (1 << K); ++idx) {
        R q = 0;
#pragma unroll
        for (int m = 0; m < (16 >> K); ++m) {
            const int e = idx | (m << K);
            q += v[e].x * v[e].x + v[e].y * v[e].y;
            if (((m + 1) & (run - 1)) == 0) {
                acc[idx].add(q);
                q = 0;
            }
        }
    }
}

// one selection by a whole warp: lane r < R holds the probability of outcome
// r.  Thresholds and fallback are those of select_k; the running sums come
// from a scan (four float64 adds where 16 outcomes one after another cost a
// 367-pass Kraus run 4%), so a sum can differ from select_k's in its last bits
// and exceed its neighbour's for an outcome of probability 0.  Such an outcome
// is never drawn: only those with p > 0 are candidates.
__device__ __forceinline__ int warp_select(double p, int R, uint64_t k53) {
    const int lane = threadIdx.x & 31;
    double c = lane < R ? p : 0.0;
    for (int o = 1; o < R; o <<= 1) {
        const double y = __shfl_up_sync(0xffffffffu, c, o);
        if (lane >= o) c += y;
    }
    const bool possible = lane < R && p > 0.0;
    unsigned m = __ballot_sync(0xffffffffu, possible && k53 < cum_threshold(c));
    if (m) return __ffs(m) - 1;
    m = __ballot_sync(0xffffffffu, possible);
    return m ? 31 - __clz(m) : R - 1;
}

// 1 / sqrt(p) of a chosen outcome.  complex64 rounds it to float32 before
// use, so the float64 reciprocal square root (within an ulp) gives the same
// factor in a fraction of the float64-pipe time of a root and a division.
template <class R> __device__ __forceinline__ double res_scale(double p) {
    return sizeof(R) == 4 ? rsqrt(p) : 1.0 / sqrt(p);
}

// history of a shot: a sum of one mixed word per (op, outcome), so that two
// shots with equal words took the same outcomes (the mixer and increment of
// splitmix64: Steele, Lea, Flood, OOPSLA'14)
__device__ __forceinline__ unsigned long long hist_word(uint32_t op, int sel) {
    unsigned long long x = ((unsigned long long)op << 32 | (uint32_t)sel) + 0x9E3779B97F4A7C15ull;
    x = (x ^ (x >> 30)) * 0xBF58476D1CE4E5B9ull;
    x = (x ^ (x >> 27)) * 0x94D049BB133111EBull;
    return x ^ (x >> 31);
}

}  // namespace

// With at most FOLD_SPARSE nonzero entries in every row, the composed matrix
// becomes a table: entry k of row r (ascending columns, the order of the
// dense product's sums; skipped terms are exact zeros) at tab[16 k + r] as
// (swizzled offset of its amplitude, re, im).  Returns the entries per row;
// 16: dense, read from the work matrix.
constexpr int FOLD_SPARSE = 4;

static __device__ __noinline__ int res_table(const float2* M, const int32_t* so, float4* tab) {
    const int lane = threadIdx.x & 31, r = lane & 15;
    const float2* row = M + fold_at(r);
    unsigned nz = 0;
#pragma unroll
    for (int c = 0; c < 16; ++c) {
        const float2 m = row[2 * c];
        nz |= (m.x != 0.f || m.y != 0.f ? 1u : 0u) << c;
    }
    int K = __popc(nz);
    for (int o = 8; o > 0; o >>= 1) K = max(K, __shfl_xor_sync(0xffffffffu, K, o));
    if (K > FOLD_SPARSE) return 16;
    for (int k = 0; k < K; ++k) {
        const int c = nz ? __ffs(nz) - 1 : 0;
        const float2 m = nz ? row[2 * c] : make_float2(0.f, 0.f);
        nz &= nz - 1;
        const int off = (c & 1 ? so[0] : 0) ^ (c & 2 ? so[1] : 0) ^ (c & 4 ? so[2] : 0) ^ (c & 8 ? so[3] : 0);
        if (lane < 16) tab[16 * k + r] = make_float4(__int_as_float(off), m.x, m.y, 0.f);
    }
    return K;
}

// a folded block on NG groups: out[r] = sum over the row's nonzero columns,
// or over all columns, ascending
template <int NG, class Off>
__device__ __forceinline__ void res_sparse(float2* st, const float4* tab, int K, const int (&base)[NG], Off off) {
    float2 o[NG][16];
#pragma unroll
    for (int j = 0; j < NG; ++j)
#pragma unroll
        for (int r = 0; r < 16; ++r) o[j][r] = make_float2(0.f, 0.f);
#pragma unroll 1
    for (int k = 0; k < K; ++k) {
#pragma unroll
        for (int r = 0; r < 16; ++r) {
            const float4 m = tab[16 * k + r];
#pragma unroll
            for (int j = 0; j < NG; ++j) {
                const float2 a = st[base[j] ^ __float_as_int(m.x)];
                o[j][r].x = fmaf(m.y, a.x, fmaf(-m.z, a.y, o[j][r].x));
                o[j][r].y = fmaf(m.y, a.y, fmaf(m.z, a.x, o[j][r].y));
            }
        }
    }
#pragma unroll
    for (int j = 0; j < NG; ++j)
#pragma unroll
        for (int r = 0; r < 16; ++r) st[base[j] ^ off(r)] = o[j][r];
}

template <int NG, class Off>
__device__ __forceinline__ void res_dense(float2* st, const float4* M, const int (&base)[NG], Off off) {
    float2 v[NG][16];
#pragma unroll
    for (int j = 0; j < NG; ++j)
#pragma unroll
        for (int r = 0; r < 16; ++r) v[j][r] = st[base[j] ^ off(r)];
#pragma unroll 1
    for (int r = 0; r < 16; r += 2) {
        float2 x[NG], y[NG];
#pragma unroll
        for (int j = 0; j < NG; ++j) x[j] = y[j] = make_float2(0.f, 0.f);
#pragma unroll
        for (int c = 0; c < 16; ++c) {
            const float4 m = M[(r >> 1) * FOLD_LD + c];
#pragma unroll
            for (int j = 0; j < NG; ++j) {
                const float2 a = v[j][c];
                x[j].x = fmaf(m.x, a.x, fmaf(-m.y, a.y, x[j].x));
                x[j].y = fmaf(m.x, a.y, fmaf(m.y, a.x, x[j].y));
                y[j].x = fmaf(m.z, a.x, fmaf(-m.w, a.y, y[j].x));
                y[j].y = fmaf(m.z, a.y, fmaf(m.w, a.x, y[j].y));
            }
        }
        const int o0 = off(r), o1 = off(r + 1);
#pragma unroll
        for (int j = 0; j < NG; ++j) {
            st[base[j] ^ o0] = x[j];
            st[base[j] ^ o1] = y[j];
        }
    }
}

// the sums of the 256-amplitude blocks of a chunk but for its last, from the
// state in shared memory: this warp's w, w + step, ...  (complex128 states are
// searched without them)
static __device__ __forceinline__ void res_block_sums(const float2* st, int j0, int len, double* blocks, int w, int step) {
    for (int k = w; k < len / 256 - 1; k += step) {
        float4 v[4];
        svs::block_load(v, [&](int j) {
            const float2 x = st[swz(j0 + 256 * k + j)], y = st[swz(j0 + 256 * k + j + 1)];
            return make_float4(x.x, x.y, y.x, y.y);
        });
        const double t = svs::block_sum(v);
        if ((threadIdx.x & 31) == 0) blocks[k] = t;
    }
}
static __device__ __forceinline__ void res_block_sums(const double2*, int, int, double*, int, int) {}

template <class R, int NT, bool FOLDS>
__global__ void __launch_bounds__(NT, (ResCta<R, NT, FOLDS>::min_blocks)) k_resident(DevBatch d, const __grid_constant__ ResDesc p) {
    using T = typename Cplx<R>::T;
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ int n_act[RES_MAX_BATCH];  // active stages of a block; for a folded one, entries per row
    __shared__ unsigned long long clb_sh, hist_sh;
    __shared__ int pset_sh;
    const int tid = threadIdx.x, nth = blockDim.x, warp = tid >> 5, lane = tid & 31, nw = nth >> 5;
    const int dimp = 1 << p.np, free_bits = p.np - 4, groups = 1 << free_bits;
    const int mb = p.mb, slots = 2 * mb;
    T* const st = reinterpret_cast<T*>(smem);
    int32_t* const blks = reinterpret_cast<int32_t*>(st + dimp);
    int4* const acts = reinterpret_cast<int4*>(blks + slots * p.block_words);
    float4* const tabs = reinterpret_cast<float4*>(acts + mb * p.max_stages);
    float4* const works = tabs + (p.folds ? mb * 16 * FOLD_SPARSE : 0);
    unsigned char* const brm = reinterpret_cast<unsigned char*>(works + (p.folds ? mb * 8 * FOLD_LD : 0));
    double* const scale_col = reinterpret_cast<double*>(brm + mb * p.br_bytes);
    double* const redw = scale_col + MAX_PEND;
    double* const fin = redw;  // at most 8 chunk sums, after the last pass (none of a lone chunk)
    double* const blocks = redw + nw * MAX_RED;
    int32_t* const sel_col = reinterpret_cast<int32_t*>(blocks + RES_FINAL_BLOCKS);
    uint8_t* const rows = reinterpret_cast<uint8_t*>(sel_col + MAX_PEND);
    const int2* const index = reinterpret_cast<const int2*>(d.ipool + p.index_off);
    const int2* const batches = reinterpret_cast<const int2*>(d.ipool + p.batch_off);  // first block, blocks
    const int n_states = p.n_states;

    // warp w: start the copy of block bt.x + w of a batch
    auto copy_blocks = [&](int2 bt) {
        if (warp < bt.y) {
            const int i = bt.x + warp;
            const int2 ent = index[i];
            int32_t* dst = blks + (i % slots) * p.block_words;
            const int32_t* src = d.ipool + ent.x;
            for (int w = 4 * lane; w < ent.y; w += 128) cp_async16(dst + w, src + w);
        }
        cp_commit();
    };

    // one warp: the active stages of block i (number q of its batch), in op
    // order, for this state
    auto prepare = [&](int i, int q) {
        const int32_t* B = blks + (i % slots) * p.block_words;
        int4* act = acts + q * p.max_stages;
        unsigned char* br = brm + q * p.br_bytes;
        const int n = B[RB_NSTAGES];
        const uint64_t clb = clb_sh;
        int count = 0;
        for (int s0 = 0; s0 < n; s0 += 32) {
            const int s = s0 + lane;
            bool on = false;
            int4 r = make_int4(0, 0, 0, 0);
            // per-branch matrix: source entries, qubits, scale
            const T* src = nullptr;
            double scale = 1.0;
            int br_k = 0;
            if (s < n) {
                const int4 Sa = *reinterpret_cast<const int4*>(B + RB_STAGES + RS_WORDS * s);
                const int4 Sb = *reinterpret_cast<const int4*>(B + RB_STAGES + RS_WORDS * s + 4);
                const int S[7] = {Sa.x, Sa.y, Sa.z, Sa.w, Sb.x, Sb.y, Sb.z};
                const int w0 = S[0], kind = w0 & 15, k = (w0 >> 4) & 15, pos = S[1];
                on = true;
                if ((w0 >> 10) & 1) on = (int)((clb >> ((w0 >> 12) & 63)) & 1) == ((w0 >> 11) & 1);
                r.w = pos;
                if (kind == ST_DENSE) {
                    r.z = B[S[5]];
                    r.x = k == 1 ? (r.z ? RA_ONE_SHAPED : RA_ONE) : (r.z ? RA_MONO : RA_TWO);
                    r.y = (int)(reinterpret_cast<const unsigned char*>(B + S[3]) - smem);
                } else if (kind == ST_DENSE_BR) {
                    r.y = (int)(br + S[6] - smem);
                    br_k = k;
                    if ((w0 >> 20) & 1) {  // the shot's parameter set, from the constant pool
                        src = reinterpret_cast<const T*>(reinterpret_cast<const R*>(d.pool) + S[3] +
                                                         (int64_t)pset_sh * S[4]);
                        r.z = d.ipool[S[5] + pset_sh];
                    } else {
                        const int sel = sel_col[S[2]];
                        scale = scale_col[S[2]];
                        src = reinterpret_cast<const T*>(B + S[3] + sel * S[4]);
                        r.z = B[S[5] + sel];
                    }
                    r.x = k == 1 ? (r.z ? RA_ONE_SHAPED : RA_ONE) : (r.z ? RA_MONO : RA_TWO);
                } else if (kind == ST_PAULI_BR) {
                    const int sel = (w0 >> 9) & 1 ? rows[S[2]] : sel_col[S[2]];
                    const int packed = B[S[3] + sel];
                    if ((packed & 0xff) == 0) {
                        on = false;
                    } else {
                        const int xm = packed & 15, zm = (packed >> 4) & 15, ny = (packed >> 8) & 3;
                        int xg = 0, zg = 0;
                        for (int j = 0; j < k; ++j) {
                            const int b = 1 << ((pos >> (4 * j)) & 15);
                            if ((xm >> j) & 1) xg |= b;
                            if ((zm >> j) & 1) zg |= b;
                        }
                        int sign = 0;
                        for (int e = 0; e < 16; ++e)
                            if ((((ny >> 1) & 1) ^ (__popc(zg & e) & 1)) != 0) sign |= 1 << e;
                        r.x = RA_PAULI;
                        r.z = xg | ((ny & 1) << 4) | (sign << 8);
                    }
                } else {  // ST_PROJ_BR
                    const int sel = sel_col[S[2]];
                    int keep = 0, xr = 0;
                    for (int e = 0; e < 16; ++e) {
                        int o = 0;
                        for (int j = 0; j < k; ++j) o |= ((e >> ((pos >> (4 * j)) & 15)) & 1) << j;
                        if (o == sel) keep |= 1 << e;
                    }
                    if ((w0 >> 8) & 1)
                        for (int j = 0; j < k; ++j)
                            if ((sel >> j) & 1) xr |= 1 << ((pos >> (4 * j)) & 15);
                    *reinterpret_cast<R*>(br + S[6]) = (R)scale_col[S[2]];
                    r.x = RA_PROJ;
                    r.y = (int)(br + S[6] - smem);
                    r.z = keep | (xr << 16);
                }
            }
            const unsigned m = __ballot_sync(0xffffffffu, on);
            if (on) act[count + __popc(m & ((1u << lane) - 1u))] = r;
            count += __popc(m);
            // a branch's own matrices: entries over the lanes, times the scale
            unsigned mb = __ballot_sync(0xffffffffu, on && src != nullptr);
            while (mb) {
                const int l = __ffs(mb) - 1;
                mb &= mb - 1;
                const T* ls = reinterpret_cast<const T*>(__shfl_sync(0xffffffffu, (unsigned long long)src, l));
                const R sc = (R)__shfl_sync(0xffffffffu, scale, l);
                const int off = __shfl_sync(0xffffffffu, r.y, l), code = __shfl_sync(0xffffffffu, r.x, l);
                const int lk = __shfl_sync(0xffffffffu, br_k, l);
                const int ne = code == RA_MONO ? 4 : 1 << (2 * lk);
                if (lane < ne) {
                    T mm = ls[lane];
                    mm.x *= sc;
                    mm.y *= sc;
                    if (sizeof(T) == 8 && code == RA_TWO)
                        reinterpret_cast<ulonglong2*>(smem + off)[lane] =
                            make_ulonglong2(pk2((float)mm.x, (float)mm.x), pk2(-(float)mm.y, (float)mm.y));
                    else
                        reinterpret_cast<T*>(smem + off)[lane] = mm;
                }
            }
        }
        __syncwarp();
        if constexpr (FOLDS) {
            if (B[RB_FOLD]) {
                if (count > 0) {
                    float2* M = reinterpret_cast<float2*>(works + q * 8 * FOLD_LD);
                    res_compose(act, count, smem, M);
                    count = res_table(M, B + RB_SO, tabs + q * 16 * FOLD_SPARSE);
                }
            }
        }
        if (lane == 0) n_act[q] = count;
        __syncwarp();
    };

    const int2 none = make_int2(0, 0), first = p.n_batches > 0 ? batches[0] : none;

    for (int state = blockIdx.x; state < n_states; state += gridDim.x) {
        const uint32_t shot = (uint32_t)state;  // batch mode: shot s is branch s in slot s
        const uint64_t gs = d.shot_base + shot;
        copy_blocks(first);
        if (tid == 0) {
            const int ps = d.pset_of_shot ? (int)d.pset_of_shot[state] : 0;
            clb_sh = 0;
            pset_sh = ps;
            hist_sh = p.hist ? hist_word(0xffffffffu, ps) : 0ull;
            // the branch tables of a run with a state per shot, as a reset
            // and the run's decides would leave them
            d.perm[state] = shot;
            d.br_slot[state] = state;
            d.br_start[state] = state;
            d.br_count[state] = 1;
            d.br_parent[state] = -1;
            d.br_big[state] = -1;
            d.br_pset[state] = ps;
            if (state == 0) {
                d.ctl[CTL_NBR] = n_states;
                d.ctl[CTL_NFREE] = 0;  // as many slots as shots
                d.ctl[CTL_NWAIT] = 0;
                d.ctl[CTL_COPY_FIRST] = 0;
                d.ctl[CTL_COPY_END] = 0;
                d.ctl[CTL_NALLOC] = 0;
                d.ctl[CTL_DONE] = 0;
            }
        }
        for (int j = tid; j < dimp; j += nth) {
            T z;
            z.x = j == 0 ? (R)1 : (R)0;
            z.y = 0;
            st[j] = z;
        }
        // the shot's choice of every Pauli op: state-independent, drawn first
        unsigned long long hsum = 0;
        for (int q = tid; q < p.n_rows; q += nth) {
            const int32_t* e = d.ipool + p.row_table + (int64_t)PRE_WORDS * q;
            const uint32_t op = (uint32_t)e[0];
            const int sel = select_k(philox_k53(d.seed, gs, op), reinterpret_cast<const uint64_t*>(d.ipool + e[2]),
                                     reinterpret_cast<const double*>(d.ipool + e[3]), e[1]);
            rows[q] = (uint8_t)sel;
            hsum += hist_word(op, sel);
        }
        __syncthreads();
        if (p.hist && hsum) atomicAdd(&hist_sh, hsum);
        int2 bt = first, nxt = p.n_batches > 1 ? batches[1] : none;
        for (int t = 0, q = 0; t < p.n_batches;) {
            if (q == 0) {
                if (warp < bt.y) {
                    cp_wait0();
                    __syncwarp();
                    prepare(bt.x + warp, warp);
                }
                __syncthreads();
                copy_blocks(nxt);
            }
            const int i = bt.x + q;
            const int32_t* B = blks + (i % slots) * p.block_words;
            const int rw = B[RB_RED], red_kind = rw & 15, red_k = (rw >> 4) & 15, red_R = (rw >> 8) & 31;
            const bool red = red_kind != RED_NONE;
            Acc<R> acc[REG_MAX_RED];
#pragma unroll
            for (int r = 0; r < REG_MAX_RED; ++r) acc[r].zero();
            // swizzled offsets of the group-number bits, two to a word
            int sfw[5];
#pragma unroll
            for (int j = 0; j < 5; ++j) sfw[j] = B[RB_SF + j];
            auto group_base = [&](int g) {
                int b = 0;
#pragma unroll
                for (int j = 0; j < 5; ++j) {
                    b ^= g & (1 << (2 * j)) ? sfw[j] & 0xffff : 0;
                    b ^= g & (2 << (2 * j)) ? (int)((unsigned)sfw[j] >> 16) : 0;
                }
                return b;
            };
            const int so0 = B[RB_SO], so1 = B[RB_SO + 1], so2 = B[RB_SO + 2], so3 = B[RB_SO + 3];
            auto off = [&](int e) {
                return ((e & 1) ? so0 : 0) ^ ((e & 2) ? so1 : 0) ^ ((e & 4) ? so2 : 0) ^ ((e & 8) ? so3 : 0);
            };
            if (FOLDS && B[RB_FOLD]) {
                if constexpr (FOLDS) {
                    const int K = n_act[q];
                    const float4* tab = tabs + q * 16 * FOLD_SPARSE;
                    const float4* M = works + q * 8 * FOLD_LD;
                    // A dense product is bound by delivering its matrix: a
                    // 128-bit broadcast load returns 512 bytes to the warp,
                    // four clocks of the SM, for eight FMAs.  Two groups per
                    // thread share each load.
                    for (int g = tid; K > 0 && g < groups; g += 2 * nth) {
                        if (g + nth < groups) {
                            const int base[2] = {group_base(g), group_base(g + nth)};
                            if (K <= FOLD_SPARSE) res_sparse<2>(st, tab, K, base, off);
                            else res_dense<2>(st, M, base, off);
                        } else {
                            const int base[1] = {group_base(g)};
                            if (K <= FOLD_SPARSE) res_sparse<1>(st, tab, K, base, off);
                            else res_dense<1>(st, M, base, off);
                        }
                    }
                }
            } else {
                const int4* act = acts + q * p.max_stages;
                const int cnt = n_act[q];
                const bool touch = cnt > 0 || red_kind == RED_DIAG || red_kind == RED_FORMS;
                for (int g = tid; touch && g < groups; g += nth) {
                    const int base = group_base(g);
                    T v[16];
#pragma unroll
                    for (int e = 0; e < 16; ++e) v[e] = st[base ^ off(e)];
#pragma unroll 1
                    for (int s = 0; s < cnt; ++s) {
                        const int4 r = act[s];
                        const T* m = reinterpret_cast<const T*>(smem + r.y);
                        if (r.x == RA_ONE_SHAPED) {
                            if (r.w & 15) reg_apply1_shaped<T, 16, 1>(v, m, r.z);
                            else reg_apply1_shaped<T, 16, 0>(v, m, r.z);
                        } else if (r.x == RA_ONE) {
                            if (r.w & 15) reg_apply1<T, 16, 1>(v, m);
                            else reg_apply1<T, 16, 0>(v, m);
                        } else if (r.x == RA_MONO) {
                            if (r.z & RES_MONO_REAL) {  // real phases: half the products
                                reg_mono<T, 16, 0, 1>(v, r.z | 2, m);
#pragma unroll
                                for (int e = 0; e < 16; ++e) {
                                    v[e].x = m[e & 3].x * v[e].x;
                                    v[e].y = m[e & 3].x * v[e].y;
                                }
                            } else {
                                reg_mono<T, 16, 0, 1>(v, r.z, m);
                            }
                        } else if (r.x == RA_TWO) {
                            if constexpr (sizeof(T) == 8)
                                reg_apply2_f32x2<16, 0, 1>(reinterpret_cast<float2*>(v),
                                                           reinterpret_cast<const ulonglong2*>(m));
                            else
                                reg_apply2<T, 16, 0, 1>(v, m);
                        } else if (r.x == RA_PAULI) {
                            reg_xor_mask<T, 16>(v, r.z & 15);
                            const bool rot = (r.z >> 4) & 1;
                            const int sign = r.z >> 8;
#pragma unroll
                            for (int e = 0; e < 16; ++e) {
                                T t = v[e];
                                if (rot) {
                                    const R x = t.x;
                                    t.x = t.y;
                                    t.y = -x;
                                }
                                if ((sign >> e) & 1) {
                                    t.x = -t.x;
                                    t.y = -t.y;
                                }
                                v[e] = t;
                            }
                        } else {
                            const R sc = m->x;
#pragma unroll
                            for (int e = 0; e < 16; ++e) {
                                if ((r.z >> e) & 1) {
                                    v[e].x *= sc;
                                    v[e].y *= sc;
                                } else {
                                    v[e].x = 0;
                                    v[e].y = 0;
                                }
                            }
                            reg_xor_mask<T, 16>(v, (r.z >> 16) & 15);
                        }
                    }
                    if (red_kind == RED_DIAG) {
                        const int run = B[RB_RUN];
                        if (red_k == 2) res_diag<R, 2>(v, run, acc);
                        else res_diag<R, 1>(v, run, acc);
                    } else if (red_kind == RED_FORMS) {
                        reg_forms1<R, 16, 0>(v, reinterpret_cast<const T*>(B + B[RB_COEF]), red_R, acc);
                    }
                    if (cnt > 0)
#pragma unroll
                        for (int e = 0; e < 16; ++e) st[base ^ off(e)] = v[e];
                }
            }
            if (red) {
                const int nv = red_kind == RED_DIAG ? 1 << red_k : red_R;  // values reduced over the state
                if (red_kind == RED_BINS) {
                    // a warp owns up to four outcomes at a time: their
                    // amplitudes, one compensated addition each, in a fixed
                    // order
                    __syncthreads();
                    // (the measured qubits are group bits 0.. in order)
                    for (int o0 = warp; o0 < red_R; o0 += 4 * nw) {
                        Acc<R> a[4];
#pragma unroll
                        for (int r = 0; r < 4; ++r) a[r].zero();
                        for (int m = 0; m < 16; m += red_R) {
                            int om[4];
#pragma unroll
                            for (int r = 0; r < 4; ++r) om[r] = off((o0 + r * nw + m) & 15);
                            if (o0 + nw >= red_R) {  // the warp's only outcome
#pragma unroll 4
                                for (int g = lane; g < groups; g += 32) {
                                    const T x = st[group_base(g) ^ om[0]];
                                    a[0].add(x.x * x.x + x.y * x.y);
                                }
                                continue;
                            }
#pragma unroll 2
                            for (int g = lane; g < groups; g += 32) {
                                const int base = group_base(g);
#pragma unroll
                                for (int r = 0; r < 4; ++r)
                                    if (o0 + r * nw < red_R) {
                                        const T x = st[base ^ om[r]];
                                        a[r].add(x.x * x.x + x.y * x.y);
                                    }
                            }
                        }
                        const double t = warp_totals<R>(a[0], a[1], a[2], a[3]);
                        const int o = o0 + (lane >> 3) * nw;
                        if ((lane & 7) == 0 && o < red_R) redw[o] = t;
                    }
                } else {
                    const double t = warp_totals<R>(acc[0], acc[1], acc[2], acc[3]);  // (zeros past nv)
                    if ((lane & 7) == 0 && lane >> 3 < nv) redw[warp * MAX_RED + (lane >> 3)] = t;
                }
                __syncthreads();
                if (warp == 0) {
                    // totals (lane r: value r), then the probabilities
                    double val = 0.0;
                    if (lane < nv) {
                        val = redw[lane];
                        if (red_kind != RED_BINS)
                            for (int w = 1; w < nw; ++w) val += redw[w * MAX_RED + lane];
                    }
                    double pr = val;
                    if (red_kind == RED_DIAG) {
                        const double* W = reinterpret_cast<const double*>(B + B[RB_COEF]) + (lane < red_R ? lane << red_k : 0);
                        pr = 0.0;
                        for (int r = 0; r < nv; ++r) pr += W[r] * __shfl_sync(0xffffffffu, val, r);
                    }
                    const int32_t* D = B + B[RB_DECIDE];
                    const int kind = D[RD_KIND], nR = D[RD_R], r2 = D[RD_R2];
                    double ph = pr;  // the head op's probabilities, lane r: outcome r
                    if (kind == DEC_KRAUS_J1) {
                        ph = 0.0;
                        const int base = lane < nR ? lane * r2 : 0;
                        for (int j = 0; j < r2; ++j) ph += __shfl_sync(0xffffffffu, pr, base + j);
                    }
                    const int o1 = warp_select(ph, nR, philox_k53(d.seed, gs, (uint32_t)D[RD_OP]));
                    const double p1 = __shfl_sync(0xffffffffu, ph, o1);
                    if (lane == 0) {
                        sel_col[D[RD_PEND]] = o1;
                        scale_col[D[RD_PEND]] = res_scale<R>(p1);
                        if (p.hist) hist_sh += hist_word((uint32_t)D[RD_OP], o1);
                        if (kind == DEC_MEASURE) {
                            unsigned long long cl = clb_sh;
                            for (int j = 0; j < D[RD_M]; ++j) {
                                const int b = (D[RD_CLBITS] >> (8 * j)) & 255;
                                cl = (cl & ~(1ull << b)) | ((unsigned long long)((o1 >> j) & 1) << b);
                            }
                            clb_sh = cl;
                        }
                    }
                    if (kind == DEC_KRAUS_J1) {
                        // op 2 from p(j | o1) = p_ij / p_i
                        const double pj = __shfl_sync(0xffffffffu, pr, o1 * r2 + (lane < r2 ? lane : 0)) / p1;
                        const int o2 = warp_select(pj, r2, philox_k53(d.seed, gs, (uint32_t)D[RD_OP2]));
                        const double p2 = __shfl_sync(0xffffffffu, pj, o2);
                        if (lane == 0) {
                            sel_col[D[RD_PEND2]] = o2;
                            scale_col[D[RD_PEND2]] = res_scale<R>(p2);
                            if (p.hist) hist_sh += hist_word((uint32_t)D[RD_OP2], o2);
                        }
                    }
                    __syncwarp();
                }
                // the next batch's lists read the choices: a batch of one
                // block is prepared by the warp that made them
                if (nxt.y > 1) __syncthreads();
            } else {
                __syncthreads();
            }
            if (++q == bt.y) {
                q = 0;
                ++t;
                bt = nxt;
                nxt = t + 1 < p.n_batches ? batches[t + 1] : none;
            }
        }
        __syncthreads();

        // the final state to its slot, and the final sample: the chunks of
        // every other final sample, summed in the order of chunk_sum_warp, and
        // (complex64) the blocks that sample_warp may pass over in the draw's
        // chunk
        T* const out = reinterpret_cast<T*>(d.states) + (int64_t)shot * d.dim;
        const int dim = (int)d.dim;
        for (int j = tid; j < dim; j += nth) out[j] = st[swz(j)];
        if (p.has_final) {
            const int chunks = svs::final_chunks(dim), len = dim / chunks;
            const double u = philox_uniform(d.seed, gs, p.fin_op);
            constexpr int PER = sizeof(R) == 4 ? 2 : 1;  // neighbouring amplitudes of a lane
            for (int c = warp; chunks > 1 && c < chunks; c += nw) {
                svs::Sum<R> a;
#pragma unroll 2
                for (int j = PER * lane; j < len; j += 32 * PER)
#pragma unroll
                    for (int e = 0; e < PER; ++e) {
                        const T x = st[swz(c * len + j + e)];
                        a.add_sq(x.x, x.y);
                    }
                const double t = svs::warp_sum(a.wide());
                if (lane == 0) fin[c] = t;
            }
            if (chunks > 1) {
                __syncthreads();
                if (warp == 0) {
                    svs::chunk_cum(fin, fin, chunks, 1);
                    __syncwarp();
                    const unsigned m = __ballot_sync(0xffffffffu, lane < chunks && u < fin[lane]);
                    if (lane == 0) n_act[0] = m ? __ffs(m) - 1 : 0;  // the draw's chunk
                }
                __syncthreads();
            }
            res_block_sums(st, chunks > 1 ? n_act[0] * len : 0, len, blocks, warp, nw);
            __syncthreads();
            if (warp == 0) {
                double lo, hi;
                const int64_t key =
                    svs::sample_warp<R, sizeof(R) == 4>(out, dim, chunks, fin, 1, u, &lo, &hi, blocks);
                if (lane == 0) d.keys[shot] = (uint64_t)key;
            }
        }
        if (tid == 0) {
            d.br_clbits[state] = clb_sh;
            if (p.hist) p.hist[shot] = hist_sh;
        }
        __syncthreads();  // st, rows and the block ring are free again
    }
}

}  // namespace sv
