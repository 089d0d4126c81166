// tn_kernels.cu -- generic node kernel, renormalisation helpers and the FP64
// cross-slice accumulation of libtn.so (sm_103a).
//
// Semantics (arXiv 2002.01935):
//   * a pairwise contraction takes the inner product over the shared
//     labels, an outer product if there are none (Sec. 2);
//   * after each contraction the tensor is renormalised by a power of two
//     and the exponent is carried along (Sec. 4.2, active renormalisation);
//     here the scale is applied when the consumer reads the tensor: the
//     stored tensor S and exponent E mean S * 2^E, and a consumer multiplies
//     S by 2^-e, e = frexp exponent of max |component| of S, which is exact;
//   * the sliced contractions are summed in FP64 with exponent alignment
//     (Sec. 4.7.1).
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <cstring>
#include <type_traits>

#include "tn_internal.h"

namespace tn {

__device__ __forceinline__ int exp_of_max(const unsigned* slot) {
    if (slot == nullptr) return 0;
    float m = __uint_as_float(*slot);
    if (!(m > 0.f)) return 0;
    int e;
    frexpf(m, &e);
    return e;
}

__device__ __forceinline__ unsigned long long global_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ int64_t slice_offset(const SliceDigits& d, int64_t slice) {
    int64_t off = 0;
    for (int i = 0; i < d.n; ++i) off += ((slice / d.div[i]) % d.dim[i]) * d.stride[i];
    return off;
}

// Block-wide max of non-negative floats, folded into *slot with atomicMax
// on the float bit pattern (order-preserving for non-negative floats).
__device__ __forceinline__ void block_max_to(float v, unsigned* slot) {
    __shared__ float red[32];
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (lane == 0) red[w] = v;
    __syncthreads();
    if (w == 0) {
        int nw = (blockDim.x + 31) >> 5;
        v = lane < nw ? red[lane] : 0.f;
        for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
        if (lane == 0 && v > 0.f) atomicMax(slot, __float_as_uint(v));
    }
}

template <bool CPLX>
__global__ void __launch_bounds__(256) k_generic(const __grid_constant__ GenericArgs a) {
    // instance blockIdx.y: offset pointers, scale slots and slice id
    const int inst = blockIdx.y;
    const InstanceInfo& in = a.in;
    const int64_t slice = a.ctl->slice + (int64_t)inst * in.slice_step;
    if (slice >= a.ctl->slice_end) return;
    const int esz = CPLX ? 8 : 4;
    const void* Ap = (const char*)a.A + (int64_t)inst * in.a_is * esz;
    const void* Bp = (const char*)a.B + (int64_t)inst * in.b_is * esz;
    void* Cp = (char*)a.C + (int64_t)inst * in.c_is * esz;
    ScaleIO sc = a.sc;
    if (sc.max_a) sc.max_a += (int64_t)inst * in.sa_is;
    if (sc.exp_a) sc.exp_a += (int64_t)inst * in.sa_is;
    if (sc.max_b) sc.max_b += (int64_t)inst * in.sb_is;
    if (sc.exp_b) sc.exp_b += (int64_t)inst * in.sb_is;
    sc.max_c += (int64_t)inst * in.sc_is;
    sc.exp_c += (int64_t)inst * in.sc_is;
    const int eA = exp_of_max(sc.max_a);
    const int eB = exp_of_max(sc.max_b);
    const int esum = eA + eB;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        int64_t s = (sc.exp_a ? *sc.exp_a : 0) + (sc.exp_b ? *sc.exp_b : 0) + esum;
        *sc.exp_c = s;
    }
    const int64_t baseA = slice_offset(a.sla, slice);
    const int64_t baseB = slice_offset(a.slb, slice);
    float lmax = 0.f;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t o = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; o < a.n_out; o += stride) {
        int64_t ia = baseA, ib = baseB, rem = o;
        for (int i = 0; i < a.n_od; ++i) {
            int64_t d = a.od_dim[i];
            int64_t v = rem % d;
            rem /= d;
            ia += v * a.od_sa[i];
            ib += v * a.od_sb[i];
        }
        int cnt[kMaxDigits];
        for (int i = 0; i < a.n_kd; ++i) cnt[i] = 0;
        float re = 0.f, im = 0.f;
        for (int64_t k = 0; k < a.n_sum; ++k) {
            if (CPLX) {
                float2 x = reinterpret_cast<const float2*>(Ap)[ia];
                float2 y = reinterpret_cast<const float2*>(Bp)[ib];
                if (a.conj_a) x.y = -x.y;
                if (a.conj_b) y.y = -y.y;
                re = fmaf(x.x, y.x, re);
                re = fmaf(-x.y, y.y, re);
                im = fmaf(x.x, y.y, im);
                im = fmaf(x.y, y.x, im);
            } else {
                re = fmaf(reinterpret_cast<const float*>(Ap)[ia],
                          reinterpret_cast<const float*>(Bp)[ib], re);
            }
            for (int i = 0; i < a.n_kd; ++i) {
                ia += a.kd_sa[i];
                ib += a.kd_sb[i];
                if (++cnt[i] < a.kd_dim[i]) break;
                ia -= a.kd_sa[i] * a.kd_dim[i];
                ib -= a.kd_sb[i] * a.kd_dim[i];
                cnt[i] = 0;
            }
        }
        re = ldexpf(re, -esum);
        if (CPLX) {
            im = ldexpf(im, -esum);
            reinterpret_cast<float2*>(Cp)[o] = make_float2(re, im);
            lmax = fmaxf(lmax, fmaxf(fabsf(re), fabsf(im)));
        } else {
            reinterpret_cast<float*>(Cp)[o] = re;
            lmax = fmaxf(lmax, fabsf(re));
        }
    }
    block_max_to(lmax, sc.max_c);
    if (a.t_done && threadIdx.x == 0) atomicMax(a.t_done, global_ns());
}

int sm_count() {
    constexpr int kMaxDev = 64;
    static int cache[kMaxDev] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDev) {
        cudaGetLastError();
        return 152;
    }
    if (cache[dev] <= 0) {
        int n = 0;
        if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0) {
            cudaGetLastError();
            n = 152;
        }
        cache[dev] = n;
    }
    return cache[dev];
}

cudaError_t launch_generic(const GenericArgs& a, bool is_c, cudaStream_t s) {
    if (a.cfg) return launch_tile_any(a, is_c, s);
    int64_t blocks = (a.n_out + 255) / 256;
    if (blocks > sm_count() * 16) blocks = sm_count() * 16;
    if (blocks < 1) blocks = 1;
    const unsigned ni = a.in.n_inst > 1 ? (unsigned)a.in.n_inst : 1u;
    if (is_c)
        k_generic<true><<<dim3((unsigned)blocks, ni), 256, 0, s>>>(a);
    else
        k_generic<false><<<dim3((unsigned)blocks, ni), 256, 0, s>>>(a);
    return cudaGetLastError();
}

// --------------------------------------------------------------------------
// FP64 cross-slice accumulation (Sec. 4.7.1) with exponent alignment
// --------------------------------------------------------------------------

// Common part of the folds: the roots of one launch are slices ctl->slice + i
// (i < n, in order; zero roots and idle slices are skipped) and are folded
// with one common exponent.  The call's first group starts from zero instead
// of reading the accumulator, and (direct folds) its last group writes the
// caller's output instead of the accumulator: a call of one group, which is
// every unsliced one, moves each output once.
constexpr int kFoldInst = 64;  // instances whose maxima and exponents are kept in shared memory

struct FoldState {
    int64_t slice, slice_end, newE;
    double fa;         // factor of the accumulator
    int n;             // instances of this group that are live
    int par;
    bool any, first, last;
    const double* src;  // accumulator to read, nullptr: zero
    double* dst;
    bool idle;          // nothing to write: all roots zero, accumulator stays
    bool vec;           // dst is 16-byte aligned
    bool plain;         // one root into zero: its values as they are
    const double* fac;  // shared memory: factor of each instance, negative for a zero root (n <= kFoldInst)
};

// Maximum and exponent of instance i of the group.
__device__ __forceinline__ unsigned fold_max(const AccumArgs& a, int i) { return a.max_r[(int64_t)i * a.s_is]; }
__device__ __forceinline__ int64_t fold_exp(const AccumArgs& a, int i) { return a.exp_r[(int64_t)i * a.s_is]; }
__device__ __forceinline__ double fold_pow2(int64_t d) { return ldexp(1.0, (int)(d < -2000 ? -2000 : d)); }

// The accumulator's exponent, after the call's last group the result's, and the
// slice counter: written by the last block to have read the control block, so
// that no launch of its own is needed for them.  The fences order each block's
// reads before its ticket, and the last ticket before the writes; they come
// before the block's own stores, which they would otherwise wait for (2.2 us at
// the end of a fold of 2^20 to 2^22 outputs).
__device__ __forceinline__ void fold_control(const AccumArgs& a, const FoldState& f) {
    if (gridDim.x > 1) {
        __threadfence();
        const unsigned ticket = atomicInc(&a.ctl->ticket, gridDim.x - 1);  // wraps to 0 at the last block
        __threadfence();
        if (ticket != gridDim.x - 1) return;
    }
    a.ctl->acc_exp[f.par ^ 1] = f.newE;
    if (f.last) {
        const int64_t e = f.newE == INT64_MIN ? 0 : f.newE;
        a.ctl->final_exp = e;
        if (a.direct) *a.ctl->out_exp = e;
    }
    a.ctl->slice = f.slice + a.advance;
}

__device__ __forceinline__ FoldState fold_state(const AccumArgs& a) {
    __shared__ unsigned smax[kFoldInst];
    __shared__ int64_t sexp[kFoldInst];
    __shared__ double sfac[kFoldInst];
    FoldState f;
    const Control* ctl = a.ctl;
    const int group = a.n_inst > 1 ? a.n_inst : 1;
    // one round trip for the control block and the instances' slots
    if (threadIdx.x < kFoldInst && (int)threadIdx.x < group) {
        smax[threadIdx.x] = fold_max(a, threadIdx.x);
        sexp[threadIdx.x] = fold_exp(a, threadIdx.x);
    }
    f.slice = ctl->slice;
    f.slice_end = ctl->slice_end;
    const int64_t begin = ctl->slice_begin, acc_exp0 = ctl->acc_exp[0], acc_exp1 = ctl->acc_exp[1];
    double* const out_ptr = ctl->out;
    __syncthreads();
    f.n = (int)(f.slice_end - f.slice < group ? f.slice_end - f.slice : group);
    f.par = group == 1 ? (int)((f.slice - begin) & 1) : (int)(((f.slice - begin) / group) & 1);
    f.first = a.direct && f.slice == begin;
    f.last = f.slice + group >= f.slice_end;
    const int64_t accE = f.par ? acc_exp1 : acc_exp0;
    const bool empty = accE == INT64_MIN;
    f.newE = accE;
    f.any = false;
    for (int i = 0; i < f.n; ++i) {
        if (!(__uint_as_float(i < kFoldInst ? smax[i] : fold_max(a, i)) > 0.f)) continue;
        const int64_t S = i < kFoldInst ? sexp[i] : fold_exp(a, i);
        f.newE = (empty && !f.any) ? S : (S > f.newE ? S : f.newE);
        f.any = true;
    }
    f.fa = f.any && !empty ? fold_pow2(accE - f.newE) : 1.0;
    f.src = f.first ? nullptr : a.acc;
    const bool out = a.direct && f.last;
    f.dst = out ? out_ptr : a.acc;
    f.idle = !f.any && !f.first && !out;
    f.vec = (reinterpret_cast<uintptr_t>(f.dst) & 15) == 0;
    f.plain = f.first && f.n == 1 && f.any;
    f.fac = nullptr;
    if (threadIdx.x == 0) fold_control(a, f);  // (every thread's reads came before the barrier above)
    if (f.n > 1 && f.n <= kFoldInst) {  // the same factors for every output
        if ((int)threadIdx.x < f.n)
            sfac[threadIdx.x] =
                __uint_as_float(smax[threadIdx.x]) > 0.f ? fold_pow2(sexp[threadIdx.x] - f.newE) : -1.0;
        __syncthreads();
        f.fac = sfac;
    }
    return f;
}

// Root factor of instance i; false for a zero root.  A factor may be zero (a
// root far below the others): its infinities and NaN still reach the sum.
__device__ __forceinline__ bool fold_factor(const AccumArgs& a, const FoldState& f, int i, double& fr) {
    if (f.fac) {
        fr = f.fac[i];
        return fr >= 0.0;
    }
    if (!(__uint_as_float(fold_max(a, i)) > 0.f)) return false;
    fr = fold_pow2(fold_exp(a, i) - f.newE);
    return true;
}

// (double)x + 0.0 in integer operations: the FP64 pipe converts and adds about
// two values per clock and SM, which bounds a fold of many outputs in the
// root's order (67 us for 2^22 complex ones, 35 to 42 with this).  Zeros of either sign give +0; subnormal,
// infinite and NaN values take the conversion.
__device__ __forceinline__ double widen(float x) {
    const unsigned u = __float_as_uint(x), e = (u >> 23) & 0xffu;
    if ((u << 1) == 0u) return 0.0;
    if (e == 0u || e == 255u) return (double)x;
    return __hiloint2double((int)((u & 0x80000000u) | (((u & 0x7fffffffu) >> 3) + 0x38000000u)), (int)(u << 29));
}

template <bool CPLX>
__device__ __forceinline__ double2 fold_start(const FoldState& f, int64_t o) {
    if (!f.src) return make_double2(0.0, 0.0);
    if constexpr (CPLX) {
        const double2 v = reinterpret_cast<const double2*>(f.src)[o];
        return make_double2(v.x * f.fa, v.y * f.fa);
    } else {
        return make_double2(f.src[o] * f.fa, 0.0);
    }
}

__device__ __forceinline__ void fold_add(double2& v, float2 r, double fr) {
    v.x += (double)r.x * fr;
    v.y += (double)r.y * fr;
}
__device__ __forceinline__ void fold_add(double2& v, float r, double fr) { v.x += (double)r * fr; }
__device__ __forceinline__ double2 fold_plain(float2 r) { return make_double2(widen(r.x), widen(r.y)); }
__device__ __forceinline__ double2 fold_plain(float r) { return make_double2(widen(r), 0.0); }

template <bool CPLX>
__device__ __forceinline__ void fold_store(const FoldState& f, int64_t o, double2 v) {
    if constexpr (CPLX) {
        if (f.vec) {
            reinterpret_cast<double2*>(f.dst)[o] = v;
        } else {  // a caller's buffer that only has the alignment of a double
            f.dst[2 * o] = v.x;
            f.dst[2 * o + 1] = v.y;
        }
    } else {
        f.dst[o] = v.x;
    }
}

// Root offset of output o: digits fastest first, shifts where a size is a
// power of two, 32-bit division otherwise (outputs beyond 2^31 entries: 64).
__device__ __forceinline__ int64_t fold_offset(const AccumArgs& a, int64_t o) {
    int64_t src = 0;
    if (a.n_out >= (int64_t(1) << 31)) {
        for (int i = 0; i < a.n_od; ++i) {
            const int64_t d = a.od_dim[i];
            src += (o % d) * a.od_s[i];
            o /= d;
        }
        return src;
    }
    unsigned rem = (unsigned)o;
    for (int i = 0; i < a.n_od; ++i) {
        const unsigned d = (unsigned)a.od_dim[i];
        if ((d & (d - 1)) == 0) {
            src += (int64_t)(rem & (d - 1)) * a.od_s[i];
            rem >>= __ffs(d) - 1;
        } else {
            const unsigned q = rem / d;
            src += (int64_t)(rem - q * d) * a.od_s[i];
            rem = q;
        }
    }
    return src;
}

// One thread per output; consecutive threads write consecutive outputs.
// Bound by memory when the outputs follow the root's order (the digits are
// merged on the host: one digit then), by latency for the few outputs of a
// network with few or no open labels: FEW loads the roots of the first eight
// instances before anything else, so that they share one round trip with the
// control block and the scale slots (16 outputs of eight slices side by side:
// 19 us with one load after the other, 7 now; one output: 7.5 and 4).
template <bool CPLX, bool FEW>
__global__ void __launch_bounds__(256, 3) k_accumulate(const __grid_constant__ AccumArgs a) {
    using T = typename std::conditional<CPLX, float2, float>::type;
    const T* const root = reinterpret_cast<const T*>(a.R);
    constexpr int R = FEW ? 1 : 4;  // outputs in flight per thread
    constexpr int C = FEW ? 8 : 1;  // instances
    const int64_t stride = (int64_t)gridDim.x * blockDim.x, o_first = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int group = a.n_inst > 1 ? a.n_inst : 1;  // every instance of a group has its root, live or not
    T head[C];
    if (FEW && o_first < a.n_out) {
        const int64_t at = fold_offset(a, o_first);
#pragma unroll
        for (int c = 0; c < C; ++c)
            if (c < group) head[c] = __ldcs(root + at + (int64_t)c * a.r_is);
    }
    const FoldState f = fold_state(a);
    if (!f.idle) {
        for (int64_t o0 = o_first; o0 < a.n_out; o0 += R * stride) {
            double2 v[R];
            int64_t src[R];
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const int64_t o = o0 + r * stride;
                if (o >= a.n_out) break;
                src[r] = fold_offset(a, o);
                if (!f.plain) v[r] = fold_start<CPLX>(f, o);
            }
            if (f.plain) {
                T ld[R];
#pragma unroll
                for (int r = 0; r < R; ++r)
                    if (o0 + r * stride < a.n_out) ld[r] = FEW && o0 == o_first ? head[0] : __ldcs(root + src[r]);
#pragma unroll
                for (int r = 0; r < R; ++r)
                    if (o0 + r * stride < a.n_out) v[r] = fold_plain(ld[r]);
            } else {
                for (int i0 = 0; i0 < f.n; i0 += C) {
                    T ld[R][C];
#pragma unroll
                    for (int r = 0; r < R; ++r)
#pragma unroll
                        for (int c = 0; c < C; ++c)
                            if (o0 + r * stride < a.n_out && i0 + c < f.n)
                                ld[r][c] = FEW && o0 == o_first && i0 == 0 ? head[c]
                                                                          : __ldcs(root + src[r] + (int64_t)(i0 + c) * a.r_is);
#pragma unroll
                    for (int c = 0; c < C; ++c) {
                        double fr;
                        if (i0 + c >= f.n || !fold_factor(a, f, i0 + c, fr)) continue;
#pragma unroll
                        for (int r = 0; r < R; ++r)
                            if (o0 + r * stride < a.n_out) fold_add(v[r], ld[r][c], fr);
                    }
                }
            }
#pragma unroll
            for (int r = 0; r < R; ++r)
                if (o0 + r * stride < a.n_out) fold_store<CPLX>(f, o0 + r * stride, v[r]);
        }
    }
}

// Outputs in another order than the root's (power-of-two sizes): tiles of up
// to 2^10 entries holding the lowest five index bits of either order, read
// in root order and written in output order through shared memory, so that
// both sides move whole 128-byte lines.  Bound by memory: 12 bytes read and
// written per real output, 24 per complex one.  A call whose 2^13 x 2^12
// complex root is transposed: 2146 us with one thread per output and a digit
// loop, a cleared and re-read accumulator and a copy to the caller (947, 75
// and 255 us of it), 851 us with this fold, which writes the output itself
// (159 us of it; 345 with one tile's loads and stores after the other).
template <bool CPLX>
__global__ void __launch_bounds__(256, 5) k_accumulate_perm(const __grid_constant__ AccumArgs a,
                                                         const __grid_constant__ FoldPlan p) {
    using T = typename std::conditional<CPLX, float2, float>::type;
    __shared__ T stage[kFoldTile + kFoldTile / 32];
    __shared__ int64_t tsrc[kFoldTile], tdst[kFoldTile];
    __shared__ uint16_t tidx[kFoldTile];
    const FoldState f = fold_state(a);
    if (!f.idle) {
        const int tsz = 1 << p.t;
        for (int i = threadIdx.x; i < tsz; i += blockDim.x) {
            int64_t so = 0, dd = 0;
            int idx = 0;
            for (int j = 0; j < p.t; ++j)
                if ((i >> j) & 1) {
                    so += p.src_add[j];
                    dd += p.dst_add[j];
                    idx += p.idx_add[j];
                }
            tsrc[i] = so;                            // i counts the tile in root order
            tdst[i] = dd;                            // ... and in output order
            tidx[i] = (uint16_t)(idx + (idx >> 5));  // its place in the stage
        }
        __syncthreads();
        constexpr int R = kFoldTile / 256;
        const int64_t n_tiles = int64_t(1) << p.u;
        // tile bases, one bit per lane and a warp-wide sum
        const int lane = threadIdx.x & 31;
        auto bases = [&](int64_t tile, int64_t& sb, int64_t& db) {
            sb = db = 0;
            for (int j = lane; j < p.u; j += 32)
                if ((tile >> j) & 1) {
                    sb += p.rest_src[j];
                    db += p.rest_dst[j];
                }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                sb += __shfl_xor_sync(0xffffffffu, sb, o);
                db += __shfl_xor_sync(0xffffffffu, db, o);
            }
        };
        if (f.plain) {
            // one root into zero: the next tile's loads are in flight while
            // this one is written
            const T* root = reinterpret_cast<const T*>(a.R);
            T ld[R];
            int64_t sb, db = 0, nsb = 0, ndb = 0;
            if (blockIdx.x < n_tiles) {
                bases(blockIdx.x, sb, db);
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    const int i = threadIdx.x + r * 256;
                    if (i < tsz) ld[r] = __ldcs(root + sb + tsrc[i]);
                }
            }
            for (int64_t tile = blockIdx.x; tile < n_tiles; tile += gridDim.x) {
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    const int i = threadIdx.x + r * 256;
                    if (i < tsz) stage[i + (i >> 5)] = ld[r];
                }
                __syncthreads();
                if (tile + gridDim.x < n_tiles) {
                    bases(tile + gridDim.x, nsb, ndb);
#pragma unroll
                    for (int r = 0; r < R; ++r) {
                        const int i = threadIdx.x + r * 256;
                        if (i < tsz) ld[r] = __ldcs(root + nsb + tsrc[i]);
                    }
                }
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    const int i = threadIdx.x + r * 256;
                    if (i < tsz) fold_store<CPLX>(f, db + tdst[i], fold_plain(stage[tidx[i]]));
                }
                db = ndb;
                __syncthreads();
            }
        }
        for (int64_t tile = f.plain ? n_tiles : blockIdx.x; tile < n_tiles; tile += gridDim.x) {
            int64_t sb, db;
            bases(tile, sb, db);
            double2 v[R];
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const int i = threadIdx.x + r * 256;
                if (i < tsz) v[r] = fold_start<CPLX>(f, db + tdst[i]);
            }
            for (int q = 0; q < f.n; ++q) {
                double fr;
                if (!fold_factor(a, f, q, fr)) continue;
                const T* root = reinterpret_cast<const T*>(a.R) + (int64_t)q * a.r_is + sb;
                T ld[R];
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    const int i = threadIdx.x + r * 256;
                    if (i < tsz) ld[r] = __ldcs(root + tsrc[i]);
                }
                __syncthreads();  // the stage's previous entries have been read
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    const int i = threadIdx.x + r * 256;
                    if (i < tsz) stage[i + (i >> 5)] = ld[r];
                }
                __syncthreads();
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    const int i = threadIdx.x + r * 256;
                    if (i < tsz) {
                        fold_add(v[r], stage[tidx[i]], fr);
                    }
                }
            }
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const int i = threadIdx.x + r * 256;
                if (i < tsz) fold_store<CPLX>(f, db + tdst[i], v[r]);
            }
        }
    }
}

// Tile plan of the permuted fold; false where the plain fold serves as well:
// few outputs, sizes other than powers of two, or outputs whose lowest 32
// entries are contiguous in the root.
static bool make_fold_plan(const AccumArgs& a, FoldPlan& p) {
    if (a.n_out < kFoldTile) return false;
    int64_t add[64];  // root stride of every output index bit
    int n = 0;
    for (int i = 0; i < a.n_od; ++i) {
        const int64_t d = a.od_dim[i];
        if (d & (d - 1)) return false;
        for (int64_t b = 1; b < d; b <<= 1) {
            if (n >= kMaxBits) return false;
            add[n++] = a.od_s[i] * b;
        }
    }
    bool contiguous = true;
    for (int j = 0; j < 5; ++j) contiguous &= add[j] == (int64_t(1) << j);
    if (contiguous) return false;
    memset(&p, 0, sizeof(p));
    bool in[64] = {};
    for (int j = 0; j < 5; ++j) in[j] = true;
    int cnt = 5;
    int by_src[64];
    for (int j = 0; j < n; ++j) by_src[j] = j;
    std::sort(by_src, by_src + n, [&](int x, int y) { return add[x] < add[y]; });
    for (int j = 0; j < 5; ++j)
        if (!in[by_src[j]]) {
            in[by_src[j]] = true;
            ++cnt;
        }
    for (int j = 5; j < n && cnt < 10; ++j)
        if (!in[j]) {
            in[j] = true;
            ++cnt;
        }
    int rank[64], r = 0;  // place of a tile bit in root order
    for (int j = 0; j < n; ++j)
        if (in[by_src[j]]) {
            p.src_add[r] = add[by_src[j]];
            rank[by_src[j]] = r++;
        }
    int t = 0;
    for (int j = 0; j < n; ++j) {
        if (in[j]) {
            p.dst_add[t] = int64_t(1) << j;
            p.idx_add[t] = 1 << rank[j];
            ++t;
        } else {
            p.rest_src[p.u] = add[j];
            p.rest_dst[p.u] = int64_t(1) << j;
            ++p.u;
        }
    }
    p.t = t;
    return true;
}

cudaError_t launch_accumulate(const AccumArgs& a0, bool is_c, cudaStream_t s, int advance) {
    AccumArgs a = a0;
    a.advance = advance;
    FoldPlan p;
    if (make_fold_plan(a, p)) {
        const int64_t tiles = a.n_out >> p.t;
        const unsigned blocks = (unsigned)(tiles < sm_count() * 5 ? tiles : sm_count() * 5);  // one round
        if (is_c)
            k_accumulate_perm<true><<<blocks, 256, 0, s>>>(a, p);
        else
            k_accumulate_perm<false><<<blocks, 256, 0, s>>>(a, p);
        return cudaGetLastError();
    }
    int64_t blocks = (a.n_out + 255) / 256;
    if (blocks > sm_count() * 8) blocks = sm_count() * 8;
    if (blocks < 1) blocks = 1;
    const bool few = a.n_out <= 256 * blocks;
    if (is_c && few)
        k_accumulate<true, true><<<(unsigned)blocks, 256, 0, s>>>(a);
    else if (is_c)
        k_accumulate<true, false><<<(unsigned)blocks, 256, 0, s>>>(a);
    else if (few)
        k_accumulate<false, true><<<(unsigned)blocks, 256, 0, s>>>(a);
    else
        k_accumulate<false, false><<<(unsigned)blocks, 256, 0, s>>>(a);
    return cudaGetLastError();
}

__global__ void k_begin_call(Control* ctl, int64_t slice_begin, int64_t slice_end, double* acc,
                             int64_t n) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i == 0) {
        ctl->slice = slice_begin;
        ctl->slice_begin = slice_begin;
        ctl->slice_end = slice_end;
        ctl->acc_exp[0] = INT64_MIN;
        ctl->acc_exp[1] = INT64_MIN;
        ctl->status = 0;
        ctl->ticket = 0;
    }
    for (; i < n; i += (int64_t)gridDim.x * blockDim.x) acc[i] = 0.0;
}

cudaError_t launch_begin_call(Control* ctl, int64_t slice_begin, int64_t slice_end, double* acc,
                              int64_t n, cudaStream_t s) {
    int64_t blocks = (n + 255) / 256;
    if (blocks > 1024) blocks = 1024;
    if (blocks < 1) blocks = 1;
    k_begin_call<<<(unsigned)blocks, 256, 0, s>>>(ctl, slice_begin, slice_end, acc, n);
    return cudaGetLastError();
}

cudaError_t launch_begin_slice(unsigned* maxabs, int n_nodes, cudaStream_t s) {
    return cudaMemsetAsync(maxabs, 0, sizeof(unsigned) * (size_t)n_nodes, s);
}

__global__ void k_advance(Control* ctl, int step) { ctl->slice += step; }

cudaError_t launch_advance(Control* ctl, cudaStream_t s, int step) {
    k_advance<<<1, 1, 0, s>>>(ctl, step);
    return cudaGetLastError();
}

constexpr int kTablePart = 500;  // pointers per launch: 4 KB of parameters
struct LeafTablePart {
    const void* ptr[kTablePart];
};

__global__ void __launch_bounds__(512) k_leaf_table(const __grid_constant__ LeafTablePart p, int n, const void** table) {
    if ((int)threadIdx.x < n) table[threadIdx.x] = p.ptr[threadIdx.x];
}

cudaError_t launch_leaf_table(const void* const* ptrs, int n, const void** table, cudaStream_t s) {
    for (int i = 0; i < n; i += kTablePart) {
        LeafTablePart p;
        const int m = std::min(kTablePart, n - i);
        memcpy(p.ptr, ptrs + i, sizeof(void*) * m);
        k_leaf_table<<<1, 512, 0, s>>>(p, m, table + i);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

// Largest |component| of every leaf, so that leaves are renormalised like
// intermediates before their first contraction.  A leaf of more than two parts'
// floats is cut into parts of kLeafPart (at most 1024), one block each (2^23 and
// 2^22 complex entries: 29 us with parts of 2^14 floats, 22 with 2^13), combined
// by atomicMax on the float bits (non-negative floats order like unsigned), or
// stored directly when one block covers the leaf and `direct` allows it (no
// zeroing needed then).
// Blocks [0, n0) are part 0 of every leaf, the others the further parts of the
// large leaves listed in `big`, so that many small leaves beside a large one
// add no empty blocks (300 leaves and one of 2^26 floats: 228 us with as many
// blocks for every leaf, 40 now; 2000 and one of 2^20: 91 and 5).
// Large leaves are read 16 bytes a load, four loads in flight per thread
// (bound by memory); a leaf that is not 16-byte aligned, and the ends, by
// single floats.
constexpr int kBigLeaves = 128;
struct BigLeaves {
    int32_t n;
    int32_t leaf[kBigLeaves];
    int32_t first[kBigLeaves + 1];  // first of the leaf's further blocks
};

__host__ __device__ inline int leaf_parts(int64_t nfloat) {
    if (nfloat <= 2 * kLeafPart) return 1;  // (several would need their slot cleared by a launch of its own)
    const int64_t parts = (nfloat + kLeafPart - 1) / kLeafPart;
    return (int)(parts > 1024 ? 1024 : parts);
}

__device__ __forceinline__ void leaf_max_part(const float* const* ptrs, const int64_t* nfloat, unsigned* out, int n0,
                                              const BigLeaves& big, bool direct) {
    int v = blockIdx.x, part = 0;
    if (v >= n0) {
        const int b = v - n0;
        if (b >= big.first[big.n]) return;
        int lo = 0, hi = big.n - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) / 2;
            if (big.first[mid] <= b) lo = mid;
            else hi = mid - 1;
        }
        v = big.leaf[lo];
        part = 1 + b - big.first[lo];
    }
    const float* p = ptrs[v];
    const int64_t m = nfloat[v];
    const int parts = leaf_parts(m);
    const bool vec = (reinterpret_cast<uintptr_t>(p) & 15) == 0 && m >= 4096;
    const int64_t m4 = vec ? m / 4 : 0;
    const int64_t step = (int64_t)parts * blockDim.x, first = (int64_t)part * blockDim.x + threadIdx.x;
    float lmax = 0.f;
    const float4* p4 = reinterpret_cast<const float4*>(p);
    for (int64_t i = first; i < m4; i += 4 * step) {
        float4 x[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) x[r] = i + r * step < m4 ? p4[i + r * step] : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int r = 0; r < 4; ++r)
            lmax = fmaxf(lmax, fmaxf(fmaxf(fabsf(x[r].x), fabsf(x[r].y)), fmaxf(fabsf(x[r].z), fabsf(x[r].w))));
    }
    for (int64_t i = 4 * m4 + first; i < m; i += step) lmax = fmaxf(lmax, fabsf(p[i]));
    __shared__ float red[32];
    for (int o = 16; o > 0; o >>= 1) lmax = fmaxf(lmax, __shfl_xor_sync(0xffffffffu, lmax, o));
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = lmax;
    __syncthreads();
    if (threadIdx.x < 32) {
        const int nw = blockDim.x >> 5;
        lmax = threadIdx.x < nw ? red[threadIdx.x] : 0.f;
        for (int o = 16; o > 0; o >>= 1) lmax = fmaxf(lmax, __shfl_xor_sync(0xffffffffu, lmax, o));
        if (threadIdx.x == 0) {
            if (direct && parts == 1)
                out[v] = __float_as_uint(lmax);
            else
                atomicMax(&out[v], __float_as_uint(lmax));
        }
    }
}

// The next large leaves from v on; returns the number of their further blocks.
static int next_big(const int64_t* nfloat, int n, int& v, BigLeaves& big) {
    big.n = 0;
    int blocks = 0;
    for (; v < n && big.n < kBigLeaves; ++v) {
        const int parts = leaf_parts(nfloat[v]);
        if (parts == 1) continue;
        big.leaf[big.n] = v;
        big.first[big.n++] = blocks;
        blocks += parts - 1;
    }
    big.first[big.n] = blocks;
    return blocks;
}

__global__ void __launch_bounds__(256) k_leaf_max(const float* const* ptrs, const int64_t* nfloat, unsigned* out, int n0,
                                                  const __grid_constant__ BigLeaves big) {
    leaf_max_part(ptrs, nfloat, out, n0, big, false);
}

// The start of a call: leaf maxima as k_leaf_max, (block 0) the control block
// with the call's output pointers, and the FP64 accumulator cleared where the
// fold reads it (n_acc > 0).
__global__ void __launch_bounds__(256) k_call_begin(const float* const* ptrs, const int64_t* nfloat, unsigned* out, int n,
                                                    const __grid_constant__ BigLeaves big, Control* ctl,
                                                    int64_t slice_begin, int64_t slice_end, double* acc, int64_t n_acc,
                                                    double* result, int64_t* result_exp) {
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        ctl->slice = slice_begin;
        ctl->slice_begin = slice_begin;
        ctl->slice_end = slice_end;
        ctl->acc_exp[0] = INT64_MIN;
        ctl->acc_exp[1] = INT64_MIN;
        ctl->status = 0;
        ctl->ticket = 0;
        ctl->out = result;
        ctl->out_exp = result_exp;
    }
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n_acc; i += (int64_t)gridDim.x * blockDim.x)
        acc[i] = 0.0;
    leaf_max_part(ptrs, nfloat, out, n, big, true);
}

// The further parts of large leaves that one list does not hold.
static cudaError_t launch_more_big(const float* const* ptrs, const int64_t* nfloat, unsigned* out,
                                   const int64_t* nfloat_host, int n, int v, cudaStream_t s) {
    BigLeaves big;
    while (const int blocks = next_big(nfloat_host, n, v, big)) {
        k_leaf_max<<<(unsigned)blocks, 256, 0, s>>>(ptrs, nfloat, out, 0, big);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

cudaError_t launch_call_begin(const float* const* ptrs, const int64_t* nfloat, const int64_t* nfloat_host, unsigned* out,
                              int n, Control* ctl, int64_t slice_begin, int64_t slice_end, double* acc, int64_t n_acc,
                              double* result, int64_t* result_exp, cudaStream_t s) {
    BigLeaves big;
    int v = 0;
    const int more = next_big(nfloat_host, n, v, big);
    if (more) {  // several blocks per leaf combine by atomicMax from zero
        const cudaError_t e = cudaMemsetAsync(out, 0, sizeof(unsigned) * (size_t)n, s);
        if (e != cudaSuccess) return e;
    }
    k_call_begin<<<(unsigned)std::max(n + more, 1), 256, 0, s>>>(ptrs, nfloat, out, n, big, ctl, slice_begin, slice_end, acc, n_acc,
                                                      result, result_exp);
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? launch_more_big(ptrs, nfloat, out, nfloat_host, n, v, s) : e;
}

cudaError_t launch_leaf_max(const float* const* ptrs, const int64_t* nfloat, const int64_t* nfloat_host, unsigned* out,
                            int n, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    cudaError_t e = cudaMemsetAsync(out, 0, sizeof(unsigned) * (size_t)n, s);
    if (e != cudaSuccess) return e;
    BigLeaves big;
    int v = 0;
    const int more = next_big(nfloat_host, n, v, big);
    k_leaf_max<<<(unsigned)(n + more), 256, 0, s>>>(ptrs, nfloat, out, n, big);
    e = cudaGetLastError();
    return e == cudaSuccess ? launch_more_big(ptrs, nfloat, out, nfloat_host, n, v, s) : e;
}

// Leaf adjoints of one slice, all leaves in one launch: blockIdx.y picks
// the table entry, blockIdx.x a chunk of its elements.
template <bool CPLX>
__global__ void __launch_bounds__(256) k_leaf_grads(const LeafGradArgs* tab, int n_entries) {
    __shared__ LeafGradArgs a;
    if ((int)blockIdx.y >= n_entries) return;
    {
        const int* src = reinterpret_cast<const int*>(tab + blockIdx.y);
        int* dst = reinterpret_cast<int*>(&a);
        for (int i = threadIdx.x; i < (int)(sizeof(LeafGradArgs) / 4); i += blockDim.x) dst[i] = src[i];
    }
    __syncthreads();
    if ((int64_t)blockIdx.x * blockDim.x >= a.n) return;
    const int64_t inst = blockIdx.z;
    const int64_t slice = a.ctl->slice;
    const int64_t base = slice_offset(a.sl, slice);
    int64_t e = a.exp_adj[inst * a.exp_is];
    const int ex = (int)(e < -400 ? -400 : (e > 400 ? 400 : e));
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t o = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; o < a.n; o += stride) {
        int64_t g = base, s = 0, rem = o;
        for (int i = 0; i < a.n_d; ++i) {
            const int64_t d = a.dim[i];
            const int64_t v = rem % d;
            rem /= d;
            g += v * a.gstride[i];
            s += v * a.astride[i];
        }
        s += inst * a.adj_is;
        g += inst * a.grad_is;
        if (CPLX) {
            const float2 x = reinterpret_cast<const float2*>(a.adj)[s];
            float2* G = reinterpret_cast<float2*>(a.grad);
            float2 y = G[g];
            y.x += ldexpf(x.x, ex);
            y.y += ldexpf(x.y, ex);
            G[g] = y;
        } else {
            reinterpret_cast<float*>(a.grad)[g] += ldexpf(reinterpret_cast<const float*>(a.adj)[s], ex);
        }
    }
}

cudaError_t launch_leaf_grads(const LeafGradArgs* tab, int n_entries, int64_t max_n, int n_inst, bool is_c,
                              cudaStream_t s) {
    if (n_entries <= 0) return cudaSuccess;
    int64_t blocks = (max_n + 255) / 256;
    blocks = blocks < 1 ? 1 : (blocks > sm_count() * 8 ? sm_count() * 8 : blocks);
    const dim3 grid((unsigned)blocks, (unsigned)n_entries, (unsigned)(n_inst > 1 ? n_inst : 1));
    if (is_c)
        k_leaf_grads<true><<<grid, 256, 0, s>>>(tab, n_entries);
    else
        k_leaf_grads<false><<<grid, 256, 0, s>>>(tab, n_entries);
    return cudaGetLastError();
}

// dst = src (or dst += src) for every entry of the table: blockIdx.y picks
// the entry, blockIdx.x a chunk.
__global__ void __launch_bounds__(256) k_copy_table(const CopyEntry* tab, int n_entries) {
    if ((int)blockIdx.y >= n_entries) return;
    const CopyEntry e = tab[blockIdx.y];
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < e.nfloat; i += stride) {
        float v = e.src[i];
        for (int r = 1; r < e.n_sum; ++r) v += e.src[r * e.src_is + i];
        e.dst[i] = e.add ? e.dst[i] + v : v;
    }
}

cudaError_t launch_copy_table(const CopyEntry* tab, int n_entries, int64_t max_nfloat, cudaStream_t s) {
    int64_t blocks = (max_nfloat + 255) / 256;
    blocks = blocks < 1 ? 1 : (blocks > sm_count() * 4 ? sm_count() * 4 : blocks);
    for (int first = 0; first < n_entries; first += 65535) {  // grid y limit
        const int cnt = n_entries - first < 65535 ? n_entries - first : 65535;
        k_copy_table<<<dim3((unsigned)blocks, (unsigned)cnt), 256, 0, s>>>(tab + first, cnt);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

// p[i * stride + j] = 0 for i < n, j < count.
__global__ void k_zero_strided(unsigned* p, int64_t count, int64_t stride, int n) {
    const int64_t total = count * n;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < total; t += (int64_t)gridDim.x * blockDim.x)
        p[(t / count) * stride + t % count] = 0u;
}

cudaError_t launch_zero_strided(unsigned* p, int64_t count, int64_t stride, int n, cudaStream_t s) {
    const int64_t total = count * n;
    if (total <= 0) return cudaSuccess;
    int64_t blocks = (total + 255) / 256;
    if (blocks > sm_count() * 4) blocks = sm_count() * 4;
    k_zero_strided<<<(unsigned)blocks, 256, 0, s>>>(p, count, stride, n);
    return cudaGetLastError();
}

// The root adjoint in the form the sweep reads: largest |component| m of
// the FP64 adjoint, m = f * 2^e with f in [0.5, 1) (frexp), every component
// scaled by 2^-e (exact) and rounded to float into the root's layout; the
// root's scale slots get f and e plus the adjoint's own exponent.  One block.
__global__ void __launch_bounds__(1024) k_root_adjoint(RootAdjArgs a) {
    __shared__ double red[32];
    const int c = a.cplx ? 2 : 1;
    const int64_t nd = a.n_out * c;
    const int64_t inst = blockIdx.x;
    a.adj += inst * nd;
    a.dst += inst * a.dst_is;
    a.max_slot += inst * a.slot_is;
    a.exp_slot += inst * a.slot_is;
    if (a.exp_dev) a.exp_dev += inst;
    double m = 0.0;
    for (int64_t i = threadIdx.x; i < nd; i += blockDim.x) m = fmax(m, fabs(a.adj[i]));
    for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
    __syncthreads();
    if (threadIdx.x < 32) {
        m = threadIdx.x < (blockDim.x >> 5) ? red[threadIdx.x] : 0.0;
        for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
        if (threadIdx.x == 0) red[0] = m;
    }
    __syncthreads();
    m = red[0];
    int e = 0;
    if (m > 0.0) frexp(m, &e);
    for (int64_t i = threadIdx.x; i < nd; i += blockDim.x)
        a.dst[a.perm[i / c] * c + (i % c)] = (float)ldexp(a.adj[i], -e);
    if (threadIdx.x == 0) {
        const float f = m > 0.0 ? (float)ldexp(m, -e) : 0.f;
        *a.max_slot = __float_as_uint(f);
        *a.exp_slot = (int64_t)e + a.exp_host + (a.exp_dev ? *a.exp_dev : 0);
    }
}

cudaError_t launch_root_adjoint(const RootAdjArgs& a, int n_inst, cudaStream_t s) {
    k_root_adjoint<<<(unsigned)(n_inst > 1 ? n_inst : 1), 1024, 0, s>>>(a);
    return cudaGetLastError();
}

__global__ void k_batch_start(unsigned long long* t_start) { *t_start = global_ns(); }

cudaError_t launch_batch_start(unsigned long long* t_start, cudaStream_t s) {
    k_batch_start<<<1, 1, 0, s>>>(t_start);
    return cudaGetLastError();
}

__global__ void k_batch_finish(const BatchRoot* roots, int n, double* out, int64_t* out_exp,
                               const unsigned long long* t_start, const unsigned long long* t_done,
                               unsigned long long* latency) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const BatchRoot r = roots[i];
    if (r.root == nullptr) {
        // a sliced network: its slice loop runs after this kernel and writes
        // its value, exponent and latency itself
        out[2 * i] = 0.0;
        out[2 * i + 1] = 0.0;
        out_exp[i] = 0;
        if (latency) latency[i] = 0;
        return;
    }
    const bool zero = !(__uint_as_float(*r.max) > 0.f);
    if (r.is_c) {
        const float2 v = *reinterpret_cast<const float2*>(r.root);
        out[2 * i] = v.x;
        out[2 * i + 1] = v.y;
    } else {
        out[2 * i] = *reinterpret_cast<const float*>(r.root);
        out[2 * i + 1] = 0.0;
    }
    out_exp[i] = zero ? 0 : *r.exp;
    if (latency) latency[i] = t_done[i] > *t_start ? t_done[i] - *t_start : 0;
}

__global__ void k_batch_mark(const unsigned long long* t_start, unsigned long long* latency) {
    const unsigned long long t = global_ns();
    *latency = t > *t_start ? t - *t_start : 0;
}

cudaError_t launch_batch_mark(const unsigned long long* t_start, unsigned long long* latency, cudaStream_t s) {
    k_batch_mark<<<1, 1, 0, s>>>(t_start, latency);
    return cudaGetLastError();
}

cudaError_t launch_batch_finish(const BatchRoot* roots, int n, double* out, int64_t* out_exp,
                                const unsigned long long* t_start, const unsigned long long* t_done,
                                unsigned long long* latency, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    k_batch_finish<<<(n + 127) / 128, 128, 0, s>>>(roots, n, out, out_exp, t_start, t_done, latency);
    return cudaGetLastError();
}

}  // namespace tn
