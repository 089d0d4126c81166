// tn_tiled.cu -- tiled node kernels (FP32 on CUDA cores): the tile kernel for
// label sizes of any kind, the inner-product and wave kernels for powers of two.
//
// A tree node contracts A and B over the shared labels (Sec. 2 of arXiv
// 2002.01935).  With every label size a power of two, each group of labels
// (batch, M, N, K) is a set of index bits and an operand offset is a
// scatter of those bits to the operand's strides (other sizes: of mixed-radix
// digits).  The node output is laid
// out [batch][M][N], i.e. a row-major M x N matrix per batch index, so a
// node is a batched GEMM whose operands are read through bit scatters:
//   C[b, m, n] = sum_k A[sA(b) + sA(m) + sA(k)] * B[sB(b) + sB(k) + sB(n)].
// The index permutation of a classic transpose-transpose-GEMM scheme is
// folded into the operand loads: each CTA builds tile-local offset tables
// once, and the planner orders every group's bits by operand stride so
// that tiles cover the operands' contiguous bits (coalesced loads).
//
// Renormalisation (Sec. 4.2): operands are multiplied by 2^-e at load,
// e = frexp exponent of their max |component|, which is exact; the output
// max goes to the node's slot for its consumer.
#include <cuda_runtime.h>
#include <algorithm>
#include <atomic>
#include <cstring>
#include <stdint.h>
#include <type_traits>

#include "../../include/tn.h"
#include "tn_internal.h"

namespace tn {

namespace {

template <bool CPLX>
struct VT;
template <>
struct VT<true> {
    using T = float2;
};
template <>
struct VT<false> {
    using T = float;
};

__device__ __forceinline__ int64_t scatter_bits(uint64_t x, const uint8_t* sh, int nbits) {
    int64_t o = 0;
    for (int i = 0; i < nbits; ++i)
        if (((x >> i) & 1ull) && sh[i] != kNoBit) o += (int64_t)1 << sh[i];
    return o;
}

// Scale slots are read through L2 (ld.global.cg): inside a dataflow launch
// other CTAs write them, and a line an earlier item left in this SM's L1
// could be stale.
__device__ __forceinline__ int exp_of(const unsigned* slot) {
    if (slot == nullptr) return 0;
    float m = __uint_as_float(__ldcg(slot));
    if (!(m > 0.f)) return 0;
    int e;
    frexpf(m, &e);
    return e;
}

__device__ __forceinline__ int64_t slice_off(const SliceDigits& d, int64_t slice) {
    int64_t off = 0;
    for (int i = 0; i < d.n; ++i) off += ((slice / d.div[i]) % d.dim[i]) * d.stride[i];
    return off;
}

__device__ __forceinline__ int64_t min64(int64_t a, int64_t b) { return a < b ? a : b; }

// scaled load value, complex-conjugated when cj != 0 (a sign flip of Im)
__device__ __forceinline__ float2 cmul(float2 x, float f, int cj) {
    return make_float2(x.x * f, cj ? -x.y * f : x.y * f);
}
__device__ __forceinline__ float cmul(float x, float f, int) { return x * f; }
__device__ __forceinline__ float absmax(float2 x) { return fmaxf(fabsf(x.x), fabsf(x.y)); }
__device__ __forceinline__ float absmax(float x) { return fabsf(x); }
__device__ __forceinline__ void fma_acc(float2& c, float2 a, float2 b) {
    c.x = fmaf(a.x, b.x, c.x);
    c.x = fmaf(-a.y, b.y, c.x);
    c.y = fmaf(a.x, b.y, c.y);
    c.y = fmaf(a.y, b.x, c.y);
}
__device__ __forceinline__ void fma_acc(float& c, float a, float b) { c = fmaf(a, b, c); }
template <typename T>
__device__ __forceinline__ T zero();
template <>
__device__ __forceinline__ float2 zero<float2>() {
    return make_float2(0.f, 0.f);
}
template <>
__device__ __forceinline__ float zero<float>() {
    return 0.f;
}
__device__ __forceinline__ float2 add(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float add(float a, float b) { return a + b; }

__device__ __forceinline__ unsigned long long global_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ void block_max(float v, unsigned* slot) {
    __shared__ float red[32];
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (lane == 0) red[w] = v;
    __syncthreads();
    if (w == 0) {
        const int nw = (blockDim.x + 31) >> 5;
        v = lane < nw ? red[lane] : 0.f;
        for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
        if (lane == 0 && v > 0.f) atomicMax(slot, __float_as_uint(v));
    }
}

// Operand scales 2^-e (clamped so the float factor stays finite) and the
// residual exponent applied to the result.
struct Scales {
    float fa, fb;
    int resid;
};

// One instance's view of a node: operand/result pointers, scale slots and
// slice id, all offset by the instance index.
struct View {
    const void* A;
    const void* B;
    void* C;
    void* P;
    ScaleIO sc;
    int64_t slice;
    bool live;
};

template <class ARGS>
__device__ __forceinline__ View inst_view(const ARGS& a, int inst, int esz) {
    const InstanceInfo& in = a.in;
    View v;
    v.A = (const char*)a.A + (int64_t)inst * in.a_is * esz;
    v.B = (const char*)a.B + (int64_t)inst * in.b_is * esz;
    v.C = (char*)a.C + (int64_t)inst * in.c_is * esz;
    v.P = (char*)a.P + (int64_t)inst * in.p_is * esz;
    v.sc = a.sc;
    if (v.sc.max_a) v.sc.max_a += (int64_t)inst * in.sa_is;
    if (v.sc.exp_a) v.sc.exp_a += (int64_t)inst * in.sa_is;
    if (v.sc.max_b) v.sc.max_b += (int64_t)inst * in.sb_is;
    if (v.sc.exp_b) v.sc.exp_b += (int64_t)inst * in.sb_is;
    if (v.sc.max_c) v.sc.max_c += (int64_t)inst * in.sc_is;
    if (v.sc.exp_c) v.sc.exp_c += (int64_t)inst * in.sc_is;
    v.slice = a.ctl->slice + (int64_t)inst * in.slice_step;
    v.live = v.slice < a.ctl->slice_end;
    return v;
}

__device__ __forceinline__ Scales node_scales(const ScaleIO& sio, bool write_exp) {
    const int eA = exp_of(sio.max_a), eB = exp_of(sio.max_b);
    const int cA = max(-120, min(120, eA)), cB = max(-120, min(120, eB));
    if (write_exp && sio.exp_c)
        *sio.exp_c = (sio.exp_a ? __ldcg(sio.exp_a) : 0) + (sio.exp_b ? __ldcg(sio.exp_b) : 0) + eA + eB;
    Scales s;
    s.fa = ldexpf(1.f, -cA);
    s.fb = ldexpf(1.f, -cB);
    s.resid = (eA - cA) + (eB - cB);
    return s;
}

// node_scales from values already read: the children's max bits and
// exponents (0 where absent); exp_c (may be null) receives the node's
// exponent.
__device__ __forceinline__ Scales scales_from(unsigned ma, unsigned mb, int64_t ea, int64_t eb, int64_t* exp_c) {
    auto ex = [](unsigned bits) {
        const float m = __uint_as_float(bits);
        if (!(m > 0.f)) return 0;
        int e;
        frexpf(m, &e);
        return e;
    };
    const int eA = ex(ma), eB = ex(mb);
    const int cA = max(-120, min(120, eA)), cB = max(-120, min(120, eB));
    if (exp_c) *exp_c = ea + eb + eA + eB;
    Scales s;
    s.fa = ldexpf(1.f, -cA);
    s.fb = ldexpf(1.f, -cB);
    s.resid = (eA - cA) + (eB - cB);
    return s;
}

}  // namespace

template <bool CPLX>
__device__ __forceinline__ typename VT<CPLX>::T ld_cg(const typename VT<CPLX>::T* p) {
    if constexpr (CPLX) return __ldcg(reinterpret_cast<const float2*>(p));
    else return __ldcg(reinterpret_cast<const float*>(p));
}

// --------------------------------------------------------------------------
// Register-blocked tile: TM x TN outputs of one batch index and one K split;
// TK-deep steps through one shared-memory stage, 64-bit operand offsets.  This
// body serves the tile items of the persistent dataflow launch (CG: operands
// read through L2 only -- they may have been written earlier in the same launch
// by other CTAs) and k_tile_wide; the tile kernel below computes the same with
// two stages, more outputs per thread and 32-bit offsets.  A and B are the
// instance's operand bases; the epilogue writes C (or the K part's partial) and
// the maximum.
// --------------------------------------------------------------------------
template <bool CPLX, int TM, int TN, int TK, int RM, int RN, bool CG>
__device__ __forceinline__ void tile_body(const TileArgs& a, int64_t tile_x, int split_id, int64_t b,
                                          const View& vw, const typename VT<CPLX>::T* A,
                                          const typename VT<CPLX>::T* B, const Scales& sc) {
    using T = typename VT<CPLX>::T;
    constexpr int TX = TN / RN, TY = TM / RM, NT = TX * TY;
    constexpr int PB = CPLX ? 2 : 4;  // keeps sB rows 16-byte aligned
    __shared__ T sA[TK][TM + 1];
    __shared__ __align__(16) T sB[TK][TN + PB];
    __shared__ int64_t rowA[TM], colB[TN], kA[TK], kB[TK];
    auto ldx = [](const T* p) -> T {
        if constexpr (CG) return ld_cg<CPLX>(p);
        else return *p;
    };

    const int tid = threadIdx.x;
    const int64_t M = 1ll << a.nm, N = 1ll << a.nn, K = 1ll << a.nk;
    const int64_t tiles_n = (N + TN - 1) / TN;
    const int64_t m0 = (tile_x / tiles_n) * TM;
    const int64_t n0 = (tile_x % tiles_n) * TN;
    const int64_t slice = vw.slice;
    const int64_t baseA =
        slice_off(a.sla, slice) + scatter_bits(b, a.a_b, a.nb) + scatter_bits(m0, a.a_m, a.nm);
    const int64_t baseB =
        slice_off(a.slb, slice) + scatter_bits(b, a.b_b, a.nb) + scatter_bits(n0, a.b_n, a.nn);
    for (int i = tid; i < TM; i += NT) rowA[i] = scatter_bits(i, a.a_m, a.nm);
    for (int j = tid; j < TN; j += NT) colB[j] = scatter_bits(j, a.b_n, a.nn);
    for (int t = tid; t < TK; t += NT) {
        kA[t] = scatter_bits(t, a.a_k, a.nk);
        kB[t] = scatter_bits(t, a.b_k, a.nk);
    }
    __syncthreads();
    const int mlim = (int)min64(M - m0, TM);
    const int nlim = (int)min64(N - n0, TN);
    const int64_t kbeg = (int64_t)split_id * a.kchunk;
    const int64_t kend = min64(K, kbeg + a.kchunk);
    const int tx = tid % TX, ty = tid / TX;

    T acc[RM][RN];
#pragma unroll
    for (int r = 0; r < RM; ++r)
#pragma unroll
        for (int c = 0; c < RN; ++c) acc[r][c] = zero<T>();

    // global -> registers for one K step (all loads issued back to back).
    // The operand offsets of the K step's base k0 are kept incrementally:
    // k0 advances by TK, so only the bits of its carry chain change.
    constexpr int LA = (TM * TK + NT - 1) / NT, LB = (TN * TK + NT - 1) / NT;
    constexpr int LG_TK = TK == 16 ? 4 : (TK == 8 ? 3 : (TK == 4 ? 2 : 0));
    static_assert((1 << LG_TK) == TK, "TK must be a power of two");
    T ra[LA], rb[LB];
    int64_t cur_k = kbeg;
    int64_t kaA = scatter_bits(kbeg, a.a_k, a.nk), kaB = scatter_bits(kbeg, a.b_k, a.nk);
    auto step_k = [&]() {  // cur_k += TK, offsets follow
        int i = LG_TK;
        while (i < a.nk && ((cur_k >> i) & 1)) {
            if (a.a_k[i] != kNoBit) kaA -= int64_t(1) << a.a_k[i];
            if (a.b_k[i] != kNoBit) kaB -= int64_t(1) << a.b_k[i];
            ++i;
        }
        if (i < a.nk) {
            if (a.a_k[i] != kNoBit) kaA += int64_t(1) << a.a_k[i];
            if (a.b_k[i] != kNoBit) kaB += int64_t(1) << a.b_k[i];
        }
        cur_k += TK;
    };
    auto gload = [&](int64_t k0) {
        const int klim = (int)min64(kend - k0, TK);
#pragma unroll
        for (int q = 0; q < LA; ++q) {
            const int e = tid + q * NT;
            const int i = a.a_mfast ? e % TM : e / TK;
            const int t = a.a_mfast ? e / TM : e % TK;
            const bool in = e < TM * TK && i < mlim && t < klim;
            ra[q] = in ? cmul(ldx(A + baseA + rowA[i] + kaA + kA[t]), sc.fa, a.conj_a) : zero<T>();
        }
#pragma unroll
        for (int q = 0; q < LB; ++q) {
            const int e = tid + q * NT;
            const int j = a.b_nfast ? e % TN : e / TK;
            const int t = a.b_nfast ? e / TN : e % TK;
            const bool in = e < TN * TK && j < nlim && t < klim;
            rb[q] = in ? cmul(ldx(B + baseB + colB[j] + kaB + kB[t]), sc.fb, a.conj_b) : zero<T>();
        }
    };
    if (kbeg < kend) gload(kbeg);
    for (int64_t k0 = kbeg; k0 < kend; k0 += TK) {
        // kaA/kaB describe k0 here; gload of k0 + TK needs them advanced
#pragma unroll
        for (int q = 0; q < LA; ++q) {
            const int e = tid + q * NT;
            if (e < TM * TK) {
                const int i = a.a_mfast ? e % TM : e / TK;
                const int t = a.a_mfast ? e / TM : e % TK;
                sA[t][i] = ra[q];
            }
        }
#pragma unroll
        for (int q = 0; q < LB; ++q) {
            const int e = tid + q * NT;
            if (e < TN * TK) {
                const int j = a.b_nfast ? e % TN : e / TK;
                const int t = a.b_nfast ? e / TN : e % TK;
                sB[t][j] = rb[q];
            }
        }
        __syncthreads();
        if (k0 + TK < kend) {
            step_k();
            gload(k0 + TK);  // next step's loads overlap this step's FMAs
        }
#pragma unroll 4
        for (int t = 0; t < TK; ++t) {
            T af[RM], bf[RN];
#pragma unroll
            for (int r = 0; r < RM; ++r) af[r] = sA[t][ty * RM + r];
#pragma unroll
            for (int c = 0; c < RN; ++c) bf[c] = sB[t][tx + c * TX];  // conflict-free
#pragma unroll
            for (int r = 0; r < RM; ++r)
#pragma unroll
                for (int c = 0; c < RN; ++c) fma_acc(acc[r][c], af[r], bf[c]);
        }
        __syncthreads();
    }

    // epilogue: direct output (one split) or a partial for the reduce pass
    float lmax = 0.f;
    T* out = reinterpret_cast<T*>(a.split > 1 ? vw.P : vw.C);
    const int64_t plane = (a.split > 1 ? (int64_t)split_id * ((int64_t)a.nbatch) : 0) + b;
#pragma unroll
    for (int r = 0; r < RM; ++r) {
        const int i = ty * RM + r;
        if (i >= mlim) continue;
        const int64_t rowoff = (plane * M + m0 + i) * N + n0;
#pragma unroll
        for (int c = 0; c < RN; ++c) {
            const int j = tx + c * TX;
            if (j >= nlim) continue;
            T v = acc[r][c];
            if (a.split == 1) {
                if (sc.resid) {
                    if constexpr (CPLX) {
                        v.x = ldexpf(v.x, -sc.resid);
                        v.y = ldexpf(v.y, -sc.resid);
                    } else {
                        v = ldexpf(v, -sc.resid);
                    }
                }
                lmax = fmaxf(lmax, absmax(v));
            }
            out[rowoff + j] = v;
        }
    }
    if (a.split == 1) {
        block_max(lmax, vw.sc.max_c);
        if (a.t_done && threadIdx.x == 0) atomicMax(a.t_done, global_ns());
    }
}

// Operands spread over 2^31 entries (a slice of a larger leaf, so at least 8 GB
// of it): the body above, whose operand offsets are 64-bit.  Bound like k_tile by
// the FP32 pipes and shared-memory loads, at about half its rate (2^11 x 2^11 x
// 2^10, real: 523 us, 294 in k_tile): one stage and 4 x 4 outputs per thread.
template <bool CPLX, int TM, int TN, int TK>
__global__ void __launch_bounds__((TM / 4) * (TN / 4)) k_tile_wide(const __grid_constant__ TileArgs a) {
    using T = typename VT<CPLX>::T;
    const int per_inst = (int)(a.nbatch * a.split);
    const int zz = blockIdx.z % per_inst;
    const View vw = inst_view(a, blockIdx.z / per_inst, (int)sizeof(T));
    if (!vw.live) return;
    const Scales sc = node_scales(vw.sc, blockIdx.x == 0 && zz == 0 && threadIdx.x == 0);
    tile_body<CPLX, TM, TN, TK, 4, 4, false>(a, blockIdx.x, zz % a.split, zz / a.split, vw,
                                             reinterpret_cast<const T*>(vw.A), reinterpret_cast<const T*>(vw.B), sc);
}

// --------------------------------------------------------------------------
// Index groups of the two argument forms.  TileArgs (power-of-two sizes): an
// offset is a scatter of index bits.  GenericArgs (any sizes): mixed-radix
// digits, the output's fastest first (N digits, then M, then batch).
// --------------------------------------------------------------------------
__device__ __forceinline__ int64_t size_m(const TileArgs& a) { return 1ll << a.nm; }
__device__ __forceinline__ int64_t size_n(const TileArgs& a) { return 1ll << a.nn; }
__device__ __forceinline__ int64_t size_k(const TileArgs& a) { return 1ll << a.nk; }
__device__ __forceinline__ int64_t off_m(const TileArgs& a, int64_t m) { return scatter_bits(m, a.a_m, a.nm); }
__device__ __forceinline__ int64_t off_n(const TileArgs& a, int64_t n) { return scatter_bits(n, a.b_n, a.nn); }
__device__ __forceinline__ void off_k(const TileArgs& a, int64_t k, int64_t& ka, int64_t& kb) {
    ka = scatter_bits(k, a.a_k, a.nk);
    kb = scatter_bits(k, a.b_k, a.nk);
}
__device__ __forceinline__ void off_b(const TileArgs& a, int64_t b, int64_t& ba, int64_t& bb) {
    ba = scatter_bits(b, a.a_b, a.nb);
    bb = scatter_bits(b, a.b_b, a.nb);
}

__device__ __forceinline__ int64_t size_m(const GenericArgs& a) { return a.M; }
__device__ __forceinline__ int64_t size_n(const GenericArgs& a) { return a.N; }
__device__ __forceinline__ int64_t size_k(const GenericArgs& a) { return a.n_sum; }
// digits [j0, j1) of x (below 2^31: the planner's condition) with strides st
__device__ __forceinline__ int64_t digits(unsigned x, const int32_t* dim, const int64_t* st, int j0, int j1) {
    int64_t o = 0;
    for (int j = j0; j < j1; ++j) {
        const unsigned d = (unsigned)dim[j], q = x / d;
        o += (int64_t)(x - q * d) * st[j];
        x = q;
    }
    return o;
}
__device__ __forceinline__ int64_t off_m(const GenericArgs& a, int64_t m) {
    return digits((unsigned)m, a.od_dim, a.od_sa, a.n_nd, a.n_nd + a.n_md);
}
__device__ __forceinline__ int64_t off_n(const GenericArgs& a, int64_t n) {
    return digits((unsigned)n, a.od_dim, a.od_sb, 0, a.n_nd);
}
__device__ __forceinline__ void off_k(const GenericArgs& a, int64_t k, int64_t& ka, int64_t& kb) {
    ka = digits((unsigned)k, a.kd_dim, a.kd_sa, 0, a.n_kd);
    kb = digits((unsigned)k, a.kd_dim, a.kd_sb, 0, a.n_kd);
}
__device__ __forceinline__ void off_b(const GenericArgs& a, int64_t b, int64_t& ba, int64_t& bb) {
    ba = digits((unsigned)b, a.od_dim, a.od_sa, a.n_nd + a.n_md, a.n_od);
    bb = digits((unsigned)b, a.od_dim, a.od_sb, a.n_nd + a.n_md, a.n_od);
}

// --------------------------------------------------------------------------
// The tile kernel: one CTA = TM x TN outputs of one batch index and one K
// split, RM x RN of them per thread.
//
// Bound by the FP32 pipes for large K, by the operand loads from shared
// memory before that: a thread holds 8 x 4 outputs (real: 8 x 8 in the largest
// tiles), reads them 16 bytes at a time -- two complex or four real entries of
// a row of either operand -- and K is stepped by 8 through two shared-memory
// stages, the next step's global loads in flight during this step's
// multiply-adds, one barrier a step.  Per-thread operand offsets within a step
// are kept in registers; the K base follows its carry chain (power-of-two
// sizes) or a table of 1024 K offsets in shared memory (any sizes).
// 2^11 x 2^11 x 2^10, complex: 1029 us with 4 x 4 outputs per thread, 8-byte
// loads and 64-bit address sums per entry, 732 now (47 TFLOP/s; 2^12 x 2^12:
// 51); real: 421 -> 256.  The paired multiply-add fma.rn.f32x2 was tried in
// its place and is no faster here (47 TFLOP/s on the larger node): its three
// 64-bit operands issue every third cycle.
// --------------------------------------------------------------------------
constexpr int kTabK = 1024;  // K offsets held in shared memory (any sizes)

template <class ARGS, bool CPLX, int TM, int TN, int TK>
struct TileSmem {
    using T = typename VT<CPLX>::T;
    static constexpr int PAD = CPLX ? 2 : 4;  // 16 bytes a row: no bank conflicts in stores along K
    static constexpr size_t a_bytes = (size_t)TK * (TM + PAD) * sizeof(T);
    static constexpr size_t b_bytes = (size_t)TK * (TN + PAD) * sizeof(T);
    static constexpr size_t tab_bytes = std::is_same<ARGS, GenericArgs>::value ? 2 * kTabK * sizeof(int32_t) : 0;
    static constexpr size_t bytes = 2 * (a_bytes + b_bytes) + tab_bytes;
};

template <class ARGS, bool CPLX, int TM, int TN, int TK, int RM, int RN, int MINB>
__global__ void __launch_bounds__((TM / RM) * (TN / RN), MINB)
    k_tile(const __grid_constant__ ARGS a) {
    using T = typename VT<CPLX>::T;
    using SM = TileSmem<ARGS, CPLX, TM, TN, TK>;
    constexpr bool ANY = std::is_same<ARGS, GenericArgs>::value;
    constexpr int TX = TN / RN, TY = TM / RM, NT = TX * TY;
    constexpr int RP = CPLX ? RN : RN / 2;  // accumulator pairs per row
    constexpr int VB = CPLX ? 2 : 4;        // entries per 16-byte load
    static_assert(RN % VB == 0 && RM % VB == 0, "thread tile");
    extern __shared__ __align__(16) unsigned char tile_smem[];
    __shared__ int64_t rowA[TM], colB[TN];
    auto sA = [&](int st, int t) { return reinterpret_cast<T*>(tile_smem + st * SM::a_bytes) + t * (TM + SM::PAD); };
    auto sB = [&](int st, int t) {
        return reinterpret_cast<T*>(tile_smem + 2 * SM::a_bytes + st * SM::b_bytes) + t * (TN + SM::PAD);
    };
    int32_t* const tabA = reinterpret_cast<int32_t*>(tile_smem + 2 * (SM::a_bytes + SM::b_bytes));
    int32_t* const tabB = tabA + kTabK;

    const int tid = threadIdx.x;
    const int64_t M = size_m(a), N = size_n(a), K = size_k(a);
    const int64_t tiles_n = (N + TN - 1) / TN;
    const int64_t m0 = ((int64_t)blockIdx.x / tiles_n) * TM;
    const int64_t n0 = ((int64_t)blockIdx.x % tiles_n) * TN;
    const int per_inst = (int)(a.nbatch * a.split);
    const int inst = blockIdx.z / per_inst;
    const int zz = blockIdx.z % per_inst;
    const int split_id = zz % a.split;
    const int64_t b = zz / a.split;
    const View vw = inst_view(a, inst, (int)sizeof(T));
    if (!vw.live) return;
    const Scales sc = node_scales(vw.sc, blockIdx.x == 0 && zz == 0 && tid == 0);
    const int mlim = (int)min64(M - m0, TM);
    const int nlim = (int)min64(N - n0, TN);
    const int64_t kbeg = (int64_t)split_id * a.kchunk;
    const int64_t kend = min64(K, kbeg + a.kchunk);
    for (int i = tid; i < mlim; i += NT) rowA[i] = off_m(a, m0 + i);
    for (int j = tid; j < nlim; j += NT) colB[j] = off_n(a, n0 + j);
    int64_t ba, bb;
    off_b(a, b, ba, bb);
    const T* A = reinterpret_cast<const T*>(vw.A) + slice_off(a.sla, vw.slice) + ba;
    const T* B = reinterpret_cast<const T*>(vw.B) + slice_off(a.slb, vw.slice) + bb;
    __syncthreads();
    const int tx = tid % TX, ty = tid / TX;

    // this thread's entries of a K step: entry q of an operand tile of S rows
    // (columns) is row i0 + q di, K index t0 + q dt, along the rows or along K
    // as the operand is contiguous
    constexpr int LA = (TM * TK + NT - 1) / NT, LB = (TN * TK + NT - 1) / NT;
    constexpr int LG_TK = TK == 16 ? 4 : (TK == 8 ? 3 : 2);
    static_assert((1 << LG_TK) == TK, "TK must be a power of two");
    struct Walk {
        int i0, t0, di, dt;
        bool wrap;  // S > NT, along the rows: S / NT entries per K index
    };
    auto walk = [&](int S, bool along_rows) {
        Walk w;
        w.wrap = along_rows && S > NT;
        if (along_rows) {
            w.i0 = S > NT ? tid : tid % S;
            w.t0 = S > NT ? 0 : tid / S;
            w.di = 0;
            w.dt = S > NT ? 0 : NT / S;
        } else {
            w.i0 = tid / TK;
            w.t0 = tid % TK;
            w.di = NT / TK;
            w.dt = 0;
        }
        if (tid >= S * TK) w.i0 = S;  // fewer entries than threads: none for this one
        return w;
    };
    const Walk wa = walk(TM, a.a_mfast != 0), wb = walk(TN, a.b_nfast != 0);
    auto row_of = [&](const Walk& w, int q, int S) { return w.wrap ? w.i0 + q % (S > NT ? S / NT : 1) * NT : w.i0 + q * w.di; };
    auto k_of = [&](const Walk& w, int q, int S) { return w.wrap ? q / (S > NT ? S / NT : 1) : w.t0 + q * w.dt; };
    // offset in the operand without the K base (sizes of any kind: without K)
    int offA[LA], offB[LB];  // the planner sends operands that reach 2^31 entries elsewhere (TileArgs::wide)
#pragma unroll
    for (int q = 0; q < LA; ++q) {
        const int i = row_of(wa, q, TM);
        offA[q] = i < mlim ? (int)rowA[i] : 0;
        if constexpr (!ANY) offA[q] += (int)scatter_bits(k_of(wa, q, TM), a.a_k, min(a.nk, LG_TK));
    }
#pragma unroll
    for (int q = 0; q < LB; ++q) {
        const int j = row_of(wb, q, TN);
        offB[q] = j < nlim ? (int)colB[j] : 0;
        if constexpr (!ANY) offB[q] += (int)scatter_bits(k_of(wb, q, TN), a.b_k, min(a.nk, LG_TK));
    }

    float2 acc[RM][RP];
#pragma unroll
    for (int r = 0; r < RM; ++r)
#pragma unroll
        for (int c = 0; c < RP; ++c) acc[r][c] = make_float2(0.f, 0.f);

    T ra[LA], rb[LB];
    int64_t cur_k = kbeg, kaA = 0, kaB = 0;
    if constexpr (!ANY) off_k(a, kbeg, kaA, kaB);
    [[maybe_unused]] auto step_k = [&]() {  // cur_k += TK, the K base follows its carry chain
        if constexpr (!ANY) {
            int i = LG_TK;
            while (i < a.nk && ((cur_k >> i) & 1)) {
                if (a.a_k[i] != kNoBit) kaA -= int64_t(1) << a.a_k[i];
                if (a.b_k[i] != kNoBit) kaB -= int64_t(1) << a.b_k[i];
                ++i;
            }
            if (i < a.nk) {
                if (a.a_k[i] != kNoBit) kaA += int64_t(1) << a.a_k[i];
                if (a.b_k[i] != kNoBit) kaB += int64_t(1) << a.b_k[i];
            }
            cur_k += TK;
        }
    };
    // global -> registers for the K step at k0 (all loads back to back); w0:
    // first K index of the offset table
    auto gload = [&](int64_t k0, [[maybe_unused]] int64_t w0) {
        const int klim = (int)min64(kend - k0, TK);
#pragma unroll
        for (int q = 0; q < LA; ++q) {
            const int i = row_of(wa, q, TM), t = k_of(wa, q, TM);
            ra[q] = zero<T>();
            if (i < mlim && t < klim) {
                if constexpr (ANY) ra[q] = A[offA[q] + tabA[(int)(k0 - w0) + t]];
                else ra[q] = A[kaA + offA[q]];
            }
        }
#pragma unroll
        for (int q = 0; q < LB; ++q) {
            const int j = row_of(wb, q, TN), t = k_of(wb, q, TN);
            rb[q] = zero<T>();
            if (j < nlim && t < klim) {
                if constexpr (ANY) rb[q] = B[offB[q] + tabB[(int)(k0 - w0) + t]];
                else rb[q] = B[kaB + offB[q]];
            }
        }
    };
    auto stash = [&](int st) {  // registers -> shared memory, scaled
#pragma unroll
        for (int q = 0; q < LA; ++q) {
            const int i = row_of(wa, q, TM);
            if (i < TM) sA(st, k_of(wa, q, TM))[i] = cmul(ra[q], sc.fa, a.conj_a);
        }
#pragma unroll
        for (int q = 0; q < LB; ++q) {
            const int j = row_of(wb, q, TN);
            if (j < TN) sB(st, k_of(wb, q, TN))[j] = cmul(rb[q], sc.fb, a.conj_b);
        }
    };
    auto multiply = [&](int st) {
#pragma unroll
        for (int t = 0; t < TK; ++t) {
            float4 bv[RN / VB];
#pragma unroll
            for (int c = 0; c < RN / VB; ++c)
                bv[c] = *reinterpret_cast<const float4*>(sB(st, t) + (tx + c * TX) * VB);
            float4 av[RM / VB];
#pragma unroll
            for (int r = 0; r < RM / VB; ++r) av[r] = *reinterpret_cast<const float4*>(sA(st, t) + ty * RM + r * VB);
            const float* af = reinterpret_cast<const float*>(av);
            const float* bf = reinterpret_cast<const float*>(bv);
#pragma unroll
            for (int r = 0; r < RM; ++r)
#pragma unroll
                for (int c = 0; c < RP; ++c) {
                    float2& x = acc[r][c];
                    if constexpr (CPLX) {
                        fma_acc(x, make_float2(af[2 * r], af[2 * r + 1]), make_float2(bf[2 * c], bf[2 * c + 1]));
                    } else {
                        x.x = fmaf(af[r], bf[2 * c], x.x);
                        x.y = fmaf(af[r], bf[2 * c + 1], x.y);
                    }
                }
        }
    };
    // window by window of the K offset table (power-of-two sizes: one window)
    const int64_t win = ANY ? kTabK : (kend > kbeg ? kend - kbeg : 1);
    for (int64_t w0 = kbeg; w0 < kend; w0 += win) {
        const int64_t w1 = min64(kend, w0 + win);
        if constexpr (ANY) {
            __syncthreads();  // the table's and the stages' last readers are done
            for (int t = tid; t < (int)(w1 - w0); t += NT) {
                int64_t ka, kb;
                off_k(a, w0 + t, ka, kb);
                tabA[t] = (int32_t)ka;
                tabB[t] = (int32_t)kb;
            }
            __syncthreads();
        }
        gload(w0, w0);
        stash(0);
        __syncthreads();
        int st = 0;
        for (int64_t k0 = w0; k0 < w1; k0 += TK) {
            const bool more = k0 + TK < w1;
            if (more) {
                step_k();
                gload(k0 + TK, w0);
            }
            multiply(st);
            if (more) {
                st ^= 1;
                stash(st);
                __syncthreads();
            }
        }
    }

    // epilogue: direct output (one split) or a partial for the reduce pass
    float lmax = 0.f;
    T* out = reinterpret_cast<T*>(a.split > 1 ? vw.P : vw.C);
    const int64_t plane = (a.split > 1 ? (int64_t)split_id * a.nbatch : 0) + b;
    // whole 16-byte stores where every row starts on 16 bytes
    const bool vec = N % VB == 0 && (reinterpret_cast<uintptr_t>(out) & 15) == 0;
#pragma unroll
    for (int r = 0; r < RM; ++r) {
        const int i = ty * RM + r;
        if (i >= mlim) continue;
        T* row = out + (plane * M + m0 + i) * N + n0;
#pragma unroll
        for (int c = 0; c < RN / VB; ++c) {
            const int j = (tx + c * TX) * VB;
            if (j >= nlim) continue;
            float4 v = make_float4(acc[r][2 * c].x, acc[r][2 * c].y, acc[r][2 * c + 1].x, acc[r][2 * c + 1].y);
            if (a.split == 1) {
                if (sc.resid) {
                    v.x = ldexpf(v.x, -sc.resid);
                    v.y = ldexpf(v.y, -sc.resid);
                    v.z = ldexpf(v.z, -sc.resid);
                    v.w = ldexpf(v.w, -sc.resid);
                }
                // columns beyond the node's hold zeros
                lmax = fmaxf(fmaxf(lmax, fmaxf(fabsf(v.x), fabsf(v.y))), fmaxf(fabsf(v.z), fabsf(v.w)));
            }
            if (vec) {
                *reinterpret_cast<float4*>(row + j) = v;
            } else if constexpr (CPLX) {
                row[j] = make_float2(v.x, v.y);
                if (j + 1 < nlim) row[j + 1] = make_float2(v.z, v.w);
            } else {
                row[j] = v.x;
                if (j + 1 < nlim) row[j + 1] = v.y;
                if (j + 2 < nlim) row[j + 2] = v.z;
                if (j + 3 < nlim) row[j + 3] = v.w;
            }
        }
    }
    if (a.split == 1) {
        block_max(lmax, vw.sc.max_c);
        if (a.t_done && threadIdx.x == 0) atomicMax(a.t_done, global_ns());
    }
}

// Sums the K-split partials of a node in a fixed order and applies its
// epilogue.  G threads share one output (G = 1 when the outputs alone fill
// the GPU): thread g sums splits [g*split/G, (g+1)*split/G) in eight
// independent chains, then the G sums are added in g order.
template <class ARGS, bool CPLX>
__global__ void __launch_bounds__(256) k_split_reduce(const __grid_constant__ ARGS a, int G) {
    using T = typename VT<CPLX>::T;
    __shared__ T red[256];
    const int64_t plane_sz = a.nbatch * size_m(a) * size_n(a);
    const View vw = inst_view(a, blockIdx.y, (int)sizeof(T));
    if (!vw.live) return;
    const Scales sc = node_scales(vw.sc, blockIdx.x == 0 && threadIdx.x == 0);
    const T* P = reinterpret_cast<const T*>(vw.P);
    T* C = reinterpret_cast<T*>(vw.C);
    const int tid = threadIdx.x, g = tid % G, per_blk = 256 / G;
    const int s0 = (int)((int64_t)a.split * g / G), s1 = (int)((int64_t)a.split * (g + 1) / G);
    float lmax = 0.f;
    for (int64_t ob = (int64_t)blockIdx.x * per_blk; ob < plane_sz; ob += (int64_t)gridDim.x * per_blk) {
        const int64_t o = ob + tid / G;
        T v = zero<T>();
        if (o < plane_sz) {
            T part[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) part[q] = zero<T>();
            int sp = s0;
            for (; sp + 8 <= s1; sp += 8)
#pragma unroll
                for (int q = 0; q < 8; ++q) part[q] = add(part[q], P[(int64_t)(sp + q) * plane_sz + o]);
            for (int q = 0; sp < s1; ++sp, ++q) part[q] = add(part[q], P[(int64_t)sp * plane_sz + o]);
            v = add(add(add(part[0], part[1]), add(part[2], part[3])),
                    add(add(part[4], part[5]), add(part[6], part[7])));
        }
        if (G > 1) {  // uniform over the block: every thread runs the same iterations
            red[tid] = v;
            __syncthreads();
            if (g == 0)
                for (int q = 1; q < G; ++q) v = add(v, red[tid + q]);
            __syncthreads();
        }
        if (g != 0 || o >= plane_sz) continue;
        if (sc.resid) {
            if constexpr (CPLX) {
                v.x = ldexpf(v.x, -sc.resid);
                v.y = ldexpf(v.y, -sc.resid);
            } else {
                v = ldexpf(v, -sc.resid);
            }
        }
        lmax = fmaxf(lmax, absmax(v));
        C[o] = v;
    }
    block_max(lmax, vw.sc.max_c);
    if (a.t_done && threadIdx.x == 0) atomicMax(a.t_done, global_ns());
}

// Inner-product node (2 to 64 outputs, long K, more than two tiles of 1024
// products per SM: dot_each_output in tn_plan.cpp): out[b,m,n] = sum_k A[.., k] B[.., k].
// One CTA computes all outputs of a batch entry over its part of K, so that
// either operand is read once.  K is cut into tiles of 2^t entries that hold
// the lowest strides of A and of B; a tile of an operand -- its rows times the
// tile's K entries -- is read in the operand's own order (consecutive threads,
// consecutive addresses) by asynchronous copies straight into shared memory,
// where each entry lands at its row and K position.  A ring of kDotStages
// tiles keeps two tiles of copies in flight per CTA while a third is
// multiplied; the tile base offsets follow the tile index by its carry chain.
// Each thread multiplies RM x RN outputs over every LPG-th K entry (LPG threads
// share a group of outputs).  blockIdx.x: batch entry, y: `parts` consecutive K
// parts (short parts share a CTA and its setup, each with its own partial, so
// that the sum does not depend on the grid), z: instance.  The batch entries of
// a K part run together: where they are an operand's fastest label they read
// the same lines (16 entries over K = 2^20 and 4 outputs, complex: 1098 us with
// the K parts of an entry together, 458 this way).
// Bound by memory for few outputs, for many by the instructions of its copies.
// A node of 16 outputs over K = 2^18 in eight copies, 134 MB:
// 262 us with one CTA per output and K part, which read each operand once per
// row or column of the other, 61 now (89 with more CTAs than fit at a time).
constexpr int kDotStages = 3;
constexpr int kDotPer = kDotEntries / 256;   // copies per thread and tile
constexpr int kDotTile = 1 << (2 * kDotLow);  // K entries of a tile of one output
// one padding entry per 32 of a row and one a row: no bank conflicts along K or along the rows
__host__ __device__ constexpr int dot_row(int t) { return (1 << t) + (1 << t) / 32 + 1; }

// the stages, then offset (4 bytes) and stage position (2) of every entry of a tile
inline size_t dot_smem_bytes(const DotPlan& dp, int rows, size_t esz) {
    return (size_t)kDotStages * rows * dot_row(dp.t) * esz + (size_t)kDotEntries * 6;
}

// asynchronous global -> shared copy of one 4- or 8-byte element
template <int BYTES>
__device__ __forceinline__ void cp_async_elem(void* dst, const void* src) {
    const uint32_t d = static_cast<uint32_t>(__cvta_generic_to_shared(dst));
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(d), "l"(src), "n"(BYTES) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

__device__ __forceinline__ float shfl_xor(float v, int o) { return __shfl_xor_sync(0xffffffffu, v, o); }
__device__ __forceinline__ float2 shfl_xor(float2 v, int o) { return make_float2(shfl_xor(v.x, o), shfl_xor(v.y, o)); }

// CTAs per SM (registers: RM x RN sums per thread)
constexpr int dot_resident(bool cplx, int outs) { return cplx && outs >= 8 ? 2 : 3; }

template <bool CPLX, int RM, int RN>
__global__ void __launch_bounds__(256, dot_resident(CPLX, RM * RN))
    k_dot(const __grid_constant__ TileArgs a, const __grid_constant__ DotPlan dp, int parts) {
    using T = typename VT<CPLX>::T;
    extern __shared__ __align__(16) unsigned char dot_smem[];
    T* const stg = reinterpret_cast<T*>(dot_smem);  // [stage][rows of A, then of B][dot_row]
    __shared__ T red[8][64];
    const int tid = threadIdx.x;
    const int N = 1 << a.nn, M = 1 << a.nm;
    const int64_t b = blockIdx.x;
    const View vw = inst_view(a, blockIdx.z, (int)sizeof(T));
    if (!vw.live) return;
    const Scales sc = node_scales(vw.sc, blockIdx.x == 0 && blockIdx.y == 0 && tid == 0);
    const int t = dp.t, u = dp.u, tsz = 1 << t;
    const int row = dot_row(t), stage_sz = (M + N) * row;
    // the copies of a tile: entries of A in A's order, then of B
    const int n_a = M << t, n_ab = (M + N) << t;
    int32_t* const off = reinterpret_cast<int32_t*>(stg + (size_t)kDotStages * stage_sz);
    uint16_t* const pos = reinterpret_cast<uint16_t*>(off + kDotEntries);
    for (int e0 = tid; e0 < n_ab; e0 += 256) {
        const bool is_b = e0 >= n_a;
        const int e = is_b ? e0 - n_a : e0, bits = t + (is_b ? a.nn : a.nm);
        int o = 0, c = is_b ? M << 16 : 0;
        for (int w = 0; w < bits; ++w)
            if ((e >> w) & 1) {  // offsets within one operand, below 2^31 entries (TileArgs::wide)
                o += (int)(is_b ? dp.b_add : dp.a_add)[w];
                c += (is_b ? dp.cb_add : dp.ca_add)[w];
            }
        const int k = c & 0xffff;
        off[e0] = o;
        pos[e0] = (uint16_t)((c >> 16) * row + k + (k >> 5));
    }
    __syncthreads();
    const int64_t slice = vw.slice;
    const T* A = reinterpret_cast<const T*>(vw.A) + slice_off(a.sla, slice) + scatter_bits(b, a.a_b, a.nb);
    const T* B = reinterpret_cast<const T*>(vw.B) + slice_off(a.slb, slice) + scatter_bits(b, a.b_b, a.nb);
    const int64_t n_tiles = int64_t(1) << u;
    const int64_t per = (n_tiles + a.split - 1) / a.split;
    int left = (int)min64(per, 1 << 30);  // tiles to the end of the current part
    const int64_t t0 = (int64_t)blockIdx.y * parts * per, t1 = min64(n_tiles, t0 + parts * per);
    // offsets of the next tile to copy; advanced tile by tile along the carry chain
    int64_t nt = t0, ba = 0, bb = 0;
    for (int j = 0; j < u; ++j)
        if ((t0 >> j) & 1) {
            ba += dp.rest_a[j];
            bb += dp.rest_b[j];
        }
    auto issue = [&](int stage) {
        if (nt < t1) {
            T* st = stg + (size_t)stage * stage_sz;
#pragma unroll
            for (int r = 0; r < kDotPer; ++r) {
                const int e = tid + r * 256;
                if (e < n_ab) cp_async_elem<sizeof(T)>(st + pos[e], (e < n_a ? A + ba : B + bb) + off[e]);
            }
            int j = 0;
            while (j < u && ((nt >> j) & 1)) {
                ba -= dp.rest_a[j];
                bb -= dp.rest_b[j];
                ++j;
            }
            if (j < u) {
                ba += dp.rest_a[j];
                bb += dp.rest_b[j];
            }
            ++nt;
        }
        cp_async_commit();  // one group per call, empty or not: the wait counts stay uniform
    };
#pragma unroll
    for (int q = 0; q < kDotStages - 1; ++q) issue(q);
    // output groups: LPG consecutive threads share one
    const int groups = (M / RM) * (N / RN), lpg = 256 / groups;
    const int g = tid / lpg, lane = tid % lpg;
    const int gm = g / (N / RN) * RM, gn = g % (N / RN) * RN;
    T acc[RM][RN];
#pragma unroll
    for (int r = 0; r < RM; ++r)
#pragma unroll
        for (int c = 0; c < RN; ++c) acc[r][c] = zero<T>();
    int stage = 0;
    for (int64_t tile = t0; tile < t1; ++tile) {
        issue((stage + kDotStages - 1) % kDotStages);
        cp_async_wait<kDotStages - 1>();  // this thread's copies of `tile` have landed
        __syncthreads();                  // ... and every other thread's
        const T* sA = stg + (size_t)stage * stage_sz + gm * row;
        const T* sB = stg + (size_t)stage * stage_sz + (M + gn) * row;
#pragma unroll 4
        for (int i = lane; i < tsz; i += lpg) {
            const int ip = i + (i >> 5);
            T av[RM], bv[RN];
#pragma unroll
            for (int r = 0; r < RM; ++r) av[r] = cmul(sA[r * row + ip], sc.fa, a.conj_a);
#pragma unroll
            for (int c = 0; c < RN; ++c) bv[c] = cmul(sB[c * row + ip], sc.fb, a.conj_b);
#pragma unroll
            for (int r = 0; r < RM; ++r)
#pragma unroll
                for (int c = 0; c < RN; ++c) fma_acc(acc[r][c], av[r], bv[c]);
        }
        __syncthreads();  // the stage is refilled by the next iteration's copies
        stage = (stage + 1) % kDotStages;
        if (--left && tile + 1 < t1) continue;
        left = (int)min64(per, 1 << 30);
        // end of a K part.  Fixed-order reduction: the group's lanes of a
        // warp, then its warps
        const int span = lpg < 32 ? lpg : 32;
#pragma unroll
        for (int r = 0; r < RM; ++r)
#pragma unroll
            for (int c = 0; c < RN; ++c) {
                T v = acc[r][c];
                for (int o = span >> 1; o > 0; o >>= 1) v = add(v, shfl_xor(v, o));
                if (lane % 32 == 0) red[lane / 32][(gm + r) * N + gn + c] = v;
                acc[r][c] = zero<T>();
            }
        __syncthreads();
        if (tid < M * N) {
            T v = red[0][tid];
            for (int w = 1; w < (lpg + 31) / 32; ++w) v = add(v, red[w][tid]);
            const int64_t o = b * M * N + tid;
            if (a.split > 1) {
                reinterpret_cast<T*>(vw.P)[tile / per * (a.nbatch * M * N) + o] = v;
            } else {
                if (sc.resid) {
                    if constexpr (CPLX) {
                        v.x = ldexpf(v.x, -sc.resid);
                        v.y = ldexpf(v.y, -sc.resid);
                    } else {
                        v = ldexpf(v, -sc.resid);
                    }
                }
                reinterpret_cast<T*>(vw.C)[o] = v;
                const float mx = absmax(v);
                if (mx > 0.f) atomicMax(vw.sc.max_c, __float_as_uint(mx));
                if (a.t_done) atomicMax(a.t_done, global_ns());
            }
        }
        // (the next part's first barrier comes before its reduction writes red)
    }
    cp_async_wait<0>();
}

// One output per CTA: every thread multiplies its own four entries of a tile.
// blockIdx.x: batch entry and output, y: K part, z: instance.  For one-output
// nodes, several where the planner's rule says so, and (WIDE: 64-bit offsets)
// operands spread over 2^31 entries (8 x 4 outputs over K = 2^18, real: 52 us, 30
// in k_dot).  Bound by memory: one output over K = 2^28
// (4.3 GB) 726 us, 5.9 TB/s; as an instance of k_dot, whose loop over rows and
// parts costs registers and instructions per copy, 820 to 1105.
template <bool CPLX, bool WIDE>
__global__ void __launch_bounds__(256) k_dot_one(const __grid_constant__ TileArgs a, const __grid_constant__ DotPlan dp) {
    using T = typename VT<CPLX>::T;
    using O = typename std::conditional<WIDE, int64_t, int32_t>::type;  // offset within an operand
    extern __shared__ __align__(16) unsigned char dot_smem[];
    constexpr int kPad = kDotTile + kDotTile / 32;  // one padding entry per 32: no bank conflicts
    T* const stg = reinterpret_cast<T*>(dot_smem);  // [stage][A, B][kPad]
    O* const offA = reinterpret_cast<O*>(dot_smem + (size_t)kDotStages * 2 * kPad * sizeof(T));
    O* const offB = offA + kDotTile;
    uint16_t* const posA = reinterpret_cast<uint16_t*>(offB + kDotTile);
    uint16_t* const posB = posA + kDotTile;
    __shared__ T red[256];
    const int lg_out = a.nm + a.nn, out = (int)blockIdx.x & ((1 << lg_out) - 1), sp = (int)blockIdx.y;
    const int64_t b = blockIdx.x >> lg_out;
    const View vw = inst_view(a, blockIdx.z, (int)sizeof(T));
    if (!vw.live) return;
    const Scales sc = node_scales(vw.sc, blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0);
    const int t = dp.t, u = dp.u, tsz = 1 << t;
    for (int e = threadIdx.x; e < tsz; e += 256) {
        O xa = 0, xb = 0;
        int pa = 0, pb = 0;
        for (int w = 0; w < t; ++w)
            if ((e >> w) & 1) {
                xa += (O)dp.a_add[w];
                xb += (O)dp.b_add[w];
                pa += dp.ca_add[w];
                pb += dp.cb_add[w];
            }
        offA[e] = xa;
        offB[e] = xb;
        posA[e] = (uint16_t)(pa + (pa >> 5));
        posB[e] = (uint16_t)(pb + (pb >> 5));
    }
    __syncthreads();
    const int64_t slice = vw.slice;
    const T* A = reinterpret_cast<const T*>(vw.A) + slice_off(a.sla, slice) + scatter_bits(b, a.a_b, a.nb) +
                 scatter_bits(out >> a.nn, a.a_m, a.nm);
    const T* B = reinterpret_cast<const T*>(vw.B) + slice_off(a.slb, slice) + scatter_bits(b, a.b_b, a.nb) +
                 scatter_bits(out & ((1 << a.nn) - 1), a.b_n, a.nn);
    const int64_t n_tiles = int64_t(1) << u;
    const int64_t per = (n_tiles + a.split - 1) / a.split;
    const int64_t t0 = (int64_t)sp * per, t1 = min64(n_tiles, t0 + per);
    // offsets of the next tile to copy; advanced tile by tile along the carry chain
    int64_t nt = t0, ba = 0, bb = 0;
    for (int j = 0; j < u; ++j)
        if ((t0 >> j) & 1) {
            ba += dp.rest_a[j];
            bb += dp.rest_b[j];
        }
    auto issue = [&](int stage) {
        if (nt < t1) {
            T* sA = stg + (size_t)stage * 2 * kPad;
            T* sB = sA + kPad;
#pragma unroll
            for (int r = 0; r < kDotTile / 256; ++r) {
                const int e = threadIdx.x + r * 256;
                if (e < tsz) {
                    cp_async_elem<sizeof(T)>(sA + posA[e], A + ba + offA[e]);
                    cp_async_elem<sizeof(T)>(sB + posB[e], B + bb + offB[e]);
                }
            }
            int j = 0;
            while (j < u && ((nt >> j) & 1)) {
                ba -= dp.rest_a[j];
                bb -= dp.rest_b[j];
                ++j;
            }
            if (j < u) {
                ba += dp.rest_a[j];
                bb += dp.rest_b[j];
            }
            ++nt;
        }
        cp_async_commit();  // one group per call, empty or not: the wait counts stay uniform
    };
#pragma unroll
    for (int q = 0; q < kDotStages - 1; ++q) issue(q);
    T acc0 = zero<T>(), acc1 = zero<T>();
    int stage = 0;
    for (int64_t tile = t0; tile < t1; ++tile) {
        issue((stage + kDotStages - 1) % kDotStages);
        cp_async_wait<kDotStages - 1>();  // this thread's copies of `tile` have landed
        __syncthreads();                  // ... and every other thread's
        const T* sA = stg + (size_t)stage * 2 * kPad;
        const T* sB = sA + kPad;
#pragma unroll
        for (int r = 0; r < kDotTile / 256; ++r) {
            const int i = threadIdx.x + r * 256;
            if (i < tsz) {
                const int ip = i + (i >> 5);
                fma_acc(r & 1 ? acc1 : acc0, cmul(sA[ip], sc.fa, a.conj_a), cmul(sB[ip], sc.fb, a.conj_b));
            }
        }
        __syncthreads();  // the stage is refilled by the next iteration's copies
        stage = (stage + 1) % kDotStages;
    }
    cp_async_wait<0>();
    // fixed-order block reduction
    red[threadIdx.x] = add(acc0, acc1);
    __syncthreads();
    for (int s = 128; s > 0; s >>= 1) {
        if (threadIdx.x < s) red[threadIdx.x] = add(red[threadIdx.x], red[threadIdx.x + s]);
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        T v = red[0];
        const int64_t o = (b << lg_out) + out;
        if (a.split > 1) {
            reinterpret_cast<T*>(vw.P)[(int64_t)sp * (a.nbatch << lg_out) + o] = v;
            return;
        }
        if (sc.resid) {
            if constexpr (CPLX) {
                v.x = ldexpf(v.x, -sc.resid);
                v.y = ldexpf(v.y, -sc.resid);
            } else {
                v = ldexpf(v, -sc.resid);
            }
        }
        reinterpret_cast<T*>(vw.C)[o] = v;
        const float mx = absmax(v);
        if (mx > 0.f) atomicMax(vw.sc.max_c, __float_as_uint(mx));
        if (a.t_done) atomicMax(a.t_done, global_ns());
    }
}

// One launch for the small nodes of one or more consecutive tree levels.
// Each work item is a chunk of one node's outputs; descriptors live in
// device memory.  With fewer than 256 outputs in the chunk, g = 256/outputs
// threads share each output's K range and reduce it in a fixed order.
//
// Without dependencies (deps == nullptr) item i is CTA i.  With them, the
// launch covers several levels as one dataflow: persistent CTAs take items
// in order from a counter; before an item runs, the chunks of its children
// that belong to the same launch must have finished (per node and instance
// completion counters; a bounded wait that records TN_ETIMEOUT); after it,
// its own counter is raised.  Items only depend on earlier items, and every
// taken item belongs to a running CTA, so the waits always end.  Inputs that
// other CTAs of the launch produced are read through L2 (ld.global.cg).
// The persistent launch (every node of every slice of a call in one
// dataflow) adds tile items (o_count < 0): a 64 x 64 output tile of a large
// node computed by the tile kernel's body over all of K.
constexpr long long kFlowWaitCycles = 4000000000ll;  // ~2 s

// Completion counters: the producer's release add (after a CTA barrier, so
// it covers the whole CTA's writes) pairs with the consumer's acquire load.
__device__ __forceinline__ unsigned ld_acquire_gpu(const unsigned* p) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void red_release_gpu_add(unsigned* p, unsigned v) {
    asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

template <bool CPLX, bool TILES>
__global__ void __launch_bounds__(256)
    k_wave(const WaveItem* items, int n_items, const TileArgs* descs, const void* const* leaf_ptrs,
           const int4* deps, unsigned* done, unsigned* head, int G) {
    using T = typename VT<CPLX>::T;
    __shared__ TileArgs d;
    // K offsets: low 8 bits of the K index from kA / kB, the rest (at most
    // 6 more bits: wave nodes have nk <= 14) from kAh / kBh
    __shared__ int64_t kA[256], kB[256], kAh[64], kBh[64];
    // output offsets: low 8 bits of the output index, and the rest of each of
    // the item's rows of 256 outputs (at most 4): bit loops per output took
    // longer than its sum (32 copies of seven nodes 60 -> 51 us)
    __shared__ int64_t oA[256], oB[256], oAh[4], oBh[4];
    __shared__ T red[256];
    __shared__ int cur;
    __shared__ int loaded;  // node whose descriptor and K tables are in shared memory
    const int tid = threadIdx.x;
    if (tid == 0) loaded = -1;
    for (int pass = 0;; ++pass) {
        // ---- take an item
        if (deps == nullptr) {
            if (pass > 0) break;
            if (tid == 0) cur = blockIdx.x;
        } else if (tid == 0) {
            cur = (int)atomicAdd(head, 1u);
        }
        __syncthreads();
        const int idx = cur;
        if (idx >= n_items) break;
        const WaveItem it = items[idx];
        // ---- everything that does not depend on the children first: the
        // descriptor and the K offset tables (kept from the previous item
        // when it was of the same node), the instance view
        const bool fresh = it.node != loaded;
        if (fresh) {
            const int4* src = reinterpret_cast<const int4*>(descs + it.node);
            int4* dst = reinterpret_cast<int4*>(&d);
            for (int i = tid; i < (int)(sizeof(TileArgs) / 16); i += blockDim.x) dst[i] = src[i];
        }
        __syncthreads();
        if (tid == 0) loaded = it.node;  // every thread has read the old value
        const View vw = inst_view(d, it.pad, (int)sizeof(T));
        const int kt = d.nk < 8 ? (int)(1ll << d.nk) : 256;  // table covers k & 255
        const int kh = d.nk > 8 && d.nk <= 14 ? (int)(1ll << (d.nk - 8)) : 0;  // k >> 8
        auto o_scatter = [&](int64_t o, int64_t& offA, int64_t& offB) {
            const int64_t n = o & ((1ll << d.nn) - 1), m = (o >> d.nn) & ((1ll << d.nm) - 1), b = o >> (d.nn + d.nm);
            offA = scatter_bits(b, d.a_b, d.nb) + scatter_bits(m, d.a_m, d.nm);
            offB = scatter_bits(b, d.b_b, d.nb) + scatter_bits(n, d.b_n, d.nn);
        };
        // an item that is its CTA's only one, with one output per thread, enters
        // just its own outputs, high bits and all (one bit loop, not one after
        // the other: 2^14 outputs over K = 4 12.7 -> 11.3 us)
        const bool direct = deps == nullptr && it.o_count <= 256;
        if (fresh) {
            if (!direct && (!TILES || it.o_count >= 0)) o_scatter(tid, oA[tid], oB[tid]);
            for (int t = tid; t < kt; t += 256) {
                kA[t] = scatter_bits(t, d.a_k, d.nk);
                kB[t] = scatter_bits(t, d.b_k, d.nk);
            }
            for (int h = tid; h < kh; h += 256) {
                kAh[h] = scatter_bits((int64_t)h << 8, d.a_k, d.nk);
                kBh[h] = scatter_bits((int64_t)h << 8, d.b_k, d.nk);
            }
        }
        // operand bases need only the descriptor and the leaf table
        const int64_t isz = (int64_t)sizeof(T);
        const T* A = nullptr;
        const T* B = nullptr;
        int64_t sA = 0, sB = 0;
        if (vw.live) {
            A = reinterpret_cast<const T*>(
                d.a_leaf >= 0 ? (const char*)leaf_ptrs[d.a_leaf] + (int64_t)it.pad * d.in.a_is * isz : vw.A);
            B = reinterpret_cast<const T*>(
                d.b_leaf >= 0 ? (const char*)leaf_ptrs[d.b_leaf] + (int64_t)it.pad * d.in.b_is * isz : vw.B);
            sA = slice_off(d.sla, vw.slice);
            sB = slice_off(d.slb, vw.slice);
            if (direct) {
                const int g = 256 / (int)it.o_count;
                if (tid % g == 0 && tid / g < it.o_count) {
                    const int64_t o = it.o_begin + tid / g;
                    o_scatter(o, oA[o & 255], oB[o & 255]);
                }
                if (tid == 0) {
                    oAh[0] = sA;
                    oBh[0] = sB;
                }
            } else if (tid < 4 && tid * 256 < it.o_count) {
                int64_t hA, hB;
                o_scatter((it.o_begin + tid * 256) & ~255ll, hA, hB);
                oAh[tid] = sA + hA;
                oBh[tid] = sB + hB;
            }
        }
        // ---- then wait for children computed in this launch
        if (deps != nullptr && tid == 0) {
            const int4 dp = deps[it.node];
            const long long t0 = clock64();
            for (int side = 0; side < 2; ++side) {
                const int child = side ? dp.z : dp.x;
                const unsigned need = (unsigned)(side ? dp.w : dp.y);
                if (child < 0) continue;
                const unsigned* cnt = done + (int64_t)child * G + it.pad;
                while (ld_acquire_gpu(cnt) < need) {
                    if (clock64() - t0 > kFlowWaitCycles) {
                        atomicExch(const_cast<int32_t*>(&d.ctl->status), (int32_t)TN_ETIMEOUT);
                        break;
                    }
                    __nanosleep(32);
                }
            }
        }
        __syncthreads();
        if (TILES && vw.live && it.o_count < 0) {
            // a tile item of the persistent launch: 64 x 64 outputs of one
            // batch entry (o_begin = batch entry x tiles + tile), all of K
            const unsigned rma = vw.sc.max_a ? __ldcg(vw.sc.max_a) : 0u;
            const unsigned rmb = vw.sc.max_b ? __ldcg(vw.sc.max_b) : 0u;
            const int64_t rea = vw.sc.exp_a ? __ldcg(vw.sc.exp_a) : 0;
            const int64_t reb = vw.sc.exp_b ? __ldcg(vw.sc.exp_b) : 0;
            const Scales sc = scales_from(rma, rmb, rea, reb, it.o_begin == 0 && tid == 0 ? vw.sc.exp_c : nullptr);
            const int64_t tiles = ((1ll << d.nm) + 63) / 64 * (((1ll << d.nn) + 63) / 64);
            if constexpr (TILES)
                tile_body<CPLX, 64, 64, 16, 4, 4, true>(d, it.o_begin % tiles, 0, it.o_begin / tiles, vw, A, B, sc);
        } else if (vw.live) {
            const int64_t K = 1ll << d.nk;
            const int O = (int)it.o_count;
            const int g = O >= 256 ? 1 : 256 / O;
            auto k_off = [&](int64_t t, int64_t& ka, int64_t& kb2) {
                if (d.nk < 8) {
                    ka = kA[t];
                    kb2 = kB[t];
                } else if (kh > 0) {
                    ka = kA[t & 255] + kAh[t >> 8];
                    kb2 = kB[t & 255] + kBh[t >> 8];
                } else {
                    const int64_t hi = t & ~255ll;
                    ka = kA[t & 255] + (hi ? scatter_bits(hi, d.a_k, d.nk) : 0);
                    kb2 = kB[t & 255] + (hi ? scatter_bits(hi, d.b_k, d.nk) : 0);
                }
            };
            auto o_off = [&](int ol, int64_t& offA, int64_t& offB) {
                const int lo = ((int)it.o_begin + ol) & 255;
                offA = oA[lo] + oAh[ol >> 8];
                offB = oB[lo] + oBh[ol >> 8];
            };
            // the children's scale slots and this thread's first operand
            // pair are read together (one L2 round trip, not two)
            const unsigned rma = vw.sc.max_a ? __ldcg(vw.sc.max_a) : 0u;
            const unsigned rmb = vw.sc.max_b ? __ldcg(vw.sc.max_b) : 0u;
            const int64_t rea = vw.sc.exp_a ? __ldcg(vw.sc.exp_a) : 0;
            const int64_t reb = vw.sc.exp_b ? __ldcg(vw.sc.exp_b) : 0;
            bool first = tid / g < O && (int64_t)(tid % g) < K;
            T a0 = zero<T>(), b0 = zero<T>();
            if (first) {
                int64_t offA, offB, ka, kb2;
                o_off(tid / g, offA, offB);
                k_off(tid % g, ka, kb2);
                a0 = ld_cg<CPLX>(A + offA + ka);
                b0 = ld_cg<CPLX>(B + offB + kb2);
            }
            const Scales sc = scales_from(rma, rmb, rea, reb, it.o_begin == 0 && tid == 0 ? vw.sc.exp_c : nullptr);
            float lmax = 0.f;
            T* C = reinterpret_cast<T*>(vw.C);
            for (int ol = tid / g; ol < O; ol += 256 / g) {
                const int64_t o = it.o_begin + ol;
                int64_t offA, offB;
                o_off(ol, offA, offB);
                T acc = zero<T>();
#pragma unroll 4
                for (int64_t t = tid % g; t < K; t += g) {
                    T va, vb;
                    if (first) {
                        va = a0;
                        vb = b0;
                        first = false;
                    } else {
                        int64_t ka, kb2;
                        k_off(t, ka, kb2);
                        va = ld_cg<CPLX>(A + offA + ka);
                        vb = ld_cg<CPLX>(B + offB + kb2);
                    }
                    fma_acc(acc, cmul(va, sc.fa, d.conj_a), cmul(vb, sc.fb, d.conj_b));
                }
                if (g > 1) {
                    red[tid] = acc;
                    __syncthreads();
                    const int j = tid % g;
                    for (int s2 = g / 2; s2 > 0; s2 >>= 1) {
                        if (j < s2) red[tid] = add(red[tid], red[tid + s2]);
                        __syncthreads();
                    }
                    if (j != 0) continue;
                    acc = red[tid];
                }
                if (sc.resid) {
                    if constexpr (CPLX) {
                        acc.x = ldexpf(acc.x, -sc.resid);
                        acc.y = ldexpf(acc.y, -sc.resid);
                    } else {
                        acc = ldexpf(acc, -sc.resid);
                    }
                }
                lmax = fmaxf(lmax, absmax(acc));
                C[o] = acc;
            }
            block_max(lmax, vw.sc.max_c);
            if (d.t_done && tid == 0) atomicMax(d.t_done, global_ns());
        }
        // ---- publish: outputs, maximum and exponent before the counter
        __syncthreads();
        if (deps != nullptr && tid == 0) red_release_gpu_add(done + (int64_t)it.node * G + it.pad, 1u);
    }
}

// --------------------------------------------------------------------------
// launchers
// --------------------------------------------------------------------------

inline int64_t host_m(const TileArgs& a) { return int64_t(1) << a.nm; }
inline int64_t host_n(const TileArgs& a) { return int64_t(1) << a.nn; }
inline int64_t host_m(const GenericArgs& a) { return a.M; }
inline int64_t host_n(const GenericArgs& a) { return a.N; }
inline int64_t host_k(const TileArgs& a) { return int64_t(1) << a.nk; }
inline int64_t host_k(const GenericArgs& a) { return a.n_sum; }

template <class ARGS, bool CPLX, int TM, int TN, int TK, int RM, int RN, int MINB>
static cudaError_t launch_cfg(const ARGS& a, cudaStream_t s) {
    const int64_t M = host_m(a), N = host_n(a);
    const int64_t tiles = ((M + TM - 1) / TM) * ((N + TN - 1) / TN);
    const int ni = a.in.n_inst > 1 ? a.in.n_inst : 1;
    dim3 grid((unsigned)tiles, 1, (unsigned)(a.nbatch * a.split * ni));
    constexpr size_t smem = TileSmem<ARGS, CPLX, TM, TN, TK>::bytes;
    auto* kern = k_tile<ARGS, CPLX, TM, TN, TK, RM, RN, MINB>;
    static std::atomic<uint64_t> ready{0};
    const cudaError_t e = allow_shared(kern, smem, ready);
    if (e != cudaSuccess) return e;
    kern<<<grid, (TM / RM) * (TN / RN), smem, s>>>(a);
    return cudaGetLastError();
}

template <class ARGS, bool CPLX>
static cudaError_t launch_shape(const ARGS& a, cudaStream_t s) {
    switch (a.cfg) {
        case kTile64x64:
            // short sums are bound by loads and stores: twice the threads with
            // half the outputs (complex, 2^12 x 2^12 outputs: K = 16 123 us with
            // 8 x 4 outputs per thread, 109 with 4 x 4)
            if (host_k(a) <= 32) return launch_cfg<ARGS, CPLX, 64, 64, 8, 4, 4, 3>(a, s);
            return launch_cfg<ARGS, CPLX, 64, 64, 8, 8, 4, CPLX ? 3 : 4>(a, s);
        case kTile16x256: return launch_cfg<ARGS, CPLX, 16, 256, 8, 4, 4, 2>(a, s);
        case kTile4x1024: return launch_cfg<ARGS, CPLX, 4, 1024, 4, 4, 4, 2>(a, s);
        case kTile256x16: return launch_cfg<ARGS, CPLX, 256, 16, 8, 4, 4, 2>(a, s);
        case kTile128x64: return launch_cfg<ARGS, CPLX, 128, 64, 8, 8, CPLX ? 4 : 8, CPLX ? 2 : 3>(a, s);
        case kTile128x128:
            if constexpr (!CPLX) return launch_cfg<ARGS, CPLX, 128, 128, 8, 8, 8, 2>(a, s);
            else return cudaErrorInvalidValue;
        default: return cudaErrorInvalidValue;
    }
}

// The K parts' partials summed in a fixed order.
template <class ARGS, bool CPLX>
static cudaError_t launch_reduce(const ARGS& a, cudaStream_t s) {
    const int64_t n = a.nbatch * host_m(a) * host_n(a);
    const int ni = a.in.n_inst > 1 ? a.in.n_inst : 1;
    // threads per output: enough that outputs x G fill the GPU's threads;
    // chosen from one instance's outputs, so that every instance sums in the
    // same order however many run side by side (results independent of the
    // slice batch)
    int G = 1;
    while (G < 32 && G * 2 <= a.split && n * G < (int64_t)sm_count() * 256 * 4) G *= 2;
    int64_t blocks = (n + 256 / G - 1) / (256 / G);
    if (blocks > sm_count() * 8) blocks = sm_count() * 8;
    k_split_reduce<ARGS, CPLX><<<dim3((unsigned)blocks, (unsigned)ni), 256, 0, s>>>(a, G);
    return cudaGetLastError();
}

// Tile plan of an inner-product node.  Tile bits of K: those among the kDotLow
// lowest strides of either operand (its row bits, which are in every tile, take
// part in that), the operands in turn, then the lowest K positions.  Then each
// operand's order of its row and tile bits (ascending stride, absent bits last).
// (One output per CTA: no row bits, they are in the operand's base.)
static DotPlan make_dot_plan(const TileArgs& a) {
    DotPlan dp;
    memset(&dp, 0, sizeof(dp));
    const int nm = a.dot_each ? 0 : a.nm, nn = a.dot_each ? 0 : a.nn;
    const int nk = a.nk, t_max = dot_tile_bits(nm, nn, nk);
    // by stride: K position, or -2 - i for row bit i; -1: none
    int by[2][64];
    for (int q = 0; q < 64; ++q) by[0][q] = by[1][q] = -1;
    for (int p = 0; p < nk; ++p) {
        if (a.a_k[p] < 64) by[0][a.a_k[p]] = p;
        if (a.b_k[p] < 64) by[1][a.b_k[p]] = p;
    }
    for (int i = 0; i < nm; ++i) by[0][a.a_m[i]] = -2 - i;
    for (int i = 0; i < nn; ++i) by[1][a.b_n[i]] = -2 - i;
    bool in[kMaxBits] = {};
    int cnt = 0, q[2] = {0, 0}, low[2] = {0, 0};
    for (bool more = true; more && cnt < t_max;) {
        more = false;
        for (int side = 0; side < 2; ++side) {
            while (q[side] < 64 && by[side][q[side]] == -1) ++q[side];
            if (q[side] >= 64 || low[side] >= kDotLow || cnt >= t_max) continue;
            const int p = by[side][q[side]++];
            ++low[side];
            more = true;
            if (p >= 0 && !in[p]) {
                in[p] = true;
                ++cnt;
            }
        }
    }
    for (int p = 0; p < nk && cnt < t_max; ++p)
        if (!in[p]) {
            in[p] = true;
            ++cnt;
        }
    int tk[2 * kDotLow], pos[kMaxBits];
    int t = 0, u = 0;
    for (int p = 0; p < nk; ++p) {
        if (in[p]) {
            pos[p] = t;
            tk[t++] = p;
        } else {
            dp.rest_a[u] = a.a_k[p] != kNoBit ? int64_t(1) << a.a_k[p] : 0;
            dp.rest_b[u] = a.b_k[p] != kNoBit ? int64_t(1) << a.b_k[p] : 0;
            ++u;
        }
    }
    for (int side = 0; side < 2; ++side) {
        int64_t* add = side ? dp.b_add : dp.a_add;
        int32_t* cad = side ? dp.cb_add : dp.ca_add;
        int w = 0;
        for (int s = 0; s < 64; ++s) {
            const int p = by[side][s];
            if (p == -1 || (p >= 0 && !in[p])) continue;
            add[w] = int64_t(1) << s;
            cad[w++] = p >= 0 ? 1 << pos[p] : 1 << (16 - 2 - p);  // K position, or row << 16
        }
        for (int j = 0; j < t; ++j)  // tile bits the operand lacks repeat its entries
            if ((side ? a.b_k : a.a_k)[tk[j]] >= 64) {
                add[w] = 0;
                cad[w++] = 1 << j;
            }
    }
    dp.t = t;
    dp.u = u;
    return dp;
}

template <bool CPLX, int RM, int RN>
static cudaError_t launch_dot_rc(const TileArgs& a, const DotPlan& dp, cudaStream_t s) {
    using T = typename VT<CPLX>::T;
    const size_t smem = dot_smem_bytes(dp, (1 << a.nm) + (1 << a.nn), sizeof(T));
    static std::atomic<uint64_t> ready{0};
    const cudaError_t e = allow_shared(k_dot<CPLX, RM, RN>, kDotStages * (kDotEntries + kDotEntries / 16) * sizeof(T) +
                                                                kDotEntries * 6, ready);
    if (e != cudaSuccess) return e;
    const int ni = a.in.n_inst > 1 ? a.in.n_inst : 1;
    // parts of fewer than eight tiles: as many per CTA as make one round of
    // resident CTAs (longer ones balance better over many rounds)
    const int64_t slots = (int64_t)sm_count() * dot_resident(CPLX, RM * RN), total = (int64_t)a.split * a.nbatch * ni;
    int parts = 1;
    if (((int64_t(1) << dp.u) + a.split - 1) / a.split < 8)
        parts = (int)std::min<int64_t>((total + slots - 1) / slots, a.split);
    const unsigned blocks = (unsigned)((a.split + parts - 1) / parts);
    k_dot<CPLX, RM, RN><<<dim3((unsigned)a.nbatch, blocks, (unsigned)ni), 256, smem, s>>>(a, dp, parts);
    return cudaGetLastError();
}

template <bool CPLX, bool WIDE>
static cudaError_t launch_dot_one(const TileArgs& a, const DotPlan& dp, cudaStream_t s) {
    using T = typename VT<CPLX>::T;
    constexpr size_t smem = (size_t)kDotStages * 2 * (kDotTile + kDotTile / 32) * sizeof(T) + kDotTile * (WIDE ? 20 : 12);
    static std::atomic<uint64_t> ready{0};
    const cudaError_t e = allow_shared(k_dot_one<CPLX, WIDE>, smem, ready);
    if (e != cudaSuccess) return e;
    const int ni = a.in.n_inst > 1 ? a.in.n_inst : 1;
    const dim3 grid((unsigned)a.nbatch << (a.nm + a.nn), (unsigned)a.split, (unsigned)ni);
    k_dot_one<CPLX, WIDE><<<grid, 256, smem, s>>>(a, dp);
    return cudaGetLastError();
}

template <bool CPLX, int RM>
static cudaError_t launch_dot_r(const TileArgs& a, const DotPlan& dp, cudaStream_t s) {
    if (a.nn == 0) {
        if constexpr (RM > 1) return launch_dot_rc<CPLX, RM, 1>(a, dp, s);
        else return cudaErrorInvalidValue;  // one output: k_dot_one
    }
    if (a.nn == 1) return launch_dot_rc<CPLX, RM, 2>(a, dp, s);
    return launch_dot_rc<CPLX, RM, 4>(a, dp, s);
}

template <bool CPLX>
static cudaError_t launch_dot(const TileArgs& a, cudaStream_t s) {
    const DotPlan dp = make_dot_plan(a);
    if (a.wide) return launch_dot_one<CPLX, true>(a, dp, s);
    if (a.dot_each) return launch_dot_one<CPLX, false>(a, dp, s);
    if (a.nm == 0) return launch_dot_r<CPLX, 1>(a, dp, s);
    if (a.nm == 1) return launch_dot_r<CPLX, 2>(a, dp, s);
    return launch_dot_r<CPLX, 4>(a, dp, s);
}

template <bool CPLX, int TM, int TN, int TK>
static cudaError_t launch_wide_cfg(const TileArgs& a, cudaStream_t s) {
    const int64_t tiles = ((host_m(a) + TM - 1) / TM) * ((host_n(a) + TN - 1) / TN);
    const int ni = a.in.n_inst > 1 ? a.in.n_inst : 1;
    const dim3 grid((unsigned)tiles, 1, (unsigned)(a.nbatch * a.split * ni));
    k_tile_wide<CPLX, TM, TN, TK><<<grid, (TM / 4) * (TN / 4), 0, s>>>(a);
    return cudaGetLastError();
}

template <bool CPLX>
static cudaError_t launch_wide(const TileArgs& a, cudaStream_t s) {
    switch (a.cfg) {
        case kTile16x256: return launch_wide_cfg<CPLX, 16, 256, 16>(a, s);
        case kTile4x1024: return launch_wide_cfg<CPLX, 4, 1024, 4>(a, s);
        case kTile256x16: return launch_wide_cfg<CPLX, 256, 16, 16>(a, s);
        default: return launch_wide_cfg<CPLX, 64, 64, 16>(a, s);  // K parts do not depend on the tile
    }
}

template <bool CPLX>
static cudaError_t launch_tile_t(const TileArgs& a, cudaStream_t s) {
    const cudaError_t e = a.cfg == kTileDot ? launch_dot<CPLX>(a, s)
                          : a.wide          ? launch_wide<CPLX>(a, s)
                                            : launch_shape<TileArgs, CPLX>(a, s);
    if (e != cudaSuccess || a.split == 1) return e;
    return launch_reduce<TileArgs, CPLX>(a, s);
}

cudaError_t launch_tile(const TileArgs& a, bool is_c, cudaStream_t s) {
    return is_c ? launch_tile_t<true>(a, s) : launch_tile_t<false>(a, s);
}

cudaError_t launch_tile_any(const GenericArgs& a, bool is_c, cudaStream_t s) {
    const cudaError_t e = is_c ? launch_shape<GenericArgs, true>(a, s) : launch_shape<GenericArgs, false>(a, s);
    if (e != cudaSuccess || a.split == 1) return e;
    return is_c ? launch_reduce<GenericArgs, true>(a, s) : launch_reduce<GenericArgs, false>(a, s);
}

cudaError_t launch_wave(const WaveItem* items, int n_items, const TileArgs* descs,
                        const void* const* leaf_ptrs, bool is_c, cudaStream_t s, const int4* deps,
                        unsigned* done, unsigned* head, int G, bool tiles) {
    if (n_items <= 0) return cudaSuccess;
    // dataflow: persistent CTAs (8 per SM for the plain waves), else one per item
    const int grid = deps ? std::min(n_items, sm_count() * 8) : n_items;
    if (tiles) {
        if (is_c)
            k_wave<true, true><<<grid, 256, 0, s>>>(items, n_items, descs, leaf_ptrs, deps, done, head, G);
        else
            k_wave<false, true><<<grid, 256, 0, s>>>(items, n_items, descs, leaf_ptrs, deps, done, head, G);
    } else if (is_c) {
        k_wave<true, false><<<grid, 256, 0, s>>>(items, n_items, descs, leaf_ptrs, deps, done, head, G);
    } else {
        k_wave<false, false><<<grid, 256, 0, s>>>(items, n_items, descs, leaf_ptrs, deps, done, head, G);
    }
    return cudaGetLastError();
}

}  // namespace tn
