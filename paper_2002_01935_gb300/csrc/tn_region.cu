// tn_region.cu -- subtrees of small nodes computed in shared memory.
//
// Most nodes of a circuit or spin network contract a few entries (300 to 400
// of the 370 to 480 nodes of a 20- to 25-qubit circuit have at most 2^8
// multiply-adds): as work items of a dataflow wave each of them pays for an
// item, a descriptor, completion counters and scale slots read through L2,
// about 3 us per tree level.  Here one CTA takes a whole connected piece of
// the tree (a region: at most 2^16 multiply-adds): it loads the region's
// program -- every output's operand offsets and every node's K offsets, laid
// out once on the host -- and the operands from outside, and goes through the
// piece level by level with one barrier each, intermediates, maxima and
// exponents in shared memory; only the nodes read from outside are stored.
// Offsets come from tables, so label sizes of any kind are alike.  Bound by the
// chain of levels (about a microsecond each; a multiply-add costs some twenty
// instructions) after three dependent round trips for header, program and
// operands, which come by asynchronous copies.  The steps of a level (outputs
// of one shape of sum) are dealt to the block's warps, not run one after another.
//
// Every output is summed in the order of the wave kernel (partial sums of
// every g-th entry, then their tree), so the results are the same bits.
// Launch times (waves alone before): 16-qubit, 8-cycle amplitude 77 -> 54 us in
// three region launches, 32 copies of a 25-qubit one 221 -> 84, eight
// slices of a 25-qubit tree 139 -> 76 (20 of it the regions), 69 nodes of
// three-valued labels 10 instead of one launch each, forward and reverse sweep
// of a 20-qubit circuit in 64 copies 1022 -> 333 (104 the regions).
#include <cuda_runtime.h>
#include <atomic>
#include <stdint.h>

#include "tn_internal.h"

namespace tn {

namespace {


template <bool CPLX>
struct RT {
    using T = float2;
};
template <>
struct RT<false> {
    using T = float;
};

__device__ __forceinline__ float2 scaled(float2 x, float f, bool cj) {
    return make_float2(x.x * f, cj ? -x.y * f : x.y * f);
}
__device__ __forceinline__ float scaled(float x, float f, bool) { return x * f; }
__device__ __forceinline__ void mac(float2& c, float2 a, float2 b) {
    c.x = fmaf(a.x, b.x, c.x);
    c.x = fmaf(-a.y, b.y, c.x);
    c.y = fmaf(a.x, b.y, c.y);
    c.y = fmaf(a.y, b.x, c.y);
}
__device__ __forceinline__ void mac(float& c, float a, float b) { c = fmaf(a, b, c); }
__device__ __forceinline__ float2 plus(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float plus(float a, float b) { return a + b; }
__device__ __forceinline__ float2 down(float2 v, int o) {
    return make_float2(__shfl_down_sync(0xffffffffu, v.x, o), __shfl_down_sync(0xffffffffu, v.y, o));
}
__device__ __forceinline__ float down(float v, int o) { return __shfl_down_sync(0xffffffffu, v, o); }
__device__ __forceinline__ float largest(float2 v) { return fmaxf(fabsf(v.x), fabsf(v.y)); }
__device__ __forceinline__ float largest(float v) { return fabsf(v); }
__device__ __forceinline__ float2 shifted(float2 v, int e) { return make_float2(ldexpf(v.x, e), ldexpf(v.y, e)); }
__device__ __forceinline__ float shifted(float v, int e) { return ldexpf(v, e); }

// asynchronous global -> shared copies (all of a thread's are in flight at once)
template <int BYTES>
__device__ __forceinline__ void copy_async(void* dst, const void* src) {
    const uint32_t d = static_cast<uint32_t>(__cvta_generic_to_shared(dst));
    if constexpr (BYTES == 16)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src) : "memory");
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(d), "l"(src), "n"(BYTES) : "memory");
}
__device__ __forceinline__ void copies_done() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// frexpf's exponent of a maximum, 0 for 0 and NaN
__device__ __forceinline__ int exponent_of(unsigned bits) {
    const unsigned e = bits >> 23;  // (maxima have no sign)
    if (e - 1u < 254u) return (int)e - 126;
    const float m = __uint_as_float(bits);
    if (!(m > 0.f)) return 0;
    int x;
    frexpf(m, &x);
    return x;
}
__device__ __forceinline__ float power_of_two(int e) { return __uint_as_float((unsigned)(127 + e) << 23); }  // |e| <= 126

// Outputs [q0, q1) of a step: 2^lg threads and A partial sums per thread each.
// K index t belongs to partial sum t mod (A 2^lg); the sums are added as a
// tree over their index, highest bit first.  This warp's lanes are the step's
// threads i0 .. i0 + 31, i0 + THREADS ...
template <bool CPLX, int A, int THREADS>
__device__ __forceinline__ void region_step(const RegionStep& st, int lg, int i0, const uint2* outs, const int32_t* ktab,
                                            const RegionNode* nodes, typename RT<CPLX>::T* arena, int out0,
                                            unsigned* maxs, int64_t* exps, int n_ext) {
    using T = typename RT<CPLX>::T;
    const int lanes = 1 << lg, lane = threadIdx.x & (lanes - 1), n = (st.q1 - st.q0) << lg;
    for (; i0 < n; i0 += THREADS) {  // uniform over the warp: shuffles below
        const int i = i0 + (threadIdx.x & 31);
        const bool on = i < n;
        const int q = st.q0 + ((on ? i : 0) >> lg);
        const uint2 rec = outs[q];
        const RegionNode nd = nodes[rec.y];
        const int eA = exponent_of(maxs[nd.sa]), eB = exponent_of(maxs[nd.sb]);
        const int cA = max(-120, min(120, eA)), cB = max(-120, min(120, eB));
        const float fa = power_of_two(-cA), fb = power_of_two(-cB);
        const int resid = (eA - cA) + (eB - cB);
        const T* a = arena + nd.a + (rec.x & 0xffffu);
        const T* b = arena + nd.b + (rec.x >> 16);
        T acc[A];
#pragma unroll
        for (int j = 0; j < A; ++j) acc[j] = T{};
        if (on) {
            for (int t0 = lane; t0 < nd.k; t0 += A << lg)
#pragma unroll
                for (int j = 0; j < A; ++j) {
                    const int t = t0 + (j << lg);
                    if (t < nd.k) {
                        const unsigned ko = (unsigned)ktab[nd.kbase + t];
                        mac(acc[j], scaled(a[ko & 0xffffu], fa, nd.conj & 1), scaled(b[ko >> 16], fb, nd.conj & 2));
                    }
                }
        }
#pragma unroll
        for (int s = A / 2; s > 0; s >>= 1)
#pragma unroll
            for (int j = 0; j < s; ++j) acc[j] = plus(acc[j], acc[j + s]);
        T v = acc[0];
        for (int o = lanes >> 1; o > 0; o >>= 1) v = plus(v, down(v, o));
        if (on && lane == 0) {
            if (resid) v = shifted(v, -resid);
            arena[out0 + q] = v;
            if (q == nd.q0) exps[n_ext + rec.y] = exps[nd.sa] + exps[nd.sb] + eA + eB;
        }
        // the node's maximum: one shared atomic per warp where it holds one node.
        // fmaxf leaves NaN out, as the other kernels' maxima do (as bits it would
        // be above every number, and the fold take the node for a zero one).
        const unsigned m = on && lane == 0 ? __float_as_uint(fmaxf(largest(v), 0.f)) : 0u;
        if (__all_sync(0xffffffffu, rec.y == __shfl_sync(0xffffffffu, rec.y, 0))) {
            const unsigned w = __reduce_max_sync(0xffffffffu, m);
            if ((threadIdx.x & 31) == 0 && w) atomicMax(&maxs[n_ext + rec.y], w);
        } else if (m) {
            atomicMax(&maxs[n_ext + rec.y], m);
        }
    }
}

template <bool CPLX, int THREADS>
__global__ void __launch_bounds__(THREADS, THREADS > 256 ? 2 : 3) k_region(const __grid_constant__ RegionArgs a) {
    using T = typename RT<CPLX>::T;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ RegionHdr h;
    __shared__ const T* ext_ptr[kRegionExt];
    __shared__ int64_t exps[kRegionExt + kRegionNodes];
    __shared__ unsigned maxs[kRegionExt + kRegionNodes];
    int32_t* const blob = reinterpret_cast<int32_t*>(smem);
    T* const arena = reinterpret_cast<T*>(smem + sizeof(int32_t) * a.words);
    const int tid = threadIdx.x;
    const int region = blockIdx.x % a.n_regions, inst = blockIdx.x / a.n_regions;
    if (tid < (int)(sizeof(RegionHdr) / 4))
        reinterpret_cast<int32_t*>(&h)[tid] = reinterpret_cast<const int32_t*>(a.hdr + region)[tid];
    const int64_t slice = a.ctl->slice + (int64_t)inst * a.slice_step, slice_end = a.ctl->slice_end;
    __syncthreads();
    if (slice >= slice_end) return;
    {
        const int4* src = reinterpret_cast<const int4*>(a.prog + h.blob);
        for (int i = tid; i < h.words / 4; i += THREADS) copy_async<16>(reinterpret_cast<int4*>(blob) + i, src + i);
    }
    copies_done();
    __syncthreads();
    const uint2* outs = reinterpret_cast<const uint2*>(blob);
    const int32_t* ktab = blob + h.o_k;
    RegionNode* nodes = reinterpret_cast<RegionNode*>(blob + h.o_nodes);
    RegionExt* ext = reinterpret_cast<RegionExt*>(blob + h.o_ext);
    const uint16_t* elem = reinterpret_cast<const uint16_t*>(blob + h.o_elem);
    const RegionStep* steps = reinterpret_cast<const RegionStep*>(blob + h.o_steps);
    const RegionStore* stores = reinterpret_cast<const RegionStore*>(blob + h.o_store);
    // operands from outside: pointer, scale, and the slice offset of a leaf
    // (kept as its arena base for the nodes that read it)
    for (int e = tid; e < h.n_ext; e += THREADS) {
        const RegionExt x = ext[e];
        int base = x.first;
        if (x.leaf >= 0) {
            ext_ptr[e] = reinterpret_cast<const T*>(a.leaf_ptrs[x.leaf]) +
                         (a.leaf_is ? (int64_t)inst * a.leaf_is[x.leaf] : 0);
            maxs[e] = a.leafmax[x.leaf];
            exps[e] = 0;
            if (a.leaf_sl) {
                const SliceDigits& d = a.leaf_sl[x.leaf];
                for (int i = 0; i < d.n; ++i) base += (int)(((slice / d.div[i]) % d.dim[i]) * d.stride[i]);
            }
        } else {
            ext_ptr[e] = reinterpret_cast<const T*>(a.ws) + (int64_t)inst * a.ws_is + x.ws_off;
            maxs[e] = a.maxabs[(int64_t)inst * a.slot_is + x.node];
            exps[e] = a.exps[(int64_t)inst * a.slot_is + x.node];
        }
        ext[e].pad = base;
    }
    for (int k = tid; k < h.n_nodes; k += THREADS) maxs[h.n_ext + k] = 0u;
    __syncthreads();
    for (int i = tid; i < h.n_elem; i += THREADS) {
        const int e = elem[i];
        copy_async<sizeof(T)>(arena + i, ext_ptr[e] + (i - ext[e].first));
    }
    for (int k = tid; k < h.n_nodes; k += THREADS) {
        nodes[k].a = nodes[k].a >= 0 ? ext[nodes[k].a].pad : ~nodes[k].a;
        nodes[k].b = nodes[k].b >= 0 ? ext[nodes[k].b].pad : ~nodes[k].b;
    }
    copies_done();
    // the steps of a level are independent: their warps' shares are dealt round
    // robin over the block, so that a level takes as long as its longest step
    int dealt = 0;
    for (int s = 0; s < h.n_steps; ++s) {
        const RegionStep st = steps[s];
        if (st.accs < 0) {
            __syncthreads();
            dealt = 0;
        }
        const int A = st.accs < 0 ? -st.accs : st.accs, lg = st.lg_lanes;
        const int i0 = (((tid >> 5) - dealt) & (THREADS / 32 - 1)) * 32;
        dealt += (((st.q1 - st.q0) << lg) + 31) / 32;
        switch (A) {
            case 1: region_step<CPLX, 1, THREADS>(st, lg, i0, outs, ktab, nodes, arena, h.n_elem, maxs, exps, h.n_ext); break;
            case 2: region_step<CPLX, 2, THREADS>(st, lg, i0, outs, ktab, nodes, arena, h.n_elem, maxs, exps, h.n_ext); break;
            case 4: region_step<CPLX, 4, THREADS>(st, lg, i0, outs, ktab, nodes, arena, h.n_elem, maxs, exps, h.n_ext); break;
            default: region_step<CPLX, 8, THREADS>(st, lg, i0, outs, ktab, nodes, arena, h.n_elem, maxs, exps, h.n_ext); break;
        }
    }
    __syncthreads();
    // nodes that others read: one warp each
    for (int r = tid >> 5; r < h.n_store; r += THREADS / 32) {
        const RegionStore so = stores[r];
        const int q0 = nodes[so.node].q0, q1 = so.node + 1 < h.n_nodes ? nodes[so.node + 1].q0 : h.n_out;
        T* dst = reinterpret_cast<T*>(a.ws) + (int64_t)inst * a.ws_is + so.ws_off;
        for (int i = tid & 31; i < q1 - q0; i += 32) dst[i] = arena[h.n_elem + q0 + i];
        if ((tid & 31) == 0) {
            a.maxabs[(int64_t)inst * a.slot_is + so.slot] = maxs[h.n_ext + so.node];
            a.exps[(int64_t)inst * a.slot_is + so.slot] = exps[h.n_ext + so.node];
            if (so.done >= 0 && a.t_done) {
                unsigned long long now;
                asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(now));
                atomicMax(a.t_done + so.done, now);
            }
        }
    }
}

template <bool CPLX, int THREADS>
cudaError_t launch_t(const RegionArgs& a, unsigned blocks, cudaStream_t s) {
    constexpr size_t esz = sizeof(typename RT<CPLX>::T);
    static std::atomic<uint64_t> ready{0};
    const cudaError_t e =
        allow_shared(k_region<CPLX, THREADS>, sizeof(int32_t) * kRegionWords + kRegionArena * esz, ready);
    if (e != cudaSuccess) return e;
    k_region<CPLX, THREADS><<<blocks, THREADS, sizeof(int32_t) * a.words + a.entries * esz, s>>>(a);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_regions(const RegionArgs& a, bool is_c, cudaStream_t s) {
    if (a.n_regions <= 0) return cudaSuccess;
    const unsigned blocks = (unsigned)(a.n_regions * (a.n_inst > 1 ? a.n_inst : 1));
    // one block per SM or fewer: twice the threads for its levels (a 16-qubit
    // amplitude's three regions 60 -> 54 us); more: more blocks side by side
    // (both halves of a 64-copy sweep 104 us, 134 with 512 threads)
    if (blocks <= (unsigned)sm_count()) return is_c ? launch_t<true, 512>(a, blocks, s) : launch_t<false, 512>(a, blocks, s);
    return is_c ? launch_t<true, 256>(a, blocks, s) : launch_t<false, 256>(a, blocks, s);
}

}  // namespace tn
