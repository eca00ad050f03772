// CUDA kernels of the D3Q19 flux-boundary step (sm_103a).
//
//   k_step          one full time step for every pore node: pull streaming with
//                   halfway bounce-back (Eq. LBE), the Appendix B closures at the
//                   inlet/outlet planes with the inlet density of Eq. (potential),
//                   collision (Appendix A) and the store.  The same launch also
//                   forms the NEXT step's inlet density: every stored value that
//                   the next step pulls into an inlet node's known sum (Eq.
//                   inlet) is added by the node that produces it (FP32 values
//                   without error in FP32 words, FP64 values in FP64), and each
//                   warp or tile stores its FP64 part of the sum, which the next
//                   step adds in a fixed order.
//   k_step_pair     the same for the 16-bit formats, two nodes per thread.
//   k_inlet_reduce  the same density by a pull over the inlet plane, for states
//                   set from outside a step (creation, set_*, a new Q).
//   k_step_aa       the same step on ONE buffer (AA pattern), with the layout swaps
//                   k_aa_swap / k_aa_unstream around a call; k_aa_odd_pair and
//                   k_aa_even_pair for the 16-bit formats.
//   k_monitors      FP64 mass / flux / max|u| / NaN reductions of a state.
//   k_export, k_init_eq, k_encode, k_decode   field and state conversions.
#include <algorithm>
#include <cstdlib>
#include <utility>

#include "lbm_device.cuh"
#include "lbm_internal.h"
#include "lbm_pair.cuh"

namespace lbm {

namespace {

constexpr int kBlock = 256;
constexpr int kReduceBlock = 256;
// Resident 256-thread blocks per SM the step kernel is compiled for (caps its
// registers at 65536 / (256 * n)); FP64 arithmetic is left unconstrained.  On the row
// windows FP32 fits 48 registers without spills: 100 steps of a 100^3 pack 1142, 1101
// and 1101 us at 4, 5 and 6 blocks, of a 180x160x200 one 5817, 5595 and 5640.
#ifndef LBM_STEP_MIN_BLOCKS
#define LBM_STEP_MIN_BLOCKS 4
#endif
#ifndef LBM_STEP_WIN_BLOCKS
#define LBM_STEP_WIN_BLOCKS 5
#endif
template <class S, bool WIN>
constexpr int step_min_blocks() {
    return sizeof(typename S::M) == 8 ? 1 : WIN ? LBM_STEP_WIN_BLOCKS : LBM_STEP_MIN_BLOCKS;
}

template <int... Qs, class F>
__device__ __forceinline__ void for_q(std::integer_sequence<int, Qs...>, F&& f) {
    (f(std::integral_constant<int, Qs>{}), ...);
}
using AllQ = std::make_integer_sequence<int, 19>;
template <int Q>
using qc_t = std::integral_constant<int, Q>;

// Reference profile of the 16-bit formats at the plane of padded voxel p, and
// its slope (both 0 for the formats that store d directly).
template <class S>
__device__ __forceinline__ typename S::M own_ref(const BcState* bc, const DevLattice& L, int64_t p) {
    using M = typename S::M;
    if constexpr (S::kRef) return ref_at<M>(bc, plane_of((uint64_t)p, L.sz_magic));
    else return M(0);
}
template <class S>
__device__ __forceinline__ typename S::M own_ref_word(const BcState* bc, const DevLattice& L, uint32_t word) {
    using M = typename S::M;
    if constexpr (S::kRef) return ref_at<M>(bc, plane_of((uint64_t)(word >> 5), L.wz_magic));
    else return M(0);
}
template <class S>
__device__ __forceinline__ typename S::M own_slope(const BcState* bc) {
    using M = typename S::M;
    if constexpr (S::kRef) return ref_slope<M>(bc);
    else return M(0);
}

// ---------------------------------------------------- step-kernel access ---
// Per-direction row pointers of the two distribution buffers, passed as kernel
// parameters: every gather address is one multiply-add with a constant-bank
// operand, and no register is spent on 19 hoisted row bases.
template <class T>
struct StepPtrs {
    const T* in[19];
    T* out[19];
};

// The per-node kernel forms the next step's inlet contribution from the
// registers (FP32/FP64: measured faster) or by reloading the values it has just
// stored (16-bit formats, which it serves where there are no row windows: frees the
// decode state, measured faster).
// LBM_CONTRIB_RELOAD = 0 / 1 forces one way for every format.
template <class S>
__host__ __device__ constexpr bool contrib_reload() {
#ifdef LBM_CONTRIB_RELOAD
    return LBM_CONTRIB_RELOAD != 0;
#else
    return S::kRef;
#endif
}

// LBM_L2_HINTS: 0 = no hints; 1 = index structures evict-last; 2 = also the
// distribution streams evict-first.
#ifndef LBM_L2_HINTS
#define LBM_L2_HINTS 1
#endif

template <class T>
__device__ __forceinline__ T ld_index(const T* a, uint64_t pol) {
#if LBM_L2_HINTS >= 1
    return ld_hint(a, pol);
#else
    (void)pol;
    return __ldg(a);
#endif
}
template <class T>
__device__ __forceinline__ T ld_stream(const T* a, uint64_t pol) {
#if LBM_L2_HINTS >= 2
    return ld_hint(a, pol);
#else
    (void)pol;
    return __ldg(a);
#endif
}
template <class T>
__device__ __forceinline__ void st_stream(T* a, T v, uint64_t pol) {
#if LBM_L2_HINTS >= 2
    st_hint(a, v, pol);
#else
    (void)pol;
    *a = v;
#endif
}

// Pull all 19 values of node i (padded voxel p): a pore source gives its own
// value, a solid or outside source the node's opposite value (halfway
// bounce-back; the z-outside ones are replaced by the closure).
template <class S, bool OFF32>
__device__ __forceinline__ void pull_step(typename S::M* d, const StepPtrs<typename S::T>& P,
                                          const DevLattice& L, uint32_t p, int i, uint64_t pol_f,
                                          uint64_t pol_idx, typename S::M r_own, typename S::M g) {
    using M = typename S::M;
    for_q(AllQ{}, [&](auto qc) {
        constexpr int Q = decltype(qc)::value;
        if constexpr (Q == 0) {
            d[0] = S::template dec<0>(ld_stream(P.in[0] + i, pol_f), r_own);
        } else {
            // padded voxel indices fit in 32 bits (checked at creation)
            const int id = ld_index(L.grid + (uint32_t)(p + (uint32_t)L.goff[Q]), pol_idx);
            const typename S::T* a;
            if constexpr (OFF32)
                a = P.in[0] + (id >= 0 ? (uint32_t)Q * (uint32_t)L.ns + (uint32_t)id
                                       : (uint32_t)opp(Q) * (uint32_t)L.ns + (uint32_t)i);
            else
                a = id >= 0 ? P.in[Q] + id : P.in[opp(Q)] + i;
            // a pulled value was written on plane z - xi_z (reference r_own - g xi_z)
            const M r = (cz(Q) != 0 && id >= 0) ? r_own - M(cz(Q)) * g : r_own;
            d[Q] = S::template dec<Q>(ld_stream(a, pol_f), r);
        }
    });
}

// The same from the row windows: every source is row 0 plus one 32-bit element
// offset (rows are ns apart, buffers of fewer than 2^32 elements).  FP32 and FP64: the
// 16-bit formats take two nodes per thread there.
template <class S>
__device__ __forceinline__ void pull_step_win(typename S::M* d, const StepPtrs<typename S::T>& P, const DevLattice& L,
                                              uint32_t word, int i, uint64_t pol_f) {
    static_assert(!S::kRef, "k_step_pair");
    d[0] = ld_stream(P.in[0] + i, pol_f);
    for_links(L.win, word, L.wy, L.wz, (uint32_t)i, [&](auto qc, bool pore, uint32_t id) {
        constexpr int Q = decltype(qc)::value;
        const uint32_t off = pore ? (uint32_t)Q * (uint32_t)L.ns + id : (uint32_t)opp(Q) * (uint32_t)L.ns + (uint32_t)i;
        d[Q] = ld_stream(P.in[0] + off, pol_f);
    });
}

template <class S>
__device__ __forceinline__ void store_step(const typename S::M* d, const StepPtrs<typename S::T>& P,
                                           int i, uint64_t pol_f, typename S::M r_own, uint32_t seed) {
    encode_node<S>(d, seed, i, [&](auto) { return r_own; }, [&](auto qc, typename S::T v) {
        constexpr int Q = decltype(qc)::value;
        st_stream(P.out[Q] + i, v, pol_f);
    });
}

// Stochastic-rounding seed of this step (16-bit formats), and the next one.
template <class S>
__device__ __forceinline__ uint32_t step_seed(const BcState* bc, int slot) {
    if constexpr (S::kRef) return bc->sr_seed[slot];
    else return 0u;
}

// ------------------------------------------------------------ reductions ---
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
}
__device__ __forceinline__ double warp_max(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_down_sync(0xffffffffu, v, o));
    return v;
}
// Warp sums in the storage's arithmetic type (FP32 for the FP32/16-bit
// formats): FP64 arithmetic is scarce on GB300, so per-node values and the
// first 32-way level stay in M and only the block level runs in FP64.
template <class M>
__device__ __forceinline__ M warp_sum_m(M v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
}
template <class M>
__device__ __forceinline__ M warp_max_m(M v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const M w = __shfl_down_sync(0xffffffffu, v, o);  // every lane shuffles, then compares
        v = v > w ? v : w;
    }
    return v;
}
template <int NT, class M>
__device__ __forceinline__ double block_sum_m(M v, double* sh) {
    v = warp_sum_m(v);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (lane == 0) sh[wid] = (double)v;
    __syncthreads();
    double r = 0.0;
    if (wid == 0) {
        r = lane < NT / 32 ? sh[lane] : 0.0;
        r = warp_sum(r);
    }
    __syncthreads();
    return r;  // valid in thread 0
}
template <int NT, class M>
__device__ __forceinline__ double block_max_m(M v, double* sh) {
    v = warp_max_m(v);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (lane == 0) sh[wid] = (double)v;
    __syncthreads();
    double r = 0.0;
    if (wid == 0) {
        r = lane < NT / 32 ? sh[lane] : 0.0;
        r = warp_max(r);
    }
    __syncthreads();
    return r;
}

// Fixed-shape block sum: the result depends only on the inputs, not on timing.
template <int NT>
__device__ __forceinline__ double block_sum(double v, double* sh) {
    v = warp_sum(v);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (lane == 0) sh[wid] = v;
    __syncthreads();
    double r = 0.0;
    if (wid == 0) {
        r = lane < NT / 32 ? sh[lane] : 0.0;
        r = warp_sum(r);
    }
    __syncthreads();
    return r;  // valid in thread 0
}
template <int NT>
__device__ __forceinline__ double block_max(double v, double* sh) {
    v = warp_max(v);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (lane == 0) sh[wid] = v;
    __syncthreads();
    double r = 0.0;
    if (wid == 0) {
        r = lane < NT / 32 ? sh[lane] : 0.0;
        r = warp_max(r);
    }
    __syncthreads();
    return r;
}

// ------------------------------------------------------- inlet reduction ---
// One thread per inlet pore node (pore indices [0, A)).  K'_i is the known sum
// of Eq. (inlet) on shifted values, formed in FP64; S' = sum_i K'_i; then
// rho_in - 1 = (Q + S') / A  (Eq. potential with rho0 = 1, since K = 1 + K').
template <class S>
__global__ void __launch_bounds__(kReduceBlock)
k_inlet_reduce(const typename S::T* __restrict__ fin, int slot, DevLattice L, BcState* bc,
               double* __restrict__ partials, unsigned* __restrict__ counter) {
    __shared__ double sh[32];
    __shared__ bool last;
    const int64_t i64 = (int64_t)blockIdx.x * kReduceBlock + threadIdx.x;
    double k = 0.0;
    if (i64 < L.a_in) {
        const int i = (int)i64;
        const int64_t p = L.vox[i];
        using M = typename S::M;
        const M r_own = own_ref<S>(bc, L, p), g = own_slope<S>(bc);
        M d[19];
        for_q(std::integer_sequence<int, 0, 1, 2, 3, 4, 6, 7, 8, 9, 10, 12, 13, 16, 17>{},
              [&](auto qc) {
                  constexpr int Q = decltype(qc)::value;
                  d[Q] = pull<S, Q>(fin, L.ns, L.grid, p, i, L.sy, L.sz, r_own, g);
              });
        k = (double)d[0] + (double)d[1] + (double)d[2] + (double)d[3] + (double)d[4] +
            (double)d[7] + (double)d[8] + (double)d[9] + (double)d[10] +
            2.0 * ((double)d[6] + (double)d[12] + (double)d[13] + (double)d[16] + (double)d[17]);
    }
    const double b = block_sum<kReduceBlock>(k, sh);
    if (threadIdx.x == 0) {
        partials[blockIdx.x] = b;
        __threadfence();
        last = atomicAdd(counter, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    double s = 0.0;
    for (int j = threadIdx.x; j < (int)gridDim.x; j += kReduceBlock) s += __ldcg(partials + j);
    s = block_sum<kReduceBlock>(s, sh);
    if (threadIdx.x == 0) {
        bc->drho_in[slot] = (bc->Q + s) / (double)L.a_in;
        bc->parts[slot] = 0;
        *counter = 0u;
    }
}

// ---------------------------------------------------------- the step ---
// Contribution of pore node i (on plane z = 0 or z = 1) to the next step's
// inlet known sum S' = sum over inlet nodes of K'.  A value stored in direction
// p lands, at the next pull, on node i + xi_p (if that is a pore) or bounces
// back to i as direction opp(p).  It enters S' when it lands on the plane z = 0
// in a direction with xi_z = 0 (weight 1) or xi_z = -1 (weight 2):
//   z = 0:  all xi_z = 0 values (they stay on the plane either way), plus twice
//           each xi_z = +1 value whose destination on z = 1 is solid;
//   z = 1:  twice each xi_z = -1 value whose destination on z = 0 is a pore.
// `val(Q)` returns the stored value of direction Q exactly as the next step
// will decode it.
template <class S, class V>
__device__ __forceinline__ double inlet_contribution(const DevLattice& L, uint32_t p, int i, V&& val) {
    using M = typename S::M;
    InletSum<M> s;
    auto dest_is_pore = [&](auto qc) -> bool {
        constexpr int Q = decltype(qc)::value;  // destination i + xi_Q = pull source of opp(Q)
        return __ldg(L.grid + (uint32_t)(p + (uint32_t)L.goff[opp(Q)])) >= 0;
    };
    if (i < L.a_in) {
        for_q(std::integer_sequence<int, 0, 1, 2, 3, 4, 7, 8, 9, 10>{},
              [&](auto qc) { s.add(val(qc)); });
        for_q(std::integer_sequence<int, 5, 11, 14, 15, 18>{},
              [&](auto qc) { if (!dest_is_pore(qc)) s.add(M(2) * val(qc)); });
    } else {
        for_q(std::integer_sequence<int, 6, 12, 13, 16, 17>{},
              [&](auto qc) { if (dest_is_pore(qc)) s.add(M(2) * val(qc)); });
    }
    return s.value();
}

// From values still in registers (the pipelined kernel).
template <class S>
__device__ __forceinline__ double next_inlet_part(const typename S::M* d, const DevLattice& L,
                                                  int64_t p, int i, typename S::M r_own, uint32_t seed) {
    return inlet_contribution<S>(L, (uint32_t)p, i, [&](auto qc) {
        constexpr int Q = decltype(qc)::value;
        return S::template dec<Q>(S::template enc_sr<Q>(d[Q], r_own, sr_key<S>(seed, i)), r_own);
    });
}

// From the values this thread has just stored (the per-node kernel): the
// registers of the collision are free again, and only the ~2 % of nodes on the
// planes next to the inlet pay the reload.
template <class S>
__device__ __forceinline__ double next_inlet_part_stored(const StepPtrs<typename S::T>& P, const DevLattice& L,
                                                         uint32_t p, int i, typename S::M r_own) {
    return inlet_contribution<S>(L, (uint32_t)p, i, [&](auto qc) {
        constexpr int Q = decltype(qc)::value;
        const typename S::T v = *(volatile const typename S::T*)(P.out[Q] + i);
        return S::template dec<Q>(v, r_own);
    });
}

// LBM_STEP_PREFETCH: each block asks L2 (a bulk prefetch, nothing waited for)
// for the 19 input rows and the voxel list of the block that many blocks ahead,
// as the gather-scatter AA step does; 0 = off.  Measured on the 256^3 pack
// (same-call A/B, bitwise equal states): FP32 step 0.1953 ms without, 0.1764,
// 0.1745 and 0.1773 ms at 128, 224 and 320 blocks ahead; FP16-dev 0.1730,
// 0.1640, 0.1620 and 0.1614 ms.
#ifndef LBM_STEP_PREFETCH
#define LBM_STEP_PREFETCH 224
#endif

// The inlet sum of the next step leaves a step as parts, one per warp of the tiles
// that hold plane z = 0 or z = 1 nodes (tile number `tile`, of NT / 32 warps), and
// the blocks of the next step that hold inlet nodes add them while their gathers
// are on the way.  (Adding them here, in the tile that finishes last, put a memory
// fence, a ticket and a second round of loads at the end of every step: 8.5 us per
// step of a 10k-node FP32 lattice against 6.7, 8.8 against 7.5 at 173k nodes, 11.0
// against 9.1 at 365k.)
//   Every block with inlet nodes adds all parts, which costs the square of the inlet
// area: with one part per warp throughout, an open FP32 lattice of 1024x1024x3 took
// 602 us per step, of 512x512x16 139.  Above LBM_WARP_PARTS warps of nodes on the planes
// (FP64: twice as many, its steps being longer) a tile therefore leaves one part for
// all its warps (FP32 packs, AA pattern: 140x160x100, 1,400 warps 21.4 us per step with
// a part per warp and 21.7 with one per tile, 250x250x24, 3,906 warps 24.7 and 24.2;
// FP64 241.8 and 243.7 there), and above LBM_PARTS_DIRECT of those a kernel behind the
// step adds them to kFolded ones first (512x512x16, 2,048 parts: 117.4 us without that
// kernel and 118.7 with it, 600x600x16, 2,813 parts: 167.5 and 165.2; 1024x1024x3 125,
// 2047x2047x4 8,590 -> 613).
#ifndef LBM_WARP_PARTS
#define LBM_WARP_PARTS 2048
#endif
#ifndef LBM_PARTS_DIRECT
#define LBM_PARTS_DIRECT 2048
#endif
constexpr int kPartsDirect = LBM_PARTS_DIRECT;
constexpr int kFolded = 128;
// TILES: one part per tile.  Both forms are compiled: as a branch of one kernel it cost
// the steps of small lattices up to 2 % (61x67x72 FP32 7.05 -> 7.15 us).  f(TILES).
template <class M, class F>
cudaError_t with_parts(const DevLattice& L, F&& f) {
    constexpr int64_t kNodes = 32 * LBM_WARP_PARTS * (sizeof(M) == 8 ? 2 : 1);
    return L.a_01 > kNodes ? f(std::true_type{}) : f(std::false_type{});
}
// Parts that a step in blocks of NT threads and `nodes` nodes leaves.
template <int NT, bool TILES>
__host__ __device__ __forceinline__ int step_parts(const DevLattice& L, int nodes) {
    return (int)((L.a_01 + nodes - 1) / nodes) * (TILES ? 1 : NT / 32);
}
// The parts of a step that folds them lie behind the two parities.
__global__ void __launch_bounds__(kReduceBlock)
k_inlet_fold(DevLattice L, int n, int slot, double* __restrict__ partials) {
    __shared__ double sh[32];
    const double* p = partials + 2 * L.part_stride;
    double s = 0.0;
    for (int j = blockIdx.x * kReduceBlock + threadIdx.x; j < n; j += kFolded * kReduceBlock) s += p[j];
    s = block_sum<kReduceBlock>(s, sh);
    if (threadIdx.x == 0) partials[slot * L.part_stride + blockIdx.x] = s;
}
// Behind a step that reads buffer `slot`, in blocks of NT threads and `nodes` nodes.
template <int NT, bool TILES>
inline cudaError_t fold_parts(const DevLattice& L, int slot, double* partials, int nodes, cudaStream_t st) {
    const int n = step_parts<NT, TILES>(L, nodes);
    if (TILES && n > kPartsDirect) k_inlet_fold<<<kFolded, kReduceBlock, 0, st>>>(L, n, slot ^ 1, partials);
    return cudaGetLastError();
}
template <class S, int NT, int NODES, bool TILES>
__device__ __forceinline__ void store_inlet_part(double part, int64_t tile, const DevLattice& L, BcState* bc, int slot,
                                                 double* __restrict__ partials, double* sh) {
    constexpr int W = TILES ? 1 : NT / 32;
    double v;
    if constexpr (TILES) v = block_sum<NT>(part, sh);
    else v = warp_sum(part);
    const int n = step_parts<NT, TILES>(L, NODES);
    const bool fold = TILES && n > kPartsDirect;
    if ((threadIdx.x & 31) == 0 && (!TILES || threadIdx.x == 0))
        partials[(fold ? 2 : slot ^ 1) * L.part_stride + tile * W + (threadIdx.x >> 5)] = v;
    if (tile == 0 && threadIdx.x == 0) {
        bc->parts[slot ^ 1] = fold ? kFolded : n;
        if constexpr (S::kRef) bc->sr_seed[slot ^ 1] = sr_next(bc->sr_seed[slot]);
    }
}

// Inlet density - 1 of this step, for every thread of a block that holds inlet
// nodes; the block `first` records it.  The parts are added in an order that does
// not depend on NT -- part j on virtual lane j mod 256, then the trees of 8 virtual
// warps, then one of the 8 sums.
template <class M, int NT>
__device__ __forceinline__ M density_of_parts(const DevLattice& L, BcState* bc, int slot,
                                              const double* __restrict__ partials, double* sh, bool first) {
    constexpr int W = NT / 32;
    const int n = bc->parts[slot];
    if (n == 0) return M(bc->drho_in[slot]);
    // a 32-bit offset in the two-node kernels (NT = 128): with a pointer k_aa_even_pair
    // spilled 40 bytes (2 % of a 45x50x60 pack's step); with an offset the FP32
    // gather-scatter kernel spilled 8
    using Row = std::conditional_t<NT == kBlock / 2, int, const double*>;
    Row row;
    if constexpr (std::is_same<Row, int>::value) row = slot * (int)L.part_stride;
    else row = partials + slot * L.part_stride;
    const auto part = [&](int j) {
        if constexpr (std::is_same<Row, int>::value) return partials[row + j];
        else return row[j];
    };
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    for (int vw = wid; vw < 8; vw += W) {
        double s = 0.0;
        for (int j = vw * 32 + lane; j < n; j += 256) s += part(j);
        s = warp_sum(s);
        if (lane == 0) sh[vw] = s;
    }
    __syncthreads();
    if (wid == 0) {
        const double s = warp_sum(lane < 8 ? sh[lane] : 0.0);
        if (lane == 0) {
            const double drho = (bc->Q + s) / (double)L.a_in;
            sh[8] = drho;
            if (first) bc->drho_in[slot] = drho;
        }
    }
    __syncthreads();
    return M(sh[8]);
}

template <class M, int NT>
__device__ __forceinline__ M inlet_density(const DevLattice& L, BcState* bc, int slot, const double* __restrict__ partials,
                                           double* sh, bool first) {
    // in pressure mode the first block still records the density that the flux would need
    const int fixed = bc->inlet_mode;
    if (fixed && !first) return M(bc->drho_in_fixed);
    const M drho = density_of_parts<M, NT>(L, bc, slot, partials, sh, first);
    return fixed ? M(bc->drho_in_fixed) : drho;
}

// drho_in[slot] from its parts, for readers between steps (the 16-bit reference,
// which takes it in pressure mode too).
__global__ void __launch_bounds__(kReduceBlock)
k_inlet_finish(DevLattice L, BcState* bc, int slot, const double* __restrict__ partials) {
    __shared__ double sh[32];
    density_of_parts<double, kReduceBlock>(L, bc, slot, partials, sh, true);
}

// FORM: see Form in lbm_device.cuh.  NT nodes per block.
template <class S, int FORM, int NT, bool TILES>
__global__ void __launch_bounds__(NT, step_min_blocks<S, FORM == kWindows>())
k_step(const StepPtrs<typename S::T> P, int slot, DevLattice L, Rates<typename S::M> rates,
       BcState* bc, double* __restrict__ partials) {
    using M = typename S::M;
    constexpr bool WIN = FORM == kWindows;
    __shared__ double sh[32];
    const int64_t i64 = (int64_t)blockIdx.x * NT + threadIdx.x;
    const int i = (int)i64;
    double part = 0.0;
    if constexpr (LBM_STEP_PREFETCH > 0 && NT == kBlock) {
        // threads 0..18: input row q (rows are P.in[0] + q ns; the 128-element
        // padding keeps every range 16-byte aligned); thread 19: the voxel list,
        // cut to a multiple of 4 entries
        const int64_t s = ((int64_t)blockIdx.x + LBM_STEP_PREFETCH) * kBlock;
        const int t = (int)threadIdx.x;
        if (t < 19) l2_prefetch_range(P.in[0] + (int64_t)t * L.ns, s, kBlock, L.ns);
        else if (t == 19) l2_prefetch_range(WIN ? L.nodew : L.vox, s, kBlock, L.n & ~(int64_t)3);
    }
#if LBM_L2_HINTS >= 2
    const uint64_t pol_f = l2_policy_evict_first();
#else
    const uint64_t pol_f = 0;
#endif
#if LBM_L2_HINTS >= 1
    const uint64_t pol_idx = l2_policy_evict_last();
#else
    const uint64_t pol_idx = 0;
#endif
    uint32_t p = 0;  // node word or padded voxel
    M r_own = M(0), drin = M(0);
    uint32_t seed = 0;
    M d[19];
    if (i64 < L.n) {
        p = ld_index((WIN ? L.nodew : L.vox) + i, pol_idx);  // node word or padded voxel
        const M g = own_slope<S>(bc);
        if constexpr (!WIN) r_own = own_ref<S>(bc, L, p);
        seed = step_seed<S>(bc, slot);
        if constexpr (WIN) pull_step_win<S>(d, P, L, p, i, pol_f);
        else pull_step<S, FORM == kGrid32>(d, P, L, p, i, pol_f, pol_idx, r_own, g);
    }
    if ((int64_t)blockIdx.x * NT < L.a_in) drin = inlet_density<M, NT>(L, bc, slot, partials, sh, blockIdx.x == 0);
    if (i64 < L.n) {
        if (i < L.a_in) {
            // Section 2: after streaming, before collision.  u_z from Eq. (inlet)
            // with the density of Eq. (potential); then the Appendix B closure.
            close_inlet(d, drin - inlet_known(d));
        } else if (i64 >= L.n - L.a_out) {
            const M uz = outlet_known(d) - M(bc->drho_out);
            close_outlet(d, uz);
        }
        collide(d, rates);
        store_step<S>(d, P, i, pol_f, r_own, seed);
        if (i64 < L.a_01) {
            const uint32_t pv = WIN ? __ldg(L.vox + i) : p;
            if constexpr (contrib_reload<S>()) part = next_inlet_part_stored<S>(P, L, pv, i, r_own);
            else part = next_inlet_part<S>(d, L, pv, i, r_own, seed);
        }
    }
    if ((int64_t)blockIdx.x * NT < L.a_01)
        store_inlet_part<S, NT, NT, TILES>(part, blockIdx.x, L, bc, slot, partials, sh);
}

// ------------------------------------------------------ AA-pattern step ---
// Single-buffer variant (every storage format).  At rest the state has the pull
// layout of k_step, F[q][x] = f*_q(x) (post-collision values at their own node).
// The library first swaps every node's opposite pairs (layout S:
// F[opp q][x] = f*_q(x)), then alternates
//   odd step:  in_q(x) = F[opp q][x - xi_q] for a pore source, else F[q][x]
//              (halfway bounce-back); closures, collision; f*_q(x) goes to
//              F[q][x + xi_q] for a pore destination, else to F[opp q][x]
//              (layout S -> I, I[q][x] = the value arriving at x in direction q);
//   even step: in_q(x) = F[q][x]; closures, collision; f*_q(x) -> F[opp q][x]
//              (layout I -> S);
// and swaps the pairs back before anything else reads the state (after an odd
// count, k_aa_unstream first turns layout I into S); consecutive step calls stay
// in the in-place layouts.  Within a step every slot is read and then written by
// one node only, so the update runs in place.  Values leaving through the z
// faces are kept like bounced ones; the closures overwrite them.  The next
// step's inlet density is formed exactly as in k_step: the landing rule of a
// post-collision value does not depend on where it is stored.
// Row pointers of the single buffer as kernel parameters (constant bank), as
// for k_step: no registers spent on 19 row addresses.
template <class T>
struct AAPtrs {
    T* row[19];
};

// Resident blocks per SM the two AA kernels are compiled for (register caps).
// On the 256^3 pack the FP32 gather-scatter step measured best at 5 (48 registers):
// 171 us against 180 at 4 and 186 at 6; the node-local one at 5: 143.8 us against
// 145.2 at 6 and 160.6 at 7.
#ifndef LBM_AA_MIN_BLOCKS
#define LBM_AA_MIN_BLOCKS 5
#endif
#ifndef LBM_AA_EVEN_MIN_BLOCKS
#define LBM_AA_EVEN_MIN_BLOCKS 5
#endif
// LBM_AA_ID_HINT: 1 = the id grid is read with the L2 evict-last policy, 0 = plain.
#ifndef LBM_AA_ID_HINT
#define LBM_AA_ID_HINT 1
#endif
// The 16-bit formats carry the reference profile and the rounding seed too.
#ifndef LBM_AA16_MIN_BLOCKS
#define LBM_AA16_MIN_BLOCKS 5
#endif
#ifndef LBM_AA16_EVEN_MIN_BLOCKS
#define LBM_AA16_EVEN_MIN_BLOCKS 5
#endif
// LBM_AA_PREFETCH: the FP32/FP64 gather-scatter step asks L2 for the rows of the
// block that many blocks ahead (a bulk prefetch, nothing waited for), so that
// the DRAM requests in flight no longer depend on how many warps are waiting on
// their own gathers; 0 = off.  Measured on the 256^3 pack: the gain is flat from
// about 160 to 288 blocks ahead and falls off outside; at 224 the AA step pair is
// 4.7 % shorter than without (with the cap of 4 blocks).
#ifndef LBM_AA_PREFETCH
#define LBM_AA_PREFETCH 224
#endif
// LBM_AA16_PREFETCH: the same bulk L2 prefetch for the 16-bit gather-scatter
// step, that many blocks ahead; 0 = off.  Measured on the 256^3 pack: FP16-dev
// step 0.1735 against 0.1763 ms without, BF16-dev 0.1742 against 0.1826 ms (a
// 4-block register cap or reloaded ids with it were 10-14 % slower).
#ifndef LBM_AA16_PREFETCH
#define LBM_AA16_PREFETCH 224
#endif
template <class S, bool ODD>
constexpr int aa_min_blocks() {
    if constexpr (sizeof(typename S::M) == 8) return 1;
    else if constexpr (S::kRef) return ODD ? LBM_AA16_MIN_BLOCKS : LBM_AA16_EVEN_MIN_BLOCKS;
    else return ODD ? LBM_AA_MIN_BLOCKS : LBM_AA_EVEN_MIN_BLOCKS;
}
template <class T>
__device__ __forceinline__ T ld_aa_index(const T* a, uint64_t pol) {
#if LBM_AA_ID_HINT
    return ld_index(a, pol);
#else
    (void)pol;
    return __ldg(a);
#endif
}
__device__ __forceinline__ uint64_t aa_index_policy() {
#if LBM_AA_ID_HINT
    return l2_policy_evict_last();
#else
    return 0;
#endif
}

// FORM (of the gather-scatter launch; see lbm_device.cuh): with 32-bit offsets, each
// direction's gather offset is staged in shared memory.  The scatter
// destination of q is the gather source of opp(q) -- F[q][x + xi_q] for a pore
// there, else the bounce-back slot F[opp q][x], both read by the gather of
// opp(q) -- so the scatter reads its offset as it is and needs no id test or
// offset arithmetic (the launch on the 256^3 pack, ids staged -> offsets staged:
// 0.2006 -> 0.1825 ms FP16-dev, 0.2013 -> 0.1972 ms FP32).  Otherwise the ids of
// the id grid are staged and the rows addressed by 64-bit pointers.
template <class S, bool ODD, int FORM, int NT, bool TILES>
__global__ void __launch_bounds__(NT, aa_min_blocks<S, ODD>())
k_step_aa(const AAPtrs<typename S::T> F, int slot, DevLattice L, Rates<typename S::M> rates,
          BcState* bc, double* __restrict__ partials) {
    using M = typename S::M;
    __shared__ double sh[32];
    constexpr bool WIN = FORM == kWindows, OFF32 = FORM != kGrid64;
    __shared__ int sid[ODD ? 18 : 1][NT];  // gather offset (OFF32) or pore id per direction
    const int64_t i64 = (int64_t)blockIdx.x * NT + threadIdx.x;
    // threads past the last node of a gather-scatter launch load its values and write
    // nothing: straight-line loads up to the barrier of inlet_density (0.9 us of 171)
    const int i = ODD ? (int)min(i64, L.n - 1) : (int)i64;
    double part = 0.0;
    constexpr int kAhead = S::kRef ? LBM_AA16_PREFETCH : LBM_AA_PREFETCH;
    if constexpr (ODD && kAhead > 0 && NT == kBlock) {
        // threads 0..18: row q of the buffer (rows are F.row[0] + q ns, as
        // launched; 128-element padding keeps every range 16-byte aligned for
        // 2-byte values too); thread 19: the node list, cut to a multiple of 4 entries
        const int64_t s = ((int64_t)blockIdx.x + kAhead) * kBlock;
        const int t = (int)threadIdx.x;
        if (t < 19) l2_prefetch_range(F.row[0] + (int64_t)t * L.ns, s, kBlock, L.ns);
        else if (t == 19) l2_prefetch_range(WIN ? L.nodew : L.vox, s, kBlock, L.n & ~(int64_t)3);
    }
    M d[19];
    M r_own = M(0), g = M(0), drin = M(0);
    uint32_t seed = 0;
    if (ODD || i64 < L.n) {
        // 16-bit formats: every stored value is encoded with the reference of the
        // plane of the node that holds it (the even step writes its own slots; the
        // odd step encodes a scattered value with its destination's plane), so a
        // value read from the neighbour x - xi_q decodes with r(z - xi_z).
        seed = step_seed<S>(bc, slot);
        if constexpr (ODD && WIN) {
            static_assert(!S::kRef, "k_aa_odd_pair");
            const uint32_t word = ld_aa_index(L.nodew + i, aa_index_policy());
            d[0] = F.row[0][i];
            for_links(L.win, word, L.wy, L.wz, (uint32_t)i, [&](auto qc, bool pore, uint32_t id) {
                constexpr int Q = decltype(qc)::value;
                const uint32_t off =
                    pore ? (uint32_t)opp(Q) * (uint32_t)L.ns + id : (uint32_t)Q * (uint32_t)L.ns + (uint32_t)i;
                sid[Q - 1][threadIdx.x] = (int)off;
                d[Q] = F.row[0][off];
            });
        } else if constexpr (ODD) {
            const uint64_t pol_idx = aa_index_policy();
            const uint32_t p = ld_aa_index(L.vox + i, pol_idx);
            r_own = own_ref<S>(bc, L, p);
            g = own_slope<S>(bc);
            d[0] = S::template dec<0>(F.row[0][i], r_own);
            for_q(std::make_integer_sequence<int, 18>{}, [&](auto qc) {
                constexpr int Q = decltype(qc)::value + 1;
                const int id = ld_aa_index(L.grid + (uint32_t)(p + (uint32_t)L.goff[Q]), pol_idx);
                if constexpr (OFF32) {
                    const uint32_t off = id >= 0 ? (uint32_t)opp(Q) * (uint32_t)L.ns + (uint32_t)id
                                                 : (uint32_t)Q * (uint32_t)L.ns + (uint32_t)i;
                    sid[Q - 1][threadIdx.x] = (int)off;
                    d[Q] = S::template dec<Q>(F.row[0][off], id >= 0 ? r_own - M(cz(Q)) * g : r_own);
                } else {
                    sid[Q - 1][threadIdx.x] = id;
                    d[Q] = id >= 0 ? S::template dec<Q>(F.row[opp(Q)][id], r_own - M(cz(Q)) * g)
                                   : S::template dec<Q>(F.row[Q][i], r_own);
                }
            });
        } else {
            if constexpr (S::kRef)
                r_own = L.nodew ? own_ref_word<S>(bc, L, __ldg(L.nodew + i)) : own_ref<S>(bc, L, __ldg(L.vox + i));
            for_q(AllQ{}, [&](auto qc) {
                constexpr int Q = decltype(qc)::value;
                d[Q] = S::template dec<Q>(F.row[Q][i], r_own);
            });
        }
    }
    if ((int64_t)blockIdx.x * NT < L.a_in) drin = inlet_density<M, NT>(L, bc, slot, partials, sh, blockIdx.x == 0);
    if (i64 < L.n) {
        if (i < L.a_in) {
            close_inlet(d, drin - inlet_known(d));
        } else if (i64 >= L.n - L.a_out) {
            close_outlet(d, outlet_known(d) - M(bc->drho_out));
        }
        collide(d, rates);
        // an opaque copy of i for the stores: sharing the load addresses would keep
        // 19 64-bit addresses live across the collision
        int j;
        asm volatile("mov.b32 %0, %1;" : "=r"(j) : "r"(i));
        if constexpr (ODD && OFF32) {
            F.row[0][j] = S::template enc_sr<0>(d[0], r_own, sr_key<S>(seed, i));
            // a pore destination lies in row Q, a bounce-back one in row opp(Q)
            for_q(std::make_integer_sequence<int, 18>{}, [&](auto qc) {
                constexpr int Q = decltype(qc)::value + 1;
                const uint32_t off = *(volatile uint32_t*)&sid[opp(Q) - 1][threadIdx.x];
                M r = r_own;
                if constexpr (S::kRef && cz(Q) != 0) {
                    const bool pore = (Q & 1) ? off < (uint32_t)(Q + 1) * (uint32_t)L.ns
                                              : off >= (uint32_t)Q * (uint32_t)L.ns;
                    r = pore ? r_own + M(cz(Q)) * g : r_own;
                }
                F.row[0][off] = S::template enc_sr<Q>(d[Q], r, sr_key<S>(seed, i));
            });
        } else if constexpr (ODD) {
            F.row[0][j] = S::template enc_sr<0>(d[0], r_own, sr_key<S>(seed, i));
            for_q(std::make_integer_sequence<int, 18>{}, [&](auto qc) {
                constexpr int Q = decltype(qc)::value + 1;
                const int dst = sid[opp(Q) - 1][threadIdx.x];  // x + xi_Q is the pull source of opp(Q)
                const uint32_t key = sr_key<S>(seed, i);
                if (dst >= 0) F.row[Q][dst] = S::template enc_sr<Q>(d[Q], r_own + M(cz(Q)) * g, key);
                else F.row[opp(Q)][j] = S::template enc_sr<Q>(d[Q], r_own, key);
            });
        } else {
            encode_node<S>(d, seed, i, [&](auto) { return r_own; }, [&](auto qc, typename S::T v) {
                constexpr int Q = decltype(qc)::value;
                F.row[opp(Q)][j] = v;
            });
        }
        if (i64 < L.a_01) {
            // the counted values land on plane 0: from plane 1 (xi_z = -1, stored
            // with plane 0's reference in the odd step) or staying on plane 0
            part = inlet_contribution<S>(L, L.vox[i], i, [&](auto qc) {
                constexpr int Q = decltype(qc)::value;
                const M rq = (ODD && cz(Q) < 0) ? r_own - g : r_own;
                return S::template dec<Q>(S::template enc_sr<Q>(d[Q], rq, sr_key<S>(seed, i)), rq);
            });
        }
    }
    if ((int64_t)blockIdx.x * NT < L.a_01)
        store_inlet_part<S, NT, NT, TILES>(part, blockIdx.x, L, bc, slot, partials, sh);
}

// ------------------------------------------- two nodes per thread (16-bit) ---
// The 16-bit steps of k_step and k_step_aa with the slots i and i + 1 (i even) on
// one thread: 128 threads per 256-node tile.  See lbm_pair.cuh for why.  A row
// ends in padding (rows are multiples of 128 elements, and their node words name
// an interior window), so the slot i + 1 of an odd last node exists; what is
// written there is never read by another node.
// Resident blocks per SM (register caps), measured on those packs: two-buffer step
// 33.6, 33.1 and 34.0 us at 5, 6 and 7; gather-scatter 149, 144 and 148 us at 4, 5
// and 6; node-local 77.6, 76.9 and 98 us at 6, 7 and 8, with the L2 prefetch 448
// tiles ahead (86 us without, 79 at 224).  The staged offsets are read back through
// a volatile pointer: otherwise the compiler keeps all 36 in registers (200 bytes
// of spills, 195 us).
constexpr int kPair = kBlock / 2;  // threads per tile
#ifndef LBM_PAIR_STEP_BLOCKS
#define LBM_PAIR_STEP_BLOCKS 6
#endif
#ifndef LBM_PAIR_ODD_BLOCKS
#define LBM_PAIR_ODD_BLOCKS 5
#endif
#ifndef LBM_PAIR_EVEN_BLOCKS
#define LBM_PAIR_EVEN_BLOCKS 7
#endif
#ifndef LBM_PAIR_EVEN_PREFETCH
#define LBM_PAIR_EVEN_PREFETCH 448
#endif

// Inlet and outlet closures of the nodes i0 < i1 of a thread (both planes are rare).
__device__ __forceinline__ void close_nodes(F2* d, int64_t i0, int64_t i1, const DevLattice& L, const BcState* bc,
                                            float drin) {
    if (i0 < L.a_in || i1 >= L.n - L.a_out) {
        float a[2][19];
#pragma unroll
        for (int q = 0; q < 19; ++q) split(d[q], a[0][q], a[1][q]);
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const int64_t i = k ? i1 : i0;
            if (i < L.a_in) {
                close_inlet(a[k], drin - inlet_known(a[k]));
            } else if (i >= L.n - L.a_out) {
                close_outlet(a[k], outlet_known(a[k]) - float(bc->drho_out));
            }
        }
#pragma unroll
        for (int q = 0; q < 19; ++q) d[q] = f2(a[0][q], a[1][q]);
    }
}

// Their part of the next inlet sum (see inlet_contribution); ref(k, Q): the
// reference density that direction Q's value of node k is stored with.
template <class S, class Ref>
__device__ __forceinline__ double inlet_part_nodes(const F2* d, int64_t i0, int64_t i1, const DevLattice& L,
                                                   uint32_t seed, Ref&& ref) {
    double s = 0.0;
    if (i0 >= L.a_01) return s;
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const int64_t i = k ? i1 : i0;
        if (i < L.a_01) {
            const uint32_t u = sr_key<S>(seed, i);
            s += inlet_contribution<S>(L, L.vox[i], (int)i, [&](auto qc) {
                constexpr int Q = decltype(qc)::value;
                float v[2];
                split(d[Q], v[0], v[1]);
                const float r = ref(k, qc);
                return S::template dec<Q>(S::template enc_sr<Q>(v[k], r, u), r);
            });
        }
    }
    return s;
}

template <class S, bool TILES>
__global__ void __launch_bounds__(kPair, LBM_PAIR_STEP_BLOCKS)
k_step_pair(const StepPtrs<typename S::T> P, int slot, DevLattice L, Rates<float> rates, BcState* bc,
            double* __restrict__ partials) {
    using T = typename S::T;
    __shared__ double sh[32];
    {
        const int64_t s = ((int64_t)blockIdx.x + LBM_STEP_PREFETCH) * kBlock;
        const int t = (int)threadIdx.x;
        if (t < 19) l2_prefetch_range(P.in[0] + (int64_t)t * L.ns, s, kBlock, L.ns);
        else if (t == 19) l2_prefetch_range(L.nodew, s, kBlock, L.n & ~(int64_t)3);
    }
    const int64_t i64 = (int64_t)blockIdx.x * kBlock + 2 * threadIdx.x;
    double part = 0.0;
    const uint32_t i = (uint32_t)i64, ns = (uint32_t)L.ns;
    float r0 = 0.f, r1 = 0.f;
    uint32_t seed = 0;
    F2 d[19];
    if (i64 < L.n) {
        const uint2 w = __ldg(reinterpret_cast<const uint2*>(L.nodew + i));
        const float g = own_slope<S>(bc);
        r0 = own_ref_word<S>(bc, L, w.x);
        r1 = own_ref_word<S>(bc, L, w.y);
        seed = step_seed<S>(bc, slot);
        {
            float v[2][19];
            split(dec2<S, 0>(widen2<S>(__ldg(reinterpret_cast<const uint32_t*>(P.in[0] + i))),
                             f2(float(wq(0)) * r0, float(wq(0)) * r1)), v[0][0], v[1][0]);
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                const float r = k ? r1 : r0;
                const uint32_t ik = i + k;
                for_links(L.win, k ? w.y : w.x, L.wy, L.wz, ik, [&](auto qc, bool pore, uint32_t id) {
                    constexpr int Q = decltype(qc)::value;
                    const uint32_t off = pore ? (uint32_t)Q * ns + id : (uint32_t)opp(Q) * ns + ik;
                    v[k][Q] = S::template dec<Q>(__ldg(P.in[0] + off), (cz(Q) != 0 && pore) ? r - float(cz(Q)) * g : r);
                });
            }
#pragma unroll
            for (int q = 0; q < 19; ++q) d[q] = f2(v[0][q], v[1][q]);
        }
    }
    float drin = 0.f;
    if ((int64_t)blockIdx.x * kBlock < L.a_in)
        drin = inlet_density<float, kPair>(L, bc, slot, partials, sh, blockIdx.x == 0);
    if (i64 < L.n) {
        close_nodes(d, i64, i64 + 1, L, bc, drin);
        collide2<true>(d, rates.sp, rates.sm);
        const F2 nr = f2(-1024.0f * r0, -1024.0f * r1);
        const uint32_t u = sr_key2(seed, i, i + 1u);
        for_q(AllQ{}, [&](auto qc) {
            constexpr int Q = decltype(qc)::value;
            *reinterpret_cast<uint32_t*>(P.out[Q] + i) = enc_sr2<S, Q>(d[Q], nr, u);
        });
        part = inlet_part_nodes<S>(d, i64, i64 + 1, L, seed, [&](int k, auto) { return k ? r1 : r0; });
    }
    if ((int64_t)blockIdx.x * kBlock < L.a_01)
        store_inlet_part<S, kPair, kBlock, TILES>(part, blockIdx.x, L, bc, slot, partials, sh);
}

// Gather-scatter launch: thread t of a warp owns the nodes 64 w + t and
// 64 w + 32 + t, so that a warp's 2-byte gathers and scatters of one node each
// cover consecutive slots (with neighbouring nodes on a thread every store leaves
// half of each sector to the next one: L2 throughput 65 % and the launch slower
// than one node per thread).
template <class S, bool TILES>
__global__ void __launch_bounds__(kPair, LBM_PAIR_ODD_BLOCKS)
k_aa_odd_pair(typename S::T* __restrict__ f, int slot, DevLattice L, Rates<float> rates, BcState* bc,
              double* __restrict__ partials) {
    __shared__ double sh[32];
    // gather offsets: the scatter destination of q is the gather source of opp(q)
    __shared__ uint32_t soff[2][18][kPair];
    {
        const int64_t s = ((int64_t)blockIdx.x + LBM_AA16_PREFETCH) * kBlock;
        const int t = (int)threadIdx.x;
        if (t < 19) l2_prefetch_range(f + (int64_t)t * L.ns, s, kBlock, L.ns);
        else if (t == 19) l2_prefetch_range(L.nodew, s, kBlock, L.n & ~(int64_t)3);
    }
    const int64_t i64 = (int64_t)blockIdx.x * kBlock + 2 * (threadIdx.x & ~31u) + (threadIdx.x & 31u);
    double part = 0.0;
    const uint32_t ns = (uint32_t)L.ns;
    const uint32_t i = (uint32_t)i64;
    // an absent second node repeats the first one's reads and writes nothing
    const bool two = i64 + 32 < L.n;
    const uint32_t i1 = two ? i + 32u : i;
    float g = 0.f, r0 = 0.f, r1 = 0.f;
    uint32_t seed = 0;
    F2 d[19];
    if (i64 < L.n) {
        const uint32_t w0 = __ldg(L.nodew + i), w1 = __ldg(L.nodew + i1);
        g = own_slope<S>(bc);
        r0 = own_ref_word<S>(bc, L, w0);
        r1 = own_ref_word<S>(bc, L, w1);
        seed = step_seed<S>(bc, slot);
        {
            float v[2][19];
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                const float r = k ? r1 : r0;
                const uint32_t ik = k ? i1 : i;
                v[k][0] = S::template dec<0>(f[ik], r);
                for_links(L.win, k ? w1 : w0, L.wy, L.wz, ik, [&](auto qc, bool pore, uint32_t id) {
                    constexpr int Q = decltype(qc)::value;
                    const uint32_t o = pore ? (uint32_t)opp(Q) * ns + id : (uint32_t)Q * ns + ik;
                    soff[k][Q - 1][threadIdx.x] = o;
                    v[k][Q] = S::template dec<Q>(f[o], (cz(Q) != 0 && pore) ? r - float(cz(Q)) * g : r);
                });
            }
#pragma unroll
            for (int q = 0; q < 19; ++q) d[q] = f2(v[0][q], v[1][q]);
        }
    }
    float drin = 0.f;
    if ((int64_t)blockIdx.x * kBlock < L.a_in)
        drin = inlet_density<float, kPair>(L, bc, slot, partials, sh, blockIdx.x == 0);
    if (i64 < L.n) {
        close_nodes(d, i64, i64 + 32, L, bc, drin);
        collide2<false>(d, rates.sp, rates.sm);
        const float m0 = -1024.0f * r0, m1 = -1024.0f * r1;
        const uint32_t u = sr_key2(seed, i, i + 32u);
        {
            const uint32_t h = enc_sr2<S, 0>(d[0], f2(m0, m1), u);
            f[i] = S::half_of(h, false);
            if (two) f[i1] = S::half_of(h, true);
        }
        // a value for a pore on another plane is encoded with that plane's reference
        const float up0 = -1024.0f * (r0 + g), up1 = -1024.0f * (r1 + g);
        const float dn0 = -1024.0f * (r0 - g), dn1 = -1024.0f * (r1 - g);
        for_q(std::make_integer_sequence<int, 18>{}, [&](auto qc) {
            constexpr int Q = decltype(qc)::value + 1;
            const uint32_t o0 = *(volatile uint32_t*)&soff[0][opp(Q) - 1][threadIdx.x];
            const uint32_t o1 = *(volatile uint32_t*)&soff[1][opp(Q) - 1][threadIdx.x];
            F2 n = f2(m0, m1);
            if constexpr (cz(Q) != 0) {
                // a pore destination lies in row Q, a bounce-back one in row opp(Q)
                const bool p0 = (Q & 1) ? o0 < (uint32_t)(Q + 1) * ns : o0 >= (uint32_t)Q * ns;
                const bool p1 = (Q & 1) ? o1 < (uint32_t)(Q + 1) * ns : o1 >= (uint32_t)Q * ns;
                n = f2(p0 ? (cz(Q) > 0 ? up0 : dn0) : m0, p1 ? (cz(Q) > 0 ? up1 : dn1) : m1);
            }
            const uint32_t h = enc_sr2<S, Q>(d[Q], n, u);
            f[o0] = S::half_of(h, false);
            if (two) f[o1] = S::half_of(h, true);
        });
        part = inlet_part_nodes<S>(d, i64, i64 + 32, L, seed, [&](int k, auto qc) {
            const float r = k ? r1 : r0;
            return cz(decltype(qc)::value) < 0 ? r - g : r;
        });
    }
    if ((int64_t)blockIdx.x * kBlock < L.a_01)
        store_inlet_part<S, kPair, kBlock, TILES>(part, blockIdx.x, L, bc, slot, partials, sh);
}

// Node-local launch: neighbouring nodes on a thread, one 4-byte load and store per row.
template <class S, bool TILES>
__global__ void __launch_bounds__(kPair, LBM_PAIR_EVEN_BLOCKS)
k_aa_even_pair(const AAPtrs<typename S::T> F, int slot, DevLattice L, Rates<float> rates, BcState* bc,
               double* __restrict__ partials) {
    __shared__ double sh[32];
    if constexpr (LBM_PAIR_EVEN_PREFETCH > 0) {
        const int64_t s = ((int64_t)blockIdx.x + LBM_PAIR_EVEN_PREFETCH) * kBlock;
        const int t = (int)threadIdx.x;
        if (t < 19) l2_prefetch_range(F.row[0] + (int64_t)t * L.ns, s, kBlock, L.ns);
        else if (t == 19) l2_prefetch_range(L.nodew, s, kBlock, L.n & ~(int64_t)3);
    }
    const int64_t i64 = (int64_t)blockIdx.x * kBlock + 2 * threadIdx.x;
    double part = 0.0;
    const uint32_t i = (uint32_t)i64;
    float r0 = 0.f, r1 = 0.f;
    uint32_t seed = 0;
    F2 d[19];
    if (i64 < L.n) {
        uint32_t raw[19];
        for_q(AllQ{}, [&](auto qc) {
            constexpr int Q = decltype(qc)::value;
            raw[Q] = *reinterpret_cast<const uint32_t*>(F.row[Q] + i);
        });
        const uint2 w = __ldg(reinterpret_cast<const uint2*>(L.nodew + i));
        r0 = own_ref_word<S>(bc, L, w.x);
        r1 = own_ref_word<S>(bc, L, w.y);
        seed = step_seed<S>(bc, slot);
        for_q(AllQ{}, [&](auto qc) {
            constexpr int Q = decltype(qc)::value;
            d[Q] = dec2<S, Q>(widen2<S>(raw[Q]), f2(float(wq(Q)) * r0, float(wq(Q)) * r1));
        });
    }
    float drin = 0.f;
    if ((int64_t)blockIdx.x * kBlock < L.a_in)
        drin = inlet_density<float, kPair>(L, bc, slot, partials, sh, blockIdx.x == 0);
    if (i64 < L.n) {
        close_nodes(d, i64, i64 + 1, L, bc, drin);
        collide2<false>(d, rates.sp, rates.sm);
        const F2 nr = f2(-1024.0f * r0, -1024.0f * r1);
        const uint32_t u = sr_key2(seed, i, i + 1u);
        uint32_t j;  // an opaque copy: the store addresses must not stay live from the loads
        asm volatile("mov.b32 %0, %1;" : "=r"(j) : "r"(i));
        for_q(AllQ{}, [&](auto qc) {
            constexpr int Q = decltype(qc)::value;
            *reinterpret_cast<uint32_t*>(F.row[opp(Q)] + j) = enc_sr2<S, Q>(d[Q], nr, u);
        });
        part = inlet_part_nodes<S>(d, i64, i64 + 1, L, seed, [&](int k, auto) { return k ? r1 : r0; });
    }
    if ((int64_t)blockIdx.x * kBlock < L.a_01)
        store_inlet_part<S, kPair, kBlock, TILES>(part, blockIdx.x, L, bc, slot, partials, sh);
}

// Pull layout <-> layout S: swap F[q][x] and F[opp q][x] at every node.
// All 18 loads are issued before any store (the rows of one buffer could alias
// as far as the compiler knows, which would serialise load-store pairs).
template <class T>
__global__ void k_aa_swap(T* __restrict__ f, int64_t n, int64_t ns) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    T v[19];
#pragma unroll
    for (int q = 1; q < 19; ++q) v[q] = f[(int64_t)q * ns + i];
#pragma unroll
    for (int q = 1; q < 19; q += 2) {  // opposite pairs are (q, q + 1), q odd
        f[(int64_t)q * ns + i] = v[q + 1];
        f[(int64_t)(q + 1) * ns + i] = v[q];
    }
}

// Layout I -> layout S after an odd step: the value that arrived at x in
// direction q from the pore x - xi_q belongs in F[opp q][x - xi_q], and that
// slot holds the value that arrived at x - xi_q in direction opp q from x,
// which belongs in F[q][x]: one swap per pair, done by the node with odd q.
// A value that arrived by bounce-back is already in place.
// 16-bit formats: a moved value is re-encoded from its old holder's plane to
// the new one's (opposite directions share the weight).
template <class S>
__global__ void k_aa_unstream(typename S::T* __restrict__ f, DevLattice L, const BcState* bc) {
    using T = typename S::T;
    using M = typename S::M;
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= L.n) return;
    const uint32_t p = L.vox[i];
    const M r_own = own_ref<S>(bc, L, p), g = own_slope<S>(bc);
    // ids and values first, stores after (see k_aa_swap)
    int id[19];
    T ta[19], tb[19];
    for_q(std::integer_sequence<int, 1, 3, 5, 7, 9, 11, 13, 15, 17>{}, [&](auto qc) {
        constexpr int Q = decltype(qc)::value;
        id[Q] = __ldg(L.grid + (uint32_t)(p + (uint32_t)L.goff[Q]));
    });
    for_q(std::integer_sequence<int, 1, 3, 5, 7, 9, 11, 13, 15, 17>{}, [&](auto qc) {
        constexpr int Q = decltype(qc)::value;
        if (id[Q] >= 0) {
            ta[Q] = f[(int64_t)Q * L.ns + i];
            tb[Q] = f[(int64_t)(Q + 1) * L.ns + id[Q]];
        }
    });
    for_q(std::integer_sequence<int, 1, 3, 5, 7, 9, 11, 13, 15, 17>{}, [&](auto qc) {
        constexpr int Q = decltype(qc)::value;
        if (id[Q] >= 0) {
            T* a = f + (int64_t)Q * L.ns + i;
            T* b = f + (int64_t)(Q + 1) * L.ns + id[Q];
            if constexpr (S::kRef) {
                const M r_src = r_own - M(cz(Q)) * g;  // plane of x - xi_Q
                *a = S::template enc<Q>(S::template dec<Q>(tb[Q], r_src), r_own);
                *b = S::template enc<Q>(S::template dec<Q>(ta[Q], r_own), r_src);
            } else {
                *a = tb[Q];
                *b = ta[Q];
            }
        }
    });
}

// ------------------------------------------------ pipelined step kernel ---
// The same step as k_step, restructured for memory-level parallelism: a
// persistent grid walks 256-node tiles (tile t, t + G, t + 2G, ...), and every
// gather goes through cp.async into shared memory one tile ahead of its use:
//   A(t): the 18 neighbour ids of tile t        (id grid -> smem, L2 evict-last)
//   B(t): the 19 pulled values of tile t         (distributions -> smem)
// While tile t is collided, B(t + G) and A(t + 2G) are in flight, so the loads
// outstanding per SM no longer cost registers.  Each thread only reads back the
// shared-memory slots its own copies filled, so the pipeline needs no barrier.
// 16-bit values are fetched as the aligned 4-byte pair that contains them.

__device__ __forceinline__ unsigned smem_u32(const void* p) {
    return (unsigned)__cvta_generic_to_shared(p);
}
template <int BYTES>
__device__ __forceinline__ void cp_async(unsigned dst, const void* src) {
    if constexpr (BYTES == 8)
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(dst), "l"(src) : "memory");
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_hint4(unsigned dst, const void* src, uint64_t pol) {
    asm volatile("cp.async.ca.shared.global.L2::cache_hint [%0], [%1], 4, 4, %2;" ::"r"(dst), "l"(src), "l"(pol)
                 : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }

template <class S>
struct AsyncSlot {
    using T = typename S::T;
    static constexpr int kBytes = sizeof(T) >= 4 ? (int)sizeof(T) : 4;  // bytes fetched per value
};

template <int NT>
constexpr size_t async_smem_bytes(int slot_bytes) {
    return (size_t)18 * NT * 4 + (size_t)2 * 19 * NT * slot_bytes;
}

// A(t): neighbour ids of this thread's node of tile t into ids[q-1][tid].
template <int NT>
__device__ __forceinline__ void issue_ids(int* ids, const DevLattice& L, uint32_t p, uint64_t pol) {
    for_q(std::make_integer_sequence<int, 18>{}, [&](auto qc) {
        constexpr int Q = decltype(qc)::value + 1;
        cp_async_hint4(smem_u32(ids + (Q - 1) * NT + threadIdx.x), L.grid + (int64_t)p + L.goff[Q], pol);
    });
}

// B(t): the 19 pulled values of node i into vals[q][tid]; returns the bit mask
// of 16-bit values that sit in the upper half of their fetched 4-byte pair.
template <class S, int NT>
__device__ __forceinline__ unsigned issue_vals(unsigned char* vals, const int* ids,
                                               const StepPtrs<typename S::T>& P, int i, unsigned& nbr) {
    using T = typename S::T;
    constexpr int SB = AsyncSlot<S>::kBytes;
    unsigned hi = 0;
    nbr = 0;
    for_q(AllQ{}, [&](auto qc) {
        constexpr int Q = decltype(qc)::value;
        const T* a;
        if constexpr (Q == 0) {
            a = P.in[0] + i;
        } else {
            const int id = ids[(Q - 1) * NT + threadIdx.x];
            a = id >= 0 ? P.in[Q] + id : P.in[opp(Q)] + i;
            if constexpr (S::kRef && cz(Q) != 0) nbr |= (unsigned)(id >= 0) << Q;
        }
        const unsigned dst = smem_u32(vals + ((size_t)Q * NT + threadIdx.x) * SB);
        if constexpr (sizeof(T) == 2) {
            const uintptr_t u = reinterpret_cast<uintptr_t>(a);
            hi |= (unsigned)((u >> 1) & 1u) << Q;
            cp_async<4>(dst, reinterpret_cast<const void*>(u & ~(uintptr_t)3));
        } else {
            cp_async<SB>(dst, a);
        }
    });
    return hi;
}

template <class S, int NT>
__device__ __forceinline__ void read_vals(typename S::M* d, const unsigned char* vals, unsigned hi,
                                          unsigned nbr, typename S::M r_own, typename S::M g) {
    using T = typename S::T;
    using M = typename S::M;
    constexpr int SB = AsyncSlot<S>::kBytes;
    for_q(AllQ{}, [&](auto qc) {
        constexpr int Q = decltype(qc)::value;
        const unsigned char* slot = vals + ((size_t)Q * NT + threadIdx.x) * SB;
        const M r = (cz(Q) != 0 && ((nbr >> Q) & 1u)) ? r_own - M(cz(Q)) * g : r_own;
        if constexpr (sizeof(T) == 2) {
            const T* pair = reinterpret_cast<const T*>(slot);
            d[Q] = S::template dec<Q>(pair[(hi >> Q) & 1u], r);
        } else {
            d[Q] = S::template dec<Q>(*reinterpret_cast<const T*>(slot), r);
        }
    });
}

template <class S, int NT, bool TILES>
__global__ void __launch_bounds__(NT)
k_step_async(const StepPtrs<typename S::T> P, int slot, DevLattice L, Rates<typename S::M> rates, BcState* bc, double* __restrict__ partials) {
    using M = typename S::M;
    constexpr int SB = AsyncSlot<S>::kBytes;
    extern __shared__ __align__(16) unsigned char smem[];
    int* ids = reinterpret_cast<int*>(smem);
    unsigned char* vals0 = smem + (size_t)18 * NT * 4;
    unsigned char* vals1 = vals0 + (size_t)19 * NT * SB;
    __shared__ double sh[32];

    const int64_t ntiles = (L.n + NT - 1) / NT;
    const int64_t nt01 = (L.a_01 + NT - 1) / NT;
    const int64_t G = gridDim.x;
    const uint64_t pol_idx = l2_policy_evict_last();
    auto node = [&](int64_t t) -> int64_t { return t * NT + threadIdx.x; };

    int64_t t = blockIdx.x;
    if (t >= ntiles) return;
    // prologue: A(t); wait; B(t); A(t + G)
    uint32_t p_cur = 0, p_next = 0, p_next2 = 0;
    if (node(t) < L.n) p_cur = __ldg(L.vox + node(t));
    if (t + G < ntiles && node(t + G) < L.n) p_next = __ldg(L.vox + node(t + G));
    if (t + 2 * G < ntiles && node(t + 2 * G) < L.n) p_next2 = __ldg(L.vox + node(t + 2 * G));
    if (node(t) < L.n) issue_ids<NT>(ids, L, p_cur, pol_idx);
    cp_async_commit();
    cp_async_wait_all();
    unsigned hi_cur = 0, hi_next = 0, nb_cur = 0, nb_next = 0;
    if (node(t) < L.n) hi_cur = issue_vals<S, NT>(vals0, ids, P, (int)node(t), nb_cur);
    cp_async_commit();
    if (t + G < ntiles && node(t + G) < L.n) issue_ids<NT>(ids, L, p_next, pol_idx);
    cp_async_commit();
    M drin = M(0);
    if (t * NT < L.a_in) drin = inlet_density<M, NT>(L, bc, slot, partials, sh, t == 0);

    for (int k = 0; t < ntiles; ++k, t += G) {
        unsigned char* vcur = (k & 1) ? vals1 : vals0;
        unsigned char* vnext = (k & 1) ? vals0 : vals1;
        cp_async_wait_all();  // B(t) and A(t + G) have landed
        const int64_t tn = t + G, tn2 = t + 2 * G;
        if (tn < ntiles && node(tn) < L.n) hi_next = issue_vals<S, NT>(vnext, ids, P, (int)node(tn), nb_next);
        cp_async_commit();
        if (tn2 < ntiles && node(tn2) < L.n) issue_ids<NT>(ids, L, p_next2, pol_idx);
        cp_async_commit();
        const int64_t tn3 = t + 3 * G;
        const uint32_t p_after = (tn3 < ntiles && node(tn3) < L.n) ? __ldg(L.vox + node(tn3)) : 0u;

        // ---- collide tile t (its values are in vcur)
        const int64_t i64 = node(t);
        double part = 0.0;
        if (i64 < L.n) {
            const int i = (int)i64;
            const M r_own = own_ref<S>(bc, L, p_cur), g = own_slope<S>(bc);
            const uint32_t seed = step_seed<S>(bc, slot);
            M d[19];
            read_vals<S, NT>(d, vcur, hi_cur, nb_cur, r_own, g);
            if (i < L.a_in) {
                close_inlet(d, drin - inlet_known(d));
            } else if (i64 >= L.n - L.a_out) {
                const M uz = outlet_known(d) - M(bc->drho_out);
                close_outlet(d, uz);
            }
            collide(d, rates);
            encode_node<S>(d, seed, i, [&](auto) { return r_own; }, [&](auto qc, typename S::T v) {
                constexpr int Q = decltype(qc)::value;
                P.out[Q][i] = v;
            });
            if (i64 < L.a_01) part = next_inlet_part<S>(d, L, p_cur, i, r_own, seed);
        }
        if (t < nt01)  // tile holds plane z = 0 / z = 1 nodes (block-uniform)
            store_inlet_part<S, NT, NT, TILES>(part, t, L, bc, slot, partials, sh);
        hi_cur = hi_next;
        nb_cur = nb_next;
        p_cur = p_next;
        p_next = p_next2;
        p_next2 = p_after;
    }
    cp_async_wait_all();
}

// ---------------------------------------------------------- monitors ---
template <class S>
__global__ void __launch_bounds__(kReduceBlock)
k_monitors(const typename S::T* __restrict__ f, DevLattice L, const BcState* bc,
           double* __restrict__ partials, unsigned* __restrict__ counter, MonitorOut* out) {
    using M = typename S::M;
    __shared__ double sh[32];
    __shared__ bool last;
    const int64_t i64 = (int64_t)blockIdx.x * kReduceBlock + threadIdx.x;
    M v[5] = {M(0), M(0), M(0), M(0), M(0)};
    if (i64 < L.n) {
        const int i = (int)i64;
        const M r_own = own_ref<S>(bc, L, L.vox[i]);
        M d[19];
        for_q(AllQ{}, [&](auto qc) {
            constexpr int Q = decltype(qc)::value;
            d[Q] = S::template dec<Q>(f[(int64_t)Q * L.ns + i], r_own);
        });
        M drho, jx, jy, jz;
        moments(d, drho, jx, jy, jz);
        const M u2 = jx * jx + jy * jy + jz * jz;
        const bool bad = !isfinite((double)drho) || !isfinite((double)u2);
        v[0] = bad ? M(0) : drho;
        if (i64 < L.a_in && !bad) v[1] = jz;
        if (i64 >= L.n - L.a_out && !bad) v[2] = jz;
        v[3] = bad ? M(0) : u2;
        v[4] = bad ? M(1) : M(0);
    }
    const int nb = gridDim.x;
    double r[5];
    r[0] = block_sum_m<kReduceBlock>(v[0], sh);
    r[1] = block_sum_m<kReduceBlock>(v[1], sh);
    r[2] = block_sum_m<kReduceBlock>(v[2], sh);
    r[3] = block_max_m<kReduceBlock>(v[3], sh);
    r[4] = block_sum_m<kReduceBlock>(v[4], sh);
    if (threadIdx.x == 0) {
        for (int c = 0; c < 5; ++c) partials[(int64_t)c * nb + blockIdx.x] = r[c];
        __threadfence();
        last = atomicAdd(counter, 1u) == (unsigned)nb - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    double acc[5] = {0, 0, 0, 0, 0};
    for (int j = threadIdx.x; j < nb; j += kReduceBlock) {
        acc[0] += __ldcg(partials + j);
        acc[1] += __ldcg(partials + (int64_t)nb + j);
        acc[2] += __ldcg(partials + 2 * (int64_t)nb + j);
        acc[3] = fmax(acc[3], __ldcg(partials + 3 * (int64_t)nb + j));
        acc[4] += __ldcg(partials + 4 * (int64_t)nb + j);
    }
    const double t0 = block_sum<kReduceBlock>(acc[0], sh);
    const double t1 = block_sum<kReduceBlock>(acc[1], sh);
    const double t2 = block_sum<kReduceBlock>(acc[2], sh);
    const double t3 = block_max<kReduceBlock>(acc[3], sh);
    const double t4 = block_sum<kReduceBlock>(acc[4], sh);
    if (threadIdx.x == 0) {
        out->drho_sum = t0;
        out->q_in = t1;
        out->q_out = t2;
        out->umax2 = t3;
        out->nan_count = t4;
        *counter = 0u;
    }
}

// ------------------------------------------------- steady residual ---
// Section 3.1 stopping criterion: sum_x |u(x,t) - u(x,t_ref)| and sum_x |u(x,t)|
// (|.| the Euclidean norm per node), FP64; u_ref <- u(t) for the next call.
template <class S>
__global__ void __launch_bounds__(kReduceBlock)
k_velocity_change(const typename S::T* __restrict__ f, DevLattice L, const BcState* bc,
                  double* __restrict__ u_ref,
                  double* __restrict__ partials, unsigned* __restrict__ counter, MonitorOut* out) {
    using M = typename S::M;
    __shared__ double sh[32];
    __shared__ bool last;
    const int64_t i64 = (int64_t)blockIdx.x * kReduceBlock + threadIdx.x;
    M dn = M(0), un = M(0);
    if (i64 < L.n) {
        const M r_own = own_ref<S>(bc, L, L.vox[i64]);
        M d[19];
        for_q(AllQ{}, [&](auto qc) {
            constexpr int Q = decltype(qc)::value;
            d[Q] = S::template dec<Q>(f[(int64_t)Q * L.ns + i64], r_own);
        });
        M drho, jx, jy, jz;
        moments(d, drho, jx, jy, jz);
        const M u[3] = {jx, jy, jz};
        M d2 = M(0), u2 = M(0);
        for (int c = 0; c < 3; ++c) {
            const M r = (M)u_ref[(int64_t)c * L.n + i64];
            d2 += (u[c] - r) * (u[c] - r);
            u2 += u[c] * u[c];
            u_ref[(int64_t)c * L.n + i64] = (double)u[c];
        }
        dn = sqrt(d2);
        un = sqrt(u2);
    }
    const int nb = gridDim.x;
    const double b0 = block_sum_m<kReduceBlock>(dn, sh);
    const double b1 = block_sum_m<kReduceBlock>(un, sh);
    if (threadIdx.x == 0) {
        partials[blockIdx.x] = b0;
        partials[(int64_t)nb + blockIdx.x] = b1;
        __threadfence();
        last = atomicAdd(counter, 1u) == (unsigned)nb - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    double a0 = 0.0, a1 = 0.0;
    for (int j = threadIdx.x; j < nb; j += kReduceBlock) {
        a0 += __ldcg(partials + j);
        a1 += __ldcg(partials + (int64_t)nb + j);
    }
    const double t0 = block_sum<kReduceBlock>(a0, sh);
    const double t1 = block_sum<kReduceBlock>(a1, sh);
    if (threadIdx.x == 0) {
        out->drho_sum = t0;  // sum |u - u_ref|
        out->q_in = t1;      // sum |u|
        *counter = 0u;
    }
}

// ---------------------------------------------------------- re-encode ---
// 16-bit formats: move the reference profile to r(z) = r0 + g z with r0 = the
// inlet density of the next step (drho_in[slot]) and g from there to the
// outlet density, re-encoding every stored value in place (each node owns its
// values).  Reads profile slot e, writes slot e ^ 1 and selects it.
template <class S>
__global__ void k_reencode(typename S::T* __restrict__ f, DevLattice L, BcState* bc, int e, int slot) {
    using M = typename S::M;
    const float r0n = (float)bc->drho_in[slot];
    const float gn = (float)((bc->drho_out - bc->drho_in[slot]) / (double)(L.nz - 1));
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i == 0) {
        bc->ref_r0[e ^ 1] = r0n;
        bc->ref_g[e ^ 1] = gn;
        bc->ref_cur = e ^ 1;
    }
    if (i >= L.n) return;
    const int z = plane_of((uint64_t)L.vox[i], L.sz_magic);
    const M r_old = M(bc->ref_r0[e]) + M(bc->ref_g[e]) * M(z);
    const M r_new = M(r0n) + M(gn) * M(z);
    for_q(AllQ{}, [&](auto qc) {
        constexpr int Q = decltype(qc)::value;
        typename S::T* a = f + (int64_t)Q * L.ns + i;
        *a = S::template enc<Q>(S::template dec<Q>(*a, r_old), r_new);
    });
}

// ---------------------------------------------------- conversions ---
__device__ __forceinline__ int64_t unpadded(const DevLattice& L, int64_t p) {
    const int64_t z = p / L.sz - 1;
    const int64_t rem = p % L.sz;
    const int64_t y = rem / L.sy - 1;
    const int64_t x = rem % L.sy - 1;
    return (z * L.ny + y) * L.nx + x;
}

template <class S, class O>
__global__ void k_export(const typename S::T* __restrict__ f, DevLattice L, const BcState* bc, O* rho,
                         O* ux, O* uy, O* uz) {
    using M = typename S::M;
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= L.n) return;
    const M r_own = own_ref<S>(bc, L, L.vox[i]);
    M d[19];
    for_q(AllQ{}, [&](auto qc) {
        constexpr int Q = decltype(qc)::value;
        d[Q] = S::template dec<Q>(f[(int64_t)Q * L.ns + i], r_own);
    });
    M drho, jx, jy, jz;
    moments(d, drho, jx, jy, jz);
    const int64_t o = unpadded(L, L.vox[i]);
    if (rho) rho[o] = (O)(1.0 + (double)drho);
    if (ux) ux[o] = (O)jx;
    if (uy) uy[o] = (O)jy;
    if (uz) uz[o] = (O)jz;
}

template <class S>
__global__ void k_init_eq(typename S::T* __restrict__ f, DevLattice L, const BcState* bc, const double* rho,
                          const double* ux, const double* uy, const double* uz) {
    using M = typename S::M;
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= L.n) return;
    const M r_own = own_ref<S>(bc, L, L.vox[i]);
    const M dr = rho ? M(rho[i] - 1.0) : M(0);
    const M u[3] = {ux ? M(ux[i]) : M(0), uy ? M(uy[i]) : M(0), uz ? M(uz[i]) : M(0)};
    const M uu15 = M(1.5) * (u[0] * u[0] + u[1] * u[1] + u[2] * u[2]);
    for_q(AllQ{}, [&](auto qc) {
        constexpr int Q = decltype(qc)::value;
        const M xu = M(cx(Q)) * u[0] + M(cy(Q)) * u[1] + M(cz(Q)) * u[2];
        const M dq = M(wq(Q)) * (dr + M(3) * xu + M(4.5) * xu * xu - uu15);
        f[(int64_t)Q * L.ns + i] = S::template enc<Q>(dq, r_own);
    });
}

template <class S>
__global__ void k_encode(typename S::T* __restrict__ f, DevLattice L, const BcState* bc,
                         const double* __restrict__ d) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= L.n) return;
    const typename S::M r_own = own_ref<S>(bc, L, L.vox[i]);
    for_q(AllQ{}, [&](auto qc) {
        constexpr int Q = decltype(qc)::value;
        f[(int64_t)Q * L.ns + i] = S::template enc<Q>((typename S::M)d[(int64_t)Q * L.n + i], r_own);
    });
}

template <class S>
__global__ void k_decode(const typename S::T* __restrict__ f, DevLattice L, const BcState* bc,
                         double* __restrict__ d) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= L.n) return;
    const typename S::M r_own = own_ref<S>(bc, L, L.vox[i]);
    for_q(AllQ{}, [&](auto qc) {
        constexpr int Q = decltype(qc)::value;
        d[(int64_t)Q * L.n + i] = (double)S::template dec<Q>(f[(int64_t)Q * L.ns + i], r_own);
    });
}

// Row windows (lbm_device.cuh) of one padded box from its id grid, one thread per window.
__global__ void k_windows(const int* __restrict__ grid, int sy, int rows, int nw, uint2* __restrict__ win) {
    const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= (int64_t)rows * nw) return;
    const int64_t row = k / nw;
    const int x0 = 30 * (int)(k - row * nw);
    uint32_t bits = 0, first = 0;
    for (int b = 31; b >= 0; --b) {  // a bit past the padded row stays 0
        const int id = x0 + b < sy ? grid[row * sy + x0 + b] : SOLID;
        if (id >= 0) {
            bits |= 1u << b;
            first = (uint32_t)id;
        }
    }
    win[k] = make_uint2(bits, first);
}
// Words of n nodes; those of the padding slots up to n_pad name an interior window.
__global__ void k_node_words(const uint32_t* __restrict__ vox, uint32_t vox0, int64_t n, int64_t n_pad, int sy, int nw,
                             uint32_t w0, uint32_t w_pad, uint32_t* __restrict__ nodew) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n_pad) return;
    uint32_t word = w_pad << 5 | 1u;
    if (i < n) {
        const uint32_t p = vox[i] - vox0, row = p / (uint32_t)sy, x = p - row * (uint32_t)sy, w = (x - 1u) / 30u;
        word = (w0 + row * (uint32_t)nw + w) << 5 | (x - 30u * w);
    }
    nodew[i] = word;
}

// FP64 lattices of at most one wave of 256-node blocks (152 SMs, one such block
// resident) run in small blocks, so that every SM's FP64 units get an even share:
// 16x16x64 duct, 12,544 nodes, 100 steps 2.05 -> 1.64 ms.  Near the line, per step in
// small blocks and before them: 30x30x48 duct, 37,632 nodes 16.5 and 22.2 us; above it
// (32x32x48, 43,200 nodes, two waves of 256-node blocks) 23.8 and 31.8 us.  FP32 (61x67x72 pack,
// 112 k nodes) measured slower: 1.01 ms in blocks of 256, 1.02 in 128, 1.17 in 64.
constexpr int64_t kSmallNodes = 152 * 256;
constexpr int kSmallBlock = 32;
static_assert(kSmallNodes / kSmallBlock <= LBM_PARTS_DIRECT, "a step in small blocks leaves no parts to fold");

inline unsigned blocks_for(int64_t n, int b) { return (unsigned)((n + b - 1) / b); }

template <class F>
cudaError_t dispatch(int prec, F&& f) {
    switch (prec) {
        case 0: return f(StoreF64{});
        case 1: return f(StoreF32{});
        case 2: return f(StoreF16{});
        case 3: return f(StoreBF16{});
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace

cudaError_t launch_build_windows(const int* grid, const uint32_t* vox, uint32_t vox0, int64_t n, int64_t n_pad,
                                 int nx, int ny, int nz, uint32_t w0, uint2* win, uint32_t* nodew, cudaStream_t st) {
    const int nw = windows_per_row(nx), rows = (ny + 2) * (nz + 2);
    k_windows<<<blocks_for((int64_t)rows * nw, 256), 256, 0, st>>>(grid, nx + 2, rows, nw, win + w0);
    const uint32_t w_pad = w0 + (uint32_t)nw * (uint32_t)(ny + 3);  // row y = 0 of plane z = 0
    k_node_words<<<blocks_for(n_pad, 256), 256, 0, st>>>(vox, vox0, n, n_pad, nx + 2, nw, w0, w_pad, nodew);
    return cudaGetLastError();
}

int elem_size(int prec) { return prec == 0 ? 8 : prec == 1 ? 4 : 2; }
int inlet_reduce_blocks(const DevLattice& L) { return (int)blocks_for(L.a_in, kReduceBlock); }
int monitor_blocks(const DevLattice& L) { return (int)blocks_for(L.n, kReduceBlock); }

cudaError_t launch_inlet_reduce(int prec, const void* fin, int slot, const DevLattice& L, BcState* bc,
                                double* partials, unsigned* counter, cudaStream_t st) {
    return dispatch(prec, [&](auto s) {
        using S = decltype(s);
        k_inlet_reduce<S><<<inlet_reduce_blocks(L), kReduceBlock, 0, st>>>(
            (const typename S::T*)fin, slot, L, bc, partials, counter);
        return cudaGetLastError();
    });
}

cudaError_t launch_step(int prec, const void* fin, void* fout, int slot, const DevLattice& L, Relax r,
                        BcState* bc, double* partials, cudaStream_t st) {
    return dispatch(prec, [&](auto s) {
        using S = decltype(s);
        using M = typename S::M;
        using T = typename S::T;
        StepPtrs<T> P;
        for (int q = 0; q < 19; ++q) {
            P.in[q] = (const T*)fin + (int64_t)q * L.ns;
            P.out[q] = (T*)fout + (int64_t)q * L.ns;
        }
        // GB300_LBM_STEP_ADDR64 forces the id-grid form with 64-bit addresses (tests)
        const bool off32 = 19 * (uint64_t)L.ns <= 0xFFFFFFFFull && !std::getenv("GB300_LBM_STEP_ADDR64");
        const bool win = L.win && off32;
        const unsigned nb = blocks_for(L.n, kBlock);
        const auto rates = make_rates<M>(r.sp, r.sm);
        if constexpr (sizeof(M) == 8) {
            if (win && L.n < kSmallNodes) {
                k_step<S, kWindows, kSmallBlock, false><<<blocks_for(L.n, kSmallBlock), kSmallBlock, 0, st>>>(
                    P, slot, L, rates, bc, partials);
                return cudaGetLastError();
            }
        }
        return with_parts<M>(L, [&](auto tiles) {
            constexpr bool TILES = decltype(tiles)::value;
            if (win) {
                if constexpr (S::kRef) {
                    k_step_pair<S, TILES><<<nb, kPair, 0, st>>>(P, slot, L, rates, bc, partials);
                    return fold_parts<kPair, TILES>(L, slot, partials, kBlock, st);
                } else {
                    k_step<S, kWindows, kBlock, TILES><<<nb, kBlock, 0, st>>>(P, slot, L, rates, bc, partials);
                }
            } else if (off32) {
                k_step<S, kGrid32, kBlock, TILES><<<nb, kBlock, 0, st>>>(P, slot, L, rates, bc, partials);
            } else {
                k_step<S, kGrid64, kBlock, TILES><<<nb, kBlock, 0, st>>>(P, slot, L, rates, bc, partials);
            }
            return fold_parts<kBlock, TILES>(L, slot, partials, kBlock, st);
        });
    });
}

template <class S, int NT>
cudaError_t launch_async_t(const void* fin, void* fout, int slot, const DevLattice& L, Relax r, BcState* bc,
                           double* partials, cudaStream_t st, int grid) {
    using T = typename S::T;
    using M = typename S::M;
    StepPtrs<T> P;
    for (int q = 0; q < 19; ++q) {
        P.in[q] = (const T*)fin + (int64_t)q * L.ns;
        P.out[q] = (T*)fout + (int64_t)q * L.ns;
    }
    const size_t smem = async_smem_bytes<NT>(AsyncSlot<S>::kBytes);
    return with_parts<M>(L, [&](auto tiles) {
        constexpr bool TILES = decltype(tiles)::value;
        k_step_async<S, NT, TILES><<<grid, NT, smem, st>>>(P, slot, L, make_rates<M>(r.sp, r.sm), bc, partials);
        return fold_parts<NT, TILES>(L, slot, partials, NT, st);
    });
}

template <class S, int NT>
cudaError_t config_async_t(int* grid, const DevLattice& L) {
    using M = typename S::M;
    const size_t smem = async_smem_bytes<NT>(AsyncSlot<S>::kBytes);
    return with_parts<M>(L, [&](auto tiles) {
        auto* kernel = k_step_async<S, NT, decltype(tiles)::value>;
        cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        int per_sm = 0, dev = 0, sms = 0;
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, NT, smem);
        if (e != cudaSuccess) return e;
        if (per_sm < 1) return cudaErrorInvalidConfiguration;
        if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
        if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
        const int64_t ntiles = (L.n + NT - 1) / NT;
        *grid = (int)std::min<int64_t>((int64_t)per_sm * sms, ntiles);
        return cudaSuccess;
    });
}

cudaError_t launch_inlet_finish(const DevLattice& L, BcState* bc, int slot, const double* partials, cudaStream_t st) {
    k_inlet_finish<<<1, kReduceBlock, 0, st>>>(L, bc, slot, partials);
    return cudaGetLastError();
}

cudaError_t launch_monitors(int prec, const void* f, const DevLattice& L, const BcState* bc, double* partials,
                            unsigned* counter, MonitorOut* out, cudaStream_t st) {
    return dispatch(prec, [&](auto s) {
        using S = decltype(s);
        k_monitors<S><<<monitor_blocks(L), kReduceBlock, 0, st>>>((const typename S::T*)f, L, bc,
                                                                   partials, counter, out);
        return cudaGetLastError();
    });
}

cudaError_t launch_velocity_change(int prec, const void* f, const DevLattice& L, const BcState* bc, double* u_ref,
                                   double* partials, unsigned* counter, MonitorOut* out, cudaStream_t st) {
    return dispatch(prec, [&](auto s) {
        using S = decltype(s);
        k_velocity_change<S><<<monitor_blocks(L), kReduceBlock, 0, st>>>((const typename S::T*)f, L, bc, u_ref,
                                                                         partials, counter, out);
        return cudaGetLastError();
    });
}

cudaError_t launch_reencode(int prec, void* f, const DevLattice& L, BcState* bc, int e, int slot,
                            cudaStream_t st) {
    return dispatch(prec, [&](auto s) {
        using S = decltype(s);
        if constexpr (S::kRef) {
            k_reencode<S><<<blocks_for(L.n, 256), 256, 0, st>>>((typename S::T*)f, L, bc, e, slot);
            return cudaGetLastError();
        } else {
            return cudaSuccess;
        }
    });
}

cudaError_t launch_export(int prec, const void* f, const DevLattice& L, const BcState* bc, void* rho, void* ux,
                          void* uy, void* uz, int out_double, cudaStream_t st) {
    return dispatch(prec, [&](auto s) {
        using S = decltype(s);
        if (out_double)
            k_export<S, double><<<blocks_for(L.n, 256), 256, 0, st>>>(
                (const typename S::T*)f, L, bc, (double*)rho, (double*)ux, (double*)uy, (double*)uz);
        else
            k_export<S, float><<<blocks_for(L.n, 256), 256, 0, st>>>(
                (const typename S::T*)f, L, bc, (float*)rho, (float*)ux, (float*)uy, (float*)uz);
        return cudaGetLastError();
    });
}

cudaError_t launch_init_eq(int prec, void* f, const DevLattice& L, const BcState* bc, const double* rho,
                           const double* ux, const double* uy, const double* uz, cudaStream_t st) {
    return dispatch(prec, [&](auto s) {
        using S = decltype(s);
        k_init_eq<S><<<blocks_for(L.n, 256), 256, 0, st>>>((typename S::T*)f, L, bc, rho, ux, uy, uz);
        return cudaGetLastError();
    });
}

cudaError_t launch_encode(int prec, void* f, const DevLattice& L, const BcState* bc, const double* d,
                          cudaStream_t st) {
    return dispatch(prec, [&](auto s) {
        using S = decltype(s);
        k_encode<S><<<blocks_for(L.n, 256), 256, 0, st>>>((typename S::T*)f, L, bc, d);
        return cudaGetLastError();
    });
}

cudaError_t launch_decode(int prec, const void* f, const DevLattice& L, const BcState* bc, double* d,
                          cudaStream_t st) {
    return dispatch(prec, [&](auto s) {
        using S = decltype(s);
        k_decode<S><<<blocks_for(L.n, 256), 256, 0, st>>>((const typename S::T*)f, L, bc, d);
        return cudaGetLastError();
    });
}

cudaError_t launch_aa_step(int prec, void* f, int odd, int slot, const DevLattice& L, Relax r, BcState* bc,
                           double* partials, cudaStream_t st) {
    return dispatch(prec, [&](auto s) {
        using S = decltype(s);
        using M = typename S::M;
        {
            AAPtrs<typename S::T> F;
            for (int q = 0; q < 19; ++q) F.row[q] = (typename S::T*)f + (int64_t)q * L.ns;
            // every element offset of the buffer in 32 bits; the environment variable
            // GB300_LBM_AA_ADDR64 forces the id-grid form with 64-bit addresses (tests)
            const bool off32 = 19 * (uint64_t)L.ns <= 0xFFFFFFFFull && !std::getenv("GB300_LBM_AA_ADDR64");
            const bool win = L.win && off32;
            const unsigned nb = blocks_for(L.n, kBlock);
            const auto rates = make_rates<M>(r.sp, r.sm);
            if constexpr (sizeof(M) == 8) {
                if (win && L.n < kSmallNodes) {
                    const unsigned nbs = blocks_for(L.n, kSmallBlock);
                    if (odd)
                        k_step_aa<S, true, kWindows, kSmallBlock, false><<<nbs, kSmallBlock, 0, st>>>(F, slot, L, rates, bc, partials);
                    else
                        k_step_aa<S, false, kGrid64, kSmallBlock, false><<<nbs, kSmallBlock, 0, st>>>(F, slot, L, rates, bc, partials);
                    return cudaGetLastError();
                }
            }
            return with_parts<M>(L, [&](auto tiles) {
                constexpr bool TILES = decltype(tiles)::value;
                if constexpr (S::kRef) {
                    if (win) {
                        if (odd)
                            k_aa_odd_pair<S, TILES><<<nb, kPair, 0, st>>>((typename S::T*)f, slot, L, rates, bc, partials);
                        else
                            k_aa_even_pair<S, TILES><<<nb, kPair, 0, st>>>(F, slot, L, rates, bc, partials);
                        return fold_parts<kPair, TILES>(L, slot, partials, kBlock, st);
                    }
                } else if (odd && win) {
                    k_step_aa<S, true, kWindows, kBlock, TILES><<<nb, kBlock, 0, st>>>(F, slot, L, rates, bc, partials);
                    return fold_parts<kBlock, TILES>(L, slot, partials, kBlock, st);
                }
                if (odd && off32) k_step_aa<S, true, kGrid32, kBlock, TILES><<<nb, kBlock, 0, st>>>(F, slot, L, rates, bc, partials);
                else if (odd) k_step_aa<S, true, kGrid64, kBlock, TILES><<<nb, kBlock, 0, st>>>(F, slot, L, rates, bc, partials);
                else k_step_aa<S, false, kGrid64, kBlock, TILES><<<nb, kBlock, 0, st>>>(F, slot, L, rates, bc, partials);
                return fold_parts<kBlock, TILES>(L, slot, partials, kBlock, st);
            });
        }
    });
}

cudaError_t launch_aa_swap(int prec, void* f, const DevLattice& L, cudaStream_t st) {
    return dispatch(prec, [&](auto s) {
        using S = decltype(s);
        k_aa_swap<typename S::T><<<blocks_for(L.n, 256), 256, 0, st>>>((typename S::T*)f, L.n, L.ns);
        return cudaGetLastError();
    });
}

cudaError_t launch_aa_unstream(int prec, void* f, const DevLattice& L, const BcState* bc, cudaStream_t st) {
    return dispatch(prec, [&](auto s) {
        using S = decltype(s);
        k_aa_unstream<S><<<blocks_for(L.n, 256), 256, 0, st>>>((typename S::T*)f, L, bc);
        return cudaGetLastError();
    });
}

cudaError_t configure_step(int prec, int variant, const DevLattice& L, StepConfig* cfg) {
    cfg->variant = variant;
    cfg->grid = 0;
    if (variant == 0) return cudaSuccess;
    return dispatch(prec, [&](auto s) {
        using S = decltype(s);
        if (variant == 1) return config_async_t<S, 256>(&cfg->grid, L);
        if (variant == 2) return config_async_t<S, 128>(&cfg->grid, L);
        return cudaErrorInvalidValue;
    });
}

cudaError_t launch_step_cfg(int prec, const StepConfig& cfg, const void* fin, void* fout, int slot,
                            const DevLattice& L, Relax r, BcState* bc, double* partials,
                            cudaStream_t st) {
    if (cfg.variant == 0) return launch_step(prec, fin, fout, slot, L, r, bc, partials, st);
    return dispatch(prec, [&](auto s) {
        using S = decltype(s);
        if (cfg.variant == 1)
            return launch_async_t<S, 256>(fin, fout, slot, L, r, bc, partials, st, cfg.grid);
        if (cfg.variant == 2)
            return launch_async_t<S, 128>(fin, fout, slot, L, r, bc, partials, st, cfg.grid);
        return cudaErrorInvalidValue;
    });
}

}  // namespace lbm
