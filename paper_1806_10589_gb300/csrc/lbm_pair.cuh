// Two pore nodes per thread: FP32 arithmetic on packed pairs (add / mul / fma
// .f32x2, sm_100 and later) and the 16-bit codecs on two neighbouring slots.
//
// The 16-bit steps are bound by the instructions they issue, not by memory: one
// FP16-dev node took 736 (gather-scatter launch) and 470 (node-local launch)
// instructions per node at 33 % and 49 % of the DRAM rate.  A thread that owns
// the slots i and i + 1 (i even) reads and writes both with one 4-byte access
// wherever a slot is its own, rounds both with one conversion, and issues one
// packed instruction for two nodes' arithmetic.  Measured on a 251x243x262 pack,
// FP16-dev, one -> two nodes per thread: node-local launch 112 -> 77 us (470 -> 260
// instructions per node, 0.89 of the copy rate), gather-scatter launch 168 -> 144 us
// (736 -> 540); two-buffer step of a 157x149x171 pack, BF16-dev, 39.0 -> 33.1 us.
//
// The packed operations round each half exactly as the scalar ones do, and the
// collision below is spelled out operation by operation, so the states are bitwise
// those of one node per thread (tests/test_gpu_windows.py).
#pragma once

#include <type_traits>

#include "lbm_device.cuh"

namespace lbm {

struct F2 {
    unsigned long long v;  // low half: node i, high half: node i + 1
};
__device__ __forceinline__ F2 f2(float lo, float hi) {
    F2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ F2 f2(float a) { return f2(a, a); }
__device__ __forceinline__ void split(F2 a, float& lo, float& hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(a.v));
}
__device__ __forceinline__ F2 vadd(F2 a, F2 b) {
    F2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ F2 vmul(F2 a, F2 b) {
    F2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ F2 vfma(F2 a, F2 b, F2 c) {
    F2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
    return r;
}
// a - b as one rounding of a + (-1) b: there is no packed subtraction
__device__ __forceinline__ F2 vsub(F2 a, F2 b) { return vfma(b, f2(-1.0f), a); }

// The FP32 collision of lbm_device.cuh for two nodes, each half rounded as the
// scalar kernels round it (operation by operation what the compiler makes of
// collide there); xi.u takes only the components a direction has.
template <int A>
__device__ __forceinline__ void relax_pair2(F2* d, const F2* m, F2 drho, F2 ux, F2 uy, F2 uz, F2 uu, F2 nsp, F2 sm,
                                            F2 nsm) {
    constexpr int B = A + 1;
    F2 xu;
    if constexpr (A == 1) xu = ux;
    else if constexpr (A == 3) xu = uy;
    else if constexpr (A == 5) xu = uz;
    else if constexpr (A == 7) xu = vadd(ux, uy);
    else if constexpr (A == 9) xu = vsub(ux, uy);
    else if constexpr (A == 11) xu = vadd(ux, uz);
    else if constexpr (A == 13) xu = vsub(ux, uz);
    else if constexpr (A == 15) xu = vadd(uy, uz);
    else xu = vsub(uy, uz);
    constexpr float w = float(wq(A));
    const F2 h = f2(0.5f);
    const F2 y = vfma(f2(-1.5f), uu, vfma(vmul(f2(4.5f), xu), xu, drho));
    const F2 p = vfma(h, vadd(d[A], d[B]), vmul(f2(-w), y));            // f+ - feq+
    const F2 q = vfma(h, m[A / 2], vmul(f2(-(w * 3.0f)), xu));          // f- - feq-
    d[A] = vfma(nsm, q, vfma(nsp, p, d[A]));
    d[B] = vfma(sm, q, vfma(nsp, p, d[B]));
}
// XX: u.u starts from the rounded u_x^2, otherwise from u_y^2.  The two-buffer
// steps use the first, the in-place steps the second, as their scalar kernels do
// (a 16-bit state follows every last bit).
template <bool XX>
__device__ __forceinline__ void collide2(F2* d, float sp_, float sm_) {
    const F2 nsp = f2(-sp_), sm = f2(sm_), nsm = f2(-sm_);
    F2 m[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) m[k] = vsub(d[2 * k + 1], d[2 * k + 2]);
    F2 drho = vadd(vadd(vadd(d[0], d[1]), vadd(d[2], d[3])), vadd(vadd(d[4], d[5]), vadd(d[6], d[7])));
    drho = vadd(drho, vadd(vadd(d[8], d[9]), vadd(d[10], d[11])));
    drho = vadd(drho, vadd(vadd(d[12], d[13]), vadd(d[14], d[15])));
    drho = vadd(drho, vadd(vadd(d[16], d[17]), d[18]));
    const F2 ux = vadd(vadd(vadd(vadd(m[0], m[3]), m[4]), m[5]), m[6]);
    const F2 uy = vadd(vadd(vsub(vadd(m[1], m[3]), m[4]), m[7]), m[8]);
    const F2 uz = vsub(vadd(vsub(vadd(m[2], m[5]), m[6]), m[7]), m[8]);
    const F2 uu = vfma(uz, uz, XX ? vfma(uy, uy, vmul(ux, ux)) : vfma(ux, ux, vmul(uy, uy)));
    const F2 t = vfma(f2(-1.5f), uu, drho);
    d[0] = vfma(nsp, vfma(f2(-float(wq(0))), t, d[0]), d[0]);
    relax_pair2<1>(d, m, drho, ux, uy, uz, uu, nsp, sm, nsm);
    relax_pair2<3>(d, m, drho, ux, uy, uz, uu, nsp, sm, nsm);
    relax_pair2<5>(d, m, drho, ux, uy, uz, uu, nsp, sm, nsm);
    relax_pair2<7>(d, m, drho, ux, uy, uz, uu, nsp, sm, nsm);
    relax_pair2<9>(d, m, drho, ux, uy, uz, uu, nsp, sm, nsm);
    relax_pair2<11>(d, m, drho, ux, uy, uz, uu, nsp, sm, nsm);
    relax_pair2<13>(d, m, drho, ux, uy, uz, uu, nsp, sm, nsm);
    relax_pair2<15>(d, m, drho, ux, uy, uz, uu, nsp, sm, nsm);
    relax_pair2<17>(d, m, drho, ux, uy, uz, uu, nsp, sm, nsm);
}

// ------------------------------------------------------ 16-bit pair codec ---
// Two stored values (low half: node i) as floats.
template <class S>
__device__ __forceinline__ F2 widen2(uint32_t v) {
    if constexpr (std::is_same<typename S::T, __half>::value) {
        const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&v));
        return f2(f.x, f.y);
    } else {
        return f2(__uint_as_float(v << 16), __uint_as_float(v & 0xFFFF0000u));
    }
}
template <class S>
__device__ __forceinline__ F2 widen2(typename S::T a, typename S::T b) {
    if constexpr (std::is_same<typename S::T, __half>::value) return f2(__half2float(a), __half2float(b));
    else return f2(__bfloat162float(a), __bfloat162float(b));
}
// dec of lbm_device.cuh for both nodes; wr = w r.
template <class S, int Q>
__device__ __forceinline__ F2 dec2(F2 v, F2 wr) {
    return vfma(v, f2(float(wq(Q) / 1024.0)), wr);
}
// enc_sr of both nodes, node i in the low half; nr = -1024 r.  u holds node i's
// random field in its low 16 bits and node i + 1's in the high ones.
template <class S, int Q>
__device__ __forceinline__ uint32_t enc_sr2(F2 d, F2 nr, uint32_t u) {
    float lo, hi;
    split(vfma(d, f2(float(1024.0 / wq(Q))), nr), lo, hi);
    return S::cvt_rs(hi, lo, u);
}
// Random fields of nodes i and j (sr_key of each, one half each).
__device__ __forceinline__ uint32_t sr_key2(uint32_t seed, uint32_t i, uint32_t j) {
    return __byte_perm(sr_hash(seed ^ i), sr_hash(seed ^ j), 0x7632);
}

}  // namespace lbm
