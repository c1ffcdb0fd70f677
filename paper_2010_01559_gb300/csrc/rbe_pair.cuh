// rbe_pair.cuh -- the real-space pair terms of the mixed path (Eq. force,
// second term, truncated at r_c; Eq. Ljpotential with r_off = 0), shared by the
// real-space kernels (rbe_real.cu) and the fused structure-factor + list-pass
// launch (rbe_fourier.cu).
#pragma once

#include "rbe_internal.cuh"

namespace rbe {

constexpr int kPartFourier = 1, kPartReal = 2, kPartLJ = 4;

__device__ __forceinline__ int wrapc(int c, int n) { return c < 0 ? c + n : (c >= n ? c - n : c); }

// The 27 neighbour cells as 9 rows (dz, dy) of three x-adjacent cells.  Cells
// are numbered x fastest, so a row is one contiguous range of the sorted
// particles unless it wraps around the box edge; then it is two ranges.
__device__ __forceinline__ void row_ranges(const int* __restrict__ cs, int base, int cx, int ncd,
                                           int& s0, int& e0, int& s1, int& e1) {
    if (ncd < 3) {                                  // one cell per edge: the whole row once
        s0 = __ldg(cs + base); e0 = __ldg(cs + base + ncd); s1 = 0; e1 = 0;
    } else if (cx > 0 && cx < ncd - 1) {
        s0 = __ldg(cs + base + cx - 1); e0 = __ldg(cs + base + cx + 2); s1 = 0; e1 = 0;
    } else if (cx == 0) {
        s0 = __ldg(cs + base); e0 = __ldg(cs + base + 2);
        s1 = __ldg(cs + base + ncd - 1); e1 = __ldg(cs + base + ncd);
    } else {
        s0 = __ldg(cs + base + ncd - 2); e0 = __ldg(cs + base + ncd);
        s1 = __ldg(cs + base); e1 = __ldg(cs + base + 1);
    }
}

// Deterministic block sum of two doubles (fixed shuffle tree, then warps in
// order); the result is valid in thread 0.
__device__ __forceinline__ double2 block_sum2_real(double a, double b) {
    __shared__ double sa[32], sb[32];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        a += __shfl_down_sync(0xffffffffu, a, o);
        b += __shfl_down_sync(0xffffffffu, b, o);
    }
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (lane == 0) { sa[w] = a; sb[w] = b; }
    __syncthreads();
    double2 r = make_double2(0.0, 0.0);
    if (threadIdx.x == 0) {
        const int nw = (blockDim.x + 31) >> 5;
        for (int k = 0; k < nw; ++k) { r.x += sa[k]; r.y += sb[k]; }
    }
    return r;
}

struct PairAcc {
    float fx, fy, fz, phr, ec, elj, wc, wlj;     // wc, wlj: half the pair virials r.F
};

// erfc(x) for x >= 0 given e = exp(-x^2): the rational approximation of
// Abramowitz & Stegun, Handbook of Mathematical Functions, formula 7.1.26
// (after Hastings), |error| <= 1.5e-7.  It reuses the Gaussian the force needs
// anyway, so erfc costs one reciprocal and five FMAs.
__device__ __forceinline__ float erfc_as(float e, float x) {
    const float t = __fdividef(1.0f, fmaf(0.3275911f, x, 1.0f));
    float p = 1.061405429f;
    p = fmaf(p, t, -1.453152027f);
    p = fmaf(p, t, 1.421413741f);
    p = fmaf(p, t, -0.284496736f);
    p = fmaf(p, t, 0.254829592f);
    return p * t * e;
}

// Per-system constants of the pair terms, in registers.
struct PairConst {
    float rc2, lj_rc2, alpha, sa, two_sa_spi, lB, lj_s2, lj_eps, lj_shift;
    bool vir;                                   // accumulate the virials
};

// Pair terms for displacement r_ij = (dx, dy, dz), |r_ij|^2 = r2 > 0.
__device__ __forceinline__ void pair_terms(float dx, float dy, float dz, float r2, float qj,
                                           float lbqi, const PairConst& k, PairAcc& acc) {
    const float inv_r = rsqrtf(r2);
    if (r2 < k.rc2) {
        const float x = k.sa * (r2 * inv_r);
        const float ex = __expf(-k.alpha * r2);                  // exp(-x^2)
        const float pot = erfc_as(ex, x) * inv_r;                 // erfc(sqrt(a) r) / r
        const float g_over_r = fmaf(k.two_sa_spi, ex, pot) * inv_r * inv_r;   // G(r) / r
        const float s_ = -lbqi * qj * g_over_r;
        acc.fx = fmaf(s_, dx, acc.fx);
        acc.fy = fmaf(s_, dy, acc.fy);
        acc.fz = fmaf(s_, dz, acc.fz);
        acc.phr = fmaf(k.lB * qj, pot, acc.phr);
        acc.ec = fmaf(0.5f * lbqi * qj, pot, acc.ec);
        // r.F of the pair: lB q_i q_j (erfc(sqrt(a) r)/r + 2 sqrt(a/pi) e^{-a r^2})
        if (k.vir) acc.wc = fmaf(0.5f * lbqi * qj, fmaf(k.two_sa_spi, ex, pot), acc.wc);
    }
    if (r2 < k.lj_rc2) {
        const float inv_r2 = inv_r * inv_r;
        const float sr2 = k.lj_s2 * inv_r2;
        const float sr6 = sr2 * sr2 * sr2;
        const float mag = 24.f * k.lj_eps * (2.f * sr6 * sr6 - sr6) * inv_r2;
        acc.fx = fmaf(-mag, dx, acc.fx);
        acc.fy = fmaf(-mag, dy, acc.fy);
        acc.fz = fmaf(-mag, dz, acc.fz);
        acc.elj += 0.5f * (4.f * k.lj_eps * (sr6 * sr6 - sr6) + k.lj_shift);
        if (k.vir) acc.wlj = fmaf(0.5f * mag, r2, acc.wlj);   // r.F = 24 eps (2 (s/r)^12 - (s/r)^6)
    }
}

// Pair terms from two fixed-point records: the displacement is the 32-bit
// difference of the coordinates, which is the minimum image (|r_ij| < L / 2),
// rounded once to FP32 and scaled to length units.  A zero displacement (the
// particle itself) adds nothing.
__device__ __forceinline__ void pair_fixed(const uint4& si, const uint4& sj, float Lu,
                                           float lbqi, const PairConst& kc, PairAcc& acc) {
    const float dx = (float)(int32_t)(sj.x - si.x) * Lu;
    const float dy = (float)(int32_t)(sj.y - si.y) * Lu;
    const float dz = (float)(int32_t)(sj.z - si.z) * Lu;
    const float r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
    if (r2 > 0.f) pair_terms(dx, dy, dz, r2, __uint_as_float(sj.w), lbqi, kc, acc);
}

// ---- two pairs at a time (MD steps: the force alone)
// The list pass of an MD step is bound by instruction issue: with two pairs per
// packed FP32 instruction a pair takes about 32 instructions instead of 70.  Same
// formulas as pair_terms (erfc as in erfc_as) from the same displacements and r^2
// to the last bit, so that a pair at a cutoff falls on the same side (the truncated
// force jumps by 7e-5 there at the parameters of the benchmark).  Pairs beyond the
// cutoff and the particle itself (a zero displacement) get the factor 0.
struct Pair2Acc {
    f32x2 x, y, z;                               // Coulomb / (-lB q_i), the two pairs' sums apart
    float lx, ly, lz;                            // Lennard-Jones
};

__device__ __forceinline__ void pair2_fixed(const uint4& si, const uint4& sa, const uint4& sb,
                                            const SysDev& S, Pair2Acc& acc) {
    const f32x2 Lu = pack2(S.L_over_2_32, S.L_over_2_32);
    const f32x2 dx = mul2(pack2((float)(int32_t)(sa.x - si.x), (float)(int32_t)(sb.x - si.x)), Lu);
    const f32x2 dy = mul2(pack2((float)(int32_t)(sa.y - si.y), (float)(int32_t)(sb.y - si.y)), Lu);
    const f32x2 dz = mul2(pack2((float)(int32_t)(sa.z - si.z), (float)(int32_t)(sb.z - si.z)), Lu);
    const f32x2 r2 = fma2(dx, dx, fma2(dy, dy, mul2(dz, dz)));
    const float2 q2 = unpack2(r2);
    const bool ina = q2.x < S.f_rc2 && q2.x > 0.f, inb = q2.y < S.f_rc2 && q2.y > 0.f;
    if (!(ina || inb)) return;
    const float ia = rsqrtf(q2.x), ib = rsqrtf(q2.y);
    const f32x2 inv = pack2(ia, ib), inv2 = mul2(inv, inv);
    // t = 1 / (1 + 0.3275911 x), x = sqrt(alpha) r
    const float2 den = unpack2(
        fma2(mul2(r2, inv), pack2(S.f_erfc_x, S.f_erfc_x), pack2(1.f, 1.f)));
    const f32x2 t = pack2(__fdividef(1.0f, den.x), __fdividef(1.0f, den.y));
    const float2 e2 = unpack2(mul2(r2, pack2(S.f_gauss_ex2, S.f_gauss_ex2)));
    const f32x2 ex = pack2(exp2f(e2.x), exp2f(e2.y));            // exp(-alpha r^2)
    f32x2 p = fma2(t, pack2(1.061405429f, 1.061405429f), pack2(-1.453152027f, -1.453152027f));
    p = fma2(p, t, pack2(1.421413741f, 1.421413741f));
    p = fma2(p, t, pack2(-0.284496736f, -0.284496736f));
    p = fma2(p, t, pack2(0.254829592f, 0.254829592f));
    // q_j (erfc / r + 2 sqrt(alpha / pi) exp(-alpha r^2)) / r^2
    const f32x2 g = mul2(fma2(mul2(p, t), inv, pack2(S.f_two_sa_spi, S.f_two_sa_spi)),
                         mul2(ex, inv2));
    const float2 f =
        unpack2(mul2(g, pack2(__uint_as_float(sa.w), __uint_as_float(sb.w))));
    const f32x2 s = pack2(ina ? f.x : 0.f, inb ? f.y : 0.f);
    acc.x = fma2(s, dx, acc.x);
    acc.y = fma2(s, dy, acc.y);
    acc.z = fma2(s, dz, acc.z);
    if (fminf(q2.x, q2.y) < S.f_lj_rc2_on) {     // a few pairs per particle, one at a time
        const float2 x = unpack2(dx), y = unpack2(dy), z = unpack2(dz);
        auto lj = [&](float r2s, float inv_r, float ux, float uy, float uz) {
            if (r2s < S.f_lj_rc2_on && r2s > 0.f) {
                const float inv_r2 = inv_r * inv_r;
                const float sr2 = S.f_lj_sigma2 * inv_r2;
                const float sr6 = sr2 * sr2 * sr2;
                const float mag = 24.f * S.f_lj_eps * (2.f * sr6 * sr6 - sr6) * inv_r2;
                acc.lx = fmaf(-mag, ux, acc.lx);
                acc.ly = fmaf(-mag, uy, acc.ly);
                acc.lz = fmaf(-mag, uz, acc.lz);
            }
        };
        lj(q2.x, ia, x.x, y.x, z.x);
        lj(q2.y, ib, x.y, y.y, z.y);
    }
}

// The particle's force from its sums.
__device__ __forceinline__ float3 pair2_force(const Pair2Acc& a, const uint4& si,
                                              const SysDev& S) {
    const float2 x = unpack2(a.x), y = unpack2(a.y), z = unpack2(a.z);
    const float c = -S.f_lB * __uint_as_float(si.w);
    return make_float3(fmaf(c, x.x + x.y, a.lx), fmaf(c, y.x + y.y, a.ly),
                       fmaf(c, z.x + z.y, a.lz));
}

}  // namespace rbe
