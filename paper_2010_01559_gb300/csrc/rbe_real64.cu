// rbe_real64.cu -- real-space Coulomb, shifted Lennard-Jones, the assembly of
// the total force / dE/dq and the MD update on the FP64 path (formulas:
// rbe_real.cu), over the cell list.
//
// What bounds it: the FP64 pipe (two lanes per SM and clock).  The pair terms
// cost about a hundred FP64 instructions, and only about one candidate of the
// 27 cells in ten is within the cutoff, so a warp that tested and evaluated in
// one loop spent them on nearly every candidate.  Here G lanes per particle
// first test the candidates' 32-bit fixed-point records (integer and FP32 work
// only, with a margin that keeps every pair the FP64 test would) and collect
// the survivors' indices in shared memory; then the G lanes evaluate them
// densely in FP64, which applies the cutoffs themselves.  erfc is
// e^{-x^2} erfcx(x) with the Gaussian the force needs anyway, and one
// reciprocal square root serves every division.
//
// erfcx is a polynomial of about 30 terms for the usual cutoffs (alpha r_c^2 <= 16,
// rbe_poly64.cuh), the library's beyond.  Every factor of a term keeps its relative
// accuracy, so that a pair near the cutoff, where erfc has fallen by up to seven
// orders, is as good as a close one (1 / r minus a polynomial of erf(x) / x takes a
// term less, but is good to 1e-16 / r only).
//
// Below some 10^4 particles the latency of an FP64 instruction (about a hundred
// cycles) and of dependent loads bounds it instead: the lanes fetch the bounds of
// a particle's nine neighbour rows side by side and walk them as one range with
// kCand candidates in flight each, evaluate two listed pairs at a time, and a warp
// of its own fetches what the closing update needs and draws the thermostat's
// noise meanwhile.
// Measured (events around the kernel, launch included): N = 1000, r_c = 5, MD
// step: 298 -> 27 us; N = 8001, r_c = 6, forces with energy and dE/dq: 930 ->
// 139 us.  Error against an 80-bit evaluation, now / before, geometric means over 40
// systems of 400 to 19124: forces 0.88, dE/dq 0.49.
#include <cmath>

#include "rbe_internal.cuh"
#include "rbe_pair.cuh"

namespace rbe {

constexpr int kHitCap = 96;           // listed candidates per particle before a flush
constexpr int kCand = 2;              // candidates in flight per lane
constexpr int kReal64Threads = kBlockP + 32;

struct Pair64 {
    double fx, fy, fz, phr, ec, elj, wc, wlj;
};

struct Const64 {
    double rc2, lj_rc2, lj_sigma2, lj_eps, lj_shift, alpha, sqrt_alpha, two_sa_spi, lB, lBqi;
    double L, halfL, t_scale;
    double far2;                         // r_c^2
    const double* poly;                  // highest power first
    int npoly;
};

__device__ __forceinline__ double min_image(double d, const Const64& c) {
    return fabs(d) > c.halfL ? d - copysign(c.L, d) : d;
}

// How a launch's systems get erfcx: a system alone by its polynomial or, beyond its
// range, the library's function; a batch of either kind alone likewise, a batch of
// both by each block's own system, so that no system's results depend on the others.
enum { kErfcxLib, kErfcxPoly, kErfcxEach };             // RealArgs.poly64_form

// EN: also the potential, energies and virials.  Without branches on the Coulomb
// part, so that two calls in a row overlap; pj of a pair that is not one (live
// false) is any record, and its distance stands at r_c: within the polynomials'
// range in any unit of length (a charge of 0 does not cancel an infinity).
template <bool EN, int POLY>
__device__ __forceinline__ void pair64(const double4& pi, const double4& pj, bool live,
                                       const Const64& c, Pair64& a) {
    const double dx = min_image(pj.x - pi.x, c), dy = min_image(pj.y - pi.y, c),
                 dz = min_image(pj.z - pi.z, c);
    const double r2 = live ? dx * dx + dy * dy + dz * dz : c.far2;
    const bool in = live && r2 < c.rc2, lj = live && r2 < c.lj_rc2;
    // the square of rsqrt's last-place error would enter the Lennard-Jones force
    // seven times: one Newton step makes 1 / r^2 good to its rounding
    const double inv_r = rsqrt(r2), sq = inv_r * inv_r;
    const double inv_r2 = fma(sq, fma(-r2, sq, 1.0), sq);
    const double r = r2 * inv_r;
    double ecx;                          // erfcx(sqrt(alpha) r)
    if (POLY == kErfcxPoly || (POLY == kErfcxEach && c.npoly > 0)) {
        const double t = fma(r, c.t_scale, -1.0);
        ecx = c.poly[0];
#pragma unroll 4
        for (int k = 1; k < c.npoly; ++k) ecx = fma(ecx, t, c.poly[k]);
    } else {
        ecx = erfcx(c.sqrt_alpha * r);
    }
    const double ex = exp(-c.alpha * r2);
    const double pot = ex * ecx * inv_r;                       // erfc / r
    const double g = fma(c.two_sa_spi, ex, pot);               // + 2 sqrt(alpha / pi) e^{-alpha r^2}
    const double qq = in ? c.lBqi * pj.w : 0.0;
    double s = -qq * g * inv_r2;
    if constexpr (EN) {
        a.phr = fma(in ? c.lB * pj.w : 0.0, pot, a.phr);
        a.ec = fma(0.5 * qq, pot, a.ec);
        a.wc = fma(0.5 * qq, g, a.wc);
    }
    if (lj) {
        const double sr2 = c.lj_sigma2 * inv_r2;
        const double sr6 = sr2 * sr2 * sr2;
        const double mag = 24.0 * c.lj_eps * fma(2.0 * sr6, sr6, -sr6) * inv_r2;
        s -= mag;
        if constexpr (EN) {
            a.elj += 0.5 * fma(4.0 * c.lj_eps, fma(sr6, sr6, -sr6), c.lj_shift);
            a.wlj = fma(0.5 * mag, r2, a.wlj);
        }
    }
    a.fx = fma(s, dx, a.fx);
    a.fy = fma(s, dy, a.fy);
    a.fz = fma(s, dz, a.fz);
}

// r wrapped into [0, L): inside the box floor(r / L) is 0, so the division is
// only taken outside it
__device__ __forceinline__ double wrap_box(double r, double L) {
    return (r >= 0.0 && r < L) ? r : r - L * floor(r / L);
}

template <int G, bool ONE, bool EN, int POLY>
__global__ void __launch_bounds__(kReal64Threads)
k_real_f64(const __grid_constant__ RealArgs a) {
    constexpr int T = kBlockP / G;               // particles per block
    __shared__ int s_hit[T][kHitCap];
    __shared__ int s_pre[T][10], s_s0[T][9], s_n0[T][9], s_s1[T][9];   // rows as one range
    __shared__ double4 s_f[T];
    __shared__ double s_poly[POLY ? kPoly64 : 1];        // highest power first
    // block (x, y): particles T y .. T y + T - 1 of tile x (kBlockP particles)
    Tile tl = tile_of<ONE>(a.w);
    tl.first += (int)blockIdx.y * T;
    tl.count = max(0, min(T, tl.count - (int)blockIdx.y * T));
    const int blk = blockIdx.x * G + blockIdx.y;         // its energy / virial partials
    const SysDev& S = sys_of<ONE>(a.w, tl.sys);
    const bool do_real = (a.parts & kPartReal) != 0;
    const bool do_lj = (a.parts & kPartLJ) != 0 && S.lj_eps != 0.0;
    Pair64 acc{0, 0, 0, 0, 0, 0, 0, 0};
    bool owner = false;
    int npoly = 0;
    if constexpr (POLY) {
        const Poly64& P = a.poly64[tl.sys];
        npoly = P.n;
        for (int k = threadIdx.x; k < npoly; k += kReal64Threads)
            s_poly[npoly - 1 - k] = P.c[k];
        __syncthreads();
    }
    if (threadIdx.x < kBlockP) {
        // ---- the pair sums: G lanes per particle
        const int g = threadIdx.x % G, t = threadIdx.x / G;
        const bool active = t < tl.count;
        owner = active && g == 0;
        const int i = tl.first + (tl.count > 0 ? min(t, tl.count - 1) : 0);
        if (tl.count > 0 && (do_real || do_lj)) {
            const double4 pi = a.spos64[i];
            Const64 c;
            c.far2 = S.r_c * S.r_c;
            c.rc2 = do_real ? c.far2 : 0.0;
            c.lj_rc2 = do_lj ? S.lj_rcut2 : 0.0;
            c.lj_sigma2 = S.lj_sigma2;
            c.lj_eps = S.lj_eps;
            c.lj_shift = S.lj_shift;
            c.alpha = S.alpha;
            c.sqrt_alpha = S.sqrt_alpha;
            c.two_sa_spi = 2.0 * S.sqrt_alpha * 0.5641895835477563;      // 1 / sqrt(pi)
            c.lB = S.lB;
            c.lBqi = S.lB * pi.w;
            c.L = S.L;
            c.halfL = 0.5 * S.L;
            c.poly = s_poly;
            c.npoly = npoly;
            c.t_scale = POLY ? a.poly64[tl.sys].scale : 0.0;
            // the candidate test: fixed-point records are within a unit of the FP64
            // positions (a displacement within two, whatever the box measures in
            // cutoffs), and the cutoff widened by 5e-5 covers the FP32 rounding
            const float Lu = S.L_over_2_32;
            const float cut = fmaf(sqrtf(fmaxf(do_real ? S.f_rc2 : 0.f,
                                               do_lj ? S.f_lj_rc2 : 0.f)), 1.00005f, 2.f * Lu);
            const float cut2 = cut * cut;
            const uint4 si = a.spos[i];
            const unsigned lane = threadIdx.x & 31;
            const unsigned gmask = G == 32 ? 0xffffffffu : ((1u << G) - 1u) << (lane & ~(G - 1u));
            const unsigned below = gmask & ((1u << lane) - 1u);
            int* hit = s_hit[t];
            int nhit = 0;                        // the same in every lane of the group
            auto dense = [&](int k0, int n) {    // two listed pairs per lane from k0 on
                const int ka = k0 + g, kb = ka + G;
                const bool la = ka < n, lb = kb < n;
                const double4 pa = a.spos64[la ? hit[ka] : i], pb = a.spos64[lb ? hit[kb] : i];
                pair64<EN, POLY>(pi, pa, la, c, acc);
                pair64<EN, POLY>(pi, pb, lb, c, acc);
            };
            const int ncd = S.ncd;
            auto cell = [&](double w) {
                const double u = w * S.invL * (double)ncd;
                return (u >= 0.0 && u < (double)ncd) ? (int)u : 0;
            };
            if (active) {
                const int cx = cell(pi.x), cy = cell(pi.y), cz = cell(pi.z);
                const int nrow = ncd < 3 ? 1 : 9;         // one cell: every pair once
                for (int r = g; r < nrow; r += G) {
                    const int dz = ncd < 3 ? 0 : r / 3 - 1, dy = ncd < 3 ? 0 : r % 3 - 1;
                    const int zz = wrapc(cz + dz, ncd), yy = wrapc(cy + dy, ncd);
                    int b0, e0, b1, e1;
                    row_ranges(a.cell_start, S.off_c + (zz * ncd + yy) * ncd, cx, ncd, b0, e0, b1,
                               e1);
                    s_s0[t][r] = b0;
                    s_n0[t][r] = e0 - b0;
                    s_s1[t][r] = b1;
                    s_pre[t][r + 1] = (e0 - b0) + (e1 - b1);
                }
                __syncwarp(gmask);
                if (g == 0) {
                    int run = 0;
                    s_pre[t][0] = 0;
                    for (int r = 1; r <= nrow; ++r) s_pre[t][r] = run += s_pre[t][r];
                }
                __syncwarp(gmask);
                const int tot = s_pre[t][nrow];
                int r = 0;                                // row of this lane's candidate
                for (int k0 = 0; k0 < tot; k0 += G * kCand) {
                    uint4 sj[kCand];
                    int jj[kCand];
#pragma unroll
                    for (int u = 0; u < kCand; ++u) {
                        const int k = k0 + u * G + g;
                        jj[u] = i;                        // not a pair
                        if (k < tot) {
                            while (k >= s_pre[t][r + 1]) ++r;
                            const int o = k - s_pre[t][r], n0 = s_n0[t][r];
                            jj[u] = o < n0 ? s_s0[t][r] + o : s_s1[t][r] + (o - n0);
                            if (!RBE_IN_BOUNDS(jj[u], a.nbr_stride, a.err)) jj[u] = i;
                        }
                        sj[u] = __ldg(a.spos + jj[u]);
                    }
#pragma unroll
                    for (int u = 0; u < kCand; ++u) {
                        const float dx = (float)(int32_t)(sj[u].x - si.x) * Lu;
                        const float dyy = (float)(int32_t)(sj[u].y - si.y) * Lu;
                        const float dzz = (float)(int32_t)(sj[u].z - si.z) * Lu;
                        const bool near =
                            fmaf(dx, dx, fmaf(dyy, dyy, dzz * dzz)) < cut2 && jj[u] != i;
                        const unsigned m = __ballot_sync(gmask, near) & gmask;
                        if (near) hit[nhit + __popc(m & below)] = jj[u];
                        nhit += __popc(m);
                        if (nhit > kHitCap - G) {         // crowded: evaluate what is listed
                            __syncwarp(gmask);
                            for (int k = 0; k < nhit; k += 2 * G) dense(k, nhit);
                            __syncwarp(gmask);
                            nhit = 0;
                        }
                    }
                }
            }
            __syncwarp();
            // dense rounds, the warp's groups together
            const int rounds =
                (int)__reduce_max_sync(0xffffffffu, (unsigned)(nhit + 2 * G - 1) / (2 * G));
            for (int q = 0; q < rounds; ++q) dense(q * 2 * G, nhit);
        }
#pragma unroll
        for (int o = G / 2; o > 0; o >>= 1) {
            acc.fx += __shfl_down_sync(0xffffffffu, acc.fx, o, G);
            acc.fy += __shfl_down_sync(0xffffffffu, acc.fy, o, G);
            acc.fz += __shfl_down_sync(0xffffffffu, acc.fz, o, G);
            if constexpr (EN) {
                acc.phr += __shfl_down_sync(0xffffffffu, acc.phr, o, G);
                acc.ec += __shfl_down_sync(0xffffffffu, acc.ec, o, G);
                acc.elj += __shfl_down_sync(0xffffffffu, acc.elj, o, G);
                acc.wc += __shfl_down_sync(0xffffffffu, acc.wc, o, G);
                acc.wlj += __shfl_down_sync(0xffffffffu, acc.wlj, o, G);
            }
        }
        if (owner) s_f[t] = make_double4(acc.fx, acc.fy, acc.fz, acc.phr);
    }
    // ---- the closing warp, a lane per particle: what does not depend on the sums
    const int tc = (int)threadIdx.x - kBlockP;
    bool closes = tc >= 0 && tc < tl.count;
    const bool nhm = a.md_pos64 && a.nh && S.thermostat == RBE_THERMO_NOSE_HOOVER;
    const bool andersen = S.thermostat == RBE_THERMO_ANDERSEN;
    int o = 0;
    double4 f = make_double4(0, 0, 0, 0), v = f, rp = f;
    double xi[3] = {0.0, 0.0, 0.0};
    bool coll = false;
    if (closes) {
        o = a.perm[tl.first + tc];
        if (!RBE_IN_BOUNDS(o, a.nbr_stride, a.err)) closes = false;
    }
    if (closes) {
        if (a.parts & kPartFourier) {
            f = a.fs64[o];
            if (a.phi_out64) {
                const double qs = (double)(long long)__ldcg(a.qsum_fx + tl.sys) / kQScale;
                f.w -= 2.0 * S.self_coef * a.spos64[tl.first + tc].w + S.bg_coef * qs;
            }
        } else {
            f.w = 0.0;
        }
        if (a.md_pos64) {
            v = a.md_vel64[o];
            rp = a.md_pos64[o];
            if (!nhm) {
                // Langevin: normals of the OU step; Andersen: collision word, then normals
                const uint64_t step = *a.cur_step;
                const uint2 key = make_uint2((uint32_t)S.seed, (uint32_t)(S.seed >> 32));
                const uint32_t pid = (uint32_t)(o - S.off_p);
                const uint4 cw =
                    philox4x32_10(make_uint4(pid, 0u, (uint32_t)step,
                                             (S.stream << 8) | (andersen ? 0x07u : 0x02u)), key);
                coll = andersen && (uint64_t)cw.x < S.andersen_thr;
                if (!andersen || coll) {
                    const uint4 w = andersen
                                        ? philox4x32_10(make_uint4(pid, 1u, (uint32_t)step,
                                                                   (S.stream << 8) | 0x07u), key)
                                        : cw;
                    const double u1 = ((double)w.x + 1.0) * 0x1p-32, u2 = (double)w.y * 0x1p-32;
                    const double u3 = ((double)w.z + 1.0) * 0x1p-32, u4 = (double)w.w * 0x1p-32;
                    const double r1 = sqrt(-2.0 * log(u1)), r3 = sqrt(-2.0 * log(u3));
                    double s2, c2;
                    sincospi(2.0 * u2, &s2, &c2);
                    xi[0] = r1 * c2;
                    xi[1] = r1 * s2;
                    xi[2] = r3 * cospi(2.0 * u4);
                }
            }
        }
    }
    __syncthreads();
    if (closes) {
        const double4 fr = s_f[tc];
        const double F3[3] = {fr.x + f.x, fr.y + f.y, fr.z + f.z};
        if (a.F_out64) a.F_out64[o] = make_double4(F3[0], F3[1], F3[2], 0.0);
        if (a.phi_out64) a.phi_out64[o] = fr.w + f.w;
        if (a.md_pos64) {
            double* vv[3] = {&v.x, &v.y, &v.z};
            double* rr[3] = {&rp.x, &rp.y, &rp.z};
            if (nhm) {
                // Nose-Hoover leapfrog: v <- (v a + (dt/m) F) b, drift, wrap
                const double na = a.nh[tl.sys].a, nb = a.nh[tl.sys].b;
                double v2 = 0.0;
#pragma unroll
                for (int d = 0; d < 3; ++d) {
                    const double vd = (*vv[d] * na + S.dt_over_m * F3[d]) * nb;
                    *rr[d] = wrap_box(*rr[d] + S.dt * vd, S.L);
                    *vv[d] = vd;
                    v2 += vd * vd;
                }
                atomicAdd(&a.nh[tl.sys].k2, __double2ull_rn(v2 * S.nh_k2scale));
            } else {
#pragma unroll
                for (int d = 0; d < 3; ++d) {
                    double vd = *vv[d] + S.dt_over_m * F3[d];
                    if (!andersen) vd = S.c1 * vd + S.c2 * xi[d];
                    *rr[d] = wrap_box(*rr[d] + S.dt * vd, S.L);
                    if (coll) vd = S.vsd * xi[d];          // Andersen collision after the drift
                    *vv[d] = vd;
                }
            }
            a.md_vel64[o] = v;
            a.md_pos64[o] = rp;
        }
    }
    if constexpr (EN) {
        if (a.blk_e) {
            const double2 r = block_sum2_real(owner ? acc.ec : 0.0, owner ? acc.elj : 0.0);
            if (threadIdx.x == 0) a.blk_e[blk] = r;
        }
        if (a.blk_w) {
            __syncthreads();                            // the partial buffers are reused
            const double2 r = block_sum2_real(owner ? acc.wc : 0.0, owner ? acc.wlj : 0.0);
            if (threadIdx.x == 0) a.blk_w[blk] = r;
        }
    }
}

template <int G, bool ONE, bool EN>
static void real_f64_e(cudaStream_t st, const RealArgs& a) {
    const dim3 grid(a.npblk, G);
    if constexpr (!ONE)
        if (a.poly64_form == kErfcxEach) {
            k_real_f64<G, ONE, EN, kErfcxEach><<<grid, kReal64Threads, 0, st>>>(a);
            return;
        }
    if (a.poly64_form == kErfcxPoly)
        k_real_f64<G, ONE, EN, kErfcxPoly><<<grid, kReal64Threads, 0, st>>>(a);
    else
        k_real_f64<G, ONE, EN, kErfcxLib><<<grid, kReal64Threads, 0, st>>>(a);
}

template <int G>
static void real_f64_g(cudaStream_t st, bool one, const RealArgs& a) {
    const bool en = a.phi_out64 || a.blk_e || a.blk_w;
    if (one) {
        if (en) real_f64_e<G, true, true>(st, a);
        else real_f64_e<G, true, false>(st, a);
    } else {
        if (en) real_f64_e<G, false, true>(st, a);
        else real_f64_e<G, false, false>(st, a);
    }
}

void launch_real_f64(cudaStream_t st, bool one, const RealArgs& a) {
    if (a.npblk <= 0) return;
    switch (a.split64) {
        case 4: real_f64_g<4>(st, one, a); break;
        case 8: real_f64_g<8>(st, one, a); break;
        case 32: real_f64_g<32>(st, one, a); break;
        default: real_f64_g<16>(st, one, a); break;
    }
}

}  // namespace rbe
