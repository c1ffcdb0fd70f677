// rbe_fourier.cu -- the Fourier (long-range) part of one RBE evaluation.
//
//  k-sampling   P i.i.d. m in Z^3 \ {0} from P_k ~ exp(-k^2 / 4 alpha)   (Eq. probexpression)
//               by a per-axis integer inverse-CDF table indexed with Philox words;
//  k_rho        partial structure factors of a tile of particles
//                 rho_tile(k_l) = sum_{j in tile} q_j exp(i k_l . r_j)           (Sec. 2)
//               particles (caller's order, so this branch does not wait for
//               the cell sort) staged in shared memory and read as broadcasts;
//               each block adds its sums to rho(k_l) with 64-bit fixed-point
//               atomics: integer addition is associative, so the cross-block
//               sum is bitwise reproducible, with no separate reduction pass;
//  k_force      per particle: F*_i = -q_i sum_l coef_l k_l Im(e^{-i k_l.r_i} rho_l)
//               (Eq. rbmapprox) and the Fourier part of dE/dq_i, with the k-batch
//               and coef_l rho_l, coef_l = (S/P) 4 pi / (V k^2) formed in FP64, staged
//               in shared memory; the mixed path holds coef_l rho_l in polar form
//               (R_l, phi_l), so that an MD step's force takes one sine per pair.
//
// Mixed path phases: theta = 2 pi (m . s mod 1) with s the 32-bit fixed-point
// fraction of the position; the product is exact in 32-bit integer arithmetic,
// so the only phase error is the conversion of a 32-bit integer to FP32
// (2^-25 turns).  sin/cos then run on the special-function unit for arguments
// in [-pi, pi).  No FP32 work grows with |m| or L.
#include <algorithm>
#include <cmath>

#include "rbe_internal.cuh"
#include "rbe_list_body.cuh"

namespace rbe {

constexpr float kTwoPiOver2p32 = 1.4629180792671596e-09f;   // 2 pi / 2^32
constexpr int kStage = 512;                                 // particles staged per pass

__global__ void k_sample(const SysDev* __restrict__ sysv, int nsys, int ktot,
                         const int* __restrict__ kstart, const uint64_t* __restrict__ table,
                         const uint64_t* __restrict__ cur_step, int4* __restrict__ ksamp,
                         int* __restrict__ err) {
    const int g = blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= ktot) return;
    const int s = find_sys(kstart, nsys, g);
    const SysDev& S = sysv[s];
    ksamp[g] = sample_one(S, table + S.off_t, g - S.off_k, *cur_step, err);
}

// ----------------------------------------------------------------- rho (mixed)
// Blocks of T = 128 or 256 threads: a tile of particles against a tile of up to
// 2 T wave vectors, two per thread (one shared-memory read of a particle serves
// two pairs), so a system with P of them fills ceil(P / 2) threads; the block holds
// floor(T / that) such groups ("subs"), which share the particles.  That keeps
// the lanes busy at any P: with one thread row of 128 per 256 wave vectors a
// batch of P = 100 used 39 % of them, P = 137 54 %, and P = 10 4 %.
//
// What bounds it: the special-function unit (a sine and a cosine per pair, 16
// cycles per warp), so the sums must cost little beside it.  A thread adds every
// other particle of a run of `run` particles in FP32, then carries the run's sum
// into a float pair (a few FP32 operations; FP64 additions and conversions are
// two lanes per clock on this part and, done per 32 particles, took as long as
// the sines).  Each block adds its sums to the fixed-point rho(k) with integer
// work, once per wave vector.  The result depends on `run` and on the runs'
// boundaries only through FP32 rounding; an evaluation that returns energies
// keeps the run its tuning names.
//
// Measured (events around the kernel, about 5 us of them launch, before -> now):
// N = 8001, P = 200 14.3 -> 10.9 us; 50021, P = 137 39.3 -> 13.9; 100003, P = 200 40.9 ->
// 20.9; 2^20, P = 100 129 -> 60.7; 262144, P = 500 70.6 -> 70.2 (full lanes already).

// round(f 2^e) as a 64-bit integer, in integer arithmetic (|f| 2^e < 2^63; beyond, the
// words saturate as a conversion of the double would)
__device__ __forceinline__ long long fixed64(float f, int e) {
    const uint32_t b = __float_as_uint(f);
    const int ex = (int)((b >> 23) & 255u);
    const long long m = ex ? (long long)((b & 0x7FFFFFu) | 0x800000u) : 0ll;
    const int sh = ex - 150 + e;
    const long long v = sh >= 0 ? (sh <= 39 ? m << sh : 0x7FFFFFFFFFFFFFFFll)
                                : (sh > -25 ? (m + (1ll << (-sh - 1))) >> -sh : 0ll);
    return (b >> 31) ? -v : v;
}

// Sums of one wave vector as float pairs: (Re hi, Re lo, Im hi, Im lo).
__device__ __forceinline__ void carry(float4& s, float re, float im) {
    const float2 x = two_sum(s.x, re), y = two_sum(s.z, im);
    s = make_float4(x.x, s.y + x.y, y.x, s.w + y.y);
}

__device__ __forceinline__ void carry(float4& s, f32x2 v) {
    const float2 c = unpack2(v);
    carry(s, c.x, c.y);
}

__device__ __forceinline__ void rho_add(unsigned long long* dst, const float4& s, int e) {
    atomicAdd(dst, (unsigned long long)(fixed64(s.x, e) + fixed64(s.y, e)));
    atomicAdd(dst + 1, (unsigned long long)(fixed64(s.z, e) + fixed64(s.w, e)));
}

// rho_body: particle tile ctile, wave-vector tile ktile (the whole block), for
// the kernel of its own and for the fused structure-factor + list launch.
template <int T, bool ONE>
__device__ __forceinline__ void rho_body(const Work& w, const int4* __restrict__ ksamp,
                                         const double* __restrict__ kcoef,
                                         const uint4* __restrict__ fx,
                                         unsigned long long* __restrict__ rho_fx,
                                         int* __restrict__ kcnt, float2* __restrict__ kab,
                                         int ctile, int ktile, int run) {
    __shared__ uint4 sp[kRhoStage];                  // 8 KB, then the subs' sums
    static_assert(sizeof(sp) >= sizeof(float4) * 2 * T, "sums alias the stage");
    const Tile ch = tile_at<ONE>(w, ctile);
    const SysDev& S = sys_of<ONE>(w, ch.sys);
    const int k0 = ktile * (2 * T);
    if (k0 >= S.P) return;                           // whole block beyond this system's P
    const int nk = min(S.P - k0, (2 * T));            // wave vectors of this tile
    const int slots = (nk + 1) / 2;
    const int subs = T / slots;
    const int sub = threadIdx.x / slots, slot = threadIdx.x - sub * slots;
    const bool work = sub < subs;
    uint32_t mx[2], my[2], mz[2];
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        const int4 m = ksamp[S.off_k + k0 + min(slot + r * slots, nk - 1)];   // prep drew them
        mx[r] = (uint32_t)m.x;
        my[r] = (uint32_t)m.y;
        mz[r] = (uint32_t)m.z;
    }
    float4 sum[2] = {make_float4(0.f, 0.f, 0.f, 0.f), make_float4(0.f, 0.f, 0.f, 0.f)};
    // particles per pass: a whole number of runs for every sub where that fits
    const int per = run * subs;
    const int stage = per <= kRhoStage ? per * (kRhoStage / per) : kRhoStage;
    for (int base = 0; base < ch.count; base += stage) {
        const int cnt = min(stage, ch.count - base);
        __syncthreads();
        for (int u = threadIdx.x; u < cnt; u += T) sp[u] = fx[ch.first + base + u];
        __syncthreads();
        // (cos, sin) of both wave vectors for one particle, added times its charge
        auto terms = [&](const uint4 p, f32x2* c) {
            const float q = __uint_as_float(p.w);
            const f32x2 qq = pack2(q, q);
            const float2 th = unpack2(
                mul2(pack2((float)(int32_t)(mx[0] * p.x + my[0] * p.y + mz[0] * p.z),
                           (float)(int32_t)(mx[1] * p.x + my[1] * p.y + mz[1] * p.z)),
                     pack2(kTwoPiOver2p32, kTwoPiOver2p32)));
            float sn, cs;
            __sincosf(th.x, &sn, &cs);
            c[0] = fma2(qq, pack2(cs, sn), c[0]);
            __sincosf(th.y, &sn, &cs);
            c[1] = fma2(qq, pack2(cs, sn), c[1]);
        };
        if (subs == 1) {
            // one thread takes a run's even and odd particles side by side
            if (work)
                for (int j0 = 0; j0 < cnt; j0 += run) {
                    const int j1 = min(cnt, j0 + run);
                    f32x2 even[2] = {0ull, 0ull}, odd[2] = {0ull, 0ull};
                    int j = j0;
#pragma unroll 8
                    for (; j + 1 < j1; j += 2) {
                        terms(sp[j], even);
                        terms(sp[j + 1], odd);
                    }
                    if (j < j1) terms(sp[j], even);
#pragma unroll
                    for (int r = 0; r < 2; ++r) {
                        carry(sum[r], even[r]);
                        carry(sum[r], odd[r]);
                    }
                }
        } else if (work) {
            // a run's even particles, then its odd ones, are a unit of work each
            for (int u = sub; (u >> 1) * run < cnt; u += subs) {
                const int j0 = (u >> 1) * run + (u & 1), j1 = min(cnt, ((u >> 1) + 1) * run);
                f32x2 c[2] = {0ull, 0ull};
#pragma unroll 8
                for (int j = j0; j < j1; j += 2) terms(sp[j], c);
                carry(sum[0], c[0]);
                carry(sum[1], c[1]);
            }
        }
    }
    unsigned long long* dst =
        rho_fx + (size_t)(ctile % kRhoCopies) * S.rho_stride + 2 * (S.off_k + k0);
    if (subs == 1) {
        if (work) {
            rho_add(dst + 2 * slot, sum[0], S.rho_exp);
            if (slot + slots < nk) rho_add(dst + 2 * (slot + slots), sum[1], S.rho_exp);
        }
    } else {
        float4* red = (float4*)sp;                   // [wave vector][sub]
        __syncthreads();
        if (work) {
            red[slot * subs + sub] = sum[0];
            red[(slot + slots) * subs + sub] = sum[1];
        }
        __syncthreads();
        for (int l = threadIdx.x; l < nk; l += T) {
            float4 s = red[l * subs];
            for (int u = 1; u < subs; ++u) {
                const float4 v = red[l * subs + u];
                carry(s, v.x, v.z);
                s.y += v.y;
                s.w += v.w;
            }
            rho_add(dst + 2 * l, s, S.rho_exp);
        }
    }
    // The last of the system's tiles to add its sums for this tile of
    // wave vectors finds rho(k) complete and turns it into the force
    // coefficient of Eq. rbmapprox in polar form, once per k instead of once
    // per force block: with A = coef Im rho and B = coef Re rho,
    // A cos(theta) - B sin(theta) = R sin(phi - theta) for R = |(A, B)| and
    // phi = atan2(A, B), stored as (R, phi in 2^-32 turns).  Fence, then
    // count: every tile's atomics are visible to the block that takes the
    // last count (no waiting on other blocks).
    __shared__ int s_last;
    __threadfence();
    __syncthreads();
    int* cnt_k = kcnt + S.off_k + k0;
    if (threadIdx.x == 0) s_last = atomicAdd(cnt_k, 1) == S.nrt - 1;
    __syncthreads();
    if (s_last) {
        __threadfence();
        for (int l = k0 + threadIdx.x; l < k0 + nk; l += T) {
            const double2 r =
                rho_total(rho_fx + 2 * (S.off_k + l), S.rho_stride, S.rho_inv_scale);
            const double c = kcoef[S.off_k + l];
            const float A = (float)(c * r.y), B = (float)(c * r.x);
            const float turns = atan2f(A, B) * 0.15915494309189535f;      // (-1/2, 1/2]
            const uint32_t phi = (uint32_t)(long long)llrintf(turns * 4294967296.0f);
            kab[S.off_k + l] = make_float2(hypotf(A, B), __uint_as_float(phi));
        }
        if (threadIdx.x == 0) *cnt_k = 0;            // ready for the next evaluation
    }
}

template <int T, bool ONE>
__global__ void __launch_bounds__(T, 1024 / T)
k_rho_mixed(const __grid_constant__ Work w, const int4* __restrict__ ksamp,
            const double* __restrict__ kcoef, const uint4* __restrict__ fx,
            unsigned long long* __restrict__ rho_fx, int* __restrict__ kcnt,
            float2* __restrict__ kab, int run) {
    pdl_wait();                                       // the prep kernel's samples and records
    pdl_trigger();                                    // the force kernel may be scheduled (and
                                                      // finds the prep kernel complete)
    rho_body<T, ONE>(w, ksamp, kcoef, fx, rho_fx, kcnt, kab, blockIdx.x, blockIdx.y, run);
}

// ------------------------------------------- structure factors + list pass
// The MD step's structure factors and its real-space pass over a standing
// neighbour list in one launch of T-thread blocks: block b takes
// structure-factor work when floor((b + 1) nrho / total) > floor(b nrho /
// total), else T / kBlockP tiles of the list pass, so that the two kinds are spread evenly
// over the grid and each SM holds both at once -- the structure factors keep
// the special-function unit busy while the pair terms use the ALU and FMA
// pipes and wait on their gathers.  The list tiles work only when the list
// stands (over a rebuilt list the build adds the pair terms itself).  The list
// pass is that of its own kernel (list_step), with as many entries in flight as the
// registers beside the structure factors allow.
template <int T, int R, bool ONE>
__global__ void __launch_bounds__(T, T == 128 ? 9 : 4)
k_rho_list(const __grid_constant__ Work w, const int4* __restrict__ ksamp,
           const double* __restrict__ kcoef, const uint4* __restrict__ fx,
           unsigned long long* __restrict__ rho_fx, int* __restrict__ kcnt,
           float2* __restrict__ kab, const __grid_constant__ RealArgs a, int ntiles, int run,
           int nrho, int nlist) {
    pdl_wait();                                       // the prep kernel's samples and records
    pdl_trigger();                                    // the force kernel may be scheduled (and
                                                      // finds the prep kernel complete)
    const int b = blockIdx.x, total = nrho + nlist;
    const int r0 = (int)((long long)b * nrho / total);
    const int r1 = (int)((long long)(b + 1) * nrho / total);
    if (r1 > r0) {
        rho_body<T, ONE>(w, ksamp, kcoef, fx, rho_fx, kcnt, kab, r0 % ntiles, r0 / ntiles, run);
        return;
    }
    if (*a.list_flag) return;
    const int tile = (T / kBlockP) * (b - r1) + (int)(threadIdx.x / kBlockP);
    if (tile < a.nlblk)
        list_step<R, ONE, false, T == 128 ? 4 : 8, T == 128>(a, tile, threadIdx.x % kBlockP);
}

// ----------------------------------------------------------------- force (mixed)
// Shared-memory record per wave vector: -m and phi (the phase of the
// coefficient, 2^-32 turns) as integers, and R m (the direction scaled by the
// coefficient's magnitude) with R as floats.  phi - m.s is exact in 32-bit
// arithmetic, so one sine per (particle, k) pair gives the force term
// R m sin(phi - theta) = m coef Im(e^{-i k.r} rho) (and the cosine, in the
// same SFU pair, the dE/dq term R cos(phi - theta)).
struct KPhase { uint32_t nmx, nmy, nmz, phi; };
struct KForce { float rmx, rmy, rmz, R; };
// SPLIT threads per particle (each a 1/SPLIT share of the wave vectors), or
// with SPLIT = 1 PT = 2 particles per thread, which share each wave vector's
// shared-memory loads and the loop overhead (the pass is issue-bound at large
// N).  A block holds a tile of kBlockP / SPLIT particles and kBlockP / PT
// threads.  A: sums of its own per thread, each over every A-th term of its share, so
// that fewer threads per particle do not mean longer FP32 chains.  PHI: also dE/dq (the
// forces path); MD steps need only the force.
template <int SPLIT, int PT, int A, bool PHI, bool ONE>
__global__ void __launch_bounds__(kBlockP / PT)
k_force_mixed(const __grid_constant__ Work w, const uint4* __restrict__ rec,
              const int4* __restrict__ ksamp, const float2* __restrict__ kab,
              float4* __restrict__ fs, const __grid_constant__ MdOut md) {
    static_assert(PT == 1 || SPLIT == 1, "two particles per thread only with one thread each");
    constexpr int NT = kBlockP / PT;                // threads per block
    constexpr int TILE = kBlockP / SPLIT;           // particles per block
    constexpr int EP = (TILE + NT - 1) / NT;        // closing updates per thread
    constexpr int kKT = 256;                        // wave vectors staged per pass
    __shared__ KPhase kp[kKT];
    __shared__ KForce kf[kKT];
    const Tile tl = tile_of<ONE>(w);
    const SysDev& S = sys_of<ONE>(w, tl.sys);
    const int sub = threadIdx.x % SPLIT;            // lane within the particle's group
    if constexpr (SPLIT == 1) pdl_wait();           // rho(k), kab and the real-space forces
    // Before the structure factors are complete (SPLIT > 1: in the large systems of
    // SPLIT 1 there is nothing to hide, and the order costs registers): what the prep kernel and the
    // previous step left -- the records, and (MD step) the inputs of the closing
    // update (thread t: particles t, t + NT, .. of the tile) and the thermostat's
    // noise.  With a programmatic launch the blocks get here when every block of
    // the structure-factor kernel has found the prep kernel complete; loads past
    // L1, which may hold an earlier step's lines.
    int tq[PT];
    uint4 p[PT];
#pragma unroll
    for (int q = 0; q < PT; ++q) {
        tq[q] = threadIdx.x / SPLIT + q * (NT / SPLIT);
        p[q] = make_uint4(0, 0, 0, 0);
        if (tl.count > 0) p[q] = __ldcg(rec + tl.first + min(tq[q], tl.count - 1));
    }
    const bool nhm = md.md_pos && md.nh && S.thermostat == RBE_THERMO_NOSE_HOOVER;
    float4 e_fr[EP], e_v[EP], e_r[EP];
    MdNoise e_z[EP];
#pragma unroll
    for (int e = 0; e < EP; ++e) {
        e_fr[e] = make_float4(0.f, 0.f, 0.f, 0.f);
        e_v[e] = e_fr[e];
        e_r[e] = e_fr[e];
        e_z[e] = MdNoise{0.f, 0.f, 0.f, false};
        const int te = threadIdx.x + e * NT;
        if (md.freal && te < tl.count) {
            const int o = tl.first + te;
            if constexpr (SPLIT == 1) e_fr[e] = md.freal[o];
            if (md.md_pos) {
                e_v[e] = __ldcg(md.vel_in + o);
                e_r[e] = __ldcg(md.pos_in + o);
                if (!nhm) e_z[e] = md_noise(S, __ldcg((const unsigned long long*)md.cur_step), o);
            }
        }
    }
    if constexpr (SPLIT > 1) {
        pdl_wait();
        pdl_trigger();                              // the next step's prep kernel may be scheduled
        if (md.freal) {
#pragma unroll
            for (int e = 0; e < EP; ++e) {
                const int te = threadIdx.x + e * NT;
                if (te < tl.count) e_fr[e] = md.freal[tl.first + te];
            }
        }
    }
    float cx[PT][A], cy[PT][A], cz[PT][A], cp[PT][A];      // sums of every A-th term
#pragma unroll
    for (int q = 0; q < PT; ++q)
#pragma unroll
        for (int u = 0; u < A; ++u) cx[q][u] = cy[q][u] = cz[q][u] = cp[q][u] = 0.f;
    for (int base = 0; base < S.P; base += kKT) {
        const int cnt = min(kKT, S.P - base);
        __syncthreads();
        for (int k = threadIdx.x; k < cnt; k += blockDim.x) {
            const int4 m = ksamp[S.off_k + base + k];
            const float2 rp = kab[S.off_k + base + k];
            kp[k] = KPhase{0u - (uint32_t)m.x, 0u - (uint32_t)m.y, 0u - (uint32_t)m.z,
                           __float_as_uint(rp.y)};
            kf[k] = KForce{rp.x * (float)m.x, rp.x * (float)m.y, rp.x * (float)m.z, rp.x};
        }
        __syncthreads();
        auto term = [&](int k, int u) {
            const KPhase a = kp[k];
            const KForce f = kf[k];
#pragma unroll
            for (int q = 0; q < PT; ++q) {
                const uint32_t d = a.phi + a.nmx * p[q].x + a.nmy * p[q].y + a.nmz * p[q].z;
                const float t = (float)(int32_t)d * kTwoPiOver2p32;          // phi - theta
                float sn;                                   // Im(e^{-i theta} rho) coef / R
                if constexpr (PHI) {
                    float cs;
                    __sincosf(t, &sn, &cs);
                    cp[q][u] = fmaf(f.R, cs, cp[q][u]);     // Re(e^{-i theta} rho) * coef
                } else {
                    sn = __sinf(t);
                }
                cx[q][u] = fmaf(sn, f.rmx, cx[q][u]);
                cy[q][u] = fmaf(sn, f.rmy, cy[q][u]);
                cz[q][u] = fmaf(sn, f.rmz, cz[q][u]);
            }
        };
        int k = sub;
#pragma unroll 8 / A
        for (; k + (A - 1) * SPLIT < cnt; k += A * SPLIT)
#pragma unroll
            for (int u = 0; u < A; ++u) term(k + u * SPLIT, u);
#pragma unroll
        for (int u = 0; u < A - 1; ++u)
            if (k + u * SPLIT < cnt) term(k + u * SPLIT, u);
    }
    float fx[PT], fy[PT], fz[PT], ph[PT];
#pragma unroll
    for (int q = 0; q < PT; ++q) {
#pragma unroll
        for (int d = A / 2; d > 0; d >>= 1)
#pragma unroll
            for (int u = 0; u < d; ++u) {
                cx[q][u] += cx[q][u + d];
                cy[q][u] += cy[q][u + d];
                cz[q][u] += cz[q][u + d];
                cp[q][u] += cp[q][u + d];
            }
        fx[q] = cx[q][0];
        fy[q] = cy[q][0];
        fz[q] = cz[q][0];
        ph[q] = cp[q][0];
    }
#pragma unroll
    for (int o = SPLIT / 2; o > 0; o >>= 1) {
        fx[0] += __shfl_down_sync(0xffffffffu, fx[0], o, SPLIT);
        fy[0] += __shfl_down_sync(0xffffffffu, fy[0], o, SPLIT);
        fz[0] += __shfl_down_sync(0xffffffffu, fz[0], o, SPLIT);
        ph[0] += __shfl_down_sync(0xffffffffu, ph[0], o, SPLIT);
    }
    if (!md.freal) {
#pragma unroll
        for (int q = 0; q < PT; ++q)
            if (tq[q] < tl.count && sub == 0) {
                const float qc = __uint_as_float(p[q].w);
                const float sc = -qc * (float)(2.0 * M_PI) * S.f_invL;
                fs[tl.first + tq[q]] = make_float4(sc * fx[q], sc * fy[q], sc * fz[q], ph[q]);
            }
        return;
    }
    // neighbour-list MD step: the total force and the thermostat
    if (md.list_flag && blockIdx.x == 0 && threadIdx.x == 0) *md.list_flag = 0;   // consumed
    __shared__ float4 s_t[TILE];
#pragma unroll
    for (int q = 0; q < PT; ++q)
        if (tq[q] < tl.count && sub == 0) {
            const float qc = __uint_as_float(p[q].w);
            const float sc = -qc * (float)(2.0 * M_PI) * S.f_invL;
            s_t[tq[q]] = make_float4(sc * fx[q], sc * fy[q], sc * fz[q], 0.f);
        }
    __syncthreads();
    unsigned long long k2 = 0ull;
#pragma unroll
    for (int e = 0; e < EP; ++e) {
        const int te = threadIdx.x + e * NT;
        if (te < tl.count) {
            const int o = tl.first + te;
            const float4 ff = s_t[te];
            const float Fx = e_fr[e].x + ff.x, Fy = e_fr[e].y + ff.y, Fz = e_fr[e].z + ff.z;
            if (md.F_out) md.F_out[o] = make_float4(Fx, Fy, Fz, 0.f);
            if (md.md_pos) {
                if (nhm)
                    k2 += nose_hoover_apply(S, md.nh[tl.sys].f_va, md.nh[tl.sys].f_vf, Fx, Fy,
                                            Fz, e_v[e], e_r[e]);
                else
                    md_apply(S, e_z[e], Fx, Fy, Fz, e_v[e], e_r[e]);
                md.md_vel[o] = e_v[e];
                md.md_pos[o] = e_r[e];
            }
        }
    }
    if (nhm) warp_add_u64(k2, &md.nh[tl.sys].k2);
    if (md.done_host) {
        __threadfence_system();                     // this thread's pos / vel stores
        __syncthreads();
        if (threadIdx.x == 0 && atomicAdd(md.done_cnt, 1u) == gridDim.x - 1) {
            __threadfence_system();                 // every block's stores, then the words
            *md.done_cnt = 0u;
            *(volatile int*)md.err_host = *(const volatile int*)md.err;
            __threadfence_system();
            *(volatile unsigned long long*)md.done_host = *md.cur_step + 1ull;
        }
    }
}

// ------------------------------------------------------------- launchers
void launch_sample(cudaStream_t st, const SysDev* sys, int nsys, int ktot, const int* kstart,
                   const uint64_t* table, const uint64_t* cur_step, int4* ksamp, int* err) {
    if (ktot <= 0) return;
    k_sample<<<(ktot + 127) / 128, 128, 0, st>>>(sys, nsys, ktot, kstart, table, cur_step, ksamp,
                                                 err);
}

// The k-batch (ksamp) and coef_scale / k^2 (kcoef) come from the prep kernel.
template <int T>
static void rho_mixed_t(cudaStream_t st, bool one, const Work& w, int ntiles, int ktiles, int run,
                        const int4* ksamp, const double* kcoef, const uint4* fx,
                        unsigned long long* rho_fx, int* kcnt, float2* kab, bool pdl) {
    PdlConfig c(dim3(ntiles, ktiles), dim3(T), 0, st, pdl);
    if (one)
        cudaLaunchKernelEx(&c.cfg, k_rho_mixed<T, true>, w, ksamp, kcoef, fx, rho_fx, kcnt, kab,
                           run);
    else
        cudaLaunchKernelEx(&c.cfg, k_rho_mixed<T, false>, w, ksamp, kcoef, fx, rho_fx, kcnt, kab,
                           run);
}

void launch_rho_mixed(cudaStream_t st, bool one, const Work& w, const RhoGrid& g,
                      const int4* ksamp, const double* kcoef, const uint4* fx,
                      unsigned long long* rho_fx, int* kcnt, float2* kab, bool pdl) {
    if (g.ntiles <= 0 || g.ktiles <= 0) return;
    if (g.threads == 128)
        rho_mixed_t<128>(st, one, w, g.ntiles, g.ktiles, g.run, ksamp, kcoef, fx, rho_fx, kcnt, kab, pdl);
    else
        rho_mixed_t<256>(st, one, w, g.ntiles, g.ktiles, g.run, ksamp, kcoef, fx, rho_fx, kcnt, kab, pdl);
}

template <int T, int R>
static void rho_list_r(cudaStream_t st, bool one, const Work& w, const RhoGrid& g,
                       const int4* ksamp, const double* kcoef, const uint4* fx,
                       unsigned long long* rho_fx, int* kcnt, float2* kab, const RealArgs& a,
                       bool pdl) {
    constexpr int LT = T / kBlockP;
    const int nrho = g.ntiles * g.ktiles, nlist = (a.nlblk + LT - 1) / LT;
    PdlConfig c(dim3(nrho + nlist), dim3(T), 0, st, pdl);
    if (one)
        cudaLaunchKernelEx(&c.cfg, k_rho_list<T, R, true>, w, ksamp, kcoef, fx, rho_fx, kcnt, kab,
                           a, g.ntiles, g.run, nrho, nlist);
    else
        cudaLaunchKernelEx(&c.cfg, k_rho_list<T, R, false>, w, ksamp, kcoef, fx, rho_fx, kcnt,
                           kab, a, g.ntiles, g.run, nrho, nlist);
}

template <int T>
static void rho_list_t(cudaStream_t st, bool one, const Work& w, const RhoGrid& g,
                       const int4* ksamp, const double* kcoef, const uint4* fx,
                       unsigned long long* rho_fx, int* kcnt, float2* kab, const RealArgs& a,
                       bool pdl) {
    switch (a.lsplit) {
        case 2: rho_list_r<T, 2>(st, one, w, g, ksamp, kcoef, fx, rho_fx, kcnt, kab, a, pdl); break;
        case 4: rho_list_r<T, 4>(st, one, w, g, ksamp, kcoef, fx, rho_fx, kcnt, kab, a, pdl); break;
        case 8: rho_list_r<T, 8>(st, one, w, g, ksamp, kcoef, fx, rho_fx, kcnt, kab, a, pdl); break;
        default: rho_list_r<T, 1>(st, one, w, g, ksamp, kcoef, fx, rho_fx, kcnt, kab, a, pdl); break;
    }
}

void launch_rho_list(cudaStream_t st, bool one, const Work& w, const RhoGrid& g,
                     const int4* ksamp, const double* kcoef, const uint4* fx,
                     unsigned long long* rho_fx, int* kcnt, float2* kab, const RealArgs& a,
                     bool pdl) {
    if (g.ntiles <= 0 || g.ktiles <= 0) return;
    if (g.threads == 128)
        rho_list_t<128>(st, one, w, g, ksamp, kcoef, fx, rho_fx, kcnt, kab, a, pdl);
    else
        rho_list_t<256>(st, one, w, g, ksamp, kcoef, fx, rho_fx, kcnt, kab, a, pdl);
}

template <int SPLIT, int PT, int A>
static void force_mixed_a(cudaStream_t st, bool one, const Work& w, int nblk, const uint4* fx,
                          const int4* ksamp, const float2* kab, float4* fs, const MdOut& md,
                          bool pdl) {
    PdlConfig c(dim3(nblk), dim3(kBlockP / PT), 0, st, pdl);
    if (md.freal) {
        if (one) cudaLaunchKernelEx(&c.cfg, k_force_mixed<SPLIT, PT, A, false, true>, w, fx, ksamp, kab, fs, md);
        else cudaLaunchKernelEx(&c.cfg, k_force_mixed<SPLIT, PT, A, false, false>, w, fx, ksamp, kab, fs, md);
    } else {
        if (one) cudaLaunchKernelEx(&c.cfg, k_force_mixed<SPLIT, PT, A, true, true>, w, fx, ksamp, kab, fs, md);
        else cudaLaunchKernelEx(&c.cfg, k_force_mixed<SPLIT, PT, A, true, false>, w, fx, ksamp, kab, fs, md);
    }
}

template <int SPLIT, int PT>
static void force_mixed_split(cudaStream_t st, bool one, const Work& w, int nblk, int sums,
                              const uint4* fx, const int4* ksamp, const float2* kab, float4* fs,
                              const MdOut& md, bool pdl) {
    if constexpr (SPLIT <= 2)
        if (sums >= 4) return force_mixed_a<SPLIT, PT, 4>(st, one, w, nblk, fx, ksamp, kab, fs, md, pdl);
    if constexpr (SPLIT <= 4)
        if (sums >= 2) return force_mixed_a<SPLIT, PT, 2>(st, one, w, nblk, fx, ksamp, kab, fs, md, pdl);
    force_mixed_a<SPLIT, PT, 1>(st, one, w, nblk, fx, ksamp, kab, fs, md, pdl);
}

void launch_fourier_force_mixed(cudaStream_t st, bool one, const Work& w, int nblk, int split,
                                int sums, const uint4* fx, const int4* ksamp, const float2* kab,
                                float4* fs, const MdOut& md, bool pdl) {
    if (nblk <= 0) return;
    switch (split) {
        case 2: force_mixed_split<2, 1>(st, one, w, nblk, sums, fx, ksamp, kab, fs, md, pdl); break;
        case 4: force_mixed_split<4, 1>(st, one, w, nblk, sums, fx, ksamp, kab, fs, md, pdl); break;
        case 8: force_mixed_split<8, 1>(st, one, w, nblk, sums, fx, ksamp, kab, fs, md, pdl); break;
        default: force_mixed_split<1, 2>(st, one, w, nblk, sums, fx, ksamp, kab, fs, md, pdl); break;
    }
}

}  // namespace rbe

namespace rbe {

// ----------------------------------------------------------------- observables
// Full (non-random) Ewald structure factors of one system over a half space of
// wave vectors (m and -m give conjugate rho(k)): the phases as in the
// structure-factor pass (exact 32-bit phase, FP32 sin/cos), the sums in the
// 64-bit fixed-point accumulators.  Grid: (particle chunks, k tiles).
__global__ void __launch_bounds__(kLTile)
k_struct_full(const uint4* __restrict__ fx, int first, int n, int chunk,
              const int4* __restrict__ mlist, int K, double scale,
              unsigned long long* __restrict__ rho_fx) {
    __shared__ uint4 sp[kStage];
    const int l = blockIdx.y * kLTile + threadIdx.x;
    const bool active = l < K;
    const int4 m = active ? mlist[l] : make_int4(0, 0, 0, 0);
    const uint32_t mx = (uint32_t)m.x, my = (uint32_t)m.y, mz = (uint32_t)m.z;
    const int b0 = blockIdx.x * chunk;
    const int cnt_all = min(chunk, n - b0);
    float re = 0.f, im = 0.f;
    for (int base = 0; base < cnt_all; base += kStage) {
        const int cnt = min(kStage, cnt_all - base);
        __syncthreads();
        for (int t = threadIdx.x; t < cnt; t += blockDim.x) sp[t] = fx[first + b0 + base + t];
        __syncthreads();
        if (active) {
#pragma unroll 4
            for (int j = 0; j < cnt; ++j) {
                const uint4 p = sp[j];
                const uint32_t ph = mx * p.x + my * p.y + mz * p.z;
                float sn, cs;
                __sincosf((float)(int32_t)ph * kTwoPiOver2p32, &sn, &cs);
                const float q = __uint_as_float(p.w);
                re = fmaf(q, cs, re);
                im = fmaf(q, sn, im);
            }
        }
    }
    if (active && cnt_all > 0) rho_accumulate(rho_fx + 2 * l, (double)re, (double)im, scale);
}

// Energy and virial terms of the full structure factors, one thread per wave
// vector, FP64, summed per block in a fixed order: part[b] = (sum e_k, sum w_k)
// with e_k = 2 A_k |rho_k|^2 (half space: each k stands for +-k),
// A_k = (2 pi lB / V) e^{-k^2/(4 alpha)} / k^2, w_k = e_k (1 - k^2 / (2 alpha)).
__global__ void __launch_bounds__(256)
k_obs_terms(const __grid_constant__ SysDev S, const int4* __restrict__ mlist, int K,
            const unsigned long long* __restrict__ rho_fx, double2* __restrict__ part) {
    __shared__ double sa[256], sb[256];
    const int l = blockIdx.x * blockDim.x + threadIdx.x;
    double e = 0.0, wv = 0.0;
    if (l < K) {
        const double tp = 2.0 * M_PI * S.invL;
        const int4 m = mlist[l];
        const double k2 = tp * tp * ((double)m.x * m.x + (double)m.y * m.y + (double)m.z * m.z);
        const double2 r = rho_read(rho_fx + 2 * l, S.rho_inv_scale);
        e = 2.0 * (2.0 * M_PI * S.lB / S.V) * exp(-k2 / (4.0 * S.alpha)) / k2 *
            (r.x * r.x + r.y * r.y);
        wv = e * (1.0 - k2 / (2.0 * S.alpha));
    }
    sa[threadIdx.x] = e;
    sb[threadIdx.x] = wv;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if ((int)threadIdx.x < o) {
            sa[threadIdx.x] += sa[threadIdx.x + o];
            sb[threadIdx.x] += sb[threadIdx.x + o];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) part[blockIdx.x] = make_double2(sa[0], sb[0]);
}

// One block: the true energy and the virial of one system from the per-block
// wave-vector partials, the real-space Coulomb / LJ energies and virials of the
// preceding evaluation, the charges and the velocities, all summed in FP64 in
// a fixed order.  out[12]: E_total, E_fourier (incl. self and background),
// E_real, E_lj, E_kin, W_fourier, W_real, W_lj, W_background, pressure,
// kinetic temperature, 0.  P = (2 E_kin + W) / (3 V); W_bg = 3 E_bg.
__global__ void __launch_bounds__(256)
k_observables(const __grid_constant__ SysDev S, const double2* __restrict__ part, int nparts,
              const float4* __restrict__ pos_q, const float4* __restrict__ vel, int n,
              const double* __restrict__ E_in, const double* __restrict__ W_in, double mass,
              double* __restrict__ out) {
    __shared__ double sa[256], sb[256], sc[256], sd[256], se[256];
    double ef = 0.0, wf = 0.0, q1 = 0.0, q2 = 0.0, ke = 0.0;
    for (int b = threadIdx.x; b < nparts; b += blockDim.x) {
        const double2 v = part[b];
        ef += v.x;
        wf += v.y;
    }
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        const double q = (double)pos_q[i].w;
        q1 += q;
        q2 += q * q;
        if (vel) {
            const float4 v = vel[i];
            ke += 0.5 * mass * ((double)v.x * v.x + (double)v.y * v.y + (double)v.z * v.z);
        }
    }
    sa[threadIdx.x] = ef; sb[threadIdx.x] = wf; sc[threadIdx.x] = q1; sd[threadIdx.x] = q2;
    se[threadIdx.x] = ke;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if ((int)threadIdx.x < o) {
            sa[threadIdx.x] += sa[threadIdx.x + o];
            sb[threadIdx.x] += sb[threadIdx.x + o];
            sc[threadIdx.x] += sc[threadIdx.x + o];
            sd[threadIdx.x] += sd[threadIdx.x + o];
            se[threadIdx.x] += se[threadIdx.x + o];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        const double ebg = -S.lB * M_PI * sc[0] * sc[0] / (2.0 * S.V * S.alpha);
        const double eself = -S.self_coef * sd[0];
        const double Ef = sa[0] + eself + ebg;
        const double Er = E_in[2], El = E_in[3];
        const double W = sb[0] + W_in[0] + W_in[1] + 3.0 * ebg;
        out[0] = Ef + Er + El;
        out[1] = Ef;
        out[2] = Er;
        out[3] = El;
        out[4] = se[0];
        out[5] = sb[0];
        out[6] = W_in[0];
        out[7] = W_in[1];
        out[8] = 3.0 * ebg;
        out[9] = (2.0 * se[0] + W) / (3.0 * S.V);
        out[10] = n > 0 ? 2.0 * se[0] / (3.0 * (double)n) : 0.0;
        out[11] = 0.0;
    }
}

void launch_observables(cudaStream_t st, const SysDev& S, const uint4* fx, int first, int n,
                        const int4* mlist, int K, unsigned long long* rho_fx, double2* part,
                        const float4* pos_q, const float4* vel, const double* E_in,
                        const double* W_in, double mass, double* out) {
    const int nparts = (K + 255) / 256;
    if (K > 0) {
        const int chunk = 1024;
        const int nch = std::max(1, (n + chunk - 1) / chunk);
        dim3 grid(nch, (K + kLTile - 1) / kLTile);
        cudaMemsetAsync(rho_fx, 0, sizeof(unsigned long long) * 2 * (size_t)K, st);
        if (n > 0)
            k_struct_full<<<grid, kLTile, 0, st>>>(fx, first, n, chunk, mlist, K, S.rho_scale,
                                                   rho_fx);
        k_obs_terms<<<nparts, 256, 0, st>>>(S, mlist, K, rho_fx, part);
    }
    k_observables<<<1, 256, 0, st>>>(S, part, nparts, pos_q + first,
                                     vel ? vel + first : nullptr, n, E_in, W_in, mass, out);
}

}  // namespace rbe
