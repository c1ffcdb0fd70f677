// rbe_fourier64.cu -- the Fourier part of the FP64 path: structure factors
//   rho(k_l) = sum_j q_j exp(i k_l . r_j)                                  (Sec. 2)
// and the force F*_i = -q_i sum_l coef_l k_l Im(e^{-i k_l.r_i} rho_l)     (Eq. rbmapprox)
// with the phase factors taken from per-particle tables of powers
//   e^{2 pi i m x / L},  m = 0 .. max |m| of the batch,  for each axis,
// so that a (particle, wave vector) pair costs two complex products instead
// of an FP64 sine and cosine.
//
// What bounds it: the FP64 pipe, two lanes per SM and clock on this part, so
// the count of FP64 instructions is everything and shared-memory gathers ride
// along for free.  A pair costs 8 (structure factor) or 13 (force) of them
// against about 50 with sincos; a table entry costs 4 (a power is the product
// of two smaller ones, log2 max|m| rounds) and is shared by all P wave vectors.
// The phase of the first power is exact to an ulp (its rounding error is
// recovered with an FMA), so the m-th power is off by about m ulp: less than
// the rounding of k.r in the direct form, whose size is |k.r| ulp.
//
// Split: a block holds the tables of kTabP particles at a time.  Structure
// factors: one thread per KR wave vectors, the block's particles in turn.
// Force: 16 lanes per particle, each a sixteenth of the wave vectors.  With 8
// particles per block a system of 1000 is 125 blocks, so that most SMs work
// (one thread per particle left 8 blocks of 128).
// Measured (events around one kernel, launch included), structure factors and
// force: N = 1000, P = 100: 41 -> 12 and 133 -> 14 us against one sincos per
// pair; N = 8001, P = 200: 132 -> 41 and 261 -> 67 us.  Error of forces / dE/dq
// against an 80-bit evaluation, geometric mean over 16 systems of 9000 to 20000:
// 0.56 / 0.79 of the direct form's.
#include <algorithm>

#include "rbe_internal.cuh"

namespace rbe {

constexpr int kTabP = 8;            // particles whose tables a block holds at a time
constexpr int kTabThreads = 128;
constexpr int kTabLanes = kTabThreads / kTabP;     // lanes per particle of the force
constexpr int kTabK = 128;          // wave vectors staged per pass of the force

// Direct form: tables that do not fit in shared memory or do not pay (large alpha L^2).
constexpr int kDirectStage = 256;

size_t tab_smem(int mcap) { return sizeof(double2) * kTabP * 3 * (size_t)(mcap + 1); }

__device__ __forceinline__ double2 cmul(const double2 a, const double2 b) {
    return make_double2(fma(a.x, b.x, -(a.y * b.y)), fma(a.x, b.y, a.y * b.x));
}

// b with its sign bit flipped where neg is 0x80000000 (integer work)
__device__ __forceinline__ double flip(double v, uint32_t neg) {
    return __hiloint2double((int)((uint32_t)__double2hiint(v) ^ neg), __double2loint(v));
}

// Largest |m| over the system's batch (the whole block; synchronises it).
__device__ __forceinline__ int batch_mmax(const int4* __restrict__ ksamp, int P) {
    __shared__ int s_mm;
    if (threadIdx.x == 0) s_mm = 1;
    __syncthreads();
    int mm = 1;
    for (int l = threadIdx.x; l < P; l += blockDim.x) {
        const int4 m = ksamp[l];
        mm = max(mm, max(abs(m.x), max(abs(m.y), abs(m.z))));
    }
    mm = __reduce_max_sync(0xffffffffu, mm);
    if ((threadIdx.x & 31) == 0) atomicMax(&s_mm, mm);
    __syncthreads();
    return s_mm;
}

// tab[(3 p + axis) * (mm + 1) + m] = e^{2 pi i m x / L} of cnt records, axis 0
// scaled by the charge if fold_q.  Ends with a block synchronisation.
__device__ __forceinline__ void build_tables(double2* __restrict__ tab, int mm, int cnt,
                                             const double4* __restrict__ rec, const SysDev& S,
                                             bool fold_q) {
    const int st = mm + 1, rows = 3 * cnt;
    for (int e = threadIdx.x; e < rows; e += blockDim.x) {
        const double4 p = rec[e / 3];
        const int ax = e % 3;
        const double x = ax == 0 ? p.x : (ax == 1 ? p.y : p.z);
        const double f = x * S.invL;
        const double d = 2.0 * M_PI * (fma(-f, S.L, x) * S.invL);    // what f's rounding lost
        double sn, cs;
        sincospi(2.0 * f, &sn, &cs);
        tab[e * st] = make_double2(1.0, 0.0);
        tab[e * st + 1] = make_double2(fma(-sn, d, cs), fma(cs, d, sn));
    }
    for (int h = 1; h < mm; h <<= 1) {
        __syncthreads();
        const int w = min(h, mm - h);
        for (int e = threadIdx.x; e < rows * w; e += blockDim.x) {
            const int r = e / w, j = e - r * w + 1;
            double2* T = tab + r * st;
            T[h + j] = cmul(T[h], T[j]);
        }
    }
    __syncthreads();
    if (fold_q) {
        for (int e = threadIdx.x; e < cnt * st; e += blockDim.x) {
            const int p = e / st;
            double2* T = tab + 3 * p * st + (e - p * st);
            const double q = rec[p].w;
            *T = make_double2(T->x * q, T->y * q);
        }
        __syncthreads();
    }
}

// ----------------------------------------------------------------- rho
// Block (x, y, z): share y of chunk x (the chunk cut into gridDim.y equal
// parts) and tile z of kTabThreads * KR wave vectors.
template <bool ONE, int KR>
__global__ void __launch_bounds__(kTabThreads)
k_rho_f64_tab(const __grid_constant__ Work w, const int4* __restrict__ ksamp,
              const double4* __restrict__ fx64, unsigned long long* __restrict__ rho_fx) {
    extern __shared__ __align__(16) unsigned char smem64[];
    double2* tab = (double2*)smem64;
    const Tile ch = tile_of<ONE>(w);
    const SysDev& S = sys_of<ONE>(w, ch.sys);
    const int l0 = blockIdx.z * kTabThreads * KR;
    const int per = (ch.count + gridDim.y - 1) / gridDim.y;
    const int b0 = blockIdx.y * per, b1 = min(ch.count, b0 + per);
    if (l0 >= S.P || b0 >= b1) return;
    pdl_trigger();                                  // the force kernel may build its tables
    const int mm = batch_mmax(ksamp + S.off_k, S.P), st = mm + 1;
    int ox[KR], oy[KR], oz[KR];
    uint32_t nx[KR], ny[KR], nz[KR];
    double re[KR], im[KR];
#pragma unroll
    for (int r = 0; r < KR; ++r) {
        const int l = l0 + r * kTabThreads + threadIdx.x;
        const int4 m = ksamp[S.off_k + min(l, S.P - 1)];
        ox[r] = abs(m.x); oy[r] = st + abs(m.y); oz[r] = 2 * st + abs(m.z);
        nx[r] = m.x < 0 ? 0x80000000u : 0u;
        ny[r] = m.y < 0 ? 0x80000000u : 0u;
        nz[r] = m.z < 0 ? 0x80000000u : 0u;
        re[r] = im[r] = 0.0;
    }
    const bool any = l0 + (int)threadIdx.x < S.P;
    for (int base = b0; base < b1; base += kTabP) {
        const int cnt = min(kTabP, b1 - base);
        if (base > b0) __syncthreads();
        build_tables(tab, mm, cnt, fx64 + ch.first + base, S, true);
        if (any) {
            for (int p = 0; p < cnt; ++p) {
                const double2* T = tab + 3 * p * st;
#pragma unroll
                for (int r = 0; r < KR; ++r) {
                    if (l0 + r * kTabThreads + ((int)threadIdx.x & ~31) >= S.P) break;  // no lane
                    double2 X = T[ox[r]], Y = T[oy[r]], Z = T[oz[r]];
                    X.y = flip(X.y, nx[r]);
                    Y.y = flip(Y.y, ny[r]);
                    Z.y = flip(Z.y, nz[r]);
                    const double2 E = cmul(X, Y);
                    re[r] = fma(E.x, Z.x, fma(-E.y, Z.y, re[r]));
                    im[r] = fma(E.x, Z.y, fma(E.y, Z.x, im[r]));
                }
            }
        }
    }
    unsigned long long* dst =
        rho_fx + (size_t)((blockIdx.x * gridDim.y + blockIdx.y) % kRhoCopies) * S.rho_stride +
        2 * S.off_k;
#pragma unroll
    for (int r = 0; r < KR; ++r) {
        const int l = l0 + r * kTabThreads + threadIdx.x;
        if (l < S.P) rho_accumulate(dst + 2 * l, re[r], im[r], S.rho_scale);
    }
}

// Direct form, one sincos per pair: where the tables do not fit or do not pay.
template <bool ONE>
__global__ void __launch_bounds__(kLTile)
k_rho_f64(const __grid_constant__ Work w, const int4* __restrict__ ksamp,
          const double4* __restrict__ fx64, unsigned long long* __restrict__ rho_fx) {
    __shared__ double4 sp[kDirectStage];
    const Tile ch = tile_of<ONE>(w);
    const SysDev& S = sys_of<ONE>(w, ch.sys);
    const int l = blockIdx.y * kLTile + threadIdx.x;
    if (blockIdx.y * kLTile >= S.P) return;
    const bool active = l < S.P;
    int4 m = make_int4(0, 0, 0, 0);
    if (active) m = ksamp[S.off_k + l];
    const double tp = 2.0 * M_PI * S.invL;
    const double kx = tp * m.x, ky = tp * m.y, kz = tp * m.z;
    double re = 0.0, im = 0.0;
    for (int base = 0; base < ch.count; base += kDirectStage) {
        const int cnt = min(kDirectStage, ch.count - base);
        __syncthreads();
        for (int t = threadIdx.x; t < cnt; t += blockDim.x) sp[t] = fx64[ch.first + base + t];
        __syncthreads();
        if (active) {
            for (int j = 0; j < cnt; ++j) {
                const double4 p = sp[j];
                const double th = kx * p.x + ky * p.y + kz * p.z;
                double sn, cs;
                sincos(th, &sn, &cs);
                re += p.w * cs;
                im += p.w * sn;
            }
        }
    }
    if (active) rho_accumulate(rho_fx + 2 * (S.off_k + l), re, im, S.rho_scale);
}

// ----------------------------------------------------------------- force
// Block (x, y): particles 8 y .. 8 y + 7 of tile x (kBlockP particles);
// kTabLanes adjacent lanes per particle.  PHI: also dE/dq.
template <bool ONE, bool PHI>
__global__ void __launch_bounds__(kTabThreads)
k_force_f64_tab(const __grid_constant__ Work w, const double4* __restrict__ rec64,
                const int4* __restrict__ ksamp, const double* __restrict__ kcoef,
                const unsigned long long* __restrict__ rho_fx, double4* __restrict__ fs64) {
    extern __shared__ __align__(16) unsigned char smem64[];
    double2* tab = (double2*)smem64;
    __shared__ double2 s_ab[kTabK];                // coef (Im rho, Re rho)
    __shared__ double s_mx[kTabK], s_my[kTabK], s_mz[kTabK];
    __shared__ uint4 s_o[kTabK];                   // table offsets, signs in w
    const Tile tl = tile_of<ONE>(w);
    const SysDev& S = sys_of<ONE>(w, tl.sys);
    const int b0 = blockIdx.y * kTabP;
    const int cnt = min(kTabP, tl.count - b0);
    if (cnt <= 0) return;
    const int mm = batch_mmax(ksamp + S.off_k, S.P), st = mm + 1;
    build_tables(tab, mm, cnt, rec64 + tl.first + b0, S, false);
    pdl_wait();                                     // rho(k)
    const int p = threadIdx.x / kTabLanes, sub = threadIdx.x % kTabLanes;
    const double2* T = tab + 3 * min(p, cnt - 1) * st;
    double fx = 0.0, fy = 0.0, fz = 0.0, ph = 0.0;
    for (int base = 0; base < S.P; base += kTabK) {
        const int nk = min(kTabK, S.P - base);
        if (base > 0) __syncthreads();
        for (int k = threadIdx.x; k < nk; k += kTabThreads) {
            const int l = S.off_k + base + k;
            const int4 m = ksamp[l];
            const double2 r = rho_total(rho_fx + 2 * l, S.rho_stride, S.rho_inv_scale);
            const double c = kcoef[l];
            s_ab[k] = make_double2(c * r.y, c * r.x);
            s_mx[k] = m.x; s_my[k] = m.y; s_mz[k] = m.z;
            s_o[k] = make_uint4(abs(m.x), st + abs(m.y), 2 * st + abs(m.z),
                                (m.x < 0 ? 1u : 0u) | (m.y < 0 ? 2u : 0u) | (m.z < 0 ? 4u : 0u));
        }
        __syncthreads();
        for (int k = sub; k < nk; k += kTabLanes) {
            const uint4 o = s_o[k];
            double2 X = T[o.x], Y = T[o.y], Z = T[o.z];
            X.y = flip(X.y, o.w << 31);
            Y.y = flip(Y.y, (o.w << 30) & 0x80000000u);
            Z.y = flip(Z.y, (o.w << 29) & 0x80000000u);
            // (A + iB) e^{i theta}: the real part is A cos - B sin (force), the
            // imaginary part A sin + B cos (dE/dq)
            const double2 V = cmul(cmul(s_ab[k], X), Y);
            const double g = fma(V.x, Z.x, -(V.y * Z.y));
            fx = fma(g, s_mx[k], fx);
            fy = fma(g, s_my[k], fy);
            fz = fma(g, s_mz[k], fz);
            if constexpr (PHI) ph = fma(V.x, Z.y, fma(V.y, Z.x, ph));
        }
    }
#pragma unroll
    for (int o = kTabLanes / 2; o > 0; o >>= 1) {
        fx += __shfl_down_sync(0xffffffffu, fx, o, kTabLanes);
        fy += __shfl_down_sync(0xffffffffu, fy, o, kTabLanes);
        fz += __shfl_down_sync(0xffffffffu, fz, o, kTabLanes);
        if constexpr (PHI) ph += __shfl_down_sync(0xffffffffu, ph, o, kTabLanes);
    }
    if (sub == 0 && p < cnt) {
        const int i = tl.first + b0 + p;
        const double sc = -rec64[i].w * (2.0 * M_PI * S.invL);
        fs64[i] = make_double4(sc * fx, sc * fy, sc * fz, ph);
    }
}

// Direct form, one thread per particle: where the tables do not fit or do not pay.
template <bool ONE>
__global__ void __launch_bounds__(kBlockP)
k_force_f64(const __grid_constant__ Work w, const double4* __restrict__ rec64,
            const int4* __restrict__ ksamp, const double* __restrict__ kcoef,
            const unsigned long long* __restrict__ rho_fx, double4* __restrict__ fs64) {
    constexpr int kKT = 256;
    __shared__ double4 kk[kKT];     // kx, ky, kz, A
    __shared__ double kb[kKT];      // B
    const Tile tl = tile_of<ONE>(w);
    const SysDev& S = sys_of<ONE>(w, tl.sys);
    const int t = threadIdx.x;
    const bool active = t < tl.count;
    double4 p = make_double4(0, 0, 0, 0);
    if (active) p = rec64[tl.first + t];
    const double tp = 2.0 * M_PI * S.invL;
    double fx = 0, fy = 0, fz = 0, ph = 0;
    for (int base = 0; base < S.P; base += kKT) {
        const int cnt = min(kKT, S.P - base);
        __syncthreads();
        for (int k = threadIdx.x; k < cnt; k += blockDim.x) {
            const int l = S.off_k + base + k;
            const int4 m = ksamp[l];
            const double2 r = rho_total(rho_fx + 2 * l, S.rho_stride, S.rho_inv_scale);
            const double c = kcoef[l];
            kk[k] = make_double4(tp * m.x, tp * m.y, tp * m.z, c * r.y);
            kb[k] = c * r.x;
        }
        __syncthreads();
        if (active) {
            for (int k = 0; k < cnt; ++k) {
                const double4 kv = kk[k];
                const double th = kv.x * p.x + kv.y * p.y + kv.z * p.z;
                double sn, cs;
                sincos(th, &sn, &cs);
                const double B = kb[k];
                const double g = cs * kv.w - sn * B;
                fx += g * kv.x;
                fy += g * kv.y;
                fz += g * kv.z;
                ph += cs * B + sn * kv.w;
            }
        }
    }
    if (active) fs64[tl.first + t] = make_double4(-p.w * fx, -p.w * fy, -p.w * fz, ph);
}

// ------------------------------------------------------------- launchers
// Tables where they fit in a block's shared memory (half width M of the sampler up to
// kTabMaxM) and cost less than a sine and a cosine per pair.  A table's cost grows with
// M (its length and, by the shared memory it takes, the blocks that share an SM), the
// direct form's with P, in whole warps for the structure factors.  Fitted and measured
// (us, table / direct; events around the kernel):
//                             structure factors    force
//   N = 1000, M = 168, P = 5      13 / 38           12 / 13
//   20000, 79, 10                 38 / 52           43 / 31
//   20000, 250, 40               123 / 91          109 / 106
//   140000, 151, 20              406 / 272         448 / 206
//   2^20, 295, 50               5453 / 3749       9838 / 3365
//   2^20, 295, 500             12944 / 29389     25147 / 33453
constexpr int kTabMaxM = 560;               // 8 * 3 * 561 * 16 B = 210 KB

static bool rho_tables_pay(double n, int P, int M) {
    return M <= kTabMaxM && 11.0 + n * (1.9e-5 * M + 1.7e-5 * P) <=
                                30.0 + 1.73e-3 * n * ((P + 31) / 32);
}

static bool force_tables_pay(double n, int P, int M) {
    return M <= kTabMaxM && 8.0 + n * (1.8e-5 * M + 3.6e-5 * P) <= 6.0 + P * (1.1 + 7e-5 * n);
}

template <bool ONE, int KR>
static void rho_f64_kr(cudaStream_t st, const Work& w, dim3 grid, size_t smem, const int4* ksamp,
                       const double4* fx64, unsigned long long* rho_fx) {
    static KernelLimits limits;
    limits.set((const void*)k_rho_f64_tab<ONE, KR>);
    k_rho_f64_tab<ONE, KR><<<grid, kTabThreads, smem, st>>>(w, ksamp, fx64, rho_fx);
}

void launch_rho_f64(cudaStream_t st, bool one, const Work& w, int nchunks, int chunk, int n,
                    int pmax, int mcap, const int4* ksamp, const double4* fx64,
                    unsigned long long* rho_fx) {
    if (nchunks <= 0 || pmax <= 0) return;
    if (!rho_tables_pay(n, pmax, mcap)) {
        dim3 grid(nchunks, (pmax + kLTile - 1) / kLTile);
        if (one) k_rho_f64<true><<<grid, kLTile, 0, st>>>(w, ksamp, fx64, rho_fx);
        else k_rho_f64<false><<<grid, kLTile, 0, st>>>(w, ksamp, fx64, rho_fx);
        return;
    }
    // chunks cut into shares of at least kTabP particles until there are
    // several blocks per SM
    int parts = 1;
    while (parts * kTabP * 2 <= chunk && (long long)nchunks * parts < 152LL * 4) parts <<= 1;
    const int kr = pmax <= kTabThreads ? 1 : (pmax <= 2 * kTabThreads ? 2 : 4);
    dim3 grid(nchunks, parts, (pmax + kTabThreads * kr - 1) / (kTabThreads * kr));
    const size_t sm = tab_smem(mcap);
    if (one) {
        if (kr == 1) rho_f64_kr<true, 1>(st, w, grid, sm, ksamp, fx64, rho_fx);
        else if (kr == 2) rho_f64_kr<true, 2>(st, w, grid, sm, ksamp, fx64, rho_fx);
        else rho_f64_kr<true, 4>(st, w, grid, sm, ksamp, fx64, rho_fx);
    } else {
        if (kr == 1) rho_f64_kr<false, 1>(st, w, grid, sm, ksamp, fx64, rho_fx);
        else if (kr == 2) rho_f64_kr<false, 2>(st, w, grid, sm, ksamp, fx64, rho_fx);
        else rho_f64_kr<false, 4>(st, w, grid, sm, ksamp, fx64, rho_fx);
    }
}

template <bool ONE, bool PHI>
static void force_f64_tab(cudaStream_t st, const Work& w, int nblk, size_t smem,
                          const double4* fx64, const int4* ksamp, const double* kcoef,
                          const unsigned long long* rho_fx, double4* fs64, bool pdl) {
    static KernelLimits limits;
    limits.set((const void*)k_force_f64_tab<ONE, PHI>);
    PdlConfig c(dim3(nblk, kBlockP / kTabP), dim3(kTabThreads), smem, st, pdl);
    cudaLaunchKernelEx(&c.cfg, k_force_f64_tab<ONE, PHI>, w, fx64, ksamp, kcoef, rho_fx, fs64);
}

void launch_fourier_force_f64(cudaStream_t st, bool one, const Work& w, int nblk, int n,
                              int pmax, int mcap, bool phi, const double4* fx64, const int4* ksamp,
                              const double* kcoef, const unsigned long long* rho_fx,
                              double4* fs64, bool pdl) {
    if (nblk <= 0) return;
    if (!force_tables_pay(n, pmax, mcap)) {
        if (one)
            k_force_f64<true><<<nblk, kBlockP, 0, st>>>(w, fx64, ksamp, kcoef, rho_fx, fs64);
        else
            k_force_f64<false><<<nblk, kBlockP, 0, st>>>(w, fx64, ksamp, kcoef, rho_fx, fs64);
        return;
    }
    const size_t sm = tab_smem(mcap);
    if (one) {
        if (phi) force_f64_tab<true, true>(st, w, nblk, sm, fx64, ksamp, kcoef, rho_fx, fs64, pdl);
        else force_f64_tab<true, false>(st, w, nblk, sm, fx64, ksamp, kcoef, rho_fx, fs64, pdl);
    } else {
        if (phi) force_f64_tab<false, true>(st, w, nblk, sm, fx64, ksamp, kcoef, rho_fx, fs64, pdl);
        else force_f64_tab<false, false>(st, w, nblk, sm, fx64, ksamp, kcoef, rho_fx, fs64, pdl);
    }
}

}  // namespace rbe
