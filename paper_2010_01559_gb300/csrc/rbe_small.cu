// rbe_small.cu -- MD steps of a small system in one launch: one thread-block
// cluster runs all the steps of a call.
//
// What bounds a step of a few hundred to a few thousand particles is latency:
// as separate kernels it is nine dependent launches of about 2 us each for
// well under a microsecond of arithmetic.  Here the sixteen blocks of a
// cluster keep the whole system in their shared memory and exchange it twice
// per step with asynchronous remote stores that complete on an mbarrier of the
// receiving block (no cluster-wide barrier in the loop):
//
//   records    rank c owns n/16 particles (position, velocity and build record
//              stay in registers of one thread each for the whole call); the
//              block sends their fixed-point records to all ranks
//   k-batch    rank c holds P/16 wave vectors, drawn a step ahead; each warp sums the structure factors of two of them
//              over a share of all n records (no sum crosses blocks); then a
//              warp per wave vector adds the shares, forms the force
//              coefficient and sends it to all ranks
//   pairs      meanwhile R lanes per owned particle walk its neighbour list,
//              then (coefficients in) its wave vectors; the particle's thread
//              applies the thermostat.  (A lane per particle with a warp per
//              share of the wave vectors reads a coefficient once per warp, but
//              needs another pass to add the shares: 7.2 against 7.0 us at
//              N = 1000, P = 100, 12.5 against 13.5 at P = 500.)
//
// A block that runs ahead cannot overwrite what another still reads, nor count
// on a barrier phase that has not begun: to send the records of step s + 1 it
// needs every rank's coefficients of step s, to send coefficients every rank's
// records (a rank without particles or wave vectors sends a message all the
// same), and the records alternate between two buffers.
//
// Serial chains are what counts.  FP64 instructions are kept out of the loop but for
// the Nose-Hoover friction and kinetic energies (their latency on this part is over a
// hundred cycles; summing a wave vector's shares and its coefficient in FP64 took 3500
// to 10700 cycles a step); one thread sending to 16 ranks in turn or adding 32 partial
// forces took 1200 to 4000, which a thread per message and shuffles take to a few
// hundred.  Partial sums are added as float pairs, and the coefficient
// (lB S/P 4 pi / V) / k^2 is a float-pair constant over the integer |m|^2.
//
// Neighbour list: the owned particles' neighbours within r_c + skin as 16-bit
// caller indices in shared memory, read from the handle's list when that
// stands and rebuilt (all pairs, in ascending order) when a particle has moved
// more than skin/2 since the build, which also writes the handle's list
// arrays (in the caller's order: perm is the identity).  List, displacement
// test and build count thus carry over between calls and to the other paths
// of the handle.
//
// Measured (us per step, 64 steps in a call, replayed kernels before -> now):
// N = 300, P = 10 15.4 -> 4.1; N = 1000, P = 100 16.3 -> 6.5 and P = 500 18.3 -> 14.0;
// N = 2000, P = 100 16.3 -> 9.5.
// A call costs about 10 us beside its steps (the cluster's launch, the list taken over,
// a first pass through the code), the price of a path that does not depend on how many
// steps a call has (calls of any length give the same bits).  One step per call, back to
// back, replayed kernels before -> now: N = 300, P = 10 14.4 -> 13.6; 1000, 100 16.8 -> 16.9;
// 2000, 100 20.6 -> 21.2; 3000, 10 18.6 -> 20.8 (22.7 with the list's entries taken over one
// by one); 1000, 500 20.6 -> 25.1.
#include <algorithm>

#include "rbe_cluster.cuh"
#include "rbe_internal.cuh"
#include "rbe_pair.cuh"

namespace rbe {

constexpr int kSmallThreads = 1024;
constexpr int kSmallWarps = kSmallThreads / 32;

// 16 bytes into a block's shared memory, counted on that block's mbarrier
__device__ __forceinline__ void send(uint32_t dst, const uint4& v, uint32_t bar) {
    asm volatile(
        "st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.u32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(
            dst),
        "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w), "r"(bar)
        : "memory");
}
__device__ __forceinline__ void bar_init(uint32_t bar) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar) : "memory");
}
// this phase of the barrier completes when `bytes` have come in
__device__ __forceinline__ void bar_expect(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ unsigned long long now_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
// Whether the phase of the given parity has completed, at once (test_wait) or after a
// wait of the hardware's choosing (try_wait).
template <bool TEST>
__device__ __forceinline__ bool bar_poll(uint32_t bar, uint32_t parity) {
    uint32_t done;
    if constexpr (TEST)
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(done)
            : "r"(bar), "r"(parity)
            : "memory");
    else
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(done)
            : "r"(bar), "r"(parity)
            : "memory");
    return done != 0u;
}
// Waits for the phase of the given parity, limit_ns at most (a step takes
// microseconds; 0: one look): false if it did not complete.
__device__ __forceinline__ bool bar_wait(uint32_t bar, uint32_t parity,
                                         unsigned long long limit_ns) {
    if (limit_ns == 0ull) return bar_poll<true>(bar, parity);
    unsigned long long t0 = 0ull;
    for (unsigned t = 0;; ++t) {
        if (bar_poll<false>(bar, parity)) return true;
        if ((t & 63u) == 0u) {
            const unsigned long long now = now_ns();
            if (t == 0u) t0 = now;
            else if (now - t0 > limit_ns) return false;
        }
    }
}

constexpr float kTurn = 1.4629180792671596e-09f;                     // 2 pi / 2^32
constexpr int kSmallMaxKc = 2 * kSmallWarps;                         // wave vectors per rank
constexpr int kSmallMaxCs = 16;                                      // blocks per cluster

// Shared-memory layout of a block (byte offsets, 16-byte aligned).
struct SmallLayout {
    int np, kc, tab;             // owned particles, wave vectors per rank, table entries
    size_t rec, kv, own, frc, list, table, end;
};

__host__ __device__ inline size_t small_align(size_t x) { return (x + 15) & ~size_t(15); }

__host__ __device__ inline SmallLayout small_layout(int n, int P, int M, int cap, int cs) {
    SmallLayout L;
    L.np = (n + cs - 1) / cs;
    L.kc = (P + cs - 1) / cs;
    L.tab = 2 * M + 1;
    L.rec = 0;                                                       // uint4 [2][n]
    L.kv = L.rec + 32 * (size_t)n;                                   // uint4 [2][P]
    L.own = L.kv + 32 * (size_t)P;                                   // uint4 [np]
    L.frc = L.own + 16 * (size_t)L.np;                               // float4 [np]
    L.list = L.frc + 16 * (size_t)L.np;                              // u16 [np][cap]
    L.table = L.list + small_align(2 * (size_t)L.np * cap);          // u32 [2M + 1]
    L.end = L.table + small_align(4 * (size_t)L.tab);
    return L;
}

// A warp's structure factors: FP32 chains per lane, then the lanes' sums.  Their
// rounding is kept at that of chains of 16 terms added exactly, a variance of 8 n in
// units of one term's (c / 2 per term of a chain of c, one per term and level of a
// sum of the lanes).  Up to kSmallPlain terms per lane an FP32 sum over the five levels
// stays at it, (6 / 2 + 5) n; beyond, the lanes' sums are float pairs, of chains of
// kSmallChain terms at most.  Fourier force against 64 bits (RMS, 16 to 24 systems),
// FP32 sums throughout / now: N = 2000, P = 100 2.83e-7 / 2.74e-7; 1150, 500 3.25e-7 /
// 3.14e-7; 890, 1000 2.88e-7 / 2.72e-7.
constexpr int kSmallPlain = 6, kSmallChain = 16;

__device__ __forceinline__ float sum_of(float a, float b) { return a + b; }
__device__ __forceinline__ float2 sum_of(float2 a, float2 b) {
    const float2 x = two_sum(a.x, b.x);
    return make_float2(x.x, a.y + b.y + x.y);
}
__device__ __forceinline__ float lane_xor(float v, int d) {
    return __shfl_xor_sync(0xffffffffu, v, d);
}
__device__ __forceinline__ float2 lane_xor(float2 v, int d) {
    return make_float2(lane_xor(v.x, d), lane_xor(v.y, d));
}
// Four sums over the warp, halving the values with the lanes: lanes 0, 8, 16, 24 end
// with re0, im0, re1, im1.
template <class V>
__device__ __forceinline__ V warp_sum4(V re0, V im0, V re1, V im1, int lane) {
    const bool up = lane & 16, up2 = lane & 8;
    const V a = sum_of(up ? re1 : re0, lane_xor(up ? re0 : re1, 16));
    const V b = sum_of(up ? im1 : im0, lane_xor(up ? im0 : im1, 16));
    V v = sum_of(up2 ? b : a, lane_xor(up2 ? a : b, 8));
    v = sum_of(v, lane_xor(v, 4));
    v = sum_of(v, lane_xor(v, 2));
    return sum_of(v, lane_xor(v, 1));
}

// (ch + cl) (h + l) to FP32
__device__ __forceinline__ float pair_mul(float ch, float cl, float2 v) {
    const float p = __fmul_rn(ch, v.x);
    return __fadd_rn(p, fmaf(ch, v.x, -p) + fmaf(ch, v.y, cl * v.x));
}

// Samples la and lb of the step's k-batch (as sample_one_smem draws them), by a
// whole warp: six lanes look up one axis of one sample each.
__device__ __forceinline__ void warp_sample2(const SysDev& S, const uint32_t* T, int la, int lb,
                                             uint64_t step, int* err, int4& ma, int4& mb) {
    const int lane = threadIdx.x & 31, ax = lane % 3;
    const uint2 key = make_uint2((uint32_t)S.seed, (uint32_t)(S.seed >> 32));
    bool oka = false, okb = false;
    for (int a = 0; a < kMaxAttempts && !(oka && okb); ++a) {
        const uint4 w = philox4x32_10(make_uint4((uint32_t)(lane < 3 ? la : lb), (uint32_t)a,
                                                 (uint32_t)step, (S.stream << 8) | 0x01u), key);
        const uint32_t u = ax == 0 ? w.x : (ax == 1 ? w.y : w.z);
        int lo = 0, hi = 2 * S.M;                   // smallest j with u < T[j]
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if (u < T[mid]) hi = mid; else lo = mid + 1;
        }
        const int v = lo - S.M;
        const int x0 = __shfl_sync(0xffffffffu, v, 0), y0 = __shfl_sync(0xffffffffu, v, 1),
                  z0 = __shfl_sync(0xffffffffu, v, 2), x1 = __shfl_sync(0xffffffffu, v, 3),
                  y1 = __shfl_sync(0xffffffffu, v, 4), z1 = __shfl_sync(0xffffffffu, v, 5);
        if (!oka) { ma = make_int4(x0, y0, z0, a + 1); oka = (x0 | y0 | z0) != 0; }
        if (!okb) { mb = make_int4(x1, y1, z1, a + 1); okb = (x1 | y1 | z1) != 0; }
    }
    if (!oka) ma = make_int4(1, 0, 0, kMaxAttempts + 1);
    if (!okb) mb = make_int4(1, 0, 0, kMaxAttempts + 1);
    if (!(oka && okb) && lane == 0) atomicOr(err, kErrSampler);
}

template <int R>
__global__ void __launch_bounds__(kSmallThreads, 1) k_small_md(const __grid_constant__ SmallArgs a) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ __align__(8) unsigned long long s_bar[2];        // records in, coefficients in
    __shared__ float2 s_part[kSmallWarps][4];                   // structure-factor partials (pairs)
    __shared__ int4 s_m[2][kSmallMaxKc];                        // this rank's wave vectors and
    __shared__ float2 s_c[2][kSmallMaxKc];                      // (float pairs) coef / rho, by parity
    __shared__ uint4 s_token;                                   // from ranks without wave vectors
    // from every rank, by step parity: (flags, 0, Nose-Hoover kinetic sum); flags:
    // 1 a particle moved beyond half the skin, 2 non-finite input
    __shared__ uint4 s_msg[2][kSmallMaxCs];
    __shared__ unsigned long long s_k2;                         // this rank's kinetic sum
    __shared__ int s_flags[2];                                  // its flags, by step parity
    __shared__ int s_late[kSmallMaxCs];                         // the ranks that gave up
    const SysDev& S = a.S;
    const uint32_t rank = cluster_rank();
    const int cs = a.cs, n = a.n, P = S.P, tid = threadIdx.x;
    const int lane = tid & 31, warp = tid >> 5;
    const SmallLayout L = small_layout(n, P, S.M, a.cap, cs);
    uint4* rec = (uint4*)(smem + L.rec);
    uint4* kv = (uint4*)(smem + L.kv);              // [l]: -m and phi; [P + l]: R m and R
    uint4* own = (uint4*)(smem + L.own);            // owned records, to be sent
    float4* frc = (float4*)(smem + L.frc);          // owned particles' total forces
    uint16_t* list = (uint16_t*)(smem + L.list);
    uint32_t* table = (uint32_t*)(smem + L.table);
    const int first = (int)rank * L.np;
    const int np = max(0, min(L.np, n - first));    // owned particles (caller's order)
    const int k0 = (int)rank * L.kc;
    const int nk = max(0, min(L.kc, P - k0));       // owned wave vectors
    const bool nhm = S.thermostat == RBE_THERMO_NOSE_HOOVER;
    const bool owner = tid < np;                    // thread tid closes particle first + tid
    const int o = first + tid;
    const int p = tid / R, l = tid % R;             // pair lanes: particle p, lane l of R
    const bool pairs = p < np;
    const int pn = first + p;
    const uint32_t bar_rec = local_addr(&s_bar[0]), bar_kv = local_addr(&s_bar[1]);
    const uint64_t step0 = *a.step_dev;
    const bool stale = *a.list_flag != 0;           // the handle's list does not stand
    float4 pos = make_float4(0.f, 0.f, 0.f, 0.f), vel = pos;
    uint4 ref = make_uint4(0, 0, 0, 0);
    if (owner) {
        pos = a.pos[o];
        vel = a.vel[o];
        ref = a.sref[o];
    }
    for (int j = tid; j < L.tab; j += kSmallThreads) table[j] = (uint32_t)a.table[j];
    if (tid < 2 * kSmallMaxCs) (&s_msg[0][0])[tid] = make_uint4(0, 0, 0, 0);
    int cnt = 0;                                    // list entries of particle p
    if (pairs && !stale) {
        // the handle's list, in sorted indices of its last build: kTake entries per lane
        // in flight at a time, the first ones alongside the count (slots within the
        // capacity always hold valid indices)
        constexpr int kTake = 8;
        const int i = a.iperm[pn];
        if (RBE_IN_BOUNDS(i, a.stride, a.err)) {
            const int* nb = a.nbr + i;
            int j[kTake], c[kTake];
            const int have = a.ncnt[i];
#pragma unroll
            for (int u = 0; u < kTake; ++u) {
                const int k = l + u * R;
                j[u] = k < a.cap ? nb[(size_t)k * a.stride] : 0;
            }
            cnt = min(have, a.cap);
            for (int k0 = l; k0 < cnt; k0 += kTake * R) {
                if (k0 > l) {
#pragma unroll
                    for (int u = 0; u < kTake; ++u) {
                        const int k = k0 + u * R;
                        j[u] = k < cnt ? nb[(size_t)k * a.stride] : 0;
                    }
                }
#pragma unroll
                for (int u = 0; u < kTake; ++u)
                    c[u] = RBE_IN_BOUNDS(j[u], a.stride, a.err) ? a.perm[j[u]] : pn;
#pragma unroll
                for (int u = 0; u < kTake; ++u) {
                    const int k = k0 + u * R;
                    if (k < cnt)
                        list[p * a.cap + k] = (uint16_t)(RBE_IN_BOUNDS(c[u], n, a.err) ? c[u] : pn);
                }
            }
        }
    }
    NhState nh{};
    if (nhm) nh = *a.nh;
    if (tid == 0) {
        s_k2 = 0ull;
        s_flags[0] = s_flags[1] = 0;
        bar_init(bar_rec);
        bar_init(bar_kv);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    cluster_sync();                                 // every rank's barriers are initialised

    const int kp = (nk + 1) / 2;                    // pairs of wave vectors, a group of warps each
    const int wpp = kp > 0 ? kSmallWarps / kp : 0;
    const bool sums = warp < kp * wpp;              // this warp sums pair pr, share sub of wpp
    const int pr = sums ? warp % kp : 0, sub = sums ? warp / kp : 0;
    // bytes a block receives per step: all records and a message from every rank
    const uint32_t rec_bytes = 16u * (uint32_t)(n + cs);
    const uint32_t kv_bytes = 32u * (uint32_t)P + 16u * (uint32_t)(cs - (P + L.kc - 1) / L.kc);
    // the k-batch of a step: a warp per pair of wave vectors, from warp w0 on
    auto draw = [&](uint64_t step, int w0) {
        const int u = warp - w0;
        if (u < 0 || u >= kp) return;
        const int q = 2 * u, b = (int)(step & 1);
        int4 m0, m1;
        warp_sample2(S, table, k0 + q, k0 + min(q + 1, nk - 1), step, a.err, m0, m1);
        if (lane < 2) {
            // c = coefficient scale / |m|^2 as a float pair (|m|^2 is exact)
            const int4 m = lane ? m1 : m0;
            const float m2 = (float)(m.x * m.x + m.y * m.y + m.z * m.z);
            const float ch = a.kscale_hi / m2;
            s_m[b][q + lane] = m;
            s_c[b][q + lane] =
                make_float2(ch, (fmaf(-ch, m2, a.kscale_hi) + a.kscale_lo) / m2);
        }
    };
    // (the warps below those that form the coefficients: the last ones hold few
    // particles or none)
    const int w_draw = max(0, kSmallWarps - min(nk, kSmallWarps) - kp);
    draw(step0, w_draw);
    // where this thread's first record of every step goes
    const int q_snd = np > 0 ? tid % np : 0, t_snd = np > 0 ? tid / np : 0;
    const uint32_t rec_snd = remote(local_addr(rec + first + q_snd), min(t_snd, cs - 1));
    const uint32_t bar_snd = remote(bar_rec, min(t_snd, cs - 1));
    bool bad_seen = false;                          // some position or charge was not finite
    bool gave_up = false;                           // a wait of this block ran out

    for (int s = 0; s < a.nsteps; ++s) {
        const uint64_t step = step0 + (uint64_t)s;
        uint4* R_ = rec + (s & 1) * n;              // this step's records
        const uint32_t par = (uint32_t)(s & 1);
        if (tid == 0) {
            bar_expect(bar_rec, rec_bytes);
            bar_expect(bar_kv, kv_bytes);
        }
        // ---- fixed-point records and displacement test, to every rank
        uint4 cur = make_uint4(0, 0, 0, 0);
        int flags = 0;
        if (owner) {
            cur = make_uint4(to_fixed(pos.x, S.fx_hi, S.fx_lo), to_fixed(pos.y, S.fx_hi, S.fx_lo),
                             to_fixed(pos.z, S.fx_hi, S.fx_lo), __float_as_uint(pos.w));
            own[tid] = cur;
            const float dx = (float)(int32_t)(cur.x - ref.x) * S.L_over_2_32;
            const float dy = (float)(int32_t)(cur.y - ref.y) * S.L_over_2_32;
            const float dz = (float)(int32_t)(cur.z - ref.z) * S.L_over_2_32;
            if ((s == 0 && stale) || fmaf(dx, dx, fmaf(dy, dy, dz * dz)) > S.f_half_skin2)
                flags = 1;
            if (!(isfinite(pos.x) && isfinite(pos.y) && isfinite(pos.z) && isfinite(pos.w))) {
                flags |= 2;
                atomicOr(a.err, kErrNonfinite);
            }
        }
        if (flags) atomicOr(&s_flags[par], flags);
        __syncthreads();                            // own, s_flags, s_k2
        if (tid < np * cs) send(rec_snd + 16u * (uint32_t)(par * n), own[q_snd], bar_snd);
        for (int e = tid + kSmallThreads; e < np * cs; e += kSmallThreads) {
            const int t = e / np, q = e - t * np;
            send(remote(local_addr(R_ + first + q), t), own[q], remote(bar_rec, t));
        }
        if (warp == kSmallWarps / 2) {
            // one message to every rank, from a warp of the middle (the first
            // ones own particles, the last ones draw wave vectors)
            const unsigned long long k2 = s_k2;
            if (lane < cs)
                send(remote(local_addr(&s_msg[par][rank]), lane),
                     make_uint4((uint32_t)s_flags[par], 0u, (uint32_t)k2, (uint32_t)(k2 >> 32)),
                     remote(bar_rec, lane));
        }
        const bool rec_in = bar_wait(bar_rec, par, a.wait_ns);
        const uint32_t seen = __reduce_or_sync(0xffffffffu, lane < cs ? s_msg[par][lane].x : 0u);
        const bool rebuild = (seen & 1u) != 0u;
        bad_seen |= (seen & 2u) != 0u;
        // ---- structure factors of two wave vectors over a share of all records
        if (sums) {
            const int4 m0 = s_m[step & 1][2 * pr], m1 = s_m[step & 1][2 * pr + 1];
            const int stride = wpp * 32, j0 = sub * 32 + lane;
            // the sums of a lane's records j0 .. je - 1 (every stride-th): q cos, q sin of
            // both wave vectors
            auto chain = [&](int jb, int je) {
                float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 4
                for (int j = jb; j < je; j += stride) {
                    const uint4 r = R_[j];
                    const float q = __uint_as_float(r.w);
                    float sn, cn;
                    __sincosf((float)(int32_t)((uint32_t)m0.x * r.x + (uint32_t)m0.y * r.y +
                                               (uint32_t)m0.z * r.z) * kTurn, &sn, &cn);
                    a.x = fmaf(q, cn, a.x);
                    a.y = fmaf(q, sn, a.y);
                    __sincosf((float)(int32_t)((uint32_t)m1.x * r.x + (uint32_t)m1.y * r.y +
                                               (uint32_t)m1.z * r.z) * kTurn, &sn, &cn);
                    a.z = fmaf(q, cn, a.z);
                    a.w = fmaf(q, sn, a.w);
                }
                return a;
            };
            float2 v;
            if (n <= kSmallPlain * stride) {
                const float4 a = chain(j0, n);
                v = make_float2(warp_sum4(a.x, a.y, a.z, a.w, lane), 0.f);
            } else {
                float2 re0{}, im0{}, re1{}, im1{};
                for (int jb = j0; jb < n; jb += kSmallChain * stride) {
                    const float4 a = chain(jb, min(n, jb + kSmallChain * stride));
                    re0 = sum_of(re0, make_float2(a.x, 0.f));
                    im0 = sum_of(im0, make_float2(a.y, 0.f));
                    re1 = sum_of(re1, make_float2(a.z, 0.f));
                    im1 = sum_of(im1, make_float2(a.w, 0.f));
                }
                v = warp_sum4(re0, im0, re1, im1, lane);
            }
            if ((lane & 7) == 0) s_part[sub * kp + pr][lane >> 3] = v;
        }
        if (__syncthreads_or(!rec_in)) {            // the whole block leaves the steps, before
            gave_up = true;                         // it uses or sends anything of this one
            break;
        }
        if (tid == 0) {                             // (read above, written after the next barrier)
            s_k2 = 0ull;
            s_flags[par] = 0;
        }
        // ---- a warp per wave vector: its force coefficient, to every rank
        for (int q = kSmallWarps - 1 - warp; q < nk; q += kSmallWarps) {
            // lanes 0-15 add the shares' real parts, lanes 16-31 the imaginary
            // ones, as float pairs
            const int u = lane & 15, c = (q & 1) * 2 + (lane >> 4);
            float2 v = make_float2(0.f, 0.f);
            if (u < wpp) v = s_part[u * kp + (q >> 1)][c];
            if (u + 16 < wpp) v = sum_of(v, s_part[(u + 16) * kp + (q >> 1)][c]);
#pragma unroll
            for (int d = 8; d > 0; d >>= 1) v = sum_of(v, lane_xor(v, d));
            const int4 m = s_m[step & 1][q];
            const float2 cf = s_c[step & 1][q];
            const float AB = pair_mul(cf.x, cf.y, v);
            const float A = __shfl_sync(0xffffffffu, AB, 16), B = __shfl_sync(0xffffffffu, AB, 0);
            const float Rk = hypotf(A, B);
            // phi in 2^-32 turns; half a turn is 2^31 (the conversion saturates below it)
            const float turns = atan2f(A, B) * 0.15915494309189535f * 4294967296.0f;
            const uint32_t phi =
                turns >= 2147483648.0f ? 0x80000000u : (uint32_t)__float2int_rn(turns);
            const uint4 x = make_uint4(0u - (uint32_t)m.x, 0u - (uint32_t)m.y, 0u - (uint32_t)m.z,
                                       phi);
            const uint4 y = make_uint4(__float_as_uint(Rk * (float)m.x),
                                       __float_as_uint(Rk * (float)m.y),
                                       __float_as_uint(Rk * (float)m.z), __float_as_uint(Rk));
            const int t = lane & 15;                // lanes 0-15 send x, 16-31 send y
            if (t < cs)
                send(remote(local_addr(kv + (lane < 16 ? 0 : P) + k0 + q), t), lane < 16 ? x : y,
                     remote(bar_kv, t));
        }
        if (s + 1 < a.nsteps) draw(step + 1, w_draw);   // the next step's wave vectors
        MdNoise z{0.f, 0.f, 0.f, false};
        if (owner && !nhm) z = md_noise(S, step, o);
        if (nk == 0 && tid == 0)
            for (int t = 0; t < cs; ++t)
                send(remote(local_addr(&s_token), t), make_uint4(0u, 0u, 0u, 0u),
                     remote(bar_kv, t));
        if (nhm && owner) {
            // the friction, from the kinetic sums the messages carried
            unsigned long long k2 = 0ull;
            for (int t = 0; t < cs; ++t) {
                const uint4 v = s_msg[par][t];
                k2 += (unsigned long long)v.z | ((unsigned long long)v.w << 32);
            }
            if (s > 0) nh.k2 = k2;
            if (!nh.first) nh.xi += S.nh_rate * ((double)nh.k2 * 0x1p-32 - 3.0 * (double)S.n);
            nh.first = 0;
            const double hx = 0.5 * nh.xi * S.dt;
            nh.a = 1.0 - hx;
            nh.b = 1.0 / (1.0 + hx);
            nh.f_va = (float)(nh.a * nh.b);
            nh.f_vf = (float)(S.dt_over_m * nh.b);
        }
        // ---- the list, rebuilt if any particle moved beyond half the skin
        if (rebuild) {
            const uint4 si = R_[min(pn, n - 1)];
            cnt = 0;
            // 32 candidates per lane at a time, then the lanes' hits one after another
            for (int jb = l; jb < n + l; jb += 32 * R) {
                uint32_t bits = 0;
                if (pairs)
                    for (int b = 0, j = jb; b < 32 && j < n; ++b, j += R) {
                        const uint4 sj = R_[j];
                        const float dx = (float)(int32_t)(sj.x - si.x) * S.L_over_2_32;
                        const float dy = (float)(int32_t)(sj.y - si.y) * S.L_over_2_32;
                        const float dz = (float)(int32_t)(sj.z - si.z) * S.L_over_2_32;
                        const float r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
                        if (r2 < S.f_list_cut2 && j != pn) bits |= 1u << b;
                    }
                int incl = __popc(bits), slot = cnt - incl;
#pragma unroll
                for (int d = 1; d < R; d <<= 1) {
                    const int y = __shfl_up_sync(0xffffffffu, incl, d, R);
                    if (l >= d) incl += y;
                }
                slot += incl;
                cnt += __shfl_sync(0xffffffffu, incl, R - 1, R);
                for (; bits; bits &= bits - 1, ++slot) {
                    const int j = jb + (__ffs(bits) - 1) * R;
                    if (slot < a.cap) {
                        list[p * a.cap + slot] = (uint16_t)j;
                        a.nbr[(size_t)slot * a.stride + pn] = j;
                    }
                }
            }
            if (pairs && l == 0) {
                a.ncnt[pn] = min(cnt, a.cap);
                // (non-finite input has its own error; its neighbour counts mean nothing)
                if (cnt > a.cap && !bad_seen) atomicOr(a.err, kErrList);
                atomicMax(a.stats + 1, (unsigned long long)cnt);
            }
            cnt = min(cnt, a.cap);
            if (owner) {
                ref = cur;
                a.sref[o] = cur;
                a.perm[o] = o;
                a.iperm[o] = o;
            }
            if (rank == 0 && tid == 0) atomicAdd(a.stats, 1ull);
            __syncwarp();
        }
        // ---- real-space pairs
        float fx = 0.f, fy = 0.f, fz = 0.f;
        if (pairs) {
            Pair2Acc acc{0ull, 0ull, 0ull, 0.f, 0.f, 0.f};
            const uint4 si = R_[pn];
            auto rec_of = [&](int k) {              // (the particle itself is no pair)
                const int j = list[p * a.cap + k];
                return RBE_IN_BOUNDS(j, n, a.err) ? R_[j] : si;
            };
            for (int k = l; k < cnt; k += 2 * R) {
                const uint4 sb = k + R < cnt ? rec_of(k + R) : si;
                pair2_fixed(si, rec_of(k), sb, S, acc);
            }
            const float3 f = pair2_force(acc, si, S);
            fx = f.x;
            fy = f.y;
            fz = f.z;
        }
        // ---- Fourier force
        const bool kv_in = bar_wait(bar_kv, par, a.wait_ns);
        if (pairs) {
            const uint4 si = R_[pn];
            float gx = 0.f, gy = 0.f, gz = 0.f;
#pragma unroll 4
            for (int k = l; k < P; k += R) {
                const uint4 A = kv[k], B = kv[P + k];
                const uint32_t d = A.w + A.x * si.x + A.y * si.y + A.z * si.z;
                const float sn = __sinf((float)(int32_t)d * kTurn);
                gx = fmaf(sn, __uint_as_float(B.x), gx);
                gy = fmaf(sn, __uint_as_float(B.y), gy);
                gz = fmaf(sn, __uint_as_float(B.z), gz);
            }
            const float sc = -__uint_as_float(si.w) * (float)(2.0 * M_PI) * S.f_invL;
            fx = fmaf(sc, gx, fx);
            fy = fmaf(sc, gy, fy);
            fz = fmaf(sc, gz, fz);
        }
#pragma unroll
        for (int d = R / 2; d > 0; d >>= 1) {
            fx += __shfl_down_sync(0xffffffffu, fx, d, R);
            fy += __shfl_down_sync(0xffffffffu, fy, d, R);
            fz += __shfl_down_sync(0xffffffffu, fz, d, R);
        }
        if (pairs && l == 0) frc[p] = make_float4(fx, fy, fz, 0.f);
        if (__syncthreads_or(!kv_in)) {
            gave_up = true;
            break;
        }
        // ---- thermostat and drift
        if (warp * 32 < np) {
            unsigned long long k2 = 0ull;
            if (owner) {
                const float4 F = frc[tid];
                if (nhm) k2 = nose_hoover_apply(S, nh.f_va, nh.f_vf, F.x, F.y, F.z, vel, pos);
                else md_apply(S, z, F.x, F.y, F.z, vel, pos);
            }
            if (nhm) {
                for (int d = 16; d > 0; d >>= 1) k2 += __shfl_xor_sync(0xffffffffu, k2, d);
                if (lane == 0) atomicAdd(&s_k2, k2);
            }
        }
    }
    // the last step's kinetic sums, for the friction of the next call (slots
    // of the parity that no rank reads any more), and whether this rank gave up
    __syncthreads();
    if (nhm && tid == 0) {
        const uint32_t d = remote(local_addr(&s_msg[a.nsteps & 1][rank]), 0);
        asm volatile("st.shared::cluster.v2.u32 [%0], {%1, %2};" ::"r"(d + 8u),
                     "r"((uint32_t)s_k2), "r"((uint32_t)(s_k2 >> 32))
                     : "memory");
    }
    if (tid < cs)
        asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(
                         remote(local_addr(&s_late[rank]), (uint32_t)tid)),
                     "r"((int)gave_up)
                     : "memory");
    cluster_sync();
    int any = 0;
    for (int t = 0; t < cs; ++t) any |= s_late[t];
    if (!any) {
        if (owner) {
            a.pos[o] = pos;
            a.vel[o] = vel;
            if (a.F_out) a.F_out[o] = frc[tid];
        }
    } else if (tid == 0) {
        // some rank gave up: none stores its state.  No rank sends any more; what is
        // still under way to this one lands before the block goes
        const unsigned long long t0 = now_ns();
        while (now_ns() - t0 < 100000ull) {
        }
    }
    if (a.done_host) __threadfence_system();        // this thread's outputs
    // orders those stores, and keeps every rank's shared memory alive until all are done
    cluster_sync();
    if (rank == 0 && tid == 0) {
        if (any) {
            // positions, velocities, friction and step index stay as they were; the
            // list may have been rebuilt in part
            atomicOr(a.err, kErrWait);
            *a.list_flag = 1;
        } else {
            if (nhm) {
                unsigned long long k2 = 0ull;
                for (int t = 0; t < cs; ++t) {
                    const uint4 v = s_msg[a.nsteps & 1][t];
                    k2 += (unsigned long long)v.z | ((unsigned long long)v.w << 32);
                }
                nh.k2 = k2;
                *a.nh = nh;
            }
            *a.list_flag = 0;
            *a.step_dev = step0 + (uint64_t)a.nsteps;
        }
        if (a.done_host) {
            __threadfence_system();
            *(volatile int*)a.err_host = *(const volatile int*)a.err;
            __threadfence_system();
            *(volatile unsigned long long*)a.done_host = a.done_value;
        }
    }
}

// Lanes per particle: as many as 1024 threads allow.
static int small_lanes(int n, int cs) {
    const int np = (n + cs - 1) / cs;
    int r = 32;
    while (r > 4 && np * r > kSmallThreads) r >>= 1;
    return r;
}

template <int R>
static cudaError_t small_config(cudaLaunchConfig_t& cfg, cudaLaunchAttribute* attr, cudaStream_t st,
                         int cs, size_t smem) {
    cfg = cudaLaunchConfig_t{};
    cfg.gridDim = dim3(cs);
    cfg.blockDim = dim3(kSmallThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = cs;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    static KernelLimits limits;
    return limits.set((const void*)k_small_md<R>, true);
}

template <int R>
static bool small_fits(int cs, size_t smem) {
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr[1];
    int clusters = 0;
    const bool ok = small_config<R>(cfg, attr, nullptr, cs, smem) == cudaSuccess &&
                    cudaOccupancyMaxActiveClusters(&clusters, k_small_md<R>, &cfg) == cudaSuccess;
    if (!ok) cudaGetLastError();
    return ok && clusters >= 1;
}

// Whether a system of n particles, P wave vectors, half width M and cap list
// entries per particle runs as one cluster: it fits in the blocks' shared memory and the GPU can place the
// cluster.  cs: blocks of the cluster.
bool small_md_fits(int n, int P, int M, int cap, int cs) {
    const int R = small_lanes(n, cs);
    if (n < 1 || (n + cs - 1) / cs * R > kSmallThreads) return false;
    if ((P + cs - 1) / cs > kSmallMaxKc || cs > kSmallMaxCs || M > 2000) return false;
    const size_t smem = small_layout(n, P, M, cap, cs).end;
    if (smem > 216 * 1024) return false;
    switch (R) {
        case 4: return small_fits<4>(cs, smem);
        case 8: return small_fits<8>(cs, smem);
        case 16: return small_fits<16>(cs, smem);
        default: return small_fits<32>(cs, smem);
    }
}

template <int R>
static cudaError_t small_launch(cudaStream_t st, const SmallArgs& a, size_t smem) {
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr[1];
    const cudaError_t e = small_config<R>(cfg, attr, st, a.cs, smem);
    if (e != cudaSuccess) return e;
    return cudaLaunchKernelEx(&cfg, k_small_md<R>, a);
}

cudaError_t launch_small_md(cudaStream_t st, const SmallArgs& a) {
    const int R = small_lanes(a.n, a.cs);
    const size_t smem = small_layout(a.n, a.S.P, a.S.M, a.cap, a.cs).end;
    switch (R) {
        case 4: return small_launch<4>(st, a, smem);
        case 8: return small_launch<8>(st, a, smem);
        case 16: return small_launch<16>(st, a, smem);
        default: return small_launch<32>(st, a, smem);
    }
}

}  // namespace rbe
