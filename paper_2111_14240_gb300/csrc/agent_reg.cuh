// The fused agent sweep (steps S0-S5 of one PMACE iteration, the arithmetic
// of agent.cuh) with whole windows in registers.
//
// A thread holds 32 complex values, so 512 threads (16 warps of 128
// registers a thread, all that an SM holds) hold one 128 x 128 window, four
// 64 x 64 windows or sixteen 32 x 32 windows.  128 x 128 and 64 x 64 windows
// take a CTA each, 32 x 32 windows a warp (see the end of this file).
//
// A 2-D DFT of 128 x 128 has 14 binary levels; a thread's values cover five
// at a time, so the forward transform takes three register passes and two
// exchanges through shared memory, the inverse the same two back.  With W
// warps a window (16, or 4 for 64 x 64; the numbers are for 128 x 128), warp w
// (0..15), lane l, thread registers:
//   pass 1  rows w + 16 rr (rr = 0..7), columns l + 32 cc (cc = 0..3):
//           radix 4 over cc, radix 8 over rr (first DIF stages of both axes),
//           both twiddles;
//   E1      between the lanes of a warp: registers (kr, kc) <-> lanes l;
//   pass 2  lane m = 4 kr + kc, registers l = 0..31: radix 32, which ends the
//           column axis (frequency kc + 4 k);
//   E2      between the warps: registers k = 2 w' + b <-> warps w;
//   pass 3  warp w', lane m, registers (w = 0..15, b = 0..1): two radix-16
//           DFTs, which end the row axis (frequency kr + 8 i), the magnitude
//           replacement (S3), the two inverse radix-16 DFTs;
// then E2, pass 2, E1 and pass 1 back, the agent update and the stores.
//
// Against the cluster form (agent_xpose.cuh: two radix stages per axis, each
// through shared memory, and two exchanges between eight CTAs) a value
// crosses shared memory 4 times in and 4 times out instead of 12 passes and
// 4 bulk-copy passes, there is no wait for other CTAs, and a window takes two
// block barriers.  E1 needs none: a warp's 8704-byte region of the exchange
// buffer is its own from the second barrier of a window to the first of the
// next.  In that time the region also receives the warp's rows of the next
// window's stack (bulk copies issued before the update, awaited after the
// consensus loads of the next copy-in).
//
// Layouts in a warp's region (all accesses free of bank conflicts):
//   stack  row rr at 1024 rr bytes;
//   E1     row l of 34 values (rows 16-byte aligned, 16-byte accesses of a
//          row side and 8-byte accesses of a column side);
//   E2     values (k, k + 1) of lane m side by side at 16 (32 (k / 2) + m)
//          bytes; the thread that reads them writes them back in place.
//
// v and 1/d live in tensor memory (all 512 columns of an SM: 2 x 64 a
// thread), d of a thread's first kDSmem values in shared memory, of the others
// in L2.
//
// A CTA takes every ceil(J / wpc)-th window.  Waits are bounded as in
// agent_xpose.cuh: a warp whose wait for its copies gives up sets bit 2 of
// *err, and the CTA's threads agree at the next block barrier and stop.
//
// Measured (GB300, FP16 amplitudes, one sweep, against the cluster form): 64009
// windows 5.07-5.21 against 7.19 ms (3.7 TB/s of the 18 bytes a pixel the sweep
// must move: read q and y, write q), 14641 windows 1.17-1.20 against 1.68 ms, 900
// windows 86 against 125 us; 3600 windows of 64 x 64 92 against 164 us, of 32 x 32
// (both formats) 24 against 41 us for one CTA a window in place.  What bounds the 128 x 128 sweep: about 13.5 k of a window's 26 k
// cycles are instruction issue (75 % of it on the FP32 pipes), 8 k the
// shared-memory passes, and the store of 128 KB takes 4.1 k at the 32 bytes a
// cycle an SM can store; the block barriers keep the warps in step, so these
// overlap only in part.  Bulk stores of q' with plain loads of q, the other
// way round from what is built, were no faster (1.24 ms against 1.22 then).
#pragma once

#include "agent_xpose.cuh"
#include "pdl.cuh"

namespace pmace {

// W warps hold a window; thread registers e = CC rr + cc, rr = 0 .. RR - 1.
template <int N>
struct RegGeom {
    static constexpr int kPer = N == 128 ? 1 : 4;                     // CTAs an SM: 512 threads of 128 registers
    static constexpr int W = N * N / 1024;
    static constexpr int T = 32 * W;
    static constexpr int CC = N / 32;                                 // columns l + 32 cc of a thread
    static constexpr int RR = N / W;                                  // its rows w + W rr
    static constexpr int IR = W;                                      // radix of pass 3
    static constexpr int KB = 32 / IR;                                // its DFTs a thread
    static constexpr int kRow = 34;                                   // values per row of E1
    static constexpr int kRegion = 32 * kRow * (int)sizeof(float2);   // bytes of a warp's region
    static constexpr int kDSmem = N == 128 ? 22 : 20;                 // values of d per thread in shared memory
    static constexpr int kOffD = W * kRegion;
    static constexpr int kOffU = kOffD + kDSmem * T * (int)sizeof(float2);
    static constexpr int kOffV = kOffU + W * RR * (int)sizeof(float2);
    static constexpr int kOffBar = kOffV + 32 * CC * (int)sizeof(float2);
    static constexpr int kOffRed = kOffBar + W * 8;
    static constexpr int kOffConst = kOffRed + W * 4 * (int)sizeof(double);
    static constexpr int kOffTm = kOffConst + 32;
    static constexpr int kSmem = kOffTm + 16;
    static constexpr uint32_t kTmCols = 512 / kPer;
    static_assert(CC * RR == 32 && KB * IR == 32 && IR * RR == N, "32 values a thread, two radices an axis");
    static_assert(kRegion % 16 == 0 && kOffD % 16 == 0 && kOffU % 16 == 0 && kOffV % 16 == 0 && kOffConst % 16 == 0,
                  "16-byte accesses");
    static_assert(RR * N * (int)sizeof(float2) <= kRegion, "the stack rows of a warp fit its region");
    // exactly kPer CTAs an SM (1 KB reserved each), which share its TMEM
    static_assert(kPer * (kSmem + 1024) <= 228 * 1024 && (kPer + 1) * (kSmem + 1024) > 228 * 1024, "CTAs an SM");
};

// Copy `bytes` from global memory to this CTA's shared memory, counted on `bar`.
__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
                 "l"(src), "r"(bytes), "r"(bar)
                 : "memory");
}

// Bounded wait of a whole warp: the lanes poll one by one and may reach the
// limit at different polls, so they vote, and all of them take the way of a
// wait that gave up if any did.  What follows a wait is warp-wide (.sync.aligned
// tensor-memory accesses, full-mask shuffles and warp barriers); the vote also
// brings the lanes back together for it.
__device__ __forceinline__ bool mbar_wait_warp(uint32_t bar, uint32_t parity, int* err) {
    return __all_sync(0xffffffffu, mbar_wait_bounded(bar, parity, err));
}

// A load of a probe table (read-only while the kernel runs) that stays where it
// is written (the compiler moves plain ones up, which costs the registers they
// are meant to wait for).
__device__ __forceinline__ float2 ld_here(const float2* p) {
    float2 v;
    asm volatile("ld.global.nc.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "l"(p));
    return v;
}

// The consensus values of a thread's next window.  A launch that may start while
// the gather before it still writes the image (LIVE, pdl.cuh) takes plain loads.
// Where the kernel before has ended, read-only ones: with plain loads, which stay
// in order with the stores around them, the 64009-window sweep of 128 x 128
// windows spills 150 bytes more a thread (two iterations 15.9 ms against 14.9,
// 3600 windows of 64 x 64 276 us against 272).
template <bool LIVE>
__device__ __forceinline__ float2 ld_next(const float2* p) {
    if constexpr (LIVE) return ld_live(p);
    else return ld_here(p);
}

// Pass 1 forward on x[CC rr + cc]: radix CC over cc with the lane's twiddles
// v[kc] = W^(l kc), radix RR over rr with the warp's u[kr] = W^(w kr); the
// result x[CC kr + kc].
template <int CC, int RR>
__device__ __forceinline__ void reg_pass1(float2 (&x)[32], const float2* __restrict__ v, const float2* __restrict__ u) {
    const float4* v4 = reinterpret_cast<const float4*>(v);
    const float4 v01 = v4[0], v23 = CC == 4 ? v4[1] : v01;
#pragma unroll
    for (int rr = 0; rr < RR; ++rr) {
        float2 s[CC];
#pragma unroll
        for (int cc = 0; cc < CC; ++cc) s[cc] = x[CC * rr + cc];
        Dft<CC, false>::run(s);
        x[CC * rr] = s[0];
        x[CC * rr + 1] = cmul(s[1], make_float2(v01.z, v01.w));
        if constexpr (CC == 4) {
            x[CC * rr + 2] = cmul(s[2], make_float2(v23.x, v23.y));
            x[CC * rr + 3] = cmul(s[3], make_float2(v23.z, v23.w));
        }
    }
    const float4* u4 = reinterpret_cast<const float4*>(u);
#pragma unroll
    for (int kc = 0; kc < CC; ++kc) {
        float2 s[RR];
#pragma unroll
        for (int rr = 0; rr < RR; ++rr) s[rr] = x[CC * rr + kc];
        Dft<RR, false>::run(s);
#pragma unroll
        for (int p = 0; p < RR / 2; ++p) {
            const float4 f = u4[p];
            x[CC * (2 * p) + kc] = p ? cmul(s[2 * p], make_float2(f.x, f.y)) : s[0];
            x[CC * (2 * p + 1) + kc] = cmul(s[2 * p + 1], make_float2(f.z, f.w));
        }
    }
}

// Pass 1 back: the conjugate twiddles and inverse DFTs in reverse order.
template <int CC, int RR>
__device__ __forceinline__ void reg_pass1_inv(float2 (&x)[32], const float2* __restrict__ v,
                                              const float2* __restrict__ u) {
    const float4* u4 = reinterpret_cast<const float4*>(u);
#pragma unroll
    for (int kc = 0; kc < CC; ++kc) {
        float2 s[RR];
#pragma unroll
        for (int p = 0; p < RR / 2; ++p) {
            const float4 f = u4[p];
            s[2 * p] = p ? cmulc(x[CC * (2 * p) + kc], make_float2(f.x, f.y)) : x[kc];
            s[2 * p + 1] = cmulc(x[CC * (2 * p + 1) + kc], make_float2(f.z, f.w));
        }
        Dft<RR, true>::run(s);
#pragma unroll
        for (int rr = 0; rr < RR; ++rr) x[CC * rr + kc] = s[rr];
    }
    const float4* v4 = reinterpret_cast<const float4*>(v);
    const float4 v01 = v4[0], v23 = CC == 4 ? v4[1] : v01;
#pragma unroll
    for (int rr = 0; rr < RR; ++rr) {
        float2 s[CC];
        s[0] = x[CC * rr];
        s[1] = cmulc(x[CC * rr + 1], make_float2(v01.z, v01.w));
        if constexpr (CC == 4) {
            s[2] = cmulc(x[CC * rr + 2], make_float2(v23.x, v23.y));
            s[3] = cmulc(x[CC * rr + 3], make_float2(v23.z, v23.w));
        }
        Dft<CC, true>::run(s);
#pragma unroll
        for (int cc = 0; cc < CC; ++cc) x[CC * rr + cc] = s[cc];
    }
}

// Eight amplitudes of a thread from raw 16-byte chunks (one of FP16 codes,
// two of FP32 values).
template <int AMP>
__device__ __forceinline__ void unpack_amps8(const uint4* raw, float (&out)[8]) {
    constexpr int NCH = AMP ? 1 : 2;
#pragma unroll
    for (int k = 0; k < NCH; ++k) {
        const uint32_t w[4] = {raw[k].x, raw[k].y, raw[k].z, raw[k].w};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            if constexpr (AMP == 1) {
                const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&w[q]));
                out[8 * k + 2 * q] = f.x;
                out[8 * k + 2 * q + 1] = f.y;
            } else {
                out[4 * k + q] = __uint_as_float(w[q]);
            }
        }
    }
}

// Named barriers id (1..15): wait for `count` threads to arrive, or arrive only.
__device__ __forceinline__ void named_sync(int id, int count) { asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(count) : "memory"); }
__device__ __forceinline__ void named_arrive(int id, int count) {
    asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(count) : "memory");
}

// Windows j0, j0 + step, ... below J of the job `a` on one CTA, with
// FP16 amplitudes (agent_impl).  LIVE: the launch may start while the kernel
// before it runs.
template <int N, bool LIVE>
__device__ __forceinline__ void reg_body(const AgentArgs& a, const int j0, const int step) {
    using G = RegGeom<N>;
    constexpr int T = G::T, W = G::W, CC = G::CC, RR = G::RR, IR = G::IR, KB = G::KB;
    constexpr uint32_t kCopyBytes = RR * N * sizeof(float2);

    extern __shared__ float4 smem_raw[];
    char* sm = reinterpret_cast<char*>(smem_raw);
    float2* s_d = reinterpret_cast<float2*>(sm + G::kOffD);
    float2* s_u = reinterpret_cast<float2*>(sm + G::kOffU);
    float2* s_v = reinterpret_cast<float2*>(sm + G::kOffV);
    double* red = reinterpret_cast<double*>(sm + G::kOffRed);
    uint32_t* s_tm = reinterpret_cast<uint32_t*>(sm + G::kOffTm);

    const int t = (int)threadIdx.x, l = t & 31;
    const int w = __shfl_sync(0xffffffffu, t >> 5, 0);
    char* region = sm + w * G::kRegion;
    const uint32_t region_s = smem_addr(region), bar = smem_addr(sm + G::kOffBar) + 8u * (uint32_t)w;

    // the window corner is loaded a window ahead
    int2 off_next = window_corner<N>(a, j0);
    if (t < 32) tmem_alloc(smem_addr(s_tm), G::kTmCols);
    // the step's constants wait in shared memory: registers are short
    float4* s_const = reinterpret_cast<float4*>(sm + G::kOffConst);
    if (t == 0) {
        const float two_rho = 2.0f * a.rho_cur, inv1pa = 1.0f / (1.0f + a.alpha), two_rho_prev = 2.0f * a.rho_prev;
        const float keep = 1.0f - inv1pa;                  // alpha / (1 + alpha)
        const float data = inv1pa * (1.0f / (float)N);     // the orthonormal F^* of the data term, over 1 + alpha
        s_const[0] = make_float4(keep, keep, -two_rho, -two_rho);
        s_const[1] = make_float4(two_rho_prev, two_rho_prev, data, 0.f);
    }
    if (l == 0) mbar_init(bar, 1);
    for (int i = t; i < W * RR; i += T) s_u[i] = a.tw[(i / RR) * (i % RR)];            // [w][kr]
    for (int i = t; i < 32 * CC; i += T) s_v[i] = a.tw[((i / CC) * (i % CC)) & (N - 1)];   // [l][kc]
    mbar_fence_init();
    fence_proxy_async_smem();
    tmem_fence_before_sync();
    __syncthreads();
    tmem_fence_after_sync();

    // the warp's stack rows of window j into its region (a row a lane)
    auto load_stack = [&](int j) {
        if (l == 0) mbar_arrive_expect_tx(bar, kCopyBytes);
        __syncwarp();
        if (l < RR)
            bulk_load(region_s + (uint32_t)(N * sizeof(float2)) * (uint32_t)l, a.q + ((size_t)j * N + w + W * l) * N,
                      (uint32_t)(N * sizeof(float2)), bar);
    };
    // v in columns 0..63 of the warp's lanes, 1/d in 64..127.  The tables are
    // loaded all at once, while the kernel before this one ends.
    const uint32_t tm_v = *s_tm + ((uint32_t)(32 * (w & 3)) << 16) + 128u * (uint32_t)(w >> 2), tm_i = tm_v + 64u;
    const float2* __restrict__ d_l2 = a.probe + w * N + l;   // value e = CC rr + cc at W N rr + 32 cc
    bool absent = false;   // whether one of the thread's pixels has its probe value treated as absent (1/d = 0)
    float2 x[32];
#pragma unroll
    for (int e = 0; e < 32; ++e) x[e] = __ldg(a.dinv + w * N + l + W * N * (e / CC) + 32 * (e % CC));
#pragma unroll
    for (int g = 0; g < 8; ++g) {
        uint32_t r[8];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const float2 di = x[4 * g + k];
            absent |= di.x == 0.f && di.y == 0.f;
            r[2 * k] = __float_as_uint(di.x);
            r[2 * k + 1] = __float_as_uint(di.y);
        }
        tmem_st8(tm_i + 8u * g, r);
    }
#pragma unroll
    for (int e = 0; e < G::kDSmem; ++e) x[e] = __ldg(d_l2 + W * N * (e / CC) + 32 * (e % CC));
#pragma unroll
    for (int e = 0; e < G::kDSmem; ++e) s_d[e * T + t] = x[e];
    tmem_wait_st();
    pdl_wait();   // the stacks and the consensus image from here on
    load_stack(j0);

    constexpr float inv_n = 1.0f / (float)N;
    const bool first = a.first != 0;
    const bool res = a.residual != 0;
    const bool wu = a.u != nullptr;
    uint32_t parity = 0;

    // L2 prefetch of the warp's stack rows and amplitudes of a window
    auto prefetch = [&](int j) {
        if (l < RR) prefetch_l2(a.q + ((size_t)j * N + w + W * l) * N, (uint32_t)(N * sizeof(float2)));
        else if (l == RR) {
            constexpr uint32_t yb = 1024 * sizeof(__half);
            prefetch_l2(static_cast<const char*>(a.y) + (size_t)j * N * N * sizeof(__half) + (size_t)w * yb, yb);
        }
    };
    // Where a window takes sixteen warps, four groups of four take turns (a
    // chain of named barriers) at the reads that follow each block barrier, so
    // that one group computes while the next still reads: with all sixteen
    // warps reading and then computing together the 14641-window sweep of
    // 128 x 128 windows took 1296 us instead of 1217.
    const int grp = w >> 2;
    auto turn_begin = [&](int id) {
        if (W == 16 && grp > 0) named_sync(id + grp - 1, T / 2);
    };
    auto turn_end = [&](int id) {
        if (W == 16 && grp < 3) named_arrive(id + grp, T / 2);
    };

    const size_t rows_w = (size_t)W * a.n2;
    // where the thread's consensus values of the window at `off` start
    auto xbar_at = [&](int2 off) { return a.xbar + (size_t)(off.x + w) * a.n2 + off.y + l; };
    {
        const float2* xr = xbar_at(off_next);
#pragma unroll
        for (int e = 0; e < 32; ++e) x[e] = ld_live(xr + (e / CC) * rows_w + 32 * (e % CC));
    }
#pragma unroll 1
    for (int j = j0; j < a.J; j += step) {
        const int2 off = off_next;
        const bool more = j + step < a.J;
        if (more) {
            off_next = window_corner<N>(a, j + step);
            prefetch(j + step);
        }
        const size_t wbase = (size_t)j * N * N;
        // ---- S0 + S1: the consensus values are in x (loaded by the update
        // of the previous window as it freed the registers)
        const bool got = mbar_wait_warp(bar, parity, a.err);
        {
            const float2* st = reinterpret_cast<const float2*>(region) + l;
            const float2 trp2 = make_float2(s_const[1].x, s_const[1].y);
            float2 dl[32 - G::kDSmem];
            static_assert(G::kDSmem >= 20 && G::kDSmem < 32, "groups 5 to 7 are loaded four groups ahead");
#pragma unroll
            for (int g = 0; g < 8; ++g) {   // four values at a time
                if (g >= 1 && g <= 3) {     // the values of d that shared memory does not hold, four groups ahead
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const int e = 4 * (g + 4) + k;
                        if (e >= G::kDSmem) dl[e < G::kDSmem ? 0 : e - G::kDSmem] = ld_here(d_l2 + W * N * (e / CC) + 32 * (e % CC));
                    }
                }
                uint32_t r[8];
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const int e = 4 * g + k;
                    x[e] = mann_close2(st[N * (e / CC) + 32 * (e % CC)], x[e], trp2);
                    r[2 * k] = __float_as_uint(x[e].x);
                    r[2 * k + 1] = __float_as_uint(x[e].y);
                }
                tmem_st8(tm_v + 8u * g, r);   // v, for the update
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const int e = 4 * g + k;
                    x[e] = cmul(e < G::kDSmem ? s_d[e * T + t] : dl[e < G::kDSmem ? 0 : e - G::kDSmem], x[e]);
                }
            }
        }
        reg_pass1<CC, RR>(x, s_v + CC * l, s_u + RR * w);
        // ---- E1
        __syncwarp();   // every lane has read its stack values
        {
            float4* row = reinterpret_cast<float4*>(region) + (G::kRow / 2) * l;
#pragma unroll
            for (int p = 0; p < 16; ++p) row[p] = make_float4(x[2 * p].x, x[2 * p].y, x[2 * p + 1].x, x[2 * p + 1].y);
            __syncwarp();
            const float2* col = reinterpret_cast<const float2*>(region) + l;
#pragma unroll
            for (int i = 0; i < 32; ++i) {   // in the order the radix-32 DFT takes them
                const int k = 4 * (i % 8) + i / 8;
                x[k] = col[G::kRow * k];
            }
        }
        Dft<32, false>::run(x);
        // ---- E2
        __syncwarp();
        {
            float4* mine = reinterpret_cast<float4*>(region) + l;
#pragma unroll
            for (int p = 0; p < 16; ++p) mine[32 * p] = make_float4(x[2 * p].x, x[2 * p].y, x[2 * p + 1].x, x[2 * p + 1].y);
        }
        uint4 raw[4];   // eight codes each
        const float yscale = __ldg(a.yscale + j);
        {
            const uint4* yp = reinterpret_cast<const uint4*>(static_cast<const char*>(a.y) + wbase * sizeof(__half)) + t;
            const uint64_t pol_first = l2_policy_evict_first();
#pragma unroll
            for (int k = 0; k < 4; ++k) raw[k] = ld_nc_l2_hint(yp + k * T, pol_first);
        }
        if (__syncthreads_or(!got)) {
            // a wait that gave up stops the CTA; its warp's copies may still
            // be in flight: one more (bounded) wait before shared memory goes
            if (!got) mbar_wait_warp(bar, parity, a.err);
            break;
        }
        parity ^= 1u;
        // ---- pass 3: row axis, S3 and back
        float acc_d = 0.f, acc_y = 0.f;
        {
            float4* mine = reinterpret_cast<float4*>(sm) + 32 * (KB / 2) * w + l;
            constexpr int RS4 = G::kRegion / 16;
            float2 z[32];   // DFT kb: z[IR kb + i]
            turn_begin(1);
#pragma unroll
            for (int p = 0; p < KB / 2; ++p) {
#pragma unroll
                for (int k = 0; k < IR; ++k) {
                    const int i = IR == 16 ? 4 * (k % 4) + k / 4 : k;   // in the order the DFT takes them
                    const float4 f = mine[RS4 * i + 32 * p];
                    z[IR * (2 * p) + i] = make_float2(f.x, f.y);
                    z[IR * (2 * p + 1) + i] = make_float2(f.z, f.w);
                }
            }
            turn_end(1);
            auto rows = [&](auto with_res) {
                constexpr bool kRes = decltype(with_res)::value;
                constexpr int B = IR < 8 ? 8 / IR : 1;   // DFTs per step of at least eight values
#pragma unroll
                for (int k0 = 0; k0 < KB; k0 += B) {
#pragma unroll
                    for (int b = 0; b < B; ++b) Dft<IR, false>::run(reinterpret_cast<float2(&)[IR]>(z[IR * (k0 + b)]));
                    if (a.spectrum) {   // check of the forward transform, natural order
#pragma unroll
                        for (int i = 0; i < IR * B; ++i)
                            a.spectrum[wbase + (size_t)(l / CC + RR * (i % IR)) * N + l % CC + CC * (KB * w + k0 + i / IR)] =
                                z[IR * k0 + i];
                    }
#pragma unroll
                    for (int h = 0; h < IR * B / 8; ++h) {   // eight at a time: registers
                        float yv[8];
                        unpack_amps8<1>(raw + IR * k0 / 8 + h, yv);
                        replace_magnitudes<kRes>(reinterpret_cast<float2(&)[8]>(z[IR * k0 + 8 * h]), yv, inv_n, acc_d, acc_y,
                                                 yscale);
                    }
#pragma unroll
                    for (int b = 0; b < B; ++b) Dft<IR, true>::run(reinterpret_cast<float2(&)[IR]>(z[IR * (k0 + b)]));
                }
            };
            if (res) rows(std::true_type{});
            else rows(std::false_type{});
#pragma unroll
            for (int p = 0; p < KB / 2; ++p)
#pragma unroll
                for (int i = 0; i < IR; ++i)
                    mine[RS4 * i + 32 * p] = make_float4(z[IR * (2 * p) + i].x, z[IR * (2 * p) + i].y,
                                                         z[IR * (2 * p + 1) + i].x, z[IR * (2 * p + 1) + i].y);
        }
        __syncthreads();
        // ---- E2, pass 2, E1 back
        {
            const float4* mine = reinterpret_cast<const float4*>(region) + l;
            turn_begin(4);
#pragma unroll
            for (int i = 0; i < 16; ++i) {
                const int p = 2 * (i % 8) + i / 8;
                const float4 f = mine[32 * p];
                x[2 * p] = make_float2(f.x, f.y);
                x[2 * p + 1] = make_float2(f.z, f.w);
            }
            turn_end(4);
        }
        Dft<32, true>::run(x);
        __syncwarp();
        {
            float2* col = reinterpret_cast<float2*>(region) + l;
#pragma unroll
            for (int i = 0; i < 32; ++i) col[G::kRow * i] = x[i];
            __syncwarp();
            const float4* row = reinterpret_cast<const float4*>(region) + (G::kRow / 2) * l;
#pragma unroll
            for (int i = 0; i < 16; ++i) {
                const int p = 2 * (i % 8) + i / 8;
                const float4 f = row[p];
                x[2 * p] = make_float2(f.x, f.y);
                x[2 * p + 1] = make_float2(f.z, f.w);
            }
        }
        // the region is free: the next window's stack rows
        fence_proxy_async_smem();
        __syncwarp();
        if (more) load_stack(j + step);
        reg_pass1_inv<CC, RR>(x, s_v + CC * l, s_u + RR * w);
        // ---- S4 + S5, four values at a time; the registers a group frees take the consensus values of the next window (its own again
        // after the last one, which keeps the loads unconditional)
        float acc_z = 0.f, acc_w = 0.f;
        tmem_wait_st();   // v of the copy-in has landed
        {
            const float4 c0 = s_const[0], c1 = s_const[1];
            const float2 keep2 = make_float2(c0.x, c0.y), m2rho2 = make_float2(c0.z, c0.w);
            const float ds = c1.z * yscale;
            const float2 data2 = make_float2(ds, ds);
            const uint64_t pol_next = a.keep ? l2_policy_evict_last() : l2_policy_evict_normal();
            const uint64_t pol_q = wu ? l2_policy_evict_first() : pol_next;
            float2* qr = a.q + wbase + w * N + l;
            float2* __restrict__ ur = a.u + wbase + w * N + l;
            const float2* xr = xbar_at(off);
            const float2* xn = xbar_at(off_next);
#pragma unroll
            for (int g = 0; g < 8; ++g) {
                uint32_t rv[8], ri[8];
                tmem_ld8x2(tm_v + 8u * g, rv, tm_i + 8u * g, ri);
                float2 v[4], wv[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    v[k] = make_float2(__uint_as_float(rv[2 * k]), __uint_as_float(rv[2 * k + 1]));
                    const float2 dv = make_float2(__uint_as_float(ri[2 * k]), __uint_as_float(ri[2 * k + 1]));
                    wv[k] = __ffma2_rn(keep2, v[k], cmul(dv, __fmul2_rn(x[4 * g + k], data2)));
                }
                if (absent) {
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        if (ri[2 * k] << 1 == 0u && ri[2 * k + 1] << 1 == 0u) wv[k] = v[k];   // 1/d is +-0
                }
                if (res) {
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const int e = 4 * g + k;
                        residual_sums(first ? v[k] : ld_live(xr + (e / CC) * rows_w + 32 * (e % CC)), wv[k], acc_z, acc_w);
                    }
                }
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const int e = 4 * g + k, at = W * N * (e / CC) + 32 * (e % CC);
                    if (wu) st_l2_hint(ur + at, agent_u2(v[k], wv[k]), pol_next);
                    st_l2_hint(qr + at, __ffma2_rn(m2rho2, wv[k], v[k]), pol_q);
                }
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    x[4 * g + k] = ld_next<LIVE>(xn + 32 * ((4 * g + k) % CC));
                    if ((4 * g + k) % CC == CC - 1) xn += rows_w;
                }
            }
        }
        if (res) {
            float acc[4] = {acc_z, acc_w, acc_d, acc_y};
            block_reduce4<T>(acc, red, a.partials + (size_t)j * 4);
        }
    }
    tmem_wait_st();   // a stopped run may leave its last v stores outstanding
    tmem_fence_before_sync();
    __syncthreads();
    if (t < 32) {
        tmem_fence_after_sync();
        tmem_dealloc(*s_tm, G::kTmCols);
    }
}

// ---- 32 x 32 windows: a warp holds a window (thread l: column l, x[r] row r),
// so the 2-D DFT is a radix-32 pass over the registers, one exchange inside
// the warp and a second radix-32 pass (thread kr, x[kc]), without a twiddle
// or a block barrier; the warps of a CTA share only the probe tables.
struct RegGeom32 {
    static constexpr int N = 32;
    static constexpr int W = 4;                       // warps (windows) per CTA
    static constexpr int T = 32 * W;
    static constexpr int kPer = 4;                    // CTAs an SM
    static constexpr int kRow = 34;
    static constexpr int kRegion = 32 * kRow * (int)sizeof(float2);
    static constexpr int kOffD = W * kRegion;
    static constexpr int kOffI = kOffD + N * N * (int)sizeof(float2);
    static constexpr int kOffConst = kOffI + N * N * (int)sizeof(float2);
    static constexpr int kOffBar = kOffConst + 32;
    static constexpr int kOffTm = kOffBar + W * 8;
    static constexpr int kSmem = kOffTm + 16;
    static_assert(kOffD % 16 == 0 && kOffI % 16 == 0 && kOffConst % 16 == 0, "16-byte accesses");
    static_assert(kPer * (kSmem + 1024) <= 228 * 1024 && (kPer + 1) * (kSmem + 1024) > 228 * 1024, "CTAs an SM");
};

// Windows j0, j0 + step, ... below J of the job `a` on one warp of a CTA.
template <int AMP>
__device__ __forceinline__ void reg32_body(const AgentArgs& a, const int cta, const int nctas) {
    using G = RegGeom32;
    constexpr int N = G::N, T = G::T, W = G::W;
    constexpr int NCH = AMP ? 1 : 2;          // 16-byte chunks of eight amplitudes
    constexpr uint32_t kCopyBytes = N * N * sizeof(float2);
    extern __shared__ float4 smem_raw[];
    char* sm = reinterpret_cast<char*>(smem_raw);
    const int t = (int)threadIdx.x, l = t & 31;
    const int w = __shfl_sync(0xffffffffu, t >> 5, 0);
    char* region = sm + w * G::kRegion;
    float4* s_const = reinterpret_cast<float4*>(sm + G::kOffConst);
    uint32_t* s_tm = reinterpret_cast<uint32_t*>(sm + G::kOffTm);
    const uint32_t region_s = smem_addr(region), bar = smem_addr(sm + G::kOffBar) + 8u * (uint32_t)w;
    const int j0 = cta * W + w, step = nctas * W;

    int2 off_next = window_corner<N>(a, min(j0, a.J - 1));
    if (t < 32) tmem_alloc(smem_addr(s_tm), 64u);
    if (l == 0) {
        mbar_init(bar, 1);
        mbar_fence_init();
    }
    fence_proxy_async_smem();
    __syncwarp();
    auto load_stack = [&](int j) {
        if (l == 0) {
            mbar_arrive_expect_tx(bar, kCopyBytes);
            bulk_load(region_s, a.q + (size_t)j * (N * N), kCopyBytes, bar);
        }
    };
    if (t == 0) {
        const float two_rho = 2.0f * a.rho_cur, inv1pa = 1.0f / (1.0f + a.alpha), two_rho_prev = 2.0f * a.rho_prev;
        const float keep = 1.0f - inv1pa, data = inv1pa * (1.0f / (float)N);   // as in reg_body
        s_const[0] = make_float4(keep, keep, -two_rho, -two_rho);
        s_const[1] = make_float4(two_rho_prev, two_rho_prev, data, 0.f);
    }
    bool absent = false;
    {
        float4* dst = reinterpret_cast<float4*>(sm + G::kOffD);
        constexpr int H = N * N / 2;   // 16-byte pieces per table
        float4 f[2 * H / T];
#pragma unroll
        for (int i = 0; i < H / T; ++i) {
            f[i] = __ldg(reinterpret_cast<const float4*>(a.probe) + t + i * T);
            f[H / T + i] = __ldg(reinterpret_cast<const float4*>(a.dinv) + t + i * T);
        }
#pragma unroll
        for (int i = 0; i < H / T; ++i) {
            const float4 di = f[H / T + i];
            absent |= (di.x == 0.f && di.y == 0.f) || (di.z == 0.f && di.w == 0.f);
            dst[t + i * T] = f[i];
            dst[H + t + i * T] = di;
        }
    }
    const float2* s_d = reinterpret_cast<const float2*>(sm + G::kOffD) + l;
    const float2* s_i = reinterpret_cast<const float2*>(sm + G::kOffI) + l;
    constexpr float inv_n = 1.0f / (float)N;
    const bool first = a.first != 0;
    const bool res = a.residual != 0;
    const bool wu = a.u != nullptr;
    const size_t n2 = (size_t)a.n2;
    auto xbar_at = [&](int2 off) { return a.xbar + (size_t)off.x * a.n2 + off.y + l; };
    pdl_wait();   // the stacks and the consensus image from here on
    if (j0 < a.J) load_stack(j0);
    float2 x[32];
    {
        const float2* xr = xbar_at(off_next);
#pragma unroll
        for (int e = 0; e < 32; ++e) x[e] = ld_live(xr + e * n2);
    }
    tmem_fence_before_sync();
    absent = __syncthreads_or(absent);
    tmem_fence_after_sync();
    const uint32_t tm_v = *s_tm + ((uint32_t)(32 * w) << 16);   // v in the 64 columns of the warp's lanes
    uint32_t parity = 0;
#pragma unroll 1
    for (int j = j0; j < a.J; j += step) {
        const int2 off = off_next;
        const bool more = j + step < a.J;
        if (more) {
            off_next = window_corner<N>(a, j + step);
            if (l == 0) prefetch_l2(a.q + (size_t)(j + step) * (N * N), kCopyBytes);
            else if (l == 1)
                prefetch_l2(static_cast<const char*>(a.y) + (size_t)(j + step) * (N * N * (AMP ? 2 : 4)), N * N * (AMP ? 2 : 4));
        }
        const size_t wbase = (size_t)j * N * N;
        // ---- S0 + S1, and the first radix-32 pass (rows)
        if (!mbar_wait_warp(bar, parity, a.err)) {
            mbar_wait_warp(bar, parity, a.err);   // the warp stops: see reg_body
            break;
        }
        parity ^= 1u;
        {
            const float2* st = reinterpret_cast<const float2*>(region) + l;
            const float2 trp2 = make_float2(s_const[1].x, s_const[1].y);
#pragma unroll
            for (int g = 0; g < 8; ++g) {
                uint32_t r[8];
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const int e = 4 * g + k;
                    x[e] = mann_close2(st[N * e], x[e], trp2);
                    r[2 * k] = __float_as_uint(x[e].x);
                    r[2 * k + 1] = __float_as_uint(x[e].y);
                }
                tmem_st8(tm_v + 8u * g, r);   // v, for the update
#pragma unroll
                for (int k = 0; k < 4; ++k) x[4 * g + k] = cmul(s_d[N * (4 * g + k)], x[4 * g + k]);
            }
        }
        Dft<32, false>::run(x);
        __syncwarp();
        float2* col = reinterpret_cast<float2*>(region) + l;
        float4* row = reinterpret_cast<float4*>(region) + (G::kRow / 2) * l;
#pragma unroll
        for (int p = 0; p < 16; ++p) row[p] = make_float4(x[2 * p].x, x[2 * p].y, x[2 * p + 1].x, x[2 * p + 1].y);
        uint4 raw[4 * NCH];
        float yscale = 1.0f;
        {
            const uint4* yp = reinterpret_cast<const uint4*>(static_cast<const char*>(a.y) + wbase * (AMP ? 2 : 4)) + l;
            const uint64_t pol_first = l2_policy_evict_first();
#pragma unroll
            for (int k = 0; k < 4 * NCH; ++k) raw[k] = ld_nc_l2_hint(yp + k * 32, pol_first);
            if constexpr (AMP == 1) yscale = __ldg(a.yscale + j);
        }
        __syncwarp();
#pragma unroll
        for (int i = 0; i < 32; ++i) {
            const int k = 4 * (i % 8) + i / 8;
            x[k] = col[G::kRow * k];
        }
        // ---- second pass (columns), S3 and back
        float acc_d = 0.f, acc_y = 0.f;
        Dft<32, false>::run(x);
        auto replace = [&](auto with_res) {
            constexpr bool kRes = decltype(with_res)::value;
#pragma unroll
            for (int h = 0; h < 4; ++h) {
                float yv[8];
                unpack_amps8<AMP>(raw + NCH * h, yv);
                replace_magnitudes<kRes>(reinterpret_cast<float2(&)[8]>(x[8 * h]), yv, inv_n, acc_d, acc_y,
                                         AMP == 1 ? yscale : 1.0f);
            }
        };
        if (res) replace(std::true_type{});
        else replace(std::false_type{});
        Dft<32, true>::run(x);
#pragma unroll
        for (int i = 0; i < 32; ++i) col[G::kRow * i] = x[i];
        __syncwarp();
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            const int p = 2 * (i % 8) + i / 8;
            const float4 f = row[p];
            x[2 * p] = make_float2(f.x, f.y);
            x[2 * p + 1] = make_float2(f.z, f.w);
        }
        fence_proxy_async_smem();
        __syncwarp();   // the region is free: the next window's stack
        if (more) load_stack(j + step);
        Dft<32, true>::run(x);
        // ---- S4 + S5, as in reg_body
        float acc_z = 0.f, acc_w = 0.f;
        tmem_wait_st();
        {
            const float4 c0 = s_const[0], c1 = s_const[1];
            const float2 keep2 = make_float2(c0.x, c0.y), m2rho2 = make_float2(c0.z, c0.w);
            const float ds = AMP == 1 ? c1.z * yscale : c1.z;
            const float2 data2 = make_float2(ds, ds);
            const uint64_t pol_next = a.keep ? l2_policy_evict_last() : l2_policy_evict_normal();
            const uint64_t pol_q = wu ? l2_policy_evict_first() : pol_next;
            float2* qr = a.q + wbase + l;
            float2* __restrict__ ur = a.u + wbase + l;
            const float2* xr = xbar_at(off);
            const float2* xn = xbar_at(off_next);
#pragma unroll
            for (int g = 0; g < 8; ++g) {
                uint32_t rv[8];
                tmem_ld8(tm_v + 8u * g, rv);
                float2 v[4], wv[4], dv[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) dv[k] = s_i[N * (4 * g + k)];
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    v[k] = make_float2(__uint_as_float(rv[2 * k]), __uint_as_float(rv[2 * k + 1]));
                    wv[k] = __ffma2_rn(keep2, v[k], cmul(dv[k], __fmul2_rn(x[4 * g + k], data2)));
                }
                if (absent) {
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        if (dv[k].x == 0.f && dv[k].y == 0.f) wv[k] = v[k];
                }
                if (res) {
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        residual_sums(first ? v[k] : ld_live(xr + (4 * g + k) * n2), wv[k], acc_z, acc_w);
                }
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const int at = N * (4 * g + k);
                    if (wu) st_l2_hint(ur + at, agent_u2(v[k], wv[k]), pol_next);
                    st_l2_hint(qr + at, __ffma2_rn(m2rho2, wv[k], v[k]), pol_q);
                }
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    x[4 * g + k] = ld_live(xn);
                    xn += n2;
                }
            }
        }
        if (res) {
            float acc[4] = {acc_z, acc_w, acc_d, acc_y};
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
                for (int i = 0; i < 4; ++i) acc[i] += __shfl_xor_sync(0xffffffffu, acc[i], o);
            }
            if (l == 0) {
#pragma unroll
                for (int i = 0; i < 4; ++i) a.partials[(size_t)j * 4 + i] = (double)acc[i];
            }
        }
    }
    tmem_wait_st();
    tmem_fence_before_sync();
    __syncthreads();
    if (t < 32) {
        tmem_fence_after_sync();
        tmem_dealloc(*s_tm, 64u);
    }
}

template <int AMP>
__global__ void __launch_bounds__(RegGeom32::T, RegGeom32::kPer) agent_reg32_kernel(const __grid_constant__ AgentArgs a) {
    reg32_body<AMP>(a, (int)blockIdx.x, (int)gridDim.x);
}
template <int AMP>
__global__ void __launch_bounds__(RegGeom32::T, RegGeom32::kPer)
agent_reg32_kernel_batched(const AgentArgs* __restrict__ descs, const int2* __restrict__ work) {
    const int2 wk = work[blockIdx.x];
    const AgentArgs& a = descs[wk.x];
    reg32_body<AMP>(a, wk.y / a.wpc, (a.J + a.wpc - 1) / a.wpc);
}

// One job: CTA k of G processes windows k, k + G, k + 2 G, ..., so that the
// CTAs are always within a few windows of one another in scan order and the
// consensus image they read stays in L2 (with contiguous runs the 64009-window
// sweep of 128 x 128 windows took 7.24 ms instead of 5.62).
template <int N, bool LIVE>
__global__ void __launch_bounds__(RegGeom<N>::T, RegGeom<N>::kPer) agent_reg_kernel(const __grid_constant__ AgentArgs a) {
    reg_body<N, LIVE>(a, (int)blockIdx.x, (int)gridDim.x);
}

// Several jobs: CTA k takes the share of job work[k].x that starts at window
// work[k].y / wpc, every ceil(J / wpc)-th window.
template <int N>
__global__ void __launch_bounds__(RegGeom<N>::T, RegGeom<N>::kPer)
agent_reg_kernel_batched(const AgentArgs* __restrict__ descs, const int2* __restrict__ work) {
    const int2 wk = work[blockIdx.x];
    const AgentArgs& a = descs[wk.x];
    reg_body<N, false>(a, wk.y / a.wpc, (a.J + a.wpc - 1) / a.wpc);
}

// Query (a == nullptr: fills info; a "cluster" is one CTA) or launch
// ceil(J / a->wpc) CTAs of `threads` threads, `per` an SM.
inline cudaError_t reg_query(cudaError_t e, int threads, int smem, int per, AgentPlanInfo* info) {
    int dev = 0, nsm = 0;
    if (e == cudaSuccess) e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    cudaGetLastError();
    info->threads = threads;
    info->smem_bytes = smem;
    info->max_clusters = e == cudaSuccess ? nsm * per : 0;
    info->launchable = info->max_clusters > 0;
    return cudaSuccess;
}

template <int N>
cudaError_t agent_reg(const AgentArgs* a, int amp_f16, cudaStream_t s, AgentPlanInfo* info) {
    using G = RegGeom<N>;
    const bool live = a != nullptr && a->overlap != 0;
    if (!amp_f16) return cudaErrorInvalidValue;   // agent_impl
    void (*fn)(const AgentArgs) = live ? agent_reg_kernel<N, true> : agent_reg_kernel<N, false>;
    const cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, G::kSmem);
    if (a == nullptr) return reg_query(e, G::T, G::kSmem, G::kPer, info);
    if (e != cudaSuccess) return e;
    if (a->wpc <= 0) return cudaErrorInvalidValue;
    return pdl_launch(live, fn, (unsigned)((a->J + a->wpc - 1) / a->wpc), G::T, G::kSmem, s, *a);
}

template <int N>
cudaError_t agent_reg_batched(const AgentArgs* descs, const int2* work, int nctas, int amp_f16, cudaStream_t s) {
    using G = RegGeom<N>;
    if (nctas <= 0) return cudaSuccess;
    if (!amp_f16) return cudaErrorInvalidValue;   // agent_impl
    void (*fn)(const AgentArgs*, const int2*) = agent_reg_kernel_batched<N>;
    const cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, G::kSmem);
    if (e != cudaSuccess) return e;
    fn<<<(unsigned)nctas, G::T, G::kSmem, s>>>(descs, work);
    return cudaGetLastError();
}

inline cudaError_t agent_reg32(const AgentArgs* a, int amp_f16, cudaStream_t s, AgentPlanInfo* info) {
    using G = RegGeom32;
    void (*fn)(const AgentArgs) = amp_f16 ? agent_reg32_kernel<1> : agent_reg32_kernel<0>;
    const cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, G::kSmem);
    if (a == nullptr) return reg_query(e, G::T, G::kSmem, G::kPer, info);
    if (e != cudaSuccess) return e;
    if (a->wpc <= 0) return cudaErrorInvalidValue;
    return pdl_launch(a->overlap != 0, fn, (unsigned)((a->J + a->wpc - 1) / a->wpc), G::T, G::kSmem, s, *a);
}

inline cudaError_t agent_reg32_batched(const AgentArgs* descs, const int2* work, int nctas, int amp_f16,
                                       cudaStream_t s) {
    using G = RegGeom32;
    if (nctas <= 0) return cudaSuccess;
    void (*fn)(const AgentArgs*, const int2*) = amp_f16 ? agent_reg32_kernel_batched<1> : agent_reg32_kernel_batched<0>;
    const cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, G::kSmem);
    if (e != cudaSuccess) return e;
    fn<<<(unsigned)nctas, G::T, G::kSmem, s>>>(descs, work);
    return cudaGetLastError();
}

}  // namespace pmace
