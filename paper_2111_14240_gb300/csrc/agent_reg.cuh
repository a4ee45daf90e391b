// The fused agent sweep (steps S0-S5 of one PMACE iteration, the arithmetic
// of agent.cuh) with a whole 128 x 128 window in the registers of one CTA.
//
// 512 threads hold 32 complex values each (the 128 KB of a window are half
// of an SM's register file).  A 2-D DFT of 128 x 128 has 14 binary levels; a
// thread's 32 values cover five at a time, so the forward transform takes
// three register passes and two exchanges through shared memory, the inverse
// the same two back.  Warp w (0..15), lane l, thread registers:
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
// v and 1/d live in tensor memory (all 512 columns: 2 x 64 a thread), d of
// a thread's first kDSmem values in shared memory, of the others in L2.
//
// 128 registers a thread and 227 KB of shared memory: one CTA an SM, which
// takes every ceil(J / wpc)-th window.  Waits are bounded as in
// agent_xpose.cuh: a warp whose wait for its copies gives up sets bit 2 of
// *err, and the CTA's threads agree at the next block barrier and stop.
//
// Measured (GB300, FP16 amplitudes, one sweep): 64009 windows 5.38 ms against
// 7.10 for the cluster form (3.5 TB/s of the 18 bytes a pixel the sweep must
// move: read q and y, write q), 14641 windows 1.22 against 1.66 ms, 900 windows
// (FP32) 91 against 125 us.  What bounds it: about 13.5 k of a window's 26 k
// cycles are instruction issue (75 % of it on the FP32 pipes), 8 k the
// shared-memory passes, and the store of 128 KB takes 4.1 k at the 32 bytes a
// cycle an SM can store; the block barriers keep the warps in step, so these
// overlap only in part.  Bulk stores of q' with plain loads of q, the other
// way round from what is built, were no faster (1.24 ms).
#pragma once

#include "agent_xpose.cuh"

namespace pmace {

struct RegGeom128 {
    static constexpr int N = 128;
    static constexpr int kThreads = 512;
    static constexpr int kWarps = 16;
    static constexpr int kRow = 34;                                   // values per row of E1
    static constexpr int kRegion = 32 * kRow * (int)sizeof(float2);   // bytes of a warp's region
    static constexpr int kDSmem = 22;                                 // values of d per thread in shared memory
    static constexpr int kOffD = kWarps * kRegion;
    static constexpr int kOffU = kOffD + kDSmem * kThreads * (int)sizeof(float2);
    static constexpr int kOffV = kOffU + kWarps * 8 * (int)sizeof(float2);
    static constexpr int kOffBar = kOffV + 32 * 4 * (int)sizeof(float2);
    static constexpr int kOffRed = kOffBar + kWarps * 8;
    static constexpr int kOffTm = kOffRed + kWarps * 4 * (int)sizeof(double);
    static constexpr int kOffConst = kOffTm + 16;
    static constexpr int kSmem = kOffConst + 32;
    static_assert(kRegion % 16 == 0 && kOffD % 16 == 0 && kOffU % 16 == 0 && kOffV % 16 == 0, "16-byte accesses");
    static_assert(8 * N * (int)sizeof(float2) <= kRegion, "the stack rows of a warp fit its region");
    static_assert(kSmem <= 227 * 1024, "shared memory of one CTA");
    // no second CTA of any kernel that allocates TMEM fits beside this one
    static_assert(2 * (kSmem + 1024) > 228 * 1024, "one CTA an SM");
};

// Copy `bytes` from global memory to this CTA's shared memory, counted on `bar`.
__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
                 "l"(src), "r"(bytes), "r"(bar)
                 : "memory");
}

// A read-only load that stays where it is written (the compiler moves plain
// ones up, which costs the registers they are meant to wait for).
__device__ __forceinline__ float2 ld_here(const float2* p) {
    float2 v;
    asm volatile("ld.global.nc.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "l"(p));
    return v;
}

// Pass 1 forward on x[4 rr + cc]: radix 4 over cc with the lane's twiddles
// v[kc] = W^(l kc), radix 8 over rr with the warp's u[kr] = W^(w kr); the
// result x[4 kr + kc].
__device__ __forceinline__ void reg_pass1(float2 (&x)[32], const float2* __restrict__ v, const float2* __restrict__ u) {
    const float4 v01 = reinterpret_cast<const float4*>(v)[0], v23 = reinterpret_cast<const float4*>(v)[1];
#pragma unroll
    for (int rr = 0; rr < 8; ++rr) {
        float2 s[4] = {x[4 * rr], x[4 * rr + 1], x[4 * rr + 2], x[4 * rr + 3]};
        Dft<4, false>::run(s);
        x[4 * rr] = s[0];
        x[4 * rr + 1] = cmul(s[1], make_float2(v01.z, v01.w));
        x[4 * rr + 2] = cmul(s[2], make_float2(v23.x, v23.y));
        x[4 * rr + 3] = cmul(s[3], make_float2(v23.z, v23.w));
    }
    const float4* u4 = reinterpret_cast<const float4*>(u);
    const float4 ua = u4[0], ub = u4[1], uc = u4[2], ud = u4[3];
#pragma unroll
    for (int kc = 0; kc < 4; ++kc) {
        float2 s[8];
#pragma unroll
        for (int rr = 0; rr < 8; ++rr) s[rr] = x[4 * rr + kc];
        Dft<8, false>::run(s);
        x[kc] = s[0];
        x[4 + kc] = cmul(s[1], make_float2(ua.z, ua.w));
        x[8 + kc] = cmul(s[2], make_float2(ub.x, ub.y));
        x[12 + kc] = cmul(s[3], make_float2(ub.z, ub.w));
        x[16 + kc] = cmul(s[4], make_float2(uc.x, uc.y));
        x[20 + kc] = cmul(s[5], make_float2(uc.z, uc.w));
        x[24 + kc] = cmul(s[6], make_float2(ud.x, ud.y));
        x[28 + kc] = cmul(s[7], make_float2(ud.z, ud.w));
    }
}

// Pass 1 back: the conjugate twiddles and inverse DFTs in reverse order.
__device__ __forceinline__ void reg_pass1_inv(float2 (&x)[32], const float2* __restrict__ v,
                                              const float2* __restrict__ u) {
    const float4* u4 = reinterpret_cast<const float4*>(u);
    const float4 ua = u4[0], ub = u4[1], uc = u4[2], ud = u4[3];
#pragma unroll
    for (int kc = 0; kc < 4; ++kc) {
        float2 s[8] = {x[kc],
                       cmulc(x[4 + kc], make_float2(ua.z, ua.w)),
                       cmulc(x[8 + kc], make_float2(ub.x, ub.y)),
                       cmulc(x[12 + kc], make_float2(ub.z, ub.w)),
                       cmulc(x[16 + kc], make_float2(uc.x, uc.y)),
                       cmulc(x[20 + kc], make_float2(uc.z, uc.w)),
                       cmulc(x[24 + kc], make_float2(ud.x, ud.y)),
                       cmulc(x[28 + kc], make_float2(ud.z, ud.w))};
        Dft<8, true>::run(s);
#pragma unroll
        for (int rr = 0; rr < 8; ++rr) x[4 * rr + kc] = s[rr];
    }
    const float4 v01 = reinterpret_cast<const float4*>(v)[0], v23 = reinterpret_cast<const float4*>(v)[1];
#pragma unroll
    for (int rr = 0; rr < 8; ++rr) {
        float2 s[4] = {x[4 * rr], cmulc(x[4 * rr + 1], make_float2(v01.z, v01.w)),
                       cmulc(x[4 * rr + 2], make_float2(v23.x, v23.y)), cmulc(x[4 * rr + 3], make_float2(v23.z, v23.w))};
        Dft<4, true>::run(s);
#pragma unroll
        for (int cc = 0; cc < 4; ++cc) x[4 * rr + cc] = s[cc];
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

// Windows j0, j0 + step, ... below J of the job `a` on one CTA.
template <int AMP>
__device__ __forceinline__ void reg128_body(const AgentArgs& a, const int j0, const int step) {
    using G = RegGeom128;
    constexpr int N = G::N, T = G::kThreads;
    constexpr int NCH = AMP ? 1 : 2;          // 16-byte chunks of eight amplitudes
    constexpr uint32_t kCopyBytes = 8 * N * sizeof(float2);

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

    if (t < 32) tmem_alloc(smem_addr(s_tm), 512u);
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
    if (t < 128) s_u[t] = a.tw[((t >> 3) * (t & 7)) & (N - 1)];                      // [w][kr]
    else if (t < 256) s_v[t - 128] = a.tw[(((t - 128) >> 2) * ((t - 128) & 3)) & (N - 1)];   // [l][kc]
    mbar_fence_init();
    fence_proxy_async_smem();
    tmem_fence_before_sync();
    __syncthreads();
    tmem_fence_after_sync();

    // v in columns 0..63 of the warp's lanes, 1/d in 64..127
    const uint32_t tm_v = *s_tm + ((uint32_t)(32 * (w & 3)) << 16) + 128u * (uint32_t)(w >> 2), tm_i = tm_v + 64u;
    const float2* __restrict__ d_l2 = a.probe + w * N + l;   // value e = 4 rr + cc at 16 N rr + 32 cc
    bool absent = false;   // whether one of the thread's pixels has its probe value treated as absent (1/d = 0)
#pragma unroll
    for (int h = 0; h < 4; ++h) {
        uint32_t r[16];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const int e = 8 * h + k, at = 16 * N * (e >> 2) + 32 * (e & 3);
            const float2 di = __ldg(a.dinv + w * N + l + at);
            absent |= di.x == 0.f && di.y == 0.f;
            r[2 * k] = __float_as_uint(di.x);
            r[2 * k + 1] = __float_as_uint(di.y);
            if (e < G::kDSmem) s_d[e * T + t] = __ldg(d_l2 + at);
        }
        tmem_st16(tm_i + 16u * h, r);
    }
    tmem_wait_st();

    constexpr float inv_n = 1.0f / (float)N;
    const bool first = a.first != 0;
    const bool res = a.residual != 0;
    const bool wu = a.u != nullptr;
    uint32_t parity = 0;

    // the warp's stack rows of window j into its region (lanes 0..7 a row each)
    auto load_stack = [&](int j) {
        if (l == 0) mbar_arrive_expect_tx(bar, kCopyBytes);
        __syncwarp();
        if (l < 8) bulk_load(region_s + 1024u * (uint32_t)l, a.q + ((size_t)j * N + w + 16 * l) * N, 1024u, bar);
    };
    // L2 prefetch of the warp's stack rows and amplitudes of a window
    auto prefetch = [&](int j) {
        if (l < 8) prefetch_l2(a.q + ((size_t)j * N + w + 16 * l) * N, 1024u);
        else if (l == 8) {
            constexpr uint32_t yb = N * N / G::kWarps * (AMP ? 2 : 4);
            prefetch_l2(static_cast<const char*>(a.y) + (size_t)j * N * N * (AMP ? 2 : 4) + (size_t)w * yb, yb);
        }
    };
    load_stack(j0);
    // Four groups of four warps take turns (a chain of named barriers) at the
    // reads that follow each block barrier, so that one group computes while
    // the next still reads: with all sixteen warps reading and then computing
    // together the 14641-window sweep took 1296 us instead of 1217.
    const int grp = w >> 2;
    auto turn_begin = [&](int id) {
        if (grp > 0) named_sync(id + grp - 1, T / 2);
    };
    auto turn_end = [&](int id) {
        if (grp < 3) named_arrive(id + grp, T / 2);
    };

    const size_t row16 = (size_t)16 * a.n2;
    // where the thread's consensus values of the window at `off` start
    auto xbar_at = [&](int2 off) { return a.xbar + (size_t)(off.x + w) * a.n2 + off.y + l; };
    // the window corner is loaded a window ahead
    int2 off_next = window_corner<N>(a, j0);
    float2 x[32];
    {
        const float2* __restrict__ xr = xbar_at(off_next);
#pragma unroll
        for (int e = 0; e < 32; ++e) x[e] = __ldg(xr + (e >> 2) * row16 + 32 * (e & 3));
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
        const bool got = mbar_wait_bounded(bar, parity, a.err);
        {
            const float2* st = reinterpret_cast<const float2*>(region) + l;
            const float2 trp2 = make_float2(s_const[1].x, s_const[1].y);
            float2 dl[32 - G::kDSmem];
            static_assert(G::kDSmem >= 20 && G::kDSmem < 32, "rows 5 to 7 are loaded four rows ahead");
#pragma unroll
            for (int rr = 0; rr < 8; ++rr) {
                if (rr >= 1 && rr <= 3) {   // the values of d that shared memory does not hold, four rows ahead
#pragma unroll
                    for (int cc = 0; cc < 4; ++cc)
                        if (4 * rr + 16 + cc >= G::kDSmem)
                            dl[4 * rr + 16 + cc - G::kDSmem] = ld_here(d_l2 + 16 * N * (rr + 4) + 32 * cc);
                }
                uint32_t r[8];
#pragma unroll
                for (int cc = 0; cc < 4; ++cc) {
                    const int e = 4 * rr + cc;
                    x[e] = mann_close2(st[N * rr + 32 * cc], x[e], trp2);
                    r[2 * cc] = __float_as_uint(x[e].x);
                    r[2 * cc + 1] = __float_as_uint(x[e].y);
                }
                tmem_st8(tm_v + 8u * rr, r);   // v, for the update
#pragma unroll
                for (int cc = 0; cc < 4; ++cc) {
                    const int e = 4 * rr + cc;
                    x[e] = cmul(e < G::kDSmem ? s_d[e * T + t] : dl[e < G::kDSmem ? 0 : e - G::kDSmem], x[e]);
                }
            }
        }
        reg_pass1(x, s_v + 4 * l, s_u + 8 * w);
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
        uint4 raw[4 * NCH];
        float yscale = 1.0f;
        {
            const uint4* yp = reinterpret_cast<const uint4*>(static_cast<const char*>(a.y) + wbase * (AMP ? 2 : 4)) + t;
            const uint64_t pol_first = l2_policy_evict_first();
#pragma unroll
            for (int k = 0; k < 4 * NCH; ++k) raw[k] = ld_nc_l2_hint(yp + k * T, pol_first);
            if constexpr (AMP == 1) yscale = __ldg(a.yscale + j);
        }
        if (__syncthreads_or(!got)) {
            // a wait that gave up stops the CTA; its warp's copies may still
            // be in flight: one more (bounded) wait before shared memory goes
            if (!got) mbar_wait_bounded(bar, parity, a.err);
            break;
        }
        parity ^= 1u;
        // ---- pass 3: row axis, S3 and back
        float acc_d = 0.f, acc_y = 0.f;
        {
            float4* mine = reinterpret_cast<float4*>(sm + 512 * w) + l;
            constexpr int RS4 = G::kRegion / 16;
            float2 z[2][16];
            turn_begin(1);
#pragma unroll
            for (int k = 0; k < 16; ++k) {
                const int i = 4 * (k % 4) + k / 4;   // in the order the radix-16 DFT takes them
                const float4 f = mine[RS4 * i];
                z[0][i] = make_float2(f.x, f.y);
                z[1][i] = make_float2(f.z, f.w);
            }
            turn_end(1);
            auto rows = [&](auto with_res) {
                constexpr bool kRes = decltype(with_res)::value;
#pragma unroll
                for (int b = 0; b < 2; ++b) {
                    Dft<16, false>::run(z[b]);
                    if (a.spectrum) {   // check of the forward transform, natural order
#pragma unroll
                        for (int i = 0; i < 16; ++i)
                            a.spectrum[wbase + (size_t)((l >> 2) + 8 * i) * N + (l & 3) + 4 * (2 * w + b)] = z[b][i];
                    }
#pragma unroll
                    for (int h = 0; h < 2; ++h) {   // eight at a time: registers
                        float yv[8];
                        unpack_amps8<AMP>(raw + NCH * (2 * b + h), yv);
                        replace_magnitudes<kRes>(reinterpret_cast<float2(&)[8]>(z[b][8 * h]), yv, inv_n, acc_d, acc_y,
                                                 AMP == 1 ? yscale : 1.0f);
                    }
                    Dft<16, true>::run(z[b]);
                }
            };
            if (res) rows(std::true_type{});
            else rows(std::false_type{});
#pragma unroll
            for (int i = 0; i < 16; ++i) mine[RS4 * i] = make_float4(z[0][i].x, z[0][i].y, z[1][i].x, z[1][i].y);
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
        reg_pass1_inv(x, s_v + 4 * l, s_u + 8 * w);
        // ---- S4 + S5, a row of four values at a time; the registers a row
        // frees take the consensus values of the next window (its own again
        // after the last one, which keeps the loads unconditional)
        float acc_z = 0.f, acc_w = 0.f;
        tmem_wait_st();   // v of the copy-in has landed
        {
            const float4 c0 = s_const[0], c1 = s_const[1];
            const float2 keep2 = make_float2(c0.x, c0.y), m2rho2 = make_float2(c0.z, c0.w);
            const float ds = AMP == 1 ? c1.z * yscale : c1.z;
            const float2 data2 = make_float2(ds, ds);
            const uint64_t pol_next = a.keep ? l2_policy_evict_last() : l2_policy_evict_normal();
            const uint64_t pol_q = wu ? l2_policy_evict_first() : pol_next;
            float2* qr = a.q + wbase + w * N + l;
            float2* __restrict__ ur = a.u + wbase + w * N + l;
            const float2* __restrict__ xr = xbar_at(off);
            const float2* __restrict__ xn = xbar_at(off_next);
#pragma unroll
            for (int rr = 0; rr < 8; ++rr) {
                uint32_t rv[8], ri[8];
                tmem_ld8x2(tm_v + 8u * rr, rv, tm_i + 8u * rr, ri);
                float2 v[4], wv[4];
#pragma unroll
                for (int cc = 0; cc < 4; ++cc) {
                    v[cc] = make_float2(__uint_as_float(rv[2 * cc]), __uint_as_float(rv[2 * cc + 1]));
                    const float2 dv = make_float2(__uint_as_float(ri[2 * cc]), __uint_as_float(ri[2 * cc + 1]));
                    wv[cc] = __ffma2_rn(keep2, v[cc], cmul(dv, __fmul2_rn(x[4 * rr + cc], data2)));
                }
                if (absent) {
#pragma unroll
                    for (int cc = 0; cc < 4; ++cc)
                        if (ri[2 * cc] << 1 == 0u && ri[2 * cc + 1] << 1 == 0u) wv[cc] = v[cc];   // 1/d is +-0
                }
                if (res) {
#pragma unroll
                    for (int cc = 0; cc < 4; ++cc)
                        residual_sums(first ? v[cc] : __ldg(xr + rr * row16 + 32 * cc), wv[cc], acc_z, acc_w);
                }
#pragma unroll
                for (int cc = 0; cc < 4; ++cc) {
                    const int at = 16 * N * rr + 32 * cc;
                    if (wu) st_l2_hint(ur + at, agent_u2(v[cc], wv[cc]), pol_next);
                    st_l2_hint(qr + at, __ffma2_rn(m2rho2, wv[cc], v[cc]), pol_q);
                }
#pragma unroll
                for (int cc = 0; cc < 4; ++cc) x[4 * rr + cc] = ld_here(xn + 32 * cc);
                xn += row16;
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
        tmem_dealloc(*s_tm, 512u);
    }
}

// One job: CTA k of G processes windows k, k + G, k + 2 G, ..., so that the
// CTAs are always within a few windows of one another in scan order and the
// consensus image they read stays in L2 (with contiguous runs the 64009-window
// sweep took 7.24 ms instead of 5.62).
template <int AMP>
__global__ void __launch_bounds__(RegGeom128::kThreads, 1) agent_reg128_kernel(const __grid_constant__ AgentArgs a) {
    reg128_body<AMP>(a, (int)blockIdx.x, (int)gridDim.x);
}

// Several jobs: CTA k takes the share of job work[k].x that starts at window
// work[k].y / wpc, every ceil(J / wpc)-th window.
template <int AMP>
__global__ void __launch_bounds__(RegGeom128::kThreads, 1)
agent_reg128_kernel_batched(const AgentArgs* __restrict__ descs, const int2* __restrict__ work) {
    const int2 wk = work[blockIdx.x];
    const AgentArgs& a = descs[wk.x];
    reg128_body<AMP>(a, wk.y / a.wpc, (a.J + a.wpc - 1) / a.wpc);
}

// Query (a == nullptr: fills info; a "cluster" is one CTA) or launch
// ceil(J / a->wpc) CTAs.
inline cudaError_t agent_reg128(const AgentArgs* a, int amp_f16, cudaStream_t s, AgentPlanInfo* info) {
    using G = RegGeom128;
    void (*fn)(const AgentArgs) = amp_f16 ? agent_reg128_kernel<1> : agent_reg128_kernel<0>;
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, G::kSmem);
    if (a == nullptr) {
        int dev = 0, nsm = 0;
        if (e == cudaSuccess) e = cudaGetDevice(&dev);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
        cudaGetLastError();
        info->threads = G::kThreads;
        info->smem_bytes = G::kSmem;
        info->max_clusters = e == cudaSuccess ? nsm : 0;
        info->launchable = info->max_clusters > 0;
        return cudaSuccess;
    }
    if (e != cudaSuccess) return e;
    if (a->wpc <= 0) return cudaErrorInvalidValue;
    fn<<<(unsigned)((a->J + a->wpc - 1) / a->wpc), G::kThreads, G::kSmem, s>>>(*a);
    return cudaGetLastError();
}

inline cudaError_t agent_reg128_batched(const AgentArgs* descs, const int2* work, int nctas, int amp_f16,
                                        cudaStream_t s) {
    using G = RegGeom128;
    if (nctas <= 0) return cudaSuccess;
    void (*fn)(const AgentArgs*, const int2*) = amp_f16 ? agent_reg128_kernel_batched<1> : agent_reg128_kernel_batched<0>;
    const cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, G::kSmem);
    if (e != cudaSuccess) return e;
    fn<<<(unsigned)nctas, G::kThreads, G::kSmem, s>>>(descs, work);
    return cudaGetLastError();
}

}  // namespace pmace
