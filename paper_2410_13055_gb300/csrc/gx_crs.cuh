// Cluster-resident message passing: the whole iteration loop of a scenario (forward dispatch
// or adjoint) in one launch, its state in shared memory.  The kernel template; its instances
// are compiled by gx_crs_fwd1.cu, gx_crs_fwd4.cu, gx_crs_adj1.cu and gx_crs_adj4.cu.
//
// One thread-block cluster of C CTAs per scenario; CTA r owns hours [r*H, (r+1)*H) of every
// bus, generator, load, line and battery injection.  Buses are coupled by lines only within an
// hour, so everything but the batteries stays in the CTA's own shared memory.  A battery couples
// all hours: it is owned by one CTA (b mod C), where kW warps run its prox.  One iteration:
//   A  every device prox, all of them depending only on the previous iteration's bus values:
//      the battery groups take their batteries, and every warp its share of the line, generator
//      and load items in chunks of 32, smaller for the warps that have batteries
//   B  the bus step: sums the devices' injections, consensus and dual update
// Between A and B the new injections of a battery travel to the CTAs that own its hours, and
// after B the prox targets v = x - p_bar - u of each battery-hour travel back to its owner: as
// asynchronous remote stores that complete on a shared-memory barrier of the receiver, so a CTA
// waits for the data it needs and not for the cluster.  Every check_every iterations the CTAs
// exchange residual partials over one cluster barrier and each takes the same stop decision
// from them, in FP64.
//
// What bounds it: shared-memory wavefronts and instruction issue where a CTA carries many hours
// (100 buses, 28 hours: 40,000 instructions and 9,800 wavefronts in 17,000 cycles, the wavefronts
// alone 58 % of it), the battery sweeps' dependent chain where it carries few; there is no
// per-iteration DRAM traffic.  Microseconds per iteration, forward and adjoint, against the
// per-iteration kernels:
//     5 buses x 24 h               1.5  1.3      7.2  6.6
//     100 buses x 24 h, 4 of them  2.4  2.4     11.4 10.1   (12 CTAs each)
//     100 buses x 168 h, 2         4.6  4.4     11.2  9.9   (14 CTAs each)
//     100 buses x 168 h, 16        8.4  8.2     15.4 14.1   (6 CTAs each)
//     400 buses x 1 h, 24          4.8  4.4     13.1 13.0
// With remote loads by the batteries and two cluster barriers per iteration, the form before this
// one, the last four took 3.6, 7.0, 12.2 and 5.9 (forward): a battery waited 9,500 cycles for its
// scattered loads and each barrier took 600 to 2,300.  Hence the layout: rows of H hours per device, a thread item being kV consecutive hours (a float4 for
// kV = 4; one hour where the network is too small to fill the threads with quads); devices
// renumbered so that a bus's generators, line ends and batteries are consecutive rows, and buses
// sorted by device count, so that a warp's lanes walk lists of equal length; every per-device
// constant (line coefficients, capacities, reciprocal pivots, scan multipliers) computed once at
// entry.
//
// The arithmetic of every step is that of the per-iteration kernels (gx_kernels.cu), in the same
// order, so a scenario takes bitwise the same iterates on either path; only the residual
// partials are summed in another order: FP32 within an item (at most four hours of a device or bus),
// pairs of floats over a thread's items and a warp's lanes (about 48 bits), FP64 from there on.
// State is read from and written back to the workspace rows at entry and exit, so the reset,
// mask, extraction and gradient kernels work unchanged.
#pragma once
#include "gx_async.cuh"
#include "gx_internal.cuh"

#include <cfloat>
#include <cooperative_groups.h>
#include <type_traits>

namespace cg = cooperative_groups;

namespace gx {

namespace {

__device__ __forceinline__ float clampf(float x, float lo, float hi) { return fminf(fmaxf(x, lo), hi); }

// ---------------------------------------------------------------- cluster primitives
__device__ __forceinline__ unsigned map_rank(unsigned a, int rank) {
    unsigned r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
    return r;
}
__device__ __forceinline__ float ld_cluster(unsigned a) {
    float v;
    asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(a) : "memory");
    return v;
}
// Remote stores that count their bytes on the receiver's mbarrier.
__device__ __forceinline__ void st_async1(unsigned a, float v, unsigned bar) {
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.f32 [%0], %1, [%2];" ::"r"(a), "f"(v), "r"(bar)
                 : "memory");
}
__device__ __forceinline__ void st_async4(unsigned a, float x, float y, float z, float w, unsigned bar) {
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.f32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(a),
                 "f"(x), "f"(y), "f"(z), "f"(w), "r"(bar)
                 : "memory");
}
// One bounded probe, acquiring what the cluster's remote stores wrote.
__device__ __forceinline__ bool mbar_try_cluster(unsigned long long* bar, unsigned parity) {
    unsigned ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, "
        "0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_addr(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

// kV consecutive hours of a row
template <int kV>
__device__ __forceinline__ void ldv(const float* p, float (&v)[kV]) {
    if constexpr (kV == 4) {
        const float4 q = *reinterpret_cast<const float4*>(p);
        v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
    } else {
        v[0] = *p;
    }
}
template <int kV>
__device__ __forceinline__ void stv(float* p, const float (&v)[kV]) {
    if constexpr (kV == 4) *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
    else *p = v[0];
}

// Integer division by a small constant of the launch (q < 2^16): multiply-high by
// ceil(2^32 / d); d = 1 is kept apart.
struct FastDiv {
    unsigned d, m;
    __device__ __forceinline__ explicit FastDiv(int n) : d((unsigned)n), m(n > 1 ? (unsigned)((0x100000000ULL + n - 1) / n) : 0u) {}
    __device__ __forceinline__ int div(int q) const { return d == 1 ? q : (int)__umulhi((unsigned)q, m); }
};

// Items 0 to n - 1 over the block's threads, kU of a thread's at a time: ld(q) reads from global
// memory, st(q, v) stores.  The compiler keeps a load behind a store that might alias it, so a plain
// copy loop waits for one round trip to L2 per value; here a thread's kU items are in flight together
// (16 x 168 h of 100 buses, a launch more per loop: 43 us, 52 with plain loops).
template <int kU, class V, class Ld, class St>
__device__ __forceinline__ void batched(int n, int tid, int nt, Ld ld, St st) {
    for (int q0 = tid; q0 < n; q0 += kU * nt) {
        V v[kU];
#pragma unroll
        for (int k = 0; k < kU; ++k) v[k] = ld(min(q0 + k * nt, n - 1));
#pragma unroll
        for (int k = 0; k < kU; ++k)
            if (q0 + k * nt < n) st(q0 + k * nt, v[k]);
    }
}
struct BusIn { float pbar, u, thb, xl, ld; };
struct LineIn { float dl, vf, vt; int from, to; };
struct BatIn { float xb; int slot; };

// Operand order of the fused multiply-adds.  The iterates of this path equal those of the
// per-iteration kernels bit for bit, so every sum of products that the compiler could fuse either
// way is written out: fma_first fuses a x and rounds b y, fma_second the reverse.
__device__ __forceinline__ float fma_first(float a, float x, float b, float y) { return __fmaf_rn(a, x, __fmul_rn(b, y)); }
__device__ __forceinline__ float fma_second(float a, float x, float b, float y) { return __fmaf_rn(b, y, __fmul_rn(a, x)); }

// a / b from the correctly rounded reciprocal r of b: two residual corrections, each a fused
// multiply-add pair; by Markstein's theorem (IBM J. Res. Dev. 34, 1990) the second one's result is the correctly
// rounded quotient, as the division of the per-iteration kernels gives it (away from overflow and
// the subnormals).  No branch, and half the instructions.
__device__ __forceinline__ float quotient(float a, float b, float r) {
    float q = __fmul_rn(a, r);
    q = __fmaf_rn(__fmaf_rn(-b, q, a), r, q);
    return __fmaf_rn(__fmaf_rn(-b, q, a), r, q);
}

// A residual sum: the rounding errors of hi, each exact (Knuth's two-sum), are summed in lo.  Most
// of a scenario's terms meet in one CTA, so plain FP32 sums would round some 40 times on the way to
// the total where the per-iteration kernels go to FP64 after 128 threads; and the dual residual's
// device and bus parts, which cancel, meet here only in the sum.  0.2 to 1.5 % of a pass.
struct Sum2 {
    float hi, lo;
    __device__ __forceinline__ void add(float v) {
        const float s = __fadd_rn(hi, v), b = __fsub_rn(s, hi);
        lo = __fadd_rn(lo, __fadd_rn(__fsub_rn(hi, __fsub_rn(s, b)), __fsub_rn(v, b)));
        hi = s;
    }
    __device__ __forceinline__ void add(float h, float l) {
        add(h);
        lo = __fadd_rn(lo, l);
    }
};

// The sums of a residual check: |n| pbar^2 and the phase mismatch; the adjoint scale; |z^k - z^{k-1}|^2
// (devices' dx^2 less the buses' part); dthbar^2 w; |rho u|^2; and x^2, which is there for the test
// of finiteness alone and so a plain FP32 sum.
struct ResSums {
    Sum2 n, scale, dz, dth, u;
    float x;
};

// The warp's totals, sum k of ResSums in lanes 4 k to 4 k + 3: a step that can halves the sums that
// a lane carries.
__device__ __forceinline__ Sum2 warp_sums(const ResSums& a, int lane) {
    Sum2 v[8] = {a.n, a.scale, a.dz, a.dth, a.u, Sum2{a.x, 0.f}, Sum2{0.f, 0.f}, Sum2{0.f, 0.f}};
#pragma unroll
    for (int n = 4; n >= 1; n >>= 1) {
        const int bit = 4 * n;
        const bool up = lane & bit;
#pragma unroll
        for (int q = 0; q < n; ++q) {
            const Sum2 out = up ? v[q] : v[q + n];
            if (up) v[q] = v[q + n];
            v[q].add(__shfl_xor_sync(0xffffffffu, out.hi, bit), __shfl_xor_sync(0xffffffffu, out.lo, bit));
        }
    }
#pragma unroll
    for (int bit = 2; bit >= 1; bit >>= 1)
        v[0].add(__shfl_xor_sync(0xffffffffu, v[0].hi, bit), __shfl_xor_sync(0xffffffffu, v[0].lo, bit));
    return v[0];
}

struct GState {
    float *xg, *xl, *dl, *sg, *vf, *vt, *xb, *zc, *u, *pbar, *thb;
    long long zstride;  // zc, zd, zs, yc, yd, ys lie this many floats apart
};

struct Sm {
    double* red;     // [2][C][kCrsRed] residual partials of every rank (two chunks' slots)
    Sum2* wred;      // [warps][kCrsRed - 1]
    float* xch;      // [warps][8] two-warp exchange of the battery prox
    unsigned long long* bar;  // [0] battery injections have arrived, [1] prox targets have arrived
    int* flag;       // [0] stop, [1] a bounded wait gave up, [2] that as of a residual check
    int4* busr;      // [N] generator rows, first line-end slot, first battery slot, counts (12, 12, 8 bits)
    float4* busf;    // [N] 1/terminals, 1/sum of phase weights, dual-residual weight
    int2* genr;      // [G] bus row offset, cost
    int4* endr;      // [2L + 1] line row offset, signed beta, phase weight; a zero entry
    int4* liner;     // [L] from / to bus row offsets, from / to end row offsets
    float4* linef;   // [L] beta, rho beta, rho_theta / 2, denominator
    float4* linec;   // [L] flow / angle cap, phase weight, 1 / denominator
    int2* bslot;     // [B] the prox-target row of each injection slot's battery at its owner, its barrier there
    int4* batr;      // [nbo][2] injection row offset, its bytes, pivot row, index; P, E, a, k
    float2* batg;    // [nbo] dc/dmu, dd/dmu
    float* idd;      // [rows][T] reciprocal pivots
    float* scan;     // [rows][12][lanes] multipliers of the battery sweeps' scans
    float *pbar, *u, *thb, *xl, *ld, *xg, *cap, *dl, *q, *xb, *vrow, *bst;
    uint8_t* lmask;
};

__device__ __forceinline__ Sm sm_at(unsigned char* b, const CrsOff& o) {
    Sm m;
    m.red = reinterpret_cast<double*>(b + o.red);
    m.wred = reinterpret_cast<Sum2*>(b + o.wred);
    m.xch = reinterpret_cast<float*>(b + o.xch);
    m.bar = reinterpret_cast<unsigned long long*>(b + o.bar);
    m.flag = reinterpret_cast<int*>(b + o.flag);
    m.busr = reinterpret_cast<int4*>(b + o.busr);
    m.busf = reinterpret_cast<float4*>(b + o.busf);
    m.genr = reinterpret_cast<int2*>(b + o.genr);
    m.endr = reinterpret_cast<int4*>(b + o.endr);
    m.liner = reinterpret_cast<int4*>(b + o.liner);
    m.linef = reinterpret_cast<float4*>(b + o.linef);
    m.linec = reinterpret_cast<float4*>(b + o.linec);
    m.bslot = reinterpret_cast<int2*>(b + o.bslot);
    m.batr = reinterpret_cast<int4*>(b + o.batr);
    m.batg = reinterpret_cast<float2*>(b + o.batg);
    m.idd = reinterpret_cast<float*>(b + o.idd);
    m.scan = reinterpret_cast<float*>(b + o.scan);
    m.pbar = reinterpret_cast<float*>(b + o.pbar);
    m.u = reinterpret_cast<float*>(b + o.u);
    m.thb = reinterpret_cast<float*>(b + o.thb);
    m.xl = reinterpret_cast<float*>(b + o.xl);
    m.ld = reinterpret_cast<float*>(b + o.ld);
    m.xg = reinterpret_cast<float*>(b + o.xg);
    m.cap = reinterpret_cast<float*>(b + o.cap);
    m.dl = reinterpret_cast<float*>(b + o.dl);
    m.q = reinterpret_cast<float*>(b + o.q);
    m.xb = reinterpret_cast<float*>(b + o.xb);
    m.vrow = reinterpret_cast<float*>(b + o.vrow);
    m.bst = reinterpret_cast<float*>(b + o.bst);
    m.lmask = b + o.lmask;
    return m;
}

// Wait for phase `parity` of one of the CTA's barriers.  The wait is bounded: on expiry the CTA's
// failure flag and the workspace's error word are set, the iteration goes on with what is there,
// and every rank stops at the chunk's reduction, which carries the flag.
__device__ __forceinline__ void res_wait(const Ctx& c, const Sm& m, int which, unsigned parity) {
    for (int k = 0; k < kWaitProbes; ++k) {
        if (mbar_try_cluster(m.bar + which, parity)) return;
        if ((k & 1023) == 1023 && *reinterpret_cast<volatile int*>(m.flag + 1)) return;
    }
    *reinterpret_cast<volatile int*>(m.flag + 1) = 1;
    atomicExch(c.err, GX_ERR_TIMEOUT);
}

// Constants of the battery prox, the same for every battery.
struct BatConst {
    float rho, ri, iri, Ah, idet;
};

// One prox of an owned battery (the battery kernel's inner ADMM: box copy z, scaled duals y,
// the equality-constrained step through the constant tridiagonal system, its two sweeps as
// affine scans over the lanes).  The scans' multipliers depend on the pivots alone: they come
// from a table (per direction the multiplier of each of the five steps, 0 for lanes without a
// partner, then the whole prefix's), so a step is one shuffle and one multiply-add.  Hours past
// the horizon carry zero pivots and zero state, which the sweeps leave at zero.
// s6: the lane's hours of the state (z then y), kept in registers by the caller (kReg) or read
// from and written to st (rows sstride apart).  The prox targets come from the battery's row
// (m.vrow); the new injections go to the owners of the hours: lane by lane (kV = 1), or through
// the same row as float4s.  qa, qb: per lane the address of its hours (kV = 1) or quad (kV = 4) in
// the owner's injection array, and the owner's barrier.
template <int WANT, int ADJ, int kHpl, int kW, int kV, int kReg>
__device__ __forceinline__ void res_battery(const Ctx& c, const Sm& m, const BatConst& K, int T, int TR, int HS, bool multi,
                                            const unsigned (&qa)[kV == 4 ? 1 : kHpl],
                                            const unsigned (&qb)[kV == 4 ? 1 : kHpl], int slot, int group,
                                            float (&s6)[6][kHpl], float* st, long long sstride, long long row0,
                                            ResSums& acc) {
    constexpr int NL = 32 * kW;
    const int Lx = threadIdx.x & (NL - 1);
    const int lane = Lx & 31, wb = Lx >> 5;
    float* xch = m.xch + group * 8;
    auto sync = [&]() {
        if (kW == 2) asm volatile("bar.sync %0, %1;" ::"r"(group + 1), "n"(NL) : "memory");
        else __syncwarp();
    };
    const int4 br = m.batr[2 * slot];
    const int4 bp = m.batr[2 * slot + 1];
    const float2 bg = m.batg[slot];
    const float P = __int_as_float(bp.x), E = __int_as_float(bp.y), a = __int_as_float(bp.z), k = __int_as_float(bp.w);
    const float gc = bg.x, gd = bg.y;
    float* vr = m.vrow + slot * TR;
    const float* ird = m.idd + br.z * T;
    const float* sc = m.scan + br.z * (12 * NL) + Lx;
    const int t0 = Lx * kHpl, nv = T - t0;  // the lane's first hour; valid hours j < nv
    const float rho = K.rho, ri = K.ri, iri = K.iri, Ah = K.Ah, idet = K.idet;

    float v[kHpl], idd[kHpl], iddp[kHpl], qc[kHpl], qd[kHpl];
    int mk[kHpl];  // adjoint: active-set code of the hour (c, d, s two bits each)
#pragma unroll
    for (int j = 0; j < kHpl; ++j) {
        const int t = t0 + j, tc = min(t, T - 1);
        const bool ok = j < nv;
        v[j] = vr[tc];
        if (!kReg)
#pragma unroll
            for (int r = 0; r < 6; ++r) s6[r][j] = st[r * sstride + tc];
        idd[j] = ird[tc];
        iddp[j] = ird[max(tc - 1, 0)];
        qc[j] = qd[j] = 0.f;
        mk[j] = 0;
        if (ADJ) {
            mk[j] = c.m_bat[row0 + tc];
            qc[j] = -c.eps * c.zc[row0 + tc];
            qd[j] = -c.eps * c.zd[row0 + tc];
        }
        v[j] = ok ? v[j] : 0.f;
        if (!kReg)
#pragma unroll
            for (int r = 0; r < 6; ++r) s6[r][j] = ok ? s6[r][j] : 0.f;
        idd[j] = ok ? idd[j] : 0.f;
        iddp[j] = ok && t > 0 ? iddp[j] : 0.f;
        if (ADJ) {
            qc[j] = ok ? qc[j] : 0.f;
            qd[j] = ok ? qd[j] : 0.f;
        }
    }
    float(&zc)[kHpl] = s6[0];
    float(&zd)[kHpl] = s6[1];
    float(&zs)[kHpl] = s6[2];
    float(&yc)[kHpl] = s6[3];
    float(&yd)[kHpl] = s6[4];
    float(&ys)[kHpl] = s6[5];
    float xn[kHpl];
#pragma unroll
    for (int j = 0; j < kHpl; ++j) xn[j] = 0.f;

    for (int it = 0; it < c.inner_iters; ++it) {
        float c0[kHpl], d0[kHpl], rs[kHpl], rhs[kHpl];
#pragma unroll
        for (int j = 0; j < kHpl; ++j) {
            const float rc = __fsub_rn(zc[j], __fmul_rn(yc[j], iri)), rd = __fsub_rn(zd[j], __fmul_rn(yd[j], iri));
            rs[j] = __fsub_rn(zs[j], __fmul_rn(ys[j], iri));
            float b1 = fma_first(ri, rc, -rho, v[j]);
            float b2 = fma_first(ri, rd, rho, v[j]);
            if (ADJ) { b1 = __fsub_rn(b1, qc[j]); b2 = __fsub_rn(b2, qd[j]); }
            if (kHpl == 1 && kW == 1 && !ADJ) {
                // (the forward battery kernel for horizons up to 32 hours fuses this pair the other way round)
                const bool sw = c.max_bat_T <= 32;
                const float p = sw ? rho : Ah, x = sw ? b2 : b1, q = sw ? Ah : rho, y = sw ? b1 : b2;
                c0[j] = __fmul_rn(fma_first(p, x, q, y), idet);
                d0[j] = __fmul_rn(fma_first(q, x, p, y), idet);
            } else {
                c0[j] = __fmul_rn(fma_first(Ah, b1, rho, b2), idet);
                d0[j] = __fmul_rn(fma_first(rho, b1, Ah, b2), idet);
            }
        }
        // previous hour's r_s for the first hour of the chunk (0 before hour 0)
        float rs_prev = __shfl_up_sync(0xffffffffu, rs[kHpl - 1], 1);
        if (kW == 2) {
            if (Lx == 31) xch[0] = rs[kHpl - 1];
            sync();
        }
        if (lane == 0) rs_prev = (kW == 2 && wb == 1) ? xch[0] : 0.f;
        // forward sweep y_t = rhs_t + y_{t-1} / dd_{t-1}
        float Bv = 0.f;
#pragma unroll
        for (int j = 0; j < kHpl; ++j) {
            const float prev = j == 0 ? rs_prev : rs[j > 0 ? j - 1 : 0];
            rhs[j] = __fmul_rn(ri, __fsub_rn(__fsub_rn(rs[j], prev), fma_first(a, c0[j], -k, d0[j])));
            Bv = __fmaf_rn(iddp[j], Bv, rhs[j]);
        }
#pragma unroll
        for (int o = 0; o < 5; ++o) {
            const float Bo = __shfl_up_sync(0xffffffffu, Bv, 1 << o);
            Bv = __fmaf_rn(sc[o * NL], Bo, Bv);
        }
        float yin = __shfl_up_sync(0xffffffffu, Bv, 1);
        if (kW == 2) {
            // the second warp's prefixes start from the first warp's total
            if (Lx == 31) xch[2] = Bv;
            sync();
            if (wb == 1) {
                const float B0 = xch[2];
                Bv = __fmaf_rn(sc[5 * NL], B0, Bv);
                const float yw = __shfl_up_sync(0xffffffffu, Bv, 1);
                yin = lane == 0 ? B0 : yw;
            }
        }
        if (lane == 0 && !(kW == 2 && wb == 1)) yin = 0.f;
        float yv[kHpl];
#pragma unroll
        for (int j = 0; j < kHpl; ++j) {
            yin = __fmaf_rn(iddp[j], yin, rhs[j]);
            yv[j] = yin;
        }
        // backward sweep mu_t = (y_t + mu_{t+1}) / dd_t, mu_T = 0
        Bv = 0.f;
#pragma unroll
        for (int j = kHpl - 1; j >= 0; --j) Bv = fma_first(idd[j], Bv, idd[j], yv[j]);
#pragma unroll
        for (int o = 0; o < 5; ++o) {
            const float Bo = __shfl_down_sync(0xffffffffu, Bv, 1 << o);
            Bv = __fmaf_rn(sc[(6 + o) * NL], Bo, Bv);
        }
        float min_ = __shfl_down_sync(0xffffffffu, Bv, 1);
        if (kW == 2) {
            // the first warp's suffixes continue into the second warp's total
            if (Lx == 32) xch[4] = Bv;
            sync();
            if (wb == 0) {
                const float B1 = xch[4];
                Bv = __fmaf_rn(sc[11 * NL], B1, Bv);
                const float mw = __shfl_down_sync(0xffffffffu, Bv, 1);
                min_ = lane == 31 ? B1 : mw;
            }
        }
        if (lane == 31 && !(kW == 2 && wb == 0)) min_ = 0.f;
        float mu[kHpl];
        float mnext = min_;
#pragma unroll
        for (int j = kHpl - 1; j >= 0; --j) {
            mnext = __fmul_rn(idd[j], __fadd_rn(yv[j], mnext));
            mu[j] = mnext;
        }
        // x = (c, d, s), then the box projection and the inner dual step
#pragma unroll
        for (int j = 0; j < kHpl; ++j) {
            const float mu_n = j + 1 < kHpl ? mu[j + 1 < kHpl ? j + 1 : j] : min_;
            const float cc = __fmaf_rn(mu[j], gc, c0[j]);
            const float dd_ = __fmaf_rn(mu[j], gd, d0[j]);
            const float ss = __fmaf_rn(-__fsub_rn(mu[j], mu_n), iri, rs[j]);
            const float tc = __fadd_rn(cc, __fmul_rn(yc[j], iri)), td = __fadd_rn(dd_, __fmul_rn(yd[j], iri)),
                        ts = __fadd_rn(ss, __fmul_rn(ys[j], iri));
            float nzc, nzd, nzs;
            if (ADJ) {
                // fixed components of the active set stay at 0; free ones are unbounded
                nzc = (mk[j] & 3) != A_FREE ? 0.f : clampf(tc, -FLT_MAX, FLT_MAX);
                nzd = ((mk[j] >> 2) & 3) != A_FREE ? 0.f : clampf(td, -FLT_MAX, FLT_MAX);
                nzs = ((mk[j] >> 4) & 3) != A_FREE ? 0.f : clampf(ts, -FLT_MAX, FLT_MAX);
            } else {
                nzc = clampf(tc, 0.f, P);
                nzd = clampf(td, 0.f, P);
                nzs = clampf(ts, 0.f, E);
            }
            yc[j] = __fmaf_rn(ri, __fsub_rn(cc, nzc), yc[j]);
            yd[j] = __fmaf_rn(ri, __fsub_rn(dd_, nzd), yd[j]);
            ys[j] = __fmaf_rn(ri, __fsub_rn(ss, nzs), ys[j]);
            zc[j] = nzc; zd[j] = nzd; zs[j] = nzs;
            xn[j] = __fsub_rn(dd_, cc);
        }
    }
    // Before the new injections are sent: once they have arrived, the buses' new prox targets may
    // come back into the row.
    if (!kReg)
#pragma unroll
        for (int j = 0; j < kHpl; ++j)
            if (j < nv)
#pragma unroll
                for (int r = 0; r < 6; ++r) st[r * sstride + t0 + j] = s6[r][j];
    float* xl = m.xb + br.x;  // local row of the battery's injections (multi: this rank's hours)
    if (WANT) {
        float dx2 = 0.f, x2 = 0.f;
#pragma unroll
        for (int j = 0; j < kHpl; ++j) {
            if (j >= nv) continue;
            const int t = t0 + j, rk = t / HS;
            const float old = multi ? ld_cluster(map_rank(smem_addr(xl + (t - rk * HS)), rk)) : xl[t];
            dx2 += (xn[j] - old) * (xn[j] - old);
            x2 += xn[j] * xn[j];
        }
        acc.dz.add(dx2);
        acc.x += x2;
        sync();  // every lane has read the old injections before a lane of another order sends new ones
    }
    if (!multi) {
#pragma unroll
        for (int j = 0; j < kHpl; ++j)
            if (j < nv) xl[t0 + j] = xn[j];
    } else if (kV == 1) {
#pragma unroll
        for (int j = 0; j < kHpl; ++j)
            if (j < nv) st_async1(qa[j] + br.y, xn[j], qb[j]);
    } else {
#pragma unroll
        for (int j = 0; j < kHpl; ++j)
            if (j < nv) vr[t0 + j] = xn[j];
        sync();
        if (4 * Lx < TR) {
            const float4 x = *reinterpret_cast<const float4*>(vr + 4 * Lx);
            st_async4(qa[0] + br.y, x.x, x.y, x.z, x.w, qb[0]);
        }
    }
}

// The scan multipliers of one pivot row (see res_battery), by the lanes of one warp group.
template <int kHpl, int kW>
__device__ __forceinline__ void res_scan_table(const float* ird, float* sc, int T) {
    constexpr int NL = 32 * kW;
    const int Lx = threadIdx.x & (NL - 1), lane = Lx & 31, t0 = Lx * kHpl;
    float A = 1.f, D = 1.f;
#pragma unroll
    for (int j = 0; j < kHpl; ++j) A = __fmul_rn(t0 + j < T && t0 + j > 0 ? ird[t0 + j - 1] : 0.f, A);
#pragma unroll
    for (int j = kHpl - 1; j >= 0; --j) D = __fmul_rn(t0 + j < T ? ird[t0 + j] : 0.f, D);
#pragma unroll
    for (int o = 0; o < 5; ++o) {
        const float Ao = __shfl_up_sync(0xffffffffu, A, 1 << o), Do = __shfl_down_sync(0xffffffffu, D, 1 << o);
        const bool up = lane >= (1 << o), down = lane + (1 << o) < 32;
        sc[o * NL + Lx] = up ? A : 0.f;
        sc[(6 + o) * NL + Lx] = down ? D : 0.f;
        if (up) A = __fmul_rn(A, Ao);
        if (down) D = __fmul_rn(D, Do);
    }
    sc[5 * NL + Lx] = A;
    sc[11 * NL + Lx] = D;
}

// One line item (phase-dual update and the clipped 1-D minimiser).  sigma is read only by the
// residual: it stays in the workspace row, written in the iteration before a residual (store_sg)
// and in the residual iteration.
template <int WANT, int ADJ, int kV>
__device__ __forceinline__ void res_line(const Ctx& c, const Sm& m, float* sg, long long row, int HS, int l, int hq,
                                         int store_sg, ResSums& acc) {
    float dx2 = 0.f, x2 = 0.f, th2 = 0.f;
    const int hl = hq * kV;
    const int4 lr = m.liner[l];
    const float4 lf = m.linef[l];
    const float4 lc = m.linec[l];
    const float beta = lf.x, cap = lc.x, lw = lc.y;
    float d[kV], qf[kV], qt[kV], pbf[kV], uf[kV], zf[kV], pbt[kV], ut[kV], zt[kV];
    float* pd = m.dl + l * HS + hl;
    float* pqf = m.q + lr.z + hl;
    float* pqt = m.q + lr.w + hl;
    ldv<kV>(pd, d); ldv<kV>(pqf, qf); ldv<kV>(pqt, qt);
    ldv<kV>(m.pbar + lr.x + hl, pbf); ldv<kV>(m.u + lr.x + hl, uf); ldv<kV>(m.thb + lr.x + hl, zf);
    ldv<kV>(m.pbar + lr.y + hl, pbt); ldv<kV>(m.u + lr.y + hl, ut); ldv<kV>(m.thb + lr.y + hl, zt);
    const bool dc = lw == 0.f;  // HVDC transport line: no phase coupling, eps/2 f^2 cost
    const unsigned mk = ADJ ? m.lmask[l * (HS / kV) + hq] : 0u;  // one bit per hour
    const long long gr = row + hl;
    float fs[kV], g[kV];
#pragma unroll
    for (int h = 0; h < kV; ++h) fs[h] = g[h] = 0.f;
    if (ADJ && dc) ldv<kV>(c.dl + gr, fs);  // adjoint of a transport line: eps f* of grad h
    if (WANT) ldv<kV>(sg + gr, g);
    float dn[kV], gn[kV], nf[kV], nt[kV];
#pragma unroll
    for (int h = 0; h < kV; ++h) {
        const float vf = qf[h] - zf[h], vt = qt[h] - zt[h];
        if (WANT && !dc) {
            const float ef = 0.5f * (g[h] + d[h]) - zf[h], et = 0.5f * (g[h] - d[h]) - zt[h];
            th2 += beta * beta * (ef * ef + et * et);
        }
        const float wf = zf[h] - vf, wt = zt[h] - vt;
        const float tf = __fsub_rn(__fmaf_rn(-beta, d[h], -pbf[h]), uf[h]);
        const float tt = __fsub_rn(__fmaf_rn(beta, d[h], -pbt[h]), ut[h]);
        float num = fma_second(lf.y, __fsub_rn(tt, tf), lf.z, __fsub_rn(wf, wt));
        if (ADJ) num = __fmaf_rn(c.eps, fs[h], num);
        const float dun = quotient(num, lf.w, lc.z);
        if (ADJ) dn[h] = (mk >> h) & 1u ? 0.f : dun;
        else dn[h] = clampf(dun, -cap, cap);
        gn[h] = wf + wt;
        nf[h] = __fmaf_rn(0.5f, __fadd_rn(gn[h], dn[h]), vf);
        nt[h] = __fmaf_rn(0.5f, __fsub_rn(gn[h], dn[h]), vt);
        if (WANT) {
            const float dd = dn[h] - d[h];
            dx2 += 2.f * beta * beta * dd * dd;
            x2 += 2.f * beta * beta * dn[h] * dn[h];
        }
    }
    if (WANT) {
        acc.dz.add(dx2);
        acc.x += x2;
        acc.n.add(th2);
    }
    stv<kV>(pd, dn); stv<kV>(pqf, nf); stv<kV>(pqt, nt);
    if (WANT || store_sg) stv<kV>(sg + gr, gn);
}

// One generator item: clip (forward) or masked step (adjoint).
template <int WANT, int ADJ, int kV>
__device__ __forceinline__ void res_gen(const Sm& m, float rho, float inv_re, int HS, int g, int hl, ResSums& acc) {
    float dx2 = 0.f, x2 = 0.f, scale = 0.f;
    const int2 gr = m.genr[g];
    const float cost = __int_as_float(gr.y);
    float x[kV], a[kV], pb[kV], uu[kV], xn[kV];
    float* px = m.xg + g * HS + hl;
    ldv<kV>(px, x); ldv<kV>(m.cap + g * HS + hl, a);
    ldv<kV>(m.pbar + gr.x + hl, pb); ldv<kV>(m.u + gr.x + hl, uu);
#pragma unroll
    for (int h = 0; h < kV; ++h) {
        const float v = x[h] - pb[h] - uu[h];
        if (ADJ) {
            const float gh = a[h];  // NaN: bound active, the variable is fixed at 0
            const bool fixed = gh != gh;
            xn[h] = fixed ? 0.f : __fmul_rn(__fmaf_rn(rho, v, gh), inv_re);
            if (WANT && !fixed) scale += (gh * inv_re) * (gh * inv_re);
        } else {
            xn[h] = clampf(__fmul_rn(__fmaf_rn(rho, v, -cost), inv_re), 0.f, a[h]);
        }
        if (WANT) {
            dx2 += (xn[h] - x[h]) * (xn[h] - x[h]);
            x2 += xn[h] * xn[h];
        }
    }
    if (WANT) {
        if (ADJ) acc.scale.add(scale);
        acc.dz.add(dx2);
        acc.x += x2;
    }
    stv<kV>(px, xn);
}

// One load item (shed variable; terminal injection shed - L).
template <int WANT, int ADJ, int kV>
__device__ __forceinline__ void res_load(const Sm& m, float rho, float inv_re, float voll, int i, ResSums& acc) {
    float dx2 = 0.f, x2 = 0.f, scale = 0.f;
    float x[kV], Ld[kV], pb[kV], uu[kV], xn[kV];
    ldv<kV>(m.xl + i, x); ldv<kV>(m.ld + i, Ld); ldv<kV>(m.pbar + i, pb); ldv<kV>(m.u + i, uu);
#pragma unroll
    for (int h = 0; h < kV; ++h) {
        const float v = x[h] - pb[h] - uu[h];
        if (ADJ) {
            const float gsh = Ld[h];  // adjoint coefficient; NaN: bound active
            const bool fixed = gsh != gsh;
            xn[h] = fixed ? 0.f : __fmul_rn(__fmaf_rn(rho, v, gsh), inv_re);
            if (WANT && !fixed) scale += (gsh * inv_re) * (gsh * inv_re);
        } else {
            xn[h] = clampf(__fmul_rn(__fmaf_rn(rho, __fadd_rn(v, Ld[h]), -voll), inv_re), 0.f, Ld[h]) - Ld[h];
        }
        if (WANT) {
            dx2 += (xn[h] - x[h]) * (xn[h] - x[h]);
            x2 += xn[h] * xn[h];
        }
    }
    if (WANT) {
        if (ADJ) acc.scale.add(scale);
        acc.dz.add(dx2);
        acc.x += x2;
    }
    stv<kV>(m.xl + i, xn);
}

// The prox targets of a bus's batteries at this item's hours, to their owners.
template <int kV>
__device__ __forceinline__ void push_targets(const Sm& m, int HS, int t, bool multi, int b0, int nb, const float* xbr,
                                             const float (&pb)[kV], const float (&uu)[kV]) {
    for (int b = 0; b < nb; ++b, xbr += HS) {
        const int2 bs = m.bslot[b0 + b];
        float xb[kV], v[kV];
        ldv<kV>(xbr, xb);
#pragma unroll
        for (int h = 0; h < kV; ++h) v[h] = xb[h] - pb[h] - uu[h];
        if (!multi) stv<kV>(m.vrow + bs.x + t, v);
        else if constexpr (kV == 4) st_async4((unsigned)bs.x + 4u * t, v[0], v[1], v[2], v[3], (unsigned)bs.y);
        else st_async1((unsigned)bs.x + 4u * t, v[0], (unsigned)bs.y);
    }
}

// One bus item: the devices' injections summed (generators, load, batteries, line ends: the bus
// kernels' order), then the consensus and the dual update.
template <int WANT, int kV>
__device__ __forceinline__ void res_bus(const Ctx& c, const Sm& m, float rho, int HS, int n, int hl, int t, bool multi,
                                        ResSums& acc) {
    const int i = n * HS + hl;
    const int4 br = m.busr[n];
    const float4 bf = m.busf[n];
    const int ng = br.w & 0xfff, ne = (br.w >> 12) & 0xfff, nb = (int)((unsigned)br.w >> 24);
    // The lists are walked in batches whose loads are all issued before the first sum, without
    // branches: an entry past a list's end reads the list's last one with factor 0 (an empty
    // list the next bus's first, or the zero entry past the last), so the lanes of a warp stay
    // together whatever their lengths.
    constexpr int kGB = kV == 4 ? 3 : 4, kEB = kV == 4 ? 2 : 4;
    const float* xg = m.xg + br.x + hl;
    const float* xbr = m.xb + br.z * HS + hl;
    const int4* endr = m.endr + br.y;
    const float* qr = m.q + br.y * HS + hl;
    float xl[kV], uu[kV], sum[kV], ths[kV], x[kGB][kV], d[kEB][kV], qv[kEB][kV], sb[kEB], w[kEB];
    auto gens = [&](int g) {
#pragma unroll
        for (int k = 0; k < kGB; ++k) {
            ldv<kV>(xg + max(min(g + k, ng - 1), 0) * HS, x[k]);
#pragma unroll
            for (int h = 0; h < kV; ++h) x[k][h] = g + k < ng ? x[k][h] : 0.f;
        }
    };
    auto add_gens = [&]() {
#pragma unroll
        for (int k = 0; k < kGB; ++k)
#pragma unroll
            for (int h = 0; h < kV; ++h) sum[h] += x[k][h];
    };
    auto ends = [&](int e) {
#pragma unroll
        for (int k = 0; k < kEB; ++k) {
            const int ek = max(min(e + k, ne - 1), 0);
            const int4 er = endr[ek];
            sb[k] = e + k < ne ? __int_as_float(er.y) : 0.f;
            w[k] = e + k < ne ? __int_as_float(er.z) : 0.f;
            ldv<kV>(m.dl + er.x + hl, d[k]);
            ldv<kV>(qr + ek * HS, qv[k]);
        }
    };
    float x2 = 0.f;
    auto add_ends = [&]() {
#pragma unroll
        for (int k = 0; k < kEB; ++k)
#pragma unroll
            for (int h = 0; h < kV; ++h) {
                const float p = __fmul_rn(sb[k], d[k][h]);
                sum[h] = __fadd_rn(sum[h], p);
                if (WANT) x2 += p * p;
                ths[h] = __fmaf_rn(w[k], qv[k][h], ths[h]);
            }
    };
    gens(0);
    ends(0);
    ldv<kV>(m.xl + i, xl);
    ldv<kV>(m.u + i, uu);
#pragma unroll
    for (int h = 0; h < kV; ++h) sum[h] = ths[h] = 0.f;
    add_gens();
    for (int g = kGB; g < ng; g += kGB) {
        gens(g);
        add_gens();
    }
#pragma unroll
    for (int h = 0; h < kV; ++h) sum[h] += xl[h];
    for (int b = 0; b < nb; ++b) {
        float xb[kV];
        ldv<kV>(xbr + b * HS, xb);
#pragma unroll
        for (int h = 0; h < kV; ++h) {
            sum[h] += xb[h];
            if (WANT) x2 += xb[h] * xb[h];
        }
    }
    add_ends();
    for (int e = kEB; e < ne; e += kEB) {
        ends(e);
        add_ends();
    }
    float pbn[kV], un[kV], thn[kV];
#pragma unroll
    for (int h = 0; h < kV; ++h) {
        pbn[h] = __fmul_rn(sum[h], bf.x);
        thn[h] = __fmul_rn(ths[h], bf.y);
        un[h] = __fadd_rn(uu[h], pbn[h]);
    }
    if (WANT) {
        const float cnt = 1.f / bf.x;
        float p2 = 0.f, dp2 = 0.f, dth2 = 0.f, u2 = 0.f;
        float pb[kV], th[kV];
        ldv<kV>(m.pbar + i, pb);
        ldv<kV>(m.thb + i, th);
#pragma unroll
        for (int h = 0; h < kV; ++h) {
            const float dpb = pbn[h] - pb[h];
            p2 += cnt * pbn[h] * pbn[h];
            dp2 += cnt * dpb * dpb;
            dth2 += (thn[h] - th[h]) * (thn[h] - th[h]) * bf.z;
            u2 += cnt * (rho * un[h]) * (rho * un[h]);
        }
        acc.n.add(p2);
        acc.dz.add(-dp2);
        acc.dth.add(dth2);
        acc.u.add(u2);
        acc.x += x2;
    }
    push_targets<kV>(m, HS, t, multi, br.z, nb, xbr, pbn, un);
    stv<kV>(m.pbar + i, pbn);
    stv<kV>(m.u + i, un);
    stv<kV>(m.thb + i, thn);
}

template <int ADJ, int kHpl, int kW, int kV, int kReg>
__global__ void __launch_bounds__(kCrsMaxThreads, 1)
    k_crs(const Ctx c, const CrsTables R, const int4* __restrict__ runs, int C, int bat_smem, double tol) {
    extern __shared__ __align__(16) unsigned char smem[];
    cg::cluster_group cl = cg::this_cluster();
    const int rank = (int)cl.block_rank();
    const int4 run = runs[blockIdx.x / C];
    const int s = run.x, it0 = run.y, it_end = run.z;  // iterations already run; pause once it_end have
    const ScenDev sd = c.scen[s];
    const int T = sd.T, N = sd.N, G = sd.G, L = sd.L, B = sd.B;
    const int HS = crs_hours(T, C, kV);
    const int h0 = rank * HS;
    const int nh = max(0, min(HS, T - h0));
    const int HQ = (nh + kV - 1) / kV;  // this rank's items per row
    const int HP = HQ * kV;             // hours carried, the padding of the last quad included
    const int TR = crs_row(T);          // prox-target row: hours rounded up to a quad
    const int nbo = (B + C - 1) / C;
    const int own = rank < B ? (B - rank + C - 1) / C : 0;  // batteries this rank owns
    const CrsOff o = crs_offsets(N, G, L, B, HS, C, T, sd.n_dd < nbo ? sd.n_dd : nbo, ADJ, bat_smem, blockDim.x, kV, kW);
    const Sm m = sm_at(smem, o);
    GState X;
    if (ADJ) X = GState{c.a_xg, c.a_xl, c.a_dl, c.a_sg, c.a_vf, c.a_vt, c.a_xb, c.a_zc, c.a_u, c.a_pbar, c.a_thb, c.a_zd - c.a_zc};
    else X = GState{c.xg, c.xl, c.dl, c.sg, c.vf, c.vt, c.xb, c.zc, c.u, c.pbar, c.thb, c.zd - c.zc};
    const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, warp = tid >> 5;
    const FastDiv dq(HQ > 0 ? HQ : 1);
    const bool multi = C > 1;
    const unsigned sbase = smem_addr(smem);

    BatConst K;
    K.rho = c.rho;
    K.ri = c.rho_in;
    K.iri = 1.f / c.rho_in;
    K.Ah = c.eps + c.rho_in + c.rho;
    K.idet = 1.f / fma_first(K.Ah, K.Ah, -c.rho, c.rho);

    // ---- static records
    if (tid == 0) {
        mbar_init(m.bar, 1);
        mbar_init(m.bar + 1, 1);
        mbar_fence_init();
        m.flag[0] = m.flag[1] = 0;
    }
    for (int n = tid; n < N; n += nt) {
        const int4 r = R.bus[sd.bus0 + n];  // generator, line-end, battery slots; original bus
        const int4 r1 = n + 1 < N ? R.bus[sd.bus0 + n + 1] : make_int4(G, 2 * L, B, 0);
        m.busr[n] = make_int4(r.x * HS, r.y, r.z, (r1.x - r.x) | ((r1.y - r.y) << 12) | (int)((unsigned)(r1.z - r.z) << 24));
        const int nb = sd.bus0 + r.w;
        m.busf[n] = make_float4(c.bus_inv_cnt[nb], c.bus_inv_wsum[nb], c.bus_dres_w[nb], 0.f);
        for (int g = r.x; g < r1.x; g += 4) {
            float cost[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) cost[k] = c.g_cost[sd.gen0 + R.gen[sd.gen0 + min(g + k, r1.x - 1)]];
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if (g + k < r1.x) m.genr[g + k] = make_int2(n * HS, __float_as_int(cost[k]));
        }
    }
    // the entry past the last list is zero, and so are the rows that it leads to
    if (tid == 0) m.endr[2 * L] = make_int4(0, 0, 0, 0);
    for (int h = tid; h < HS; h += nt) {
        m.q[2 * L * HS + h] = 0.f;
        if (L == 0) m.dl[h] = 0.f;
    }
    for (int e = tid; e < 2 * L; e += nt) {
        const int code = R.end[2 * sd.line0 + e], lg = sd.line0 + (code >> 1);
        const float beta = c.l_beta[lg];
        m.endr[e] = make_int4((code >> 1) * HS, __float_as_int((code & 1) ? beta : -beta), __float_as_int(c.l_w[lg]), 0);
    }
    for (int l = tid; l < L; l += nt) {
        const int lg = sd.line0 + l;
        const int4 r = R.line[lg];
        m.liner[l] = make_int4(r.x * HS, r.y * HS, r.z * HS, r.w * HS);
        const float beta = c.l_beta[lg], w = c.l_w[lg];
        const float rth = c.rth_c * w;
        const float den = __fmaf_rn(__fmul_rn(2.f * c.rho, beta), beta, 0.5f * rth) + (w == 0.f ? c.eps : 0.f);
        m.linef[l] = make_float4(beta, c.rho * beta, 0.5f * rth, den);
        m.linec[l] = make_float4(fminf(fmaxf(c.eta[sd.eta0 + G + l], 0.f) / beta, c.l_dth[lg]), w, 1.f / den, 0.f);
    }
    for (int b = tid; b < B; b += nt) {  // each injection slot's battery: its row at its owner
        const int row = (b / C) * TR;
        m.bslot[R.bat[sd.bat0 + b].y] =
            multi ? make_int2((int)(map_rank(sbase + (unsigned)o.vrow, b % C) + 4u * row),
                              (int)map_rank(smem_addr(m.bar + 1), b % C))
                  : make_int2(row, 0);
    }
    const bool dd_cls = sd.n_dd < nbo;  // one reciprocal-pivot row per efficiency class, else per owned battery
    for (int j = tid; j < own; j += nt) {
        const int b = rank + j * C, bg = sd.bat0 + b;
        const int2 r = R.bat[bg];  // bus position, injection slot
        const float P = fmaxf(c.eta[sd.eta0 + G + L + b], 0.f);
        const float a = c.b_effc[bg], k = 1.f / c.b_effd[bg];
        m.batr[2 * j] = make_int4(r.y * HS, 4 * r.y * HS, dd_cls ? R.bat_cls[bg] : j, b);
        m.batr[2 * j + 1] = make_int4(__float_as_int(P), __float_as_int(c.b_dur[bg] * P), __float_as_int(a), __float_as_int(k));
        m.batg[j] = make_float2(__fmul_rn(fma_first(K.Ah, a, -c.rho, k), K.idet), __fmul_rn(fma_first(c.rho, a, -K.Ah, k), K.idet));
    }
    const int rows = dd_cls ? sd.n_dd : nbo;
    batched<4, float>(
        rows * T, tid, nt,
        [&](int q) {
            const int j = q / T, t = q - j * T;
            const int b = dd_cls ? R.cls_rep[sd.bat0 + j] : rank + j * C;
            const float dd = c.bat_dd[sd.e_bat + (long long)min(b, B - 1) * sd.Tp + t];
            return b < B ? 1.f / dd : 0.f;
        },
        [&](int q, float v) { m.idd[q] = v; });

    // ---- state in
    const FastDiv dp(HP > 0 ? HP : 1);
    batched<2, BusIn>(
        N * HP, tid, nt,
        [&](int q) {
            const int n = dp.div(q), hl = q - n * HP;
            const bool in = hl < nh;
            const long long gi = sd.e_bus + (long long)R.bus[sd.bus0 + n].w * sd.Tp + h0 + (in ? hl : 0);
            BusIn v{X.pbar[gi], X.u[gi], X.thb[gi], X.xl[gi], ADJ ? c.al[gi] : c.load[gi]};
            // adjoint coefficient: NaN where the bound is active, so the hour stays 0
            if (!in) v = BusIn{0.f, 0.f, 0.f, 0.f, ADJ ? __int_as_float(0x7fc00000) : 0.f};
            return v;
        },
        [&](int q, const BusIn& v) {
            const int n = dp.div(q), li = n * HS + q - n * HP;
            m.pbar[li] = v.pbar; m.u[li] = v.u; m.thb[li] = v.thb; m.xl[li] = v.xl; m.ld[li] = v.ld;
        });
    batched<4, float2>(
        G * HP, tid, nt,
        [&](int q) {
            const int k = dp.div(q), hl = q - k * HP;
            const bool in = hl < nh;
            const int g = R.gen[sd.gen0 + k];
            const long long gi = sd.e_gen + (long long)g * sd.Tp + h0 + (in ? hl : 0);
            float2 v = make_float2(X.xg[gi], ADJ ? c.ag[gi] : c.cf[gi]);
            if (!ADJ) {
                const float etag = fmaxf(c.eta[sd.eta0 + g], 0.f);
                v.y = c.g_firm[sd.gen0 + g] ? etag : v.y * etag;
            }
            if (!in) v = make_float2(0.f, ADJ ? __int_as_float(0x7fc00000) : 0.f);
            return v;
        },
        [&](int q, const float2& v) {
            const int k = dp.div(q), li = k * HS + q - k * HP;
            m.xg[li] = v.x;
            m.cap[li] = v.y;
        });
    batched<4, LineIn>(
        L * HP, tid, nt,
        [&](int q) {
            const int l = dp.div(q), hl = q - l * HP;
            const bool in = hl < nh;
            const long long gi = sd.e_line + (long long)l * sd.Tp + h0 + (in ? hl : 0);
            const int4 r = R.line[sd.line0 + l];
            LineIn v{X.dl[gi], X.vf[gi], X.vt[gi], r.z, r.w};
            if (!in) v.dl = v.vf = v.vt = 0.f;
            return v;
        },
        [&](int q, const LineIn& v) {
            const int l = dp.div(q), hl = q - l * HP;
            m.dl[l * HS + hl] = v.dl;
            m.q[v.from * HS + hl] = v.vf;
            m.q[v.to * HS + hl] = v.vt;
        });
    if (ADJ)
        batched<4, unsigned>(
            L * HQ, tid, nt,
            [&](int q) {
                const int l = dq.div(q), hq = q - l * HQ;
                unsigned b = 0;
#pragma unroll
                for (int h = 0; h < kV; ++h) {
                    const int hl = hq * kV + h;
                    const unsigned on = c.m_line[sd.e_line + (long long)l * sd.Tp + h0 + min(hl, nh - 1)] ? 1u : 0u;
                    b |= (hl < nh ? on : 0u) << h;
                }
                return b;
            },
            [&](int q, unsigned b) {
                const int l = dq.div(q);
                m.lmask[l * (HS / kV) + q - l * HQ] = (uint8_t)b;
            });
    batched<4, BatIn>(
        B * HP, tid, nt,
        [&](int q) {
            const int b = dp.div(q), hl = q - b * HP;
            const bool in = hl < nh;
            BatIn v{X.xb[sd.e_bat + (long long)b * sd.Tp + h0 + (in ? hl : 0)], R.bat[sd.bat0 + b].y};
            if (!in) v.xb = 0.f;
            return v;
        },
        [&](int q, const BatIn& v) { m.xb[v.slot * HS + q - dp.div(q) * HP] = v.xb; });
    if (!kReg && bat_smem)
        for (int q = tid; q < own * T; q += nt) {
            const int j = q / T, t = q - j * T;
            const long long r = sd.e_bat + (long long)(rank + j * C) * sd.Tp + t;
            float z[6];
#pragma unroll
            for (int k = 0; k < 6; ++k) z[k] = X.zc[k * X.zstride + r];
#pragma unroll
            for (int k = 0; k < 6; ++k) m.bst[(j * 6 + k) * T + t] = z[k];
        }
    __syncthreads();
    constexpr int NL = 32 * kW;
    const int groups = nt / NL, group = tid / NL;
    const int Lx = tid & (NL - 1);
    for (int j = group; j < rows; j += groups) res_scan_table<kHpl, kW>(m.idd + j * T, m.scan + j * 12 * NL, T);
    // where the lane's new injections go: the owner of its hours (kV = 1) or of its quad
    constexpr int NQ = kV == 4 ? 1 : kHpl;
    unsigned qa[NQ], qb[NQ];
#pragma unroll
    for (int j = 0; j < NQ; ++j) {
        const int t = min(kV == 4 ? 4 * Lx : Lx * kHpl + j, T - 1), rk = t / HS;
        qa[j] = map_rank(sbase + (unsigned)o.xb, rk) + 4u * (unsigned)(t - rk * HS);
        qb[j] = map_rank(smem_addr(m.bar), rk);
    }
    // a battery's state in its lanes' registers, one battery per group
    float s6[6][kHpl];
#pragma unroll
    for (int r = 0; r < 6; ++r)
#pragma unroll
        for (int j = 0; j < kHpl; ++j) {
            const int t = Lx * kHpl + j;
            s6[r][j] = kReg && group < own && t < T
                           ? X.zc[r * X.zstride + sd.e_bat + (long long)(rank + group * C) * sd.Tp + t] : 0.f;
        }
    cl.sync();
    const bool wait_x = multi && B > 0, wait_v = multi && own > 0;
    const unsigned bytes_x = 4u * (unsigned)(B * HP), bytes_v = 4u * (unsigned)(own * (kV == 4 ? TR : T));
    if (tid == 0 && wait_v) mbar_expect_tx(m.bar + 1, bytes_v);
    for (int q = tid; q < N * HQ; q += nt) {  // the first prox targets
        const int n = dq.div(q), hl = (q - n * HQ) * kV;
        const int4 br = m.busr[n];
        float pb[kV], uu[kV];
        ldv<kV>(m.pbar + n * HS + hl, pb);
        ldv<kV>(m.u + n * HS + hl, uu);
        push_targets<kV>(m, HS, h0 + hl, multi, br.z, (int)((unsigned)br.w >> 24), m.xb + br.z * HS + hl, pb, uu);
    }
    __syncthreads();

    // ---- iterations
    const int max_it = c.max_it, every = c.check_every;
    const int cl_n = (L * HQ + 31) >> 5, cg_n = (G * HQ + 31) >> 5, cb_n = (N * HQ + 31) >> 5;
    const float inv_re = 1.f / (c.rho + c.eps);
    // The warp's chunks [k0, k1): the chunk list (lines, generators, loads) is cut so that every
    // warp's estimated time, its batteries' included, is the same; warps whose batteries alone take
    // longer get none.  (A shared counter instead cost 0.3 to 0.8 us per iteration in atomics.)
    int k0, k1;
    {
        // cycles of a chunk and of a battery prox with the SM busy (halving or doubling the
        // latter changes an iteration by at most 3 %)
        const float wl = kV == 4 ? 900.f : 350.f, wg = kV == 4 ? 330.f : 200.f;
        const float wb = 600.f + (float)c.inner_iters * (350.f + 120.f * kHpl + (kW == 2 ? 150.f : 0.f));
        const int W = nt / 32, per = own / groups, more = own - per * groups;  // groups < more have one battery more
        const float hi = wb * (float)(per + 1), lo = wb * (float)per, total = wl * (float)cl_n + wg * (float)(cg_n + cb_n);
        const int n_hi = more * kW, n_lo = W - n_hi;
        float level = (total + hi * (float)n_hi + lo * (float)n_lo) / (float)W;
        if (n_hi > 0 && level < hi) level = n_lo > 0 ? (total + lo * (float)n_lo) / (float)n_lo : level;
        const float cap_hi = fmaxf(level - hi, 0.f), cap_lo = fmaxf(level - lo, 0.f);
        auto first = [&](int w) {  // first chunk of warp w
            if (w >= W) return cl_n + cg_n + cb_n;
            const float s0 = w < n_hi ? cap_hi * (float)w : cap_hi * (float)n_hi + cap_lo * (float)(w - n_hi);
            const float lines = wl * (float)cl_n;
            const int k = s0 <= lines ? (int)ceilf(s0 / wl - 1e-3f) : cl_n + (int)ceilf((s0 - lines) / wg - 1e-3f);
            return min(k, cl_n + cg_n + cb_n);
        };
        k0 = first(warp);
        k1 = first(warp + 1);
    }
    int it = it0, slot = 0;
    unsigned ph = 0;  // iterations of this launch: the barriers' phases
    double best = it0 > 0 ? c.rbest[s] : 0.0;
    auto iterate = [&](auto want_c, int store_sg, ResSums& acc) {
        constexpr int W = decltype(want_c)::value;
        if (tid == 0 && wait_x) mbar_expect_tx(m.bar, bytes_x);
        // A: batteries first (the longest chain), then chunks of the other devices
        if (group < own) {
            if (wait_v) res_wait(c, m, 1, ph & 1);
            if (tid == 0 && wait_v) mbar_expect_tx(m.bar + 1, bytes_v);
            for (int j = group; j < own; j += groups) {
                const long long row0 = sd.e_bat + (long long)(rank + j * C) * sd.Tp;
                float* st = bat_smem ? m.bst + (size_t)j * 6 * T : X.zc + row0;
                res_battery<W, ADJ, kHpl, kW, kV, kReg>(c, m, K, T, TR, HS, multi, qa, qb, j, group, s6, st,
                                                        bat_smem ? T : X.zstride, row0, acc);
            }
        }
        for (int k = k0; k < k1; ++k) {
            if (k < cl_n) {
                const int q = k * 32 + lane;
                if (q < L * HQ) {
                    const int l = dq.div(q), hq = q - l * HQ;
                    res_line<W, ADJ, kV>(c, m, X.sg, sd.e_line + (long long)l * sd.Tp + h0, HS, l, hq, store_sg, acc);
                }
            } else if (k < cl_n + cg_n) {
                const int q = (k - cl_n) * 32 + lane;
                if (q < G * HQ) {
                    const int g = dq.div(q);
                    res_gen<W, ADJ, kV>(m, c.rho, inv_re, HS, g, (q - g * HQ) * kV, acc);
                }
            } else {
                const int q = (k - cl_n - cg_n) * 32 + lane;
                if (q < N * HQ) {
                    const int n = dq.div(q);
                    res_load<W, ADJ, kV>(m, c.rho, inv_re, c.voll, n * HS + (q - n * HQ) * kV, acc);
                }
            }
        }
        __syncthreads();
        if (wait_x) res_wait(c, m, 0, ph & 1);
        for (int q = tid; q < N * HQ; q += nt) {
            const int n = dq.div(q), hl = (q - n * HQ) * kV;
            res_bus<W, kV>(c, m, c.rho, HS, n, hl, h0 + hl, multi, acc);
        }
        __syncthreads();
        ++ph;
    };
    for (;;) {
        const int chunk = min(every, max_it - it);
        ResSums acc;  // (the residual iteration's alone)
        for (int jt = 0; jt < chunk - 1; ++jt) iterate(std::integral_constant<int, 0>{}, jt == chunk - 2, acc);
        acc = ResSums{};
        iterate(std::integral_constant<int, 1>{}, 1, acc);
        const Sum2 w = warp_sums(acc, lane);
        if (lane < 4 * (kCrsRed - 1) && (lane & 3) == 0) m.wred[warp * (kCrsRed - 1) + (lane >> 2)] = w;
        if (tid == 0) m.flag[2] = m.flag[1] ? 1 : 0;  // (one reading for all ranks)
        __syncthreads();
        // this rank's sums, a warp each, into every rank's reduction slots; the last slot carries its
        // failure flag
        for (int q = warp; q < kCrsRed; q += nt / 32) {
            Sum2 t = lane < nt / 32 && q < kCrsRed - 1 ? m.wred[lane * (kCrsRed - 1) + q] : Sum2{0.f, 0.f};
#pragma unroll
            for (int bit = 16; bit >= 1; bit >>= 1)
                t.add(__shfl_xor_sync(0xffffffffu, t.hi, bit), __shfl_xor_sync(0xffffffffu, t.lo, bit));
            const double tot = q < kCrsRed - 1 ? (double)t.hi + (double)t.lo : (double)m.flag[2];
            if (lane < C) cl.map_shared_rank(m.red, lane)[(slot * C + rank) * kCrsRed + q] = tot;
        }
        cl.sync();
        it += chunk;
        if (warp == 0) {
            // the convergence test of the streaming reduction kernel, on the cluster's sums: lane q
            // adds up sum q, then the square roots and the divisions run lane by lane.  Every rank
            // takes the decision from the same numbers in the same order.
            double a = 0.0;
            if (lane < kCrsRed)
                for (int r = 0; r < C; ++r) a += m.red[(slot * C + r) * kCrsRed + lane];
            // NaN / inf test on the raw sums, before the clamps (fmax would turn a NaN into 0)
            const bool finite = __all_sync(0xffffffffu, isfinite(a));
            auto sum = [&](int q) { return __shfl_sync(0xffffffffu, a, q); };
            const double s0 = sum(0), s1 = sum(1), dz2 = fmax(sum(2), 0.0), s3 = sum(3), s4 = sum(4);
            const double marks = sum(kCrsRed - 1);
            const bool pause = it >= it_end, bad = marks != 0.0;
            const double rhod = c.rho, rth = c.rth_c;
            const double arg = lane == 0 ? fmax(s0, 0.0) : lane == 1 ? s1 : lane == 2 ? rhod * rhod * dz2 + rth * rth * s3 : s4;
            const double root = sqrt(arg);
            const double r0 = __shfl_sync(0xffffffffu, root, 0), r1 = __shfl_sync(0xffffffffu, root, 1),
                         r2 = __shfl_sync(0xffffffffu, root, 2), r3 = __shfl_sync(0xffffffffu, root, 3);
            const double quo = lane == 0 ? r0 / (ADJ ? fmax(r1, 1e-30) : sd.load_norm) : r2 / fmax(r3, 1e-30);
            const double rp = __shfl_sync(0xffffffffu, quo, 0), rd = __shfl_sync(0xffffffffu, quo, 1);
            const double r = fmax(rp, rd);
            if (it <= every || !(r >= best)) best = r;
            int stop = 1, status = GX_OK;
            if (bad) status = GX_ERR_TIMEOUT;
            else if (!finite || !isfinite(rp) || !isfinite(rd) || r > 1e6 * best) status = GX_ERR_NONFINITE;
            else if (rp <= tol && rd <= tol) status = GX_OK;
            else if (it >= max_it) status = GX_NOT_CONVERGED;
            else stop = 0;
            if (lane == 0) {
                if (stop && rank == 0) {
                    c.resid[2 * s + 0] = rp;
                    c.resid[2 * s + 1] = rd;
                    c.status[s] = status;
                    c.done[s] = 1;
                    (ADJ ? c.adj_iters : c.iters)[s] = it;
                    c.rbest[s] = best;
                }
                if (rank == 0 && !stop && pause) c.rbest[s] = best;
                m.flag[0] = stop || pause;
            }
        }
        __syncthreads();
        if (m.flag[0]) break;
        slot ^= 1;  // the next chunk's partials: a rank may still be reading these
    }
    // the last prox targets are in flight: they have landed before the CTA may leave
    if (wait_v) res_wait(c, m, 1, ph & 1);

    // ---- state out
    const FastDiv dn(nh > 0 ? nh : 1);
    batched<4, int>(
        N * nh, tid, nt, [&](int q) { return R.bus[sd.bus0 + dn.div(q)].w; },
        [&](int q, int bus) {
            const int n = dn.div(q), hl = q - n * nh, li = n * HS + hl;
            const long long gi = sd.e_bus + (long long)bus * sd.Tp + h0 + hl;
            X.pbar[gi] = m.pbar[li]; X.u[gi] = m.u[li]; X.thb[gi] = m.thb[li]; X.xl[gi] = m.xl[li];
        });
    batched<8, int>(
        G * nh, tid, nt, [&](int q) { return R.gen[sd.gen0 + dn.div(q)]; },
        [&](int q, int g) {
            const int k = dn.div(q), hl = q - k * nh;
            X.xg[sd.e_gen + (long long)g * sd.Tp + h0 + hl] = m.xg[k * HS + hl];
        });
    batched<4, int2>(
        L * nh, tid, nt,
        [&](int q) {
            const int4 r = R.line[sd.line0 + dn.div(q)];
            return make_int2(r.z, r.w);
        },
        [&](int q, const int2& r) {
            const int l = dn.div(q), hl = q - l * nh;
            const long long gi = sd.e_line + (long long)l * sd.Tp + h0 + hl;
            X.dl[gi] = m.dl[l * HS + hl]; X.vf[gi] = m.q[r.x * HS + hl]; X.vt[gi] = m.q[r.y * HS + hl];
        });
    batched<4, int>(
        B * nh, tid, nt, [&](int q) { return R.bat[sd.bat0 + dn.div(q)].y; },
        [&](int q, int slot) {
            const int b = dn.div(q), hl = q - b * nh;
            X.xb[sd.e_bat + (long long)b * sd.Tp + h0 + hl] = m.xb[slot * HS + hl];
        });
    if (kReg) {
#pragma unroll
        for (int r = 0; r < 6; ++r)
#pragma unroll
            for (int j = 0; j < kHpl; ++j) {
                const int t = Lx * kHpl + j;
                if (group < own && t < T) X.zc[r * X.zstride + sd.e_bat + (long long)(rank + group * C) * sd.Tp + t] = s6[r][j];
            }
    } else if (bat_smem) {
        for (int q = tid; q < own * T; q += nt) {
            const int j = q / T, t = q - j * T;
            const long long r = sd.e_bat + (long long)(rank + j * C) * sd.Tp + t;
#pragma unroll
            for (int k = 0; k < 6; ++k) X.zc[k * X.zstride + r] = m.bst[(j * 6 + k) * T + t];
        }
    }
    // no rank leaves while another may still read or write its shared memory
    cl.sync();
}

// The instances of one direction and item width.
template <int ADJ, int kV>
CrsFn crs_pick_impl(int kw, int hpl, int reg) {
    if (kw == 1) {
        if (hpl <= 1) return k_crs<ADJ, 1, 1, kV, 0>;
        if (hpl <= 2) return k_crs<ADJ, 2, 1, kV, 0>;
        return k_crs<ADJ, 3, 1, kV, 0>;
    }
    if (hpl <= 1) return reg ? k_crs<ADJ, 1, 2, kV, 1> : k_crs<ADJ, 1, 2, kV, 0>;
    if (hpl <= 2) return reg ? k_crs<ADJ, 2, 2, kV, 1> : k_crs<ADJ, 2, 2, kV, 0>;
    if (hpl <= 3) return reg ? k_crs<ADJ, 3, 2, kV, 1> : k_crs<ADJ, 3, 2, kV, 0>;
    return k_crs<ADJ, 4, 2, kV, 0>;  // over 192 hours, on request only
}

}  // namespace
}  // namespace gx
