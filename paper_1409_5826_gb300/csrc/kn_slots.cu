// kn_slots.cu -- the mixed-form integrator with several zones per thread group.
//
// What bounds a step: a chain of phases (gather, update, decision beside the flux
// pass) whose latency the longest zone of a batch pays hundreds of thousands of
// times, and, with many zones on an SM, instruction issue and shared-memory
// wavefronts, most of them for what is the same in every step and zone: table
// words, addresses, loop counters, one lane's scalar decision.  (A branch costs a
// warp about 20 cycles, a shared load 23, an FP64 operation 64.)  So here:
//   * a group of T threads integrates NZ zones ("slots") side by side.  Its arrays
//     interleave them in blocks of 32 words (word v of zone z at word
//     (v / 32) 32 NZ + 32 z + v % 32): one offset serves all zones, whose values
//     lie 128 bytes apart in the same bank;
//   * FP32 arithmetic on two zones is packed (add/mul/fma.rn.f32x2: the same
//     roundings, one instruction for both);
//   * a worker thread keeps its reactions' and gather terms' offsets and its
//     reactions' cached rates in registers for the launch: no table word is loaded
//     and no loop counted in a step.  128 registers and 512 threads an SM: with 80
//     and 768 and tables in shared memory the 4096-zone batch took 14 % longer;
//   * the zones' scalar state lives in registers of a warp of its own, 32 / NZ
//     lanes a zone: one pass of the decision's instructions serves all zones, and
//     its FP64 work runs beside the update; the species' float-float state and
//     candidate live in registers of the species' thread;
//   * zones are independent: each accepts, rejects, ends and is replaced from the
//     queue by itself.  A rejected zone keeps its (F+, k) because the gather's
//     stores are masked by the accepted zones.
// Every sum keeps the order that the group kernel's tables give it (the pieces,
// the terms of a piece, the segmented reduction, the butterflies, the warps), so
// the results are the group kernel's bit for bit, whatever T and NZ.
//
// Measured against the group kernel: 4096 zones of 150/1604 to 1e-9 s 814 -> 627 ms, 100
// zones of it (one an SM) 7.2 -> 3.5 ms, 8001 zones of the 16/48 chain to 1e-3 s 32.6 ->
// 20.5 ms, 1000 of 365/4400 to 1e-10 s 52 -> 41 ms, 4096 QSS chains to 1e-2 s 56.9 -> 38
// ms.  Where it is not faster plan_slots (kn_api.cu) leaves the call to that kernel, except
// that it cannot see this: with 4 to 5 zones an SM and four slots the fifth zone follows
// alone, in a pair's step.  Zones of a spread fill that time (684 of 150/1604 1.5 times the
// group kernel's rate); zones that all take the same number of steps do not (0.8).
#include <cstddef>
#include <cstdint>

#include "kn_device.cuh"

namespace kn {
namespace {

// ---------------------------------------------------------------------------
// packs: the zones of a group, two to a register pair
// ---------------------------------------------------------------------------
template <int NZ> struct Pack {
    using T = float2;
    static constexpr int n = NZ / 2;
};
template <> struct Pack<1> {
    using T = float;
    static constexpr int n = 1;
};

__device__ __forceinline__ float padd(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float psub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float pmul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float pfma(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ float pneg(float a) { return -a; }
__device__ __forceinline__ float2 padd(float2 a, float2 b) {
    float2 r;
    asm("{\n\t.reg .b64 x, y, z;\n\tmov.b64 x, {%2, %3};\n\tmov.b64 y, {%4, %5};\n\tadd.rn.f32x2 z, x, y;\n\t"
        "mov.b64 {%0, %1}, z;\n\t}"
        : "=f"(r.x), "=f"(r.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return r;
}
__device__ __forceinline__ float2 pmul(float2 a, float2 b) {
    float2 r;
    asm("{\n\t.reg .b64 x, y, z;\n\tmov.b64 x, {%2, %3};\n\tmov.b64 y, {%4, %5};\n\tmul.rn.f32x2 z, x, y;\n\t"
        "mov.b64 {%0, %1}, z;\n\t}"
        : "=f"(r.x), "=f"(r.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return r;
}
__device__ __forceinline__ float2 pfma(float2 a, float2 b, float2 c) {
    float2 r;
    asm("{\n\t.reg .b64 x, y, z, w;\n\tmov.b64 x, {%2, %3};\n\tmov.b64 y, {%4, %5};\n\tmov.b64 w, {%6, %7};\n\t"
        "fma.rn.f32x2 z, x, y, w;\n\tmov.b64 {%0, %1}, z;\n\t}"
        : "=f"(r.x), "=f"(r.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
    return r;
}
// a - b is the single rounding of a + (-1) b
__device__ __forceinline__ float2 psub(float2 a, float2 b) { return pfma(b, make_float2(-1.f, -1.f), a); }
__device__ __forceinline__ float2 pneg(float2 a) { return make_float2(-a.x, -a.y); }

__device__ __forceinline__ void pset(float& p, int, float v) { p = v; }
__device__ __forceinline__ void pset(float2& p, int c, float v) { (c ? p.y : p.x) = v; }
__device__ __forceinline__ float pget(float p, int) { return p; }
__device__ __forceinline__ float pget(float2 p, int c) { return c ? p.y : p.x; }
__device__ __forceinline__ void pall(float& p, float v) { p = v; }
__device__ __forceinline__ void pall(float2& p, float v) { p = make_float2(v, v); }

template <class P>
__device__ __forceinline__ void ptwo_sum(P a, P b, P& s, P& e) {
    s = padd(a, b);
    const P bv = psub(s, a);
    const P av = psub(s, bv);
    e = padd(psub(a, av), psub(b, bv));
}

// zone z's component of a group's packs (z known at compile time)
template <int NZ> __device__ __forceinline__ float zget(const typename Pack<NZ>::T (&p)[Pack<NZ>::n], int z) {
    return NZ == 1 ? pget(p[0], 0) : pget(p[z >> 1], z & 1);
}
template <int NZ> __device__ __forceinline__ void zset(typename Pack<NZ>::T (&p)[Pack<NZ>::n], int z, float v) {
    if (NZ == 1) pset(p[0], 0, v);
    else pset(p[z >> 1], z & 1, v);
}

// ---------------------------------------------------------------------------
// shared memory by 32-bit address: the arrays of a group are its base plus a plan
// constant, so an address costs one addition and no register of its own
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint32_t saddr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
template <int OFF = 0> __device__ __forceinline__ float lds(uint32_t a) {
    float v;
    asm volatile("ld.shared.f32 %0, [%1+%2];" : "=f"(v) : "r"(a), "n"(OFF));
    return v;
}
template <int OFF = 0> __device__ __forceinline__ uint32_t ldu(uint32_t a) {
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1+%2];" : "=r"(v) : "r"(a), "n"(OFF));
    return v;
}
__device__ __forceinline__ uint2 ldu2(uint32_t a) {
    uint2 v;
    asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(a));
    return v;
}
__device__ __forceinline__ void ldp(uint32_t a, float& v) { v = lds(a); }
__device__ __forceinline__ void ldp(uint32_t a, float2& v) {
    asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(a));
}
__device__ __forceinline__ float4 ldf4(uint32_t a) {
    float4 v;
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(a));
    return v;
}
template <int OFF = 0> __device__ __forceinline__ void sts(uint32_t a, float v) {
    asm volatile("st.shared.f32 [%0+%1], %2;" ::"r"(a), "n"(OFF), "f"(v) : "memory");
}
__device__ __forceinline__ void stp(uint32_t a, float v) { sts(a, v); }
__device__ __forceinline__ void stp(uint32_t a, float2 v) {
    asm volatile("st.shared.v2.f32 [%0], {%1, %2};" ::"r"(a), "f"(v.x), "f"(v.y) : "memory");
}
// base + M times the low / high half of w: one dot product of the halves with (M, 0) / (0, M)
template <int M> __device__ __forceinline__ uint32_t lo16(uint32_t w, uint32_t base) { return __dp2a_lo(w, (uint32_t)M, base); }
template <int M> __device__ __forceinline__ uint32_t hi16(uint32_t w, uint32_t base) { return __dp2a_lo(w, (uint32_t)M << 8, base); }
// a word's value in every zone of the group
template <int NZ> __device__ __forceinline__ void ld_zones(uint32_t a, typename Pack<NZ>::T (&v)[Pack<NZ>::n]) {
    zset<NZ>(v, 0, lds<0>(a));
    if constexpr (NZ > 1) zset<NZ>(v, 1, lds<128>(a));
}
template <int NZ> __device__ __forceinline__ void st_zones(uint32_t a, const typename Pack<NZ>::T (&v)[Pack<NZ>::n]) {
    sts<0>(a, zget<NZ>(v, 0));
    if constexpr (NZ > 1) sts<128>(a, zget<NZ>(v, 1));
}
// byte address of word v (zone 0) of an interleaved array, from its base
template <int NZ> __device__ __forceinline__ int at(int v) { return (v >> 5) * (128 * NZ) + (v & 31) * 4; }

// ---------------------------------------------------------------------------
// a zone's scalars: one copy per zone in shared memory, read and written by the
// control warp (a single-warp group keeps them in registers)
// ---------------------------------------------------------------------------
struct Scal {
    double t, te, ts, ta;    // time, end, t + h, the time an accept reaches
    double rem_d;            // te - ta
    long long steps, rejects;
    float h, dt;             // the attempt's step, the controller's next one
    float rem, rem_acc;      // te - t, te - ta
    float us, ur, u;         // 1 / (tau ln 2); u of the cached rates; u of the candidate
    float tf;                // t + h, in FP32
    int nrej, status;
    bool clip, cst, last, live, refresh;
};

struct SlotCtl {
    float h[kMaxSlots];      // the attempt's step
    uint32_t acc, done;      // zones whose attempt was accepted / that ended
    uint32_t rmask;          // zones whose cached rates the flux pass recomputes
    uint32_t live;           // zones in work
    float u[kMaxSlots];      // (t + h) / (tau ln 2) of the candidate state
    int zone[kMaxSlots];     // -1: the slot is empty, -2: it has had none yet
    int valid, end;          // a zone being loaded: its inputs are valid / it ends at once
    uint32_t fresh;          // zones just loaded
    int status;
    long long fetch_ns[kMaxSlots];
    double lnT0, lnR0;
};
static_assert(sizeof(SlotCtl) <= kSlotCtlBytes, "SlotCtl");
static_assert(offsetof(SlotCtl, h) == 0 && offsetof(SlotCtl, acc) % 8 == 0 &&
                  offsetof(SlotCtl, done) == offsetof(SlotCtl, acc) + 4,
              "h is loaded as a pack, acc and done as a pair");

template <bool WARP> struct SlotSync {
    int id, n;
    __device__ __forceinline__ void sync() const {
        if (WARP) {
            asm volatile("" ::: "memory");
            __syncwarp();
            asm volatile("" ::: "memory");
        } else asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory");
    }
};

// shared addresses: the tables' base and the group's base
struct SlotBase {
    uint32_t tb, gb;
};

// ---------------------------------------------------------------------------
// What a worker thread keeps in registers for the whole launch: its reactions'
// and its gather terms' 16-bit word offsets, two to a word, and the cached rates
// of its reactions.  Capacities: reactions of F1 1-body, F2 2-body and FA blocks
// of any sort, and two gather slices of up to 2 GA and 2 GB terms.
// ---------------------------------------------------------------------------
template <int NZ, class CAP> struct Resident {
    static constexpr int F1 = CAP::F1, F2 = CAP::F2, FA = CAP::FA, GA = CAP::GA, GB = CAP::GB;
    using PK = typename Pack<NZ>::T;
    static constexpr int n = Pack<NZ>::n;
    uint32_t f1[F1 ? F1 : 1];     // a | V << 16
    uint32_t f2[F2 ? F2 : 1][3];  // a | b << 16, V | P0 << 16, P1
    uint32_t fa[FA][4];           // a | b << 16, c | V << 16, P0 | P1 << 16, P2 | reactants << 16
    PK k1[F1 ? F1 : 1][n], k2[F2 ? F2 : 1][n], ka[FA][n];
    uint32_t ga[GA], gb[GB];
    uint32_t sa, sb;              // destination from Fk | stores << 16 | (bit 17 + r: round r adds the lane 2^r up)
    uint32_t cnt;                 // blocks n1 | n2 << 4 | na << 8, words of ga / gb << 12 / 18, rounds << 24 / 28

    __device__ __forceinline__ void load(const PlanDev& P, int wt, int Tw) {
        const uint32_t* t = (const uint32_t*)(P.slot_blob + P.st.off_words) + wt;
#pragma unroll
        for (int i = 0; i < F1; ++i, t += Tw) f1[i] = *t;
#pragma unroll
        for (int i = 0; i < F2; ++i)
#pragma unroll
            for (int q = 0; q < 3; ++q, t += Tw) f2[i][q] = *t;
#pragma unroll
        for (int i = 0; i < FA; ++i)
#pragma unroll
            for (int q = 0; q < 4; ++q, t += Tw) fa[i][q] = *t;
#pragma unroll
        for (int i = 0; i < GA; ++i, t += Tw) ga[i] = *t;
#pragma unroll
        for (int i = 0; i < GB; ++i, t += Tw) gb[i] = *t;
        sa = *t;
        t += Tw;
        sb = *t;
        t += Tw;
        cnt = *t;
#pragma unroll
        for (int q = 0; q < n; ++q) {
#pragma unroll
            for (int i = 0; i < (F1 ? F1 : 1); ++i) pall(k1[i][q], 0.f);
#pragma unroll
            for (int i = 0; i < (F2 ? F2 : 1); ++i) pall(k2[i][q], 0.f);
#pragma unroll
            for (int i = 0; i < FA; ++i) pall(ka[i][q], 0.f);
        }
    }
};

// shared addresses of the group's V, Y and scalars
struct WorkAddr {
    uint32_t V, Y, ctl;
};
__device__ __forceinline__ WorkAddr work_addr(const PlanDev& P, const SlotBase& g) {
    return WorkAddr{g.gb + P.sl.off_V, g.gb + P.sl.off_Y, g.gb + P.sl.off_ctl};
}

// The cached rates K 2^(-c u) of the zones of `mask`, at the u set for them.  A
// 1-body reaction's partial is its rate, so it is stored here and nowhere else.
// wt: the worker thread, Tw of them.
template <int NZ, class CAP>
__device__ __forceinline__ void refresh_rates(const PlanDev& P, const SlotBase& g, int wt, int Tw, Resident<NZ, CAP>& r,
                                              const WorkAddr& f, uint32_t mask) {
    using PK = typename Pack<NZ>::T;
    constexpr int n = Pack<NZ>::n;
    // opaque: the blocks' addresses are formed here, not kept through the step loop
    asm volatile("" : "+r"(wt), "+r"(Tw));
    uint32_t c = g.tb + 4 * wt, K = g.gb + P.sl.off_K + 4 * NZ * wt, p0 = g.tb + P.st.off_p0 + 4 * wt;
    const int n1 = r.cnt & 15, n2 = r.cnt >> 4 & 15, na = r.cnt >> 8 & 15, cs = 4 * Tw, Ks = 4 * NZ * Tw;
    float u[NZ];
#pragma unroll
    for (int z = 0; z < NZ; ++z) u[z] = lds(f.ctl + (int)offsetof(SlotCtl, u) + 4 * z);
    auto rates = [&](PK (&k)[n]) {
        const float cj = lds(c);
        PK k0[n];
#pragma unroll
        for (int q = 0; q < n; ++q) ldp(K + (int)sizeof(PK) * q, k0[q]);
#pragma unroll
        for (int z = 0; z < NZ; ++z)
            if (mask >> z & 1) zset<NZ>(k, z, __fmul_rn(zget<NZ>(k0, z), ex2_approx(-__fmul_rn(cj, u[z]))));
    };
#pragma unroll
    for (int i = 0; i < CAP::F1; ++i, c += cs, K += Ks, p0 += cs)
        if (i < n1) {
            rates(r.k1[i]);
            st_zones<NZ>(f.V + 4 * ldu(p0), r.k1[i]);
        }
#pragma unroll
    for (int i = 0; i < CAP::F2; ++i, c += cs, K += Ks)
        if (i < n2) rates(r.k2[i]);
#pragma unroll
    for (int i = 0; i < CAP::FA; ++i, c += cs, K += Ks)
        if (i < na) rates(r.ka[i]);
}

// (a) rates, fluxes and reactant-slot partials (Eq. 1) of the states at Y
template <int NZ, class CAP>
__device__ __forceinline__ void flux_pass(const Resident<NZ, CAP>& r, const WorkAddr& f) {
    using PK = typename Pack<NZ>::T;
    constexpr int n = Pack<NZ>::n;
    const int n1 = r.cnt & 15, n2 = r.cnt >> 4 & 15, na = r.cnt >> 8 & 15;
#pragma unroll
    for (int i = 0; i < CAP::F1; ++i)
        if (i < n1) {
            PK y[n], fl[n];
            ld_zones<NZ>(lo16<4>(r.f1[i], f.Y), y);
#pragma unroll
            for (int q = 0; q < n; ++q) fl[q] = pmul(r.k1[i][q], y[q]);
            st_zones<NZ>(hi16<4>(r.f1[i], f.V), fl);
        }
#pragma unroll
    for (int i = 0; i < CAP::F2; ++i)
        if (i < n2) {
            PK ya[n], yb[n], fl[n], a0[n], a1[n];
            ld_zones<NZ>(lo16<4>(r.f2[i][0], f.Y), ya);
            ld_zones<NZ>(hi16<4>(r.f2[i][0], f.Y), yb);
#pragma unroll
            for (int q = 0; q < n; ++q) {
                a1[q] = pmul(r.k2[i][q], ya[q]);
                fl[q] = pmul(a1[q], yb[q]);
                a0[q] = pmul(r.k2[i][q], yb[q]);
            }
            st_zones<NZ>(lo16<4>(r.f2[i][1], f.V), fl);
            st_zones<NZ>(hi16<4>(r.f2[i][1], f.V), a0);
            st_zones<NZ>(f.V + 4 * r.f2[i][2], a1);
        }
    // blocks of 3-body reactions or of several classes: the 3-body products with
    // the constant 1 in an absent reactant's place (multiplying by it is exact)
#pragma unroll
    for (int i = 0; i < CAP::FA; ++i)
        if (i < na) {
            const uint32_t nr = r.fa[i][3] >> 16;
            PK ya[n], yb[n], yc[n], fl[n], a0[n], a1[n], a2[n];
            ld_zones<NZ>(lo16<4>(r.fa[i][0], f.Y), ya);
            ld_zones<NZ>(hi16<4>(r.fa[i][0], f.Y), yb);
            ld_zones<NZ>(lo16<4>(r.fa[i][1], f.Y), yc);
#pragma unroll
            for (int q = 0; q < n; ++q) {
                const PK k = r.ka[i][q], x = pmul(k, ya[q]);
                fl[q] = pmul(pmul(x, yb[q]), yc[q]);
                a0[q] = pmul(pmul(k, yb[q]), yc[q]);
                a1[q] = pmul(x, yc[q]);
                a2[q] = pmul(x, yb[q]);
            }
            if (nr > 0) {
                st_zones<NZ>(hi16<4>(r.fa[i][1], f.V), fl);
                st_zones<NZ>(lo16<4>(r.fa[i][2], f.V), a0);
            }
            if (nr > 1) st_zones<NZ>(hi16<4>(r.fa[i][2], f.V), a1);
            if (nr > 2) st_zones<NZ>(lo16<4>(r.fa[i][3], f.V), a2);
        }
}

// ---------------------------------------------------------------------------
// (b) sliced gathers of the zones of `need` into the (F+, k) rows at Fk
// ---------------------------------------------------------------------------
template <int NZ, int NW>
__device__ __forceinline__ void gather_slice(const uint32_t (&wd)[NW], int words, int rounds, uint32_t sd, uint32_t V,
                                             uint32_t Fk, uint32_t need) {
    using PK = typename Pack<NZ>::T;
    constexpr int n = Pack<NZ>::n;
    PK acc[n];
#pragma unroll
    for (int q = 0; q < n; ++q) pall(acc[q], 0.f);
#pragma unroll
    for (int i = 0; i < NW; i += 2)
        if (i < words) {
            PK v[4][n];
            ld_zones<NZ>(lo16<4>(wd[i], V), v[0]);
            ld_zones<NZ>(hi16<4>(wd[i], V), v[1]);
            ld_zones<NZ>(lo16<4>(wd[i + 1], V), v[2]);
            ld_zones<NZ>(hi16<4>(wd[i + 1], V), v[3]);
#pragma unroll
            for (int k = 0; k < 4; ++k)
#pragma unroll
                for (int q = 0; q < n; ++q) acc[q] = padd(acc[q], v[k][q]);
        }
    // the pieces of split rows
    if (rounds) {
#pragma unroll
        for (int r = 0; r < 5; ++r) {
            if (r >= rounds) break;
            PK o[n];
#pragma unroll
            for (int z = 0; z < NZ; ++z) zset<NZ>(o, z, __shfl_down_sync(0xffffffffu, zget<NZ>(acc, z), 1 << r));
            if (sd >> (17 + r) & 1)
#pragma unroll
                for (int q = 0; q < n; ++q) acc[q] = padd(acc[q], o[q]);
        }
    }
    if (sd >> 16 & 1) {
        const uint32_t d = Fk + (sd & 0xffffu);
        if (NZ > 1 && need == (1u << NZ) - 1) {
#pragma unroll
            for (int q = 0; q < n; ++q) stp(d + (int)sizeof(PK) * q, acc[q]);
        } else {
#pragma unroll
            for (int z = 0; z < NZ; ++z)
                if (need >> z & 1) sts(d + 4 * z, zget<NZ>(acc, z));
        }
    }
}
template <int NZ, class CAP>
__device__ __forceinline__ void gather_pass(const Resident<NZ, CAP>& r, uint32_t V, uint32_t Fk, uint32_t need) {
    const int wa = r.cnt >> 12 & 63, wb = r.cnt >> 18 & 63;
    if (wa) gather_slice<NZ>(r.ga, wa, (int)(r.cnt >> 24 & 7), r.sa, V, Fk, need);
    if (wb) gather_slice<NZ>(r.gb, wb, (int)(r.cnt >> 28), r.sb, V, Fk, need);
}

// ---------------------------------------------------------------------------
// (d) one species' candidate in every zone, and its share of the error measures:
// Eq. 3 with the kappa switch, or (QSS) the alpha-QSS corrector.  The arithmetic
// is update_reduce_mixed's, operation by operation.
// ---------------------------------------------------------------------------
template <int NZ, bool QSS>
__device__ __forceinline__ void candidate(const OptsDev& O, uint32_t row, uint32_t row2,
                                          float A, const typename Pack<NZ>::T (&yh)[Pack<NZ>::n],
                                          const typename Pack<NZ>::T (&yl)[Pack<NZ>::n],
                                          const typename Pack<NZ>::T (&h)[Pack<NZ>::n],
                                          typename Pack<NZ>::T (&nh)[Pack<NZ>::n], typename Pack<NZ>::T (&nl)[Pack<NZ>::n],
                                          typename Pack<NZ>::T (&ch)[Pack<NZ>::n], typename Pack<NZ>::T (&cl)[Pack<NZ>::n],
                                          unsigned (&rb)[NZ]) {
    using PK = typename Pack<NZ>::T;
    constexpr int n = Pack<NZ>::n;
    PK fp[n], kk[n], a;
    if constexpr (NZ == 2) {
        const float4 r = ldf4(row);
        fp[0] = make_float2(r.x, r.y);
        kk[0] = make_float2(r.z, r.w);
    } else {
#pragma unroll
        for (int q = 0; q < n; ++q) {
            ldp(row + (int)sizeof(PK) * q, fp[q]);
            ldp(row + (int)sizeof(PK) * (n + q), kk[q]);
        }
    }
    pall(a, A);
#pragma unroll
    for (int q = 0; q < n; ++q) {
        const PK y = yh[q], yn = pneg(y);
        PK dh, dl;
        if (!QSS) {
            // explicit branch: the change h (F+ - k y) added to the pair
            PK one;
            pall(one, 1.f);
            const PK kdt = pmul(kk[q], h[q]);
            const PK de = pmul(h[q], pfma(kk[q], yn, fp[q]));
            PK s, e, xh, xl;
            ptwo_sum(y, de, s, e);
            ptwo_sum(s, padd(e, yl[q]), xh, xl);
            // asymptotic branch: y' itself
            const PK num = pfma(h[q], fp[q], y), den = padd(one, kdt);
            PK ah, ad, al;
#pragma unroll
            for (int c = 0; c < (NZ > 1 ? 2 : 1); ++c) pset(ah, c, __fdividef(pget(num, c), pget(den, c)));
            ptwo_sum(ah, yn, ad, al);
            al = psub(al, yl[q]);
#pragma unroll
            for (int c = 0; c < (NZ > 1 ? 2 : 1); ++c) {
                const bool asy = pget(kdt, c) >= O.kappa32;
                pset(nh[q], c, asy ? pget(ah, c) : pget(xh, c));
                pset(nl[q], c, asy ? 0.f : pget(xl, c));
                pset(dh, c, asy ? pget(ad, c) : pget(de, c));
                pset(dl, c, asy ? pget(al, c) : 0.f);
            }
        } else {
            PK fq, kq;
            ldp(row2 + (int)sizeof(PK) * q, fq);
            ldp(row2 + (int)sizeof(PK) * (n + q), kq);
#pragma unroll
            for (int c = 0; c < (NZ > 1 ? 2 : 1); ++c) {
                const float yc = pget(y, c), lc = pget(yl[q], c), hc = pget(h[q], c), fc = pget(fp[q], c);
                const float kbar = 0.5f * (pget(kk[q], c) + pget(kq, c));
                const float x = __fmul_rn(kbar, hc);
                float wa, wb, rh, rl, eh, el;
                qss_weights32(x, wa, wb);
                const float ft = fmaf(wa, pget(fq, c), wb * fc);
                if (x <= 1.f) {
                    eh = __fdividef(__fmul_rn(hc, fmaf(-kbar, yc, ft)), fmaf(wa, x, 1.f));
                    el = 0.f;
                    float s, e;
                    two_sum(yc, eh, s, e);
                    two_sum(s, __fadd_rn(e, lc), rh, rl);
                } else {
                    rh = qss_update1_32(yc, ft, kbar, hc);
                    rl = 0.f;
                    two_sum(rh, -yc, eh, el);
                    el = __fsub_rn(el, lc);
                }
                pset(nh[q], c, rh);
                pset(nl[q], c, rl);
                pset(dh, c, eh);
                pset(dl, c, el);
            }
        }
        // A (dh + dl): the product A dh split exactly by an FMA
        const PK p = pmul(a, dh);
        const PK pe = pfma(a, dh, pneg(p));
        ch[q] = p;
        cl[q] = pfma(a, dl, pe);
    }
    // the accept test: on the high parts outside the guard band, on the pairs in
    // FP64 inside it; a failure is recorded as an infinite ratio
#pragma unroll
    for (int z = 0; z < NZ; ++z) {
        const float y = zget<NZ>(yh, z), x = zget<NZ>(nh, z);
        const float m = fmaxf(y, x);
        const float r = __fdividef(fabsf(__fsub_rn(x, y)), m);
        const bool tested = m > O.ymin_hi32;
        unsigned v = tested ? (r > O.thr_hi32 ? 0x7f800000u : __float_as_uint(r)) : 0u;
        const bool sure = tested ? (r < O.thr_lo32 || r > O.thr_hi32) : m < O.ymin_lo32;
        if (!sure) {
            const double yd = (double)y + (double)zget<NZ>(yl, z), xd = (double)x + (double)zget<NZ>(nl, z);
            v = 0u;
            if (tested || fmax(yd, xd) > O.y_min) {
                bool pass;
                if (r < O.thr_lo32) pass = true;
                else if (r > O.thr_hi32) pass = false;
                else pass = fabs(xd - yd) <= O.eps_r * (yd > xd ? yd : xd);
                v = pass ? __float_as_uint(r) : 0x7f800000u;
            }
        }
        rb[z] = v;
    }
}

// The warp's sums of the zones' conservation pairs.  The butterfly's first
// log2 NZ levels also hand each share of 32 / NZ lanes its zone, so the later
// levels carry one zone per lane: the same tree, zone z's total in its lanes.
template <int NZ>
__device__ __forceinline__ void butterfly(const typename Pack<NZ>::T (&ch)[Pack<NZ>::n],
                                          const typename Pack<NZ>::T (&cl)[Pack<NZ>::n], int lane, float& h, float& l) {
    float vh[NZ], vl[NZ];
#pragma unroll
    for (int z = 0; z < NZ; ++z) {
        vh[z] = zget<NZ>(ch, z);
        vl[z] = zget<NZ>(cl, z);
    }
    int off = 16;
#pragma unroll
    for (int m = NZ; m > 1; m >>= 1, off >>= 1) {
        const bool up = lane & off;
#pragma unroll
        for (int z = 0; z < m / 2; ++z) {
            const float kh = up ? vh[z + m / 2] : vh[z], sh = up ? vh[z] : vh[z + m / 2];
            const float kl = up ? vl[z + m / 2] : vl[z], sl = up ? vl[z] : vl[z + m / 2];
            const float oh = __shfl_xor_sync(0xffffffffu, sh, off), ol = __shfl_xor_sync(0xffffffffu, sl, off);
            float s, e;
            two_sum(kh, oh, s, e);
            vh[z] = s;
            vl[z] = __fadd_rn(__fadd_rn(kl, ol), e);
        }
    }
    h = vh[0];
    l = vl[0];
#pragma unroll
    for (int o = 16 / NZ; o > 0; o >>= 1) {
        const float oh = __shfl_xor_sync(0xffffffffu, h, o), ol = __shfl_xor_sync(0xffffffffu, l, o);
        float s, e;
        two_sum(h, oh, s, e);
        h = s;
        l = __fadd_rn(__fadd_rn(l, ol), e);
    }
}

// ---------------------------------------------------------------------------
// A zone's lanes: what the next decision needs and does not depend on its outcome.
// In three stages, so that a single warp can put other work between an FP64
// operation and the use of its result.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void prepare_1(Scal& S) { S.ts = S.t + (double)S.h; }
__device__ __forceinline__ void prepare_2(Scal& S) {
    S.tf = __double2float_rn(S.ts);
    S.ta = S.clip ? S.te : S.ts;
    S.rem_d = S.te - S.ta;
}
__device__ __forceinline__ void prepare_3(Scal& S, const PlanDev& P) {
    S.u = S.cst ? 0.f : __fmul_rn(S.tf, S.us);
    S.rem_acc = (float)S.rem_d;
    S.last = S.clip || !(S.ta < S.te);
    // the cached rates serve while no rate moves by a quarter ulp; without a cache
    // (large networks: every pass takes the rates at its own u) while every factor
    // 2^(-c u) is 1, as it is at the cached rates' u
    S.refresh = S.live && (P.rate_cache ? !(fabsf(S.u - S.ur) <= P.u_tol)
                                        : !(fabsf(S.u) <= P.u_one && fabsf(S.ur) <= P.u_one));
}

// accept or reject the attempt and set up the next one: decide_mixed's rules
__device__ __forceinline__ void decide_slot(Scal& S, const OptsDev& O, float cs, unsigned rbits, bool& acc, bool& done) {
    const bool fin = isfinite(cs);
    const float cons = fabsf(cs), rmax = __uint_as_float(rbits);
    acc = S.live && fin && rbits < 0x7f800000u && cons <= O.eps_c32;
    done = false;
    if (acc) {
        // min of the two rounded quotients is the rounded smaller one, so one division
        // does unless they lie within rounding of each other
        const float ra = fmaxf(rmax, 1e-30f), rb = fmaxf(cons, 1e-30f);
        const float xa = O.ga32 * rb, xb = O.gb32 * ra;  // xa < xb: ga32 / ra is the smaller
        const bool ia = xa < xb;
        float q = __fdiv_rn(ia ? O.ga32 : O.gb32, ia ? ra : rb);
        if (!(fabsf(xa - xb) > 1e-5f * xa)) q = fminf(q, __fdiv_rn(ia ? O.gb32 : O.ga32, ia ? rb : ra));
        const float dt = __fmul_rn(S.h, fminf(O.grow32, q));
        S.dt = dt;
        S.steps += 1;
        S.nrej = 0;
        if (S.last) {
            S.t = S.te;
            done = true;
        } else {
            S.t = S.ta;
            S.rem = S.rem_acc;
            if (S.steps >= O.max_steps) {
                S.status = 1;  // STEP_LIMIT
                done = true;
            } else {
                S.clip = dt >= S.rem_acc;
                S.h = S.clip ? S.rem_acc : dt;
            }
        }
    } else if (S.live) {
        S.rejects += 1;
        S.nrej += 1;
        const float dt = __fmul_rn(S.h, O.shrink32);
        if (S.nrej > O.max_reject) {
            S.status = fin ? 4 : 3;  // MAX_REJECT : NONFINITE
            done = true;
        } else if (!(dt > fmaf(4.f * O.dt_min32, S.tf, 1e-43f))) {
            // t <= t + h, so only a dt near or below the limit needs the FP64 compare
            if ((double)dt < O.dt_min_frac * S.t) {
                S.status = 2;  // DT_UNDERFLOW
                done = true;
            }
        }
        S.dt = dt;
        S.clip = dt >= S.rem;
        S.h = S.clip ? S.rem : dt;
    }
}

// ---------------------------------------------------------------------------
// End the zones of `done` and take new ones from the queue; every thread of the
// group, once per zone.  The species' pairs travel through the zone's (F+, k)
// row, which is free then, so the loops below keep nothing of this in registers.
// S: the control lanes' scalars of their zone.
// ---------------------------------------------------------------------------
template <int NZ, bool WARP>
__device__ __noinline__ void change_zones(const PlanDev& P, const OptsDev& O, SlotBase g, SlotCtl& C, int tid, int T,
                                          uint32_t done, Scal& S) {
    constexpr int LZ = 32 / NZ;
    const SlotSync<WARP> gs{WARP ? 0 : 1 + (int)threadIdx.x / T, T};
    const int lane = tid & 31, w = tid >> 5, cz = lane / LZ, cw = (T >> 5) - 1, Tw = WARP ? 32 : T - 32;
    const bool mine = tid < P.N;
    const uint32_t Yi = g.gb + P.sl.off_Y + at<NZ>(tid), row = g.gb + P.sl.off_Fk + 8 * NZ * tid;
    gs.sync();
    uint32_t live = C.live, fresh = 0;
    while (done) {
        uint32_t again = 0;
        for (int z = 0; z < NZ; ++z) {
            if (!(done >> z & 1)) continue;
            // write back (Sec. 6 step 3 outputs: abundances, energy, final dt)
            const int zo = C.zone[z];
            if (w == cw && cz == z && lane == z * LZ) C.status = S.status;
            gs.sync();
            if (zo >= 0) {
                double* Yg = P.Y + (size_t)zo * P.N;
                double e = 0.0;
                if (C.status != 5 && mine) {
                    const double y0 = Yg[tid];  // still Y(t_start)
                    // a pair that never changed returns the FP64 input bit for bit
                    const float hi = lds(row + 4 * z), lo = lds(row + 4 * (NZ + z));
                    const float hi0 = __double2float_rn(y0);
                    const float lo0 = __double2float_rn(y0 - (double)hi0);
                    const double y = (hi == hi0 && lo == lo0) ? y0 : (double)hi + (double)lo;
                    if (P.bind) e = fma(P.bind[tid], y - y0, e);
                    Yg[tid] = y;
                }
                if (P.bind) {
                    double* red = (double*)__cvta_shared_to_generic(g.gb + P.sl.off_red);
#pragma unroll
                    for (int off = 16; off > 0; off >>= 1) e += __shfl_xor_sync(0xffffffffu, e, off);
                    if (lane == 0) red[w] = e;
                    gs.sync();
                    if (tid == 0) {
                        double es = 0.0;
                        for (int i = 0; i < (T >> 5); ++i) es += red[i];
                        P.energy[zo] = es;
                    }
                }
                if (w == cw && lane == z * LZ) {
                    P.t_out[zo] = S.t;
                    P.dt_next[zo] = (double)S.dt;
                    P.steps[zo] = S.steps;
                    P.rejects[zo] = S.rejects;
                    if (P.props) P.props[zo] = 0;
                    P.status[zo] = S.status;
                    if (O.zone_ns) {
                        long long* tz = O.zone_ns + 2 * (size_t)(P.zone_base + zo);
                        tz[0] = C.fetch_ns[z];
                        tz[1] = global_ns();
                    }
                }
            }
            gs.sync();
            // the next zone
            if (tid == 0) {
                // a home CTA's slots start with zones dealt over all CTAs, then over
                // the groups, so that few zones spread over the chip
                const int b = (int)blockIdx.x - P.cta_begin;
                const bool deal = zo == -2 && (int)blockIdx.x >= P.cta_begin && (int)blockIdx.x < P.cta_end;
                const int q = deal ? (z * P.ng + (int)threadIdx.x / T) * (P.cta_end - P.cta_begin) + b
                                   : P.dealt + atomicAdd(P.queue_head, 1);
                C.zone[z] = q < P.n_zones ? P.order[q] : -1;
                C.valid = 1;
                if (O.zone_ns) C.fetch_ns[z] = global_ns();
            }
            gs.sync();
            const int zi = C.zone[z];
            if (zi < 0) {
                // an empty slot runs along on zeros
                live &= ~(1u << z);
                if (mine) {
                    sts(Yi + 128 * z, 0.f);
                    sts(row + 4 * z, 0.f);
                    sts(row + 4 * (NZ + z), 0.f);
                }
                for (int i = tid; i < P.st.slots * Tw; i += T) sts(g.gb + P.sl.off_K + 4 * (i * NZ + z), 0.f);
                if (w == cw && cz == z) {
                    S = Scal{};
                    S.cst = true;
                    if (lane == z * LZ) {
                        C.h[z] = 0.f;
                        C.u[z] = 0.f;
                    }
                }
                gs.sync();
                continue;
            }
            live |= 1u << z;
            fresh |= 1u << z;
            if (mine) {
                const double y = P.Y[(size_t)zi * P.N + tid];
                const float hi = __double2float_rn(y);
                sts(row + 4 * z, hi);
                sts(row + 4 * (NZ + z), __double2float_rn(y - (double)hi));
                sts(Yi + 128 * z, hi);
                if (!(isfinite(y) && y >= 0.0)) C.valid = 0;  // benign race: every writer stores 0
            }
            if (w == cw && cz == z) {
                const double T0 = P.T0[zi], rho0 = P.rho0[zi], tau = P.tau[zi];
                const double ts = P.t_start[zi], te = P.t_end[zi], dtt = P.dt_trial[zi];
                S = Scal{};
                S.t = ts;
                S.te = te;
                S.cst = !(tau > 0.0);
                const double inv_tau = S.cst ? 0.0 : 1.0 / tau;
                S.us = S.cst ? 0.f : __double2float_rn(inv_tau * 1.4426950408889634);
                const double dt = dtt > 0.0 ? dtt : ts;
                S.dt = (float)dt;
                S.live = true;
                // the first flux pass computes the cached rates, at u(t_start)
                S.ur = S.cst ? 0.f : __fmul_rn(__double2float_rn(ts), S.us);
                const bool ok = isfinite(T0) && T0 > 0.0 && isfinite(rho0) && rho0 > 0.0 && isfinite(tau) &&
                                isfinite(ts) && isfinite(te) && ts >= 0.0 && te > ts && isfinite(dtt) &&
                                (ts > 0.0 || dtt > 0.0);
                const double rem = te - ts;
                S.clip = dt >= rem;
                S.h = (float)(S.clip ? rem : dt);
                S.rem = (float)rem;
                if (lane == z * LZ) {
                    if (ok) {
                        C.lnT0 = log(T0);
                        C.lnR0 = log(rho0);
                    } else {
                        C.valid = 0;
                    }
                }
            }
            gs.sync();
            if (C.valid) {
                // the zone's rates at (T0, rho0), once per zone (Sec. 10 item (2))
                const double lnT0 = C.lnT0, lnR0 = C.lnR0;
                const int R1 = P.R1, R12 = P.R12;
                const uint16_t* sj = (const uint16_t*)(P.slot_blob + P.st.off_sj);
                for (int i = tid; i < P.st.slots * Tw; i += T) {
                    const int j = sj[i];  // the reaction of block i / Tw of worker thread i % Tw
                    if (j == 0xffff) continue;
                    const double2 p = P.rate0[j];
                    const double r1 = (double)((j >= R1) + (j >= R12));
                    sts(g.gb + P.sl.off_K + 4 * (i * NZ + z), (float)exp(fma(p.y, lnT0, p.x) + r1 * lnR0));
                }
            }
            if (w == cw && cz == z) {
                S.status = !C.valid ? 5 : (O.max_steps <= 0 ? 1 : 0);  // INVALID, STEP_LIMIT
                if (lane == z * LZ) {
                    C.u[z] = S.ur;
                    C.h[z] = S.h;
                    C.end = S.status != 0;
                }
            }
            gs.sync();
            if (C.end) again |= 1u << z;
        }
        fresh &= ~again;
        done = again;
    }
    if (tid == 0) {
        C.live = live;
        C.fresh = fresh;
        C.rmask = 0;
    }
    gs.sync();
}

// the warps' sums of a zone, in warp order
template <int NZ>
__device__ __forceinline__ void combine_warps(uint32_t red, int nsw, float& ch, float& cl, uint32_t& rbits) {
    float4 r0 = ldf4(red);
    ch = r0.x;
    cl = r0.y;
    rbits = __float_as_uint(r0.z);
#pragma unroll 1
    for (int i = 1; i < nsw; i += 4) {
        float4 r[4];
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (i + k < nsw) r[k] = ldf4(red + 16 * NZ * (i + k));
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (i + k < nsw) {
                float s, e;
                two_sum(ch, r[k].x, s, e);
                ch = s;
                cl = __fadd_rn(__fadd_rn(cl, r[k].y), e);
                rbits = max(rbits, __float_as_uint(r[k].z));
            }
    }
}

template <int NZ> __device__ __forceinline__ uint32_t zone_bits(bool b) {
    const uint32_t v = __ballot_sync(0xffffffffu, b);
    uint32_t m = v & 1;
#pragma unroll
    for (int z = 1; z < NZ; ++z) m |= (v >> (z * (32 / NZ)) & 1) << z;
    return m;
}

// (d) of one warp: the species' candidates, stored for the flux pass, and the
// warp's sums; zone cz's in the lanes of cz
template <int NZ, bool QSS>
__device__ __forceinline__ void update_warp(const OptsDev& O, bool mine, uint32_t row, uint32_t row2, uint32_t Yi,
                                            float A, int lane, const typename Pack<NZ>::T (&yh)[Pack<NZ>::n],
                                            const typename Pack<NZ>::T (&yl)[Pack<NZ>::n],
                                            const typename Pack<NZ>::T (&h)[Pack<NZ>::n],
                                            typename Pack<NZ>::T (&nh)[Pack<NZ>::n], typename Pack<NZ>::T (&nl)[Pack<NZ>::n],
                                            float& cs_h, float& cs_l, uint32_t& rbits) {
    constexpr int n = Pack<NZ>::n;
    typename Pack<NZ>::T ch[n], cl[n];
    uint32_t rb[NZ];
#pragma unroll
    for (int q = 0; q < n; ++q) {
        pall(ch[q], 0.f);
        pall(cl[q], 0.f);
    }
#pragma unroll
    for (int z = 0; z < NZ; ++z) rb[z] = 0;
    if (mine) {
        candidate<NZ, QSS>(O, row, row2, A, yh, yl, h, nh, nl, ch, cl, rb);
        st_zones<NZ>(Yi, nh);
    }
    butterfly<NZ>(ch, cl, lane, cs_h, cs_l);
    rbits = __reduce_max_sync(0xffffffffu, rb[0]);
#pragma unroll
    for (int z = 1; z < NZ; ++z) {
        const uint32_t m = __reduce_max_sync(0xffffffffu, rb[z]);
        if (lane / (32 / NZ) >= z) rbits = m;
    }
}

// QSS: the predicted states, stored for the flux pass
template <int NZ>
__device__ __forceinline__ void predict_species(uint32_t row, uint32_t Yi, const typename Pack<NZ>::T (&yh)[Pack<NZ>::n],
                                                const typename Pack<NZ>::T (&h)[Pack<NZ>::n]) {
    float fk[2 * NZ];
#pragma unroll
    for (int z = 0; z < 2 * NZ; ++z) fk[z] = lds(row + 4 * z);
#pragma unroll
    for (int z = 0; z < NZ; ++z) sts(Yi + 128 * z, qss_update1_32(zget<NZ>(yh, z), fk[z], fk[NZ + z], zget<NZ>(h, z)));
}

// ---------------------------------------------------------------------------
// A group of several warps: warps 0 .. W - 2 hold the species, the flux blocks and
// the gather slices; warp W - 1 keeps the zones' scalars, prepares each attempt
// beside the update and decides beside the flux pass.  Barriers per attempt:
// after the gather, the update and the decision.
// ---------------------------------------------------------------------------
template <int NZ, bool QSS, class CAP>
__device__ __forceinline__ void run_workers(const PlanDev& P, const OptsDev& O, const SlotBase g, SlotCtl& C, const int tid,
                                            const SlotSync<false> gs) {
    using PK = typename Pack<NZ>::T;
    constexpr int n = Pack<NZ>::n, LZ = 32 / NZ;
    const int lane = tid & 31, w = tid >> 5, nsw = (P.N + 31) >> 5, Tw = P.T - 32;
    const bool mine = tid < P.N;
    const uint32_t Yi = g.gb + P.sl.off_Y + at<NZ>(tid), row = g.gb + P.sl.off_Fk + 8 * NZ * tid,
                   Fk = g.gb + P.sl.off_Fk, ctl = g.gb + P.sl.off_ctl;
    const float A = mine ? ((const float*)(P.blob + P.tl.off_A))[tid] : 0.f;
    const WorkAddr f = work_addr(P, g);
    Resident<NZ, CAP> res;
    res.load(P, tid, Tw);
    PK yh[n], yl[n];
#pragma unroll
    for (int q = 0; q < n; ++q) {
        pall(yh[q], 0.f);
        pall(yl[q], 0.f);
    }
    uint32_t done = (1u << NZ) - 1;  // at first every slot is to be filled
    for (;;) {
        // ---- a zone ended: once per zone ----
        if (mine)
#pragma unroll
            for (int z = 0; z < NZ; ++z)
                if (done >> z & 1) {
                    sts(row + 4 * z, zget<NZ>(yh, z));
                    sts(row + 4 * (NZ + z), zget<NZ>(yl, z));
                }
        Scal none;
        change_zones<NZ, false>(P, O, g, C, tid, P.T, done, none);
        if (!C.live) break;
        if (mine)
#pragma unroll
            for (int z = 0; z < NZ; ++z)
                if (done >> z & 1) {
                    zset<NZ>(yh, z, lds(row + 4 * z));
                    zset<NZ>(yl, z, lds(row + 4 * (NZ + z)));
                }
        const uint32_t fresh = C.fresh;
        if (fresh) {
            // (a) and (b) of the new zones' first states (the other zones' values come
            // out as they were, and are not stored)
            refresh_rates<NZ>(P, g, tid, Tw, res, f, fresh);
            flux_pass<NZ>(res, f);
            gs.sync();
            gather_pass<NZ>(res, f.V, Fk, fresh);
            gs.sync();
        }
        // ---- steps, until a zone ends ----
        do {
            PK h[n], nh[n], nl[n];
#pragma unroll
            for (int q = 0; q < n; ++q) ldp(ctl + (int)sizeof(PK) * q, h[q]);
            if (QSS) {  // the predicted state's (F+, k)
                if (mine) predict_species<NZ>(row, Yi, yh, h);
                gs.sync();
                const uint32_t pm = C.rmask;
                if (pm) refresh_rates<NZ>(P, g, tid, Tw, res, f, pm);
                flux_pass<NZ>(res, f);
                gs.sync();
                gather_pass<NZ>(res, f.V, g.gb + P.sl.off_Fk2, (1u << NZ) - 1);
                gs.sync();
            }
            // ---- (d) update and error measures ----
            if (w < nsw) {
                float ch, cl;
                uint32_t rb;
                update_warp<NZ, QSS>(O, mine, row, g.gb + P.sl.off_Fk2 + 8 * NZ * tid, Yi, A, lane, yh, yl, h, nh, nl, ch,
                                     cl, rb);
                if ((lane & (LZ - 1)) == 0)
                    asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %3};" ::"r"(g.gb + P.sl.off_red +
                                                                                  16 * (w * NZ + lane / LZ)),
                                 "f"(ch), "f"(cl), "f"(__uint_as_float(rb))
                                 : "memory");
            }
            gs.sync();
            // ---- (a) for the candidate states, as the accepted zones' next attempts
            // need it, while the control warp decides ----
            const uint32_t rm = QSS ? 0u : ldu(ctl + (int)offsetof(SlotCtl, rmask));
            if (rm) refresh_rates<NZ>(P, g, tid, Tw, res, f, rm);
            flux_pass<NZ>(res, f);
            gs.sync();
            // ---- (b) the gathers, stored for the accepted zones ----
            const uint2 ad = ldu2(ctl + (int)offsetof(SlotCtl, acc));
            done = ad.y;
#pragma unroll
            for (int z = 0; z < NZ; ++z)
                if (ad.x >> z & 1) {
                    zset<NZ>(yh, z, zget<NZ>(nh, z));
                    zset<NZ>(yl, z, zget<NZ>(nl, z));
                }
            // (rejected zones repeat their attempts with the (F+, k) they have)
            if (ad.x) {
                gather_pass<NZ>(res, f.V, Fk, ad.x & ~ad.y);
                gs.sync();
            }
        } while (!done);
    }
}

template <int NZ, bool QSS>
__device__ __forceinline__ void run_control(const PlanDev& P, const OptsDev& O, const SlotBase g, SlotCtl& C, const int tid,
                                            const SlotSync<false> gs) {
    constexpr int LZ = 32 / NZ;
    const int lane = tid & 31, cz = lane / LZ, nsw = (P.N + 31) >> 5;
    const uint32_t red = g.gb + P.sl.off_red + 16 * cz;
    const bool head = lane == cz * LZ;
    Scal S{};
    uint32_t done = (1u << NZ) - 1;
    for (;;) {
        if (done) {
            Scal X = S;  // a copy, so that S itself stays in registers
            change_zones<NZ, false>(P, O, g, C, tid, P.T, done, X);
            S = X;
            if (!C.live) break;
            if (C.fresh) {  // the new zones' flux pass and gathers
                gs.sync();
                gs.sync();
            }
        }
        // what the decision needs and does not depend on its outcome; the flux pass
        // refreshes the cached rates whatever the outcome
        prepare_1(S);
        prepare_2(S);
        prepare_3(S, P);
        const uint32_t rm = zone_bits<NZ>(S.refresh);
        if (S.refresh) S.ur = S.u;
        if (head) C.u[cz] = S.u;
        if (lane == 0) C.rmask = rm;
        if (QSS) {
            gs.sync();
            gs.sync();
            gs.sync();
        }
        gs.sync();
        float ch, cl;
        uint32_t rb;
        combine_warps<NZ>(red, nsw, ch, cl, rb);
        bool acc, end;
        decide_slot(S, O, __fadd_rn(ch, cl), rb, acc, end);
        const uint32_t am = zone_bits<NZ>(acc), dm = zone_bits<NZ>(end);
        if (head) C.h[cz] = S.h;
        if (lane == 0) {
            C.acc = am;
            C.done = dm;
        }
        gs.sync();
        done = dm;
        if (am) gs.sync();  // the workers' gather
    }
}

// ---------------------------------------------------------------------------
// A group of one warp (small networks): everything in turn, the scalars in
// registers, a zone's in its share of the lanes.
// ---------------------------------------------------------------------------
template <int NZ, bool QSS, class CAP>
__device__ __forceinline__ void run_warp(const PlanDev& P, const OptsDev& O, const SlotBase g, SlotCtl& C, const int lane) {
    using PK = typename Pack<NZ>::T;
    constexpr int n = Pack<NZ>::n, LZ = 32 / NZ;
    const SlotSync<true> gs{0, 32};
    const int cz = lane / LZ;
    const bool mine = lane < P.N;
    const uint32_t Yi = g.gb + P.sl.off_Y + at<NZ>(lane), row = g.gb + P.sl.off_Fk + 8 * NZ * lane,
                   Fk = g.gb + P.sl.off_Fk;
    const float A = mine ? ((const float*)(P.blob + P.tl.off_A))[lane] : 0.f;
    const WorkAddr f = work_addr(P, g);
    Resident<NZ, CAP> res;
    res.load(P, lane, 32);
    PK yh[n], yl[n];
#pragma unroll
    for (int q = 0; q < n; ++q) {
        pall(yh[q], 0.f);
        pall(yl[q], 0.f);
    }
    Scal S{};
    uint32_t done = (1u << NZ) - 1, need = 0;
    for (;;) {
        uint32_t rm = 0;
        if (done) {
            if (mine)
#pragma unroll
                for (int z = 0; z < NZ; ++z)
                    if (done >> z & 1) {
                        sts(row + 4 * z, zget<NZ>(yh, z));
                        sts(row + 4 * (NZ + z), zget<NZ>(yl, z));
                    }
            Scal X = S;
            change_zones<NZ, true>(P, O, g, C, lane, 32, done, X);
            S = X;
            if (!C.live) break;
            if (mine)
#pragma unroll
                for (int z = 0; z < NZ; ++z)
                    if (done >> z & 1) {
                        zset<NZ>(yh, z, lds(row + 4 * z));
                        zset<NZ>(yl, z, lds(row + 4 * (NZ + z)));
                    }
            rm = C.fresh;
            need |= rm;
        }
        // (a) of the states just reached: only they refresh their cached rates (a new
        // zone computes them, at the u set with it); beside it the FP64 work of the
        // next attempt
        if (need) {
            const bool go = (need & ~rm) >> cz & 1;
            rm |= zone_bits<NZ>(go && S.refresh);
            if (go && S.refresh) S.ur = S.u;
            if (go && lane == cz * LZ) C.u[cz] = S.u;
            gs.sync();
        }
        prepare_1(S);
        if (need) {
            if (rm) refresh_rates<NZ>(P, g, lane, 32, res, f, rm);
            flux_pass<NZ>(res, f);
            gs.sync();
        }
        prepare_2(S);
        if (need) {
            gather_pass<NZ>(res, f.V, Fk, need);
            gs.sync();
        }
        prepare_3(S, P);
        PK h[n], nh[n], nl[n];
#pragma unroll
        for (int z = 0; z < NZ; ++z) zset<NZ>(h, z, __shfl_sync(0xffffffffu, S.h, z * LZ));
        if (QSS) {
            if (mine) predict_species<NZ>(row, Yi, yh, h);
            const uint32_t pm = zone_bits<NZ>(S.refresh);
            if (S.refresh) S.ur = S.u;
            S.refresh = false;
            if (lane == cz * LZ) C.u[cz] = S.u;
            gs.sync();
            if (pm) refresh_rates<NZ>(P, g, lane, 32, res, f, pm);
            flux_pass<NZ>(res, f);
            gs.sync();
            gather_pass<NZ>(res, f.V, g.gb + P.sl.off_Fk2, (1u << NZ) - 1);
            gs.sync();
        }
        float ch, cl;
        uint32_t rb;
        update_warp<NZ, QSS>(O, mine, row, g.gb + P.sl.off_Fk2 + 8 * NZ * lane, Yi, A, lane, yh, yl, h, nh, nl, ch, cl, rb);
        bool acc, end;
        decide_slot(S, O, __fadd_rn(ch, cl), rb, acc, end);
        const uint32_t am = zone_bits<NZ>(acc);
        done = zone_bits<NZ>(end);
#pragma unroll
        for (int z = 0; z < NZ; ++z)
            if (am >> z & 1) {
                zset<NZ>(yh, z, zget<NZ>(nh, z));
                zset<NZ>(yl, z, zget<NZ>(nl, z));
            }
        need = am & ~done;
        gs.sync();
    }
}

template <int A1, int A2, int A3, int A4, int A5> struct Cap {
    static constexpr int F1 = A1, F2 = A2, FA = A3, GA = A4, GB = A5;
};
#define CAP_OF(k) Cap<kSlotCaps[k].f1, kSlotCaps[k].f2, kSlotCaps[k].fa, kSlotCaps[k].ga, kSlotCaps[k].gb>

// one plan's groups
template <int NZ, bool QSS, int CK>
__device__ __forceinline__ void run_plan(const PlanDev& P, const OptsDev& O, const SlotBase g, SlotCtl& C, int gr, int tid) {
    if (CK == kCapWarp) {
        run_warp<NZ, QSS, CAP_OF(CK)>(P, O, g, C, tid);
    } else {
        const SlotSync<false> gs{1 + gr, P.T};
        if (tid < P.T - 32) run_workers<NZ, QSS, CAP_OF(CK)>(P, O, g, C, tid, gs);
        else run_control<NZ, QSS>(P, O, g, C, tid, gs);
    }
}

// One of several plans.  Its index is a constant, so that the plan's fields are operands
// in constant memory; through an index they were loads and spilled registers (150/1604
// alone, 1024 zones to 1e-9 s: 600 ms against 467; 365/4400, 512 zones: 522 against 304).
template <int NZ, bool QSS, int I>
__device__ __forceinline__ void run_cap(const LaunchParams& lp, const SlotBase g, SlotCtl& C, int gr, int tid) {
    const PlanDev& P = lp.plans[I];
    if (P.cap == kCapWarp) run_plan<NZ, QSS, kCapWarp>(P, lp.o, g, C, gr, tid);
    else if (P.cap == kCapWide) run_plan<NZ, QSS, kCapWide>(P, lp.o, g, C, gr, tid);
    else run_plan<NZ, QSS, kCapGroup>(P, lp.o, g, C, gr, tid);
}
static_assert(kMaxPlans == 4, "the kernel's constant plan indices");

// CK: the capacities of the one plan, or kCapMany: any mix of plans.  A CTA works on one
// plan: its home plan or, for the CTAs past the first that every SM gets (one fits on an
// SM, so these start where another has ended), one that still has zones in its queue.
// (A loop over the plans in one CTA let the compiler move every plan's set-up out of the
// loop and keep it there in registers and local memory.)  16, 150 and 365 species, 2048
// zones: 690 -> 500 ms with both.  Every plan is served: a CTA past the first ones tries
// the plans from the one of its own number on, and ends only where no queue has a zone.
template <int NZ, bool QSS, int CK>
__global__ void __launch_bounds__(kSlotThreads, 1) slots_kernel(const __grid_constant__ LaunchParams lp) {
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ int s_go;
    constexpr bool ONE = CK != kCapMany;
    if (threadIdx.x == 0) {
        const int np = ONE ? 1 : lp.n_plans;
        int home = -1;  // none: no zone is left
        for (int p = 0; p < np; ++p) {
            const PlanDev& P = lp.plans[p];
            const int b = (int)blockIdx.x - P.cta_begin;
            if (b >= 0 && (int)blockIdx.x < P.cta_end && b < P.n_zones) home = p;
        }
        for (int a = 0; a < np && !ONE && home < 0; ++a) {
            const PlanDev& P = lp.plans[((int)blockIdx.x + a) % np];
            if (P.dealt + *((volatile int*)P.queue_head) < P.n_zones) home = ((int)blockIdx.x + a) % np;
        }
        s_go = home;
    }
    __syncthreads();
    const int i = s_go;
    if (i < 0) return;
    const PlanDev& P = lp.plans[ONE ? 0 : i];
    {
        const int4* src = (const int4*)P.slot_blob;
        int4* dst = (int4*)smem;
        for (int k = threadIdx.x; k < P.st.bytes / 16; k += blockDim.x) dst[k] = src[k];
    }
    __syncthreads();
    const int gr = threadIdx.x / P.T, tid = threadIdx.x - gr * P.T;
    if (gr >= P.ng) return;
    unsigned char* gb = smem + P.st.bytes + gr * P.sl.bytes;
    SlotCtl& C = *(SlotCtl*)(gb + P.sl.off_ctl);
    const SlotBase g{saddr(smem), saddr(gb)};
    if (tid < NZ) {
        sts(g.gb + P.sl.off_V + 4 * P.st.zero + 128 * tid, 0.f);
        sts(g.gb + P.sl.off_Y + at<NZ>(P.N) + 128 * tid, 1.f);  // the factor of an absent reactant
        C.h[tid] = 0.f;
        C.u[tid] = 0.f;
        C.zone[tid] = -2;
        if (tid == 0) C.live = 0;
    }
    // (change_zones begins with a barrier)
    if constexpr (ONE) {
        run_plan<NZ, QSS, CK>(P, lp.o, g, C, gr, tid);
    } else {
        if (i == 0) run_cap<NZ, QSS, 0>(lp, g, C, gr, tid);
        else if (i == 1) run_cap<NZ, QSS, 1>(lp, g, C, gr, tid);
        else if (i == 2) run_cap<NZ, QSS, 2>(lp, g, C, gr, tid);
        else run_cap<NZ, QSS, 3>(lp, g, C, gr, tid);
    }
}

typedef void (*SlotsFn)(const LaunchParams);
template <int NZ, bool QSS> SlotsFn slots_fn(int cap) {
    switch (cap) {
        case kCapWarp: return slots_kernel<NZ, QSS, kCapWarp>;
        case kCapGroup: return slots_kernel<NZ, QSS, kCapGroup>;
        case kCapWide: return slots_kernel<NZ, QSS, kCapWide>;
        default: return slots_kernel<NZ, QSS, kCapMany>;
    }
}
SlotsFn slots_fn(int nz, bool qss, int cap) {
    if (nz == 1) return qss ? slots_fn<1, true>(cap) : slots_fn<1, false>(cap);
    return qss ? slots_fn<2, true>(cap) : slots_fn<2, false>(cap);
}

}  // namespace

cudaError_t launch_slots(const LaunchParams& lp, int grid, int block, cudaStream_t stream) {
    const int cap = lp.n_plans > 1 ? kCapMany : lp.plans[0].cap;
    slots_fn(lp.nz, lp.o.method != 0, cap)<<<grid * lp.n_plans, block, lp.smem_bytes, stream>>>(lp);
    return cudaGetLastError();
}

cudaError_t slots_set_smem_limit(int bytes) {
    for (int nz = 1; nz <= 2; ++nz)
        for (int qss = 0; qss < 2; ++qss)
            for (int cap = 0; cap <= kCapMany; ++cap) {
                const cudaError_t e = cudaFuncSetAttribute((const void*)slots_fn(nz, qss, cap),
                                                           cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
                if (e != cudaSuccess) return e;
            }
    return cudaSuccess;
}

}  // namespace kn
