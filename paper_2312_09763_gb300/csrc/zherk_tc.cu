// zherk_tc.cu -- Algorithm 2 steps (iii)-(v) of arXiv:2312.09763 (Sec. 3.1) in
// one persistent launch: the Z build (eq. "littlez" / "fullz") streams U = the
// real form of Z, split in FP16 hi + lo, through a ring that stays in L2, and
// the tensor cores expand V = Z Z^dagger from it as it is written.
//
// Why: the 350-antenna x 1e5-source instance's U is 140 MB.  Built by a launch
// of its own (or inside the HERK of the batch before) it goes to HBM and comes
// back, 280 MB per instance.  Here every SM owns one product of up to 128 x 256
// of some instance for the whole source axis, so Z is needed only in source order,
// by all products at about the same time: a ring of a thousand sources per
// instance (82 MB in all there, inside the 129 MB L2) is enough, and Z is never
// read back from HBM (ncu: 3.1 of its 4.0 GB leave L2 before they are overwritten).
//
// A wave is V virtual instances (an instance, or one of S ranges of its
// sources) whose products fill the SMs.  The ring is cut into chunks of 64
// sources.  The SMs form teams that build every teams-th chunk of the wave
// each: an SM keeps one channel group and up to 12 x ant_block antennas of it.
// A finished chunk is counted in ready[chunk]; an SM's TMA warp loads it for
// the SM's own product once every SM of the team has counted it, and counts the
// SM up in done[chunk] when the loads have landed, which frees the chunk's
// place in the ring.  Both counts are released by the SM that counts itself up and
// acquired by the warp that looks at them (once they are high enough: looking is
// relaxed, as an acquire a look made hera 1 % slower), so that the loads come after
// the stores they are to see, and the next stores after the loads.  Everybody takes the chunks
// in the same order, so the oldest one never waits for a newer one; the launch is
// cooperative (all CTAs resident).  Every wait is bounded (tc.cuh).
//
// Roles of a CTA (one per SM): warp 0 TMA, warp 1 MMA, warps 2-9 drain the
// accumulator into FP32 running sums (both in TMEM) every `flush` stages,
// COUNT_WARP publishes finished and loaded chunks, FEED_WARP copies each chunk's source
// directions and WA into shared memory for the Z warps and watches the ring,
// and 12 (8 with several components) warps build Z.
//
// What bounds it (350 antennas x 1e5 sources, 19 instances a wave): L2 traffic.  A
// 64-source chunk takes 1.38 us (256 instances 15.1 ms, of 14 waves of 782 chunks;
// 56 instances 3.33, against 4.79 with the Z build fused into the HERK of the previous
// batch through HBM); in it the SMs read 12 MB of panels and write 5.3 MB of Z, where
// L2 gives 17 TB/s to reads and 5.7 to writes, and each SM moves 0.27 MB through its
// shared memory.  Copies of the kernel without one part (before its counts were
// released and acquired, when the 56 instances took 3.25 ms): without the Z stores
// 2.81, without two of the three products 3.01; the MMAs alone are 0.84 us a chunk,
// the Z build alone 0.94.  Single-channel groups are bound by their phases
// (z_ants_one).
//
// Layout of a ring row: blocks of 32 columns, 128 bytes each, hi and lo halves of
// 64 bytes (in turn, see the Z warps), so that one 128-byte-swizzled TMA box of a
// panel's rows brings both.
#include <cuda.h>
#include <cuda_fp16.h>

#include <algorithm>
#include <cmath>
#include "common.cuh"
#include "tc.cuh"
#include "zcore.cuh"
#include "zherk.h"

namespace mv {
namespace {

using namespace tc;
using namespace zcore;

constexpr int BOX = 128 * 128;            // bytes of the largest box: 128 rows x 32 columns, hi and lo
constexpr int MAX_BOX = 3;                // boxes of a stage: A and two of B
constexpr int STAGE = MAX_BOX * BOX;      // 48 KB
constexpr int STAGES = 4;
constexpr int EPI_WARPS = 8;              // four per 128 columns: warps 2-9
constexpr int COUNT_WARP = 2 + EPI_WARPS, FEED_WARP = COUNT_WARP + 1, FIRST_Z = COUNT_WARP + 2;
constexpr int TMEM_COLS = 512;            // the accumulator and the running sums, 256 columns each
constexpr int RUN_COL = 256;
constexpr int Z_BLOCK = 16;               // antennas a Z warp may have (half with channel stepping)
constexpr int Z_APH_B = Z_BLOCK * (int)sizeof(AntPhase);  // their phase factors, per Z warp
constexpr int Z_SRC_B = 6 * kZherkChunk * 4;              // a chunk's directions: 3 x S, 3 x eps
constexpr int Z_CHAN = kZherkChan;        // channels x components of a chunk's WA in shared memory
constexpr int Z_WA_B = Z_CHAN * kZherkChunk * 8;
// The Z warps' inputs: two buffers of the most channels, four or eight of fewer:
// with two, a chunk of one channel waits for the latency of a fill (12 antennas,
// 84 pairs of 70,000 sources: 704 us, with eight buffers 505).
constexpr int Z_BUF = Z_SRC_B + Z_WA_B, MAX_BUF = 8;
constexpr int Z_BARS_B = (2 * STAGES + 2 + 3 * MAX_BUF) * 8 + 16;
// Z-build warps per SM: as many as the registers allow (24 warps of 80
// registers in all with one component, 20 of 96 with several).
__host__ __device__ constexpr int z_warps(int nc) { return nc == 1 ? 12 : 8; }
constexpr int threads_for(int nc) { return (FIRST_Z + z_warps(nc)) * 32; }
constexpr int smem_for(int nc) { return STAGES * STAGE + 2 * Z_BUF + z_warps(nc) * Z_APH_B + 1024 + Z_BARS_B; }
static_assert(smem_for(1) <= 232448 && smem_for(2) <= 232448, "227 KB of shared memory");
static_assert(Z_BUF % 16 == 0 && Z_SRC_B % 16 == 0 && Z_APH_B % 16 == 0, "16-byte copies");

__device__ __forceinline__ int ld_relaxed(const int* p) {
    int v;
    asm volatile("ld.relaxed.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ int ld_acquire(const int* p) {
    int v;
    asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
// The same within the CTA, for a word in shared memory.
__device__ __forceinline__ int ld_acquire_cta(uint32_t p) {
    int v;
    asm volatile("ld.acquire.cta.shared::cta.s32 %0, [%1];" : "=r"(v) : "r"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_release_cta(uint32_t p, int v) {
    asm volatile("st.release.cta.shared::cta.s32 [%0], %1;" ::"r"(p), "r"(v) : "memory");
}
__device__ __forceinline__ bool elect_one() {
    uint32_t p;
    asm volatile("{\n\t.reg .pred q;\n\telect.sync _|q, 0xffffffff;\n\tselp.u32 %0, 1, 0, q;\n\t}" : "=r"(p));
    return p != 0;
}
// What this thread has done and seen comes before the counts it adds next.
__device__ __forceinline__ void fence_release() { asm volatile("fence.acq_rel.gpu;" ::: "memory"); }
__device__ __forceinline__ void red_add(int* p, int v) {
    asm volatile("red.relaxed.gpu.global.add.s32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
                 "l"(src), "r"(bytes), "r"(bar)
                 : "memory");
}
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}

// -------------------------------------------------------------- Z build
// The first two products of a K step share A: the first keeps it in the collector
// buffer for the second (12 % fewer shared-memory reads; 0.95 -> 0.89 us a chunk).
template <bool FIRST>
__device__ __forceinline__ void tc_mma_shared_a(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
    if constexpr (FIRST)
        asm volatile(
            "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
            "tcgen05.mma.cta_group::1.kind::f16.collector::a::fill [%0], %1, %2, %3, p;\n\t}" ::"r"(d),
            "l"(a), "l"(b), "r"(idesc), "r"(acc)
            : "memory");
    else
        asm volatile(
            "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
            "tcgen05.mma.cta_group::1.kind::f16.collector::a::lastuse [%0], %1, %2, %3, p;\n\t}" ::"r"(d),
            "l"(a), "l"(b), "r"(idesc), "r"(acc)
            : "memory");
}

// a * b + c on two packed FP32 values (FFMA2: two products per issue slot)
struct F2 {
    unsigned long long u;
};
__device__ __forceinline__ F2 pack2(float a, float b) {
    F2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r.u) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void unpack2(F2 v, float& a, float& b) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v.u));
}
__device__ __forceinline__ F2 mul2(F2 a, F2 b) {
    F2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.u) : "l"(a.u), "l"(b.u));
    return r;
}
__device__ __forceinline__ F2 fma2(F2 a, F2 b, F2 c) {
    F2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.u) : "l"(a.u), "l"(b.u), "l"(c.u));
    return r;
}

// hi and lo halves of two values (x - hi in one mixed-precision step)
__device__ __forceinline__ void split2(float x0, float x1, uint32_t& hi, uint32_t& lo) {
    const __half2 h = __floats2half2_rn(x0, x1);
    hi = *reinterpret_cast<const uint32_t*>(&h);
    float l0, l1;
    asm("{\n\t.reg .f16 a, b, m;\n\tmov.b32 {a, b}, %2;\n\tmov.b16 m, 0xBC00;\n\t"
        "fma.rn.f32.f16 %0, a, m, %3;\n\tfma.rn.f32.f16 %1, b, m, %4;\n\t}"
        : "=f"(l0), "=f"(l1) : "r"(hi), "f"(x0), "f"(x1));
    const __half2 l = __floats2half2_rn(l0, l1);
    lo = *reinterpret_cast<const uint32_t*>(&l);
}
__device__ __forceinline__ F2 add2(F2 a, F2 b) {
    F2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.u) : "l"(a.u), "l"(b.u));
    return r;
}

// Where an item's stores go and what they are multiplied with.
struct ZOut {
    uint8_t *hi, *lo;    // this lane's columns in the first row of antenna 0, first instance
    unsigned inst_b;     // bytes of an instance's rows
    const float2* wa;    // this lane's sources, first instance, beam 0
    const float4* ws;    // the same in shared memory (one beam)
    long long wa_slot, wa_pitch;
    float scale;
};

// Two sources (times NAX columns) of one row, hi and lo.
template <int NAX>
__device__ __forceinline__ void put_row(uint8_t* ph, uint8_t* pl, const float (&v)[2 * NAX]) {
    uint32_t h[NAX], l[NAX];
#pragma unroll
    for (int k = 0; k < NAX; ++k) split2(v[2 * k], v[2 * k + 1], h[k], l[k]);
    if constexpr (NAX == 1) {
        *reinterpret_cast<uint32_t*>(ph) = h[0];
        *reinterpret_cast<uint32_t*>(pl) = l[0];
    } else {
        *reinterpret_cast<uint2*>(ph) = make_uint2(h[0], h[1]);
        *reinterpret_cast<uint2*>(pl) = make_uint2(l[0], l[1]);
    }
}

// cos_sin_turns (zcore.cuh) of two phases, as pairs.
__device__ __forceinline__ void cos_sin_turns2(unsigned long long F0, unsigned long long F1, F2& c, F2& s) {
    const unsigned X0 = (unsigned)(F0 >> 32), X1 = (unsigned)(F1 >> 32);
    const unsigned q0 = (X0 + 0x20000000u) >> 30, q1 = (X1 + 0x20000000u) >> 30;
    auto two = [](float v) { return pack2(v, v); };
    const F2 x = mul2(pack2((float)(int)(X0 - (q0 << 30)), (float)(int)(X1 - (q1 << 30))), two(2.3283064365386962890625e-10f));  // 2^-32
    const F2 x2 = mul2(x, x);
    const F2 sp = mul2(fma2(fma2(fma2(two(-75.24006652832031f), x2, two(81.58812713623047f)), x2, two(-41.34162902832031f)), x2,
                            two(6.283185005187988f)), x);
    const F2 cp = fma2(fma2(fma2(fma2(two(59.22040557861328f), x2, two(-85.44285583496094f)), x2, two(64.93931579589844f)), x2,
                            two(-19.739208221435547f)), x2, two(1.0f));
    float s0, s1, c0, c1;
    unpack2(sp, s0, s1);
    unpack2(cp, c0, c1);
    // rotated by q quarter turns
    auto turn = [](unsigned q, float cv, float sv, float& co, float& so) {
        const bool swap = (q & 1u) != 0u;
        const float a = swap ? sv : cv, b = swap ? cv : sv;
        co = __uint_as_float(__float_as_uint(a) ^ (((q + 1u) & 2u) << 30));
        so = __uint_as_float(__float_as_uint(b) ^ ((q & 2u) << 30));
    };
    float co0, co1, so0, so1;
    turn(q0, c0, s0, co0, so0);
    turn(q1, c1, s1, co1, so1);
    c = pack2(co0, co1);
    s = pack2(so0, so1);
}

// The rows of one antenna and instance at hi / lo: WA (A) times the phase (c, s),
// scaled.
template <int FORM, int NAX, int NFD>
__device__ __forceinline__ void z_rows(const float4 (&A)[NFD * NAX], F2 c, F2 s, uint8_t* hi, uint8_t* lo) {
    constexpr int NP = FORM == kZherkReal ? 2 : 3, ROW_B = zherk_row_bytes(NAX);
#pragma unroll
    for (int p = 0; p < NFD; ++p) {
        float re[2 * NAX], im[2 * NAX], sm[2 * NAX];
#pragma unroll
        for (int k = 0; k < NAX; ++k) {
            const float4 a4 = A[p * NAX + k];
            // Z = WA (c - i s): re = x c + y s, im = y c - x s
            const F2 x = pack2(a4.x, a4.y), y = pack2(a4.z, a4.w), nx = pack2(-a4.x, -a4.y);
            const F2 r2 = fma2(x, c, mul2(y, s)), i2 = fma2(y, c, mul2(nx, s));
            unpack2(r2, re[k], re[NAX + k]);
            unpack2(i2, im[k], im[NAX + k]);
            if constexpr (FORM == kZherkGauss) unpack2(add2(r2, i2), sm[k], sm[NAX + k]);
        }
        put_row<NAX>(hi + p * NP * ROW_B, lo + p * NP * ROW_B, re);
        put_row<NAX>(hi + (p * NP + 1) * ROW_B, lo + (p * NP + 1) * ROW_B, im);
        if constexpr (FORM == kZherkGauss) put_row<NAX>(hi + (p * NP + 2) * ROW_B, lo + (p * NP + 2) * ROW_B, sm);
    }
}

// Z of antennas [a0, a1) for a group of one instance, two antennas at a time: each
// phase is a chain of some 60 dependent operations, and with one at a time the
// three Z warps of a scheduler issued in a third of its cycles (48 pairs of 1e5
// sources x 350 antennas: 5.30 ms, 1.80 of them for the phases; 3.62 so).
template <int FORM, int NAX, int NFD, bool ONE>
__device__ __forceinline__ void z_ants_one(const ZherkArgs& P, const ZOut& o, const AntPhase* tab, int a0, int a1,
                                           const unsigned (&S0)[3], const unsigned (&S1)[3], const float (&E0)[3],
                                           const float (&E1)[3]) {
    constexpr int NC = NFD * NAX, NP = FORM == kZherkReal ? 2 : 3, ROW_B = zherk_row_bytes(NAX);
    float4 W[NC];
    if constexpr (ONE) {
#pragma unroll
        for (int c = 0; c < NC; ++c) W[c] = o.ws[c * (kZherkChunk / 2)];
    }
    const F2 scale = pack2(o.scale, o.scale);
#pragma unroll 1
    for (int a = a0; a < a1; a += 2) {
        const int n = min(2, a1 - a);
        F2 c[2], s[2];
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const AntPhase p = tab[a - a0 + (i < n ? i : 0)];
            cos_sin_turns2(phase64(p, S0, E0), phase64(p, S1, E1), c[i], s[i]);
            c[i] = mul2(c[i], scale);
            s[i] = mul2(s[i], scale);
        }
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            if (i >= n) break;
            if constexpr (!ONE) {
                const float2* w = o.wa + (long long)P.m.beam_idx[a + i] * NC * o.wa_pitch;
#pragma unroll
                for (int k = 0; k < NC; ++k) W[k] = *reinterpret_cast<const float4*>(w + (long long)k * o.wa_pitch);
            }
            const unsigned row = (unsigned)((a + i) * NFD * NP) * ROW_B;
            z_rows<FORM, NAX, NFD>(W, c[i], s[i], o.hi + row, o.lo + row);
        }
    }
}

// Z of antenna a for every instance of group g: each lane two adjacent sources.
// tab: the antenna's phase factors (shared memory; kappa0, then dkappa per_e
// entries on).  A row of the ring has a fixed length and an antenna-feed's rows
// (Re, Im and, with the gauss form, their sum) follow each other, so that all
// stores of an instance have fixed offsets from two pointers.  ONE: one beam,
// whose WA is in shared memory.
template <int FORM, int NAX, int NFD, bool ONE>
__device__ __forceinline__ void z_ant(const ZherkArgs& P, const ZherkGroup& g, const ZOut& o, const AntPhase* tab,
                                      int per_e, int a, const unsigned (&S0)[3], const unsigned (&S1)[3],
                                      const float (&E0)[3], const float (&E1)[3]) {
    constexpr int NC = NFD * NAX, NP = FORM == kZherkReal ? 2 : 3, ROW_B = zherk_row_bytes(NAX);
    const float2* w = ONE ? nullptr : o.wa + (long long)P.m.beam_idx[a] * NC * o.wa_pitch;
    const float4* ws = o.ws;
    uint8_t* hi = o.hi + (unsigned)(a * NFD * NP) * ROW_B;
    uint8_t* lo = o.lo + (unsigned)(a * NFD * NP) * ROW_B;
    // WA of the next instance
    auto load_wa = [&](float4 (&A)[NC]) {
        if constexpr (ONE) {
#pragma unroll
            for (int c = 0; c < NC; ++c) A[c] = ws[c * (kZherkChunk / 2)];
            ws += NC * (kZherkChunk / 2);
        } else {
#pragma unroll
            for (int c = 0; c < NC; ++c) A[c] = *reinterpret_cast<const float4*>(w + (long long)c * o.wa_pitch);
            w += o.wa_slot;
        }
    };
    auto emit = [&](const float4 (&A)[NC], F2 c, F2 s) {
        z_rows<FORM, NAX, NFD>(A, c, s, hi, lo);
        hi += o.inst_b;
        lo += o.inst_b;
    };
    const F2 scale = pack2(o.scale, o.scale);
    if (g.uniform && g.n > 1) {
        // equally spaced channels: exact fixed-point phase every kAnchor
        // channels, complex recurrence in between (as zbuild_item)
        const AntPhase p0 = tab[0], pd = tab[per_e];
        unsigned long long F0 = phase64(p0, S0, E0), F1 = phase64(p0, S1, E1);
        const unsigned long long Q0 = phase64(pd, S0, E0), Q1 = phase64(pd, S1, E1);
        F2 rc, rs;
        cos_sin_turns2(Q0, Q1, rc, rs);
        const F2 nrs = mul2(rs, pack2(-1.f, -1.f));
        constexpr int PF = NC == 1 ? 2 : 1;
        for (int left = g.n; left > 0; left -= kAnchor) {
            F2 c, s;
            cos_sin_turns2(F0, F1, c, s);
            c = mul2(c, scale);
            s = mul2(s, scale);
            F0 += Q0 * kAnchor;
            F1 += Q1 * kAnchor;
            auto turn = [&]() {  // (c + i s) e^{2 pi i dF}
                const F2 nc = fma2(c, rc, mul2(s, nrs));
                s = fma2(s, rc, mul2(c, rs));
                c = nc;
            };
            if (left >= kAnchor) {
#pragma unroll
                for (int jb = 0; jb < kAnchor; jb += PF) {
                    float4 B[PF][NC];
#pragma unroll
                    for (int jj = 0; jj < PF; ++jj) load_wa(B[jj]);
#pragma unroll
                    for (int jj = 0; jj < PF; ++jj) {
                        emit(B[jj], c, s);
                        if (jb + jj + 1 < kAnchor) turn();
                    }
                }
            } else {
#pragma unroll 1
                for (int j = 0; j < left; ++j) {
                    float4 B[NC];
                    load_wa(B);
                    emit(B, c, s);
                    turn();
                }
            }
        }
        return;
    }
    // unevenly spaced channels: the phase of each from its own factors, the next
    // channel's on their way from L2 meanwhile (233 antennas, 43,833 sources, 32
    // instances: 987 us with a load at a time, 734 so)
    const AntPhase* t = P.aph + (long long)g.aph * P.n_phase * P.m.n_ant + a;
    AntPhase p = tab[0];
    for (int j = 0; j < g.n; ++j) {
        AntPhase nx = p;
        t += P.m.n_ant;
        if (j + 1 < g.n) nx = load_phase(t);
        float4 A[NC];
        load_wa(A);
        F2 c, s;
        cos_sin_turns2(phase64(p, S0, E0), phase64(p, S1, E1), c, s);
        emit(A, mul2(c, scale), mul2(s, scale));
        p = nx;
    }
}

// The chunks this SM builds in wave w: every teams-th one from `team` on, of
// group gi, antennas from a0 on (team < 0: none).
struct ZShare {
    int teams, team, gi, a0;
};
__device__ __forceinline__ ZShare z_share(const ZherkArgs& P, int w, int ants) {
    const int n_groups = P.wave_items[w], nab = (P.m.n_ant + ants - 1) / ants, per = n_groups * nab;
    ZShare s;
    s.teams = (int)gridDim.x / per;
    s.team = (int)blockIdx.x / per;
    const int r = (int)blockIdx.x - s.team * per;
    s.gi = r / nab;
    s.a0 = (r - s.gi * nab) * ants;
    if (s.team >= s.teams) s.team = -1;
    return s;
}

// -------------------------------------------------------------- kernel
template <int FORM, int NAX, int NFD, bool ONE>
__global__ void __launch_bounds__(threads_for(NAX * NFD), 1)
k_zherk(const __grid_constant__ CUtensorMap map, const __grid_constant__ ZherkArgs P) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    constexpr int Z_WARPS = z_warps(NAX * NFD), NC = NAX * NFD;
    uint8_t* zsm = smem + STAGES * STAGE;      // input buffers, then the Z warps' phase factors
    // barriers: full[STAGES], empty[STAGES], tfull, tempty, zfull, zdone and zfree [MAX_BUF] each
    uint64_t* bars = reinterpret_cast<uint64_t*>(zsm + 2 * Z_BUF + Z_WARPS * Z_APH_B);
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * STAGES + 2 + 3 * MAX_BUF);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
    const uint32_t freed = smem_u32(tmem_slot + 2);   // chunks every SM has loaded, in a row
    const uint32_t landed = smem_u32(tmem_slot + 3);  // chunks of this SM's jobs that have landed
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    auto full = [&](int s) { return smem_u32(&bars[s]); };
    auto empty = [&](int s) { return smem_u32(&bars[STAGES + s]); };
    const uint32_t tfull = smem_u32(&bars[2 * STAGES]), tempty = smem_u32(&bars[2 * STAGES + 1]);
    auto zfull = [&](int b) { return smem_u32(&bars[2 * STAGES + 2 + b]); };
    auto zdone = [&](int b) { return smem_u32(&bars[2 * STAGES + 2 + MAX_BUF + b]); };
    auto zfree = [&](int b) { return smem_u32(&bars[2 * STAGES + 2 + 2 * MAX_BUF + b]); };
    // input k of the Z warps: buffer k & zmask, its barriers' phase
    const int zmask = (1 << P.z_shift) - 1;
    auto zphase = [&](int k) { return (uint32_t)(k >> P.z_shift) & 1u; };
    constexpr int SPC = kZherkChunk * NAX / 32, RC = zherk_ring_chunks(NAX);  // stages per chunk, chunks in the ring

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) { mbar_init(full(s), 1); mbar_init(empty(s), 1); }
        mbar_init(tfull, 1);
        mbar_init(tempty, EPI_WARPS);
        for (int b = 0; b < MAX_BUF; ++b) { mbar_init(zfull(b), 1); mbar_init(zdone(b), Z_WARPS); mbar_init(zfree(b), 1); }
        *abort_flag = 0;
        tmem_slot[2] = tmem_slot[3] = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "r"(TMEM_COLS));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
        tc_fence_before();
    }
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    const uint32_t sbase = smem_u32(smem);
    const ZherkJob& J = P.jobs[blockIdx.x];   // this SM's job, the same in every wave
    const int jn = J.n, pan = P.panel, box_b = pan * 128;
    // whether the job's instance is in wave w
    auto has_job = [&](int w) { return jn > 0 && (w < P.n_waves - 1 || J.v < P.v_last); };

    if (warp >= 2 && warp < 2 + EPI_WARPS) {
        // epilogue: TMEM lane quadrant q4, 128-column half h; FP32 running sums in TMEM
        const int q4 = warp & 3, h = (warp - 2) >> 2;
        const uint32_t tl = tmem_base + ((uint32_t)(q4 * 32) << 16) + (uint32_t)(h * 128);
        const uint32_t trun = tl + RUN_COL;
        int cg = 0;
        bool ok = true;
        for (int w = 0; w < P.n_waves && ok; ++w) {
            if (!has_job(w)) continue;
            const int4 v = P.zv[w * P.V + J.v];
            const int n_flush = (v.w * SPC + P.flush - 1) / P.flush;
            for (int f = 0; f < n_flush; ++f, ++cg) {
                if (!wait_warp(tfull, (uint32_t)cg & 1u, abort_flag, P.err, kTimeoutNs, 300u)) { ok = false; break; }
                tc_fence_after();
                if (h * 128 < jn) {
                    // both loads of a piece go out together; the MMAs wait for this
#pragma unroll
                    for (int g = 0; g < 128 / 16; ++g) {
                        if (h * 128 + g * 16 >= jn) break;
                        uint32_t acc[16];
                        tmem_ld16(tl + g * 16, acc);
                        if (f > 0) {
                            uint32_t sum[16];
                            tmem_ld16(trun + g * 16, sum);
                            tmem_wait_ld16(acc);
                            tmem_wait_ld16(sum);
#pragma unroll
                            for (int i = 0; i < 16; ++i)
                                acc[i] = __float_as_uint(__uint_as_float(sum[i]) + __uint_as_float(acc[i]));
                        } else {
                            tmem_wait_ld16(acc);
                        }
                        tmem_st16(trun + g * 16, acc);
                    }
                    tmem_wait_st();
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(tempty);
            }
            if (!ok || warp_aborted(abort_flag)) break;
            if (h * 128 < jn) {
                // partial tiles, column-major [128][128] (coalesced along rows); the second
                // product's columns follow the first one's panel
                const int ks = (w * P.V + J.v) / P.n_inst, cols = J.np * pan;
                float* const p = P.partial + (long long)v.x * P.n_tiles * P.S * (128 * 128) + (long long)ks * (128 * 128) + q4 * 32 + lane;
                float* const p0 = p + (long long)J.tile[0] * P.S * (128 * 128);
                float* const p1 = p + (long long)J.tile[1] * P.S * (128 * 128) - pan * 128;
#pragma unroll 1
                for (int g = 0; g < 8; ++g) {
                    const int c0 = h * 128 + g * 16;
                    if (c0 >= cols) break;
                    uint32_t sum[16];
                    if (n_flush > 0) {
                        tmem_ld16(trun + g * 16, sum);
                        tmem_wait_ld16(sum);
                    } else {
#pragma unroll
                        for (int i = 0; i < 16; ++i) sum[i] = 0u;
                    }
#pragma unroll
                    for (int i = 0; i < 16; ++i)
                        if (c0 + i < cols) (c0 + i < pan ? p0 : p1)[(c0 + i) * 128] = __uint_as_float(sum[i]);
                }
            }
        }
    } else if (warp == COUNT_WARP) {
        // Count this SM up for every chunk whose items its Z warps have finished (ready)
        // and for every chunk that has landed in it (done).  A warp of its own, as the
        // fence before a count waits for the SM's stores to reach L2: that would hold up
        // a Z warp, and in the TMA warp the loads (350 antennas, 1e5 sources, 256
        // instances: 19.7 ms, 15.7 so).  Landed chunks are counted with a finished one or
        // two at a time, unless no more are to land in this wave (15.6 one at a time or
        // three, 15.5 so; none of those kept back is waited for before the next one lands).
        int wb = -1, q = 0, base = 0, wlen = 0, k = 0;           // the next chunk built
        int wl = -1, lq = 0, lbase = 0, llen = 0, counted = 0;   // the next chunk landed
        ZShare z{1, -1, 0, 0};
        unsigned long long t0 = gtimer();
        for (;;) {
            while (wb < P.n_waves && q >= wlen) {
                if (++wb == P.n_waves) break;
                z = z_share(P, wb, Z_WARPS * P.ant_block);
                base = P.wave_base[wb];
                wlen = z.team < 0 ? 0 : P.wave_base[wb + 1] - base;
                q = z.team < 0 ? 0 : z.team;
            }
            while (wl < P.n_waves && lq >= llen) {
                if (++wl == P.n_waves) break;
                lbase = P.wave_base[wl];
                llen = has_job(wl) ? P.zv[wl * P.V + J.v].w : 0;
                lq = 0;
            }
            if (wb == P.n_waves && wl == P.n_waves) break;
            const bool built = wb < P.n_waves && __all_sync(0xffffffffu, mbar_test(zdone(k & zmask), zphase(k)));
            int land = min(__shfl_sync(0xffffffffu, ld_acquire_cta(landed), 0) - counted, llen - lq);
            if (!built && land < 2 && lq + land < llen) land = 0;
            if (built || land > 0) {
                if (lane == 0) {
                    if (built) mbar_arrive(zfree(k & zmask));  // (seen: the buffer's barrier may start its next phase)
                    fence_release();
                    if (built) red_add(P.ready + base + q, 1);
                    for (int i = 0; i < land; ++i) red_add(P.done + lbase + lq + i, 1);
                }
                __syncwarp();
                if (built) {
                    q += z.teams;
                    ++k;
                }
                lq += land;
                counted += land;
                t0 = gtimer();
            } else {
                if (__any_sync(0xffffffffu, *abort_flag || gtimer() - t0 > 2 * kTimeoutNs)) break;
                __nanosleep(20);
            }
        }
    } else if (warp == FEED_WARP) {
        // Feed the Z warps: each chunk's directions and (one beam) WA into the next
        // buffer.  And watch the next 32 chunks' done counts and tell the Z warps
        // through shared memory how far the ring is free (one poller per SM).
        const int last_base = P.wave_base[P.n_waves - 1], total = P.wave_base[P.n_waves];
        int next = 0, k = 0, w = -1, q = 0, base = 0, wlen = 0;
        ZShare z{1, -1, 0, 0};
        const ZherkGroup* g = nullptr;
        bool more = true;
        unsigned long long t0 = gtimer();
        while (more || next < total - RC) {
            bool any = false;
            int d = 0;
            const int c = next + lane;
            const bool look = next < total - RC && c < total;
            if (look) d = ld_relaxed(P.done + c);
            // (as many buffers as are free but for one: a look takes as long as a short chunk;
            // 12 antennas x 84 pairs x 70,000 sources 657 us with one a look, 600 so)
            for (int fed = 0; fed < zmask; ++fed) {
                while (more && q >= wlen) {  // the next wave this SM builds for
                    if (++w >= P.n_waves) {
                        more = false;
                        break;
                    }
                    z = z_share(P, w, Z_WARPS * P.ant_block);
                    base = P.wave_base[w];
                    wlen = z.team < 0 ? 0 : P.wave_base[w + 1] - base;
                    q = z.team < 0 ? 0 : z.team;
                    if (z.team >= 0) g = P.groups + P.wave_group0[w] + z.gi;
                }
                if (!more || !(k <= zmask || __all_sync(0xffffffffu, mbar_test(zfree(k & zmask), zphase(k) ^ 1u)))) break;
                any = true;
                const uint32_t bar = zfull(k & zmask), dst = smem_u32(zsm + (k & zmask) * P.z_buf_b);
                if (q < g->len) {
                    const int n = ONE ? g->n * NC : 0, src = (g->c0 + q) * kZherkChunk;
                    if (lane == 0) mbar_expect_tx(bar, (uint32_t)(Z_SRC_B + n * kZherkChunk * 8));
                    __syncwarp();
                    if (lane < 6) {
                        const long long o = ((long long)g->t * 3 + (lane < 3 ? lane : lane - 3)) * P.lt.pitch + src;
                        bulk_load(dst + lane * (kZherkChunk * 4), lane < 3 ? (const void*)(P.lt.sfix + o) : (const void*)(P.lt.seps + o),
                                  kZherkChunk * 4, bar);
                    }
                    if (lane < n)  // (one beam: the components of successive slots follow each other)
                        bulk_load(dst + Z_SRC_B + lane * (kZherkChunk * 8), P.wa + ((long long)g->slot * NC + lane) * P.wa_pitch + src,
                                  kZherkChunk * 8, bar);
                } else if (lane == 0) {
                    mbar_arrive(bar);
                }
                __syncwarp();
                q += z.teams;
                ++k;
            }
            if (next < total - RC) {
                const unsigned m = __ballot_sync(0xffffffffu, look && d >= (c >= last_base ? P.n_jobs_last : P.n_jobs));
                const int adv = m == 0xffffffffu ? 32 : __ffs(~(int)m) - 1;  // chunks done in a row
                if (adv > 0) {
                    any = true;
                    next += adv;
                    if (lane < adv) ld_acquire(P.done + c);
                    __syncwarp();  // (what the lanes acquired comes before the release)
                    if (lane == 0) st_release_cta(freed, next);
                }
            }
            if (any) {
                t0 = gtimer();
            } else {
                if (__any_sync(0xffffffffu, *abort_flag || gtimer() - t0 > 2 * kTimeoutNs)) break;
                __nanosleep(20);
            }
        }
    } else {
        if (warp == 0) {
            // The whole warp looks at the next 32 chunks' ready counts with one load, and one
            // lane issues the copies.  While it waits it tells COUNT_WARP of the chunks that
            // have landed in this SM, ahead of their MMAs, so that their place in the ring
            // is free about two chunks earlier.
            int it = 0, seen = 0, li = 0, chunks = 0;  // stages issued, stages seen landed, chunks of them
            bool ok = true;
            const int nbox = J.nbox, jv = J.v;
            for (int w = 0; w < P.n_waves && ok; ++w) {
                if (!has_job(w)) continue;
                const int len = P.zv[w * P.V + jv].w;
                const int base = P.wave_base[w], wlen = P.wave_base[w + 1] - base;
                const int items = P.wave_items[w] * ((P.m.n_ant + Z_WARPS * P.ant_block - 1) / (Z_WARPS * P.ant_block));
                if (lane == 0)  // (chunks past this job's sources: never read, nothing to order)
                    for (int q = len; q < wlen; ++q) red_add(P.done + base + q, 1);
                int y[MAX_BOX], pl[MAX_BOX];
#pragma unroll
                for (int b = 0; b < MAX_BOX; ++b) {
                    y[b] = jv * P.map_rows + J.row[b];
                    pl[b] = J.plane[b];
                }
                auto land = [&]() {
                    if (seen >= it) return false;
                    if (!__all_sync(0xffffffffu, mbar_test(full(seen % STAGES), (uint32_t)(seen / STAGES) & 1u))) return false;
                    ++seen;
                    if (++li == SPC) {
                        li = 0;
                        ++chunks;
                        __syncwarp();
                        if (lane == 0) st_release_cta(landed, chunks);
                    }
                    return true;
                };
                // spin on `ready` (warp-uniform) with the landings in between; false on a timeout
                auto wait_for = [&](auto ready) {
                    unsigned long long t0 = 0;
                    for (unsigned n = 0; !ready(); ++n) {
                        if (land()) continue;
                        if ((n & 15u) == 15u) {  // (the clock is read now and then)
                            const unsigned long long t = gtimer();
                            if (t0 == 0) t0 = t;
                            const bool late = t - t0 > kTimeoutNs;
                            if (late && lane == 0) {
                                *abort_flag = 1;
                                atomicCAS(P.err, 0, (int)kDevTimeout);
                            }
                            if (__any_sync(0xffffffffu, late || *abort_flag)) return false;
                        }
                    }
                    return true;
                };
                int have = 0;  // chunks of the wave known to be ready
                for (int q = 0; q < len && ok; ++q) {
                    if (q >= have) {
                        ok = wait_for([&]() {
                            const int c = q + lane;
                            const int r = c < len ? ld_relaxed(P.ready + base + c) : 0;
                            const unsigned m = __ballot_sync(0xffffffffu, r >= items);
                            have = q + (m == 0xffffffffu ? 32 : __ffs(~(int)m) - 1);
                            return have > q;
                        });
                        if (!ok) break;
                        // the items' stores were released before they were counted: the lanes
                        // acquire the counts they saw, and the elected lane's copies follow
                        if (q + lane < have) ld_acquire(P.ready + base + q + lane);
                        __syncwarp();
                        asm volatile("fence.proxy.async.global;" ::: "memory");
                    }
                    const int x0 = ((base + q) % RC) * SPC * 64;
#pragma unroll
                    for (int i = 0; i < SPC; ++i) {
                        const int s = it % STAGES;
                        const uint32_t ph = ((uint32_t)(it / STAGES) & 1u) ^ 1u;
                        ok = wait_for([&]() { return __all_sync(0xffffffffu, mbar_test(empty(s), ph)) != 0; });
                        if (!ok) break;
                        while (seen <= it - STAGES && land()) {}  // (the stage was consumed, so it has landed)
                        if (elect_one()) {
                            mbar_expect_tx(full(s), (uint32_t)(nbox * box_b));
#pragma unroll
                            for (int b = 0; b < MAX_BOX; ++b)
                                if (b < nbox) tma_load_3d(sbase + s * STAGE + b * box_b, &map, x0 + i * 64, pl[b], y[b], full(s));
                        }
                        __syncwarp();
                        ++it;
                    }
                }
                if (ok) ok = wait_for([&]() { return seen >= it; });
            }
        } else if (warp == 1) {
            // MMA: the whole warp walks the loop (so that descriptors and barriers stay
            // in uniform registers), one elected lane issues.  With a single-lane loop an
            // MMA took 72-83 cycles to issue, more than the 64 of an N = 128 one.
            int it = 0, cg = 0;
            bool ok = true;
            const uint64_t da = sdesc(sbase + J.a * box_b), db = sdesc(sbase + J.b * box_b);
            const uint32_t id = idesc_f16(true, 128, 0) + ((uint32_t)(jn >> 3) << 17);
            const int jv = J.v, flush = P.flush;
            for (int w = 0; w < P.n_waves && ok; ++w) {
                if (!has_job(w)) continue;
                const int len = P.zv[w * P.V + jv].w;
                int ls = 0;
                const uint32_t d = tmem_base;
                for (int q = 0; q < len && ok; ++q) {
#pragma unroll
                    for (int i = 0; i < SPC; ++i) {
                        if (ls == 0) {  // the epilogue has drained the accumulator
                            ok = wait_warp_spin(tempty, ((uint32_t)cg & 1u) ^ 1u, abort_flag, P.err);
                            tc_fence_after();
                        }
                        const int s = it % STAGES;
                        ok = ok && wait_warp(full(s), (uint32_t)(it / STAGES) & 1u, abort_flag, P.err);
                        if (!ok) break;
                        tc_fence_after();
                        const uint32_t so = (uint32_t)s * (STAGE >> 4);
                        const bool last = ls + 1 == flush || (q == len - 1 && i == SPC - 1);
                        if (elect_one()) {
#pragma unroll
                            for (int kk = 0; kk < 2; ++kk) {
                                // even blocks hold hi then lo, odd ones lo then hi
                                const uint32_t oh = so + (i & 1 ? 4 : 0) + 2 * kk, ol = so + (i & 1 ? 0 : 4) + 2 * kk;
                                const uint64_t ah = da + oh, al = da + ol, bh = db + oh, bl = db + ol;
                                tc_mma_shared_a<true>(d, ah, bh, id, kk > 0 || ls > 0 ? 1u : 0u);
                                tc_mma_shared_a<false>(d, ah, bl, id, 1);
                                tc_mma(d, al, bh, id, 1);
                            }
                            tc_commit(empty(s));
                            if (last) tc_commit(tfull);
                        }
                        __syncwarp();
                        ++it;
                        if (last) {
                            ++cg;
                            ls = 0;
                        } else {
                            ++ls;
                        }
                    }
                }
            }
        } else {
            // Z build
            const int zi = warp - FIRST_Z;
            AntPhase* const tab = reinterpret_cast<AntPhase*>(zsm + 2 * Z_BUF + zi * Z_APH_B);
            ZOut o;
            o.inst_b = (unsigned)(P.rows * zherk_row_bytes(NAX));
            o.wa_pitch = P.wa_pitch;
            o.wa_slot = (long long)P.m.n_beam * NC * P.wa_pitch;
            // this lane's columns: even blocks of 32 hold hi then lo, odd ones lo then hi,
            // so that the half warps of a store meet different banks
            const int col = 2 * lane * NAX;
            const unsigned blk_b = (unsigned)((col >> 5) * 128 + (col & 31) * 2);
            const unsigned hi_b = blk_b + ((col >> 5) & 1) * 64, lo_b = blk_b + (((col >> 5) & 1) ^ 1) * 64;
            int k = 0;
            bool ok = true;
            for (int w = 0; w < P.n_waves && ok; ++w) {
                const ZShare z = z_share(P, w, Z_WARPS * P.ant_block);
                if (z.team < 0) continue;
                const int base = P.wave_base[w], wlen = P.wave_base[w + 1] - base;
                const ZherkGroup g = P.groups[P.wave_group0[w] + z.gi];
                const int a0 = z.a0 + zi * P.ant_block, a1 = min(P.m.n_ant, a0 + P.ant_block);
                o.scale = P.scale[g.slot];
                const int per_e = g.uniform && g.n > 1 ? Z_BLOCK / 2 : Z_BLOCK;
                __syncwarp();
                {   // the antennas' phase factors, once per wave
                    const AntPhase* t = P.aph + (long long)g.aph * P.n_phase * P.m.n_ant + a0;
                    const int n16 = (a1 - a0) * 3;
                    for (int i = lane; i < n16; i += 32) cp_async16(smem_u32(tab) + i * 16, (const uint4*)t + i);
                    if (per_e < Z_BLOCK)
                        for (int i = lane; i < n16; i += 32)
                            cp_async16(smem_u32(tab + per_e) + i * 16, (const uint4*)(t + P.m.n_ant) + i);
                }
                asm volatile("cp.async.commit_group;" ::: "memory");
                asm volatile("cp.async.wait_group 0;" ::: "memory");
                __syncwarp();
                for (int q = z.team; q < wlen; q += z.teams, ++k) {
                    const int cq = base + q;
                    ok = wait_warp(zfull(k & zmask), zphase(k), abort_flag, P.err);
                    // the chunk whose place in the ring this one takes has been read by all
                    auto room = [&]() { return __all_sync(0xffffffffu, ld_acquire_cta(freed) > cq - RC) != 0; };
                    if (!room()) {
                        const unsigned long long t0 = gtimer();
                        while (!room()) {
                            __nanosleep(20);
                            const bool late = gtimer() - t0 > kTimeoutNs;
                            if (late && lane == 0) {
                                *abort_flag = 1;
                                atomicCAS(P.err, 0, (int)kDevTimeout);
                            }
                            if (__any_sync(0xffffffffu, *abort_flag || late)) { ok = false; break; }
                        }
                    }
                    if (!ok) break;
                    if (q < g.len && a0 < a1) {
                        const uint8_t* sm = zsm + (k & zmask) * P.z_buf_b;
                        unsigned S0[3], S1[3];
                        float E0[3], E1[3];
#pragma unroll
                        for (int c = 0; c < 3; ++c) {
                            const uint2 qv = *reinterpret_cast<const uint2*>(sm + c * (kZherkChunk * 4) + lane * 8);
                            const float2 r2 = *reinterpret_cast<const float2*>(sm + (3 + c) * (kZherkChunk * 4) + lane * 8);
                            S0[c] = qv.x; S1[c] = qv.y;
                            E0[c] = r2.x; E1[c] = r2.y;
                        }
                        uint8_t* at = P.ring + (unsigned long long)(unsigned)g.v0 * o.inst_b + (unsigned)((cq % RC) * (kZherkChunk * NAX * 4));
                        o.hi = at + hi_b;
                        o.lo = at + lo_b;
                        o.wa = P.wa + (long long)g.slot * o.wa_slot + (g.c0 + q) * kZherkChunk + 2 * lane;
                        o.ws = reinterpret_cast<const float4*>(sm + Z_SRC_B) + lane;
                        if (g.n == 1) {
                            z_ants_one<FORM, NAX, NFD, ONE>(P, o, tab, a0, a1, S0, S1, E0, E1);
                        } else {
                            for (int a = a0; a < a1; ++a)
                                z_ant<FORM, NAX, NFD, ONE>(P, g, o, tab + (a - a0), per_e, a, S0, S1, E0, E1);
                        }
                    }
                    __syncwarp();
                    if (lane == 0) mbar_arrive(zdone(k & zmask));
                }
            }
            __syncwarp();
        }
    }
    __syncthreads();
    if (*abort_flag) {
        // let copies and MMAs already issued land before TMEM and smem go away
        const unsigned long long t0 = gtimer();
        while (gtimer() - t0 < 2000000ull) {}
    }
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(TMEM_COLS));
    }
}

// How the |WA| of an instance is brought into FP16's range: 2^all, from the largest
// |WA| among the instances of its time (mx), which takes that to 2^13 .. 2^14, and
// where that leaves the instance's own largest below 2^6 as many times 2^8 more as
// take it to 2^6 .. 2^14, so that a rounding of FP16's smallest numbers (2^-25) stays
// below 2^-31 of it.  2^all goes into the Z build's cosines and sines, where it costs
// nothing and the channels of a group have to share it; 2^more into WA itself, as
// channels of one beam seldom differ by 2^8 (in the Z build the redundant cover took
// 4 % longer by it, unevenly spaced channels 4 to 7 %).
__device__ __forceinline__ void fp16_exponents(float mx, float own, int& all, int& more) {
    all = fp16_scale_exp(mx);
    more = own > 0.f && own < 3.0e38f ? max(fp16_scale_exp(own) - all, 0) / 8 * 8 : 0;
}

// WA of an instance times 2^more: blocks 1 on of the launch below, `per` to an
// instance.
__device__ void rescale_wa(const ZherkArgs& P, const float* __restrict__ amax, int slot, int part, int per) {
    __shared__ int mx;
    if (threadIdx.x == 0) mx = 0;
    __syncthreads();
    const int t = P.inst[P.inst0 + slot].t;
    for (int j = threadIdx.x; j < P.n_inst; j += blockDim.x) {
        const float a = amax[j];
        if (P.inst[P.inst0 + j].t == t && a > 0.f && a < 3.0e38f) atomicMax(&mx, __float_as_int(a));
    }
    __syncthreads();
    int all, more;
    fp16_exponents(__int_as_float(mx), amax[slot], all, more);
    if (more == 0) return;
    const float f = ldexpf(1.f, more / 2);  // (twice: 2^more itself may be no FP32 number)
    const int rows = P.m.n_beam * P.m.n_feed * P.m.n_ax;
    const int cols = (P.lt.n_live[t] + 1) / 2;  // source pairs
    float4* w = reinterpret_cast<float4*>(const_cast<float2*>(P.wa) + (long long)slot * rows * P.wa_pitch);
    for (int r = 0; r < rows; ++r, w += P.wa_pitch / 2)
        for (int i = part * blockDim.x + threadIdx.x; i < cols; i += per * blockDim.x) {
            const float4 v = w[i];
            w[i] = make_float4(v.x * f * f, v.y * f * f, v.z * f * f, v.w * f * f);
        }
}

// Per launch: the order of the instances (by_length: by decreasing live count),
// the FP16 scale of every instance (that of the Z build, then that of V), the
// source range of every virtual instance and group, and the chunk ranges of the
// waves.
__global__ void __launch_bounds__(1024) k_zherk_prep(ZherkArgs P, const float* __restrict__ amax, int per,
                                                     float* __restrict__ scale, int4* __restrict__ zv, int* __restrict__ wave_base,
                                                     ZherkGroup* __restrict__ groups, int n_groups, int by_length,
                                                     long long n_counters) {
    kernel_chain();
    if (blockIdx.x > 0) {
        rescale_wa(P, amax, ((int)blockIdx.x - 1) / per, ((int)blockIdx.x - 1) % per, per);
        return;
    }
    for (long long i = threadIdx.x; i < n_counters; i += blockDim.x) P.ready[i] = 0;  // (ready, then done)
    extern __shared__ int sm[];  // t, live count and max |WA| of each instance, then the waves' lengths
    int *st = sm, *sk = sm + P.n_inst, *order = sm + 3 * P.n_inst, *len = sm + 4 * P.n_inst;
    float* sa = reinterpret_cast<float*>(sm + 2 * P.n_inst);
    for (int w = threadIdx.x; w < P.n_waves; w += blockDim.x) len[w] = 0;
    for (int i = threadIdx.x; i < P.n_inst; i += blockDim.x) {
        st[i] = P.inst[P.inst0 + i].t;
        sk[i] = P.lt.n_live[st[i]];
        sa[i] = amax[i];
    }
    __syncthreads();
    for (int i = threadIdx.x; i < P.n_inst; i += blockDim.x) {
        const int ti = st[i], ki = sk[i];
        int rank = 0;
        float mx = 0.f;
        for (int j = 0; j < P.n_inst; ++j) {
            rank += (sk[j] > ki) || (sk[j] == ki && j < i);
            if (st[j] == ti && sa[j] < 3.0e38f) mx = fmaxf(mx, sa[j]);
        }
        if (by_length) order[rank] = i;
        else order[i] = i;
        int all, more;
        fp16_exponents(mx, sa[i], all, more);
        scale[i] = ldexpf(1.f, all);
        scale[P.n_inst + i] = ldexpf(1.f, all + more);
    }
    __syncthreads();
    const int total = P.n_inst * P.S;
    for (int vi = threadIdx.x; vi < total; vi += blockDim.x) {
        const int ks = vi / P.n_inst, slot = order[vi - ks * P.n_inst];
        const int nch = (sk[slot] + kZherkChunk - 1) / kZherkChunk;
        const int c0 = (int)((long long)nch * ks / P.S), c1 = (int)((long long)nch * (ks + 1) / P.S);
        zv[vi] = make_int4(slot, st[slot], c0, c1 - c0);
        atomicMax(&len[vi / P.V], c1 - c0);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < n_groups; i += blockDim.x) {
        ZherkGroup g = groups[i];
        const int4 v = zv[g.vi];
        g.slot = v.x;
        g.t = v.y;
        g.c0 = v.z;
        g.len = v.w;
        if (by_length) g.aph = v.x;
        groups[i] = g;
    }
    if (threadIdx.x == 0) {
        int acc = 0;
        for (int w = 0; w < P.n_waves; ++w) {
            wave_base[w] = acc;
            acc += len[w];
        }
        wave_base[P.n_waves] = acc;
    }
}

// Rows [r, r + 4) of column c of the sum of the S partial tiles at p (128 x
// 128 floats each): what bounds the sums is the loads' latency, so eight go out
// together (one instance in 64 ranges: 32 us with 64 x 64 pieces and a load at a
// time, 6 us with 32 x 32 pieces of four rows a thread).
__device__ __forceinline__ float4 sum_parts(const float* p, int S, int r, int c) {
    const float4* q = reinterpret_cast<const float4*>(p + c * 128 + r);
    float4 v = *q;
#pragma unroll 8
    for (int k = 1; k < S; ++k) {
        const float4 x = q[(long long)k * (128 * 128 / 4)];
        v.x += x.x;
        v.y += x.y;
        v.z += x.z;
        v.w += x.w;
    }
    return v;
}

// V from the partial tiles of the real form: one block per 32 x 32 piece of a
// tile (16 x 16 antenna-feeds), read along the tile's rows and written along
// the rows of V through shared memory.
__global__ void __launch_bounds__(256) k_zherk_final_real(ZherkFinalArgs a) {
    kernel_chain();
    __shared__ float G[32][33];  // [column][row]
    const int slot = blockIdx.x / a.n_tiles, tile = blockIdx.x - slot * a.n_tiles;
    const ZherkTile t = a.tiles[tile];
    const int br = (blockIdx.y & 3) * 32, bc = (blockIdx.y >> 2) * 32;
    const float* p = a.partial + ((long long)slot * a.n_tiles + tile) * a.S * (128 * 128);
    // the product's rows and columns this piece stands for
    const int pr = t.r0 + (t.trans ? bc : br), pc = t.c0 + (t.trans ? br : bc);
    int rlim = min(2 * a.N, t.r0 + a.panel), clim = min(2 * a.N, t.c0 + a.panel);
    if (a.limits) {
        rlim = min(rlim, a.limits[tile].x);
        clim = min(clim, a.limits[tile].y);
    }
    if (pr >= rlim || pc >= clim || (!a.ho.uidx && pr + 31 < pc)) return;
    {
        const int r = (threadIdx.x & 7) * 4, c = threadIdx.x >> 3;
        const float4 v = sum_parts(p, a.S, br + r, bc + c);
        G[c][r] = v.x;
        G[c][r + 1] = v.y;
        G[c][r + 2] = v.z;
        G[c][r + 3] = v.w;
    }
    __syncthreads();
    const float us = a.scale ? 1.f / a.scale[slot] : 1.f;
    float2* Vb = a.V + a.inst[a.inst0 + slot].v_off;
    auto entry = [&](int i, int j) {  // product entry (row, column) of the piece
        return t.trans ? G[i][j] : G[j][i];
    };
    const bool diag = t.r0 == t.c0;
    const int x = threadIdx.x & 15, y = threadIdx.x >> 4;
    for (int pass = 0; pass < (a.ho.uidx ? 1 : 2); ++pass) {
        // pass 0: along the rows of V; pass 1: the mirror image, along its rows
        const int ia = pass ? x : y, ib = pass ? y : x;
        const int A = (pr >> 1) + ia, B = (pc >> 1) + ib;
        if (2 * A >= rlim || 2 * B >= clim) continue;
        const float g00 = entry(2 * ia, 2 * ib), g01 = entry(2 * ia, 2 * ib + 1);
        const float g10 = entry(2 * ia + 1, 2 * ib), g11 = entry(2 * ia + 1, 2 * ib + 1);
        const float re = ((g00 + g11) * us) * us;
        const float im = A == B ? 0.f : ((g10 - g01) * us) * us;
        if (a.ho.uidx) {
            const int nf = a.ho.n_feed;
            const int aa = A / nf, pa = A - aa * nf, bb = B / nf, pb = B - bb * nf;
            const int e = a.ho.uidx[aa * a.ho.n_ant + bb];
            if (e < 0) continue;
            const int grp = e >> 1;
            const bool cj = (e & 1) != 0;
            Vb[((long long)grp * nf + (cj ? pb : pa)) * nf + (cj ? pa : pb)] = make_float2(re, cj ? -im : im);
            continue;
        }
        if (diag && A < B) continue;  // a diagonal tile's upper half is the mirror
        if (pass == 0) Vb[(long long)A * a.N + B] = make_float2(re, im);
        else if (A != B) Vb[(long long)B * a.N + A] = make_float2(re, -im);
    }
}

// V from the partial tiles of the gauss form: one block per 32 x 32 piece of a
// block of panels (i, j), i >= j, of V.
__global__ void __launch_bounds__(256) k_zherk_final_gauss(ZherkFinalArgs a) {
    kernel_chain();
    __shared__ float M[3][32][33];  // F_ab, F_ba, H_ab at [row of a][row of b]
    const int nb = a.np * (a.np + 1) / 2;
    const int slot = blockIdx.x / nb;
    int i = 0, j = blockIdx.x - slot * nb;
    while (j > i) j -= ++i;
    const int ar = (blockIdx.y & 3) * 32, bc = (blockIdx.y >> 2) * 32;
    const int A0 = i * a.panel + ar, B0 = j * a.panel + bc;
    const int A1 = min(a.N, (i + 1) * a.panel), B1 = min(a.N, (j + 1) * a.panel);
    if (A0 >= A1 || B0 >= B1 || A0 + 31 < B0) return;
    const float* base = a.partial + (long long)slot * a.n_tiles * a.S * (128 * 128);
#pragma unroll
    for (int m = 0; m < 3; ++m) {
        const int tile = m == 0 ? a.tile_of[i * a.np + j] : m == 1 ? a.tile_of[j * a.np + i] : a.tile_of[(a.np + i) * a.np + j];
        const ZherkTile t = a.tiles[tile];
        const float* p = base + (long long)tile * a.S * (128 * 128);
        // the tile's rows run along a (M = F_ab, H_ab) unless it is F_ba or transposed
        const bool row_is_a = (m != 1) == (t.trans == 0);
        const int r = (threadIdx.x & 7) * 4, c = threadIdx.x >> 3;
        const float4 v = row_is_a ? sum_parts(p, a.S, ar + r, bc + c) : sum_parts(p, a.S, bc + r, ar + c);
        const float f[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            if (row_is_a) M[m][r + k][c] = f[k];
            else M[m][c][r + k] = f[k];
        }
    }
    __syncthreads();
    const float us = a.scale ? 1.f / a.scale[slot] : 1.f;
    float2* Vb = a.V + a.inst[a.inst0 + slot].v_off;
    for (int pass = 0; pass < 2; ++pass)
        for (int k = threadIdx.x; k < 32 * 32; k += 256) {
            const int x = k & 31, y = k >> 5;
            const int ia = pass ? x : y, ib = pass ? y : x;
            const int A = A0 + ia, B = B0 + ib;
            if (A >= A1 || B >= B1 || A < B) continue;
            const float f = M[0][ia][ib], ft = M[1][ia][ib];
            const float re = ((M[2][ia][ib] - (f + ft)) * us) * us;
            const float im = A == B ? 0.f : ((ft - f) * us) * us;
            if (pass == 0) Vb[(long long)A * a.N + B] = make_float2(re, im);
            else if (A != B) Vb[(long long)B * a.N + A] = make_float2(re, -im);
        }
}

// The ring as [rows][planes][columns]: one plane of 2N-row instances (real), or
// the planes X, Y and S of every antenna-feed (gauss).
bool ring_map(CUtensorMap* map, const void* ring, int row_b, int planes, long long rows, int panel) {
    EncodeTiledFn enc = get_encode();
    if (!enc) return false;
    cuuint64_t dims[3] = {(cuuint64_t)row_b / 2, (cuuint64_t)planes, (cuuint64_t)rows};
    cuuint64_t strides[2] = {(cuuint64_t)row_b, (cuuint64_t)row_b * planes};
    cuuint32_t box[3] = {64, 1, (cuuint32_t)panel};
    cuuint32_t estr[3] = {1, 1, 1};
    return enc(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 3, const_cast<void*>(ring), dims, strides, box, estr,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace

cudaError_t zherk_init() {
    cudaError_t e = cudaSuccess;
    auto set = [&](auto* k, int nc) {
        if (e == cudaSuccess) e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_for(nc));
    };
#define MV_SET(F, A, D) set(k_zherk<F, A, D, false>, A * D), set(k_zherk<F, A, D, true>, A * D)
    MV_SET(kZherkReal, 1, 1);
    MV_SET(kZherkReal, 1, 2);
    MV_SET(kZherkReal, 2, 1);
    MV_SET(kZherkReal, 2, 2);
    MV_SET(kZherkGauss, 1, 1);
    MV_SET(kZherkGauss, 1, 2);
    MV_SET(kZherkGauss, 2, 1);
    MV_SET(kZherkGauss, 2, 2);
#undef MV_SET
    return e;
}

cudaError_t launch_zherk_prep(const ZherkArgs& P, const float* amax, int n_sms, float* scale, int4* zv,
                              int* wave_base, ZherkGroup* groups, int n_groups, bool by_length, long long n_counters,
                              cudaStream_t st, long long* launches) {
    *launches += 1;
    // blocks for rescale_wa: one to 8192 source pairs of an instance as long as that is
    // one an SM (one instance, or one of every time, is its time's largest: none)
    const long long pairs = P.wa_pitch / 2 * P.m.n_beam * P.m.n_feed * P.m.n_ax;
    const int per = (int)std::max(1ll, std::min<long long>((pairs + 8191) / 8192, n_sms / P.n_inst));
    const unsigned blocks = P.n_inst == 1 || by_length ? 1u : 1u + (unsigned)(P.n_inst * per);
    return launch_chained(k_zherk_prep, dim3(blocks), dim3(1024), sizeof(int) * (size_t)(P.n_waves + 4 * P.n_inst), st, P, amax,
                          per, scale, zv, wave_base, groups, n_groups, (int)by_length, n_counters);
}

int zherk_input_bytes(int chan, int nc, int n_beam) { return Z_SRC_B + (n_beam == 1 ? chan * nc * kZherkChunk * 8 : 0); }
int zherk_input_shift(int bytes) { return bytes * 8 <= 2 * Z_BUF ? 3 : bytes * 4 <= 2 * Z_BUF ? 2 : 1; }

cudaError_t launch_zherk(const ZherkArgs& P, int form, int n_ctas, cudaStream_t st, long long* launches) {
    CUtensorMap map;
    if (!ring_map(&map, P.ring, zherk_row_bytes(P.m.n_ax), P.rows / P.map_rows, (long long)P.V * P.map_rows, P.panel))
        return cudaErrorInvalidValue;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)n_ctas);
    const int nc = P.m.n_ax * P.m.n_feed;
    cfg.blockDim = dim3((unsigned)threads_for(nc));
    cfg.dynamicSmemBytes = (size_t)smem_for(nc);
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    *launches += 1;
#define MV_ZK(F, A, D)                                                                       \
    if (form == F && P.m.n_ax == A && P.m.n_feed == D)                                       \
        return P.m.n_beam == 1 ? cudaLaunchKernelEx(&cfg, k_zherk<F, A, D, true>, map, P)    \
                               : cudaLaunchKernelEx(&cfg, k_zherk<F, A, D, false>, map, P)
    MV_ZK(kZherkReal, 1, 1);
    MV_ZK(kZherkReal, 1, 2);
    MV_ZK(kZherkReal, 2, 1);
    MV_ZK(kZherkReal, 2, 2);
    MV_ZK(kZherkGauss, 1, 1);
    MV_ZK(kZherkGauss, 1, 2);
    MV_ZK(kZherkGauss, 2, 1);
    MV_ZK(kZherkGauss, 2, 2);
#undef MV_ZK
    return cudaErrorInvalidValue;
}

cudaError_t launch_zherk_final(const ZherkFinalArgs& a, int form, cudaStream_t st, long long* launches) {
    *launches += 1;
    if (form == kZherkReal)
        return launch_chained(k_zherk_final_real, dim3((unsigned)(a.n_inst * a.n_tiles), 16), dim3(256), 0, st, a);
    return launch_chained(k_zherk_final_gauss, dim3((unsigned)(a.n_inst * (a.np * (a.np + 1) / 2)), 16), dim3(256), 0, st, a);
}

// ------------------------------------------------------------ host planning
int zherk_panel(int rows) {
    const int np = (rows + 127) / 128;
    return ((rows + np - 1) / np + 7) / 8 * 8;
}

std::vector<ZherkTile> zherk_triangle(int rows, int panel) {
    std::vector<ZherkTile> t;
    for (int r = 0; r < rows; r += panel)
        for (int k = 0; k <= r; k += panel) t.push_back(ZherkTile{r, k, r, k, 0, 0});
    return t;
}

std::vector<ZherkTile> zherk_gauss_tiles(int N, int panel) {
    std::vector<ZherkTile> t;
    for (int i = 0; i < N; i += panel)
        for (int j = 0; j < N; j += panel) t.push_back(ZherkTile{i, N + j, i, j, 0, 0});
    for (int i = 0; i < N; i += panel)
        for (int j = 0; j <= i; j += panel) t.push_back(ZherkTile{2 * N + i, 2 * N + j, i, j, 1, 0});
    return t;
}

namespace {

// Pair up products that share a panel: that panel is A, the other two B (N =
// 256).  The products are edges between panels (loops on the diagonal); in a
// depth-first walk every vertex pairs the edges it has not handed on and gives
// an odd one the edge to its parent, so at most one product per connected
// component stays alone.
void make_jobs(std::vector<ZherkTile>& tiles, int plane_rows, int panel, std::vector<ZherkJob>& out) {
    std::vector<int> rows;  // vertices: first rows of panels
    auto vertex = [&](int row) {
        for (size_t i = 0; i < rows.size(); ++i)
            if (rows[i] == row) return (int)i;
        rows.push_back(row);
        return (int)rows.size() - 1;
    };
    const int T = (int)tiles.size();
    std::vector<int> u(T), v(T);
    for (int i = 0; i < T; ++i) {
        u[i] = vertex(tiles[i].ra);
        v[i] = vertex(tiles[i].rb);
    }
    const int n = (int)rows.size();
    std::vector<std::vector<int>> inc(n);
    for (int i = 0; i < T; ++i) {
        inc[u[i]].push_back(i);
        if (v[i] != u[i]) inc[v[i]].push_back(i);
    }
    std::vector<char> seen(n, 0), used(T, 0);
    auto emit = [&](int at, int e0, int e1) {  // products e0 and e1 (or -1) with A = panel `at`
        ZherkJob J{};
        auto box = [&](int row) {
            J.row[J.nbox] = row % plane_rows;
            J.plane[J.nbox] = row / plane_rows;
            return J.nbox++;
        };
        auto other = [&](int e) {  // the B panel of product e; turns it round if A was its B
            if (u[e] != at) {
                std::swap(tiles[e].ra, tiles[e].rb);
                std::swap(u[e], v[e]);
                tiles[e].trans = 1;
            }
            used[e] = 1;
            return v[e];
        };
        const int b0 = other(e0), b1 = e1 >= 0 ? other(e1) : -1;
        J.b = box(rows[b0]);
        J.tile[0] = e0;
        J.np = 1;
        J.n = (panel + 15) / 16 * 16;
        if (b1 >= 0) {
            box(rows[b1]);
            J.tile[1] = e1;
            J.np = 2;
            J.n = 2 * panel;
        }
        J.a = b0 == at ? 0 : b1 == at ? 1 : box(rows[at]);
        out.push_back(J);
    };
    // depth-first order with parents
    std::vector<int> order, parent_edge(n, -1);
    for (int s = 0; s < n; ++s) {
        if (seen[s]) continue;
        std::vector<int> stack{s};
        seen[s] = 1;
        while (!stack.empty()) {
            const int x = stack.back();
            stack.pop_back();
            order.push_back(x);
            for (int e : inc[x]) {
                const int y = u[e] == x ? v[e] : u[e];
                if (!seen[y]) {
                    seen[y] = 1;
                    parent_edge[y] = e;
                    stack.push_back(y);
                }
            }
        }
    }
    for (int k = n - 1; k >= 0; --k) {
        const int x = order[k];
        std::vector<int> free;
        for (int e : inc[x])
            if (!used[e] && e != parent_edge[x]) free.push_back(e);
        if (free.size() % 2 && parent_edge[x] >= 0 && !used[parent_edge[x]]) free.push_back(parent_edge[x]);
        for (size_t i = 0; i < free.size(); i += 2) emit(x, free[i], i + 1 < free.size() ? free[i + 1] : -1);
    }
}

}  // namespace

bool zherk_plan(int N, const std::vector<ZherkTile>& cover, int n_ax, int n_inst, double est_live, int n_sms,
                long long ring_budget, long long split_budget, ZherkPlan& out) {
    if (n_inst < 1) return false;
    const double chunks = std::max(1.0, std::ceil(est_live / kZherkChunk));
    double best = 1e300;
    for (int form = kZherkReal; form <= (cover.empty() ? kZherkGauss : kZherkReal); ++form) {
        ZherkPlan z;
        z.form = form;
        z.n_ax = n_ax;
        if (form == kZherkReal) {
            z.rows = 2 * N;
            z.panel = cover.empty() ? zherk_panel(z.rows) : 128;
            z.tiles = cover.empty() ? zherk_triangle(z.rows, z.panel) : cover;
        } else {
            z.rows = 3 * N;
            z.panel = zherk_panel(N);
            z.tiles = zherk_gauss_tiles(N, z.panel);
        }
        if ((int)z.tiles.size() > 2 * n_sms) continue;
        std::vector<ZherkJob> one;  // the jobs of one instance
        make_jobs(z.tiles, form == kZherkReal ? z.rows : N, z.panel, one);
        const int nj = (int)one.size(), T = (int)z.tiles.size();
        const int vcap = (int)std::min<long long>(n_sms / nj, ring_budget / ((long long)zherk_row_bytes(n_ax) * z.rows));
        if (vcap < 1) continue;
        for (int S = 1; S <= 64 && (S == 1 || chunks / S >= 4); ++S) {
            if (S > 1 && (long long)n_inst * T * S * (128 * 128 * 4) > split_budget) break;
            const int total = n_inst * S, V = std::min(vcap, total), waves = (total + V - 1) / V;
            if (waves > kZherkMaxWaves) continue;
            // us: a chunk of a job (its MMAs at about 80 % of the tensor rate; the Z build
            // where a wave has few products), a wave's ramp, and the partial tiles written and read once
            const double t = waves * (chunks / S * n_ax * (0.35 + 0.6 * z.panel / 128.0) + 6.0) + total * (double)T * 131072.0 / 4e6;
            if (t < best) {
                best = t;
                out = z;
                out.us = t;
                out.V = V;
                out.S = S;
                out.waves = waves;
                out.jobs.clear();
                for (int v = 0; v < V; ++v)
                    for (ZherkJob J : one) {
                        J.v = v;
                        out.jobs.push_back(J);
                    }
                out.n_jobs = nj * V;
                out.n_jobs_last = nj * (total - (waves - 1) * V);
            }
        }
    }
    if (best == 1e300) return false;
    out.jobs.resize(n_sms, ZherkJob{});
    return true;
}

int zherk_ant_block(const ZherkPlan& z, int n_ant, int nc, int groups, int chan, int n_sms) {
    const int most = chan > 1 ? Z_BLOCK / 2 : Z_BLOCK;
    const int most_teams = z.n_ax == 1 ? 6 : 4;
    int best = 0;
    double t_best = 1e300;
    for (int ab = 1; ab <= most; ++ab) {
        const int ants = z_warps(nc) * ab, teams = n_sms / (groups * ((n_ant + ants - 1) / ants));
        if (teams < 1) continue;
        // cycles per chunk: an item's fixed part and its antennas, over the chunks in
        // flight, which have to leave the tensor side most of the ring
        double t = (800.0 + ab * (250.0 + 110.0 * chan)) / teams;
        if (teams > most_teams) t *= 1.0 + 0.5 * (teams - most_teams);
        if (t < t_best) {
            t_best = t;
            best = ab;
        }
    }
    return best;
}

}  // namespace mv
