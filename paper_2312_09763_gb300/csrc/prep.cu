// prep.cu -- Algorithm 2 steps (i) and (ii) of arXiv:2312.09763 (Sec. 3.1):
// rotation of the sources to East-North-Up with R(t) of eq. "rotation"
// (Sec. 2.3), the horizon cut with stable stream compaction, and the beam
// evaluation at the live sources (Sec. 2.4), fused with sqrt(I_s(nu)).
#include "common.cuh"
#include "zcore.cuh"

namespace mv {
namespace {

constexpr int kCullThreads = 256;
// Blocks of one time up to which a scatter block sums the counts before it
// itself (at most eight loads a thread); beyond, a scan kernel does it.
constexpr int kScanBlocks = 2048;

// One component of X_hrz = R X_eq, evaluated as (R0 x + R1 y) + R2 z with
// every product and sum rounded on its own (no FMA contraction), so the
// horizon decision Up > 0 is taken on a value fixed by that expression.
__device__ __forceinline__ double rot_row(const double* r, double x, double y, double z) {
    return __dadd_rn(__dadd_rn(__dmul_rn(r[0], x), __dmul_rn(r[1], y)), __dmul_rn(r[2], z));
}

__device__ __forceinline__ bool above(const Model& m, const double* __restrict__ R, int t, long long s) {
    return s < m.n_src && rot_row(R + 9 * t + 6, m.xeq[s], m.xeq[m.n_src + s], m.xeq[2 * m.n_src + s]) > 0.0;
}

// The live sources of block blk of time t: their count and, a bit each, which.
__device__ __forceinline__ void cull_count(const Model& m, const double* __restrict__ R, const CullWork& w, int bpt, int t,
                                           int blk) {
    const long long b = (long long)t * bpt + blk;
    const bool live = above(m, R, t, (long long)blk * kCullThreads + threadIdx.x);
    if (w.masks) {
        const unsigned mask = __ballot_sync(0xffffffffu, live);
        if ((threadIdx.x & 31) == 0) w.masks[b * (kCullThreads / 32) + (threadIdx.x >> 5)] = mask;
    }
    const int c = __syncthreads_count(live);
    if (threadIdx.x == 0) w.counts[b] = c;
}

// Per-channel beam planes: P[c][b][p][k][za][az] = sum_m w_m(c) G[b][p][k][m0(c)+m][za][az]
// (the frequency axis of the gridded beam interpolated once per channel); comp:
// (b, p, k) flattened.
__device__ __forceinline__ void beam_plane(const Model& m, const float2* __restrict__ grid, const Chan* __restrict__ chan,
                                           float2* __restrict__ planes, int n_comp, int c, int comp, long long i) {
    const long long plane = (long long)m.n_za * m.n_az;
    if (i >= plane) return;
    const Chan ch = chan[c];
    const float2* g = grid + (long long)comp * m.n_nu * plane;
    float re = 0.f, im = 0.f;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        float2 v = g[(long long)(ch.m0 + j) * plane + i];
        re = fmaf(ch.w[j], v.x, re);
        im = fmaf(ch.w[j], v.y, im);
    }
    planes[((long long)c * n_comp + comp) * plane + i] = make_float2(re, im);
}

// The parts of a call that depend on none of its other results, one range of
// blocks each: the live counts, the beam planes, and the first batch's phase
// table and zeroed max |WA|.  Small calls are bound by launches (64 antennas x
// 8192 sources x 16 channels: 62 us with nine kernels and two fills, 54 with six
// kernels and one).
__global__ void __launch_bounds__(kCullThreads) k_front(FrontArgs a) {
    kernel_chain();
    long long b = blockIdx.x;
    if (b < a.cull_blocks) {
        cull_count(a.m, a.R, a.w, a.bpt, (int)(b / a.bpt), (int)(b % a.bpt));
        return;
    }
    b -= a.cull_blocks;
    if (b < a.plane_blocks) {
        const int pb = (int)(((long long)a.m.n_za * a.m.n_az + kCullThreads - 1) / kCullThreads);
        const int n_comp = a.m.n_beam * a.m.n_feed * a.m.n_ax;
        const long long rest = b / pb;
        beam_plane(a.m, a.grid, a.chan, a.planes, n_comp, (int)(rest / n_comp), (int)(rest % n_comp),
                   (b % pb) * kCullThreads + threadIdx.x);
        return;
    }
    b -= a.plane_blocks;
    const int nb = (a.m.n_ant + kCullThreads - 1) / kCullThreads;
    const long long rest = b / nb;
    if (b == 0)
        for (int i = threadIdx.x; i < a.n_amax; i += kCullThreads) a.amax[i] = 0.f;
    zcore::ant_phase_entry(a.m, a.inst, a.chan, a.groups, a.g_first, a.n_phase, a.aph, (int)(rest / a.n_phase),
                           (int)(rest % a.n_phase), (int)(b % nb) * kCullThreads + threadIdx.x);
}

// Exclusive scan of the per-block live counts of one time (one block per time).
__global__ void __launch_bounds__(1024)
k_cull_scan(const int* __restrict__ counts, int* __restrict__ offsets, int* __restrict__ n_live, int bpt) {
    kernel_chain();
    __shared__ int warp_sums[32];
    const int t = blockIdx.x;
    const int per = (bpt + blockDim.x - 1) / blockDim.x;
    const int b0 = threadIdx.x * per;
    const int* c = counts + (long long)t * bpt;
    int local = 0;
    for (int i = 0; i < per; ++i)
        if (b0 + i < bpt) local += c[b0 + i];
    // block exclusive scan of `local`
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int incl = local;
    for (int o = 1; o < 32; o <<= 1) {
        int v = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += v;
    }
    if (lane == 31) warp_sums[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        int w = lane < (int)(blockDim.x >> 5) ? warp_sums[lane] : 0;
        for (int o = 1; o < 32; o <<= 1) {
            int v = __shfl_up_sync(0xffffffffu, w, o);
            if (lane >= o) w += v;
        }
        warp_sums[lane] = w;  // inclusive over warps
    }
    __syncthreads();
    int base = (warp > 0 ? warp_sums[warp - 1] : 0) + incl - local;
    int* o = offsets + (long long)t * bpt;
    for (int i = 0; i < per; ++i)
        if (b0 + i < bpt) { o[b0 + i] = base; base += c[b0 + i]; }
    if (threadIdx.x == blockDim.x - 1) n_live[t] = warp_sums[(blockDim.x >> 5) - 1];
}

// (float)v in integer operations (round to nearest even): conversions run at the
// FP64 rate.  Results below 2^-126 take the conversion.
__device__ __forceinline__ float to_float(double v) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(v);
    if (((unsigned)(b >> 52) & 0x7ffu) <= 897u) return (float)v;
    const unsigned r = (unsigned)((b + 0x0fffffffull + (b >> 29 & 1ull)) >> 29);  // exponent's low bits and 23 places
    return __uint_as_float(((unsigned)(b >> 32) & 0x80000000u) | ((r - (896u << 23)) & 0x7fffffffu));
}

// Stable compaction of a block's live sources and their tables.  What bounds it is
// FP64 (two lanes a clock and SM): a live source costs 15 operations of its
// rotation and three per component of its fixed-point direction, one below the
// horizon none.  Count and compaction of 48 times of 1e5 sources: 390 us when
// every source was rotated and converted before the cut, 257 here.
__global__ void __launch_bounds__(kCullThreads)
k_cull_scatter(Model m, const double* __restrict__ R, CullWork w, int bpt, LiveTables lt) {
    kernel_chain();
    __shared__ unsigned masks[kCullThreads / 32];
    __shared__ int sums[kCullThreads / 32];
    __shared__ unsigned char list[kCullThreads];
    const int t = blockIdx.x / bpt, blk = blockIdx.x - t * bpt;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const long long b = (long long)t * bpt + blk;
    const long long s0 = (long long)blk * kCullThreads;
    if (!w.masks) {
        const unsigned mask = __ballot_sync(0xffffffffu, above(m, R, t, s0 + threadIdx.x));
        if (lane == 0) masks[warp] = mask;
    } else if (threadIdx.x < kCullThreads / 32) {
        masks[threadIdx.x] = w.masks[b * (kCullThreads / 32) + threadIdx.x];
    }
    // live sources of the blocks before
    int before = 0;
    if (bpt <= kScanBlocks) {
        for (int i = threadIdx.x; i < blk; i += kCullThreads) before += w.counts[(long long)t * bpt + i];
        before = __reduce_add_sync(0xffffffffu, before);
        if (lane == 0) sums[warp] = before;
    }
    __syncthreads();
    int rank = 0, total = 0;
#pragma unroll
    for (int i = 0; i < kCullThreads / 32; ++i) {
        const int c = __popc(masks[i]);
        if (i < warp) rank += c;
        total += c;
    }
    if (bpt <= kScanBlocks) {
        before = 0;
#pragma unroll
        for (int i = 0; i < kCullThreads / 32; ++i) before += sums[i];
        if (blk == bpt - 1 && threadIdx.x == 0) lt.n_live[t] = before + total;
    } else {
        before = w.offsets[b];
    }
    if (masks[warp] >> lane & 1u) list[rank + __popc(masks[warp] & ((1u << lane) - 1u))] = (unsigned char)threadIdx.x;
    __syncthreads();
    if (threadIdx.x >= total) return;
    const long long s = s0 + list[threadIdx.x];
    const double* r = R + 9 * t;
    const double x = m.xeq[s], y = m.xeq[m.n_src + s], z = m.xeq[2 * m.n_src + s];
    const double comp[3] = {rot_row(r, x, y, z), rot_row(r + 3, x, y, z), rot_row(r + 6, x, y, z)};
    const long long pos = before + (int)threadIdx.x, o = (long long)t * lt.pitch + pos;
    if (lt.e) {
        lt.e[o] = comp[0];
        lt.n[o] = comp[1];
        lt.u[o] = comp[2];
    }
    lt.idx[o] = (int)s;
    if (lt.sfix) {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            // q = comp 2^31 rounded to an integer: added to 1.5 x 2^52, whose last place is
            // one, so that q (mod 2^32) is the sum's low word
            constexpr double kShift = 6755399441055744.0;
            const double sum = fma(comp[c], 2147483648.0, kShift);
            double q = sum - kShift;
            unsigned lo = (unsigned)__double2loint(sum);
            if (lo == 0x80000000u && __double2hiint(comp[c]) >= 0) {  // 1 rounds to 2^31 - 1
                lo = 0x7fffffffu;
                q = 2147483647.0;
            }
            const long long o3 = ((long long)t * 3 + c) * lt.pitch + pos;
            lt.sfix[o3] = lo + 0x80000000u;
            lt.seps[o3] = to_float(fma(q, -4.656612873077392578125e-10, comp[c]));  // 2^-31
        }
    }
    // az = atan2(E, N) in [0, 2 pi), za = atan2(|EN|, Up): well conditioned at the pole
    const float ef = to_float(comp[0]), nf = to_float(comp[1]), uf = to_float(comp[2]);
    float az = atan2f(ef, nf);
    if (az < 0.f) az += 6.2831853071795864769f;
    const float za = atan2f(sqrtf(ef * ef + nf * nf), uf);
    lt.azza[o] = make_float2(az, za);
}

// Keys (1981) cubic-convolution kernel, a = -1/2.
__device__ __forceinline__ float keys(float x) {
    const float t = fabsf(x);
    if (t <= 1.f) return (1.5f * t - 2.5f) * t * t + 1.f;
    if (t < 2.f) return ((-0.5f * t + 2.5f) * t - 4.f) * t + 2.f;
    return 0.f;
}

// WA[slot][b][p][k][s] = sqrt(I_s(nu)) * A^{pk}_b(az_s, za_s, nu) for the live
// sources of each instance (Algorithm 2 step ii, with the flux weight of step iv),
// in pairs of sources (common.cuh).
// Max of |value| over a warp, folded into amax (non-negative floats order
// like their bit patterns).
__device__ __forceinline__ void fold_amax(float v, float* amax) {
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    if ((threadIdx.x & 31) == 0 && v > 0.f) atomicMax(reinterpret_cast<int*>(amax), __float_as_int(v));
}

__device__ float wa_eval(const Model& m, const float2* __restrict__ planes, const Chan& ch, const Inst& in,
                         LiveTables lt, int s, float2* __restrict__ out, long long wa_pitch);

__global__ void __launch_bounds__(128)
k_wa(Model m, const float2* __restrict__ planes, const Chan* __restrict__ chan,
     const Inst* __restrict__ inst, int inst0, LiveTables lt, float2* __restrict__ wa, long long wa_pitch,
     float* __restrict__ amax) {
    kernel_chain();
    const int slot = blockIdx.y;
    const Inst in = inst[inst0 + slot];
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    const int nl = lt.n_live[in.t];
    const int ncomp = m.n_beam * m.n_feed * m.n_ax;
    float mx = 0.f;
    float2* out = wa + (long long)slot * ncomp * wa_pitch;
    if (s < nl) {
        mx = wa_eval(m, planes, chan[in.c], in, lt, s, out, wa_pitch);
    } else if (s < wa_pitch) {  // zeros past the live count: the Z build reads whole source pairs
        for (int comp = 0; comp < ncomp; ++comp) put_wa(out + (long long)comp * wa_pitch, s, make_float2(0.f, 0.f));
    }
    fold_amax(mx, amax + slot);
}

// sqrt(I_s(nu)) A^{pk}_b(s) for every component of one live source; returns
// the largest magnitude written.
__device__ float wa_eval(const Model& m, const float2* __restrict__ planes, const Chan& ch, const Inst& in,
                         LiveTables lt, int s, float2* __restrict__ out, long long wa_pitch) {
    const long long o = (long long)in.t * lt.pitch + s;
    const int src = lt.idx[o];
    const float2 azza = lt.azza[o];
    const float spec = expf(m.half_alpha[src] * ch.ln_ratio);
    const float w = m.pol_m ? spec : m.sqrt_flux[src] * spec;
    const float4 M = m.pol_m ? m.pol_m[src] : make_float4(0.f, 0.f, 0.f, 0.f);
    const int ncomp = m.n_beam * m.n_feed * m.n_ax;
    if (m.beam_kind == 1) {
        const float a = w * expf(-m.gauss_c * azza.y * azza.y);
        put_wa(out, s, make_float2(a, 0.f));
        return fabsf(a);
    }
    // stencil in za (pole-reflected, clamped) and az (periodic)
    const bool cubic = m.interp == 0;
    const int nt = cubic ? 4 : 2;
    const float uz = azza.y / m.dza, ua = azza.x / m.daz;
    const float fz = floorf(uz), fa = floorf(ua);
    const float tz = uz - fz, ta = ua - fa;
    const int z0 = (int)fz - (cubic ? 1 : 0), a0 = (int)fa - (cubic ? 1 : 0);
    float wz[4], wa_[4];
    if (cubic) {
        wz[0] = keys(tz + 1.f); wz[1] = keys(tz); wz[2] = keys(1.f - tz); wz[3] = keys(2.f - tz);
        wa_[0] = keys(ta + 1.f); wa_[1] = keys(ta); wa_[2] = keys(1.f - ta); wa_[3] = keys(2.f - ta);
    } else {
        wz[0] = 1.f - tz; wz[1] = tz; wz[2] = wz[3] = 0.f;
        wa_[0] = 1.f - ta; wa_[1] = ta; wa_[2] = wa_[3] = 0.f;
    }
    int rows[4], shifts[4];
    float sg[4];
    const float pole_sign = m.n_ax == 2 ? -1.f : 1.f;
    for (int r = 0; r < nt; ++r) {
        int row = z0 + r, sh = 0;
        float g = 1.f;
        if (row < 0) { row = -row; sh = m.n_az / 2; g = pole_sign; }
        if (row > m.n_za - 1) row = m.n_za - 1;
        rows[r] = row; shifts[r] = sh; sg[r] = g * wz[r];
    }
    const long long plane = (long long)m.n_za * m.n_az;
    float mx = 0.f;
    float2 a_prev = make_float2(0.f, 0.f);
    for (int comp = 0; comp < ncomp; ++comp) {
        const float2* P = planes + ((long long)in.c * ncomp + comp) * plane;
        float re = 0.f, im = 0.f;
        for (int r = 0; r < nt; ++r) {
            const float2* rowp = P + (long long)rows[r] * m.n_az;
            float rr = 0.f, ri = 0.f;
            for (int q = 0; q < nt; ++q) {
                int col = (a0 + q + shifts[r]) % m.n_az;
                if (col < 0) col += m.n_az;
                const float2 v = rowp[col];
                rr = fmaf(wa_[q], v.x, rr);
                ri = fmaf(wa_[q], v.y, ri);
            }
            re = fmaf(sg[r], rr, re);
            im = fmaf(sg[r], ri, im);
        }
        if (!m.pol_m) {
            const float2 v = make_float2(w * re, w * im);
            put_wa(out + (long long)comp * wa_pitch, s, v);
            mx = fmaxf(mx, hypotf(v.x, v.y));
        } else if ((comp & 1) == 0) {  // axis 0 of a (beam, feed): wait for axis 1
            a_prev = make_float2(re, im);
        } else {
            float2 z0, z1;
            apply_sky_sqrt(a_prev, make_float2(re, im), M, w, z0, z1);
            put_wa(out + (long long)(comp - 1) * wa_pitch, s, z0);
            put_wa(out + (long long)comp * wa_pitch, s, z1);
            mx = fmaxf(mx, fmaxf(hypotf(z0.x, z0.y), hypotf(z1.x, z1.y)));
        }
    }
    return mx;
}

}  // namespace

cudaError_t launch_front(const FrontArgs& args, int n_times, LiveTables lt, cudaStream_t st, long long* launches) {
    FrontArgs a = args;
    const Model& m = a.m;
    a.cull_blocks = (long long)a.bpt * n_times;
    a.plane_blocks = a.planes ? ((long long)m.n_za * m.n_az + kCullThreads - 1) / kCullThreads * m.n_beam * m.n_feed * m.n_ax * a.n_chan : 0;
    const long long phase_blocks = a.aph ? (long long)((m.n_ant + kCullThreads - 1) / kCullThreads) * a.n_phase * a.n_groups : 0;
    const long long blocks = a.cull_blocks + a.plane_blocks + phase_blocks;
    if (blocks > 0x7fffffffll) return cudaErrorInvalidValue;
    if (blocks > 0) {
        k_front<<<(unsigned)blocks, kCullThreads, 0, st>>>(a);
        *launches += 1;
    }
    if (a.cull_blocks > 0) {
        if (a.bpt > kScanBlocks) {
            cudaError_t e = launch_chained(k_cull_scan, dim3(n_times), dim3(1024), 0, st, (const int*)a.w.counts, a.w.offsets,
                                           lt.n_live, a.bpt);
            if (e != cudaSuccess) return e;
            *launches += 1;
        }
        *launches += 1;
        return launch_chained(k_cull_scatter, dim3((unsigned)a.cull_blocks), dim3(kCullThreads), 0, st, m, a.R, a.w, a.bpt, lt);
    }
    return cudaGetLastError();
}

cudaError_t launch_wa(const Model& m, const float2* d_planes, const Chan* d_chan, const Inst* d_inst,
                      int inst0, int n_inst, LiveTables lt, float2* d_wa, long long wa_pitch, float* d_amax,
                      cudaStream_t st, long long* launches) {
    dim3 grid((unsigned)((lt.pitch + 127) / 128), n_inst);
    *launches += 1;
    return launch_chained(k_wa, grid, dim3(128), 0, st, m, d_planes, d_chan, d_inst, inst0, lt, d_wa, wa_pitch, d_amax);
}

}  // namespace mv
