// prep.cu -- Algorithm 2 steps (i) and (ii) of arXiv:2312.09763 (Sec. 3.1):
// rotation of the sources to East-North-Up with R(t) of eq. "rotation"
// (Sec. 2.3), the horizon cut with stable stream compaction, and the beam
// evaluation at the live sources (Sec. 2.4), fused with sqrt(I_s(nu)).
#include <algorithm>

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

// (FP64 code that is seldom reached stays out of line: inlined, it is executed under
// a predicate every time.)
__device__ __noinline__ float to_float_any(double v) { return (float)v; }
__device__ __noinline__ bool above_exact(const double* r, double x, double y, double z) { return rot_row(r, x, y, z) > 0.0; }

// (float)v in integer operations (round to nearest even): conversions run at the
// FP64 rate, two lanes a clock and SM.  What is no normal FP32 number takes the
// conversion.
__device__ __forceinline__ float to_float(double v) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(v);
    if (((unsigned)(b >> 52) & 0x7ffu) - 898u > 252u) return to_float_any(v);
    const unsigned r = (unsigned)((b + 0x0fffffffull + (b >> 29 & 1ull)) >> 29);  // exponent's low bits and 23 places
    return __uint_as_float(((unsigned)(b >> 32) & 0x80000000u) | ((r - (896u << 23)) & 0x7fffffffu));
}

// v in [-2, 2) times 2^62 (truncated below 2^-62).
__device__ __forceinline__ long long to_fixed(double v) {
    const long long b = __double_as_longlong(v);
    const int e = (int)(b >> 52) & 0x7ff, sh = e - 1013;  // the last place of a double's 53 bits is 2^(e - 1075)
    const long long m = (b & 0xfffffffffffffll) | 0x10000000000000ll;
    const long long f = sh >= 0 ? m << sh : sh > -53 ? m >> -sh : 0ll;
    return b < 0 ? -f : f;
}

// Whether source s is above the horizon at time t: the sign of rot_row, taken from
// FP32 products (within 1e-6 of their magnitudes' sum) where that is clear of zero
// and far from FP32's smallest numbers.
__device__ __forceinline__ bool above(const Model& m, const double* __restrict__ R, int t, long long s) {
    if (s >= m.n_src) return false;
    const double* r = R + 9 * t + 6;
    const double x = m.xeq[s], y = m.xeq[m.n_src + s], z = m.xeq[2 * m.n_src + s];
    const float a = to_float(r[0]) * to_float(x), b = to_float(r[1]) * to_float(y), c = to_float(r[2]) * to_float(z);
    const float up = a + b + c, sum = fabsf(a) + fabsf(b) + fabsf(c);
    return fabsf(up) > 4e-6f * sum && sum > 1e-30f ? up > 0.f : above_exact(r, x, y, z);
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

// Stable compaction of a block's live sources and their tables.  FP64 (two lanes a
// clock and SM) would bound it: rotating and converting every source before the
// cut took 390 us for 48 times of 1e5 sources (count and compaction), only the live
// ones 257.  So directions are 64-bit fixed point, rotated with integer products
// (within 5 x 2^-60, finer than FP64's 2^-53): 143 us.  FP64 East, North and Up go out
// only where the caller has asked for them.
__global__ void __launch_bounds__(kCullThreads)
k_cull_scatter(Model m, const double* __restrict__ R, CullWork w, int bpt, LiveTables lt) {
    kernel_chain();
    __shared__ unsigned masks[kCullThreads / 32];
    __shared__ int sums[kCullThreads / 32];
    __shared__ unsigned char list[kCullThreads];
    __shared__ long long rot[9];
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
    if (!lt.e && threadIdx.x < 9) rot[threadIdx.x] = to_fixed(R[9 * t + threadIdx.x]);
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
    const long long pos = before + (int)threadIdx.x, o = (long long)t * lt.pitch + pos;
    lt.idx[o] = (int)s;
    float ef, nf, uf;
    if (lt.e) {
        const double e = rot_row(r, x, y, z), n = rot_row(r + 3, x, y, z), u = rot_row(r + 6, x, y, z);
        lt.e[o] = e;
        lt.n[o] = n;
        lt.u[o] = u;
        ef = to_float(e);
        nf = to_float(n);
        uf = to_float(u);
    } else {
        const long long X = to_fixed(x), Y = to_fixed(y), Z = to_fixed(z);
        float comp[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const long long v = __mul64hi(rot[3 * c], X) + __mul64hi(rot[3 * c + 1], Y) + __mul64hi(rot[3 * c + 2], Z);  // 2^60
            const long long q = min((v + (1ll << 28)) >> 29, 2147483647ll);  // 2^31
            const long long o3 = ((long long)t * 3 + c) * lt.pitch + pos;
            lt.sfix[o3] = (unsigned)(q + 2147483648ll);
            lt.seps[o3] = (float)(int)(v - (q << 29)) * 8.67361737988403547e-19f;  // 2^-60
            comp[c] = __ll2float_rn(v) * 8.67361737988403547e-19f;
        }
        ef = comp[0];
        nf = comp[1];
        uf = comp[2];
    }
    // az = atan2(E, N) in [0, 2 pi), za = atan2(|EN|, Up): well conditioned at the pole
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

// Max of |value| over a warp, folded into amax (non-negative floats order
// like their bit patterns).
__device__ __forceinline__ void fold_amax(float v, float* amax) {
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    if ((threadIdx.x & 31) == 0 && v > 0.f) atomicMax(reinterpret_cast<int*>(amax), __float_as_int(v));
}

// What the beam evaluation of a live source keeps from one channel to the next.
// T: taps per axis (4 cubic, 2 bilinear).
template <int T>
struct SourceBeam {
    float sqrt_flux, half_alpha, za;
    float4 M;
    // stencil in za (pole-reflected, clamped) and az (periodic): weights, row offsets
    // in a plane, columns (those of a row across the pole half a turn on)
    float wa[T], sg[T];
    int row[T], col[T];
    unsigned across;  // bit r: row r lies across the pole

    __device__ __forceinline__ void load(const Model& m, const LiveTables& lt, int t, int s) {
        const long long o = (long long)t * lt.pitch + s;
        const int src = lt.idx[o];
        const float2 azza = lt.azza[o];
        za = azza.y;
        half_alpha = m.half_alpha[src];
        sqrt_flux = m.pol_m ? 1.f : m.sqrt_flux[src];
        M = m.pol_m ? m.pol_m[src] : make_float4(0.f, 0.f, 0.f, 0.f);
        if (m.beam_kind == 1) return;
        const float uz = azza.y / m.dza, ua = azza.x / m.daz;
        const float fz = floorf(uz), fa = floorf(ua);
        const float tz = uz - fz, ta = ua - fa;
        const int z0 = (int)fz - (T == 4 ? 1 : 0), a0 = (int)fa - (T == 4 ? 1 : 0);
        float wz[T];
        if constexpr (T == 4) {
            wz[0] = keys(tz + 1.f); wz[1] = keys(tz); wz[2] = keys(1.f - tz); wz[3] = keys(2.f - tz);
            wa[0] = keys(ta + 1.f); wa[1] = keys(ta); wa[2] = keys(1.f - ta); wa[3] = keys(2.f - ta);
        } else {
            wz[0] = 1.f - tz; wz[1] = tz;
            wa[0] = 1.f - ta; wa[1] = ta;
        }
        const float pole_sign = m.n_ax == 2 ? -1.f : 1.f;
        across = 0u;
#pragma unroll
        for (int r = 0; r < T; ++r) {
            int z = z0 + r;
            float g = 1.f;
            if (z < 0) {
                z = -z;
                across |= 1u << r;
                g = pole_sign;
            }
            row[r] = min(z, m.n_za - 1) * m.n_az;
            sg[r] = g * wz[r];
            int c = (a0 + r) % m.n_az;
            if (c < 0) c += m.n_az;
            col[r] = c;
        }
    }

    // One component of the beam from its plane P.
    __device__ __forceinline__ float2 eval(const float2* __restrict__ P, int n_az) const {
        float re = 0.f, im = 0.f;
#pragma unroll
        for (int r = 0; r < T; ++r) {
            const float2* rowp = P + row[r];
            float rr = 0.f, ri = 0.f;
#pragma unroll
            for (int q = 0; q < T; ++q) {
                int c = col[q];
                if (across >> r & 1u) {
                    c += n_az / 2;
                    if (c >= n_az) c -= n_az;
                }
                const float2 v = rowp[c];
                rr = fmaf(wa[q], v.x, rr);
                ri = fmaf(wa[q], v.y, ri);
            }
            re = fmaf(sg[r], rr, re);
            im = fmaf(sg[r], ri, im);
        }
        return make_float2(re, im);
    }
};

// WA[slot][b][p][k][s] = sqrt(I_s(nu)) * A^{pk}_b(az_s, za_s, nu) for the live
// sources of each instance (Algorithm 2 step ii, with the flux weight of step iv),
// in pairs of sources (common.cuh), zero up to the next multiple of 256 (as far as
// anything reads).  A thread takes `per` consecutive slots: their stencil, indices
// and divisions are those of the first one while the time stays the same.  What
// bounds it is the 16 scattered loads per channel: 350 antennas x 1e5 sources x 256
// instances 490 us with one slot a thread and zeros to the end of the pitch, 425 with
// four (438 with 16).
template <int T>
__global__ void __launch_bounds__(128, 6)
k_wa(Model m, const float2* __restrict__ planes, const Chan* __restrict__ chan,
     const Inst* __restrict__ inst, int inst0, int n_inst, int per, LiveTables lt, float2* __restrict__ wa,
     long long wa_pitch, float* __restrict__ amax) {
    kernel_chain();
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    const int ncomp = m.n_beam * m.n_feed * m.n_ax;
    const long long plane = (long long)m.n_za * m.n_az;
    SourceBeam<T> b;
    int t = -1, nl = 0;
    for (int slot = blockIdx.y * per; slot < min(n_inst, (int)(blockIdx.y + 1) * per); ++slot) {
        const Inst in = inst[inst0 + slot];
        if (in.t != t) {
            t = in.t;
            nl = lt.n_live[t];
            if (s < nl) b.load(m, lt, t, s);
        }
        float mx = 0.f;
        float2* out = wa + (long long)slot * ncomp * wa_pitch;
        if (s < nl) {
            const float spec = expf(b.half_alpha * chan[in.c].ln_ratio);
            const float w = m.pol_m ? spec : b.sqrt_flux * spec;
            if (m.beam_kind == 1) {
                const float a = w * expf(-m.gauss_c * b.za * b.za);
                put_wa(out, s, make_float2(a, 0.f));
                mx = fabsf(a);
            } else {
                const float2* P = planes + (long long)in.c * ncomp * plane;
                float2 a_prev = make_float2(0.f, 0.f);
                for (int comp = 0; comp < ncomp; ++comp, P += plane) {
                    const float2 a = b.eval(P, m.n_az);
                    if (!m.pol_m) {
                        const float2 v = make_float2(w * a.x, w * a.y);
                        put_wa(out + (long long)comp * wa_pitch, s, v);
                        mx = fmaxf(mx, hypotf(v.x, v.y));
                    } else if ((comp & 1) == 0) {  // axis 0 of a (beam, feed): wait for axis 1
                        a_prev = a;
                    } else {
                        float2 z0, z1;
                        apply_sky_sqrt(a_prev, a, b.M, w, z0, z1);
                        put_wa(out + (long long)(comp - 1) * wa_pitch, s, z0);
                        put_wa(out + (long long)comp * wa_pitch, s, z1);
                        mx = fmaxf(mx, fmaxf(hypotf(z0.x, z0.y), hypotf(z1.x, z1.y)));
                    }
                }
            }
        } else if (s < (nl + kKPad - 1) / kKPad * kKPad && s < wa_pitch) {
            for (int comp = 0; comp < ncomp; ++comp) put_wa(out + (long long)comp * wa_pitch, s, make_float2(0.f, 0.f));
        }
        fold_amax(mx, amax + slot);
    }
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
                      int n_sms, cudaStream_t st, long long* launches) {
    // slots per thread: as many as leave four blocks of 128 sources for every SM
    const long long bx = (lt.pitch + 127) / 128;
    const int per = (int)std::max(1ll, std::min<long long>(4, bx * n_inst / (4ll * n_sms)));
    const dim3 grid((unsigned)bx, (unsigned)((n_inst + per - 1) / per));
    *launches += 1;
    return launch_chained(m.interp == 0 ? k_wa<4> : k_wa<2>, grid, dim3(128), 0, st, m, d_planes, d_chan, d_inst, inst0,
                          n_inst, per, lt, d_wa, wa_pitch, d_amax);
}

}  // namespace mv
