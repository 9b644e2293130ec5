// herk_fp32.cu -- Algorithm 2 step (v) of arXiv:2312.09763 (Sec. 3.1),
// V = Z Z^dagger (eq. "zz"), on the CUDA cores in FP32.
//
// Z is held as real rows with the source axis contiguous (zbuild.cu): Re and Im
// of every antenna-feed in turn (2N rows, G = U U^T as in zherk.h's real form),
// or the planes X, Y and S = X + Y (3N rows, F = X Y^T and H = S S^T, the gauss
// form) where herk_fp32_plan expects that to be quicker.  A unit of work is one
// 128 x 128 product over one of S ranges of the sources; its sum goes out as a
// partial tile and launch_zherk_final folds the tiles into V.
//
// What bounds it: the FP32 FMA pipes (128 a clock and SM).  A thread owns 8 x 8
// entries, two FP32 sums each (even and odd sources, so that operands and sums
// are natural pairs of the packed FMA, fma.rn.f32x2, two products per issue
// slot), fed by 16-byte shared-memory reads along the source axis: per four
// sources a warp issues 128 packed FMAs and 16 reads.  The panels arrive as
// they lie in memory through a four-stage TMA ring; the 128-byte swizzle keeps
// the reads free of bank conflicts.  Blocks past a panel's end or above the
// diagonal are skipped in steps of 16 or 32 rows (350 antennas: the work of
// 11.5 whole products against 15 listed, and against 15.5 in the real form).
// Every 512 sources the pairs are added into FP32 running sums in shared
// memory, which keeps the rounding error of long source sums near sqrt(K) ulp.
// The source split fills the SMs whatever the number of products.
//
// 350 antennas, 1e5 sources (half of them live), 8 channels: 13.34 ms with
// scalar FMAs on a 16-source ring of transposed panels, one block per product
// of the triangle (168 blocks on 152 SMs); 3.38 ms here, 60 % of the FMA
// pipes' rate while a block runs (2.0 ms).  Of that, the shared-memory reads cost
// about 0.4 ms (a copy that reads once per stage), the real form 0.9 ms more,
// cp.async panels with per-thread addresses 0.4 ms more, the flushes 0.04 ms.
#include <algorithm>
#include <cmath>

#include "common.cuh"
#include "tc.cuh"
#include "zherk.h"

namespace mv {
namespace {

using namespace tc;

constexpr int BT = 128;              // tile rows and columns
constexpr int BKF = 32;              // sources per stage: a 128-byte row, as wide as the swizzle
constexpr int PANEL = BT * BKF * 4;  // bytes of a panel in shared memory
constexpr int STAGES_F = 4;
constexpr int RUN_PITCH = BT + 1;
constexpr int FLUSH = 16;            // stages per flush
constexpr int BARS_F = STAGES_F * 2 * PANEL;  // barriers and the abort flag, then the running sums
constexpr int RUN_F = BARS_F + 64;
constexpr int SMEM_F = RUN_F + BT * RUN_PITCH * 4 + 1024;  // (and up to 1024 bytes to align the panels)
static_assert(SMEM_F <= 232448, "227 KB of shared memory");

// Two FP32 numbers in a register pair.
using Pair = unsigned long long;
__device__ __forceinline__ void fma_pair(Pair& c, Pair a, Pair b) {
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(c) : "l"(a), "l"(b));
}
__device__ __forceinline__ float sum_of(Pair p) {
    float a, b;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(p));
    return a + b;
}

// The main loop for NI x 16 rows of the tile and NJ x 16 columns of it; of a
// diagonal product only the 16 x 16 blocks that reach its lower triangle.
template <int NI, int NJ, bool DIAG>
__device__ __forceinline__ void tile_loop(const CUtensorMap* map, int row_a, int row_b, int kb0, int n, uint8_t* sm,
                                          float* run, int* err) {
    const int tid = threadIdx.x, tx = (tid & 31) >> 1, ty = (tid >> 5) * 2 + (tid & 1);
    const uint32_t bars = smem_u32(sm + BARS_F);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(sm + BARS_F + 8 * STAGES_F);
    Pair acc[NI][NJ];
#pragma unroll
    for (int i = 0; i < NI; ++i)
#pragma unroll
        for (int j = 0; j < NJ; ++j) acc[i][j] = 0ull;
    // one stage: both panels (a diagonal product's B is its A)
    auto load = [&](int it) {
        const int s = it % STAGES_F;
        const uint32_t st = smem_u32(sm) + s * 2 * PANEL, bar = bars + 8 * s;
        mbar_expect_tx(bar, (DIAG ? 1 : 2) * PANEL);
        tma_load_2d(st, map, (kb0 + it) * BKF, row_a, bar);
        if (!DIAG) tma_load_2d(st + PANEL, map, (kb0 + it) * BKF, row_b, bar);
    };
    auto flush = [&]() {
#pragma unroll
        for (int j = 0; j < NJ; ++j)
#pragma unroll
            for (int i = 0; i < NI; ++i) {
                if (DIAG && i < j) continue;
                run[(tx + 16 * j) * RUN_PITCH + ty + 16 * i] += sum_of(acc[i][j]);
                acc[i][j] = 0ull;
            }
    };
    int issued = 0;
    if (tid == 0)
        for (; issued < STAGES_F - 1 && issued < n; ++issued) load(issued);
    for (int it = 0; it < n; ++it) {
        const int s = it % STAGES_F;
        // (after a wait that gave up, the rest of the loop runs through without data)
        if (!*abort_flag) wait_bounded_spin(bars + 8 * s, (uint32_t)(it / STAGES_F) & 1u, abort_flag, err);
        __syncthreads();  // everyone is done with the stage before
        if (tid == 0 && issued < n && !*abort_flag) load(issued++);
        const uint8_t* pa = sm + s * 2 * PANEL + ty * 128;
        const uint8_t* pb = sm + s * 2 * PANEL + (DIAG ? 0 : PANEL) + tx * 128;
        const int xa = (ty & 7) * 16, xb = (tx & 7) * 16;  // the swizzle of rows ty + 16 i, tx + 16 j
#pragma unroll 1
        for (int k = 0; k < 128; k += 16) {  // four sources
            ulonglong2 a[NI];
#pragma unroll
            for (int i = 0; i < NI; ++i) a[i] = *reinterpret_cast<const ulonglong2*>(pa + i * 2048 + (k ^ xa));
#pragma unroll
            for (int j = 0; j < NJ; ++j) {
                const ulonglong2 b = *reinterpret_cast<const ulonglong2*>(pb + j * 2048 + (k ^ xb));
#pragma unroll
                for (int i = DIAG ? j : 0; i < NI; ++i) fma_pair(acc[i][j], b.x, a[i].x);
#pragma unroll
                for (int i = DIAG ? j : 0; i < NI; ++i) fma_pair(acc[i][j], b.y, a[i].y);
            }
        }
        if (it % FLUSH == FLUSH - 1) flush();
    }
    flush();
    if (tid == 0 && *abort_flag) {  // copies still in flight land before the block ends (a bounded wait)
        const unsigned long long t0 = gtimer();
        for (int it = max(0, issued - STAGES_F); it < issued; ++it)
            while (!mbar_try_wait(bars + 8 * (it % STAGES_F), (uint32_t)(it / STAGES_F) & 1u) && gtimer() - t0 < kTimeoutNs) {}
    }
}

__global__ void __launch_bounds__(256, 1)
k_herk_fp32(const __grid_constant__ CUtensorMap map, const Inst* __restrict__ inst, int inst0, LiveTables lt, int n_ax,
            int rows, int plane_rows, const ZherkTile* __restrict__ tiles, int n_tiles, int S,
            float* __restrict__ partial, int* err) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* sm = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    float* run = reinterpret_cast<float*>(sm + RUN_F);  // [column][row]
    const int tile = blockIdx.x % n_tiles, rest = blockIdx.x / n_tiles, ks = rest % S, slot = rest / S;
    const ZherkTile t = tiles[tile];
    const long long K = (long long)lt.n_live[inst[inst0 + slot].t] * n_ax;
    const int KB = (int)((K + BKF - 1) / BKF);
    const int kb0 = (int)((long long)KB * ks / S), n = (int)((long long)KB * (ks + 1) / S) - kb0;
    for (int i = threadIdx.x; i < BT * RUN_PITCH; i += 256) run[i] = 0.f;
    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES_F; ++s) mbar_init(smem_u32(sm + BARS_F) + 8 * s, 1);
        *reinterpret_cast<int*>(sm + BARS_F + 8 * STAGES_F) = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    const int row_a = slot * rows + t.ra, row_b = slot * rows + t.rb;
    // rows of each panel inside its plane (a box may reach past them: those products are not
    // read), in 16 x 16 blocks and steps of two
    const int ni = (min(BT, plane_rows - t.ra % plane_rows) + 31) / 32;
    const int nj = (min(BT, plane_rows - t.rb % plane_rows) + 31) / 32;
#define MV_LOOP(I, J)                                                                                        \
    if (ni == I && nj == J) {                                                                                \
        if (I == J && t.ra == t.rb) tile_loop<2 * I, 2 * J, true>(&map, row_a, row_b, kb0, n, sm, run, err); \
        else tile_loop<2 * I, 2 * J, false>(&map, row_a, row_b, kb0, n, sm, run, err);                       \
    }
#define MV_LOOPS(I) MV_LOOP(I, 1) MV_LOOP(I, 2) MV_LOOP(I, 3) MV_LOOP(I, 4)
    MV_LOOPS(1) MV_LOOPS(2) MV_LOOPS(3) MV_LOOPS(4)
#undef MV_LOOPS
#undef MV_LOOP
    __syncthreads();
    float* p = partial + (((long long)slot * n_tiles + tile) * S + ks) * (BT * BT);
    for (int i = threadIdx.x; i < BT * BT; i += 256) p[i] = run[(i >> 7) * RUN_PITCH + (i & 127)];
}

}  // namespace

cudaError_t herk_fp32_init() {
    return cudaFuncSetAttribute(k_herk_fp32, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_F);
}

cudaError_t launch_herk_fp32(const Inst* d_inst, int inst0, int n_inst, LiveTables lt, int n_ax, const float* d_u,
                             int rows, int plane_rows, long long k_pitch, const ZherkTile* d_tiles, int n_tiles,
                             int split, float* d_partial, int* d_err, cudaStream_t st, long long* launches) {
    const long long blocks = (long long)n_inst * n_tiles * split;
    EncodeTiledFn enc = get_encode();
    if (split < 1 || n_tiles < 1 || !d_partial || !enc || blocks > 0x7fffffffll || (long long)n_inst * rows > 0x7fffffffll)
        return cudaErrorInvalidValue;
    CUtensorMap map;
    cuuint64_t dims[2] = {(cuuint64_t)k_pitch, (cuuint64_t)((long long)n_inst * rows)};
    cuuint64_t strides[1] = {(cuuint64_t)k_pitch * sizeof(float)};
    cuuint32_t box[2] = {BKF, BT}, estr[2] = {1, 1};
    if (enc(&map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<float*>(d_u), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
        return cudaErrorInvalidValue;
    k_herk_fp32<<<(unsigned)blocks, 256, SMEM_F, st>>>(map, d_inst, inst0, lt, n_ax, rows, plane_rows, d_tiles, n_tiles,
                                                       split, d_partial, d_err);
    *launches += 1;
    return cudaGetLastError();
}

// Work of a product of ra x rb rows, in 16 x 16 blocks of the kernel's tile.
static double blocks_of(int ra, int rb, bool diag) {
    const int ni = (std::min(ra, BT) + 31) / 32 * 2, nj = (std::min(rb, BT) + 31) / 32 * 2;
    return diag ? 0.5 * ni * (ni + 1) : (double)ni * nj;
}

Fp32Plan herk_fp32_plan(int N, int n_ax, int n_inst, double est_live, int n_sms, bool gauss, long long split_budget) {
    Fp32Plan best;
    double t_best = 1e300;
    for (int form = kZherkReal; form <= (gauss ? kZherkGauss : kZherkReal); ++form) {
        Fp32Plan z;
        z.form = form;
        z.tiles = form == kZherkReal ? zherk_triangle(2 * N, BT) : zherk_gauss_tiles(N, BT);
        z.rows = form == kZherkReal ? 2 * N : 3 * N;
        z.plane_rows = form == kZherkReal ? 2 * N : N;
        double area = 0;
        for (const ZherkTile& t : z.tiles)
            area += blocks_of(z.plane_rows - t.ra % z.plane_rows, z.plane_rows - t.rb % z.plane_rows, t.ra == t.rb);
        const double stages = std::max(1.0, std::ceil(est_live * n_ax / BKF));
        const double units = (double)n_inst * (double)z.tiles.size();
        double t_form = 1e300;
        for (int S = 1; S <= 64 && (S == 1 || stages / S >= 4); ++S) {
            if (S > 1 && (long long)z.tiles.size() * S * (BT * BT * 4) > split_budget) break;
            // us: rounds of units over the SMs, each a fill, its stages (2.2 us for a whole tile's) and
            // its partial tile; the partial tiles read back; the rows of Z written and read
            const double t = std::ceil(units * S / n_sms) * (4.0 + stages / S * 2.2 * area / (64.0 * z.tiles.size())) +
                             units * S * 65536.0 / 4e6 + (double)n_inst * z.rows * stages * BKF * 8.0 / 4e6;
            if (t < t_form) {
                t_form = t;
                z.split = S;
            }
        }
        if (t_form < t_best) {
            t_best = t_form;
            best = std::move(z);
        }
    }
    return best;
}

}  // namespace mv
