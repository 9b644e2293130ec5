// zherk.h -- the streamed Z build + HERK of one batch of instances
// (zherk_tc.cu): its plan (host) and launch arguments.
#pragma once
#include <vector>

#include "common.cuh"

namespace mv {

constexpr int kZherkChunk = 64;      // sources per ring chunk
// Chunks in the ring, and bytes of a ring row.  Fewer chunks leave too little
// between the oldest chunk still being read and the newest ones being built (350
// antennas, one axis, 256 instances: 17.1 ms with 13 chunks, 16.2 with 14, 15.7 with
// 15, 15.5 with 16: 82 MB; the redundant cover 6.11, 5.98, 5.85, 5.78); more outgrow
// the L2 (15.7 and 5.82 with 17).
__host__ __device__ constexpr int zherk_ring_chunks(int n_ax) { return n_ax == 1 ? 16 : 9; }
__host__ __device__ constexpr int zherk_row_bytes(int n_ax) { return zherk_ring_chunks(n_ax) * kZherkChunk * 4 * n_ax; }
constexpr int kZherkMaxWaves = 2048;
constexpr int kZherkChan = 20;       // channels x components a group may have

// How Z is laid out in the ring.
//   real   2 N rows, Re and Im of every antenna-feed in turn: V from the lower
//          triangle of G = U U^T
//   gauss  3 N rows, X = Re Z, Y = Im Z and S = X + Y of every antenna-feed in
//          turn, read as three planes: V from
//          F = X Y^T (all of it) and the lower triangle of H = S S^T:
//          Re V_ab = H_ab - (F_ab + F_ba), Im V_ab = F_ba - F_ab.
enum ZherkForm : int { kZherkReal = 0, kZherkGauss = 1 };

// A product of panels of ring rows: A rows [ra, ra + panel) of an instance times
// B rows [rb, rb + panel) (gauss: plane * N + antenna-feed).  r0, c0: the rows and columns of the product it
// stands for (antenna-feeds of F or H with the gauss form, rows of U with the
// real one); trans: its rows hold the product's columns.
struct ZherkTile {
    int ra, rb, r0, c0, kind, trans;  // kind: 0 G (real) or F, 1 H
};

// The work of one SM in one wave: one A box of a panel of ring rows (128 rows of MMA,
// the last ones unused) and one or two B boxes.  n: columns of MMA, 0: none.
struct ZherkJob {
    int n, nbox;
    int a, b;                        // A's box; B's first box (the second one follows it)
    int row[4], plane[4];            // first row of each box within the instance (and its plane)
    int tile[2];
    int v, np;                       // instance within the wave, products
};

// Channels of one time (and one source range) whose Z is built together:
// virtual instances [v0, v0 + n) of the wave.  The launch fills in the rest.
struct alignas(16) ZherkGroup {
    int v0, n;
    int aph;                         // entry of the antenna phase table
    int uniform;                     // equally spaced channels
    int slot, t, c0, len;            // first instance's slot, its time, first source chunk, chunks
    int vi, pad0, pad1, pad2;        // first virtual instance, counted over all waves
};

struct ZherkPlan {
    int form = kZherkReal, n_ax = 1;
    int rows = 0, panel = 128;       // ring rows per instance, rows of a panel
    int V = 0, S = 0, waves = 0;     // instances per wave, source ranges per instance
    int n_jobs = 0, n_jobs_last = 0;
    double us = 0;                   // what it is expected to take
    std::vector<ZherkTile> tiles;
    std::vector<ZherkJob> jobs;      // n_sms entries; the last wave runs those with v < its instances
};

struct ZherkArgs {
    Model m;
    const Inst* inst;
    int inst0, n_inst;
    LiveTables lt;
    const float2* wa;
    long long wa_pitch;
    const float* scale;              // [n_inst] FP16 scale of the Z build, then (V) [n_inst] in all
    const AntPhase* aph;
    int n_phase;
    const int4* zv;                  // virtual instances: slot, time, first source chunk, chunks
    uint8_t* ring;
    int rows, map_rows, panel;       // ring rows per instance; rows of one plane, of a panel
    int V, S, n_waves, v_last;       // v_last: instances of the last wave
    const int* wave_base;            // [n_waves + 1] first chunk of each wave
    const int* wave_items;           // [n_waves] groups
    const int* wave_group0;          // [n_waves] first group
    const ZherkGroup* groups;
    const ZherkJob* jobs;
    int n_jobs, n_jobs_last;
    int ant_block;                   // antennas per Z warp
    int z_shift, z_buf_b;            // 1 << z_shift input buffers of the Z warps, bytes of each
    int flush;                       // 32-column stages per TMEM flush
    int n_tiles;
    int *ready, *done;               // per chunk: SMs that finished building it, that loaded it
    float* partial;                  // [slot][tile][S][128][128], column-major
    int* err;
};

// Sums the partial tiles into V (or the redundant groups' values).
struct ZherkFinalArgs {
    const Inst* inst;
    int inst0, n_inst;
    const float* scale;              // [n_inst] FP16 scale of WA in all, a power of two (NULL: none)
    const float* partial;
    const ZherkTile* tiles;
    const int* tile_of;              // gauss: [2][np][np] tile of F_ij and of H_ij (i >= j), np panels
    int n_tiles, S, N, np, panel;    // np: panels of a plane (gauss)
    float2* V;
    HerkOut ho;                      // uidx NULL: the full V
    const int2* limits;              // unique: row and column limits of every tile
};

// Rows of a panel: those of a plane split evenly over as few panels of at most 128 rows
// as there can be, in eights (350 rows: three of 120, so that two products side by
// side are 240 columns of MMAs instead of 256; 131: two of 72).
int zherk_panel(int rows);
// Products of one instance: in the real form the lower triangle of 2N rows,
std::vector<ZherkTile> zherk_triangle(int rows, int panel);

// and in the gauss form of N antenna-feeds.
std::vector<ZherkTile> zherk_gauss_tiles(int N, int panel);

// Plan for n_inst instances; cover: the real-form tiles to compute (empty: the
// whole V of N antenna-feeds, in either form).  est_live: live sources
// expected per instance; ring_budget: bytes the ring may take; split_budget: bytes
// the partial tiles may take where the sources are split (one tile a product is
// always taken).  False where the tiles of one instance do not fit the SMs.
bool zherk_plan(int N, const std::vector<ZherkTile>& cover, int n_ax, int n_inst, double est_live, int n_sms,
                long long ring_budget, long long split_budget, ZherkPlan& out);
// Antennas per Z warp for groups of up to `chan` channels, `groups` of them in
// a wave (0: no choice fits); nc: feeds x axes.
int zherk_ant_block(const ZherkPlan& z, int n_ant, int nc, int groups, int chan, int n_sms);
// Bytes of an input buffer of the Z warps (groups of up to chan channels), and the log2 of their number.
int zherk_input_bytes(int chan, int nc, int n_beam);
int zherk_input_shift(int bytes);
cudaError_t zherk_init();
// (multiplies WA of instances much weaker than others of their time; scale: 2 n_inst floats)
cudaError_t launch_zherk_prep(const ZherkArgs& P, const float* amax, int n_sms, float* scale, int4* zv,
                              int* wave_base, ZherkGroup* groups, int n_groups, bool by_length, long long n_counters,
                              cudaStream_t st, long long* launches);
cudaError_t launch_zherk(const ZherkArgs& P, int form, int n_ctas, cudaStream_t st, long long* launches);
cudaError_t launch_zherk_final(const ZherkFinalArgs& a, int form, cudaStream_t st, long long* launches);

// FP32 HERK on the CUDA cores (herk_fp32.cu): the form of Z (with the gauss form
// plane_rows = N and the planes X, Y and S one after another), its products and
// the source ranges each is split into.
struct Fp32Plan {
    int form = kZherkReal, rows = 0, plane_rows = 0, split = 1;
    std::vector<ZherkTile> tiles;
};
// gauss: whether that form may be taken; split_budget: bytes of one instance's partial
// tiles up to which the sources may be split.
Fp32Plan herk_fp32_plan(int N, int n_ax, int n_inst, double est_live, int n_sms, bool gauss, long long split_budget);
cudaError_t herk_fp32_init();
// Partial tiles [n_inst][n_tiles][split][128][128] of U's products.
cudaError_t launch_herk_fp32(const Inst* d_inst, int inst0, int n_inst, LiveTables lt, int n_ax, const float* d_u,
                             int rows, int plane_rows, long long k_pitch, const ZherkTile* d_tiles, int n_tiles,
                             int split, float* d_partial, int* d_err, cudaStream_t st, long long* launches);

}  // namespace mv
