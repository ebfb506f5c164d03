// host_plan.cuh -- host-side helpers shared by the ABI translation units:
// TMA descriptor encoding, GEMM tiling / token-split planning and the
// dispatch of a GEMM launch to its tile-width instantiation.
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>

#include <cstdint>
#include <cstring>
#include <mutex>

#include "gemm_launch.cuh"
#include "splitk_cluster.cuh"
#include "thin.cuh"

namespace cola {

// Thread-block clusters of S CTAs (index S, at least 1) of the cluster-reduced
// kernel that the current device runs at once.
const int* reduce_cluster_capacity(int sms);

namespace {

// ------------------------------------------------------------ tensor maps
using EncodeFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                              const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                              CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeFn encode_fn()
{
    static EncodeFn fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q = cudaDriverEntryPointSymbolNotFound;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeFn>(p);
    });
    return fn;
}

// 2-D bf16 matrix [outer x inner] with row pitch ld (elements) and box
// {box_inner, box_outer}.  Loads read zeros outside the extents; stores are
// clipped to them.
bool make_map(CUtensorMap* m, const void* base, int64_t inner, int64_t outer, int64_t ld, int box_inner,
              int box_outer, CUtensorMapSwizzle swz)
{
    EncodeFn fn = encode_fn();
    if (!fn) return false;
    cuuint64_t dims[2] = {static_cast<cuuint64_t>(inner), static_cast<cuuint64_t>(outer)};
    cuuint64_t strides[1] = {static_cast<cuuint64_t>(ld) * 2};
    cuuint32_t box[2] = {static_cast<cuuint32_t>(box_inner), static_cast<cuuint32_t>(box_outer)};
    cuuint32_t estr[2] = {1u, 1u};
    CUresult r = fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, swz, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS;
}

// Epilogue box of 32 rows x 32 columns (64-byte rows, 64-byte swizzle): the
// unit in which the GEMM epilogue stores bf16 outputs and reads the saved Z.
bool map_box32(CUtensorMap* m, const void* base, int64_t cols, int64_t rows, int64_t ld)
{
    return make_map(m, base, cols, rows, ld, 32, 32, CU_TENSOR_MAP_SWIZZLE_64B);
}

// Box of 32 rows x 64 columns (128-byte rows, 128-byte swizzle): the chunks of
// the gated dX epilogue.
bool map_box64(CUtensorMap* m, const void* base, int64_t cols, int64_t rows, int64_t ld)
{
    return make_map(m, base, cols, rows, ld, GLU_COLS, 32, CU_TENSOR_MAP_SWIZZLE_128B);
}

// K-major operand: rows are the M (or N) index, k contiguous: box {64, rows_per_tile}.
// MN-major operand: rows are k, the M (or N) index contiguous: box {64, 64}.
bool map_kmajor(CUtensorMap* m, const void* base, int64_t k_extent, int64_t mn_extent, int64_t ld, int tile_rows)
{
    return make_map(m, base, k_extent, mn_extent, ld, 64, tile_rows, CU_TENSOR_MAP_SWIZZLE_128B);
}

bool map_mnmajor(CUtensorMap* m, const void* base, int64_t mn_extent, int64_t k_extent, int64_t ld)
{
    return make_map(m, base, mn_extent, k_extent, ld, 64, 64, CU_TENSOR_MAP_SWIZZLE_128B);
}

// ------------------------------------------------------------ planning
// Column tile: the width that pads N least; a compute-heavy GEMM with K >= 512
// (`pairs`) takes 256, because only 256-column tiles run on CTA pairs, which
// outweighs the padding where fill_bn leaves it.  Measured against 128-column tiles
// wherever 256 pads N by more than 5 % (forward + backward): 16384 tokens 2600 ->
// 2600, r = 640 396 -> 301 us; 12000, 3300 -> 3300, r = 832 427 -> 357; 65536, 1500 ->
// 1500, r = 384 479 -> 439; 67708, 1536 -> 1536, r = 320 446 -> 409.
int choose_bn(int64_t N, bool pairs = false)
{
    if (N <= 128) return 128;
    if (pairs) return 256;
    const int64_t pad256 = (N + 255) / 256 * 256;
    const int64_t pad128 = (N + 127) / 128 * 128;
    return pad256 <= pad128 ? 256 : 128;
}

// Compute-heavy: more than one 128-row block and
//   - at least 64 GFLOP, or
//   - at least 16 GFLOP at an arithmetic intensity (each operand read once, the
//     result written once) of >= 300 FLOP/B, above the ridge of the GB300 bf16
//     roofline (~287): the tensor-bound GEMMs of the 8192-token inference
//     workloads (measured: 1B forward -14 %), or
//   - at least 16 GFLOP at >= 150 FLOP/B with K >= 1024, where the walk is long
//     against the epilogue, and with K >= 2048 if 256-column tiles pad N more
//     (forward + backward: 32768 tokens 1024 -> 2736, r = 256 243 -> 227 us,
//     100000, 1000 -> 1100, r = 192 407 -> 373; but 30000, 1200 -> 1200, r = 320
//     without the second condition 215 -> 226, and the 65536-token q/k/v of the
//     60M block, K = 512, 41 -> 48 us for Z).
bool heavy_gemm(int64_t M, int64_t N, int64_t K)
{
    const double m = static_cast<double>(M), n = static_cast<double>(N), k = static_cast<double>(K);
    const double flops = 2.0 * m * n * k;
    const double intensity = flops / (2.0 * (m * k + n * k + m * n));
    if (M <= 128 || flops < 16e9) return false;
    const bool pads = (N + 255) / 256 * 256 > (N + 127) / 128 * 128;
    return flops >= 64e9 || intensity >= 300.0 || (intensity >= 150.0 && K >= (pads ? 2048 : 1024));
}

// A GEMM of one 128-row block (a few tokens: decode) streams its B operand
// through as many CTAs as it has column tiles, so it takes 128-column tiles:
// twice the CTAs of 256-column ones, up to N = 8192 (64 tiles; wider ones,
// often batched in twos, would spill into a second wave of CTAs).  Measured:
// 1B decode step 0.066 -> 0.059 ms, 7B 0.090 -> 0.081 ms.
int choose_bn_for(int64_t M, int64_t N, int64_t K)
{
    if (M <= 128 && N <= 8192) return 128;
    return choose_bn(N, heavy_gemm(M, N, K) && K >= 512);
}

// Whether 256-column tiles round N up further than 128-column ones do, and by more
// than the 5 % that CTA pairs always outweigh from N = 1024 on.
bool pairs_pad(int64_t N)
{
    const int64_t pad256 = (N + 255) / 256 * 256;
    return pad256 > (N + 127) / 128 * 128 && !(N >= 1024 && pad256 * 100 <= N * 105);
}

// Where a GEMM that pairs would pad starts taking them.
// The epilogues of Z and dZ outlast the MMAs of a shorter walk, and a pair's two CTAs
// then wait for them together: pairs against 128-column tiles, K = 512, r = 384, 832
// Z 107 / 87 and 97 / 86 us, dZ 158 / 111 and 143 / 112; K = 768 Z 85 / 82, 78 / 76, dZ
// 115 / 87, 107 / 82; K = 1024 r = 832 66 / 73 and 84 / 76.  Y and dX free their
// accumulators before they store: K = 512 to 1024 0.85 to 1.02.
constexpr int64_t PAD_K_SIGMA = 1024, PAD_K_STORE = 512;

// The column tile of `count` GEMMs of one launch: 128 columns instead of 256
//   - where those tiles still run in one wave (twice the CTAs of 256-column ones);
//   - for compute-heavy GEMMs that pairs would pad, below K = pad_k, and where the
//     padding costs more waves than pairs make up for.  A wave of pair tiles (256 x
//     256 on two SMs) and one of two 128-row sub-tiles (256 x 128 on one) hold the same
//     work per SM, and the first is some 20 % faster: us of Z, waves of pairs and of
//     128-column tiles: 12715 x 384, K = 2048 (2, 1) 36.9 / 29.2; 10926 x 832, 1100 (3, 2)
//     35.7 / 31.8; 50781 x 320, 2048 (6, 4) 81.4 / 75.4; 26702 x 640, 2048 (5, 4) 67.5 /
//     71.0; 16954 x 384, 3072 (2, 2) 47.7 / 58.0.
int fill_bn(int64_t M, int64_t N, int64_t K, int count, int sms, int64_t pad_k)
{
    const int bn = choose_bn_for(M, N, K);
    if (bn == 128) return bn;
    const int64_t n256 = (N + 255) / 256, n128 = (N + 127) / 128;
    if (!heavy_gemm(M, N, K)) return count * ((M + BM - 1) / BM) * n128 <= sms ? 128 : 256;
    if (!pairs_pad(N)) return bn;
    const int64_t units = count * ((M + 2 * BM - 1) / (2 * BM)), pairs = sms / 2;
    const int64_t waves256 = (units * n256 + pairs - 1) / pairs, waves128 = (units * n128 + sms - 1) / sms;
    return K < pad_k || 4 * waves256 > 5 * waves128 ? 128 : bn;
}

// Whether plain outputs of N columns and pitch `ld` are stored through 64-column
// boxes (EPI_STORE64, and EPI_STORE on CTA pairs) or through rings of 32-column
// ones.  64 columns where rows are not 32-byte aligned (a 64-byte row piece then
// touches a sector more, twice as often), 32 against 64: Y of 110691 x 1463, two of
// them, 306 -> 213 us; 106705 x 712, r = 64, two 98 -> 82; 4047 x 1611, three 15.5 ->
// 14.4; and for a ragged right edge (N % 8 != 0), which they store by coalesced rows
// and the ring one element at a time: 65536 x 1021, r = 256 102 -> 54 us.  Other rows
// are written faster by the ring, which keeps more stores in flight, 64 against 32:
// 106705 x 720, r = 64, two 69 -> 65 us; 8143 x 1536, three 23.5 -> 23.0; 2048 x
// 4096, K = 512 12.0 -> 11.7 (but 106705 x 720, one 32 -> 34.6).
bool store_boxes64(bool pair, int64_t N, int64_t ld)
{
    return pair || ld % 16 != 0 || N % 8 != 0;
}

// Tile modes ("msub" below): 1 = one CTA runs a 128-row tile; 2 = one CTA
// runs two 128-row sub-tiles sharing each B tile; TILE_PAIR = a CTA pair runs
// a 256-row tile with tcgen05 cta_group::2 (each CTA loads half of B).
constexpr int TILE_PAIR = 3;

int tile_rows(int msub) { return msub == 1 ? BM : 2 * BM; }        // rows of one unit
int a_box_rows(int msub) { return msub == TILE_PAIR ? BM : BM * msub; }   // rows of A one CTA loads
int b_box_rows(int bn, int msub) { return msub == TILE_PAIR ? bn / 2 : bn; }   // K-major B rows one CTA loads
int unit_slots(int msub, int sms) { return msub == TILE_PAIR ? sms / 2 : sms; }   // units in flight

// Compute-heavy GEMMs with 256-column tiles and K >= 512 run on CTA pairs:
// halving each CTA's B traffic relieves the shared-memory bandwidth that a
// single CTA's M = 128 MMAs, its TMA fills and its epilogue stores saturate
// (measured: -5 to -25 % per GEMM on the 1B layers, K = 512 to 65536).  With
// K = 256 (4 k-blocks per tile, the store-bound Y and dX GEMMs at rank 256)
// a pair was 20-40 % slower, and with 128-column tiles slower than one CTA
// running two 128-row sub-tiles (+12 to +23 %), which those keep.  The
// HBM-bound short GEMMs keep single-CTA 128-row tiles (a taller tile
// lengthens the epilogue they are limited by).
int choose_msub(int64_t M, int64_t N, int64_t K, int bn)
{
    if (!heavy_gemm(M, N, K)) return 1;
    if (bn == 256) return K >= 512 ? TILE_PAIR : 1;
    return 2;
}

// Tile grid of one GEMM, without a token split.
GemmParams base_params(int64_t M, int64_t N, int64_t K, int bn, int msub)
{
    GemmParams p;
    std::memset(&p, 0, sizeof p);
    p.M = static_cast<int>(M);
    p.N = static_cast<int>(N);
    p.k_blocks = static_cast<int>((K + BK - 1) / BK);
    p.m_tiles = static_cast<int>((M + tile_rows(msub) - 1) / tile_rows(msub));
    p.n_tiles = static_cast<int>((N + bn - 1) / bn);
    p.kb_per_split = p.k_blocks;
    p.splits = 1;
    p.units = p.m_tiles * p.n_tiles;
    return p;
}

// A reduce launch after a split weight-gradient launch, in k-block steps of
// the busiest CTA (a few microseconds).
constexpr double REDUCE_LAUNCH_KB = 16.0;

// Token split of weight-gradient GEMMs sharing one launch (same K): minimise
// (waves of persistent CTAs) x (k-blocks per unit + the cost of writing and
// re-reading its fp32 partial tile, counted in k-blocks of operand bytes:
// 8 BN rows / (128 (rows + BN)), plus 2 for the reduction pass), with at least
// 4 k-blocks per split.
int choose_splits(int tiles, int k_blocks, int bn, int msub, int sms)
{
    const int max_s = k_blocks / 4 > 1 ? k_blocks / 4 : 1;
    const int rows = tile_rows(msub);
    const double c_part = 8.0 * bn * rows / (128.0 * (rows + bn)) + 2.0;
    sms = unit_slots(msub, sms);
    double best = -1.0;
    int S = 1;
    for (int s = 1; s <= max_s; ++s) {
        const long long units = static_cast<long long>(tiles) * s;
        const long long waves = (units + sms - 1) / sms;
        const long long kb = (k_blocks + s - 1) / s;
        const double cost = static_cast<double>(waves) * (static_cast<double>(kb) + (s > 1 ? c_part : 0.0));
        if (best < 0 || cost < best) {
            best = cost;
            S = s;
        }
    }
    return S;
}

void set_splits(GemmParams& p, int S)
{
    p.kb_per_split = (p.k_blocks + S - 1) / S;
    p.splits = (p.k_blocks + p.kb_per_split - 1) / p.kb_per_split;
    p.units = p.m_tiles * p.n_tiles * p.splits;
}

// Split-K through fp32 slabs for the forward GEMMs of small launches: with fewer
// output tiles than half the SMs (a few hundred tokens or less) and K >= 1024,
// the K range of each tile is split (>= 4 k-blocks per split, up to about one
// unit per SM); the fp32 partials are reduced, and the epilogue applied, by the
// reduce kernel.  The Y GEMMs of r >= 1024 above 64 tokens, and the Z/H GEMMs of 33
// to 48 tokens at r < 256 (64 in one tile; not GELU's), or of any number while the cluster
// reduction (rank_gemm_splits) is switched off.  A shorter K
// streams too little per tile for the extra reduce launch to pay off (measured:
// the 2048-token 60M layer, K = 512 / 128, got slower).  1 = no split.
int small_launch_splits(int tiles, int k_blocks, int sms)
{
    if (2 * tiles >= sms || k_blocks < 16) return 1;
    const int s = (sms + tiles - 1) / tiles;
    return s < k_blocks / 4 ? s : k_blocks / 4;
}

// K splits of a small launch reduced inside thread-block clusters
// (splitk_cluster.cuh, 128 x 128 tiles), with at most half as many tiles as SMs,
// up to S = 8 and >= 4 k-blocks per split.  The SMs of a cluster lie in one
// partition of the GPU, so it runs fewer clusters of S at once than SMs / S (on
// GB300 76, 46, 36, 28, 23, 15, 15 for S = 2..8): S is the one whose waves of
// clusters take the fewest k-block steps, CLUSTER_WAVE_KB of them for the
// exchange and the start of each wave.  Measured (weight gradients of 15249
// tokens, 19 tiles): S = 8 in two waves 36 us, planned split and reduce 28.
// *cost (when not null): those steps, less one wave's CLUSTER_WAVE_KB.
// 1 = no split.
constexpr int CLUSTER_WAVE_KB = 8;

int cluster_splits(int tiles, int k_blocks, int sms, int* cost = nullptr)
{
    if (tiles < 1 || 2 * tiles > sms) return 1;
    const int* cap = reduce_cluster_capacity(sms);
    int best = 1, best_cost = 0;
    for (int s = 2; s <= MAX_CLUSTER && s <= k_blocks / 4 && s * tiles <= sms; ++s) {
        const int waves = (tiles + cap[s] - 1) / cap[s];
        const int c = waves * ((k_blocks + s - 1) / s + CLUSTER_WAVE_KB) - CLUSTER_WAVE_KB;
        if (best == 1 || c <= best_cost) {
            best = s;
            best_cost = c;
        }
    }
    if (cost) *cost = best_cost;
    return best;
}

// K splits, inside clusters, of the `count` rank-r GEMMs of one launch (Z of the
// forward, dZ of the backward): 128 x 128 tiles, at most half as many as SMs, not
// compute-heavy.  1 = no split.  Measured against fp32 slabs with a reduce launch
// (Z) and an unsplit dZ, whole graph-replayed passes with the schedules below:
// q/k/v of 509 tokens, d = 1024, r = 256 23.9 -> 16.4 us forward, 58.8 -> 37.4 us
// with its backward; a 150-token layer 3000 -> 3000, r = 768 66.1 -> 41.1 us; a
// 2048-token 350M-shaped block 268 -> 192 us.
//   Z   from K = 1024 on (13 k-blocks with few tiles, 12 where the last is not whole):
//       shorter ones are no slower unsplit (forward of 2 to 74 tiles, split against
//       unsplit: 8 k-blocks 1.12 to 1.27, 12 1.04 to 1.21, but K = 712 0.92 to 0.98 up
//       to 24 tiles, 13 and 14 0.97 to 1.02 up to 24 and 1.05 to 1.17 above; from 16 on
//       the other way is the slabs', 0.65 to 0.97, and above 48 tokens, or 64 in one
//       tile: with fewer rows their reduce is the shorter way: one tile of 40 tokens, K =
//       1024 to 11008 1.05 to 1.11, of 128 tokens 0.88 to 0.95; three tiles of 40 tokens
//       1.04, of 64 0.94 to 0.96).
//   dZ  where the split takes enough k-blocks off the longest CTA to pay for the
//       exchange (whole backward, split against unsplit: 5 fewer 1.00 to 1.04, 8
//       0.93 to 1.03; in two splits, whose SMs the unsplit tiles half fill, 8 fewer
//       1.01 to 1.03, 10 1.00), and always up to 64 tokens, of whose rows the exchange
//       moves few (three of 1 to 9 tokens, K = 576 to 689 0.93 to 0.95).
// Both hold for SiLU and the identity.  GELU's elementwise work outweighs the
// exchange, and the splits share it out: split for every K that can be (gated MLP
// of 783 tokens, 960 -> 2176, r = 192 15.9 -> 14.0 us, 585 tokens, 696 -> 1536, r =
// 128, two projections 14.9 -> 12.7; 52 tokens, 862 -> 2304 14.0 -> 9.8), but for a dZ
// of many tiles and few k-blocks (us, unsplit and split, 56 tiles of 9 13.4, 15.9; a
// backward with 76 of 13 51.8, 49.6, with 54 of 16 42.6, 39.8).
int rank_gemm_splits(int64_t n, int64_t N, int64_t K, int count, int sigma, int sms, bool dz)
{
    if (heavy_gemm(n, N, K)) return 1;
    const int64_t tiles = count * ((n + BM - 1) / BM) * ((N + CBN - 1) / CBN);
    if (2 * tiles > sms) return 1;
    const int kb = static_cast<int>((K + BK - 1) / BK);
    const bool cheap = sigma != SIG_GELU;
    const bool few_kb = kb < (K % BK == 0 ? 13 : 12);
    if (cheap && !dz && (kb < 16 ? few_kb || tiles > 24 : n <= (tiles == 1 ? 64 : 48))) return 1;
    const int S = cluster_splits(static_cast<int>(tiles), kb, sms);
    const int least = cheap ? (S == 2 ? 9 : 8) : (tiles >= 48 ? 5 : 0);   // k-blocks saved
    if (dz && n > THIN_MAX_TOKENS && kb - (kb + S - 1) / S < least) return 1;
    return S;
}

// Split of a thin launch (thin.cuh): `tiles` 128-row weight tiles over k_blocks
// (per half of a gated product).  Clusters of up to 16 CTAs with at least two
// k-blocks each, 1.6 CTAs per SM at most (measured, 7B-shaped block of one
// token: 61.3 us at 1.25, 58.6 at 1.6, 64.4 at 2; 1B-shaped, 32 tokens: 45.1,
// 44.0, 44.9); the operand ring as deep as lets two CTAs, or one and a CTA of
// the kernel before, share an SM.  A gated product of more than 48 tokens in
// splits takes more shared memory than that, so its splits are counted for one CTA
// per SM: 43 tiles of 57 tokens, r = 512 21.1 us a call for 1.6 and 14.8 for one.
// The SMs of a cluster lie in one partition of the GPU, so it runs at most 14
// clusters of more than 13 CTAs at once, two a partition, and three of 13: Z of 16
// tokens, 15 tiles of 86 k-blocks 14.8 us in fifteens and 9.3 for 14 tiles, 17 tiles
// in thirteens 10.0.
constexpr int THIN_WIDE_CLUSTER = 13, THIN_WIDE_CLUSTERS = 14;

void thin_splits(ThinBatch& b, bool glu, int sms, bool one_per_sm = false)
{
    b.NT = (b.n + 15) / 16 * 16;
    int s = (one_per_sm ? sms : sms * 8 / 5) / b.tiles;
    if (s > (b.k_blocks + 1) / 2) s = (b.k_blocks + 1) / 2;
    if (s > THIN_MAX_CLUSTER) s = THIN_MAX_CLUSTER;
    if (s > THIN_WIDE_CLUSTER && b.tiles > THIN_WIDE_CLUSTERS) s = THIN_WIDE_CLUSTER;
    if (s < 1) s = 1;
    b.kps = (b.k_blocks + s - 1) / s;
    b.S = (b.k_blocks + b.kps - 1) / b.kps;   // no empty split
    b.TB = (b.n + b.S - 1) / b.S;
    const int left = THIN_SMEM_BUDGET - 1024 - THIN_BAR_BYTES - thin_recv_bytes(b.S, b.TB, glu);
    b.stages = left / thin_stage_bytes(b.NT);
    const int iters = b.kps * (glu ? 2 : 1);
    if (b.stages > iters) b.stages = iters;
    if (b.stages > THIN_MAX_STAGES) b.stages = THIN_MAX_STAGES;
    if (b.stages < 2) b.stages = 2;
    if (!one_per_sm && thin_smem_bytes(b.stages, b.NT, b.S, b.TB, glu) > THIN_SMEM_BUDGET) thin_splits(b, glu, sms, true);
}

int64_t partial_elems(const GemmParams& p, int bn, int msub)
{
    return static_cast<int64_t>(p.m_tiles) * tile_rows(msub) * p.n_tiles * bn;
}

// Weight-gradient group plan: count GEMMs D_i[M_i x N_i] = sum over the same
// ntok tokens, run by one launch with one tile configuration and one split.
struct WgradPlan {
    int bn, msub, splits, count;
    GemmParams p[MAX_GROUP];
    int64_t slab[MAX_GROUP];       // fp32 elements per split slab of each GEMM
    int64_t part_elems;            // all slabs of all splits
    double cost;                   // choose_splits' cost of the chosen split
};

// The plan with tiles of bn columns in mode msub.
WgradPlan plan_wgrad_tiles(const int64_t* M, const int64_t* N, int count, int64_t ntok, int bn, int msub, int sms)
{
    WgradPlan w;
    std::memset(&w, 0, sizeof w);
    w.count = count;
    w.bn = bn;
    w.msub = msub;
    int tiles = 0;
    for (int i = 0; i < count; ++i) {
        w.p[i] = base_params(M[i], N[i], ntok, w.bn, w.msub);
        // the token-major operands are read along the whole reduction: walk
        // the tiles so that a wave shares the panels of the larger one
        w.p[i].n_major = N[i] > M[i] ? 1 : 0;
        tiles += w.p[i].m_tiles * w.p[i].n_tiles;
    }
    const int S = choose_splits(tiles, w.p[0].k_blocks, w.bn, w.msub, sms);
    w.part_elems = 0;
    for (int i = 0; i < count; ++i) {
        set_splits(w.p[i], S);
        w.slab[i] = partial_elems(w.p[i], w.bn, w.msub);
        w.part_elems += static_cast<int64_t>(w.p[i].splits) * w.slab[i];
    }
    w.splits = w.p[0].splits;
    {
        const int rows = tile_rows(w.msub);
        const double c_part = 8.0 * w.bn * rows / (128.0 * (rows + w.bn)) + 2.0;
        const int sl = unit_slots(w.msub, sms);
        const long long units = static_cast<long long>(tiles) * w.splits;
        const long long waves = (units + sl - 1) / sl;
        w.cost = static_cast<double>(waves) * (w.p[0].kb_per_split + (w.splits > 1 ? c_part : 0.0)) + REDUCE_LAUNCH_KB;
    }
    return w;
}

// Split-tail schedule of a weight-gradient launch with bf16 outputs
// (EPI_TAIL).  The output tiles run whole in waves of `slots` CTAs (CTA
// pairs); the CTAs of a wave walk the token range in step, so the operand
// panels their tiles share are read from HBM about once.  The R < slots
// tiles of the last, partial wave are split over the tokens into `pieces`
// pieces each (R x pieces <= slots, >= 4 k-blocks per piece), so that the
// last wave is as short as the others allow; the tail reduce sums their
// partial slots.  Only the tail tiles write fp32 partials.  (Walking every
// CTA's equal share of all tile-and-token steps instead, stream-K style, was
// measured 1.4 to 1.6x slower at 60M to 7B: the CTAs drift apart in the token
// range, and the shared panels are then read from HBM once per tile.)
struct TailPlan {
    int body;                  // whole tiles (full waves)
    int tail;                  // tiles of the last wave
    int ntiles;                // tail tiles the reduce finishes (tail when split, else 0)
    int pieces, kps;           // pieces per tail tile, k-blocks per piece
    int units;                 // body + ntiles x pieces
    int kb;
    int tile_begin[MAX_GROUP];
    int64_t part_elems;        // ntiles x pieces x tile_rows x bn fp32 (0 when pieces == 1)
    double cost;               // k-blocks of the busiest CTA, plus the partial round trip
    TailTile tile[MAX_TAIL_TILES];
};

TailPlan plan_tail(const GemmParams* p, int count, int bn, int msub, int sms)
{
    TailPlan s;
    std::memset(&s, 0, sizeof s);
    int tiles = 0;
    for (int g = 0; g < count; ++g) {
        s.tile_begin[g] = tiles;
        tiles += p[g].m_tiles * p[g].n_tiles;
    }
    s.kb = p[0].k_blocks;
    const int slots = unit_slots(msub, sms);
    const int waves = tiles / slots;
    const int R = tiles - waves * slots;
    s.body = waves * slots;
    s.tail = R;
    s.pieces = 1;
    s.kps = s.kb;
    const int rows = tile_rows(msub);
    const double c_part = 8.0 * bn * rows / (128.0 * (rows + bn)) + 2.0;   // as in choose_splits
    if (R > 0 && R <= MAX_TAIL_TILES) {
        const int most = s.kb / 4 > 1 ? s.kb / 4 : 1;
        int St = slots / R < most ? slots / R : most;
        if (St > 1) {
            s.kps = (s.kb + St - 1) / St;
            St = (s.kb + s.kps - 1) / s.kps;   // no empty piece
        }
        // the pieces' partials and the reduce launch have to pay for themselves
        s.pieces = St > 1 && s.kps + c_part + REDUCE_LAUNCH_KB < s.kb ? St : 1;
        if (s.pieces == 1) s.kps = s.kb;
    }
    s.units = s.body + R * s.pieces;
    s.cost = static_cast<double>(waves) * s.kb + (R > 0 ? s.kps + (s.pieces > 1 ? c_part + REDUCE_LAUNCH_KB : 0.0) : 0.0);
    if (s.pieces > 1) {
        s.part_elems = static_cast<int64_t>(R) * s.pieces * rows * bn;
        s.ntiles = R;
        for (int i = 0; i < R; ++i) {
            const int t = s.body + i;
            int g = 0;
            for (int j = 1; j < count; ++j)
                if (t >= s.tile_begin[j]) g = j;
            int mb = 0, nb = 0;
            tile_coords(p[g], t - s.tile_begin[g], mb, nb);
            TailTile& e = s.tile[i];
            e.g = g;
            e.m0 = mb * rows;
            e.n0 = nb * bn;
            e.lo_slot = i * s.pieces;
            e.count = s.pieces;
        }
    }
    return s;
}

// The split-tail schedule of a planned group (bf16 gradients), with its tiles.  It runs
// when its cost is no higher than the uniform token split's (tail_wins).
TailPlan wgrad_tail_plan(const WgradPlan& w, int64_t ntok, int sms)
{
    GemmParams p[MAX_GROUP];
    for (int j = 0; j < w.count; ++j) {
        p[j] = base_params(w.p[j].M, w.p[j].N, ntok, w.bn, w.msub);
        p[j].n_major = w.p[j].n_major;
    }
    return plan_tail(p, w.count, w.bn, w.msub, sms);
}

bool tail_wins(const WgradPlan& w, const TailPlan& t) { return t.cost <= w.cost; }

// k-block steps of a planned group by the schedule it runs (`uniform`: fp32 gradients
// never take the split tail), for comparing tile sizes: a tail's few tiles are reduced
// in about half of REDUCE_LAUNCH_KB.
double wgrad_cost(const WgradPlan& w, int64_t ntok, bool uniform, int sms)
{
    if (uniform) return w.cost;
    const TailPlan t = wgrad_tail_plan(w, ntok, sms);
    return tail_wins(w, t) ? t.cost - (t.pieces > 1 ? 0.5 * REDUCE_LAUNCH_KB : 0.0) : w.cost;
}

// The plan of a group with the widest tiles all its GEMMs would take.  CTA pairs that pad
// a width (by more than fill_bn lets pass) run it where their schedule takes no more
// than 5/4 of the steps of 128-column tiles, which are of equal work per SM and some 20 %
// slower; steps, pairs and 128 columns, and us with the reduce: 16276 tokens 2560 -> 2560,
// r = 384 (199, 151) 83.7 / 72.0; 8877, 1100 -> 1100, r = 1024 (130, 93) 57.1 / 50.5; 25431,
// 2560 -> 2560, r = 384 (284, 222) 112.5 / 100.3; 14305, 5461 -> 5461, r = 384 (280, 224)
// 102.6 / 104.3; 23475, 1024 -> 1024, r = 832 (205, 179) 83.8 / 85.9.
WgradPlan plan_wgrad(const int64_t* M, const int64_t* N, int count, int64_t ntok, bool uniform, int sms)
{
    int bn = 256;
    for (int i = 0; i < count; ++i) {
        const int b = choose_bn_for(M[i], N[i], ntok);
        bn = b < bn ? b : bn;
    }
    const auto tile_mode = [&](int cols) {   // the smallest tile any GEMM of the group would take
        int msub = TILE_PAIR;
        for (int i = 0; i < count; ++i) {
            const int ms = choose_msub(M[i], N[i], ntok, cols);
            if (ms == 1 || (ms == 2 && msub == TILE_PAIR)) msub = ms;
        }
        return msub;
    };
    const int msub = tile_mode(bn);
    const WgradPlan w = plan_wgrad_tiles(M, N, count, ntok, bn, msub, sms);
    if (bn == 256 && msub == 1) {
        // 128 columns where those tiles run in one wave unsplit, unless 256 take far fewer
        // steps by splits (of 3 operand bytes to 2): 293 to 5662 tokens 0.84 to 1.0 of the
        // time of 256 columns up to 1.6 times the steps, from there on 0.99 to 1.06
        int64_t t = 0;
        for (int i = 0; i < count; ++i) t += ((M[i] + BM - 1) / BM) * ((N[i] + 127) / 128);
        if (t > sms) return w;
        const WgradPlan narrow = plan_wgrad_tiles(M, N, count, ntok, 128, 1, sms);
        return wgrad_cost(narrow, ntok, uniform, sms) > 1.6 * wgrad_cost(w, ntok, uniform, sms) ? w : narrow;
    }
    bool padded = false;
    for (int i = 0; i < count; ++i) padded = padded || pairs_pad(N[i]);
    if (msub != TILE_PAIR || !padded) return w;
    const WgradPlan narrow = plan_wgrad_tiles(M, N, count, ntok, 128, tile_mode(128), sms);
    return wgrad_cost(w, ntok, uniform, sms) > 1.25 * wgrad_cost(narrow, ntok, uniform, sms) ? narrow : w;
}

// The plan of one gradient whose partial tile grid has to fit `limit` bytes even
// unsplit, with the token split reduced until its slabs do.  Wide tiles round M and
// N up further: when their grid is too large, 128-column tiles, and then 128 x 128
// ones, whose grid is the smallest.  false: not even that fits.
bool plan_wgrad_within(int64_t M, int64_t N, int64_t ntok, size_t limit, int sms, WgradPlan* w)
{
    const auto slab = [&] { return static_cast<size_t>(w->slab[0]) * 4; };
    *w = plan_wgrad(&M, &N, 1, ntok, true, sms);
    if (slab() > limit) *w = plan_wgrad_tiles(&M, &N, 1, ntok, 128, choose_msub(M, N, ntok, 128), sms);
    if (slab() > limit) *w = plan_wgrad_tiles(&M, &N, 1, ntok, 128, 1, sms);
    if (slab() > limit) return false;
    const int max_splits = static_cast<int>(limit / slab());
    if (w->p[0].splits > max_splits) set_splits(w->p[0], max_splits);
    return true;
}

// The tile configuration dispatch() launches for a planned (bn, msub): bit 2
// set when the launch runs on CTA pairs (clusters of two, cta_group::2), bit
// 3 when one CTA runs two 128-row sub-tiles.  These are the launch-trace
// flag bits of the same meaning (include/cola.h).
constexpr int TRACE_PAIR = 4;
constexpr int TRACE_MSUB2 = 8;
constexpr int TRACE_TAIL = 16;   // weight gradients with a split tail
constexpr int TRACE_GLU = 32;    // the dX epilogue stored the gated-MLP gradients dY_gate, dY_up
constexpr int TRACE_Z = 64;      // the fused forward stored Z
constexpr int TRACE_CLUSTER = 128;   // K splits reduced inside thread-block clusters (no reduce launch)

template <bool A_MN, int EPI>
int tile_flags(int bn, int msub)
{
    constexpr bool small_only = EPI == EPI_F32 && !A_MN;   // split-K forward partials: 128-row tiles only
    if (small_only) return 0;
    if (msub == TILE_PAIR && bn == 256) return TRACE_PAIR;
    if (msub == 2 && bn == 128) return TRACE_MSUB2;
    return 0;
}

// Launch one batch (all problems of one configuration).  Programmatic
// dependent launch hides launch latency and the prologue of short GEMMs
// (measured: -8 % step time on the HBM-bound 60M block) but costs ~1 % on
// long ones, so it is used below 64 GFLOP per launch.
template <bool A_MN, bool B_MN, int EPI, int SIG>
cudaError_t dispatch_sig(int bn, int msub, GemmBatch& b, int sms, cudaStream_t s)
{
    double flops = 0.0;
    int units = 0;
    for (int g = 0; g < b.count; ++g) {
        b.prob[g].unit_begin = units;
        units += b.prob[g].p.units;
        flops += 2.0 * b.prob[g].p.M * b.prob[g].p.N * (static_cast<double>(b.prob[g].p.k_blocks) * BK);
    }
    if constexpr (EPI == EPI_TAIL) units = b.tail_body + b.tail_tiles * b.tail_pieces;
    b.units = units;
    const bool pdl = flops < 64e9;
    // the split-K forward GEMMs of small launches (K-major fp32 partials) run
    // on 128 x 128 tiles only; the gated dX GEMM on CTA pairs or on 128 x 128
    // tiles (its long-K form on pairs only)
    constexpr bool small_only = EPI == EPI_F32 && !A_MN;
    constexpr bool glu_bwd = epi_glu_bwd(EPI);
    if constexpr (!small_only && EPI != EPI_STORE64) {
        if (msub == TILE_PAIR && bn == 256) {
            const int pairs = units < sms / 2 ? units : sms / 2;
            return launch_gemm<256, 1, A_MN, B_MN, EPI, true, SIG>(b, 2 * pairs, pdl, s);
        }
    }
    // planned tiles exist as above and below only
    if (msub != 1 && (bn == 256 || small_only || glu_bwd)) return cudaErrorInvalidValue;
    const int grid = units < sms ? units : sms;
    if constexpr (glu_bwd || small_only) {
        if (bn == 256) return cudaErrorInvalidValue;
    } else {
        if (bn == 256) return launch_gemm<256, 1, A_MN, B_MN, EPI, false, SIG>(b, grid, pdl, s);
    }
    if constexpr (!small_only && !glu_bwd) {
        if (msub != 1) return launch_gemm<128, 2, A_MN, B_MN, EPI, false, SIG>(b, grid, pdl, s);
    }
    if constexpr (EPI == EPI_GLU_BWD_LONG) return cudaErrorInvalidValue;
    else return launch_gemm<128, 1, A_MN, B_MN, EPI, false, SIG>(b, grid, pdl, s);
}

// The launch of a batch whose epilogue applies sigma (EPI_ZH, EPI_DSIGMA,
// EPI_DSIGMA_H) goes to the kernel compiled for its activation (the problems
// of one batch share it); the other kinds have one kernel.
template <bool A_MN, bool B_MN, int EPI>
cudaError_t dispatch(int bn, int msub, GemmBatch& b, int sms, cudaStream_t s)
{
    if constexpr (EPI == EPI_ZH || EPI == EPI_DSIGMA || EPI == EPI_DSIGMA_H) {
        switch (b.prob[0].p.sigma) {
        case SIG_SILU: return dispatch_sig<A_MN, B_MN, EPI, SIG_SILU>(bn, msub, b, sms, s);
        case SIG_GELU: return dispatch_sig<A_MN, B_MN, EPI, SIG_GELU>(bn, msub, b, sms, s);
        case SIG_IDENTITY: return dispatch_sig<A_MN, B_MN, EPI, SIG_IDENTITY>(bn, msub, b, sms, s);
        default: return cudaErrorInvalidValue;
        }
    } else {
        return dispatch_sig<A_MN, B_MN, EPI, SIG_IDENTITY>(bn, msub, b, sms, s);
    }
}

// The gated-MLP forward launch (EPI_GLU): 256 x 256 tiles on CTA pairs (when
// `pair`), with one TMEM slot whose gate and up accumulators are handed over
// apart, or 128 x 128 tiles with two slots on single CTAs.
cudaError_t dispatch_glu(bool pair, GemmBatch& b, int sms, cudaStream_t s)
{
    b.prob[0].unit_begin = 0;
    b.units = b.prob[0].p.units;
    const GemmParams& p = b.prob[0].p;
    const bool pdl = 2.0 * p.M * p.N * (static_cast<double>(p.k_blocks) * BK) < 64e9;
    if (pair) {
        const int pairs = b.units < sms / 2 ? b.units : sms / 2;
        return launch_gemm<256, 1, false, false, EPI_GLU, true>(b, 2 * pairs, pdl, s);
    }
    return launch_gemm<128, 1, false, false, EPI_GLU>(b, b.units < sms ? b.units : sms, pdl, s);
}

}  // namespace
}  // namespace cola
