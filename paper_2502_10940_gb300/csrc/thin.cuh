// thin.cuh -- the forward GEMMs of a handful of tokens (decode; sm_103a):
//
//   D[t, m] = sum_k T[t, k] W[m, k]        t < n <= THIN_MAX_TOKENS
//
// (Z = X A^T with H = sigma(Z), Y = H B^T, and the gated product
// M = (H_gate B_gate^T) * (H_up B_up^T); Eq. (main-fwd), Fig. 4.)
//
// Such a GEMM streams its weights W once and does next to nothing with them,
// so what bounds it is the latency of getting the weight rows into the SMs
// and of finishing a split reduction.  Two things follow:
//   - The weights are the M operand (128 rows of W per tile) and the tokens the
//     N operand (n rounded up to 16): a tile's fp32 result is 128 x 16..64
//     instead of the 128 x 128 of a token-major tile that is mostly padding, so
//     the K splits of a tile, on one thread-block cluster, exchange 8 to 32 KB
//     per CTA on chip (twice that for the gated product's two halves) and no
//     reduce launch follows.
//   - Weights do not depend on the kernel before.  The second GEMM of a call
//     issues its weight loads before it waits for the first one (programmatic
//     dependent launch; every kernel of the library lets its successor start
//     only after its own wait, so what preceded the call has completed by
//     then).  The first GEMM of a call may follow any kernel of the caller's,
//     which may still be writing the weights, so it only hints them into L2.
//
// CTA s of a cluster of S accumulates the k-blocks [s kps, (s + 1) kps) of its
// tile in TMEM (lane = row of W, column = token).  The tokens are dealt out in
// bands of ceil(n / S); each CTA stages its partial token by token (128 fp32,
// so a warp's 32 lanes write 32 consecutive words), sends every owner its band
// with one bulk copy, and each owner sums its band in rank order, applies the
// epilogue and stores: deterministic, as splitk_cluster.cuh, whose exchange
// protocol (armed receive barriers, `done` signals, bounded waits that outlast
// the main loop's) this follows.
//
// Measured (graph-replayed blocks, against the token-major GEMMs with fp32 slabs
// and reduce launches): 1B-shaped, 32 tokens 57.4 -> 45.5 us (12 -> 8
// launches); 7B-shaped, 1 token 83 -> 58 us (14 -> 8), 16 tokens 82 -> 62 us.  A launch of
// the 1B-shaped o layer takes 4.5 us: 0.5 us from the wait to the first k-block,
// 0.5 us main loop, 1 us staging and exchange, 0.5 us sums and stores, 1.3 us
// until the next kernel's wait returns; 7B-shaped ones stream their weights at
// 6 to 7 TB/s between those.  More tokens summed side by side per warp (4) cost
// more in cold instructions than they save: block of 32 tokens 47 us.
//
// Warp roles (192 threads): warp 0 TMA producer, warp 1 MMA issuer (allocates
// TMEM), warps 2..5 exchange and epilogue, one per TMEM lane quarter.
#pragma once
#include "splitk_cluster.cuh"

namespace cola {

constexpr int THIN_MAX_TOKENS = 64;
constexpr int THIN_THREADS = 192;
constexpr int THIN_MAX_STAGES = 8;
constexpr int THIN_MAX_PROBS = 3;
constexpr int THIN_MAX_CLUSTER = 16;   // beyond the portable 8: opted in at launch

enum ThinKind : int { THIN_STORE = 0, THIN_ZH = 1, THIN_GLU = 2 };

struct ThinProblem {
    CUtensorMap map_w;    // W [M x K], K-major, box {64, 128} (THIN_GLU: B_gate)
    CUtensorMap map_w2;   // THIN_GLU: B_up
    int M;                // features (rows of W)
    int tile_begin;       // first batch-wide tile of this problem
    int t_x, t_x2;        // first column of the token operand (THIN_GLU: of the gate and the up half)
    __nv_bfloat16* o0;    // THIN_STORE: Y; THIN_ZH: Z or null; THIN_GLU: M
    __nv_bfloat16* o1;    // THIN_ZH: H; THIN_GLU: Y_gate or null
    __nv_bfloat16* o2;    // THIN_GLU: Y_up or null
    long long ldo;        // row pitch of the outputs
};

struct ThinBatch {
    CUtensorMap map_t;    // tokens [n x K...], K-major, box {64, NT}
    ThinProblem prob[THIN_MAX_PROBS];
    int count, tiles;
    int n, NT;            // tokens; rounded up to 16
    int k_blocks;         // of one product (THIN_GLU: of each half)
    int S, kps;           // cluster size = K splits, k-blocks per split (none empty)
    int TB;               // tokens per band = ceil(n / S)
    int stages;           // operand ring
    int early_weights;    // 1: load weights before the wait for the preceding kernel
    unsigned int* status;
    // failure-detection self-test: 1 = CTA rank 1 of the first cluster issues
    // no loads, so its MMA issuer's first wait runs out while the other CTAs
    // of the cluster complete normally
    int selftest;
};

// Dynamic shared memory: the ring (16 KB of W and NT tokens per k-block),
// which the partial is staged in afterwards, and the receive buffer.
__host__ __device__ constexpr int thin_stage_bytes(int NT) { return BM * BK * 2 + NT * BK * 2; }
__host__ __device__ constexpr int thin_ring_bytes(int stages, int NT, bool glu)
{
    const int ring = stages * thin_stage_bytes(NT), staged = NT * BM * 4 * (glu ? 2 : 1);
    return ((ring > staged ? ring : staged) + 1023) / 1024 * 1024;
}
__host__ __device__ constexpr int thin_recv_bytes(int S, int TB, bool glu) { return S > 1 ? S * TB * BM * 4 * (glu ? 2 : 1) : 0; }
constexpr int THIN_BAR_BYTES = 256;
constexpr int THIN_SMEM_BUDGET = 110 * 1024;   // two CTAs per SM (one where the gated product takes more: thin_splits)
__host__ __device__ constexpr int thin_smem_bytes(int stages, int NT, int S, int TB, bool glu)
{
    return 1024 + thin_ring_bytes(stages, NT, glu) + thin_recv_bytes(S, TB, glu) + THIN_BAR_BYTES;
}

#ifdef COLA_DEFINE_THIN_KERNEL
// Hint one box of a tensor into L2.
__device__ __forceinline__ void tma_prefetch_l2_2d(const CUtensorMap* map, int x, int y)
{
    asm volatile("cp.async.bulk.prefetch.tensor.2d.L2.global.tile [%0, {%1, %2}];" ::"l"(reinterpret_cast<uint64_t>(map)),
                 "r"(x), "r"(y)
                 : "memory");
}

__device__ __forceinline__ void thin_warps_sync() { asm volatile("bar.sync 1, 128;" ::: "memory"); }

__device__ __forceinline__ void tmem_ld_32x32b_x16(uint32_t taddr, uint32_t (&v)[16])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
          "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]),
          "=r"(v[15])
        : "r"(taddr)
        : "memory");
}

// The epilogue of four consecutive features m.. of token t: a (and a2, THIN_GLU:
// the gate and up sums).  Row pitches are multiples of 8 elements.
struct ThinOut {
    __nv_bfloat16 *o0, *o1, *o2;
    long long ldo;
    int M;
};

template <int KIND, int SIG>
__device__ __forceinline__ void thin_store(const ThinOut& P, int t, int m, const float4& a, const float4& a2)
{
    const long long off = static_cast<long long>(t) * P.ldo + m;
    auto put = [&](__nv_bfloat16* o, uint32_t lo, uint32_t hi) {
        if (m + 4 <= P.M)
            *reinterpret_cast<uint2*>(o + off) = make_uint2(lo, hi);
        else
            store_row8(o + off, make_uint4(lo, hi, 0u, 0u), P.M - m);
    };
    const uint32_t lo = pack_bf16x2(a.x, a.y), hi = pack_bf16x2(a.z, a.w);
    if (KIND == THIN_STORE) {
        put(P.o0, lo, hi);
    } else if (KIND == THIN_ZH) {   // H = bf16(sigma(bf16 Z)), as the GEMM epilogue
        if (P.o0) put(P.o0, lo, hi);
        put(P.o1, pack_bf16x2(act_sigma<SIG>(bf16_lo(lo)), act_sigma<SIG>(bf16_hi(lo))),
            pack_bf16x2(act_sigma<SIG>(bf16_lo(hi)), act_sigma<SIG>(bf16_hi(hi))));
    } else {                        // M = bf16(Y_gate * Y_up) of the rounded outputs
        const uint32_t ulo = pack_bf16x2(a2.x, a2.y), uhi = pack_bf16x2(a2.z, a2.w);
        put(P.o0, mul_bf16x2(lo, ulo), mul_bf16x2(hi, uhi));
        if (P.o1) {
            put(P.o1, lo, hi);
            put(P.o2, ulo, uhi);
        }
    }
}

constexpr int SUM_TOKENS = 2;   // of a warp's tokens summed side by side

template <int KIND, int SIG>
__global__ void __launch_bounds__(THIN_THREADS) thin_kernel(const __grid_constant__ ThinBatch b)
{
    constexpr bool GLU = KIND == THIN_GLU;
    constexpr int HALVES = GLU ? 2 : 1;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    const int NT = b.NT, S = b.S, stages = b.stages, n = b.n, TB = b.TB;
    const uint32_t stage_bytes = static_cast<uint32_t>(thin_stage_bytes(NT));
    uint8_t* recv_gen = smem + thin_ring_bytes(stages, NT, GLU);   // [half][S][band tokens][128] fp32
    const uint32_t recv = smem_u32(recv_gen);
    uint64_t* bars = reinterpret_cast<uint64_t*>(recv_gen + thin_recv_bytes(S, TB, GLU));
    uint64_t* full_bar = bars;                         // [THIN_MAX_STAGES]
    uint64_t* empty_bar = bars + THIN_MAX_STAGES;      // [THIN_MAX_STAGES]
    uint64_t* tfull = bars + 2 * THIN_MAX_STAGES;      // the partial accumulated (MMA commit)
    uint64_t* data = tfull + 1;                        // this CTA's band has arrived from every CTA
    uint64_t* done = data + 1;                         // every owner has received this CTA's bands
    uint64_t* drain_bar = done + 1;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(drain_bar + 1);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    unsigned int* const status = b.status;
    const WaitCtx wc{abort_flag, status};
    const int rank = static_cast<int>(cluster_ctarank());
    const int tile = static_cast<int>(blockIdx.x) / S;
    int g = 0;
#pragma unroll
    for (int j = 1; j < THIN_MAX_PROBS; ++j)
        if (j < b.count && tile >= b.prob[j].tile_begin) g = j;
    const ThinProblem& P = b.prob[g];
    const int m0 = (tile - P.tile_begin) * BM;
    const int kb0 = rank * b.kps;
    const int kb1 = min(kb0 + b.kps, b.k_blocks);
    const int iters = (kb1 - kb0) * HALVES;            // GLU: gate and up k-blocks in turn
    const int owners = (n + TB - 1) / TB;              // CTAs that own a token band
    auto band = [&](int p) { return max(0, min(TB, n - p * TB)); };
    const int my_tokens = band(rank);
    const int tmem_cols = HALVES * NT <= 32 ? 32 : (HALVES * NT <= 64 ? 64 : 128);
    const uint32_t tx_bytes = stage_bytes;

    auto load_w = [&](int i) {
        const int kb = kb0 + i / HALVES, s = i % stages;
        tma_load_2d(GLU && (i & 1) ? &P.map_w2 : &P.map_w, &full_bar[s], smem + s * stage_bytes, kb * BK, m0);
    };
    auto load_t = [&](int i) {
        const int kb = kb0 + i / HALVES, s = i % stages;
        tma_load_2d(&b.map_t, &full_bar[s], smem + s * stage_bytes + BM * BK * 2,
                    (GLU && (i & 1) ? P.t_x2 : P.t_x) + kb * BK, 0);
    };
    const int early = b.early_weights ? min(iters, stages) : 0;
    if (threadIdx.x == 0) {
        for (int s = 0; s < stages; ++s) {
            mbar_init(&full_bar[s], 1);
            mbar_init(&empty_bar[s], 1);
        }
        mbar_init(tfull, 1);
        mbar_init(data, 1);
        mbar_init(done, static_cast<uint32_t>(owners));
        mbar_init(drain_bar, 1);
        *abort_flag = 0;
        fence_mbar_init();
        // armed before any CTA of the cluster can send: my band from each of the S CTAs
        if (S > 1 && my_tokens > 0)
            mbar_arrive_expect_tx(data, static_cast<uint32_t>(HALVES * S * my_tokens * BM * 4));
        tma_prefetch_desc(&b.map_t);
        for (int i = 0; i < early; ++i) {
            mbar_arrive_expect_tx(&full_bar[i], tx_bytes);
            load_w(i);
        }
        if (!b.early_weights)
            for (int i = 0; i < iters; ++i)
                tma_prefetch_l2_2d(GLU && (i & 1) ? &P.map_w2 : &P.map_w, (kb0 + i / HALVES) * BK, m0);
    }
    if (warp == 1) {
        tmem_alloc(tmem_slot, static_cast<uint32_t>(tmem_cols));
        tmem_relinquish();
    }
    tc_fence_before();
    cluster_sync();   // every CTA's barriers initialised before any arrives from another
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    grid_dependency_wait();
    grid_launch_dependents();

    if (warp == 0) {
        // ------------------------------------------------ TMA producer
        if (lane == 0) {
            int issued = 0;
            const bool no_loads = b.selftest == 1 && tile == 0 && rank == 1;
            for (int i = 0; i < iters && !no_loads; ++i) {
                const int s = i % stages;
                if (i >= stages &&
                    !wait_bounded(&empty_bar[s], static_cast<uint32_t>((i / stages) - 1) & 1u, wc, ST_TIMEOUT_PRODUCER))
                    break;
                if (i >= early) {
                    mbar_arrive_expect_tx(&full_bar[s], tx_bytes);
                    load_w(i);
                }
                load_t(i);
                ++issued;
            }
            // every load has landed before the CTA can exit, also when the MMA
            // issuer gave up waiting for it
            for (int i = issued > stages ? issued - stages : 0; i < issued; ++i) {
                const uint64_t t0 = global_timer_ns();
                while (!mbar_try_wait(&full_bar[i % stages], static_cast<uint32_t>(i / stages) & 1u)) {
                    if (global_timer_ns() - t0 > WAIT_LIMIT_NS) {
                        if (status) atomicOr(status, ST_TIMEOUT_DRAIN);
                        break;
                    }
                }
            }
        }
    } else if (warp == 1) {
        // ------------------------------------------------ MMA issuer
        if (lane == 0) {
            const uint32_t idesc = idesc_bf16_f32(BM, NT, 0, 0);
            const DescWords desc_w = operand_desc<false>(smem_u32(smem)), desc_t = operand_desc<false>(smem_u32(smem) + BM * BK * 2);
            bool ok = true, issued_any = false;
            for (int i = 0; i < iters; ++i) {
                const int s = i % stages;
                if (!wait_bounded(&full_bar[s], static_cast<uint32_t>(i / stages) & 1u, wc, ST_TIMEOUT_MMA)) {
                    ok = false;
                    break;
                }
                tc_fence_after();
                const uint32_t off = (s * stage_bytes) >> 4;
                const uint32_t acc = tmem_base + static_cast<uint32_t>(GLU && (i & 1) ? NT : 0);
#pragma unroll
                for (int ks = 0; ks < BK / UMMA_K; ++ks)
                    umma_f16(acc, desc_at(desc_w.lo + off + ks * (UMMA_K * 2 >> 4), desc_w.hi),
                             desc_at(desc_t.lo + off + ks * (UMMA_K * 2 >> 4), desc_t.hi), idesc,
                             (i >= HALVES || ks > 0) ? 1u : 0u);
                issued_any = true;
                umma_commit(&empty_bar[s]);
            }
            umma_commit(tfull);
            if ((!ok || *abort_flag) && issued_any) {
                umma_commit(drain_bar);
                const uint64_t t0 = global_timer_ns();
                while (!mbar_try_wait(drain_bar, 0)) {
                    if (global_timer_ns() - t0 > WAIT_LIMIT_NS) {
                        if (status) atomicOr(status, ST_TIMEOUT_DRAIN);
                        break;
                    }
                }
            }
        }
    } else {
        // ------------------------------------------------ exchange and epilogue (warps 2..5)
        const int q = warp & 3;                  // TMEM lane quarter
        const int f = q * 32 + lane;             // this thread's feature of the tile
        const int tid = threadIdx.x - 64;
        const ThinOut out{P.o0, P.o1, P.o2, P.ldo, P.M};   // in registers before the wait
        const uint32_t tq = tmem_base + (static_cast<uint32_t>(q * 32) << 16);
        const uint32_t ring = smem_u32(smem);
        const float* src = reinterpret_cast<const float*>(S > 1 ? recv_gen : smem);   // [half][rank][token][128]
        const int step = S > 1 ? my_tokens * BM : 0;                                  // floats from rank to rank
        const int half = S > 1 ? S * step : NT * BM;                                  // floats from gate to up
        const bool acc_ok = wait_bounded(tfull, 0, wc, ST_TIMEOUT_EPILOGUE);
        tc_fence_after();
        // an accumulator this CTA gave up on sends zeros (tcgen05.ld is warp-wide)
        const bool use_acc = __all_sync(0xffffffffu, acc_ok && !*abort_flag);
        // stage the partial in the (idle) ring: token by token, 128 fp32 each
#pragma unroll 1
        for (int h = 0; h < HALVES; ++h) {
#pragma unroll 1
            for (int t0 = 0; t0 < n; t0 += 16) {
                uint32_t v[16];
                if (use_acc) {
                    tmem_ld_32x32b_x16(tq + static_cast<uint32_t>(h * NT + t0), v);
                    tmem_ld_wait();
                } else {
#pragma unroll
                    for (int j = 0; j < 16; ++j) v[j] = 0u;
                }
#pragma unroll
                for (int j = 0; j < 16; ++j)
                    asm volatile("st.shared.b32 [%0], %1;" ::"r"(ring + static_cast<uint32_t>(((h * NT + t0 + j) * BM + f) * 4)),
                                     "r"(v[j])
                                     : "memory");
            }
        }
        tc_fence_before();
        if (S > 1) fence_proxy_async_smem();   // the staged partial visible to the copy engine
        thin_warps_sync();
        bool dok = use_acc;
        if (S > 1) {
            if (tid < owners) {
                // this CTA's part of band `tid` into slot `rank` of its owner
                const uint32_t bytes = static_cast<uint32_t>(band(tid) * BM * 4);
#pragma unroll
                for (int h = 0; h < HALVES; ++h)
                    bulk_copy_to_cluster(mapa_shared(recv + static_cast<uint32_t>(h * S + rank) * bytes, static_cast<uint32_t>(tid)),
                                         ring + static_cast<uint32_t>((h * NT + tid * TB) * BM * 4), bytes,
                                         mapa_shared(smem_u32(data), static_cast<uint32_t>(tid)));
            }
            if (my_tokens > 0) {
                dok = exchange_wait(data, 2 * WAIT_LIMIT_NS, status);
                // every copy into this CTA has landed: tell each sender that its band has been read
                if (tid < S) mbar_arrive_cluster_relaxed(mapa_shared(smem_u32(done), static_cast<uint32_t>(tid)));
            }
        }
        if (dok && !*abort_flag && m0 + 4 * lane < out.M) {
            // four features a thread; a warp takes every fourth token, SUM_TOKENS
            // of them at a time; the partials in rank order
#pragma unroll 1
            for (int t = warp - 2; t < my_tokens; t += 4 * SUM_TOKENS) {
                float4 a[HALVES][SUM_TOKENS];
#pragma unroll
                for (int h = 0; h < HALVES; ++h)
#pragma unroll
                    for (int j = 0; j < SUM_TOKENS; ++j) a[h][j] = make_float4(0.f, 0.f, 0.f, 0.f);
                const float* at = src + t * BM + 4 * lane;
#pragma unroll 2
                for (int s = 0; s < S; ++s, at += step) {
#pragma unroll
                    for (int h = 0; h < HALVES; ++h)
#pragma unroll
                        for (int j = 0; j < SUM_TOKENS; ++j) {
                            if (t + 4 * j < my_tokens) {
                                const float4 v = *reinterpret_cast<const float4*>(at + h * half + 4 * j * BM);
                                a[h][j].x += v.x;
                                a[h][j].y += v.y;
                                a[h][j].z += v.z;
                                a[h][j].w += v.w;
                            }
                        }
                }
#pragma unroll
                for (int j = 0; j < SUM_TOKENS; ++j)
                    if (t + 4 * j < my_tokens)
                        thin_store<KIND, SIG>(out, rank * TB + t + 4 * j, m0 + 4 * lane, a[0][j], a[HALVES - 1][j]);
            }
        }
        // the bands this CTA sent have been read by their owners: its staging may
        // go away with it
        if (S > 1 && tid == 0) exchange_wait(done, 3 * WAIT_LIMIT_NS, status);
    }

    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem_base, static_cast<uint32_t>(tmem_cols));
    }
}
#endif  // COLA_DEFINE_THIN_KERNEL

}  // namespace cola
