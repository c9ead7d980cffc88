// e4m3 decode kernel for slices of 33..128 heads: a CLUSTER OF TWO CTAs per KV worker that
// issues its MMAs with tcgen05 cta_group::2.  H = 64 or 32 heads per CTA.
//
// Why pairs: with both operands in shared memory a small MMA costs what its operands cost to
// stream ((A + B bytes) / 128 B per cycle).  Two independent CTAs each stream every
// K row and every V row themselves.  A CTA pair shares them.  A "supertile" is two consecutive
// page tiles of a segment; each CTA supplies ONE page (64 tokens) as its half of the B operand.
// bf16 x e4m3 is not an MMA type pair, so q (one scale per head) and P are each split into two
// 8-bit terms, hi + lo:
//
//   H = 64:  S [128 heads x 128 tokens]  = q hi K^T + q lo K^T    M = 128 (64 heads per CTA), N = 128, 36 MMAs of K = 32
//            O [128 heads x 256 dv]     += P hi V + P lo V        M = 128, N = 256 (x 2 halves of dv): each CTA supplies
//                                                                  its 64 heads of P and 128 of the 256 dv columns
//   H = 32:  the same shapes, but the two terms are ROWS of one A operand (16 hi rows and the 16 lo rows of the same
//            heads in turn: a TMEM lane quadrant holds both terms of its heads), half as many MMAs:
//            S [(hi, lo) x 64 heads x 128 tokens] = [q hi; q lo] K^T,  O [(hi, lo) x 64 heads x 256 dv] += [P hi; 16 P lo] V
//            the softmax adds the two halves of a logit, the epilogue hi + lo / 16
//
// so per 128 tokens and per CTA the tensor cores read 72 + 96 KB (H = 64) or 36 + 48 KB (H = 32).
// CTA r loads page r
// (all 9 chunks of 64 columns) into a stage for QK^T.  For P.V CTA r supplies dv columns
// [256 n + 128 r, + 128) of BOTH pages, at the same shared-memory offsets in both CTAs (the
// two CTAs of an MMA share one descriptor).  Its own page already has them in chunk slots
// 4 n + 2 r, 4 n + 2 r + 1 of the stage; the other four latent chunk slots of the stage hold
// columns only the peer needs, so once QK^T of the stage has retired they are overwritten
// with the peer page's chunks 4 n + 2 r, 4 n + 2 r + 1.  The MMAs over page g then start at
// slot 4 n + 2 g in both CTAs.  That second load hides behind the softmax of the supertile.
// Accumulators: CTA r holds its 64 rows; row i is TMEM lane i (tokens / dv of the
// first half of N) and lane 64 + i (second half).
//
// Roles per CTA (512 threads): K-page + scale producer, QK^T issuer and P.V issuer
// (leader CTA only), 8 softmax warps, 4 query converters, 1 producer of the peer chunks.
// An issuer warp stays converged and one elected lane issues: what the MMAs take is the same in all lanes then and lives
// in uniform registers.  Issued from a branch that lane 0 alone takes, an MMA costs 65 to 90 cycles, because every
// descriptor has to be moved there first; converged, 35 to 48, and one warp does what took two.
// Barriers that the issuers wait on live in the leader; the peer's warps arrive on them across
// the cluster (relaxed arrivals: what they announce is already in place on the peer's SM), and
// TMA loads of the peer complete on them too.
// The query rows come by TMA once the last QK^T of the request before has read their predecessors, and are split in place.
#include "splash_fp8.cuh"
#include "splash_pair.cuh"

namespace splash {

namespace {

using namespace umma;

constexpr int kIssuerWarps = 2, kSoftmaxWarps = 8, kConvertWarps = 4;
constexpr int kWarpProducer = 0;
constexpr int kWarpQk = 1;
constexpr int kWarpPv = 2;
constexpr int kWarpSoftmax = kWarpQk + kIssuerWarps;
constexpr int kWarpConvert = kWarpSoftmax + kSoftmaxWarps;
constexpr int kWarpVProducer = kWarpConvert + kConvertWarps;
constexpr int kThreads = (kWarpVProducer + 1) * 32;    // 16 warps = 512 threads
constexpr uint32_t kSlab = 64 * 64;                 // 64 rows x 64 B
constexpr uint32_t kPageBytes = 9 * kSlab;          // 36,864
constexpr uint32_t kPeerBytes = 4 * kSlab;          // the peer page's chunks this CTA multiplies: 16,384
constexpr uint32_t kScaleBytes = 256;
constexpr int kPrefetchAhead = 1;                    // supertiles between the L2 prefetch of a page and its use (4: 1.5 % slower; none: 5 %)
constexpr float kTau = 7.0f;                          // (6 / 2.75: 0.3 % slower on the rollout workload, 4 / 4.75 more)
constexpr float kLift = 1.75f;

// H = 64: three stages are what shared memory holds beside 73,728 B of query operands; H = 32: four.
template <int H>
struct Layout {
    static constexpr int kStages = H == 64 ? 3 : 4;
    enum BarrierId {
        kBarKFull = 0,                        // [stages] leader: both CTAs' pages landed (tx bytes of both)
        kBarQkDone = kBarKFull + kStages,     // [stages] QK^T of the stage retired (multicast commit): peer chunks may land
        kBarVFull = kBarQkDone + kStages,     // [stages] leader: both CTAs' peer chunks landed
        kBarStageEmpty = kBarVFull + kStages, // [stages] P.V of the stage retired (multicast commit): stage, its scales and
                                              //     the P buffer are free, O is up to date
        kBarScFull = kBarStageEmpty + kStages,// [stages] local: scale pages of the stage landed
        kBarQRaw = kBarScFull + kStages,      // local: the request's query rows landed
        kBarQFull,                            // leader: query operands of both CTAs written
        kBarQLocal,                           // local: this CTA's query scales written
        kBarQEmpty,                           // last QK^T of the request retired (multicast commit)
        kBarQsRead,                           // local: the softmax warps have picked up the request's query scales
        kBarSFull,                            // [2] S buffer written (multicast commit)
        kBarSEmpty = kBarSFull + 2,           // [2] S buffer read (leader: by both CTAs)
        kBarPFull = kBarSEmpty + 2,           // [2] P buffer written (leader: by both CTAs)
        kBarOFull = kBarPFull + 2,            // last P.V of the request retired (multicast commit)
        kBarOEmpty,                           // O drained (leader: by both CTAs)
        kNumBarriers
    };
    // query operand: 9 chunk slabs of 2 H rows x 64 B, eight hi rows and the same heads' eight lo rows in turn (QueryRows).  H = 64: two
    // operands, 1,024 bytes from one group of eight rows to the next; H = 32: one
    static constexpr uint32_t kQSlab = 2 * H * 64;
    static constexpr uint32_t kPTerm = H == 64 ? 2 * kSlab : 16 * 64;        // from a head's hi row of P to its lo row
    static constexpr uint32_t kPBuf = H == 64 ? 4 * kSlab : 2 * kSlab;
    static constexpr uint32_t kOffK = 0;                            // [stages] 9 chunk slots
    static constexpr uint32_t kOffQ = kOffK + kStages * kPageBytes;
    static constexpr uint32_t kOffP = kOffQ + 2 * H * kDQK;         // [2 buffers] ([hi, lo]) [2 page slabs] x 4096
    static constexpr uint32_t kOffScale = kOffP + 2 * kPBuf;        // float [stages][2 pages][64]
    static constexpr uint32_t kOffQs = kOffScale + kStages * 2 * kScaleBytes;    // float [4][H]
    static constexpr uint32_t kOffAlpha = kOffQs + 4 * H * 4;       // float [H]
    static constexpr uint32_t kOffL = kOffAlpha + H * 4;            // float [H]
    static constexpr uint32_t kOffXch = kOffL + H * 4;              // float [H][4]
    static constexpr uint32_t kTokBytes = 32 * 8 + 32 * 4;          // per warp: (scale, log2 scale) x 32, 1 / scale x 32
    static constexpr uint32_t kOffTok = kOffXch + H * 16;
    static constexpr uint32_t kOffBar = kOffTok + kSoftmaxWarps * kTokBytes;
    static constexpr uint32_t kOffMisc = (kOffBar + kNumBarriers * 8 + 15) / 16 * 16;
    static constexpr uint32_t kOffPlan = kOffMisc + 32;             // inline plan
    static constexpr uint32_t kSmemBytes = kOffPlan + kInlinePlanBytes;
    static_assert(kSmemBytes <= 232448, "shared memory overflow");
    static_assert(kOffQ % 1024 == 0 && kOffP % 1024 == 0 && kOffTok % 16 == 0 && kTokBytes % 16 == 0, "alignment");
    // tensor memory: O two halves of dv x 128 columns, then 2 S buffers x 64 columns
    static constexpr uint32_t kColO = 0, kColS = 256;
};

// Issued by the elected lane of a converged warp; the operands are uniform.  `a_at`, `b_at`: 16-byte units added to the descriptors'
// addresses.  Only the low words of the descriptors move with them, and what they start from is said to be uniform: with 64-bit sums, and
// addresses that only happen to be the same in all lanes, an issuer is slower than the tensor pipe (this alone, 128 heads: 150 requests of
// 6,000 tokens 306 and 248 us, one of 500,000 166 and 129, 512 rollout requests 720 and 577; 64 heads, half the MMAs: no difference).
__device__ __forceinline__ void umma_e4m3_pair(uint32_t elected, uint32_t d_tmem, uint64_t a_desc, uint32_t a_at, uint64_t b_desc, uint32_t b_at, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t.reg .b64 a, b;\n\t"
        "setp.ne.b32 p, %6, 0;\n\t"
        "setp.ne.b32 q, %7, 0;\n\t"
        "mov.b64 a, {%1, %2};\n\t"
        "mov.b64 b, {%3, %4};\n\t"
        "@q tcgen05.mma.cta_group::2.kind::f8f6f4 [%0], a, b, %5, p;\n\t}"
        ::"r"(d_tmem), "r"((uint32_t)a_desc + a_at), "r"((uint32_t)(a_desc >> 32)), "r"((uint32_t)b_desc + b_at), "r"((uint32_t)(b_desc >> 32)),
          "r"(idesc), "r"(accumulate), "r"(elected) : "memory");
}

template <int H>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kThreads, 1)
decode_umma_fp8_pair_kernel(const __grid_constant__ DecodeParams p, const __grid_constant__ CUtensorMap tmap_page,
                            const __grid_constant__ CUtensorMap tmap_pair, const __grid_constant__ CUtensorMap tmap_out,
                            const __grid_constant__ CUtensorMap tmap_part, const __grid_constant__ CUtensorMap tmap_q) {
    using L = Layout<H>;
    constexpr int kStages = L::kStages;
    extern __shared__ __align__(1024) uint8_t smem[];
    const uint32_t sbase = smem_u32(smem);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t rank = cluster_ctarank();             // 0 = leader: issues the MMAs
    const int pair_id = blockIdx.x >> 1;                // CTA pair: (KV worker, group of 2 H heads)
    const int worker = pair_id / p.pair_groups;
    const int head0 = p.head_begin + (pair_id % p.pair_groups) * (2 * H) + (int)rank * H;
    const int h = p.head_end - p.head_begin;

    volatile uint32_t *misc = reinterpret_cast<volatile uint32_t *>(smem + L::kOffMisc);
    Ctx ctx{misc + 1, p.status};
    auto bar = [&](int id) -> uint32_t { return sbase + L::kOffBar + 8u * (uint32_t)id; };
    auto leader_bar = [&](int id) -> uint32_t { return map_to_cta(sbase + L::kOffBar + 8u * (uint32_t)id, 0); };
    // one arrival of a warp of either CTA on a barrier that lives in the leader
    auto arrive_on_leader = [&](int id) {
        if (rank == 0) mbar_arrive(bar(id));
        else mbar_arrive_cluster_relaxed(leader_bar(id));
    };

    if (tid == 0) {
        // barriers the leader's issuers wait on count the warps of both CTAs (the peer's copies are unused)
        for (int s = 0; s < kStages; ++s) {
            mbar_init(bar(L::kBarKFull + s), 1); mbar_init(bar(L::kBarQkDone + s), 1);
            mbar_init(bar(L::kBarVFull + s), 1); mbar_init(bar(L::kBarStageEmpty + s), 1);
            mbar_init(bar(L::kBarScFull + s), 1);
        }
        mbar_init(bar(L::kBarQRaw), 1);
        mbar_init(bar(L::kBarQFull), 2 * kConvertWarps); mbar_init(bar(L::kBarQLocal), kConvertWarps); mbar_init(bar(L::kBarQEmpty), 1);
        mbar_init(bar(L::kBarQsRead), kSoftmaxWarps);
        for (int b = 0; b < 2; ++b) {
            mbar_init(bar(L::kBarSFull + b), 1); mbar_init(bar(L::kBarSEmpty + b), 2 * kSoftmaxWarps);
            mbar_init(bar(L::kBarPFull + b), 2 * kSoftmaxWarps);
        }
        mbar_init(bar(L::kBarOFull), 1); mbar_init(bar(L::kBarOEmpty), 2 * kSoftmaxWarps);
        misc[1] = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(sbase + L::kOffMisc), "r"(512u) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    tcgen05_fence_before();
    __syncthreads();
    cluster_sync_all();                                   // barriers of both CTAs exist before anyone signals them
    tcgen05_fence_after();
    const uint32_t tmem_base = misc[0];
    SegmentIter<L::kOffPlan> it;
    start_plan<false>(p, worker, kThreads / 32 - 1, it, FirstLoads{kPageBytes, 0u, kPageBytes, kStages, head0, H});
    const long long t_start = clock64();
    const unsigned long long ns_start = global_timer_ns();

    Segment seg;
    seg.lo = seg.hi = seg.tile_begin = seg.tile_end = 0;
    // geometry of supertile s of the current segment: page tiles 2s (page A, CTA 0) and 2s + 1 (page B, CTA 1)
    auto pair_geom = [&](int s) -> PairGeom {
        PairGeom g;
        const int first_page = seg.lo / kPage;
        const int ta = seg.tile_begin + 2 * s, tb = ta + 1;
        g.a = tile_geom(seg.lo, seg.hi, (first_page + ta) * kPage);
        g.has_b = tb < seg.tile_end;
        if (g.has_b) g.b = tile_geom(seg.lo, seg.hi, (first_page + tb) * kPage);
        else { g.b.tok0 = 0; g.b.r_lo = 0; g.b.r_hi = 0; g.b.a = 0; g.b.b = 0; g.b.both = false; }
        return g;
    };

    if (warp == kWarpProducer || warp == kWarpVProducer) {
        // ===================================================== TMA producers
        // warp 0: this CTA's page and the scale pages of both pages, up to three supertiles ahead;
        // last warp: the peer page's chunks, into the dead half of the stage once QK^T has read it
        const bool is_v = warp == kWarpVProducer;
        uint32_t st_it = 0;                               // supertile counter
        bool ok = true;
        while (ok && it.next(p, seg)) {
            const int first_page = seg.lo / kPage;
            const int32_t *table = p.block_table + (int64_t)seg.request * p.table_stride;
            const int nsuper = (seg.tile_end - seg.tile_begin + 1) >> 1;
            for (int s = 0; ok && s < nsuper; ++s, ++st_it) {
                const PairGeom g = pair_geom(s);
                const int ta = seg.tile_begin + 2 * s;
                const uint32_t stage = st_it % kStages, ph = (st_it / kStages) & 1;
                const uint32_t k0 = sbase + L::kOffK + stage * kPageBytes;
                // the page this warp fetches: its CTA's own for QK^T, the other CTA's for the P.V chunks.  A tile cut at
                // both ends inside its page is written by hand instead (zeros outside the range); only a request whose
                // whole range lies inside one page has such a tile, and it is page A.
                const TileGeom &tg = (rank == 0) != is_v ? g.a : g.b;
                int page_a = 0, page_b = 0;
                if (lane == 0) {
                    page_a = table[first_page + ta];
                    page_b = g.has_b ? table[first_page + ta + 1] : p.num_pool_pages;   // a page past the pool reads as zeros
                    if (!is_v) {
                        ok = mbar_wait(ctx, bar(L::kBarStageEmpty + stage), ph ^ 1, L::kBarStageEmpty + stage);
                        if (ok) {
                            // the leader's barrier expects the pages of both CTAs
                            if (rank == 0) mbar_expect_tx(bar(L::kBarKFull + stage), 2 * kPageBytes);
                            if (!tg.both)
                                tma_load_4d_pair(k0, &tmap_page, leader_bar(L::kBarKFull + stage), 0, tg.tok0, 0, rank == 0 ? page_a : page_b);
                            // scale pages of both pages, for this CTA's softmax warps
                            const bool in_a = page_a >= 0 && page_a < p.num_pool_pages;
                            const bool in_b = g.has_b && page_b >= 0 && page_b < p.num_pool_pages;
                            if (!in_a || (g.has_b && !in_b)) {     // a page outside the pool reads as zeros; give its tokens the scale 1
                                float *sc1 = reinterpret_cast<float *>(smem + L::kOffScale + stage * 2 * kScaleBytes);
                                for (int t = 0; t < kPage; ++t) {
                                    if (!in_a) sc1[t] = 1.0f;
                                    if (g.has_b && !in_b) sc1[kPage + t] = 1.0f;
                                }
                            }
                            mbar_expect_tx(bar(L::kBarScFull + stage), (in_a ? kScaleBytes : 0u) + (in_b ? kScaleBytes : 0u));
                            const uint32_t sdst = sbase + L::kOffScale + stage * 2 * kScaleBytes;
                            if (in_a) bulk_load(sdst, p.kv_scales + (int64_t)page_a * kPage, kScaleBytes, bar(L::kBarScFull + stage));
                            if (in_b) bulk_load(sdst + kScaleBytes, p.kv_scales + (int64_t)page_b * kPage, kScaleBytes, bar(L::kBarScFull + stage));
                            // A stage is held from its load until P.V has read it, about three supertiles, so the
                            // load of supertile s + 3 starts only when the issuers are about to need it: have its
                            // page in L2 by then.
                            const int tf = ta + 2 * kPrefetchAhead + (int)rank;
                            if (tf < seg.tile_end) {
                                const int page_f = table[first_page + tf];
                                if (page_f >= 0 && page_f < p.num_pool_pages) tma_prefetch_4d(&tmap_page, 0, 0, 0, page_f);
                            }
                        }
                    } else {
                        ok = mbar_wait(ctx, bar(L::kBarQkDone + stage), ph, L::kBarQkDone + stage);
                        if (ok) {
                            if (rank == 0) mbar_expect_tx(bar(L::kBarVFull + stage), 2 * kPeerBytes);
                            // peer page chunks 4n + 2 rank, + 1 -> slots 4n + 2 (1 - rank), + 1
                            if (!tg.both) {
#pragma unroll
                                for (int n = 0; n < 2; ++n)
                                    tma_load_4d_pair(k0 + (4 * n + 2 * (1 - (int)rank)) * kSlab, &tmap_pair, leader_bar(L::kBarVFull + stage), 0,
                                                     tg.tok0, 4 * n + 2 * (int)rank, rank == 0 ? page_b : page_a);
                            }
                        }
                    }
                }
                ok = __shfl_sync(0xffffffffu, ok ? 1 : 0, 0) != 0;
                if (ok && tg.both) {
                    const int page = __shfl_sync(0xffffffffu, (rank == 0) != is_v ? page_a : page_b, 0);
                    const uint8_t *src = page >= 0 && page < p.num_pool_pages
                        ? static_cast<const uint8_t *>(p.kv_pool) + (size_t)page * (kPage * kDQK) : nullptr;
                    uint8_t *slabs = smem + L::kOffK + stage * kPageBytes;
                    if (!is_v) {
                        fill_rows_by_hand<64>(slabs, kSlab, kPage, src, tg.tok0, tg.a, tg.b, 0, 0, 9, lane);
                    } else {
                        for (int n = 0; n < 2; ++n)
                            fill_rows_by_hand<64>(slabs, kSlab, kPage, src, tg.tok0, tg.a, tg.b, 4 * n + 2 * (int)rank,
                                                  4 * n + 2 * (1 - (int)rank), 2, lane);
                    }
                    fence_proxy_async();
                    __syncwarp();
                    if (lane == 0) mbar_complete_tx_cluster(leader_bar(is_v ? L::kBarVFull + stage : L::kBarKFull + stage), is_v ? kPeerBytes : kPageBytes);
                }
            }
        }
    } else if (warp == kWarpQk && rank == 0) {
        // ===================================================== QK^T issuer (leader CTA)
        constexpr uint32_t kIdescQK = make_idesc_e4m3(128, 128, 0);
        const uint32_t elected = elect_one(), tmem_u = uniform(tmem_base);
        uint32_t st_it = 0, seg_it = 0;
        bool ok = true;
        while (ok && it.next(p, seg)) {
            const int nsuper = (int)uniform((uint32_t)((seg.tile_end - seg.tile_begin + 1) >> 1));
            mbar_wait_cluster(ctx, bar(L::kBarQFull), seg_it & 1, L::kBarQFull);       // (its answer goes unused: past a wait that gave up nothing counts, and a wait below ends the walk)
            for (int s = 0; ok && s < nsuper; ++s, ++st_it) {
                const uint32_t stage = st_it % kStages, b = st_it & 1;
                ok = mbar_wait_cluster(ctx, bar(L::kBarKFull + stage), (st_it / kStages) & 1, L::kBarKFull + stage) &&
                     mbar_wait_cluster(ctx, bar(L::kBarSEmpty + b), ((st_it >> 1) & 1) ^ 1, L::kBarSEmpty + b);
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) break;
                tcgen05_fence_after();
                const uint32_t d = uniform(tmem_u + L::kColS + b * 64);
                const uint64_t dq = make_desc_sw64(uniform(sbase + L::kOffQ), 16, H == 64 ? 1024 : 512);           // A: 2 x 64 rows x 32
                const uint64_t dk = make_desc_sw64(uniform(sbase + L::kOffK + stage * kPageBytes), 16, 512);       // B: 2 x 64 tokens x 32
                // 18 K = 32 steps, for H = 64 with q hi and then with q lo
#pragma unroll
                for (int t = 0; t < (H == 64 ? 36 : 18); ++t) {
                    const uint32_t ks = t % 18, at = (ks >> 1) * kSlab + (ks & 1) * 32, at_q = (ks >> 1) * L::kQSlab + (ks & 1) * 32;
                    umma_e4m3_pair(elected, d, dq, ((t / 18) * 512 + at_q) >> 4, dk, at >> 4, kIdescQK, t != 0);
                }
                if (elected) { umma_commit_pair(bar(L::kBarSFull + b)); umma_commit_pair(bar(L::kBarQkDone + stage)); }
                __syncwarp();
            }
            if (ok && elected) umma_commit_pair(bar(L::kBarQEmpty));
            __syncwarp();
            ++seg_it;
        }
    } else if (warp == kWarpPv && rank == 0) {
        // ===================================================== P.V issuer (leader CTA)
        constexpr uint32_t kIdescPV = make_idesc_e4m3(128, 256, 0, 0, 1, 0);
        constexpr uint32_t kIdescPVLo = make_idesc_e4m3(128, 256, 0, 0, 1, 1);   // P lo is e5m2 (A operand; H = 64)
        const uint32_t elected = elect_one(), tmem_u = uniform(tmem_base);
        uint32_t st_it = 0, seg_it = 0;
        bool ok = true;
        while (ok && it.next(p, seg)) {
            const int ntiles = (int)uniform((uint32_t)(seg.tile_end - seg.tile_begin));
            const int nsuper = (ntiles + 1) >> 1;
            for (int s = 0; ok && s < nsuper; ++s, ++st_it) {
                const uint32_t stage = st_it % kStages, pb = st_it & 1;
                ok = mbar_wait_cluster(ctx, bar(L::kBarVFull + stage), (st_it / kStages) & 1, L::kBarVFull + stage) &&
                     mbar_wait_cluster(ctx, bar(L::kBarPFull + pb), (st_it >> 1) & 1, L::kBarPFull + pb);
                if (ok && s == 0) ok = mbar_wait_cluster(ctx, bar(L::kBarOEmpty), (seg_it & 1) ^ 1, L::kBarOEmpty);
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) break;
                tcgen05_fence_after();
                const int pages = 2 * s + 1 < ntiles ? 2 : 1;     // page B's MMAs are skipped when it does not exist
                // A: P rows, slab = page, 32 tokens; B: slots 4n + 2 page, + 1 (two 64-wide dv chunks, LBO), 32 tokens
                const uint64_t da = make_desc_sw64(uniform(sbase + L::kOffP + pb * L::kPBuf), 16, 512);
                const uint64_t db = make_desc_sw64(uniform(sbase + L::kOffK + stage * kPageBytes), kSlab, 512);
#pragma unroll
                for (int hl = 0; hl < (H == 64 ? 2 : 1); ++hl) {
                    for (int pg = 0; pg < pages; ++pg) {
#pragma unroll
                        for (int k = 0; k < 2; ++k) {
#pragma unroll
                            for (int n = 0; n < 2; ++n)           // dv half: columns [256 n, 256 n + 256)
                                umma_e4m3_pair(elected, tmem_u + L::kColO + n * 128, da, (hl * L::kPTerm + pg * kSlab + k * 32) >> 4,
                                               db, ((4 * n + 2 * pg) * kSlab + k * 2048) >> 4, hl ? kIdescPVLo : kIdescPV,
                                               (uint32_t)s | (uint32_t)(hl | pg | k));
                        }
                    }
                }
                if (elected) {
                    umma_commit_pair(bar(L::kBarStageEmpty + stage));
                    if (s + 1 == nsuper) umma_commit_pair(bar(L::kBarOFull));
                }
                __syncwarp();
            }
            ++seg_it;
        }
    } else if (warp >= kWarpQk && warp < kWarpSoftmax) {
        // (the issuer warps of the peer CTA have nothing to do)
    } else if (warp >= kWarpConvert && warp < kWarpConvert + kConvertWarps) {
        // ===================================================== query converters (this CTA's heads)
        using Rows = QueryRows<H, kConvertWarps>;
        const int cw = warp - kWarpConvert;
        float *qs_s = reinterpret_cast<float *>(smem + L::kOffQs);
        uint32_t seg_it = 0;
        bool ok = true;
        while (ok && it.next(p, seg)) {
            {
                // the operand buffer is free once the last QK^T of the previous request has retired
                // (the rows asked into L2 here, in front of the wait: 300 requests of 64 to 500 tokens 0.8 to 1.4 % slower, no call faster)
                Rows rows(smem + L::kOffQ, cw, lane);
                if (p.q_by_hand) {
                    ok = warp_wait(ctx, bar(L::kBarQEmpty), (seg_it & 1) ^ 1, L::kBarQEmpty);
                    if (!ok) break;
                    rows.copy_by_hand(static_cast<const uint16_t *>(p.q) + (int64_t)seg.request * p.q_stride_request + (int64_t)head0 * p.q_stride_head,
                                      p.q_stride_head, p.head_end - head0, lane);
                } else {
                    if (cw == 0) {
                        if (lane == 0) {
                            ok = mbar_wait(ctx, bar(L::kBarQEmpty), (seg_it & 1) ^ 1, L::kBarQEmpty);
                            if (ok) {
                                mbar_expect_tx(bar(L::kBarQRaw), Rows::kBytes);
                                tma_load_4d(sbase + L::kOffQ, &tmap_q, bar(L::kBarQRaw), 0, head0, 0, seg.request);
                            }
                        }
                        ok = __shfl_sync(0xffffffffu, ok ? 1 : 0, 0) != 0;
                        if (!ok) break;
                    }
                    ok = warp_wait(ctx, bar(L::kBarQRaw), seg_it & 1, L::kBarQRaw);
                    if (!ok) break;
                }
                const float amax = rows.largest();
                if (rows.part == 0) qs_s[(seg_it & 3) * H + rows.row] = amax > 0.f ? amax * (1.0f / 448.0f) : 1.0f;
                rows.split(amax > 0.f ? 448.0f / amax : 1.0f);
                fence_proxy_async();
                __syncwarp();
                // The softmax warps wait on QLocal by phase parity, so it must never complete two phases
                // ahead of them: hold this request's arrival until they have entered the previous one.
                if (lane == 0) {
                    if (seg_it > 0) ok = mbar_wait(ctx, bar(L::kBarQsRead), (seg_it - 1) & 1, L::kBarQsRead);
                    mbar_arrive(bar(L::kBarQLocal)); arrive_on_leader(L::kBarQFull);
                }
                ok = __shfl_sync(0xffffffffu, ok ? 1 : 0, 0) != 0;
            }
            ++seg_it;
        }
    } else if constexpr (H == 64) {
        // ===================================================== softmax + epilogue warps
        // S layout per CTA: TMEM lane L < 64 = head L, tokens of page A in 64 columns;
        // lane 64 + L = head L, tokens of page B.  Two warps per quadrant take 32 columns each,
        // so a thread owns ONE head and 32 tokens of one page.
        const int sw = warp - kWarpSoftmax;             // 0..7
        const int q4 = warp & 3;                        // TMEM lane quadrant
        const int cf = sw >> 2;                         // column half: tokens [32 cf, 32 cf + 32) of the page
        const int pg = q4 >> 1;                         // 0: page A, 1: page B
        const int hd = 32 * (q4 & 1) + lane;            // this thread's head (0..63 within the CTA)
        const int half_id = q4 & 1;                     // heads 0-31 or 32-63: the four warps that share them sync on bar 2 + half_id
        const uint32_t lane_addr = (uint32_t)(32 * q4) << 16;
        float *qs_s = reinterpret_cast<float *>(smem + L::kOffQs);
        float *alpha_s = reinterpret_cast<float *>(smem + L::kOffAlpha);
        float *l_s = reinterpret_cast<float *>(smem + L::kOffL);
        float *xch = reinterpret_cast<float *>(smem + L::kOffXch);
        // per-warp table of its 32 tokens, read back as 16-byte broadcasts:
        // tok_a[j / 2] = (scale_j, log2 scale_j, scale_j+1, log2 scale_j+1), tok_r[j / 4] = 1 / scale of four tokens
        float4 *tok_a = reinterpret_cast<float4 *>(smem + L::kOffTok + sw * L::kTokBytes);
        float4 *tok_r = tok_a + 16;
        const float *scale_s = reinterpret_cast<const float *>(smem + L::kOffScale);
        const float scale_log2 = p.softmax_scale * kLog2e;
        const int slot4 = pg * 2 + cf;                  // this thread's slot among the 4 threads of its head
        uint32_t st_it = 0, seg_it = 0;
        // A failed (timed-out) wait only clears `ok`; the role keeps walking its supertiles so that every
        // thread still meets the named barriers -- once the CTA aborts, waits return at once.
        bool ok = true;
        while (it.next(p, seg)) {
            ok &= mbar_wait(ctx, bar(L::kBarQLocal), seg_it & 1, L::kBarQLocal);
            const float cq = scale_log2 * qs_s[(seg_it & 3) * H + hd];
            __syncwarp();
            if (lane == 0) mbar_arrive(bar(L::kBarQsRead));
            float m = -INFINITY, l = 0.f;
            const int nsuper = (seg.tile_end - seg.tile_begin + 1) >> 1;
            // several query rows per request: this thread's (virtual) head is row (head mod R) and sees the
            // tokens below causal_end only
            const int causal_end = p.q_rows > 1 ? p.seq_lens[seg.request] - (p.q_rows - 1 - (head0 + hd) % p.q_rows) : 0x3fffffff;   // (far above any token index, and safe to subtract a negative offset from)
            for (int s = 0; s < nsuper; ++s, ++st_it) {
                const PairGeom g = pair_geom(s);
                const TileGeom geo = pg ? g.b : g.a;
                const uint32_t stage = st_it % kStages, b = st_it & 1;
                ok &= mbar_wait(ctx, bar(L::kBarSFull + b), (st_it >> 1) & 1, L::kBarSFull + b);
                ok &= mbar_wait(ctx, bar(L::kBarScFull + stage), (st_it / kStages) & 1, L::kBarScFull + stage);
                tcgen05_fence_after();
                float sv[32];
                {
                    tmem_ld32(tmem_base + lane_addr + L::kColS + b * 64 + 32 * cf, sv);
                    // meanwhile: lane j prepares token 32 cf + j.  A token outside the range gets scale 0 and
                    // log2 scale -inf; its row of K may hold anything, so its logit is also forced below.
                    const int r = 32 * cf + lane;
                    const bool v = r >= geo.r_lo && r < geo.r_hi;
                    const float ts = v ? scale_s[(stage * 2 + pg) * 64 + geo.tok0 + r] : 0.f;
                    reinterpret_cast<float2 *>(tok_a)[lane] = make_float2(ts, v ? fast_log2(ts) : -INFINITY);
                    reinterpret_cast<float *>(tok_r)[lane] = v ? fast_rcp(ts) : 0.f;
                    tmem_wait_ld();
                }
                tcgen05_fence_before();
                __syncwarp();
                if (lane == 0) arrive_on_leader(L::kBarSEmpty + b);
                uint32_t valid = __ballot_sync(0xffffffffu, 32 * cf + lane >= geo.r_lo && 32 * cf + lane < geo.r_hi);
                {
                    // how many of this thread's 32 tokens lie below its head's causal end: token j of the thread is
                    // token (page index) * 64 + tok0 + 32 cf + j of the request
                    const int lim = causal_end - ((seg.lo / kPage + seg.tile_begin + 2 * s + pg) * kPage + geo.tok0 + 32 * cf);
                    if (lim < 32) valid &= lim <= 0 ? 0u : (1u << lim) - 1u;
                }
                float mt = -INFINITY;
                if (__all_sync(0xffffffffu, valid == 0xffffffffu)) {
#pragma unroll
                    for (int j2 = 0; j2 < 16; ++j2) {
                        const float4 t = tok_a[j2];
                        sv[2 * j2] = fmaf(sv[2 * j2], cq * t.x, t.y);
                        sv[2 * j2 + 1] = fmaf(sv[2 * j2 + 1], cq * t.z, t.w);
                        mt = fmaxf(mt, fmaxf(sv[2 * j2], sv[2 * j2 + 1]));
                    }
                } else {
#pragma unroll
                    for (int j2 = 0; j2 < 16; ++j2) {
                        const float4 t = tok_a[j2];
                        sv[2 * j2] = (valid >> (2 * j2)) & 1u ? fmaf(sv[2 * j2], cq * t.x, t.y) : -INFINITY;
                        sv[2 * j2 + 1] = (valid >> (2 * j2 + 1)) & 1u ? fmaf(sv[2 * j2 + 1], cq * t.z, t.w) : -INFINITY;
                        mt = fmaxf(mt, fmaxf(sv[2 * j2], sv[2 * j2 + 1]));
                    }
                }
                // row maximum over the 4 threads of this head (2 pages x 2 column halves, 4 different warps)
                xch[hd * 4 + slot4] = mt;
                named_bar_sync_dyn<128>(2 + half_id);
                {
                    const float4 x4 = *reinterpret_cast<const float4 *>(&xch[hd * 4]);
                    mt = fmaxf(fmaxf(x4.x, x4.y), fmaxf(x4.z, x4.w));
                }
                bool grew = false;
                float al = 1.f;
                if (mt > m + kTau) { al = (m == -INFINITY) ? 0.f : fast_exp2(m - mt); m = mt; l *= al; grew = true; }
                if (slot4 == 0) alpha_s[hd] = al;
                const float off = kLift - (m == -INFINITY ? 0.f : m);   // a head that has seen no token yet: all weights 0, not NaN
                uint32_t phi[8], plo[8];
#pragma unroll
                for (int j4 = 0; j4 < 8; ++j4) {
                    const float4 rt = tok_r[j4];
                    const float rts[4] = {rt.x, rt.y, rt.z, rt.w};
                    float u[4];
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        u[e] = fast_exp2(sv[4 * j4 + e] + off);
                        l = fmaf(u[e], rts[e], l);
                    }
                    uint16_t h01, h23, r01, r23;
                    split_e4m3_e5m2_x2(u[0], u[1], h01, r01);
                    split_e4m3_e5m2_x2(u[2], u[3], h23, r23);
                    phi[j4] = (uint32_t)h01 | ((uint32_t)h23 << 16);
                    plo[j4] = (uint32_t)r01 | ((uint32_t)r23 << 16);
                }
                const bool rescale = named_bar_or<1, kSoftmaxWarps * 32>(grew);
                // P.V of the supertile that last used this P buffer (two back) must be done; a rescale
                // of O also needs the previous supertile's P.V
                if (st_it > 1) ok &= mbar_wait(ctx, bar(L::kBarStageEmpty + (st_it - 2) % kStages), ((st_it - 2) / kStages) & 1, L::kBarStageEmpty);
                if (rescale && s > 0) {
                    ok &= mbar_wait(ctx, bar(L::kBarStageEmpty + (st_it - 1) % kStages), ((st_it - 1) / kStages) & 1, L::kBarStageEmpty);
                    tcgen05_fence_after();
                    // O rows are TMEM lanes: this thread scales its lane's columns [128 cf, 128 cf + 128)
                    const float a_row = alpha_s[hd];
#pragma unroll 1
                    for (int c = 0; c < 4; ++c) {
                        float o[32];
                        const uint32_t addr = tmem_base + lane_addr + L::kColO + 128 * cf + c * 32;
                        tmem_ld32(addr, o);
                        tmem_wait_ld();
#pragma unroll
                        for (int k = 0; k < 32; ++k) o[k] *= a_row;
                        tmem_st16(addr, *reinterpret_cast<float(*)[16]>(&o[0]));
                        tmem_st16(addr + 16, *reinterpret_cast<float(*)[16]>(&o[16]));
                    }
                    tmem_wait_st();
                }
                {
                    // P hi / lo: K-major, 64-byte swizzle; slab = page, row = head, bytes [32 cf, 32 cf + 32)
                    uint8_t *ph = smem + L::kOffP + ((b * 2 + 0) * 2 + pg) * kSlab;
                    uint8_t *pl = smem + L::kOffP + ((b * 2 + 1) * 2 + pg) * kSlab;
#pragma unroll
                    for (int u16 = 0; u16 < 2; ++u16) {
                        const uint32_t o = sw64((uint32_t)hd, (uint32_t)(32 * cf + 16 * u16));
                        *reinterpret_cast<uint4 *>(ph + o) = make_uint4(phi[4 * u16], phi[4 * u16 + 1], phi[4 * u16 + 2], phi[4 * u16 + 3]);
                        *reinterpret_cast<uint4 *>(pl + o) = make_uint4(plo[4 * u16], plo[4 * u16 + 1], plo[4 * u16 + 2], plo[4 * u16 + 3]);
                    }
                }
                fence_proxy_async();
                tcgen05_fence_before();
                __syncwarp();
                if (lane == 0) arrive_on_leader(L::kBarPFull + b);
            }
            // ---- row sums of the 4 threads of a head
            xch[hd * 4 + slot4] = l;
            named_bar_sync<1, kSoftmaxWarps * 32>();
            if (slot4 == 0) {
                const float4 x4 = *reinterpret_cast<const float4 *>(&xch[hd * 4]);
                const float lt = (x4.x + x4.y) + (x4.z + x4.w);
                // no token at all (an empty causal range): O = 0, LSE = -inf.  Exactly 0: a NaN in the request's data stays one.
                l_s[hd] = lt == 0.f ? 0.f : 1.f / lt;
                const int gh = head0 + hd;
                if (gh < p.head_end) {
                    float lse = lt == 0.f ? -INFINITY : (m - kLift + log2f(lt)) * kLn2;
                    if (seg.slot < 0) p.lse[(int64_t)seg.request * p.lse_stride_request + gh] = lse;
                    else p.partial_lse[(int64_t)seg.slot * h + (gh - p.head_begin)] = lse;
                }
            }
            named_bar_sync<1, kSoftmaxWarps * 32>();
            // ---- epilogue: lane L < 64 holds head L, dv [256 n, 256 n + 128) in columns n * 128 + j;
            // lane 64 + L holds head L, dv [256 n + 128, 256 n + 256).  The two warps of a quadrant
            // take one n each.
            ok &= mbar_wait(ctx, bar(L::kBarOFull), seg_it & 1, L::kBarOFull);
            tcgen05_fence_after();
            // Every warp drains its [32 heads x 128 dv] block in four rounds of 32 columns through a
            // 4 KB tile of the P buffers (idle now: the last P.V has retired): a thread writes its row
            // in the 128-byte swizzle (conflict-free), one TMA store moves the tile out in whole lines
            // and clips the rows past the head slice.
            {
                const int n = cf;
                const int dv0 = 256 * n + 128 * pg;
                const int row0 = 32 * (q4 & 1);
                uint8_t *stg = smem + L::kOffP + sw * 4096;
                const float inv_l = l_s[hd];
                const bool final_out = seg.slot < 0;
                const CUtensorMap *omap = final_out ? &tmap_out : &tmap_part;
                const int rowc = final_out ? head0 + row0 : head0 - p.head_begin + row0;
                const int outer = final_out ? seg.request : seg.slot;
#pragma unroll 1
                for (int c = 0; c < 4; ++c) {
                    float o[32];
                    tmem_ld32(tmem_base + lane_addr + L::kColO + n * 128 + c * 32, o);
                    tmem_wait_ld();
                    if (c > 0) {                          // the previous round's store has read the tile
                        if (lane == 0) bulk_wait_group_read();
                        __syncwarp();
                    }
#pragma unroll
                    for (int i = 0; i < 8; ++i)
                        *reinterpret_cast<float4 *>(stg + lane * 128 + ((i ^ (lane & 7)) << 4)) =
                            make_float4(o[4 * i] * inv_l, o[4 * i + 1] * inv_l, o[4 * i + 2] * inv_l, o[4 * i + 3] * inv_l);
                    fence_proxy_async();
                    __syncwarp();
                    if (lane == 0) { tma_store_3d(omap, smem_u32(stg), dv0 + 32 * c, rowc, outer); bulk_commit_group(); }
                }
                if (lane == 0) bulk_wait_group_read();    // the tile goes back to being a P buffer
                __syncwarp();
            }
            tcgen05_fence_before();
            __syncwarp();
            if (lane == 0) arrive_on_leader(L::kBarOEmpty);
            ++seg_it;
        }
    } else {
        // ===================================================== softmax + epilogue warps, 32 heads
        // Two heads per thread, in the accumulator fragment layout: hA and hA + 8 of a quadrant's sixteen, hi terms in
        // lanes 0..15 of the quadrant and lo terms in lanes 16..31, so both terms of a logit arrive in the same register of two
        // loads.  Quadrants 0, 1 hold page A and 2, 3 page B of 16 heads each; the two warps of a quadrant take 32 tokens
        // each, a thread tokens 8 k + 2 tq + {0, 1} of them.
        const int sw = warp - kWarpSoftmax;             // 0..7
        const int q4 = warp & 3;                        // TMEM lane quadrant
        const int cf = sw >> 2;                         // tokens [32 cf, 32 cf + 32) of the page
        const int pg = q4 >> 1;                         // 0: page A, 1: page B
        const int head16 = q4 & 1;                      // heads 0-15 or 16-31: the four warps that share them sync on bar 2 + head16
        const int hA = 16 * head16 + (lane >> 2), tq = lane & 3;
        const int slot4 = pg * 2 + cf;                  // this warp's slot among the four
        const uint32_t lane_addr = (uint32_t)(32 * q4) << 16;
        float *qs_s = reinterpret_cast<float *>(smem + L::kOffQs);
        float *alpha_s = reinterpret_cast<float *>(smem + L::kOffAlpha);
        float *l_s = reinterpret_cast<float *>(smem + L::kOffL);
        float *xch = reinterpret_cast<float *>(smem + L::kOffXch);
        // what the four warps that share a head have found
        auto exchange = [&](float (&v)[2], auto op) {
            if (tq == 0) { xch[hA * 4 + slot4] = v[0]; xch[(hA + 8) * 4 + slot4] = v[1]; }
            named_bar_sync_dyn<128>(2 + head16);
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const float4 x = *reinterpret_cast<const float4 *>(&xch[(hA + 8 * e) * 4]);
                v[e] = op(op(x.x, x.y), op(x.z, x.w));
            }
        };
        // per-warp table of its 32 tokens: tok_a[j / 2] = (scale_j, log2 scale_j, scale_j+1, log2 scale_j+1), tok_r[j] = 1 / scale_j
        float4 *tok_a = reinterpret_cast<float4 *>(smem + L::kOffTok + sw * L::kTokBytes);
        float *tok_r = reinterpret_cast<float *>(tok_a + 16);
        const float *scale_s = reinterpret_cast<const float *>(smem + L::kOffScale);
        const float scale_log2 = p.softmax_scale * kLog2e;
        uint32_t st_it = 0, seg_it = 0;
        bool ok = true;                                 // (a failed wait only clears it, as above)
        while (it.next(p, seg)) {
            ok &= mbar_wait(ctx, bar(L::kBarQLocal), seg_it & 1, L::kBarQLocal);
            const float cqA = scale_log2 * qs_s[(seg_it & 3) * H + hA], cqB = scale_log2 * qs_s[(seg_it & 3) * H + hA + 8];
            __syncwarp();
            if (lane == 0) mbar_arrive(bar(L::kBarQsRead));
            float mA = -INFINITY, mB = -INFINITY, lA = 0.f, lB = 0.f;
            const int nsuper = (seg.tile_end - seg.tile_begin + 1) >> 1;
            // causal ends of the two (virtual) heads' rows
            int endA = 0x3fffffff, endB = 0x3fffffff;
            if (p.q_rows > 1) {
                const int len = p.seq_lens[seg.request] - (p.q_rows - 1);
                endA = len + (head0 + hA) % p.q_rows; endB = len + (head0 + hA + 8) % p.q_rows;
            }
            for (int s = 0; s < nsuper; ++s, ++st_it) {
                const PairGeom g = pair_geom(s);
                const TileGeom geo = pg ? g.b : g.a;
                const uint32_t stage = st_it % kStages, b = st_it & 1;
                ok &= mbar_wait(ctx, bar(L::kBarSFull + b), (st_it >> 1) & 1, L::kBarSFull + b);
                ok &= mbar_wait(ctx, bar(L::kBarScFull + stage), (st_it / kStages) & 1, L::kBarScFull + stage);
                tcgen05_fence_after();
                float sv[16];                     // [4 k + e]: head hA, token 8 k + 2 tq + e; [4 k + 2 + e]: head hA + 8
                {
                    // a load has eight heads' hi rows and their lo rows
                    float xa[16], xb[16];
                    const uint32_t sb = tmem_base + lane_addr + L::kColS + b * 64 + 32 * cf;
                    tmem_ld_frag<32>(sb, xa);
                    tmem_ld_frag<32>(sb + (16u << 16), xb);
                    // meanwhile: lane j prepares token 32 cf + j.  A token outside the range gets scale 0 and
                    // log2 scale -inf; its row of K may hold anything, so its logit is also forced below.
                    const int r = 32 * cf + lane;
                    const bool v = r >= geo.r_lo && r < geo.r_hi;
                    const float ts = v ? scale_s[(stage * 2 + pg) * 64 + geo.tok0 + r] : 0.f;
                    reinterpret_cast<float2 *>(tok_a)[lane] = make_float2(ts, v ? fast_log2(ts) : -INFINITY);
                    tok_r[lane] = v ? fast_rcp(ts) : 0.f;
                    tmem_wait_ld();
#pragma unroll
                    for (int k = 0; k < 4; ++k)
#pragma unroll
                        for (int e = 0; e < 2; ++e) { sv[4 * k + e] = xa[4 * k + e] + xa[4 * k + 2 + e]; sv[4 * k + 2 + e] = xb[4 * k + e] + xb[4 * k + 2 + e]; }
                }
                tcgen05_fence_before();
                __syncwarp();
                if (lane == 0) arrive_on_leader(L::kBarSEmpty + b);
                // the warp's tokens [first, limA) / [first, limB) count for its two heads
                float mt[2] = {-INFINITY, -INFINITY};
                const int t_first = (seg.lo / kPage + seg.tile_begin + 2 * s + pg) * kPage + geo.tok0;    // token of row 0
                const int limA = min(geo.r_hi, endA - t_first) - 32 * cf, limB = min(geo.r_hi, endB - t_first) - 32 * cf;
                const int first = geo.r_lo - 32 * cf;
                if (__all_sync(0xffffffffu, first <= 0 && limA >= 32 && limB >= 32)) {
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const float4 t = tok_a[4 * k + tq];
                        sv[4 * k] = fmaf(sv[4 * k], cqA * t.x, t.y);
                        sv[4 * k + 1] = fmaf(sv[4 * k + 1], cqA * t.z, t.w);
                        sv[4 * k + 2] = fmaf(sv[4 * k + 2], cqB * t.x, t.y);
                        sv[4 * k + 3] = fmaf(sv[4 * k + 3], cqB * t.z, t.w);
                    }
                } else {
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const float4 t = tok_a[4 * k + tq];
                        const int j0 = 8 * k + 2 * tq, j1 = j0 + 1;
                        sv[4 * k] = j0 >= first && j0 < limA ? fmaf(sv[4 * k], cqA * t.x, t.y) : -INFINITY;
                        sv[4 * k + 1] = j1 >= first && j1 < limA ? fmaf(sv[4 * k + 1], cqA * t.z, t.w) : -INFINITY;
                        sv[4 * k + 2] = j0 >= first && j0 < limB ? fmaf(sv[4 * k + 2], cqB * t.x, t.y) : -INFINITY;
                        sv[4 * k + 3] = j1 >= first && j1 < limB ? fmaf(sv[4 * k + 3], cqB * t.z, t.w) : -INFINITY;
                    }
                }
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    mt[0] = fmaxf(mt[0], fmaxf(sv[4 * k], sv[4 * k + 1]));
                    mt[1] = fmaxf(mt[1], fmaxf(sv[4 * k + 2], sv[4 * k + 3]));
                }
                // row maximum: the four threads of a head in this warp, then the four warps
#pragma unroll
                for (int o = 1; o < 4; o <<= 1) {
                    mt[0] = fmaxf(mt[0], __shfl_xor_sync(0xffffffffu, mt[0], o));
                    mt[1] = fmaxf(mt[1], __shfl_xor_sync(0xffffffffu, mt[1], o));
                }
                exchange(mt, [](float x, float y) { return fmaxf(x, y); });
                bool grew = false;
                float alA = 1.f, alB = 1.f;
                if (mt[0] > mA + kTau) { alA = (mA == -INFINITY) ? 0.f : fast_exp2(mA - mt[0]); mA = mt[0]; lA *= alA; grew = true; }
                if (mt[1] > mB + kTau) { alB = (mB == -INFINITY) ? 0.f : fast_exp2(mB - mt[1]); mB = mt[1]; lB *= alB; grew = true; }
                if (tq == 0 && slot4 == 0) { alpha_s[hA] = alA; alpha_s[hA + 8] = alB; }
                // a head that has seen no token yet: all weights 0, not NaN
                const float offA = kLift - (mA == -INFINITY ? 0.f : mA), offB = kLift - (mB == -INFINITY ? 0.f : mB);
                uint32_t wA[4], wB[4];            // two tokens each: hi bytes below, lo bytes above
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const float2 rt = *reinterpret_cast<const float2 *>(&tok_r[8 * k + 2 * tq]);
                    const float a0 = fast_exp2(sv[4 * k] + offA), a1 = fast_exp2(sv[4 * k + 1] + offA);
                    const float b0 = fast_exp2(sv[4 * k + 2] + offB), b1 = fast_exp2(sv[4 * k + 3] + offB);
                    lA = fmaf(a1, rt.y, fmaf(a0, rt.x, lA));
                    lB = fmaf(b1, rt.y, fmaf(b0, rt.x, lB));
                    uint16_t main, rest;
                    split_e4m3_e4m3x16_x2(a0, a1, main, rest);
                    wA[k] = (uint32_t)main | ((uint32_t)rest << 16);
                    split_e4m3_e4m3x16_x2(b0, b1, main, rest);
                    wB[k] = (uint32_t)main | ((uint32_t)rest << 16);
                }
                const bool rescale = named_bar_or<1, kSoftmaxWarps * 32>(grew);
                // P.V of the supertile that last used this P buffer (two back) must be done; a rescale
                // of O also needs the previous supertile's P.V
                if (st_it > 1) ok &= mbar_wait(ctx, bar(L::kBarStageEmpty + (st_it - 2) % kStages), ((st_it - 2) / kStages) & 1, L::kBarStageEmpty);
                if (rescale && s > 0) {
                    ok &= mbar_wait(ctx, bar(L::kBarStageEmpty + (st_it - 1) % kStages), ((st_it - 1) / kStages) & 1, L::kBarStageEmpty);
                    tcgen05_fence_after();
                    // O rows are TMEM lanes (hi and lo rows of the same sixteen heads): this thread scales its lane's columns
                    // [128 cf, 128 cf + 128)
                    const float a_row = alpha_s[16 * head16 + (lane & 15)];
#pragma unroll 1
                    for (int c = 0; c < 4; ++c) {
                        float o[32];
                        const uint32_t addr = tmem_base + lane_addr + L::kColO + 128 * cf + c * 32;
                        tmem_ld32(addr, o);
                        tmem_wait_ld();
#pragma unroll
                        for (int k = 0; k < 32; ++k) o[k] *= a_row;
                        tmem_st16(addr, *reinterpret_cast<float(*)[16]>(&o[0]));
                        tmem_st16(addr + 16, *reinterpret_cast<float(*)[16]>(&o[16]));
                    }
                    tmem_wait_st();
                }
                {
                    // P: K-major, 64-byte swizzle; slab = page, byte = token, rows like the query operand's.  Neighbouring lanes swap
                    // so that a thread holds four consecutive tokens, of group k (even lanes) or k + 1 (odd lanes): 4-byte
                    // stores without conflicts.
                    const bool odd = tq & 1;
                    uint8_t *const ph = smem + L::kOffP + b * L::kPBuf + pg * kSlab + (odd ? 8 : 0) + 4 * (tq >> 1);
#pragma unroll
                    for (int k = 0; k < 4; k += 2) {
                        const uint32_t o = sw64((uint32_t)(2 * hA - (hA & 15)), (uint32_t)(32 * cf + 8 * k));
#pragma unroll
                        for (int e = 0; e < 2; ++e) {
                            const uint32_t w0 = e ? wB[k] : wA[k], w1 = e ? wB[k + 1] : wA[k + 1];
                            const uint32_t got = __shfl_xor_sync(0xffffffffu, odd ? w0 : w1, 1);
                            const uint32_t lower = odd ? got : w0, upper = odd ? w1 : got;
                            uint8_t *const dst = ph + o + e * (8 * 64);          // head hA + 8: same swizzle phase
                            *reinterpret_cast<uint32_t *>(dst) = __byte_perm(lower, upper, 0x5410);
                            *reinterpret_cast<uint32_t *>(dst + L::kPTerm) = __byte_perm(lower, upper, 0x7632);
                        }
                    }
                }
                fence_proxy_async();
                tcgen05_fence_before();
                __syncwarp();
                if (lane == 0) arrive_on_leader(L::kBarPFull + b);
            }
            // ---- row sums of a head: its four threads here, then the four warps
            float lt[2] = {lA, lB};
#pragma unroll
            for (int o = 1; o < 4; o <<= 1) {
                lt[0] += __shfl_xor_sync(0xffffffffu, lt[0], o);
                lt[1] += __shfl_xor_sync(0xffffffffu, lt[1], o);
            }
            exchange(lt, [](float x, float y) { return x + y; });
            if (tq == 0 && slot4 == 0) {
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const int hh = hA + 8 * e, gh = head0 + hh;
                    l_s[hh] = lt[e] == 0.f ? 0.f : 1.f / lt[e];      // no token at all: O = 0, LSE = -inf, as above
                    if (gh < p.head_end) {
                        const float lse = lt[e] == 0.f ? -INFINITY : ((e ? mB : mA) - kLift + log2f(lt[e])) * kLn2;
                        if (seg.slot < 0) p.lse[(int64_t)seg.request * p.lse_stride_request + gh] = lse;
                        else p.partial_lse[(int64_t)seg.slot * h + (gh - p.head_begin)] = lse;
                    }
                }
            }
            named_bar_sync<1, kSoftmaxWarps * 32>();
            // ---- epilogue: quadrants 0, 1 hold dv [256 n, 256 n + 128) in columns n * 128 + j, quadrants 2, 3
            // dv [256 n + 128, 256 n + 256).  The two warps of a quadrant take one n each: [16 heads x 128 dv] as hi and lo
            // rows, in four rounds of 32 columns through a 2 KB tile of the P buffers (idle now) and a TMA store per round.
            ok &= mbar_wait(ctx, bar(L::kBarOFull), seg_it & 1, L::kBarOFull);
            tcgen05_fence_after();
            {
                const int n = cf;
                const int dv0 = 256 * n + 128 * pg;
                const int row0 = 16 * head16;
                uint8_t *stg = smem + L::kOffP + sw * 2048;
                const bool final_out = seg.slot < 0;
                const CUtensorMap *omap = final_out ? &tmap_out : &tmap_part;
                const int rowc = final_out ? head0 + row0 : head0 - p.head_begin + row0;
                const int outer = final_out ? seg.request : seg.slot;
                const int r = lane >> 2;                      // rows r and r + 8: same swizzle phase
                const float inv_a = l_s[row0 + r], inv_b = l_s[row0 + r + 8];
#pragma unroll 1
                for (int c = 0; c < 4; ++c) {
                    const uint32_t addr = tmem_base + lane_addr + L::kColO + n * 128 + c * 32;
                    float o[16], lo[16];
                    tmem_ld_frag<32>(addr, o);
                    tmem_ld_frag<32>(addr + (16u << 16), lo);
                    tmem_wait_ld();
                    if (c > 0) {                              // the previous round's store has read the tile
                        if (lane == 0) bulk_wait_group_read();
                        __syncwarp();
                    }
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        uint8_t *const dst = stg + r * 128 + (((2 * k + (tq >> 1)) ^ r) << 4) + (tq & 1) * 8;
                        *reinterpret_cast<float2 *>(dst) =
                            make_float2(fmaf(lo[4 * k], 0.0625f, o[4 * k]) * inv_a, fmaf(lo[4 * k + 1], 0.0625f, o[4 * k + 1]) * inv_a);
                        *reinterpret_cast<float2 *>(dst + 8 * 128) =
                            make_float2(fmaf(lo[4 * k + 2], 0.0625f, o[4 * k + 2]) * inv_b, fmaf(lo[4 * k + 3], 0.0625f, o[4 * k + 3]) * inv_b);
                    }
                    fence_proxy_async();
                    __syncwarp();
                    if (lane == 0) { tma_store_3d(omap, smem_u32(stg), dv0 + 32 * c, rowc, outer); bulk_commit_group(); }
                }
                if (lane == 0) bulk_wait_group_read();        // the tile goes back to being a P buffer
                __syncwarp();
            }
            tcgen05_fence_before();
            __syncwarp();
            if (lane == 0) arrive_on_leader(L::kBarOEmpty);
            ++seg_it;
        }
    }

    fill_empty_requests(p, it.tile_start(p), worker, head0, H, tid, kThreads);
    if (p.trace != nullptr && tid == 0) {   // per-CTA cycles and nanoseconds
        p.trace[512 + blockIdx.x] = clock64() - t_start;
        if (blockIdx.x < 256) p.trace[768 + blockIdx.x] = (long long)(global_timer_ns() - ns_start);
    }

    // ---- teardown: nobody leaves while its partner may still touch its shared memory or barriers
    if (*ctx.abort_flag) {
        const unsigned long long t0 = global_timer_ns();
        while (global_timer_ns() - t0 < 200000ull) { __nanosleep(1000); }
    }
    tcgen05_fence_before();
    __syncthreads();
    cluster_sync_all();
    if (warp == 0) {
        tcgen05_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512u) : "memory");
    }
}

template <int H>
cudaError_t launch_pair(const DecodeParams &p, cudaStream_t stream) {
    alignas(64) CUtensorMap mpage, mpair, mq;
    const uint64_t pages = (uint64_t)(p.num_pool_pages > 0 ? p.num_pool_pages : 1);
    if (!make_map_4d(&mpage, CU_TENSOR_MAP_DATA_TYPE_UINT8, CU_TENSOR_MAP_SWIZZLE_64B, p.kv_pool, kPage, pages,
                     (uint64_t)kDQK, 64, (uint64_t)kPage * kDQK, 64, 9))
        return cudaErrorInvalidValue;
    if (!make_map_4d(&mpair, CU_TENSOR_MAP_DATA_TYPE_UINT8, CU_TENSOR_MAP_SWIZZLE_64B, p.kv_pool, kPage, pages,
                     (uint64_t)kDQK, 64, (uint64_t)kPage * kDQK, 64, 2))
        return cudaErrorInvalidValue;
    // output maps: (512 dv, heads below head_end, requests) over `out`, (512, h, partial slots) over the workspace
    alignas(64) CUtensorMap mout, mpart;
    if (p.out_stride_head % 4 || p.out_stride_request % 4) return cudaErrorNotSupported;   // rows must start on 16-byte boundaries
    const uint64_t hbytes = (uint64_t)p.out_stride_head * 4;
    if (!make_store_map_3d(&mout, p.out, kDV, (uint64_t)p.head_end, (uint64_t)p.B, hbytes,
                           p.B > 1 ? (uint64_t)p.out_stride_request * 4 : hbytes * (uint64_t)p.head_end, H / 2))
        return cudaErrorNotSupported;
    const uint64_t h = (uint64_t)(p.head_end - p.head_begin);
    if (!make_store_map_3d(&mpart, p.partial_out, kDV, h, (uint64_t)2 * p.num_workers, (uint64_t)kDV * 4, h * kDV * 4, H / 2))
        return cudaErrorInvalidValue;
    DecodeParams args = p;
    args.q_by_hand = make_query_map(&mq, p, H) ? 0 : 1;
    if (args.q_by_hand) mq = mpage;
    const int smem = (int)Layout<H>::kSmemBytes;
    static DeviceOnce once;
    cudaError_t e = once.run([&] {
        return cudaFuncSetAttribute(decode_umma_fp8_pair_kernel<H>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    });
    if (e != cudaSuccess) return e;
    // (the cluster shape is part of the kernel's declaration)
    e = launch_dependent(decode_umma_fp8_pair_kernel<H>,
                         dim3((unsigned)(p.num_workers * p.pair_groups * 2)), dim3(kThreads), (size_t)smem, stream, args, mpage, mpair, mout, mpart, mq);
    count_launch();
    return e;
}

}  // namespace

cudaError_t launch_decode_umma_fp8_pair(const DecodeParams &p, cudaStream_t stream) {
    return p.heads_per_group == 32 ? launch_pair<32>(p, stream) : launch_pair<64>(p, stream);
}

}  // namespace splash
