// MLKV decode-attention kernels for GB300 (sm_103a).
//
// decode_kernel: single-token attention of one layer over the cache slot of the layer's owner
// (MLKV, arXiv 2406.09297, Sec. 3 Eqs. 13-18, attention of Eqs. 2-3).
//
//   Work split.  A "segment" is one (sequence beta, KV head j) pair: positions [0, L_beta) of one
//   K/V head, read by the G = h/g query heads of its group (Eq. 15).  Segments are cut into tiles
//   of T positions and all tiles of the layer are laid end to end (beta-major, j inside).  A
//   persistent grid of P CTAs takes equal contiguous runs of that tile list, so every CTA streams
//   the same number of bytes whatever the length mix.  The part of a segment inside one CTA's run
//   is a "piece"; a CTA that holds a whole segment writes its output directly, otherwise it
//   writes a normalised partial (o, log-sum-exp) and the last CTA to finish the segment (an atomic
//   counter, no spinning) merges the partials.
//
//   Data movement.  One producer warp issues TMA tensor copies (cp.async.bulk.tensor, 128-byte
//   swizzle) of each K and V tile into a STAGES-deep shared-memory ring, completion tracked by
//   mbarrier transaction counts.  Each tile is fetched from HBM exactly once and used by all G
//   query heads of the group.
//
//   Math.  Four consumer warps split every tile by positions.  Scores S = Q K^T and the update
//   O += P V run on the tensor cores (mma.sync m16n8k16, bf16 in, fp32 accumulate), the query group
//   padded to 16 rows or (at most 8 heads) to 8 columns; the softmax is online, in fp32, base 2
//   with the 1/sqrt(d) scale folded into the exponent, with shuffles for the maxima.  At the end of
//   a piece each warp leaves its raw sums in shared memory and goes on; the epilogue warp merges
//   them (the CTA's last piece: all consumer warps, after one barrier).  With the former tree over
//   the consumer warps, a barrier a level, a piece boundary cost ~2 us at head_dim 128 (measured,
//   64 uneven segments over 138 CTAs: layer calls 16.2 -> 13.4 us with the merge of up to 8 records
//   in the launch, below; 12.1 now).
//
//   Launch.  Programmatic dependent launch: barrier set-up overlaps the previous kernel of the
//   stream, and no global memory is touched before griddepcontrol.wait.
//
// append_kernel: stores the new token's K/V of an owner layer at position L_beta - 1.
//
// Every wait on an mbarrier is bounded (about 2 s); on expiry the kernel sets a bit in the
// device error word, stops issuing copies, keeps its barrier sequence intact, drains the copies
// it already issued and exits.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

#include "mlkv_internal.h"

#include "mlkv_device.cuh"

namespace mlkv {
namespace {

// ------------------------------------------------------------------------------------------------
// shared-memory plan
// ------------------------------------------------------------------------------------------------

// Whether CTAs of `bytes` shared memory are `blocks` times resident beside the largest batch's tables
// (an SM's 228 KB, 1 KB of them the system's per CTA).
constexpr bool uneven_fits(int blocks, int bytes)
{
    return blocks * (bytes + table_bytes(MLKV_MAX_BATCH) + 1024) <= 228 * 1024;
}

// kRows: query rows the CTA keeps room for, 16 or (groups of at most 8 heads) 8.
template <int D, int T, int STAGES, int NCW, bool kT>
struct Plan {
    static constexpr int kRows = kT ? 8 : 16;
    static constexpr int kThreads = (NCW + 2) * 32;   // consumers, one producer, one epilogue warp
    // Variants whose ring fits twice in an SM's shared memory are sized for two resident CTAs.
    static constexpr int kMinBlocks = (STAGES * 2 * T * D * 2 <= (kT ? 96 : 80) * 1024) ? 2 : 1;
    static constexpr int kProducer = NCW;             // warp indices
    static constexpr int kEpilogue = NCW + 1;
    static constexpr int kSub = D / 64;               // 128-byte-wide column blocks per row
    static constexpr int kTW = T / NCW;               // positions per warp per tile
    static constexpr int kTileBytes = T * D * 2;      // one K (or V) tile
    static constexpr int kStageBytes = 2 * kTileBytes;
    static constexpr int kResO = kRows * D * 4;       // a cluster rank's result: o[kRows][D] f32
    static constexpr int kResBytes = kResO + 16 * 4 + 32;   // + lse[16] (cluster slots)
    // A finished piece: every warp's raw sums o[NCW][kRows][kRawRow] f32 (rows padded so that the
    // fragment stores of a warp's 8 rows fall in distinct banks), its row maxima and sums
    // [2][16][NCW], 8 ints of metadata and, in a cluster's leader, lse[16].
    static constexpr int kRawRow = D + 8;
    static constexpr int kRawO = NCW * kRows * kRawRow * 4;
    static constexpr int kRawMeta = kRawO + 2 * 16 * NCW * 4;
    static constexpr int kRawLse = kRawMeta + 32;
    static constexpr int kRawBytes = kRawLse + 64;
    // Two buffers where shared memory has room for them: the epilogue warp takes ~1.3 us to merge a
    // piece's warps (64 uneven sequences of up to 2048 positions, 12 heads of 64: 165 us for 12
    // layers, 172 with one buffer; 145 once the buffer was freed before the counter).
    static constexpr int kMaxRawBufs = (!kT && T == 256) ? 1 : 2;
    static constexpr int kRaw = STAGES * kStageBytes;                  // the first buffer
    // records an inline merge may take (inline_merge_pieces of the largest group they are 8 for)
    static constexpr int kMaxPieces = kT ? kInlineMergeMaxPieces : inline_merge_pieces(9, D);
    static constexpr int kEpiW = kRaw + kRawBytes;              // its weights, f32 [pieces][G]
    static constexpr int kFlags = kEpiW + kMaxPieces * kRows * 4;   // int [4]
    // u64 full[S], empty[S], res_full[2], res_empty[2], cluster
    static constexpr int kBars = kFlags + 16;
    // Per-stage query slots: the G rows of the segment whose first tile the stage holds, each row
    // padded by 16 bytes so that the fragment loads (8 rows apart) fall in distinct banks.
    static constexpr int kQRow = D * 2 + 16;
    static constexpr int kQSlot = kRows * kQRow;
    static constexpr int kQ = (kBars + (2 * STAGES + 5) * 8 + 8 + 127) / 128 * 128;
    // The tail: the second raw buffer (DecodeParams::raw_bufs == 2) and, lengths differing, the
    // per-sequence tables.  A cluster's leader keeps the slots for the other ranks' results
    // ([k-1][kResBytes]) there: its CTAs hold one piece each, so in the second buffer if there is
    // one.
    static constexpr int kTail = kQ + STAGES * kQSlot;
    static constexpr int kBytes = kTail + (kMaxRawBufs - 1) * kRawBytes;
    static constexpr bool kClusterInRaw = kMaxRawBufs == 2;
    static_assert(!kClusterInRaw || 3 * kResBytes <= kRawBytes, "slots of three ranks");
    static constexpr int kAlloc = kBytes + 1024;      // base aligned up to 1024 in the kernel
    static_assert(kTW % 16 == 0, "each warp takes whole 16-position mma steps");
    static_assert(NCW == 4, "four consumer warps");
    static_assert(D == 64 || D == 128, "head_dim 64 or 128");
    static_assert(T <= 256, "TMA box height");
    static_assert(kResBytes % 16 == 0, "result slots stay 16-byte aligned");
    // Uneven lengths cost a launch no resident CTA and no tile length at any batch: where two raw
    // buffers and the tables do not fit, one does.  (While they did not, 800 uneven sequences of up
    // to 3000 positions, 12 layers of one KV head: 926 us, 670 with one.)
    static_assert(uneven_fits(kMinBlocks, kAlloc - (kMaxRawBufs - 1) * kRawBytes),
                  "shared memory of the resident CTAs");
    // Two buffers fit at every batch: their number is no run-time value (which cost 2-3% of uneven
    // layer calls over short sequences, groups of 3 heads).
    static constexpr bool kTwoFit = kMaxRawBufs == 2 && uneven_fits(kMinBlocks, kAlloc);
    static_assert(kRawBytes % 16 == 0 && kRawMeta % 16 == 0 && kTail % 16 == 0,
                  "raw buffers and tables stay 16-byte aligned");
};


// Query fragments of one (sequence, KV head) group, rows of D bf16 `stride` elements apart (global
// memory, or the group's shared-memory slot); rows >= G are zero.  As the A operand of S = Q K^T in
// the mma.m16n8k16 layout (16 rows), or, kT, as the B operand of S^T = K Q^T (8 rows).
template <int D, bool kT>
__device__ __forceinline__ void load_q_frag(uint32_t (&qf)[D / 16][kT ? 2 : 4],
                                            const __nv_bfloat16 *qb, int stride, int G, int lane)
{
    const int qr = lane >> 2, qc = (lane & 3) * 2;
    const bool r0 = qr < G, r1 = qr + 8 < G;
#pragma unroll
    for (int ks = 0; ks < D / 16; ++ks) {
        const int c = ks * 16 + qc;
        const __nv_bfloat16 *row = qb + qr * stride + c;
        if constexpr (kT) {
            qf[ks][0] = r0 ? *reinterpret_cast<const uint32_t *>(row) : 0u;
            qf[ks][1] = r0 ? *reinterpret_cast<const uint32_t *>(row + 8) : 0u;
        } else {
            qf[ks][0] = r0 ? *reinterpret_cast<const uint32_t *>(row) : 0u;
            qf[ks][1] = r1 ? *reinterpret_cast<const uint32_t *>(row + 8 * stride) : 0u;
            qf[ks][2] = r0 ? *reinterpret_cast<const uint32_t *>(row + 8) : 0u;
            qf[ks][3] = r1 ? *reinterpret_cast<const uint32_t *>(row + 8 * stride + 8) : 0u;
        }
    }
}

// Margin (log2 units) by which a score may exceed a row's reference maximum before the reference
// is raised: weights stay <= 2^8.
constexpr float kLazyMax = 8.f;
// Two bf16 ones, the B operand that turns P V's MMA into P's row sums.
constexpr uint32_t kOnesBf16x2 = 0x3f803f80u;

// ------------------------------------------------------------------------------------------------
// decode kernel
// ------------------------------------------------------------------------------------------------

// kT: query groups of at most 8 heads.  mma.m16n8k16 pads the group to 16 rows as the A operand, to
// 8 columns as the B operand: with S^T = K Q^T and O^T += V^T P^T (A = positions, then channels;
// movmatrix turns P^T's fragments) a tile takes half the MMAs, exponentials and accumulators.
// Measured on GB300 (layer calls, 16-row form -> this one): 32 layers of 8 uneven sequences, 8 KV
// heads of 128 with 4 heads each 413 -> 404 us; 12 layers of 128 uneven sequences, 4 KV heads of 64
// with 3 heads each 602 -> 579 us.
template <int D, int T, int STAGES, int NCW, bool kT>
__global__ void __launch_bounds__(Plan<D, T, STAGES, NCW, kT>::kThreads,
                                  Plan<D, T, STAGES, NCW, kT>::kMinBlocks)
    decode_kernel(const __grid_constant__ CUtensorMap tmap,
                  const __grid_constant__ CUtensorMap tmap_rows,
                  const __grid_constant__ DecodeParams p)
{
    using PL = Plan<D, T, STAGES, NCW, kT>;
    constexpr int TW = PL::kTW;
    constexpr int NT = kT ? TW / 16 : TW / 8;   // score tiles per warp (16 or 8 positions)
    constexpr int KS = D / 16;                  // 16-wide reduction steps over the head dimension
    constexpr int NO = kT ? D / 16 : D / 8;     // output tiles (16 channels x 8 heads, or 8 x 16)

    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
    const uint32_t sbase = smem_addr(smem);
    const uint32_t bar_full = sbase + PL::kBars;
    const uint32_t bar_empty = bar_full + 8 * STAGES;
    const uint32_t bar_res_full = bar_empty + 8 * STAGES;    // [2]
    const uint32_t bar_res_empty = bar_res_full + 16;        // [2]
    const uint32_t bar_cluster = bar_res_empty + 16;         // leader: k-1 remote arrivals
    volatile int *flags = reinterpret_cast<volatile int *>(smem + PL::kFlags);
    // raw sums: one or two buffers, buffer rb at raw_at(rb)
    const int two = PL::kMaxRawBufs == 1 ? 0 : PL::kTwoFit ? 1 : p.raw_bufs - 1;
    auto raw_at = [&](int rb) { return rb ? PL::kTail : PL::kRaw; };
    int *s_len = reinterpret_cast<int *>(smem + PL::kTail + two * PL::kRawBytes);
    int *s_start = s_len + p.b;

    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    const int P = gridDim.x;
    const int cta = blockIdx.x;
    const int N = p.num_tiles;
    // floor(c N / P) in 32 bits when c N fits (a 64-bit division costs ~0.1 us at CTA start).
    // A multi-layer launch numbers each CTA's own tiles from 0: its items c, c + P, ... (whole
    // segments of nt tiles each).
    const bool ml = p.ml_layers > 0;
    const bool narrow = static_cast<long long>(P) * N < (1ll << 32);
    int tile_lo, tile_hi;
    if (ml) {
        // the tiles of this CTA's items (see TileWalk::ml_rank)
        tile_lo = 0;
        tile_hi = 0;
        for (int k = 0;; ++k) {
            const int r = TileWalk<T>::ml_rank(p, k);
            if (r < 0)
                break;
            const int L = p.uniform_len > 0
                              ? p.uniform_len
                              : p.seq_len[p.tile_start[TileWalk<T>::ml_seq_pos(p, r)]];
            if (p.ml_chunks > 1) {
                int a, b;
                TileWalk<T>::ml_chunk(p, (L + T - 1) / T, r % p.ml_chunks, a, b);
                tile_hi += b - a;
            } else {
                tile_hi += (L + T - 1) / T;
            }
        }
    } else {
        tile_lo = narrow ? static_cast<int>(static_cast<uint32_t>(cta) * N / P)
                         : static_cast<int>(static_cast<long long>(cta) * N / P);
        tile_hi = narrow ? static_cast<int>(static_cast<uint32_t>(cta + 1) * N / P)
                         : static_cast<int>(static_cast<long long>(cta + 1) * N / P);
    }
    // Per-layer pointers: a multi-layer launch reads layer `layer`'s queries, writes its outputs,
    // reads its owner's slot and new token; a single-layer launch has one of each.
    auto q_of = [&](int layer) {
        return ml ? p.Q + static_cast<size_t>(layer) * p.ml_q_stride : p.Q;
    };
    auto slot_of = [&](int layer) { return ml ? static_cast<int>(p.ml_slot[layer]) : p.slot; };

    const bool early = p.early_fetch == 1;
    const bool pre_tile = p.early_fetch != 0;   // the first tile may go out before the wait
    // The producer warp's copy of one tile into stage `s` (query rows too when a later piece
    // starts); called by all 32 lanes with the same arguments.  On GB300 one issuing thread
    // completes about one bulk copy per ~0.5 us whatever its size (measured: 8 to 64 KB, from L2
    // or HBM, 2 to 8 copies outstanding), while copies from different lanes proceed side by side;
    // so the copies of a tile -- K and V boxes, query rows -- go out from different lanes, and
    // successive stages from different groups of lanes.  Lane 0 first announces the stage's bytes.
    auto issue_tile = [&](const TileWalk<T> &w, int s, bool with_q) {
        const uint32_t fb = bar_full + 8 * s;
        const uint32_t qbytes = static_cast<uint32_t>(p.G) * D * 2;
        // A segment's last tile may be partly visible: only its boxes of 64 positions that
        // hold visible rows are fetched (the rest of the stage keeps stale rows, which the
        // consumers mask in S and zero in V).
        const int vis = w.L - w.tt * T;
        const int nbox = vis < T ? (vis + 63) / 64 : 0;
        const uint32_t kv_bytes =
            nbox > 0 ? static_cast<uint32_t>(nbox) * 64u * D * 2u * 2u : PL::kStageBytes;
        if (lane == 0)
            mbar_arrive_expect_tx(fb, kv_bytes + (with_q ? qbytes : 0u));
        __syncwarp();
        // copy i of this tile goes out from lane (i + rot) mod 32
        const int per_tile = 2 * PL::kSub * (nbox > 0 ? nbox : 1);
        const int mine = (lane - s * 2 * PL::kSub) & 31;
        const int zk = ((slot_of(w.layer) * 2 + 0) * p.b + w.beta) * p.g + w.j;
        const int zv = zk + p.b * p.g;
        const int y = w.tt * T;
        const uint32_t kdst = sbase + s * PL::kStageBytes;
        const uint32_t vdst = kdst + PL::kTileBytes;
        if (mine < per_tile) {
            // copy i: box bx = i / (2 kSub), then K or V, then the 64-column block
            const int bx = mine / (2 * PL::kSub);
            const int kv = (mine / PL::kSub) & 1;
            const int sub = mine % PL::kSub;
            const uint32_t dst = (kv ? vdst : kdst) + sub * T * 128 + bx * 64 * 128;
            if (nbox == 0)
                tma_load_3d(dst, &tmap, fb, sub * 64, y, kv ? zv : zk);
            else
                tma_load_3d(dst, &tmap_rows, fb, sub * 64, y + 64 * bx, kv ? zv : zk);
        }
        if (with_q) {
            const __nv_bfloat16 *q0 = q_of(w.layer) + (static_cast<size_t>(w.beta) * p.h +
                                                       static_cast<size_t>(w.j) * p.G) * D;
            const int r = (mine - per_tile) & 31;
            if (r < p.G)
                bulk_load(sbase + PL::kQ + s * PL::kQSlot + r * PL::kQRow, q0 + r * D, D * 2, fb);
        }
    };
    // The ring's barriers belong to the producer warp's lane 0.  With early fetch (either kind) and
    // one length for every sequence the warp also sends its first tile before the CTA barrier: a
    // CTA that got its SM late (the last ones of a layer decide the layer's end), or one that
    // starts while the step's inputs are still being copied in, then has data on the way at once.
    bool pre_issued = false;
    // The trigger comes first: the next launch (inside a decode step, the next layer's decode)
    // may start as soon as every CTA of this grid is resident.  What it reads before its own
    // dependency wait is fixed by p.early_fetch, and it finishes only after this grid.  The first
    // layer of a step triggers after its own wait instead: the kernels before the step may still be
    // writing what the next layers read early.
    if (threadIdx.x == 0 && !p.trigger_late)
        grid_dependents_launch();
    if (warp == PL::kProducer) {
        if (lane == 0) {
            prefetch_tensormap(&tmap);   // kernel parameters: safe before the dependency wait
            prefetch_tensormap(&tmap_rows);
            for (int s = 0; s < STAGES; ++s) {
                mbar_init(bar_full + 8 * s, 1);
                mbar_init(bar_empty + 8 * s, NCW);
            }
            fence_barrier_init();
        }
        __syncwarp();
        if (pre_tile && p.uniform_len > 0 && tile_lo < tile_hi) {
            TileWalk<T> w0;
            w0.init(p, s_len, s_start, tile_lo);
            if (w0.tt != w0.nt - 1 || p.newest_ready) {   // not a newest row still to wait for
                issue_tile(w0, 0, false);
                pre_issued = true;
            }
        }
    }
    if (threadIdx.x == 0) {
        for (int r = 0; r < 2; ++r) {
            mbar_init(bar_res_full + 8 * r, NCW);
            mbar_init(bar_res_empty + 8 * r, 1);
        }
        mbar_init(bar_cluster, 1);
        if (p.cluster_k > 1 && cluster_ctarank() == 0) {
            // The leader expects every other rank's result: G*D outputs and G lse values, f32.
            mbar_arrive_expect_tx(bar_cluster, static_cast<uint32_t>(
                                                   (p.cluster_k - 1) * (p.G * D + p.G) * 4));
        }
        flags[0] = 0;   // abort
        fence_barrier_init();
    }
    if (p.uniform_len <= 0) {
        for (int i = threadIdx.x; i < p.b; i += blockDim.x) {
            s_len[i] = p.seq_len[i];
            s_start[i] = p.tile_start[i];
        }
        if (threadIdx.x == 0)
            s_start[p.b] = p.tile_start[p.b];
    }
    __syncthreads();
    if (p.cluster_k > 1)
        cluster_arrive();   // this CTA's barriers exist; waited on before any remote access
    // The tile walk reads only the parameters and the shared tables: set it up before the wait.
    TileWalk<T> wk;
    if (tile_lo < tile_hi)
        wk.init(p, s_len, s_start, tile_lo);
    // Everything above overlaps the previous kernels' tails.  Normally global memory is touched
    // only after the dependency wait.  When the previous kernels still running are this library's
    // decodes of the preceding layers (p.early_fetch, inside mlkv_decode_step), they write nothing
    // this one reads except the newest row (position L-1) of the slot an owner appended to, which
    // lies in the last tile of a segment, and the merge scratch (partials, counters).  So the
    // queries and every other tile are fetched at once, and a segment's last tile too when this
    // grid replaces its newest row from K_new/V_new (p.newest_ready; else the producer waits
    // before fetching it); the epilogue warp waits before it writes its first record, and the
    // consumers before they write the last piece (scratch) or, at the latest, before they exit --
    // so this grid finishes only after the previous one, as the next layer's wait expects.
    // The first piece's query fragments come straight from global memory, before the wait when
    // the queries cannot be the previous kernel's output; later pieces find theirs in a slot.
    uint32_t qa[KS][kT ? 2 : 4];
    auto q_rows = [&](int layer, int beta, int j) {
        return q_of(layer) + (static_cast<size_t>(beta) * p.h + static_cast<size_t>(j) * p.G) * D;
    };
    if (early && warp < NCW && tile_lo < tile_hi)
        load_q_frag<D, kT>(qa, q_rows(wk.layer, wk.beta, wk.j), D, p.G, lane);
    if (warp != PL::kProducer && !early)
        grid_dependency_wait();
    if (warp == PL::kEpilogue && lane == 0) {
        grid_dependency_wait();
        if (p.trigger_late)
            grid_dependents_launch();
    }

    // -------------------------------- producer warp --------------------------------------------
    // Every lane walks the same tiles; lane 0 waits (dependency, free stages) and announces each
    // stage's bytes, and the copies go out from several lanes (issue_tile).
    if (warp == PL::kProducer) {
        if (ml && p.pf_own && lane == 31)
            prefetch_slots_share<D>(p, cta, P);
        int issued = pre_issued ? 1 : 0;
        int tile = tile_lo + issued;
        if (pre_issued)
            wk.next(p, s_len, s_start);
        bool waited = !early;
        if (!early)
            grid_dependency_wait();
        // The next layer's queries (an input of the whole step) go to L2 now: its CTAs load
        // them first thing, while this layer still streams.  Each CTA takes a 128-byte-aligned
        // share.  Issued from the last lane, which issues no tile copies.
        if (p.Q_next != nullptr && lane == 31) {
            const size_t qbytes = static_cast<size_t>(p.b) * p.h * D * 2;   // a multiple of 128
            const size_t lo = (qbytes * cta / P) & ~static_cast<size_t>(127);
            const size_t hi =
                cta + 1 == P ? qbytes : (qbytes * (cta + 1) / P) & ~static_cast<size_t>(127);
            if (hi > lo)
                bulk_prefetch_l2(reinterpret_cast<const uint8_t *>(p.Q_next) + lo,
                                 static_cast<uint32_t>(hi - lo));
        }
        for (; tile < tile_hi; ++tile) {
            if (!waited && wk.tt == wk.nt - 1 && !p.newest_ready) {
                grid_dependency_wait();   // this tile holds the newest row
                waited = true;
            }
            const int s = issued % STAGES;
            int stop = 0;
            if (lane == 0) {
                if (issued >= STAGES && !flags[0] &&
                    !mbar_wait(bar_empty + 8 * s, ((issued / STAGES) & 1) ^ 1)) {
                    flags[0] = 1;
                    atomicOr(p.err, kErrWaitEmpty);
                }
                stop = flags[0];
            }
            if (__shfl_sync(0xffffffffu, stop, 0))
                break;
            // A later piece starts here: its query rows come with the tile.
            issue_tile(wk, s, wk.tt == wk.t0 && tile != tile_lo);
            ++issued;
            wk.next(p, s_len, s_start);
        }
        // No copy may still be in flight when the CTA exits.
        if (lane == 0) {
            const int first = issued > STAGES ? issued - STAGES : 0;
            for (int k = first; k < issued; ++k)
                if (!mbar_wait(bar_full + 8 * (k % STAGES), (k / STAGES) & 1))
                    atomicOr(p.err, kErrDrain);
        }
        __syncwarp();
        if (p.cluster_k > 1)
            cluster_wait();
        return;
    }

    // -------------------------------- epilogue warp --------------------------------------------
    if (warp == PL::kEpilogue) {
        // Merges the consumer warps' raw sums of every piece but the CTA's last while the
        // consumers go on with the next piece: row by row m* = max_w m_w, l* = sum_w l_w 2^(m_w -
        // m*), o = sum_w 2^(m_w - m*) o_w / l*, lse = m* + log2 l*.
        constexpr int FS = PL::kRawRow;
        for (int k = 0;; ++k) {
            const int rb = k & two;
            int ok = 1;
            if (lane == 0 && !mbar_wait(bar_res_full + 8 * rb, (k >> two) & 1)) {
                flags[0] = 1;
                atomicOr(p.err, kErrWaitFull);
                ok = 0;
            }
            ok = __shfl_sync(0xffffffffu, ok, 0);
            if (!ok)
                break;
            uint8_t *slot = smem + raw_at(rb);
            const int *meta = reinterpret_cast<const int *>(slot + PL::kRawMeta);
            if (meta[kMetaStop])
                break;
            if (early && k == 0)
                grid_dependency_wait();   // records and merges use the shared scratch
            const int G = p.G;
            const int seg = meta[kMetaSeg], whole = meta[kMetaWhole];
            const int c_first = meta[kMetaFirst], c_last = meta[kMetaLast];
            __nv_bfloat16 *ob =
                p.out + static_cast<size_t>(meta[kMetaLayer]) * p.ml_q_stride +
                (static_cast<size_t>(meta[kMetaBeta]) * p.h + static_cast<size_t>(meta[kMetaJ]) * G) * D;
            // partial record seg + cta; a multi-layer launch's travels in kMetaFirst (its merge is
            // deferred)
            const size_t piece = ml ? static_cast<size_t>(c_first) : static_cast<size_t>(seg + cta);
            const bool stop = flags[0] != 0;
            const float *raw = reinterpret_cast<const float *>(slot);
            float *st_m = reinterpret_cast<float *>(slot + PL::kRawO);   // [16][NCW]
            const float *st_l = st_m + 16 * NCW;
            if (lane < G) {
                // lane r: row r's factors 2^(m_w - m*) / l* in place of m_w
                float mw[NCW], lw[NCW];
#pragma unroll
                for (int w = 0; w < NCW; ++w) {
                    mw[w] = st_m[lane * NCW + w];
                    lw[w] = st_l[lane * NCW + w];
                }
                float ms = mw[0];
#pragma unroll
                for (int w = 1; w < NCW; ++w)
                    ms = fmaxf(ms, mw[w]);   // finite: the piece holds a visible position
                float ls = 0.f;
#pragma unroll
                for (int w = 0; w < NCW; ++w) {
                    mw[w] = fast_exp2(mw[w] - ms);
                    ls = fmaf(lw[w], mw[w], ls);
                }
                const float inv = fast_rcp(ls);
#pragma unroll
                for (int w = 0; w < NCW; ++w)
                    st_m[lane * NCW + w] = mw[w] * inv;
                if (!whole && !stop)
                    p.part_lse[piece * G + lane] = ms + fast_log2(ls);
            }
            __syncwarp();
            constexpr int E = D / 32;   // a lane's columns lane E .. lane E + E - 1 of every row
            using Vec = typename std::conditional<E == 2, float2, float4>::type;
            auto store_out = [&](int r, const float (&x)[E]) {
                if constexpr (E == 2)
                    *reinterpret_cast<uint32_t *>(ob + r * D + lane * E) = pack_bf16x2(x[0], x[1]);
                else
                    *reinterpret_cast<uint2 *>(ob + r * D + lane * E) =
                        make_uint2(pack_bf16x2(x[0], x[1]), pack_bf16x2(x[2], x[3]));
            };
#pragma unroll 4
            for (int r = 0; r < G; ++r) {
                alignas(16) float v[E] = {};
#pragma unroll
                for (int w = 0; w < NCW; ++w) {
                    const float f = st_m[r * NCW + w];
                    const Vec x = *reinterpret_cast<const Vec *>(raw + (w * PL::kRows + r) * FS +
                                                                 lane * E);
                    const float *xe = reinterpret_cast<const float *>(&x);
#pragma unroll
                    for (int e = 0; e < E; ++e)
                        v[e] = fmaf(f, xe[e], v[e]);
                }
                if (whole && !stop) {
                    store_out(r, v);
                } else if (!stop) {
                    *reinterpret_cast<Vec *>(p.part_o + (piece * G + r) * D + lane * E) =
                        *reinterpret_cast<const Vec *>(v);
                }
            }
            // The buffer is free before the counter's round trip and a merge of records.
            __syncwarp();
            if (lane == 0)
                mbar_arrive(bar_res_empty + 8 * rb);
            if (whole || stop || p.deferred_merge)
                continue;
            unsigned prev = 0;
            if (lane == 0)
                prev = atomic_add_acq_rel_gpu(&p.counters[seg], 1u);
            prev = __shfl_sync(0xffffffffu, prev, 0);
            __syncwarp();
            if (prev != static_cast<unsigned>(c_last - c_first))
                continue;
            // This CTA finished the segment last: it merges records seg + c_first .. seg + c_last (at
            // most PL::kMaxPieces), o = sum_c 2^(lse_c - M) o_c / sum_c 2^(lse_c - M), M the
            // largest lse; the weights first, then the sums in the records' order, as the consumer
            // warps do (merge4): the outputs do not depend on which CTA is last.
            float *s_w = reinterpret_cast<float *>(smem + PL::kEpiW);
            const int np = c_last - c_first + 1;
            const size_t rec0 = static_cast<size_t>(seg + c_first);
            // Lane r: row r's log-sum-exps, in flight with the first records.  (One round trip to L2
            // after the other, with the weights' chain through shared memory between them, was the
            // launch's last microsecond: 64 uneven segments over 138 CTAs, 32 heads of 128, 12.7 us a
            // layer, now 12.1.)
            float lv[PL::kMaxPieces];
#pragma unroll
            for (int c = 0; c < PL::kMaxPieces; ++c)
                lv[c] = (lane < G && c < np) ? __ldcg(&p.part_lse[(rec0 + c) * G + lane])
                                             : -__int_as_float(0x7f800000);
            bool weighed = false;
            // 4 x 4 columns a lane of 4 records in flight at a time (8 records at once: longer code,
            // fetched cold, 4% slower).
            const float *base = p.part_o + rec0 * G * D;
            constexpr int CH = 4;
            for (int cb = 0; cb < G * D; cb += 128 * CH) {
                const int c0 = cb + 4 * lane;
                float4 acc[CH];
#pragma unroll
                for (int u = 0; u < CH; ++u)
                    acc[u] = make_float4(0.f, 0.f, 0.f, 0.f);
                for (int c = 0; c < np; c += 4) {
                    float4 x[4][CH];
#pragma unroll
                    for (int q = 0; q < 4; ++q)
#pragma unroll
                        for (int u = 0; u < CH; ++u) {
                            const int i = c0 + u * 128;
                            x[q][u] = (i < G * D && c + q < np)
                                          ? __ldcg(reinterpret_cast<const float4 *>(
                                                base + static_cast<size_t>(c + q) * G * D + i))
                                          : make_float4(0.f, 0.f, 0.f, 0.f);
                        }
                    if (!weighed) {
                        weighed = true;
                        if (lane < G) {
                            float mx = lv[0];
#pragma unroll
                            for (int k = 1; k < PL::kMaxPieces; ++k)
                                mx = fmaxf(mx, lv[k]);
                            float tot = 0.f;
#pragma unroll
                            for (int k = 0; k < PL::kMaxPieces; ++k) {
                                lv[k] = fast_exp2(lv[k] - mx);   // 0 past the records
                                tot += lv[k];
                            }
                            const float inv = fast_rcp(tot);
#pragma unroll
                            for (int k = 0; k < PL::kMaxPieces; ++k)
                                s_w[k * G + lane] = lv[k] * inv;
                        }
                        __syncwarp();
                    }
#pragma unroll
                    for (int q = 0; q < 4; ++q)
#pragma unroll
                        for (int u = 0; u < CH; ++u) {
                            const int i = c0 + u * 128;
                            const float w =
                                (i < G * D && c + q < np) ? s_w[(c + q) * G + i / D] : 0.f;
                            acc[u].x = fmaf(w, x[q][u].x, acc[u].x);
                            acc[u].y = fmaf(w, x[q][u].y, acc[u].y);
                            acc[u].z = fmaf(w, x[q][u].z, acc[u].z);
                            acc[u].w = fmaf(w, x[q][u].w, acc[u].w);
                        }
                }
#pragma unroll
                for (int u = 0; u < CH; ++u) {
                    const int i = c0 + u * 128;
                    if (i < G * D)
                        *reinterpret_cast<uint2 *>(ob + i) =
                            make_uint2(pack_bf16x2(acc[u].x, acc[u].y),
                                       pack_bf16x2(acc[u].z, acc[u].w));
                }
            }
            __syncwarp();   // s_w may be rewritten
            if (lane == 0)
                p.counters[seg] = 0u;
        }
        __syncwarp();
        if (p.cluster_k > 1)
            cluster_wait();
        return;
    }

    // -------------------------------- consumer warps -------------------------------------------
    const int qr = lane >> 2;              // fragment row (query head within the group)
    const int qc = (lane & 3) * 2;         // fragment column pair
    const int G = p.G;
    const float scale = p.scale_log2;
    const float NEG_INF = -__int_as_float(0x7f800000);

    int it = 0;
    int nhand = 0;   // pieces handed to the epilogue warp (all but the CTA's last)
    int tile = tile_lo;

    while (tile < tile_hi) {
        const int beta = wk.beta;
        const int j = wk.j;
        const int L = wk.L;
        const int seg = beta * p.g + j;
        const int layer = wk.layer;
        const int rec = wk.rec;   // partial-record index of a chunked multi-layer piece
        const bool part = p.ml_chunks > 1;   // chunks are always partial records
        const int slot = slot_of(layer);
        const int store_new = ml ? static_cast<int>(p.ml_store[layer]) : p.store_new;
        const __nv_bfloat16 *k_new = p.K_new;
        const __nv_bfloat16 *v_new = p.V_new;
        if (ml && k_new != nullptr) {
            k_new += static_cast<size_t>(slot) * p.ml_kv_stride;
            v_new += static_cast<size_t>(slot) * p.ml_kv_stride;
        }
        const int seg_first = wk.seg_first;
        const int seg_end = seg_first + wk.nt;
        const int piece_first = tile;
        const int piece_end = seg_end < tile_hi ? seg_end : tile_hi;

        if (tile == tile_lo) {
            if (!early)
                load_q_frag<D, kT>(qa, q_rows(layer, beta, j), D, G, lane);
        } else {
            // A later piece: its query rows arrive with its first tile (the loop's wait for that
            // tile then returns at once).
            const int s0 = it % STAGES;
            if (!flags[0] && !mbar_wait(bar_full + 8 * s0, (it / STAGES) & 1)) {
                flags[0] = 1;
                atomicOr(p.err, kErrWaitFull);
            }
            load_q_frag<D, kT>(
                qa, reinterpret_cast<const __nv_bfloat16 *>(smem + PL::kQ + s0 * PL::kQSlot),
                PL::kQRow / 2, G, lane);
        }

        float o[NO][4];
#pragma unroll
        for (int n = 0; n < NO; ++n)
            o[n][0] = o[n][1] = o[n][2] = o[n][3] = 0.f;
        float m_run[2] = {NEG_INF, NEG_INF};
        // Row sums of P, accumulated on the tensor core: P times a block of ones (every column
        // of la holds its row's sum; kT: every row its column's), in fp32 from the same bf16
        // weights P V uses.  A thread's two statistics (m_run, la) are those of rows qr and qr + 8,
        // or (kT) of heads qc and qc + 1.
        float la[4] = {0.f, 0.f, 0.f, 0.f};

        for (; tile < piece_end; ++tile, ++it) {
            const int s = it % STAGES;
            if (!flags[0] && !mbar_wait(bar_full + 8 * s, (it / STAGES) & 1)) {
                flags[0] = 1;
                atomicOr(p.err, kErrWaitFull);
            }
            const int row0 = warp * TW;                 // this warp's first row in the tile
            const int valid = L - (wk.tt * T + row0);   // visible rows in this warp's slice
            if (!flags[0] && valid > 0) {
                const uint32_t kt = sbase + s * PL::kStageBytes;
                const uint32_t vt = kt + PL::kTileBytes;
                if (k_new != nullptr && valid <= TW) {
                    // Fused append: this warp's slice holds position L-1, the new token.  Its K/V
                    // replace the tile rows (the copy may have read the cache before the token was
                    // stored) and, in the owner layer, are stored in the cache for the layers that
                    // read this slot later.
                    const int r_new = row0 + valid - 1;
                    if (lane < 8 * PL::kSub) {
                        const size_t src = (static_cast<size_t>(beta) * p.g + j) * D + lane * 8;
                        const uint4 kn = *reinterpret_cast<const uint4 *>(k_new + src);
                        const uint4 vn = *reinterpret_cast<const uint4 *>(v_new + src);
                        uint8_t *st = smem + s * PL::kStageBytes;
                        *reinterpret_cast<uint4 *>(st + swz<T>(r_new, lane)) = kn;
                        *reinterpret_cast<uint4 *>(st + PL::kTileBytes + swz<T>(r_new, lane)) = vn;
                        if (store_new) {
                            const size_t dst =
                                ((((static_cast<size_t>(slot) * 2) * p.b + beta) * p.g + j) *
                                     static_cast<size_t>(p.max_seq) + (L - 1)) * D + lane * 8;
                            *reinterpret_cast<uint4 *>(p.cache + dst) = kn;
                            *reinterpret_cast<uint4 *>(
                                p.cache + dst + static_cast<size_t>(p.b) * p.g * p.max_seq * D) = vn;
                        }
                    }
                    fence_proxy_async_smem();
                    __syncwarp();
                }
                if (valid < TW) {
                    // Rows past the sequence end hold whatever the cache holds there; zero the V
                    // rows so that 0-weight * V stays 0 even for non-finite contents.
                    uint8_t *vrow = smem + s * PL::kStageBytes + PL::kTileBytes;
                    const int nrows = TW - valid;
                    for (int idx = lane; idx < nrows * 8 * PL::kSub; idx += 32) {
                        const int rr = row0 + valid + idx / (8 * PL::kSub);
                        const int rem = idx % (8 * PL::kSub);
                        const int sub = rem / 8;
                        *reinterpret_cast<uint4 *>(vrow + sub * T * 128 + rr * 128 +
                                                   (rem % 8) * 16) = make_uint4(0, 0, 0, 0);
                    }
                    fence_proxy_async_smem();
                    __syncwarp();
                }

                // ---- S = Q K^T for this warp's TW positions ----
                float sc[NT][4];
#pragma unroll
                for (int n = 0; n < NT; ++n)
                    sc[n][0] = sc[n][1] = sc[n][2] = sc[n][3] = 0.f;
                const int mi = lane >> 3;   // which 8x8 matrix this lane addresses
                const int mr = lane & 7;    // which row of it
                // The K fragments of a group of up to 8 shared-memory loads go out together and
                // the MMAs follow, so the loads' latency (~47 cycles each) is paid once per group.
                constexpr int KL = kT ? NT : NT / 2;   // loads per reduction step
                constexpr int KG = (KS * KL <= 8) ? KS : (8 / KL > 0 ? 8 / KL : 1);
#pragma unroll
                for (int k0 = 0; k0 < KS; k0 += KG) {
                    uint32_t kf[KG][KL][4];
#pragma unroll
                    for (int kg = 0; kg < KG; ++kg) {
#pragma unroll
                        for (int n2 = 0; n2 < KL; ++n2) {
                            const int row = row0 + 16 * n2 + 8 * (kT ? (mi & 1) : (mi >> 1)) + mr;
                            const int chunk = 2 * (k0 + kg) + (kT ? (mi >> 1) : (mi & 1));
                            ldsm_x4(kt + swz<T>(row, chunk), kf[kg][n2][0], kf[kg][n2][1],
                                    kf[kg][n2][2], kf[kg][n2][3]);
                        }
                    }
#pragma unroll
                    for (int kg = 0; kg < KG; ++kg) {
#pragma unroll
                        for (int n2 = 0; n2 < KL; ++n2) {
                            if constexpr (kT) {
                                mma_bf16_16816(sc[n2], kf[kg][n2], qa[k0 + kg][0], qa[k0 + kg][1]);
                            } else {
                                mma_bf16_16816(sc[2 * n2], qa[k0 + kg], kf[kg][n2][0],
                                               kf[kg][n2][1]);
                                mma_bf16_16816(sc[2 * n2 + 1], qa[k0 + kg], kf[kg][n2][2],
                                               kf[kg][n2][3]);
                            }
                        }
                    }
                }
                // The V fragments of the first group of P V (up to 8 loads) go out now: their
                // latency overlaps the softmax below.
                constexpr int NG = kT ? NT : NT / 2;               // groups of 16 positions
                constexpr int VQ = kT ? NO : NO / 2;               // loads per 16 positions
                constexpr int VG = (VQ * NG <= 8) ? NG : (8 / VQ > 0 ? 8 / VQ : 1);
                auto load_v = [&](int grp, int q, uint32_t (&f)[4]) {
                    const int row = row0 + 16 * grp + 8 * (kT ? (mi >> 1) : (mi & 1)) + mr;
                    const int chunk = 2 * q + (kT ? (mi & 1) : (mi >> 1));
                    ldsm_x4_trans(vt + swz<T>(row, chunk), f[0], f[1], f[2], f[3]);
                };
                uint32_t vf[VG][VQ][4];
#pragma unroll
                for (int kg = 0; kg < VG; ++kg)
#pragma unroll
                    for (int q = 0; q < VQ; ++q)
                        load_v(kg, q, vf[kg][q]);

                // ---- online softmax (base 2, scale folded into the exponent) ----
                float mx[2] = {NEG_INF, NEG_INF};
                if (valid < TW) {
#pragma unroll
                    for (int n = 0; n < NT; ++n) {
#pragma unroll
                        for (int c = 0; c < 4; ++c) {
                            const int pos_in_slice =
                                kT ? 16 * n + qr + 8 * (c >> 1) : 8 * n + qc + (c & 1);
                            if (pos_in_slice >= valid)
                                sc[n][c] = NEG_INF;
                        }
                    }
                }
#pragma unroll
                for (int n = 0; n < NT; ++n) {
                    mx[0] = fmaxf(mx[0], fmaxf(sc[n][0], sc[n][kT ? 2 : 1]));
                    mx[1] = fmaxf(mx[1], fmaxf(sc[n][kT ? 1 : 2], sc[n][3]));
                }
                // The reference maximum moves only when a score exceeds it by more than 2^8 (in
                // the exponent): weights then stay in [0, 256], exactly as accurate in bf16, and
                // most tiles need neither the quad reduction nor a rescale.  When one does, the
                // rows' exact maxima over this tile become the new references.
                const bool raise = mx[0] * scale > m_run[0] + kLazyMax ||
                                   mx[1] * scale > m_run[1] + kLazyMax;
                if (__any_sync(0xffffffffu, raise)) {
                    float alpha[2];
#pragma unroll
                    for (int hr = 0; hr < 2; ++hr) {
                        if constexpr (kT) {
                            mx[hr] = fmaxf(mx[hr], __shfl_xor_sync(0xffffffffu, mx[hr], 4));
                            mx[hr] = fmaxf(mx[hr], __shfl_xor_sync(0xffffffffu, mx[hr], 8));
                            mx[hr] = fmaxf(mx[hr], __shfl_xor_sync(0xffffffffu, mx[hr], 16));
                        } else {
                            mx[hr] = fmaxf(mx[hr], __shfl_xor_sync(0xffffffffu, mx[hr], 1));
                            mx[hr] = fmaxf(mx[hr], __shfl_xor_sync(0xffffffffu, mx[hr], 2));
                        }
                        const float m_new = fmaxf(m_run[hr], mx[hr] * scale);
                        alpha[hr] = (m_new == NEG_INF) ? 1.f : fast_exp2(m_run[hr] - m_new);
                        m_run[hr] = m_new;
                    }
#pragma unroll
                    for (int n = 0; n < NO; ++n) {
                        o[n][0] *= alpha[0];
                        o[n][1] *= alpha[kT ? 1 : 0];
                        o[n][2] *= alpha[kT ? 0 : 1];
                        o[n][3] *= alpha[1];
                    }
                    la[0] *= alpha[0];
                    la[1] *= alpha[kT ? 1 : 0];
                    la[2] *= alpha[kT ? 0 : 1];
                    la[3] *= alpha[1];
                }
                const float m_use[2] = {m_run[0] == NEG_INF ? 0.f : m_run[0],
                                        m_run[1] == NEG_INF ? 0.f : m_run[1]};
                // P in bf16: the mma A operand, or (kT) P^T as the B operand, its 8 x 8 blocks
                // turned from [position][head] pairs to position pairs of one head.
                uint32_t pa[NG][kT ? 2 : 4];
#pragma unroll
                for (int n = 0; n < NT; ++n) {
                    const float p0 = fast_exp2(fmaf(sc[n][0], scale, -m_use[0]));
                    const float p1 = fast_exp2(fmaf(sc[n][1], scale, -m_use[kT ? 1 : 0]));
                    const float p2 = fast_exp2(fmaf(sc[n][2], scale, -m_use[kT ? 0 : 1]));
                    const float p3 = fast_exp2(fmaf(sc[n][3], scale, -m_use[1]));
                    if constexpr (kT) {
                        pa[n][0] = movmatrix_trans(pack_bf16x2(p0, p1));
                        pa[n][1] = movmatrix_trans(pack_bf16x2(p2, p3));
                    } else {
                        pa[n >> 1][(n & 1) * 2 + 0] = pack_bf16x2(p0, p1);
                        pa[n >> 1][(n & 1) * 2 + 1] = pack_bf16x2(p2, p3);
                    }
                }

                // ---- O += P V ----
                const uint32_t ones[4] = {kOnesBf16x2, kOnesBf16x2, kOnesBf16x2, kOnesBf16x2};
                auto add_pv = [&](int grp, const uint32_t (&f)[VQ][4]) {
#pragma unroll
                    for (int q = 0; q < VQ; ++q) {
                        if constexpr (kT) {
                            mma_bf16_16816(o[q], f[q], pa[grp][0], pa[grp][1]);
                        } else {
                            mma_bf16_16816(o[2 * q], pa[grp], f[q][0], f[q][1]);
                            mma_bf16_16816(o[2 * q + 1], pa[grp], f[q][2], f[q][3]);
                        }
                    }
                    if constexpr (kT)
                        mma_bf16_16816(la, ones, pa[grp][0], pa[grp][1]);
                    else
                        mma_bf16_16816(la, pa[grp], kOnesBf16x2, kOnesBf16x2);
                };
#pragma unroll
                for (int kg = 0; kg < VG; ++kg)
                    add_pv(kg, vf[kg]);
                // the remaining 16-position groups (longer tiles), a group's loads first
#pragma unroll
                for (int k0 = VG; k0 < NG; k0 += VG) {
                    uint32_t vg[VG][VQ][4];
#pragma unroll
                    for (int kg = 0; kg < VG; ++kg)
#pragma unroll
                        for (int q = 0; q < VQ; ++q)
                            load_v(k0 + kg, q, vg[kg][q]);
#pragma unroll
                    for (int kg = 0; kg < VG; ++kg)
                        add_pv(k0 + kg, vg[kg]);
                }
            }
            __syncwarp();
            if (lane == 0)
                mbar_arrive(bar_empty + 8 * s);
            wk.next(p, s_len, s_start);
        }

        // ---------------- end of piece: every warp's raw sums to the piece's buffer -------------
        // Pieces before the CTA's last go to the epilogue warp, and each warp goes straight on to
        // the next piece (a tree over the warps with a barrier per level held all of them up for
        // ~2 us a piece at head_dim 128).
        constexpr int FS = PL::kRawRow;
        const int rb = nhand & two;
        uint8_t *slot_raw = smem + raw_at(rb);
        if (nhand > two && !flags[0] &&
            !mbar_wait(bar_res_empty + 8 * rb, ((nhand >> two) & 1) ^ 1)) {
            flags[0] = 1;
            atomicOr(p.err, kErrWaitEmpty);
        }
        float *fbuf = reinterpret_cast<float *>(slot_raw);                       // [NCW][kRows][FS]
        float *red_m = reinterpret_cast<float *>(slot_raw + PL::kRawO);          // [16][NCW]
        float *red_l = red_m + 16 * NCW;
        float *flse = reinterpret_cast<float *>(slot_raw + PL::kRawLse);         // [16]
#pragma unroll
        for (int hr = 0; hr < 2; ++hr) {
            const int row = kT ? qc + hr : qr + 8 * hr;
            if (row < G) {
                float *dst = fbuf + (warp * PL::kRows + row) * FS;
#pragma unroll
                for (int n = 0; n < NO; ++n) {
                    if constexpr (kT) {
                        dst[n * 16 + qr] = o[n][hr];
                        dst[n * 16 + 8 + qr] = o[n][2 + hr];
                    } else {
                        *reinterpret_cast<float2 *>(dst + n * 8 + qc) =
                            make_float2(o[n][2 * hr], o[n][2 * hr + 1]);
                    }
                }
                if (kT ? qr == 0 : qc == 0) {
                    red_m[row * NCW + warp] = m_run[hr];
                    red_l[row * NCW + warp] = la[kT ? hr : 2 * hr];
                }
            }
        }
        if (piece_end != tile_hi) {
            if (warp == 0 && lane == 0) {
                int *meta = reinterpret_cast<int *>(slot_raw + PL::kRawMeta);
                meta[kMetaBeta] = beta;
                meta[kMetaJ] = j;
                meta[kMetaSeg] = seg;
                meta[kMetaWhole] =
                    (piece_first == seg_first && piece_end == seg_end && !part) ? 1 : 0;
                meta[kMetaFirst] = ml ? rec : cta_of_tile(seg_first, N, P);
                meta[kMetaLast] = cta_of_tile(seg_end - 1, N, P);
                meta[kMetaStop] = 0;
                meta[kMetaLayer] = layer;
            }
            __syncwarp();
            if (lane == 0)
                mbar_arrive(bar_res_full + 8 * rb);
            ++nhand;
        } else {
            // ---- the CTA's last piece: after one barrier the consumer threads finish it together,
            // four columns each a pass, from every warp's statistics of their row (as the epilogue
            // warp does).
            if (p.cluster_k > 1)
                cluster_wait();   // the partner CTAs' barriers exist
            consumer_bar_sync<NCW>();
            const int ctid = threadIdx.x;
            const bool whole = (piece_first == seg_first && piece_end == seg_end && !part);
            __nv_bfloat16 *ob = p.out + static_cast<size_t>(layer) * p.ml_q_stride +
                                (static_cast<size_t>(beta) * p.h + static_cast<size_t>(j) * G) * D;
            constexpr int kPass = 4 * NCW * 32;   // outputs per pass
            // One or two passes (groups of at most 8 heads, or head_dim 64) take the shorter code,
            // which is fetched cold once a launch; up to four overlap in pairs.
            constexpr int kPassUnroll = (!kT && D == 128) ? 2 : 1;
            static_assert(D % 4 == 0, "a thread's four columns lie in one row");
            // mode: 0 whole, 1 cluster sender, 2 cluster leader, 3 partial record
            const int rank = p.cluster_k > 1 ? static_cast<int>(cluster_ctarank()) : 0;
            const int mode = whole ? 0 : (p.cluster_k > 1 ? (rank != 0 ? 1 : 2) : 3);
            if (early && mode == 3)
                grid_dependency_wait();   // partial records and counters are shared scratch
            const uint32_t cslots = sbase + PL::kTail;
            const uint8_t *cs = smem + PL::kTail;
            uint32_t remote = 0, remote_bar = 0;
            if (mode == 1) {
                remote = map_to_rank(cslots + (rank - 1) * PL::kResBytes, 0);
                remote_bar = map_to_rank(bar_cluster, 0);
            }
            const size_t piece = ml ? static_cast<size_t>(rec) : static_cast<size_t>(seg + cta);
            float *po = p.part_o + piece * G * D;
#pragma unroll kPassUnroll
            for (int i = 4 * ctid; i < G * D; i += kPass) {
                const int row = i / D, e = i - row * D;
                // independent loads of the row's statistics of every warp
                float mw[NCW], lw[NCW];
#pragma unroll
                for (int w = 0; w < NCW; ++w) {
                    mw[w] = red_m[row * NCW + w];
                    lw[w] = red_l[row * NCW + w];
                }
                float ms = mw[0];   // finite: the piece holds a visible position
#pragma unroll
                for (int w = 1; w < NCW; ++w)
                    ms = fmaxf(ms, mw[w]);
                float ls = 0.f;
                float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                for (int w = 0; w < NCW; ++w) {
                    const float ew = fast_exp2(mw[w] - ms);
                    ls = fmaf(lw[w], ew, ls);
                    const float4 x =
                        *reinterpret_cast<const float4 *>(fbuf + (w * PL::kRows + row) * FS + e);
                    v.x = fmaf(ew, x.x, v.x);
                    v.y = fmaf(ew, x.y, v.y);
                    v.z = fmaf(ew, x.z, v.z);
                    v.w = fmaf(ew, x.w, v.w);
                }
                const float inv = fast_rcp(ls);
                v.x *= inv;
                v.y *= inv;
                v.z *= inv;
                v.w *= inv;
                const float lse_row = ms + fast_log2(ls);
                const bool row_head = e == 0;   // one thread per row
                if (mode == 0) {
                    *reinterpret_cast<uint2 *>(ob + i) =
                        make_uint2(pack_bf16x2(v.x, v.y), pack_bf16x2(v.z, v.w));
                } else if (mode == 1) {
                    // the leader's barrier completes when all these bytes have landed
                    st_async_v4(remote + i * 4, v, remote_bar);
                    if (row_head)
                        st_async_f32(remote + PL::kResO + row * 4, lse_row, remote_bar);
                } else if (mode == 2) {
                    // each element is read and rewritten by this thread alone
                    *reinterpret_cast<float4 *>(fbuf + row * FS + e) = v;
                    if (row_head)
                        flse[row] = lse_row;
                } else {
                    *reinterpret_cast<float4 *>(po + i) = v;
                    if (row_head)
                        p.part_lse[piece * G + row] = lse_row;
                }
            }
            // Weighted mean of the four columns of up to K records.
            auto merge4 = [&](const auto &l, const auto &x) {
                constexpr int K = sizeof(l) / sizeof(l[0]);
                float mx = NEG_INF;
#pragma unroll
                for (int k = 0; k < K; ++k)
                    mx = fmaxf(mx, l[k]);
                float tot = 0.f, w[K];
#pragma unroll
                for (int k = 0; k < K; ++k) {
                    w[k] = fast_exp2(l[k] - mx);   // 0 past the records
                    tot += w[k];
                }
                const float inv = fast_rcp(tot);
                float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                for (int k = 0; k < K; ++k) {
                    const float f = w[k] * inv;
                    a.x = fmaf(f, x[k].x, a.x);
                    a.y = fmaf(f, x[k].y, a.y);
                    a.z = fmaf(f, x[k].z, a.z);
                    a.w = fmaf(f, x[k].w, a.w);
                }
                return make_uint2(pack_bf16x2(a.x, a.y), pack_bf16x2(a.z, a.w));
            };
            if (mode == 2) {
                // Leader: its own result is in warp 0's rows; merge the other ranks' once landed.
                if (!flags[0] && !mbar_wait_cluster(bar_cluster, 0)) {
                    flags[0] = 1;
                    atomicOr(p.err, kErrWaitFull);
                }
                consumer_bar_sync<NCW>();   // flse is complete
                const int k = p.cluster_k;   // 2 or 4
                const bool stop = flags[0] != 0;
#pragma unroll kPassUnroll
                for (int i = 4 * ctid; i < G * D; i += kPass) {
                    const int row = i / D, e = i - row * D;
                    float lr[4];
                    float4 x[4];
                    lr[0] = flse[row];
                    x[0] = *reinterpret_cast<const float4 *>(fbuf + row * FS + e);
#pragma unroll
                    for (int r = 1; r < 4; ++r) {
                        lr[r] = NEG_INF;
                        x[r] = make_float4(0.f, 0.f, 0.f, 0.f);
                        if (r < k) {
                            const uint8_t *sl = cs + (r - 1) * PL::kResBytes;
                            lr[r] = reinterpret_cast<const float *>(sl + PL::kResO)[row];
                            x[r] = *reinterpret_cast<const float4 *>(sl + static_cast<size_t>(i) * 4);
                        }
                    }
                    const uint2 o4 = merge4(lr, x);
                    if (!stop)
                        *reinterpret_cast<uint2 *>(ob + i) = o4;
                }
            } else if (mode == 3 && !p.deferred_merge) {
                const int c_first = cta_of_tile(seg_first, N, P);
                const int c_last = cta_of_tile(seg_end - 1, N, P);
                // The barrier puts every thread's record before thread 0's release.
                consumer_bar_sync<NCW>();
                if (ctid == 0) {
                    const unsigned prev = atomic_add_acq_rel_gpu(&p.counters[seg], 1u);
                    flags[1] = (prev == static_cast<unsigned>(c_last - c_first)) ? 1 : 0;
                }
                consumer_bar_sync<NCW>();
                if (flags[1]) {
                    // Last finisher of the segment: merge its <= 8 records (own included), every
                    // record's loads of a pass in flight together.
                    const int np = c_last - c_first + 1;
                    const size_t rec0 = static_cast<size_t>(seg + c_first);
#pragma unroll 1
                    for (int i = 4 * ctid; i < G * D; i += kPass) {
                        const int row = i / D;
                        float lv[PL::kMaxPieces];
                        float4 ov[PL::kMaxPieces];
#pragma unroll
                        for (int k = 0; k < PL::kMaxPieces; ++k) {
                            lv[k] = NEG_INF;
                            ov[k] = make_float4(0.f, 0.f, 0.f, 0.f);
                            if (k < np) {
                                lv[k] = __ldcg(&p.part_lse[(rec0 + k) * G + row]);
                                ov[k] = __ldcg(reinterpret_cast<const float4 *>(
                                    p.part_o + (rec0 + k) * G * D + i));
                            }
                        }
                        *reinterpret_cast<uint2 *>(ob + i) = merge4(lv, ov);
                    }
                    if (ctid == 0)
                        p.counters[seg] = 0u;
                }
                consumer_bar_sync<NCW>();   // flags[1] is reused
            }
        }
    }
    if (early)
        grid_dependency_wait();   // no-op if already waited; this grid ends after the previous
    // Tell the epilogue warp that no piece follows (the buffer is this piece's own; with no tiles at
    // all it was never used).
    {
        const int rb = nhand & two;
        if (warp == 0 && lane == 0)
            reinterpret_cast<int *>(smem + raw_at(rb) + PL::kRawMeta)[kMetaStop] = 1;
        __syncwarp();
        if (lane == 0)
            mbar_arrive(bar_res_full + 8 * rb);
    }
}


// ------------------------------------------------------------------------------------------------
// combine kernel: merge of segments split over many CTAs
// ------------------------------------------------------------------------------------------------

// One CTA per (segment, query row of its group).  The CTA turns the pieces' log-sum-exps into
// weights w_c = 2^(lse_c - M) (M = max_c lse_c) and each thread sums w_c * o_c[e] for one column
// e over a strided subset of the pieces, 16 loads in flight (the first 16 issued with the
// log-sum-exps); the subsets are added through shared memory and scaled by 1 / sum_c w_c.
constexpr int kCombineThreads = 256;
constexpr int kCombineMaxPieces = 1024;

template <int D>
__global__ void __launch_bounds__(kCombineThreads)
    combine_kernel(const __grid_constant__ DecodeParams p)
{
    __shared__ float s_w[kCombineMaxPieces];
    __shared__ float s_red[kCombineThreads];
    // The next layer's decode may start at once: it reads neither the partials nor `out`, and it
    // writes partials only after its own dependency wait (after this grid).
    grid_dependents_launch();
    // Uneven lengths wait here, the others behind the divisions (below): there it measured no gain
    // for them (3 sequences of up to 3,000 positions, 32 layers of 8 KV heads: 323 us here, 325).
    const bool uneven = p.ml_layers <= 0 && p.uniform_len <= 0;
    if (uneven)
        grid_dependency_wait();
    const int row = blockIdx.y;
    const int G = p.G;
    int seg, np;
    size_t rec0;
    __nv_bfloat16 *out = p.out;
    if (p.ml_layers > 0) {
        // a chunked multi-layer launch: blockIdx.x = layer b g + beta g + j, chunk records
        // blockIdx.x C .. blockIdx.x C + C - 1
        const int S = p.b * p.g;
        const int layer = static_cast<int>(blockIdx.x) / S;
        seg = static_cast<int>(blockIdx.x) - layer * S;
        out += static_cast<size_t>(layer) * p.ml_q_stride;
        np = p.ml_chunks;
        rec0 = static_cast<size_t>(blockIdx.x) * p.ml_chunks;
    } else {
        seg = blockIdx.x;
        const int T = p.tile_tokens;
        const int beta = seg / p.g;
        const int jj = seg - beta * p.g;
        const int L = p.uniform_len > 0 ? p.uniform_len : p.seq_len[beta];
        const int nt = (L + T - 1) / T;
        const int seg_first = p.uniform_len > 0 ? seg * nt : p.tile_start[beta] + jj * nt;
        const int c_first = cta_of_tile(seg_first, p.num_tiles, p.decode_grid);
        const int c_last = cta_of_tile(seg_first + nt - 1, p.num_tiles, p.decode_grid);
        np = c_last - c_first + 1;
        rec0 = static_cast<size_t>(seg + c_first);
    }
    // Behind the divisions, which overlap the decode grid's tail (one sequence of 5,000 positions, 32
    // layers of 8 KV heads: 304 us with the wait in front of them, 292).  A CTA that returns waits
    // too: this grid ends after the decode grid.
    if (!uneven)
        grid_dependency_wait();
    if (p.ml_layers <= 0 && np == 1)
        return;   // one CTA held the whole segment and wrote the output itself
    const int beta = seg / p.g;
    const int j = seg - beta * p.g;
    const int tid = threadIdx.x;
    const int lane = tid & 31, wid = tid >> 5;
    constexpr int kWarps = kCombineThreads / 32;
    const float NEG_INF = -__int_as_float(0x7f800000);
    constexpr int kGroups = kCombineThreads / D;   // pieces summed side by side per column
    const int e = tid % D;
    const int grp = tid / D;
    const float *src = p.part_o + rec0 * G * D + static_cast<size_t>(row) * D + e;
    // The first 16 pieces' values of this thread go out together with the pieces' log-sum-exps:
    // one round trip to memory before the weights are known.
    float v[16];
#pragma unroll
    for (int m = 0; m < 16; ++m) {
        const int k = grp + m * kGroups;
        v[m] = k < np ? __ldcg(src + static_cast<size_t>(k) * G * D) : 0.f;
    }
    float mx = NEG_INF;
    for (int k = tid; k < np; k += kCombineThreads) {
        const float l = __ldcg(&p.part_lse[(rec0 + k) * G + row]);
        s_w[k] = l;
        mx = fmaxf(mx, l);
    }
    // block reductions: within each warp by shuffles, then across the warps through s_red
#pragma unroll
    for (int off = 16; off > 0; off >>= 1)
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, off));
    if (lane == 0)
        s_red[wid] = mx;
    __syncthreads();
    mx = s_red[0];
#pragma unroll
    for (int w = 1; w < kWarps; ++w)
        mx = fmaxf(mx, s_red[w]);
    float tot = 0.f;
    for (int k = tid; k < np; k += kCombineThreads) {
        const float w = fast_exp2(s_w[k] - mx);
        s_w[k] = w;
        tot += w;
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1)
        tot += __shfl_xor_sync(0xffffffffu, tot, off);
    __syncthreads();   // every warp has read s_red's maxima; s_w holds the weights
    if (lane == 0)
        s_red[wid] = tot;
    __syncthreads();
    tot = 0.f;
#pragma unroll
    for (int w = 0; w < kWarps; ++w)
        tot += s_red[w];
    const float inv = fast_rcp(tot);
    float acc = 0.f;
#pragma unroll
    for (int m = 0; m < 16; ++m) {
        const int k = grp + m * kGroups;
        if (k < np)
            acc += s_w[k] * v[m];
    }
    for (int k0 = grp + 16 * kGroups; k0 < np; k0 += kGroups * 16) {
#pragma unroll
        for (int m = 0; m < 16; ++m) {
            const int k = k0 + m * kGroups;
            v[m] = k < np ? __ldcg(src + static_cast<size_t>(k) * G * D) : 0.f;
        }
#pragma unroll
        for (int m = 0; m < 16; ++m) {
            const int k = k0 + m * kGroups;
            if (k < np)
                acc += s_w[k] * v[m];
        }
    }
    __syncthreads();   // every thread has read the warps' sums
    s_red[tid] = acc;
    __syncthreads();
    if (grp == 0) {
        float sum = 0.f;
#pragma unroll
        for (int q = 0; q < kGroups; ++q)
            sum += s_red[q * D + e];
        out[(static_cast<size_t>(beta) * p.h + static_cast<size_t>(j) * G + row) * D + e] =
            __float2bfloat16_rn(sum * inv);
    }
}

// ------------------------------------------------------------------------------------------------
// append kernel: one thread per 16-byte vector of the new token's K/V rows
// ------------------------------------------------------------------------------------------------

__global__ void append_kernel(const __grid_constant__ AppendParams p)
{
    grid_dependency_wait();
    grid_dependents_launch();
    const int vecs = p.d / 8;
    const long long total = 2LL * p.b * p.g * vecs;
    const long long idx = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (idx >= total)
        return;
    const int v = static_cast<int>(idx % vecs);
    long long row = idx / vecs;   // (kv, beta, j)
    const int j = static_cast<int>(row % p.g);
    row /= p.g;
    const int beta = static_cast<int>(row % p.b);
    const int kv = static_cast<int>(row / p.b);
    const int pos = p.seq_len[beta] - 1;
    const uint4 *src = reinterpret_cast<const uint4 *>(kv ? p.V : p.K) +
                       (static_cast<size_t>(beta) * p.g + j) * vecs + v;
    uint4 *dst = reinterpret_cast<uint4 *>(p.cache) +
                 ((((static_cast<size_t>(p.slot) * 2 + kv) * p.b + beta) * p.g + j) *
                      static_cast<size_t>(p.max_seq) + pos) * vecs + v;
    *dst = *src;
}

template <int D, int T, int STAGES, int NCW, bool kT>
constexpr DecodeVariant make_variant()
{
    using PL = Plan<D, T, STAGES, NCW, kT>;
    return DecodeVariant{D, T, STAGES, PL::kThreads, static_cast<size_t>(PL::kAlloc),
                         PL::kClusterInRaw ? 0 : static_cast<size_t>(PL::kResBytes),
                         reinterpret_cast<const void *>(&decode_kernel<D, T, STAGES, NCW, kT>), 0,
                         static_cast<size_t>((PL::kMaxRawBufs - 1) * PL::kRawBytes), PL::kMinBlocks};
}

// (head_dim, positions per tile, ring stages, consumer warps) for groups of more than 8 heads, and
// for those of at most 8; the first match of a (head_dim, tile) pair is used.  <64, 128, 2, 4> and
// <64, 64, 4, 4> fit twice on an SM (87 to 112 KB, at most 168 registers).
const DecodeVariant kVariants[2][5] = {
    {make_variant<64, 128, 2, 4, false>(), make_variant<64, 256, 3, 4, false>(),
     make_variant<64, 64, 4, 4, false>(), make_variant<128, 64, 4, 4, false>(),
     make_variant<128, 128, 2, 4, false>()},
    {make_variant<64, 128, 2, 4, true>(), make_variant<64, 256, 3, 4, true>(),
     make_variant<64, 64, 4, 4, true>(), make_variant<128, 64, 5, 4, true>(),
     make_variant<128, 128, 2, 4, true>()},
};

}  // namespace

const DecodeVariant *find_decode_variant(int head_dim, int tile_tokens, int tc, int group)
{
    if (tc) {
        for (int i = 0; i < kNumTcVariants; ++i)
            if (kTcVariants[i].head_dim == head_dim && kTcVariants[i].tile_tokens == tile_tokens)
                return &kTcVariants[i];
        return nullptr;
    }
    for (const DecodeVariant &v : kVariants[group <= 8 ? 1 : 0])
        if (v.head_dim == head_dim && v.tile_tokens == tile_tokens)
            return &v;
    return nullptr;
}

cudaError_t prepare_decode_variant(const DecodeVariant &v, size_t max_smem)
{
    size_t tail = table_bytes(MLKV_MAX_BATCH);
    if (3 * v.res_bytes > tail)
        tail = 3 * v.res_bytes;   // cluster mode, k = 4
    size_t want = v.smem_bytes + tail;
    if (want > max_smem)
        want = max_smem;
    if (v.smem_bytes > want)
        return cudaErrorInvalidValue;
    return cudaFuncSetAttribute(v.fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                static_cast<int>(want));
}

cudaError_t launch_decode(const DecodeVariant &v, int grid, size_t smem, cudaStream_t stream,
                          const CUtensorMap *tmap, const CUtensorMap *tmap_rows,
                          const DecodeParams &p, const cudaAccessPolicyWindow *window, bool pdl)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>(grid));
    cfg.blockDim = dim3(static_cast<unsigned>(v.threads));
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[3];
    int na = 0;
    if (pdl) {
        attr[na].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[na].val.programmaticStreamSerializationAllowed = 1;
        ++na;
    }
    if (p.cluster_k > 1) {
        attr[na].id = cudaLaunchAttributeClusterDimension;
        attr[na].val.clusterDim.x = static_cast<unsigned>(p.cluster_k);
        attr[na].val.clusterDim.y = 1;
        attr[na].val.clusterDim.z = 1;
        ++na;
    }
    if (window != nullptr) {
        attr[na].id = cudaLaunchAttributeAccessPolicyWindow;
        attr[na].val.accessPolicyWindow = *window;
        ++na;
    }
    cfg.attrs = attr;
    cfg.numAttrs = na;
    void *args[] = {const_cast<CUtensorMap *>(tmap), const_cast<CUtensorMap *>(tmap_rows),
                    const_cast<DecodeParams *>(&p)};
    return cudaLaunchKernelExC(&cfg, v.fn, args);
}

int max_pieces_per_segment(const DecodeParams &p, int T, int grid)
{
    const long long N = p.num_tiles;
    if (grid <= 1 || N <= 0)
        return 1;
    if (p.uniform_len > 0) {
        // Every CTA holds at least floor(N/grid) tiles, so a segment of nt tiles meets at most
        // ceil((nt - 1) / floor(N/grid)) + 1 of them.
        const long long nt = (p.uniform_len + T - 1) / T;
        const long long per = N / grid;
        if (per <= 0)
            return grid;
        return static_cast<int>((nt - 1 + per - 1) / per + 1);
    }
    auto cta_of = [&](long long tile) { return static_cast<int>(((tile + 1) * grid - 1) / N); };
    int worst = 1;
    for (int beta = 0; beta < p.b; ++beta) {
        const int nt = (p.seq_len[beta] + T - 1) / T;
        for (int j = 0; j < p.g; ++j) {
            const long long first =
                static_cast<long long>(p.tile_start[beta]) + static_cast<long long>(j) * nt;
            const int np = cta_of(first + nt - 1) - cta_of(first) + 1;
            worst = np > worst ? np : worst;
        }
    }
    return worst;
}

cudaError_t launch_combine(const DecodeParams &p, int head_dim, cudaStream_t stream, bool pdl)
{
    cudaLaunchConfig_t cfg = {};
    const int segs = p.b * p.g * (p.ml_layers > 0 ? p.ml_layers : 1);
    cfg.gridDim = dim3(static_cast<unsigned>(segs), static_cast<unsigned>(p.G));
    cfg.blockDim = dim3(kCombineThreads);
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = pdl ? 1 : 0;
    void *args[] = {const_cast<DecodeParams *>(&p)};
    const void *fn = head_dim == 64 ? reinterpret_cast<const void *>(&combine_kernel<64>)
                                    : reinterpret_cast<const void *>(&combine_kernel<128>);
    return cudaLaunchKernelExC(&cfg, fn, args);
}

cudaError_t max_active_clusters(const DecodeVariant &v, int k, int *out)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>(k));
    cfg.blockDim = dim3(static_cast<unsigned>(v.threads));
    cfg.dynamicSmemBytes = v.smem_bytes + (k - 1) * v.res_bytes;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = static_cast<unsigned>(k);
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaOccupancyMaxActiveClusters(out, v.fn, &cfg);
}

cudaError_t launch_append(const AppendParams &p, cudaStream_t stream)
{
    const long long total = 2LL * p.b * p.g * (p.d / 8);
    const int threads = 256;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>((total + threads - 1) / threads));
    cfg.blockDim = dim3(threads);
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    void *args[] = {const_cast<AppendParams *>(&p)};
    return cudaLaunchKernelExC(&cfg, reinterpret_cast<const void *>(&append_kernel), args);
}

}  // namespace mlkv
