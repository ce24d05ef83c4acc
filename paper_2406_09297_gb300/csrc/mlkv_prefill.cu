// MLKV prefill attention on the 5th-generation tensor cores (tcgen05, tensor memory) for GB300.
//
// Prefill runs a whole prompt through one layer at once: prompt position t of query head i
// attends to positions 0 .. t of KV head j(i) = i / G of the layer's owner slot (causal
// attention, Eqs. 2-3 with the MLKV maps of Eqs. 13-18).  An owner layer attends over the prompt's
// K/V where they are and stores them in its slot (prefix_copy_kernel, launched behind this kernel
// and running in its tail), or, when its outputs would overwrite them, stores them first and attends
// over the slot, as the block's other layers do.
//
// Persistent CTAs: the grid is at most one wave, and CTA c takes units c, 2P - 1 - c, 2P + c, ... of
// the longest-first list (P CTAs).  All roles run on over the units: while a unit's last tile is in
// its softmax and its output is stored, the next unit's queries and first K/V tiles arrive and its
// first S is computed.  With a CTA per unit, every unit paid ~7,500 cycles outside its key tiles
// (barriers, TMEM, tensor-map fetch, first loads, output); now ~3,000.
//
// Work unit, head_dim 128: two query tiles A and B of 128 prompt positions that read the
// same KV head, so that every K/V tile is loaded once for both.  With an even group size G they are
// two heads of one group at the same positions (identical causal triangles); otherwise they are the
// blocks 2p and 2p+1 of one head (B sees one tile more; a last block without a partner runs alone
// as B).  Prefill at head_dim 64: one query tile (as B) per CTA and two CTAs per SM, each with half
// the tensor memory, so that one CTA's output overlaps the other's key tiles (although every K/V
// tile is then fetched once per query tile).  Units that see the most keys run first.
//
// Fused decode (one new token per sequence, every layer of an owner block at once, Sec. 3): the
// query rows of a unit are the G heads of KV head j in each of the block's L layers, row = layer * G
// + head, layers [0, L1) in tile B and [L1, L) in tile A (L1 = 128 / G); a unit takes one chunk of
// the sequence's key tiles and reads each K/V tile once for all L * G rows.  At head_dim 64 with
// L * G <= 128 a one-tile form runs it: with at most one unit per SM the deep form (one CTA per SM,
// a 12-tile ring, key tiles alternating between two softmax warpgroups), else two CTAs per SM;
// otherwise the two-tile form.
//
// Per key tile t and query tile X (all MMAs tcgen05.mma kind::f16, bf16 in, fp32 accumulate):
//   S_X = Q_X K_t^T  M = 128 queries (A = Q_X, K-major, 128-byte swizzle as TMA wrote it),
//                    N = 128 keys (B = the K tile), K = head_dim; one query row per TMEM lane.
//   softmax          a warpgroup per query tile, one thread per row: the thread owns its row's
//                    128 scores, so the running maximum needs no exchange between threads; the
//                    tensor-memory load returns it with the scores (tcgen05.ld.red), so S's
//                    columns are free for the next S before the weights are formed.  The
//                    reference maximum is raised only when a score exceeds it by more than 2^8
//                    (then the thread rescales its O row in TMEM); p = 2^(s log2(e)/sqrt(d) - m)
//                    goes back to TMEM as bf16 pairs.
//   O_X += P_X V_t   A = P_X read from TMEM, B = the V tile read MN-major from shared memory,
//                    N = head_dim, K = 128 keys; O_X stays in TMEM for the whole unit.
// While one warpgroup turns S into P, the tensor core works on the other query tile.
//
// TMEM (512 columns, 256 with one query tile): S per tile (128 columns), O per tile (head_dim).
// For head_dim 64, P has columns of its own (so S of the next tile can be computed while P of this
// one is being written); for head_dim 128, P overwrites the first 64 columns of its S (tcgen05.mma
// of one thread execute in order, so S of the next tile is written after P V has read P), and the
// product of the first 64 keys starts while the softmax forms the weights of the last 64.
//
// What bounds it, per key tile and query tile of an SM: the tensor core (head_dim 64: 4 x 66 cycles
// of S and 8 x 34 of P V; head_dim 128: 16 x 66) and the softmax warps' issue slots (~690 cycles:
// 128 exponentials, and paired multiply-adds, sums and conversions that take two slots each).
// Measured on GB300, an owner layer and a later one of its block.  First the former form (a CTA per
// unit), then persistent CTAs with early S columns and elected issuing threads, then also with the
// owner's K/V read in place and the producer one thread:
//   8 x 2048 positions x 12 heads, head_dim 64    168.6   132.1   122.7 us
//   4 x 2048 x 32 heads, head_dim 128             313.8   240.6   215 us
//   32 prompts of 1 to 777 positions, head_dim 64 103.7    83.0    54.2 us
//
// The diagonal tile masks keys after the query; keys past the prompt's end only meet such masked
// scores, and their V rows are zeroed in shared memory so that 0 * V stays 0.
//
// Warp roles: 4 softmax warps per query tile (warps 0-3 tile A, 4-7 tile B; the one-tile CTA's
// warps 0-3 take its tile), then the TMA producer (query tiles, then K_0, V_0, K_1, V_1, ...
// through a ring), the MMA issuer (for head_dim 64 only of S, the next warp issuing the P V
// products), and last a warp that loads queries held in host memory (else idle).  Registers: the
// two-tile block launches with 168 a thread and its last warpgroup gives registers back (72 or 88)
// to the softmax warpgroups (216 or 208, head_dim 64 or 128): 128 * low + 256 * high <= 384 * 168;
// the one-tile block launches with 128 (two blocks per SM) and splits 40 / 216: 128 * 40 +
// 128 * 216 = 256 * 128.
// Every wait is bounded; on expiry the kernel records an error bit, stops, lets its copies and MMAs
// land and frees its TMEM.
#include <type_traits>

#include "mlkv_device.cuh"
#include "mlkv_tcgen05.cuh"

namespace mlkv {
namespace {

// Forms of the CTA (kForm):
//   kTwoTiles  two query tiles share every K/V tile, one CTA per SM (head_dim 128; the fused
//              decode of blocks whose rows exceed one tile);
//   kOneTile   one query tile per CTA and two CTAs per SM (prefill at head_dim 64; the fused
//              decode with more units than SMs): each CTA holds half the tensor memory and a third
//              of the registers of the two-tile form, and two independent CTAs hide each other's
//              start, first loads and output;
//   kOneDeep   one query tile, one CTA per SM (the fused decode with at most one unit per SM, its
//              K/V tiles streamed from HBM): a ring of 12 tiles keeps ~6 K/V pairs in flight, and
//              the key tiles alternate between two softmax warpgroups on the same 128 query rows,
//              each with its own S, P and O columns and its own running maximum and sum, merged
//              per row at the end -- two key tiles' softmax chains run at once, and S of the next
//              tile is computed while this one's softmax runs.
constexpr int kTwoTiles = 0, kOneTile = 1, kOneDeep = 2;

template <int D, int kForm>
struct PrefillPlan {
    static constexpr bool kOne = kForm != kTwoTiles;
    static constexpr int kTiles = kOne ? 1 : 2;              // query tiles per CTA
    static constexpr int kSBuf = kForm == kOneDeep ? 2 : 1;  // S, P and O buffers per query tile
    static constexpr int kSoftWarps = 4 * kTiles * kSBuf;    // a warpgroup per tile or buffer
    static constexpr int kThreads = (kSoftWarps + 4) * 32;
    static constexpr int kMinBlocks = kForm == kOneTile ? 2 : 1;
    // registers at launch, then the other warps' share and the softmax warps' (setmaxnreg)
    static constexpr int kRegsLaunch = kForm == kOneTile ? 128 : 168;
    static constexpr int kRegsLow = kForm == kOneTile ? 40 : (D == 64 ? 72 : 88);
    static constexpr int kRegsHigh = kForm == kOneTile ? 216 : (D == 64 ? 216 : 208);
    static constexpr int kProducer = kSoftWarps, kMma = kSoftWarps + 1;
    static constexpr int kSub = D / 64;                      // 64-channel blocks of a row
    static constexpr int kTileBytes = 128 * D * 2;           // 128 rows of Q, K or V
    // K_t and V_t alternate in the ring
    static constexpr int kRingTiles = kForm == kOneDeep ? 12 : kOne ? 5 : (D == 64 ? 8 : 4);
    // Query tiles: two sets where shared memory allows it, so that a unit's queries arrive while
    // the unit before it still runs.
    static constexpr int kQBufs = D == 64 && kForm != kOneDeep ? 2 : 1;
    static constexpr int kQ = 0;                             // [kQBufs][kTiles] query tiles
    static constexpr int kRing = kQ + kQBufs * kTiles * kTileBytes;
    // Outputs are staged for coalesced stores in the unit's own query tile (head_dim 64), else in
    // 4 KB per softmax warp.
    static constexpr bool kStageInQ = D == 64;
    static constexpr int kStage = kRing + kRingTiles * kTileBytes;
    static constexpr int kFlags = kStage + (kStageInQ ? 0 : kSoftWarps * 4096);
                                                             // int [4], TMEM base at +16
    // u64 barriers: q[2], q_free[2], full[R], empty[R], s_ready[2], s_free[2], p_half[2],
    // p_ready[2], pv_done[2], fin[2] (s_ready and s_free per query tile, or per S buffer in the
    // deep form)
    static constexpr int kBars = kFlags + 32;
    static constexpr int kNumBars = 4 + 2 * kRingTiles + 10 + 2;
    // the warpgroups' running maxima and sums per row, for the merge (two buffers)
    static constexpr int kML = kBars + kNumBars * 8;
    static constexpr int kBytes = kML + (kSBuf == 2 ? 2 * 128 * 8 : 0);
    static constexpr int kAlloc = kBytes;
    static_assert(kMinBlocks * (kAlloc + 1024) <= 228 * 1024, "shared memory of the resident CTAs");
    static constexpr int kTmemCols = kForm == kOneTile ? 256 : 512;
    static constexpr bool kPSep = D == 64;                   // P in columns of its own
    static constexpr int kColS = 0;                          // + 128 per query tile or buffer
    static constexpr int kColO = 128 * kTiles * kSBuf;       // + D per query tile or buffer
    static constexpr int kColP = kColO + D * kTiles * kSBuf; // + 64 per tile or buffer (kPSep)
    static_assert(D == 64 || D == 128, "head_dim 64 or 128");
    static_assert(!kOne || D == 64, "one query tile per CTA only at head_dim 64");
    static_assert(kRing % 1024 == 0 && kTileBytes % 1024 == 0, "swizzled tiles 1024-aligned");
    static_assert((kPSep ? kColP + 64 * kTiles * kSBuf : kColO + D * kTiles) <= kTmemCols,
                  "TMEM columns overlap");
    static_assert(128 * kRegsLow + 32 * kSoftWarps * kRegsHigh <= kThreads * kRegsLaunch,
                  "register split");
    static_assert(kMinBlocks * kThreads * kRegsLaunch <= 65536, "registers of the resident CTAs");
    static_assert(kSBuf == 1 || (kTiles == 1 && kPSep), "two buffers: one tile, P apart");
};

template <int N>
__device__ __forceinline__ void setmaxnreg_inc()
{
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(N));
}

template <int N>
__device__ __forceinline__ void setmaxnreg_dec()
{
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(N));
}

__device__ __forceinline__ float max3f(float a, float b, float c)
{
    float d;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}

// A work unit as its CTA's warps see it (see PrefillParams::units).
struct Unit {
    int beta, S;          // sequence; its prompt length, or (fused decode) its length
    int chunk, blk;       // fused decode: context chunk and owner block (both 0 for prefill)
    int kt0;              // first key tile (128 positions) of the unit
    int n_a, n_b;         // key tiles of query tiles A (0: no tile A) and B, n_a <= n_b
    int qb_b;             // prefill: tile B's query block
    int head_a, head_b, j;
    int zk, zv;           // rows of the K and V tensor maps: (slot, sequence, KV head)
    bool has_end;         // the unit holds the sequence's last key tile
};

template <bool kFused, int kTiles>
__device__ __forceinline__ Unit unit_of(const PrefillParams &p, int i)
{
    Unit x;
    const uint32_t u = p.units[i];
    x.beta = static_cast<int>(u & 0x3FFu);
    const int sel = static_cast<int>(u >> 24);
    x.S = p.prompt_len[x.beta];
    if (kFused) {
        // every query row sees positions [0, S); the unit takes key tiles [kt0, kt0 + n_b)
        const int n_kt = (x.S + 127) / 128;
        x.chunk = static_cast<int>((u >> 10) & 0xFFu);
        x.blk = static_cast<int>((u >> 18) & 0x3Fu);
        x.kt0 = x.chunk * p.fused_kc;
        const int kt1 = min(x.kt0 + p.fused_kc, n_kt);
        x.has_end = kt1 == n_kt;
        x.n_b = kt1 - x.kt0;
        x.n_a = kTiles == 2 && p.fused_L > p.fused_L1 ? x.n_b : 0;
        x.qb_b = 0;
        x.head_a = x.head_b = x.j = sel;
    } else {
        x.chunk = x.blk = x.kt0 = 0;
        x.has_end = true;
        x.qb_b = static_cast<int>((u >> 10) & 0x3FFFu);
        x.n_b = x.qb_b + 1;
        x.n_a = kTiles == 1 ? 0 : p.head_pairs ? x.n_b : ((x.qb_b & 1) ? x.qb_b : 0);
        x.head_a = p.head_pairs ? 2 * sel : sel;
        x.head_b = p.head_pairs ? 2 * sel + 1 : sel;
        x.j = x.head_b / p.G;   // Eq. 15
    }
    if (!kFused && p.kv_direct) {   // the prompt's own tensors, [b][g][s_max][D] each
        x.zk = x.zv = x.beta * p.g + x.j;
    } else {
        x.zk = (((p.slot + x.blk) * 2 + 0) * p.b + x.beta) * p.g + x.j;
        x.zv = x.zk + p.b * p.g;
    }
    return x;
}

// The CTA's k-th unit, or -1 past its last: a snake deal of the units (longest first) to the
// persistent CTAs, which evens out their key tiles.
__device__ __forceinline__ int unit_index(const PrefillParams &p, int k)
{
    const int P = static_cast<int>(gridDim.x), c = static_cast<int>(blockIdx.x);
    const int i = k * P + ((k & 1) ? P - 1 - c : c);
    return i < p.n_units ? i : -1;
}

template <int D, bool kFused, int kForm>
__global__ void __launch_bounds__(PrefillPlan<D, kForm>::kThreads,
                                  PrefillPlan<D, kForm>::kMinBlocks)
    prefill_kernel(const __grid_constant__ CUtensorMap tmap_q,
                   const __grid_constant__ CUtensorMap tmap_k,
                   const __grid_constant__ CUtensorMap tmap_v,
                   const __grid_constant__ PrefillParams p)
{
    using PL = PrefillPlan<D, kForm>;
    constexpr bool kSplit = PL::kSBuf == 2;   // key tiles alternate between two warpgroups
    constexpr int NQ = PL::kQBufs;
    constexpr int R = PL::kRingTiles;
    // Query tile g's shared-memory slot and tensor-memory columns (the only tile of a one-tile CTA
    // is tile B, in slot 0).
    auto slot_of = [](int g) { return PL::kTiles == 1 ? 0 : g; };
    extern __shared__ __align__(1024) uint8_t smem[];   // swizzled tiles: 1024-byte aligned
    const uint32_t sbase = smem_addr(smem);
    const uint32_t bar_q = sbase + PL::kBars;             // [NQ] query tiles loaded
    const uint32_t bar_q_free = bar_q + 8 * 2;            // [NQ] query tiles read for the last time
    const uint32_t bar_full = bar_q_free + 8 * 2;
    const uint32_t bar_empty = bar_full + 8 * R;
    const uint32_t bar_s_ready = bar_empty + 8 * R;       // [2] per query tile or S buffer
    const uint32_t bar_s_free = bar_s_ready + 16;
    const uint32_t bar_p_half = bar_s_free + 16;          // P of the tile's first 64 keys (P over S)
    const uint32_t bar_p_ready = bar_p_half + 16;
    const uint32_t bar_pv_done = bar_p_ready + 16;
    const uint32_t bar_fin = bar_pv_done + 16;            // [2]: one per issuing thread
    volatile int *flags = reinterpret_cast<volatile int *>(smem + PL::kFlags);

    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    if ((sbase & 1023u) != 0) {   // the swizzled tiles need it; never seen
        if (threadIdx.x == 0)
            atomicOr(p.err, kErrDrain);
        return;
    }
    if (threadIdx.x == 0) {
        for (int q = 0; q < NQ; ++q) {
            // the query tiles' barrier: the producer's tensor-map copy, or the loads from host
            // memory by the last warp (deep form: by every softmax warp); freed by the unit's last
            // S and, where the outputs are staged in the query tiles, by the softmax warps
            mbar_init(bar_q + 8 * q,
                      kSplit && kFused && p.q_host != nullptr ? PL::kSoftWarps : 1);
            mbar_init(bar_q_free + 8 * q, 1 + (PL::kStageInQ ? PL::kSoftWarps : 0));
        }
        for (int s = 0; s < R; ++s) {
            mbar_init(bar_full + 8 * s, 1);
            mbar_init(bar_empty + 8 * s, 1);
        }
        for (int g = 0; g < 2; ++g) {
            mbar_init(bar_s_ready + 8 * g, 1);
            mbar_init(bar_s_free + 8 * g, 4);
            mbar_init(bar_p_half + 8 * g, 4);
            mbar_init(bar_p_ready + 8 * g, 4);
            mbar_init(bar_pv_done + 8 * g, 1);
        }
        mbar_init(bar_fin, 1);
        mbar_init(bar_fin + 8, 1);
        flags[0] = 0;
        fence_barrier_init();
    }
    if (threadIdx.x == PL::kProducer * 32) {
        prefetch_tensormap(&tmap_q);
        prefetch_tensormap(&tmap_k);
        prefetch_tensormap(&tmap_v);
    }
    if (warp == PL::kMma) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         sbase + PL::kFlags + 16),
                     "n"(PL::kTmemCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (kFused && warp < 4 * PL::kTiles) {   // one warpgroup per query tile
        // The tiles' rows past the loaded ones (the TMA box, G x min(L1, L) rows) are never
        // written; zero them so that their (discarded) scores stay finite.
        const int grp = PL::kTiles == 1 ? 1 : warp >> 2, r = threadIdx.x & 127;
        const int box_rows = (p.fused_L < p.fused_L1 ? p.fused_L : p.fused_L1) * p.G;
        // rows the load writes: the box (tensor map), or tile A's own rows (read from host)
        const int keep = (p.q_host != nullptr && grp == 0) ? (p.fused_L - p.fused_L1) * p.G
                                                           : box_rows;
        if (r >= keep) {
            for (int q = 0; q < NQ; ++q) {
                uint8_t *qrow = smem + PL::kQ + (q * PL::kTiles + slot_of(grp)) * PL::kTileBytes;
#pragma unroll
                for (int c = 0; c < 8 * PL::kSub; ++c)
                    *reinterpret_cast<uint4 *>(qrow + (c >> 3) * 16384 + r * 128 +
                                               (((c & 7) ^ (r & 7)) << 4)) = make_uint4(0, 0, 0, 0);
            }
            fence_proxy_async_smem();
        }
    }
    tmem_fence_before();
    __syncthreads();
    tmem_fence_after();
    const uint32_t tmem = *reinterpret_cast<volatile uint32_t *>(smem + PL::kFlags + 16);
    // The owner's K/V may have just been stored by the previous kernel of the stream.  In the
    // fused step that kernel stores only position L - 1 of each slot and was itself launched after
    // every earlier kernel had finished (it triggers this launch only after its own dependency
    // wait): the queries and every tile but the one holding position L - 1 are loaded at once, the
    // producer waits before that tile, and the output waits before its stores.
    const bool early = kFused && p.fused_early;
    const bool q_early = kFused && p.fused_early == 1;   // the queries before the wait too
    if (!early)
        grid_dependency_wait();
    grid_dependents_launch();
    // A unit's query rows from page-locked host memory through its device-mapped address (16 bytes a
    // load, FLY of them in flight per thread of N), written into the query tiles the way the tensor
    // map would have (128-byte swizzle); rows past them stay zero.
    auto load_q_host = [&](const Unit &x, int qb, int t, auto n_, auto fly_) {
        constexpr int N = decltype(n_)::value, FLY = decltype(fly_)::value;
        constexpr int kC = D / 8;   // 16-byte chunks of a row
        const int rows_b = (p.fused_L < p.fused_L1 ? p.fused_L : p.fused_L1) * p.G;
        uint8_t *dst = smem + PL::kQ + qb * PL::kTiles * PL::kTileBytes;
        const int total = (rows_b + (x.n_a > 0 ? (p.fused_L - p.fused_L1) * p.G : 0)) * kC;
        for (int k0 = t; k0 < total; k0 += N * FLY) {
            uint4 v[FLY];
#pragma unroll
            for (int u = 0; u < FLY; ++u) {
                const int k = k0 + u * N;
                if (k < total) {
                    const int rr = k / kC, c = k - rr * kC;
                    const int rw = rr < rows_b ? rr : rr - rows_b;
                    const int lay =
                        x.blk * p.fused_L + (rr < rows_b ? 0 : p.fused_L1) + rw / p.G;
                    v[u] = *reinterpret_cast<const uint4 *>(
                        p.q_host + ((static_cast<size_t>(lay) * p.b + x.beta) * p.h + x.j * p.G +
                                    rw % p.G) * D + c * 8);
                }
            }
#pragma unroll
            for (int u = 0; u < FLY; ++u) {
                const int k = k0 + u * N;
                if (k < total) {
                    const int rr = k / kC, c = k - rr * kC;
                    const int rw = rr < rows_b ? rr : rr - rows_b;
                    *reinterpret_cast<uint4 *>(dst + slot_of(rr < rows_b ? 1 : 0) * PL::kTileBytes +
                                               (c >> 3) * 16384 + rw * 128 +
                                               (((c & 7) ^ (rw & 7)) << 4)) = v[u];
                }
            }
        }
    };
    if (warp == PL::kProducer) {
        // ------------------------------------ producer ------------------------------------------
        // One thread waits, announces the bytes and sends the copies.
        setmaxnreg_dec<PL::kRegsLow>();
        bool waited = !early;
        int idx = 0;   // ring tiles sent so far: K_0, V_0, K_1, V_1, ... over all units
        int uc = 0;    // units whose queries were sent
        // Ring tile k of unit x (K of key tile k / 2 if k is even, else V).
        auto send_kv = [&](const Unit &x, int k) {
            const int s = idx % R;
            if (idx >= R && !flags[0] &&
                !mbar_wait(bar_empty + 8 * s, ((idx / R) & 1) ^ 1)) {
                flags[0] = 1;
                atomicOr(p.err, kErrWaitEmpty);
            }
            if (flags[0])
                return false;
            if (!waited && x.has_end && (k >> 1) == x.n_b - 1) {
                grid_dependency_wait();   // the tile that holds the new row
                waited = true;
            }
            const uint32_t fb = bar_full + 8 * s;
            mbar_arrive_expect_tx(fb, PL::kTileBytes);
#pragma unroll
            for (int sub = 0; sub < PL::kSub; ++sub)
                tma_load_3d(sbase + PL::kRing + s * PL::kTileBytes + sub * 16384,
                            (k & 1) ? &tmap_v : &tmap_k, fb, sub * 64, ((k >> 1) + x.kt0) * 128,
                            (k & 1) ? x.zv : x.zk);
            ++idx;
            return true;
        };
        auto send_q = [&](const Unit &x) {
            const int qb = uc % NQ;
            if (kFused && p.q_host != nullptr) {
                ++uc;   // other warps read the queries from host memory (load_q_host)
                return true;
            }
            if (uc >= NQ && !flags[0] &&
                !mbar_wait(bar_q_free + 8 * qb, ((uc / NQ) & 1) ^ 1)) {
                flags[0] = 1;
                atomicOr(p.err, kErrWaitEmpty);
            }
            if (flags[0])
                return false;
            const uint32_t qbar = bar_q + 8 * qb;
            const uint32_t dst = sbase + PL::kQ + qb * PL::kTiles * PL::kTileBytes;
            const int n_tiles = x.n_a > 0 ? 2 : 1;
            // fused: Q [layers][b][h][D] as (channel, head in group, group, sequence, layer); a
            // box of min(L1, L) layers x G heads = the tile's rows, layer-major (row = layer*G + i),
            // from the block's first layer (tile B) and its layer L1 (tile A)
            const int box_rows =
                kFused ? (p.fused_L < p.fused_L1 ? p.fused_L : p.fused_L1) * p.G : 128;
            mbar_arrive_expect_tx(qbar, n_tiles * PL::kSub * box_rows * 128);
            for (int g = 1; g >= 2 - n_tiles; --g)
#pragma unroll
                for (int sub = 0; sub < PL::kSub; ++sub) {
                    const uint32_t d = dst + slot_of(g) * PL::kTileBytes + sub * 16384;
                    if (kFused)
                        tma_load_5d(d, &tmap_q, qbar, sub * 64, 0, x.j, x.beta,
                                    x.blk * p.fused_L + (g ? 0 : p.fused_L1));
                    else
                        tma_load_4d(d, &tmap_q, qbar, sub * 64, g ? x.head_b : x.head_a,
                                    (g ? x.qb_b : x.n_a - 1) * 128, x.beta);
                }
            ++uc;
            return true;
        };
        if (lane == 0) {
            bool ok = true;
            for (int n = 0; ok; ++n) {
                const int i = unit_index(p, n);
                if (i < 0)
                    break;
                const Unit x = unit_of<kFused, PL::kTiles>(p, i);
                const int n_idx = 2 * x.n_b;
                int k = 0;
                if (n == 0 && early && !q_early) {
                    // mode 2: the cache tiles that hold no new row first, as far as the ring goes
                    const int n_pre = n_idx < R ? n_idx : R;
                    while (ok && k < n_pre && !(x.has_end && (k >> 1) == x.n_b - 1))
                        ok = send_kv(x, k++);
                    grid_dependency_wait();   // the step's inputs are in place
                    waited = true;
                }
                // a later unit's first key tile can go before its queries' slot is free
                if (n > 0 && NQ == 1)
                    ok = ok && send_kv(x, k++);
                ok = ok && send_q(x);
                while (ok && k < n_idx)
                    ok = send_kv(x, k++);
                if (kSplit)
                    break;   // one unit per CTA
            }
            // No copy may still be in flight when the CTA exits.
            if (!(kFused && p.q_host != nullptr))
                for (int k = uc > NQ ? uc - NQ : 0; k < uc; ++k)
                    if (!mbar_wait(bar_q + 8 * (k % NQ), (k / NQ) & 1))
                        atomicOr(p.err, kErrDrain);
            for (int k = idx > R ? idx - R : 0; k < idx; ++k)
                if (!mbar_wait(bar_full + 8 * (k % R), (k / R) & 1))
                    atomicOr(p.err, kErrDrain);
        }
        __syncwarp();
    } else if (warp == PL::kMma || (PL::kPSep && warp == PL::kMma + 1)) {
        // ------------------------------------ MMA issuers ---------------------------------------
        // With P in columns of its own (head_dim 64) warp kMma issues every S = Q K^T and warp
        // kMma + 1 every O += P V: the two never touch the same tensor-memory columns, each waits
        // only for what its own products need, and the tensor core gets both streams.  (One thread
        // issuing both spent about a third of each key tile on barrier checks while the tensor core
        // ran dry.)  With P over S (head_dim 128) one thread issues both, in order.
        setmaxnreg_dec<PL::kRegsLow>();
        const bool do_s = warp == PL::kMma;
        const uint32_t my_fin = bar_fin + (warp == PL::kMma ? 0 : 8);
        if (elect_one()) {
            constexpr uint32_t kIdS = umma_idesc(128, 128, 0, 0);
            constexpr uint32_t kIdPV = umma_idesc(128, D, 0, 1);
            constexpr uint32_t kSlot = PL::kTileBytes >> 4;   // one ring slot in descriptor units
            // Descriptors of query tile A and of ring slot 0.  A tile, a slot, a K step or a
            // 64-channel block only moves the start-address field (shared addresses < 256 KB), so
            // each MMA's descriptors are one add away; the tensor core queues little, and any
            // latency between two MMAs of this thread leaves it idle.
            const uint64_t dq0 = umma_desc(sbase + PL::kQ, 16, 1024, kLayoutSw128);
            const uint64_t dk = umma_desc(sbase + PL::kRing, 16, 1024, kLayoutSw128);
            const uint64_t dv = umma_desc(sbase + PL::kRing, 16384, 1024, kLayoutSw128);
            bool ok = true;
            auto wait = [&](uint32_t bar, int parity) {
                const uint32_t par = static_cast<uint32_t>(parity) & 1u;
                if (ok && !mbar_test_wait(bar, par) && !mbar_wait(bar, par))
                    ok = false;
                return ok;
            };
            // Each ring tile is checked once: the K tile serves both query tiles' S, the V tile
            // both P V (a check costs ~150 cycles while the MMAs keep shared memory busy).
            int seen0 = -1, seen1 = -1;
            auto tile_full = [&](int idx) {
                if (idx == seen0 || idx == seen1)
                    return ok;
                if (wait(bar_full + 8 * (idx % R), idx / R)) {
                    seen1 = seen0;
                    seen0 = idx;
                }
                return ok;
            };
            // S of key tile kt (counted over the CTA's units) into buffer sb
            auto issue_s = [&](int g, int kt, int sb, uint64_t dq) {
                const uint64_t qa = dq + slot_of(g) * kSlot;
                const uint64_t kb = dk + ((2 * kt) % R) * kSlot;
#pragma unroll
                for (int k = 0; k < D / 16; ++k) {
                    const uint32_t off = (k >> 2) * 1024 + (k & 3) * 2;   // 16384 B, 32 B
                    umma_f16(tmem + PL::kColS + 128 * (kSplit ? sb : slot_of(g)), qa + off,
                             kb + off, kIdS, k > 0 ? 1 : 0);
                }
                umma_commit(bar_s_ready + 8 * sb);
            };
            // keys [64 h0, 64 h1) of O += P V of key tile kt into buffer pb
            auto issue_pv = [&](int kt, int pb, bool first, int h0, int h1) {
                const uint64_t vb = dv + ((2 * kt + 1) % R) * kSlot;
                const int ob = kSplit ? pb : slot_of(pb);   // P and O columns
                const uint32_t pc =
                    tmem + (PL::kPSep ? PL::kColP + 64 * ob : PL::kColS + 128 * ob);
#pragma unroll
                for (int k = 0; k < 8; ++k)   // 16 keys = 2048 B of V, 8 TMEM columns of P
                    if (k >= 4 * h0 && k < 4 * h1)
                        umma_f16_ts(tmem + PL::kColO + D * ob, pc + 8 * k, vb + k * 128, kIdPV,
                                    (!first || k > 0) ? 1 : 0);
            };
            // Ring slots are released by tile B's softmax warps (they see every MMA that read them
            // complete), not by commits: a commit costs the tensor pipe about as much as a short MMA.
            int kb = 0;             // key tiles of the units before
            int used[2] = {0, 0};   // products issued so far per S (or P) buffer
            for (int n = 0; ok; ++n) {
                const int i = unit_index(p, n);
                if (i < 0)
                    break;
                const Unit x = unit_of<kFused, PL::kTiles>(p, i);
                const int qb = n % NQ;
                const uint64_t dq = dq0 + static_cast<uint32_t>(qb * PL::kTiles) * kSlot;
                if (PL::kPSep && do_s) {
                    // S(t) once its columns are free, i.e. the previous scores of the buffer have
                    // been read (right after they arrived).
                    if (!wait(bar_q + 8 * qb, n / NQ))
                        break;
                    for (int t = 0; ok && t < x.n_b; ++t) {
#pragma unroll
                        for (int g = 2 - PL::kTiles; g < 2; ++g) {
                            if (!ok || t >= (g ? x.n_b : x.n_a))
                                continue;
                            const int sb = kSplit ? (t & 1) : g;
                            if (used[sb] > 0 && !wait(bar_s_free + 8 * sb, used[sb] - 1))
                                break;
                            if (!tile_full(2 * (kb + t)))
                                break;
                            tmem_fence_after();
                            issue_s(g, kb + t, sb, dq);
                            ++used[sb];
                        }
                    }
                    umma_commit(bar_q_free + 8 * qb);
                } else if (PL::kPSep) {
                    for (int t = 0; ok && t < x.n_b; ++t) {
#pragma unroll
                        for (int g = 2 - PL::kTiles; g < 2; ++g) {
                            if (!ok || t >= (g ? x.n_b : x.n_a))
                                continue;
                            const int pb = kSplit ? (t & 1) : g;
                            if (!tile_full(2 * (kb + t) + 1) ||
                                !wait(bar_p_ready + 8 * pb, used[pb]))
                                break;
                            tmem_fence_after();
                            issue_pv(kb + t, pb, kSplit ? t < 2 : t == 0, 0, 2);
                            umma_commit(bar_pv_done + 8 * pb);
                            ++used[pb];
                        }
                    }
                } else {
                    // P over S: the first S of the unit (the P V products that read these columns
                    // were issued before), then per key tile and query tile the P V product in two
                    // halves as the halves of P arrive, and the next S right behind it.
                    if (!wait(bar_q + 8 * qb, n / NQ) || !tile_full(2 * kb))
                        break;
                    tmem_fence_after();
                    if (x.n_a > 0)
                        issue_s(0, kb, 0, dq);
                    issue_s(1, kb, 1, dq);
                    if (x.n_b == 1)
                        umma_commit(bar_q_free + 8 * qb);
                    for (int t = 0; ok && t < x.n_b; ++t) {
#pragma unroll
                        for (int g = 0; g < 2; ++g) {
                            const int ng = g ? x.n_b : x.n_a;
                            if (!ok || t >= ng)
                                continue;
                            const bool next = t + 1 < ng;
                            if (!tile_full(2 * (kb + t) + 1) ||
                                (next && !tile_full(2 * (kb + t) + 2)) ||
                                !wait(bar_p_half + 8 * g, used[g]))
                                break;
                            tmem_fence_after();
                            issue_pv(kb + t, g, t == 0, 0, 1);
                            if (!wait(bar_p_ready + 8 * g, used[g]))
                                break;
                            tmem_fence_after();
                            issue_pv(kb + t, g, t == 0, 1, 2);
                            ++used[g];
                            // the next S's completion implies this product's
                            if (!next)
                                umma_commit(bar_pv_done + 8 * g);
                            else
                                issue_s(g, kb + t + 1, g, dq);
                            if (g == 1 && t + 2 == x.n_b)
                                umma_commit(bar_q_free + 8 * qb);   // that was the unit's last S
                        }
                    }
                }
                kb += x.n_b;
                if (kSplit)
                    break;   // one unit per CTA
            }
            if (!ok) {
                flags[0] = 1;
                atomicOr(p.err, kErrWaitFull);
            }
            umma_commit(my_fin);
            if (!mbar_wait(my_fin, 0))
                atomicOr(p.err, kErrDrain);
        }
        __syncwarp();
    } else if (warp < PL::kSoftWarps) {
        // ------------------------------------ softmax warpgroups --------------------------------
        setmaxnreg_inc<PL::kRegsHigh>();
        const int grp = PL::kTiles == 1 ? 1 : warp >> 2;   // 0: query tile A, 1: query tile B
        const int r = threadIdx.x & 127;            // query row of the tile = TMEM lane
        const uint32_t lane_off = static_cast<uint32_t>((warp & 3) * 32) << 16;
        const int sg = slot_of(grp);
        // the warpgroup's buffer: the tile's own, or (split keys) this warpgroup's tiles t = wg,
        // wg + 2, ... with S, P and O buffer wg
        const int wg = kSplit ? warp >> 2 : 0;
        const int bsel = kSplit ? wg : grp;
        const uint32_t col_s = tmem + lane_off + PL::kColS + 128 * (kSplit ? wg : sg);
        const uint32_t col_o = tmem + lane_off + PL::kColO + D * (kSplit ? wg : sg);
        const uint32_t col_p =
            tmem + lane_off +
            (PL::kPSep ? PL::kColP + 64 * (kSplit ? wg : sg) : PL::kColS + 128 * sg);
        const uint32_t s_ready = bar_s_ready + 8 * bsel, s_free = bar_s_free + 8 * bsel;
        const uint32_t p_half = bar_p_half + 8 * bsel, p_ready = bar_p_ready + 8 * bsel;
        const uint32_t pv_done = bar_pv_done + 8 * bsel;
        constexpr int kStep = kSplit ? 2 : 1;   // tiles between this warpgroup's
        // Tile B's first warp frees ring slots whose readers have all completed: K_t once S_B(t)
        // is done (S_A(t) was issued before it by the same thread); V_{t-1} once S_B(t) (P over
        // S: issued after P V_{t-1}) or P_B V_{t-1} (own P) is done.
        const bool releaser = grp == 1 && (warp & 3) == 0 && lane == 0;
        const float scale = p.scale_log2;
        const float NEG_INF = -__int_as_float(0x7f800000);
        auto wait = [&](uint32_t bar, int parity) {
            const uint32_t par = static_cast<uint32_t>(parity) & 1u;
            if (!mbar_test_wait(bar, par) && !flags[0] && !mbar_wait(bar, par)) {
                flags[0] = 1;
                atomicOr(p.err, kErrWaitFull);
            }
        };
        if (kFused && kSplit && p.q_host != nullptr) {
            // The CTA's only unit: nothing to compute before its queries, so every softmax warp
            // loads, one round trip over the link (by the last warp alone, two: 64 sequences of
            // 2,048 tokens end to end 34.5 us a step, now 32.9).
            load_q_host(unit_of<kFused, PL::kTiles>(p, unit_index(p, 0)), 0, threadIdx.x,
                        std::integral_constant<int, 32 * PL::kSoftWarps>{},
                        std::integral_constant<int, 4>{});
            fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0)
                mbar_arrive(bar_q);
        }
        int kb = 0;     // key tiles of the units before
        int used = 0;   // score tiles this warpgroup has taken
        int outs = 0;   // units it has finished (P over S: phases of pv_done)
        for (int n = 0;; ++n) {
            const int i = unit_index(p, n);
            if (i < 0 || (!kSplit && __any_sync(0xffffffffu, flags[0])))
                break;
            const Unit x = unit_of<kFused, PL::kTiles>(p, i);
            const int qb = n % NQ;
            const int n_g = grp ? x.n_b : x.n_a;
            const int q0 = (x.kt0 + n_g - 1) * 128;       // first position of the unit's last tile
            // The prompt's last block holds keys past its end; the first tile to reach it zeroes
            // them.
            const bool zero_v = n_g > 0 && (kFused ? x.has_end : n_g == (x.S + 127) / 128) &&
                                (grp == 0 || x.n_a != x.n_b);
            uint8_t *q_slot = smem + PL::kQ + (qb * PL::kTiles + sg) * PL::kTileBytes;
            float m_run = NEG_INF, l_run = 0.f;
            for (int t = wg; t < n_g; t += kStep, ++used) {
                wait(s_ready, used);
                if (releaser) {
                    mbar_arrive(bar_empty + 8 * ((2 * (kb + t)) % R));   // K_t
                    if (!PL::kPSep && t > 0)
                        mbar_arrive(bar_empty + 8 * ((2 * (kb + t) - 1) % R));   // V_{t-1}
                }
                const bool diag = t == n_g - 1 && x.has_end;
                // This tile's scores and the row's maximum, which the load returns with them.
                float sv[4][32], mx[4];
                uint32_t w[2][32];
                tmem_fence_after();
#pragma unroll
                for (int c = 0; c < 4; ++c)
                    tmem_ld32_max_nowait(col_s + c * 32, sv[c], mx[c]);
                tmem_wait_ld();
                asm volatile("" : "+f"(mx[0]), "+f"(mx[1]), "+f"(mx[2]), "+f"(mx[3]));
                if (PL::kPSep) {
                    // S's columns may take the next scores.
                    tmem_fence_before();
                    __syncwarp();
                    if (lane == 0)
                        mbar_arrive(s_free);
                }
                if (diag && zero_v && q0 + r >= x.S) {
                    // Key q0 + r lies past the prompt: its V row may hold anything; zero it.
                    const int idx = 2 * (kb + t) + 1;
                    wait(bar_full + 8 * (idx % R), idx / R);
                    uint8_t *vrow = smem + PL::kRing + (idx % R) * PL::kTileBytes;
#pragma unroll
                    for (int c = 0; c < 8 * PL::kSub; ++c)
                        *reinterpret_cast<uint4 *>(vrow + (c >> 3) * 16384 + r * 128 +
                                                   (((c & 7) ^ (r & 7)) << 4)) = make_uint4(0, 0, 0, 0);
                    fence_proxy_async_smem();
                }
                if (diag) {
                    // Keys [0, lim) of the tile are visible: up to the sequence's end (fused
                    // decode) or to the query's own position (causal mask); the maximum is
                    // taken again over those.
                    const int lim = kFused ? x.S - q0 : r + 1;
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        mx[c] = NEG_INF;
#pragma unroll
                        for (int k = 0; k < 32; ++k) {
                            if (c * 32 + k >= lim)
                                sv[c][k] = NEG_INF;
                            mx[c] = fmaxf(mx[c], sv[c][k]);
                        }
                    }
                }
                // The reference maximum is raised to the tile's when a score exceeds it by more
                // than 2^8 (the thread then rescales its O row in TMEM).
                const float m_tile = max3f(mx[0], mx[1], fmaxf(mx[2], mx[3])) * scale;
                const bool raise = (m_run == NEG_INF) || (m_tile > m_run + 8.f);
                if (__any_sync(0xffffffffu, raise)) {
                    const float m_new = raise ? fmaxf(m_run, m_tile) : m_run;
                    const float alpha = fast_exp2(m_run - m_new);   // 0 while nothing is summed
                    if (t > wg) {
                        // Rescale this row of O once the previous tile's product has landed.
                        if (PL::kPSep)
                            wait(pv_done, used - 1);
                        tmem_fence_after();
#pragma unroll
                        for (int c = 0; c < D / 32; ++c) {
                            float ov[32];
                            tmem_ld32_nowait(col_o + c * 32, ov);
                            tmem_wait_ld();
#pragma unroll
                            for (int k = 0; k < 32; ++k)
                                ov[k] *= alpha;
                            tmem_st32(col_o + c * 32, ov);
                        }
                    }
                    l_run *= alpha;
                    m_run = m_new;
                }
                // p = 2^(s log2(e)/sqrt(d) - m) as bf16 pairs, and the row's sum in fp32.
                const float2 sc2 = make_float2(scale, scale);
                const float m_use = m_run == NEG_INF ? 0.f : m_run;   // all masked so far: p = 0
                const float2 nm2 = make_float2(-m_use, -m_use);
                float2 acc[4];
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    acc[q] = make_float2(0.f, 0.f);
#pragma unroll
                for (int half = 0; half < 2; ++half) {
#pragma unroll
                    for (int e = 0; e < 32; ++e) {
                        const int c = half * 64 + 2 * e;   // keys c, c + 1
                        const float2 y = __ffma2_rn(
                            make_float2(sv[c >> 5][c & 31], sv[c >> 5][(c & 31) + 1]), sc2, nm2);
                        const float2 pr = make_float2(fast_exp2(y.x), fast_exp2(y.y));
                        acc[e & 3] = __fadd2_rn(acc[e & 3], pr);
                        w[half][e] = pack_bf16x2(pr.x, pr.y);
                    }
                    if (!PL::kPSep) {
                        tmem_st32_nowait(col_p + 32 * half, w[half]);
                        if (half == 0) {
                            // the first 64 keys' product may start
                            tmem_wait_st();
                            tmem_fence_before();
                            __syncwarp();
                            if (lane == 0)
                                mbar_arrive(p_half);
                        }
                    }
                }
                const float2 s01 = __fadd2_rn(acc[0], acc[1]), s23 = __fadd2_rn(acc[2], acc[3]);
                const float2 s4 = __fadd2_rn(s01, s23);
                // The P buffer of the previous tile must have been read by its P V; the weights
                // above were computed while that product ran.
                if (PL::kPSep && t > wg) {
                    wait(pv_done, used - 1);
                    if (releaser)   // V of this warpgroup's previous tile
                        mbar_arrive(bar_empty + 8 * ((2 * (kb + t - kStep) + 1) % R));
                }
                if (PL::kPSep) {
                    tmem_fence_after();
                    tmem_st32_nowait(col_p, w[0]);
                    tmem_st32_nowait(col_p + 32, w[1]);
                }
                l_run += s4.x + s4.y;
                tmem_wait_st();
                tmem_fence_before();
                __syncwarp();
                if (lane == 0)
                    mbar_arrive(p_ready);
            }
            // ---------------- the tile's output: o = O / l ----------------
            if (early)
                grid_dependency_wait();   // earlier kernels of the stream have finished with out
            // The unit's fields that only the output needs, read again: they need no registers
            // during the loop.
            int i_out = i;
            asm volatile("" : "+r"(i_out));
            const Unit y = unit_of<kFused, PL::kTiles>(p, i_out);
            // The unit's last product, and with it the last reader of its last V.
            const int n_mine = kSplit ? (n_g - wg + 1) / 2 : n_g;   // this warpgroup's tiles
            if (n_mine > 0) {
                wait(pv_done, PL::kPSep ? used - 1 : outs);
                ++outs;
                if (releaser)
                    mbar_arrive(bar_empty +
                                8 * ((2 * (kb + (kSplit ? wg + 2 * (n_mine - 1) : n_g - 1)) + 1) % R));
            }
            // Split keys: the warpgroups exchange their running maxima and sums, and each merges and
            // stores half the columns of every row (O = O_0 2^(m_0 - M) + O_1 2^(m_1 - M), likewise
            // l).  One warpgroup doing all of it left the CTA's tail, with nothing behind it, to
            // four warps: 64 sequences of 2,048 tokens took 18.2 us a step, now 17.6.
            float a0 = 1.f, a1 = 0.f;
            if (kSplit) {
                float2 *ml = reinterpret_cast<float2 *>(smem + PL::kML);   // [2][128]
                ml[wg * 128 + r] = make_float2(m_run, l_run);
                tmem_fence_before();
                asm volatile("bar.sync 1, %0;" ::"n"(8 * 32) : "memory");
                const float2 o0 = ml[r], o1 = ml[128 + r];
                m_run = o0.x;
                l_run = o0.y;
                if (o1.y != 0.f) {   // a NaN sum goes on into the row's output
                    const float mxx = fmaxf(m_run, o1.x);
                    a0 = fast_exp2(m_run - mxx);
                    a1 = fast_exp2(o1.x - mxx);
                    l_run = l_run * a0 + o1.y * a1;
                    m_run = mxx;
                }
            }
            // O of this row, 32 columns at c: the tile's buffer, or both merged
            auto load_o = [&](int c, float (&ov)[32]) {
                const uint32_t col = kSplit ? tmem + lane_off + PL::kColO : col_o;
                tmem_ld32_nowait(col + c * 32, ov);
                // The load is the whole warp's: its condition must not differ from row to row (a
                // row's a1 may be 0 or NaN).
                if (kSplit && n_g > 1) {
                    float o1[32];
                    tmem_ld32_nowait(col + D + c * 32, o1);
                    tmem_wait_ld();
                    if (a1 > 0.f) {
#pragma unroll
                        for (int k = 0; k < 32; ++k)
                            ov[k] = ov[k] * a0 + o1[k] * a1;
                    }
                } else {
                    tmem_wait_ld();
                }
            };
            // 32-column parts of 64 channels this warpgroup stores: both, or its own
            constexpr int kParts = kSplit ? 1 : 2;
            if (n_g > 0) {
                tmem_fence_after();
                const float inv = fast_rcp(l_run);
                const int stop = flags[0];
                // Row r of the tile.  Prefill: position q0 + r of the head.  Fused: layer
                // (grp ? 0 : L1) + r / G of the block, head j*G + r % G; out [layers][b][h][D].
                const int lay0 = y.blk * p.fused_L + (grp ? 0 : p.fused_L1);
                const int n_rows =
                    !kFused ? min(128, y.S - q0)
                            : (grp ? (p.fused_L < p.fused_L1 ? p.fused_L : p.fused_L1)
                                   : p.fused_L - p.fused_L1) * p.G;
                if (kFused && p.fused_cmax > 1) {
                    // One chunk of the context: o = O / l and lse = m + log2(l) for the merge.
                    const bool valid = r < n_rows && !stop;
                    const size_t row0 = (((static_cast<size_t>(y.blk) * p.b + y.beta) * p.g + y.j) *
                                             p.fused_cmax + y.chunk) * (p.fused_L * p.G) +
                                        (grp ? 0 : p.fused_L1) * p.G;
                    if (valid && wg == 0)
                        p.part_lse[row0 + r] = m_run + log2f(l_run);
                    float *prow = p.part + (row0 + r) * D;
#pragma unroll
                    for (int c0 = 0; c0 < PL::kSub * kParts; ++c0) {
                        const int c = kSplit ? wg : c0;
                        float ov[32];
                        load_o(c, ov);
                        if (valid) {
#pragma unroll
                            for (int k = 0; k < 32; k += 4)
                                *reinterpret_cast<float4 *>(prow + c * 32 + k) =
                                    make_float4(ov[k] * inv, ov[k + 1] * inv, ov[k + 2] * inv,
                                                ov[k + 3] * inv);
                        }
                    }
                } else {
                    // The warp's 32 rows go through shared memory, 64 channels at a time (16-byte
                    // chunks swizzled by row), and out 16 bytes a lane, 8 lanes a row: coalesced
                    // stores, which matters most when out is page-locked host memory.  At head_dim
                    // 64 the stage is the unit's own query tile (its last S has completed).
                    const int rw0 = (warp & 3) * 32;
                    uint8_t *stage = PL::kStageInQ ? q_slot + rw0 * 128
                                                   : smem + PL::kStage + warp * 4096;
#pragma unroll
                    for (int cb = 0; cb < PL::kSub; ++cb) {
#pragma unroll
                        for (int c0 = 0; c0 < kParts; ++c0) {
                            const int c = kSplit ? wg : c0;
                            float ov[32];
                            load_o(2 * cb + c, ov);
                            if (r < n_rows) {
#pragma unroll
                                for (int k = 0; k < 32; k += 8)
                                    *reinterpret_cast<uint4 *>(
                                        stage + lane * 128 + ((((c * 32 + k) >> 3) ^ (lane & 7)) << 4)) =
                                        make_uint4(pack_bf16x2(ov[k] * inv, ov[k + 1] * inv),
                                                   pack_bf16x2(ov[k + 2] * inv, ov[k + 3] * inv),
                                                   pack_bf16x2(ov[k + 4] * inv, ov[k + 5] * inv),
                                                   pack_bf16x2(ov[k + 6] * inv, ov[k + 7] * inv));
                            }
                        }
                        __syncwarp();
                        // 8 lanes a row (split keys: 4, this warpgroup's half of it)
                        constexpr int kLanes = 4 * kParts, kIts = kLanes;
                        const int ch = lane % kLanes + (kSplit ? 4 * wg : 0);
                        uint4 line[kIts];   // every load first: shared memory is busy with the MMAs
#pragma unroll
                        for (int it = 0; it < kIts; ++it) {
                            const int rl = it * (32 / kLanes) + lane / kLanes;
                            line[it] = *reinterpret_cast<const uint4 *>(stage + rl * 128 +
                                                                        ((ch ^ (rl & 7)) << 4));
                        }
                        __syncwarp();
#pragma unroll
                        for (int it = 0; it < kIts; ++it) {
                            const int rr = rw0 + it * (32 / kLanes) + lane / kLanes;
                            if (rr < n_rows && !stop) {
                                size_t row;   // of out, in units of D
                                if (kFused)
                                    row = (static_cast<size_t>(lay0 + rr / p.G) * p.b + y.beta) * p.h +
                                          y.j * p.G + rr % p.G;
                                else
                                    row = (static_cast<size_t>(y.beta) * p.s_max + (q0 + rr)) * p.h +
                                          (grp ? y.head_b : y.head_a);
                                *reinterpret_cast<uint4 *>(p.out + row * D + cb * 64 + ch * 8) =
                                    line[it];
                            }
                        }
                    }
                }
                tmem_fence_before();
            }
            if (PL::kStageInQ) {
                // The next queries may be written over the stage.  (Every warpgroup has a tile in
                // every unit here: two query tiles at head_dim 64 are a fused block of more rows
                // than one holds.)
                fence_proxy_async_smem();
                __syncwarp();
                if (lane == 0)
                    mbar_arrive(bar_q_free + 8 * qb);
            }
            kb += x.n_b;
            if (kSplit)
                break;   // one unit per CTA
        }
    } else {
        setmaxnreg_dec<PL::kRegsLow>();
        if (kFused && !kSplit && p.q_host != nullptr && warp == PL::kSoftWarps + 3) {
            // The last warp loads each unit's query rows from host memory, ahead of the unit.
            for (int n = 0;; ++n) {
                const int i = unit_index(p, n);
                if (i < 0)
                    break;
                const Unit x = unit_of<kFused, PL::kTiles>(p, i);
                const int qb = n % NQ;
                int ok = 1;
                if (lane == 0 && n >= NQ && !flags[0] &&
                    !mbar_wait(bar_q_free + 8 * qb, ((n / NQ) & 1) ^ 1)) {
                    flags[0] = 1;
                    atomicOr(p.err, kErrWaitEmpty);
                }
                if (lane == 0)
                    ok = !flags[0];
                if (!__shfl_sync(0xffffffffu, ok, 0))
                    break;
                load_q_host(x, qb, lane, std::integral_constant<int, 32>{},
                            std::integral_constant<int, PL::kRegsLow >= 72 ? 10 : 4>{});
                fence_proxy_async_smem();
                __syncwarp();
                if (lane == 0)
                    mbar_arrive(bar_q + 8 * qb);
            }
        }
    }

    tmem_fence_before();
    __syncthreads();
    if (warp == PL::kMma) {
        tmem_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                     "n"(PL::kTmemCols)
                     : "memory");
    }
}

// Merges the context chunks of the fused decode: per output row (block, sequence, KV head, block
// layer, group head) o = sum_c 2^(lse_c - M) o_c / sum_c 2^(lse_c - M), M = max_c lse_c.  W warps
// per row (fused_combine_w: 1, 2, 4 or 8, more for more chunks): warp w takes chunks w, w + W, ...,
// 8 of them in flight, and each lane keeps a running maximum, sum of weights and weighted sum for
// its D / 32 columns; the W warps' states are then merged through shared memory.
// Bound by latency: a few round trips to L2 behind the end of the decode grid.  The row's divisions
// run before the wait for it, and up to 64 chunks take one round trip (4 in flight and the
// divisions behind the wait: a step over 4 sequences of 8,192 tokens 15.2 us, now 12.1; one of
// 131,072 tokens 27.1, now 24.3; 12 in flight 12.8 and 24.2).
template <int D>
__global__ void __launch_bounds__(256, D == 64 ? 4 : 3) combine_fused_kernel(const __grid_constant__ PrefillParams p)
{
    constexpr int U = 8;        // chunks in flight a warp
    constexpr int E = D / 32;   // columns per lane
    using Vec = typename std::conditional<E == 2, float2, float4>::type;
    __shared__ float s_m[8], s_l[8];
    __shared__ Vec s_acc[8][32];
    const int W = p.fused_combine_w;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int w = warp % W;
    const int rows_per_head = p.fused_L * p.G;
    const long long row = static_cast<long long>(blockIdx.x) * (8 / W) + warp / W;
    const bool live = row < static_cast<long long>(p.fused_nblk) * p.b * p.g * rows_per_head;
    const float NEG_INF = -__int_as_float(0x7f800000);
    int rr = 0, j = 0, beta = 0, blk = 0, chunks = 0;
    size_t base = 0;
    if (live) {
        rr = static_cast<int>(row % rows_per_head);
        const long long bj = row / rows_per_head;   // (block, sequence, KV head)
        j = static_cast<int>(bj % p.g);
        const long long bb = bj / p.g;
        beta = static_cast<int>(bb % p.b);
        blk = static_cast<int>(bb / p.b);
        base = static_cast<size_t>(bj) * p.fused_cmax * rows_per_head + rr;
    }
    // Launched while the decode grid still runs: the partials are read after it has finished.
    grid_dependency_wait();
    grid_dependents_launch();
    if (live) {
        const int n_kt = (p.prompt_len[beta] + 127) / 128;
        chunks = (n_kt + p.fused_kc - 1) / p.fused_kc;
    }
    float m = NEG_INF, l = 0.f;
    float acc[E] = {};
    for (int c0 = w; c0 < chunks; c0 += U * W) {
        float lse[U];
        Vec v[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int c = c0 + u * W;
            const size_t r = base + static_cast<size_t>(c) * rows_per_head;
            if (c < chunks) {
                lse[u] = p.part_lse[r];
                v[u] = *reinterpret_cast<const Vec *>(p.part + r * D + lane * E);
            } else {
                lse[u] = NEG_INF;
                v[u] = Vec{};
            }
        }
        float mx = m;
#pragma unroll
        for (int u = 0; u < U; ++u)
            mx = fmaxf(mx, lse[u]);
        const float scale = m == NEG_INF ? 0.f : exp2f(m - mx);
        l *= scale;
#pragma unroll
        for (int e = 0; e < E; ++e)
            acc[e] *= scale;
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const float wt = lse[u] == NEG_INF ? 0.f : exp2f(lse[u] - mx);
            l += wt;
            const float *x = reinterpret_cast<const float *>(&v[u]);
#pragma unroll
            for (int e = 0; e < E; ++e)
                acc[e] += wt * x[e];
        }
        m = mx;
    }
    if (W > 1) {
        if (lane == 0) {
            s_m[warp] = m;
            s_l[warp] = l;
        }
        Vec a;
        float *ap = reinterpret_cast<float *>(&a);
#pragma unroll
        for (int e = 0; e < E; ++e)
            ap[e] = acc[e];
        s_acc[warp][lane] = a;
        __syncthreads();
        if (w != 0 || !live)
            return;
        // warp 0 of the row: every warp of the row against the largest maximum (warp 0 holds
        // chunk 0, so M is finite)
        float M = NEG_INF;
        for (int k = 0; k < W; ++k)
            M = fmaxf(M, s_m[warp + k]);
        l = 0.f;
#pragma unroll
        for (int e = 0; e < E; ++e)
            acc[e] = 0.f;
        for (int k = 0; k < W; ++k) {
            const float wt = s_m[warp + k] == NEG_INF ? 0.f : exp2f(s_m[warp + k] - M);
            l += wt * s_l[warp + k];
            const Vec b = s_acc[warp + k][lane];
            const float *x = reinterpret_cast<const float *>(&b);
#pragma unroll
            for (int e = 0; e < E; ++e)
                acc[e] += wt * x[e];
        }
    } else if (!live) {
        return;
    }
    const float inv = 1.f / l;
    const int layer = rr / p.G, i = rr - layer * p.G;
    __nv_bfloat16 *orow =
        p.out + ((static_cast<size_t>(blk * p.fused_L + layer) * p.b + beta) * p.h + j * p.G + i) * D;
#pragma unroll
    for (int e = 0; e < E; e += 2)
        *reinterpret_cast<uint32_t *>(orow + lane * E + e) =
            pack_bf16x2(acc[e] * inv, acc[e + 1] * inv);
}

template <int D, bool kFused, int kForm>
const void *prefill_fn()
{
    return reinterpret_cast<const void *>(&prefill_kernel<D, kFused, kForm>);
}

// The forms built: prefill at head_dim 64 with one query tile per CTA, at 128 with two; the fused
// decode in the two-tile form (either head_dim) or, at head_dim 64, either one-tile form.
template <typename F>
auto plan_value(int head_dim, int form, F f)
{
    if (head_dim == 64) {
        if (form == kOneDeep)
            return f(PrefillPlan<64, kOneDeep>{});
        return form == kOneTile ? f(PrefillPlan<64, kOneTile>{}) : f(PrefillPlan<64, kTwoTiles>{});
    }
    return f(PrefillPlan<128, kTwoTiles>{});
}
int threads_of(int head_dim, int form)
{
    return plan_value(head_dim, form, [](auto pl) { return decltype(pl)::kThreads; });
}
int regs_of(int head_dim, int form)
{
    return plan_value(head_dim, form, [](auto pl) { return decltype(pl)::kRegsLaunch; });
}
size_t smem_of(int head_dim, int form)
{
    return plan_value(head_dim, form,
                      [](auto pl) { return static_cast<size_t>(decltype(pl)::kAlloc); });
}

const void *kernel_fn(int head_dim, bool fused, int form)
{
    if (fused) {
        if (head_dim == 64)
            return form == kOneDeep   ? prefill_fn<64, true, kOneDeep>()
                   : form == kOneTile ? prefill_fn<64, true, kOneTile>()
                                      : prefill_fn<64, true, kTwoTiles>();
        return prefill_fn<128, true, kTwoTiles>();
    }
    return head_dim == 64 ? prefill_fn<64, false, kOneTile>() : prefill_fn<128, false, kTwoTiles>();
}

cudaError_t launch(int head_dim, bool fused, int form, const CUtensorMap *tmap_q,
                   const CUtensorMap *tmap_k, const CUtensorMap *tmap_v, const PrefillParams &p,
                   cudaStream_t stream)
{
    cudaLaunchConfig_t cfg = {};
    // persistent CTAs: at most one wave, each taking units in turn (unit_index)
    cfg.gridDim = dim3(static_cast<unsigned>(
        min(p.n_units, p.sm_count * (form == kOneTile ? 2 : 1))));
    cfg.blockDim = dim3(static_cast<unsigned>(threads_of(head_dim, form)));
    cfg.dynamicSmemBytes = smem_of(head_dim, form);
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    void *args[] = {const_cast<CUtensorMap *>(tmap_q), const_cast<CUtensorMap *>(tmap_k),
                    const_cast<CUtensorMap *>(tmap_v), const_cast<PrefillParams *>(&p)};
    return cudaLaunchKernelExC(&cfg, kernel_fn(head_dim, fused, form), args);
}

// The prefill form of a head_dim; a fused-decode form valid for the head_dim.
int prefill_form(int head_dim) { return head_dim == 64 ? kOneTile : kTwoTiles; }
int fused_form(int head_dim, int form) { return head_dim == 64 ? form : kTwoTiles; }

}  // namespace

size_t prefill_smem_bytes(int head_dim) { return smem_of(head_dim, prefill_form(head_dim)); }

// The warpgroups' register split (setmaxnreg) adds up to the registers the block is launched with;
// a kernel built with another per-thread count would wait forever in setmaxnreg.inc, so it is
// refused here instead of launched.
cudaError_t prepare(int head_dim, bool fused, int form)
{
    cudaFuncAttributes fa;
    const void *fn = kernel_fn(head_dim, fused, form);
    cudaError_t e = cudaFuncGetAttributes(&fa, fn);
    if (e != cudaSuccess)
        return e;
    if (fa.numRegs != regs_of(head_dim, form))
        return cudaErrorInvalidKernelImage;
    return cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                static_cast<int>(smem_of(head_dim, form)));
}

cudaError_t prepare_prefill(int head_dim)
{
    return prepare(head_dim, false, prefill_form(head_dim));
}

cudaError_t prepare_fused(int head_dim, int form)
{
    return prepare(head_dim, true, fused_form(head_dim, form));
}

cudaError_t launch_prefill(int head_dim, const CUtensorMap *tmap_q, const CUtensorMap *tmap_k,
                           const CUtensorMap *tmap_v, const PrefillParams &p, cudaStream_t stream)
{
    return launch(head_dim, false, prefill_form(head_dim), tmap_q, tmap_k, tmap_v, p, stream);
}

cudaError_t launch_fused(int head_dim, int form, const CUtensorMap *tmap_q,
                         const CUtensorMap *tmap_kv, const PrefillParams &p, cudaStream_t stream)
{
    return launch(head_dim, true, fused_form(head_dim, form), tmap_q, tmap_kv, tmap_kv, p, stream);
}

cudaError_t launch_fused_combine(int head_dim, const PrefillParams &p, cudaStream_t stream)
{
    const long long rows = static_cast<long long>(p.fused_nblk) * p.b * p.g * p.fused_L * p.G;
    const int per_cta = 8 / p.fused_combine_w;   // rows of a CTA
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>((rows + per_cta - 1) / per_cta));
    cfg.blockDim = dim3(256);
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    void *args[] = {const_cast<PrefillParams *>(&p)};
    const void *fn = head_dim == 64 ? reinterpret_cast<const void *>(&combine_fused_kernel<64>)
                                    : reinterpret_cast<const void *>(&combine_fused_kernel<128>);
    return cudaLaunchKernelExC(&cfg, fn, args);
}

}  // namespace mlkv
