// Grouped expert GEMMs with the weight rows on the MMA's M side and the tokens on its N side, on CTA
// pairs (tcgen05 cta_group::2, M = 256), fed by TMA.
//
// Section 3.1: each routed expert is F(x) = W2 (silu(W1 x) * (W3 x)) (SwiGLU). Per expert segment of
// permuted token rows:
//   GEMM13: acc = [W1 ; W3 rows] x^T, h[token, j] = bf16(silu(acc_gate[j]) * acc_up[j])
//   GEMM2:  o[token, j] = W2[j] . h[token]                                       (fp32 out)
// A tile is 256 weight rows x up to 256 tokens. The weights are the side whose size is fixed by the
// layer (d and w are multiples of 64; rows past the end arrive as zeros and are not stored), and the
// tokens are the side whose size varies: N is the tile's token count rounded up to 32, so a segment
// pays for at most 31 columns it does not have, where a tile with the tokens on M pays for up to 127
// (or 255) rows, and segments need no padding in memory (a tile's surplus columns read the next
// segment's rows, or zeros past the end, and are dropped).
// A segment of n rows is cut into ceil(n / 256) token tiles of equal size; tiles are walked weight
// tile by weight tile with the token tiles innermost, so the pairs that run side by side read the
// same weight rows at the same time and the segment's activations stay in L2.
//
// GEMM13 loads its A tile as one 4-D box of the packed expert block, {64 columns, 16 rows, W1 / W3,
// 4 row groups}: rows 32 g .. 32 g + 15 of a CTA's 128 are W1 rows and the next 16 the W3 rows of the
// same outputs, so the gate and up values of an output sit in one warp's TMEM quarter, 16 lanes
// apart, and meet with one shuffle per pair of columns.
//
// What bounds it (GB300, CUDA events in a steady loop, against 128-row token tiles with the
// tokens on M, since removed):
// * DeepSeek-V2-Lite shape, 4096 tokens on 48 of 64 experts (512 rows each): GEMM13 355 -> 240 us
//   (1.57 PFLOP/s), GEMM2 184 -> 154 us (1.23): the MMAs and the power cap. The old tiles paid 12 % for
//   padding and read 1.28 GB of DRAM where 0.69 GB does. Narrower token tiles and weights prefetched
//   into L2 were slower.
// * 200 tokens (19 rows an expert): HBM, the weights read once: GEMM13 145 -> 97 us, GEMM2 68 -> 55 us
//   (525 and 264 MB of weights: 5.4 and 4.8 TB/s, the start and the last round of tiles included).
// * Mixtral shape, 4096 tokens (2048 rows an expert), GEMM13 1219 -> 1147 us, GEMM2 661 -> 637 us: the
//   power cap.
// The two threads that issue are what the loops wait for when they are not kept short: with the ring
// walked under a lane test (operands moved to uniform registers one by one), tokens fetched as up to
// four boxes and the peer's barrier address found per block, the rates above were GEMM13 300 and
// GEMM2 175 us at 4096 DeepSeek tokens, 106 and 61 us at 200 (six stages). One elected lane, one box per half tile
// (hence a map for each size) and the addresses found once per tile gave the rest. Two k-blocks per
// stage and per copy (5-D and 3-D boxes) were faster than the old loop and are slower than this one.
// Eight epilogue warps rather than four, and a quotient without branches (silu_branchless): the SwiGLU of a
// tile took about 28,000 cycles on four warps, more than the MMAs of a 2048-long contraction (16,400).
// d = 960, w = 704 (15 k-blocks), 16 experts: GEMM13 at T = 4096 99 -> 63 us by the quotient alone.
//
// Roles (both CTAs of a pair): warp 0 TMA producer (its 128 weight rows and its half of the tokens,
// counted on the leader's full[s]); warp 1 allocates TMEM and, in the leader, issues the MMAs; warps
// 2-9 read the CTA's 128 accumulator rows and store them from registers. Two accumulators of 256
// columns, so a tile's epilogue runs under the next tile's MMAs. All of the shared memory is the ring,
// 224 KB: the MMAs take a stage of a 256-token tile in 270 ns, so what the ring covers of a load's
// latency is short. Seven stages of 32 KB there (and up to ten of narrower tiles; twelve were slower)
// against six with a staging buffer for h beside them: 800 DeepSeek tokens 247 -> 239 us, 200 tokens
// 166 -> 162, 4096 even (476 / 475). Stages of each tile's own size (more of them where the shared
// experts' tiles are wide and the routed ones' narrow) cost the producer more than they gave: 200
// tokens 171 us, 4096 498.
//
// With LoRA adapters (Section 3.2, Stage 2) an adapted tile appends p.nx k-blocks of one MMA each,
// D += B' U^T: for GEMM13 B' is B1 on the gate rows (zeros on the up rows) with U = s A1 x, then B3 on
// the up rows with U = s A3 x (and, if kept, the other bf16 parts of U against the same B'); for GEMM2
// B' = B2, U = s A2 h. The zeros are TMA out-of-bounds fill: the adapter matrices are r columns wide
// under boxes of 64, and the W1 / W3 dimension of the box is one plane long, entered at 0 or at -1.
//
// A cached forward's launch (RowsCacheParams) finds its weights in the cache step's device table. The other
// launches carry none of that code. Per tile everything is as in the plain launch, hence the same bits.
//
// Every wait is bounded: after 2 s the kernel records MCFT_ERR_TIMEOUT, stops issuing, waits (bounded)
// for its copies and MMAs in flight, frees TMEM and returns.
#include <type_traits>

#include "common.cuh"
#include "internal.h"
#include "tc_ptx.cuh"

namespace mcft {
namespace {

constexpr int kEpiGroups = 2;                 // of four warps, one per TMEM lane quarter
constexpr int kThreads = 64 + kEpiGroups * 128;
constexpr int BK = 64;
constexpr int kTileTok = 256;                 // most tokens of a tile
constexpr int kBoxes = 8;                     // token boxes of 16, 32, .. 128 rows: one per half tile
constexpr int kUBoxes = 4;                    // adapters' U: boxes of 16, 32, 64 and 128 rows, combined
constexpr int kMaxStages = 10;
constexpr int kABytes = 128 * BK * 2;         // a CTA's weight rows of a stage
constexpr int kRingBytes = 7 * (kABytes + (kTileTok / 2) * BK * 2);
constexpr int kTmemCols = 2 * kTileTok;
// instruction descriptor without N: D fp32, A and B bf16, both K-major, M = 256
constexpr uint32_t kIdesc = (1u << 4) | (1u << 7) | (1u << 10) | (uint32_t(256 >> 4) << 24);

enum { EPI_SWIGLU = 0, EPI_F32 = 1 };

struct RowsParams {
  CUtensorMap x[kBoxes];   // permuted rows (GEMM13: gathered x; GEMM2: h), boxes of 16 (i + 1) rows
  CUtensorMap sx[kBoxes];  // GEMM13: x itself, whose rows are the shared experts' rows in order
  CUtensorMap w[kMaxSeg];
  const int* off;
  const WsHeader* hdr;
  void* out;
  unsigned* err;
  uint32_t wmask[3];  // segments that have weights
  int nseg, E, kblocks, mtiles, ldo, group_x, use_sx;
};
struct RowsLoraParams : RowsParams {
  CUtensorMap u[kUBoxes];            // U [rows, extra k-blocks, r]
  CUtensorMap lb[2][kMaxSeg];        // GEMM13: B1, B3; GEMM2: B2
  uint32_t lmask[3];                 // segments with an adapter
  int nx;
};

// A cached forward: the routed experts' blocks are in the layer's cache slots or in the staging buffers,
// where the device table of the cache step says; their maps cover all blocks of either kind, with the block
// as the last coordinate. One launch computes the segments of one phase (seg_in_phase).
struct RowsCacheParams : RowsParams {
  CUtensorMap blocks[2];  // slots, staging buffers
  const unsigned long long* wtab;   // [E] block addresses
  const unsigned long long* ready;  // hit mask
  unsigned long long base[2], bytes;
  int count[2];
  int phase;
};

static_assert(sizeof(RowsLoraParams) <= 32764 && sizeof(RowsCacheParams) <= 32764, "kernel parameters");

struct Ctl {
  uint64_t full[kMaxStages], empty[kMaxStages], tfull[2], tempty[2], drain;
  uint32_t tmem_base;
  int abort, tiles, stages, stage_bytes;
  int off[kMaxSeg + 1];
  int first[kMaxSeg + 1];  // by position (segments in reverse order): first tile
  int block[kMaxE];        // cached forward: block of each routed expert, staging buffers from kStaging
};
constexpr int kStaging = 1 << 24;  // (more blocks than a GPU can hold)
constexpr int kCtlBytes = (int(sizeof(Ctl)) + 15) / 16 * 16;
constexpr int kSmem = kRingBytes + 1024 + kCtlBytes;
static_assert(kSmem <= 227 * 1024, "shared memory");

__device__ __forceinline__ void tma_load_4d_pair(uint32_t dst, const CUtensorMap* map, int c0,
                                                 int c1, int c2, int c3, uint32_t bar_cluster) {
  asm volatile(
      "cp.async.bulk.tensor.4d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3, %4, %5}], [%6];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(bar_cluster)
      : "memory");
}

__device__ __forceinline__ void tma_load_3d_pair(uint32_t dst, const CUtensorMap* map, int c0,
                                                 int c1, int c2, uint32_t bar_cluster) {
  asm volatile(
      "cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(bar_cluster)
      : "memory");
}
__device__ __forceinline__ void tma_load_5d_pair(uint32_t dst, const CUtensorMap* map, int c0, int c1,
                                                 int c2, int c3, int c4, uint32_t bar_cluster) {
  asm volatile(
      "cp.async.bulk.tensor.5d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3, %4, %5, %6}], [%7];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(c4),
      "r"(bar_cluster)
      : "memory");
}

__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t* r) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,"
      "%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
        "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]),
        "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]),
        "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr));
}

__device__ __forceinline__ int token_tiles(int rows) { return (rows + kTileTok - 1) / kTileTok; }
// Tokens of a segment's tiles, all but the last one's: equal shares, rounded up to 32.
__device__ __forceinline__ int tile_tokens(int rows) {
  const int nt = max(token_tiles(rows), 1);
  return ((rows + nt - 1) / nt + 31) & ~31;
}

struct TileAt {
  int seg, mt, row0, n;  // segment, weight tile, first permuted row, tokens
  __device__ int cols() const { return (n + 31) & ~31; }
};

// Tile -> segment, weight tile and token tile. Segments are taken last to first (the shared
// experts, whose tiles are the largest, before the routed ones); inside a segment groups of at most
// group_x token tiles, weight tiles inside a group, token tiles innermost.
__device__ __forceinline__ TileAt tile_at(const Ctl* c, int nseg, int mtiles, int group_x, int tile) {
  int lo = 0, hi = nseg - 1;  // the last position whose first tile is <= tile: it is not empty
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (c->first[mid] <= tile) lo = mid;
    else hi = mid - 1;
  }
  TileAt t;
  t.seg = nseg - 1 - lo;
  const int local = tile - c->first[lo];
  const int rows = c->off[t.seg + 1] - c->off[t.seg];
  const int nt = token_tiles(rows);
  const int ts = tile_tokens(rows);  // (nt - 1) * ts < rows, since ts <= 256
  const int g = local / (group_x * mtiles);
  const int r = local - g * group_x * mtiles;
  const int gsz = min(group_x, nt - g * group_x);
  t.mt = r / gsz;
  const int j = g * group_x + r % gsz;
  t.row0 = c->off[t.seg] + j * ts;
  t.n = min(ts, rows - j * ts);
  return t;
}

__device__ __forceinline__ bool in_mask(const uint32_t* m, int s) { return (m[s >> 5] >> (s & 31)) & 1u; }

// The segments of a cached forward's launch: hits and shared experts (phase 1), the others (phase 2).
__device__ __forceinline__ bool rows_in_phase(const RowsCacheParams& p, int s) {
  const bool hit = s >= p.E || ((*p.ready >> s) & 1ull);
  return p.phase == 1 ? hit : !hit;
}

template <int EPI, typename P>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kThreads, 1)
    gemm_rows_kernel(const __grid_constant__ P p) {
  constexpr bool LORA = std::is_same_v<P, RowsLoraParams>;
  constexpr bool CACHED = std::is_same_v<P, RowsCacheParams>;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;  // the same offsets in both CTAs
  Ctl* ctl = reinterpret_cast<Ctl*>(smem_raw + (base - raw) + kRingBytes);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cluster_rank();
  const bool leader = rank == 0;
  const int nseg = p.nseg;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kMaxStages; ++s) {
      mbar_init(&ctl->full[s], 1);
      mbar_init(&ctl->empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&ctl->tfull[b], 1);
      mbar_init(&ctl->tempty[b], 8 * kEpiGroups);
    }
    mbar_init(&ctl->drain, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(&ctl->tmem_base)),
                 "r"(kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  pdl_wait();
  if (warp == 2) {
    // segment offsets and the first tile of every position (three positions per lane); both CTAs
    // find the same values and the same abort decision
    const int aborted = p.hdr->abort;
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      const int s = lane + 32 * j;
      if (s <= nseg) ctl->off[s] = p.off[s];
    }
    if constexpr (CACHED) {
      for (int e = lane; e < p.E; e += 32) {
        const unsigned long long addr = p.wtab[e];
        int blk = -1;
#pragma unroll
        for (int i = 0; i < 2; ++i)
          if (addr >= p.base[i] && addr < p.base[i] + p.bytes * unsigned(p.count[i]))
            blk = int((addr - p.base[i]) / p.bytes) + i * kStaging;
        ctl->block[e] = blk;
      }
    }
    __syncwarp();
    int cnt[3], sum = 0, wide = 0;
    bool bad = false;
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      const int pos = lane * 3 + j, s = nseg - 1 - pos;
      int rows = pos < nseg ? ctl->off[s + 1] - ctl->off[s] : 0;
      bool weights = rows > 0 && in_mask(p.wmask, s);
      if constexpr (CACHED) {
        if (rows > 0 && !rows_in_phase(p, s)) rows = 0;
        if (rows > 0 && s < p.E) weights = ctl->block[s] >= 0;
      }
      bad |= rows > 0 && !weights;  // a selected expert without weights
      cnt[j] = token_tiles(rows) * p.mtiles;
      sum += cnt[j];
      wide = max(wide, tile_tokens(rows));
    }
    wide = __reduce_max_sync(0xffffffffu, wide);
    int incl = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += v;
    }
    int excl = incl - sum;
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      const int pos = lane * 3 + j;
      if (pos <= nseg) ctl->first[pos] = excl;
      excl += cnt[j];
    }
    const bool any_bad = __any_sync(0xffffffffu, bad);
    if (lane == 31) {
      const bool stop = aborted != 0 || any_bad;
      if (any_bad && aborted == 0) {
        set_error(p.err, kErrInvalid);
        const_cast<WsHeader*>(p.hdr)->abort = 1;  // later kernels of the call skip their work
      }
      ctl->abort = stop ? 1 : 0;
      ctl->tiles = stop ? 0 : incl;
      ctl->stage_bytes = kABytes + wide / 2 * BK * 2;
      ctl->stages = min(kMaxStages, kRingBytes / ctl->stage_bytes);
    }
  }
  tc_fence_before();
  cluster_sync();  // barriers initialised, TMEM allocated and the tile table built in both CTAs
  tc_fence_after();

  const uint32_t tmem = ctl->tmem_base;
  const int tiles = ctl->tiles;
  const int cid = int(blockIdx.x >> 1), ncl = int(gridDim.x >> 1);  // pair, pairs
  volatile int* abort = &ctl->abort;
  const int stages = ctl->stages, stage_bytes = ctl->stage_bytes;
  // k-blocks of a segment's tiles: the contraction, then the adapter's extra ones
  auto extra_of = [&](int seg) -> int {
    if constexpr (LORA) return in_mask(p.lmask, seg) ? p.nx : 0;
    else return 0;
  };

  if (warp == 0) {
    if (cid < tiles && elect_one()) {
      const uint32_t fb0 = peer_addr(&ctl->full[0], 0);
      int s = 0, issued = 0;
      uint32_t ph = 0;
      for (int tile = cid; tile < tiles && !*abort; tile += ncl) {
        const TileAt t = tile_at(ctl, nseg, p.mtiles, p.group_x, tile);
        const int half = t.cols() / 2, mrow = t.mt * 2 + int(rank);
        const bool sx = EPI == EPI_SWIGLU && p.use_sx && t.seg >= p.E;
        const int xrow = t.row0 - (sx ? ctl->off[t.seg] : 0) + int(rank) * half;
        const uint32_t bytes = 2u * uint32_t(kABytes + half * BK * 2);
        const CUtensorMap* mw = &p.w[t.seg];
        const CUtensorMap* mx = (sx ? p.sx : p.x) + (half / 16 - 1);
        const int nkb = p.kblocks;
        int block = -1;  // of the maps over all of the cache's blocks
        if constexpr (CACHED) {
          if (t.seg < p.E) {
            block = ctl->block[t.seg];
            mw = &p.blocks[block >= kStaging ? 1 : 0];
            block -= block >= kStaging ? kStaging : 0;
          }
        }
        int kb = 0;
        for (; kb < nkb; ++kb) {
          if (!mbar_wait_cl(&ctl->empty[s], ph ^ 1u, abort, p.err)) break;
          const uint32_t sa = base + uint32_t(s * stage_bytes), fb = fb0 + uint32_t(s) * 8u;
          if (leader) mbar_expect_tx(&ctl->full[s], bytes);
          if (CACHED && block >= 0) {
            if constexpr (EPI == EPI_SWIGLU)
              tma_load_5d_pair(sa, mw, kb * BK, 0, 0, mrow * 4, block, fb);
            else
              tma_load_3d_pair(sa, mw, kb * BK, mrow * 128, block, fb);
          } else if constexpr (EPI == EPI_SWIGLU) {
            tma_load_4d_pair(sa, mw, kb * BK, 0, 0, mrow * 4, fb);
          } else {
            tma_load_2d_pair(sa, mw, kb * BK, mrow * 128, fb);
          }
          tma_load_2d_pair(sa + kABytes, mx, kb * BK, xrow, fb);
          if (issued < stages) ++issued;
          if (++s == stages) {
            s = 0;
            ph ^= 1u;
          }
        }
        if constexpr (LORA) {
          const int nx = kb == nkb ? extra_of(t.seg) : 0;
          for (int e = 0; e < nx; ++e) {
            if (!mbar_wait_cl(&ctl->empty[s], ph ^ 1u, abort, p.err)) break;
            const uint32_t sa = base + uint32_t(s * stage_bytes), fb = fb0 + uint32_t(s) * 8u;
            if (leader) mbar_expect_tx(&ctl->full[s], bytes);
            // B1 fills the gate rows of the box, B3 (entered at plane -1) the up rows
            const int m = EPI == EPI_SWIGLU ? (e & 1) : 0;
            if constexpr (EPI == EPI_SWIGLU)
              tma_load_4d_pair(sa, &p.lb[m][t.seg], 0, 0, -m, mrow * 4, fb);
            else
              tma_load_2d_pair(sa, &p.lb[m][t.seg], 0, mrow * 128, fb);
            int r = 0;
#pragma unroll
            for (int b = kUBoxes - 1; b >= 0; --b)
              if (half & (16 << b)) {
                tma_load_3d_pair(sa + kABytes + uint32_t(r) * (BK * 2), &p.u[b], 0, e,
                                 t.row0 + int(rank) * half + r, fb);
                r += 16 << b;
              }
            if (issued < stages) ++issued;
            if (++s == stages) {
              s = 0;
              ph ^= 1u;
            }
          }
        }
      }
      // Stages still in flight: the leader waits for their bytes (both CTAs'), the peer until the
      // leader's MMAs consumed them; after the first wait that runs out the rest are skipped.
      // (oldest first: the stages before s in this round of the ring, those from s on in the last one)
      for (int i = 0; i < issued; ++i) {
        const int back = issued - i, j = s - back;
        uint64_t* ring = leader ? ctl->full : ctl->empty;
        if (!mbar_wait_drain_cl(&ring[j < 0 ? j + stages : j], j < 0 ? ph ^ 1u : ph, p.err)) break;
      }
    }
  } else if (warp == 1) {
    if (leader && cid < tiles && elect_one()) {
      int s = 0;
      uint32_t ph = 0, lt = 0;
      for (int tile = cid; tile < tiles && !*abort; tile += ncl) {
        const TileAt t = tile_at(ctl, nseg, p.mtiles, p.group_x, tile);
        const uint32_t idesc = kIdesc | (uint32_t(t.cols() >> 3) << 17);
        const int nkb = p.kblocks + extra_of(t.seg);
        const uint32_t b = lt & 1u;
        if (!mbar_wait_cl(&ctl->tempty[b], ((lt >> 1) & 1u) ^ 1u, abort, p.err)) break;
        tc_fence_after();
        const uint32_t dt = tmem + b * kTileTok;
        bool ok = true;
        for (int kb = 0; kb < nkb; ++kb) {
          if (!mbar_wait_cl(&ctl->full[s], ph, abort, p.err)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t sa = base + uint32_t(s * stage_bytes), sb = sa + kABytes;
          const uint64_t da = sw128_desc(sa), db = sw128_desc(sb);
          if (!LORA || kb < p.kblocks) {
#pragma unroll
            for (int k = 0; k < BK / 16; ++k)
              tc_mma_pair(dt, da + uint64_t(2 * k), db + uint64_t(2 * k), idesc,
                          (kb | k) != 0 ? 1u : 0u);
          } else {  // an adapter's k-block: r <= 16 columns, the rest zeros
            tc_mma_pair(dt, da, db, idesc, 1u);
          }
          tc_commit_pair_both(&ctl->empty[s]);
          if (++s == stages) {
            s = 0;
            ph ^= 1u;
          }
        }
        if (!ok) break;
        tc_commit_pair_both(&ctl->tfull[b]);
        ++lt;
      }
      tc_commit_pair(&ctl->drain);  // arrives once every MMA issued above has completed
      mbar_wait_drain_cl(&ctl->drain, 0, p.err);
    }
  } else {
    const int q = warp & 3, grp = (warp - 2) >> 2;  // TMEM lane quarter this warp may access; group
    uint32_t lt = 0;
    for (int tile = cid; tile < tiles; tile += ncl) {
      const TileAt t = tile_at(ctl, nseg, p.mtiles, p.group_x, tile);
      const uint32_t b = lt & 1u;
      int ok = 1;
      if (lane == 0) ok = mbar_wait_cl(&ctl->tfull[b], (lt >> 1) & 1u, abort, p.err) ? 1 : 0;
      if (!__shfl_sync(0xffffffffu, ok, 0)) break;
      tc_fence_after();
      const uint32_t taddr = tmem + b * kTileTok + (uint32_t(q * 32) << 16);
      // the groups take the 32-token chunks in turn
      for (int c0 = grp * 32; c0 < t.n; c0 += 32 * kEpiGroups) {
        uint32_t v[32];
        tmem_ld32(taddr + c0, v);
        tmem_ld_wait();
        if constexpr (EPI == EPI_SWIGLU) {
          // lanes 0-15 hold the gate and lanes 16-31 the up values of 16 outputs: lane pairs
          // exchange, so that a low lane finishes the even tokens and a high lane the odd ones, and
          // a store writes one 32-byte sector of each of two rows
          const bool low = lane < 16;
          const int col = (t.mt * 2 + int(rank)) * 64 + q * 16 + (lane & 15);
          const int m = t.n - c0 - (low ? 0 : 1);
          uint16_t* dst = reinterpret_cast<uint16_t*>(p.out) +
                          size_t(t.row0 + c0 + (low ? 0 : 1)) * p.ldo + col;
          const bool in = col < p.ldo;
          bool regular = true;
#pragma unroll
          for (int i = 0; i < 16; ++i) {
            const uint32_t mine = low ? v[2 * i] : v[2 * i + 1];
            const uint32_t got = __shfl_xor_sync(0xffffffffu, low ? v[2 * i + 1] : v[2 * i], 16);
            v[2 * i] = low ? mine : got;
            v[2 * i + 1] = low ? got : mine;
            const float g = __uint_as_float(v[2 * i]);
            regular &= silu_regular(g);
            const uint16_t h = f2bf(silu_branchless(g) * __uint_as_float(v[2 * i + 1]));
            if (in && 2 * i < m) dst[2 * i * size_t(p.ldo)] = h;
          }
          if (!regular) {  // rare: this lane's values again, by IEEE division
#pragma unroll
            for (int i = 0; i < 16; ++i)
              if (in && 2 * i < m)
                dst[2 * i * size_t(p.ldo)] = f2bf(silu(__uint_as_float(v[2 * i])) * __uint_as_float(v[2 * i + 1]));
          }
        } else {
          const int col = t.mt * 256 + int(rank) * 128 + q * 32 + lane;
          if (col < p.ldo) {
            float* dst = reinterpret_cast<float*>(p.out) + size_t(t.row0 + c0) * p.ldo + col;
            const int m = t.n - c0;
#pragma unroll
            for (int i = 0; i < 32; ++i, dst += p.ldo)
              if (i < m) *dst = __uint_as_float(v[i]);
          }
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive_cluster(peer_addr(&ctl->tempty[b], 0));
      ++lt;
    }
  }

  tc_fence_before();
  cluster_sync();  // the leader's MMAs drained, every copy landed, both epilogues done
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols)
                 : "memory");
  }
}

// ---- host ----

bool encode(CUtensorMap* m, const void* base, int rank, const cuuint64_t* dims,
            const cuuint64_t* strides, const cuuint32_t* box) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  const cuuint32_t es[5] = {1, 1, 1, 1, 1};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, cuuint32_t(rank), const_cast<void*>(base), dims,
            strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
            CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// bf16 rows [rows, cols] with a row stride of `stride` elements; boxes of 64 columns x box_rows.
bool encode_rows(CUtensorMap* m, const void* base, uint64_t cols, uint64_t rows, uint64_t stride,
                 uint32_t box_rows) {
  const cuuint64_t dims[2] = {cols, rows}, strides[1] = {stride * 2};
  const cuuint32_t box[2] = {BK, box_rows};
  return encode(m, base, 2, dims, strides, box);
}
bool encode_boxes(CUtensorMap* m, const void* base, uint64_t cols, uint64_t rows, uint64_t stride) {
  for (int b = 0; b < kBoxes; ++b)
    if (!encode_rows(m + b, base, cols, rows, stride, 16u * uint32_t(b + 1))) return false;
  return true;
}
// Rows of `planes` matrices [rows, cols] (plane stride in elements), interleaved 16 by 16: box of 64
// columns x 16 rows x 2 planes x 4 groups = the 128 A rows of a GEMM13 CTA.
bool encode_gate_up(CUtensorMap* m, const void* base, uint64_t cols, uint64_t rows, uint64_t planes,
                    uint64_t plane_stride) {
  const cuuint64_t dims[4] = {cols, 16, planes, rows / 16};
  const cuuint64_t strides[3] = {cols * 2, plane_stride * 2, 16 * cols * 2};
  const cuuint32_t box[4] = {BK, 16, 2, 4};
  return encode(m, base, 4, dims, strides, box);
}

template <int EPI, typename P>
cudaError_t launch_rows(const P& p, int num_sms, cudaStream_t s) {
  static SmemOptIn smem;
  static ResidentClusters resident;  // a persistent grid of pairs that all run at once
  const void* fn = reinterpret_cast<const void*>(gemm_rows_kernel<EPI, P>);
  cudaError_t e = smem.allow(fn, kSmem);
  if (e != cudaSuccess) return e;
  const int pairs = resident.get(fn, num_sms & ~1, kThreads, kSmem);
  if (pairs < 1) return cudaErrorInvalidConfiguration;
  const int kid = EPI == EPI_SWIGLU ? kProfGemm13 : kProfGemm2;
  prof_begin(kid, s);
  e = launch_pdl(gemm_rows_kernel<EPI, P>, dim3(2 * pairs), dim3(kThreads), kSmem, s, p);
  prof_end(kid, s);
  return e != cudaSuccess ? e : cudaGetLastError();
}

// Token tiles per group: as many as keep this many bytes of activations in L2.
constexpr size_t kGroupBytes = size_t(24) << 20;
int group_for(int K) {
  const size_t tile = size_t(kTileTok) * K * 2, g = kGroupBytes / tile;
  return g < 1 ? 1 : int(g);
}

// The parameters of one of the two GEMMs (stage 1: GEMM13, stage 2: GEMM2); 0 on failure.
bool fill(RowsParams& p, const FfnArgs& a, const void* xp, int mcap, int stage) {
  const uint64_t d = uint64_t(a.d), w = uint64_t(a.w);
  const uint64_t K = stage == 1 ? d : w;
  if (!encode_boxes(p.x, stage == 1 ? xp : a.h, K, uint64_t(mcap), K)) return false;
  if (stage == 1 && !encode_boxes(p.sx, a.x, d, uint64_t(a.T), d)) return false;
  for (int s = 0; s < a.nseg; ++s) {
    const char* blk = reinterpret_cast<const char*>(a.wblk[s]);
    if (!blk) continue;
    const bool ok = stage == 1 ? encode_gate_up(&p.w[s], blk, d, w, 2, w * d)
                               : encode_rows(&p.w[s], blk + 2 * w * d * 2, w, d, w, 128);
    if (!ok) return false;
    p.wmask[s >> 5] |= 1u << (s & 31);
  }
  p.off = a.off;
  p.hdr = a.hdr;
  p.out = stage == 1 ? a.h : static_cast<void*>(a.o);
  p.err = a.err;
  p.nseg = a.nseg;
  p.E = a.E;
  p.kblocks = int(K / BK);
  p.mtiles = stage == 1 ? (a.w + 127) / 128 : (a.d + 255) / 256;
  p.ldo = stage == 1 ? a.w : a.d;
  p.group_x = group_for(int(K));
  p.use_sx = stage == 1 ? 1 : 0;
  return true;
}

// The adapters of one GEMM. U planes of r columns side by side: GEMM13 [s A1 x | s A3 x], GEMM2 s A2 h, then
// the same of each further bf16 part; 16-byte rows and offsets for r = 8 and 16.
bool fill_lora(RowsLoraParams& p, const FfnArgs& a, int mcap, int stage, int split) {
  const LoraOffsets lo = lora_offsets(a.d, a.w, a.lrank);
  const uint64_t r = uint64_t(a.lrank);
  p.nx = (stage == 1 ? 2 : 1) * split;
  const cuuint64_t nx = cuuint64_t(p.nx), dims[3] = {r, nx, uint64_t(mcap)}, strides[2] = {r * 2, nx * r * 2};
  for (int b = 0; b < kUBoxes; ++b) {
    const cuuint32_t box[3] = {BK, 1, 16u << b};
    if (!encode(&p.u[b], stage == 1 ? a.u13 : a.u2, 3, dims, strides, box)) return false;
  }
  for (int s = 0; s < a.nseg; ++s) {
    const char* blk = reinterpret_cast<const char*>(a.lblk[s]);
    if (!blk || !a.wblk[s]) continue;
    const bool ok = stage == 1
                        ? encode_gate_up(&p.lb[0][s], blk + lo.b1 * 2, r, uint64_t(a.w), 1, a.w * r) &&
                              encode_gate_up(&p.lb[1][s], blk + lo.b3 * 2, r, uint64_t(a.w), 1, a.w * r)
                        : encode_rows(&p.lb[0][s], blk + lo.b2 * 2, r, uint64_t(a.d), r, 128);
    if (!ok) return false;
    p.lmask[s >> 5] |= 1u << (s & 31);
  }
  return true;
}

// The cache's blocks: encode_gate_up's and encode_rows' maps with the block as one dimension more.
bool fill_cache(RowsCacheParams& p, const FfnArgs& a, const CacheBlocks& c, int stage) {
  const uint64_t d = uint64_t(a.d), w = uint64_t(a.w);
  for (int i = 0; i < 2; ++i) {
    p.base[i] = reinterpret_cast<unsigned long long>(c.base[i]);
    p.count[i] = c.count[i];
    if (c.count[i] >= kStaging) return false;
    if (c.count[i] == 0) continue;
    const cuuint64_t n = cuuint64_t(c.count[i]), bytes = c.bytes;
    const char* base = static_cast<const char*>(c.base[i]);
    if (stage == 1) {
      const cuuint64_t dims[5] = {d, 16, 2, w / 16, n}, strides[4] = {d * 2, w * d * 2, 16 * d * 2, bytes};
      const cuuint32_t box[5] = {BK, 16, 2, 4, 1};
      if (!encode(&p.blocks[i], base, 5, dims, strides, box)) return false;
    } else {
      const cuuint64_t dims[3] = {w, d, n}, strides[2] = {w * 2, bytes};
      const cuuint32_t box[3] = {BK, 128, 1};
      if (!encode(&p.blocks[i], base + 2 * w * d * 2, 3, dims, strides, box)) return false;
    }
  }
  p.bytes = c.bytes;
  p.wtab = a.wtab;
  p.ready = a.ready;
  p.phase = a.phase;
  return true;
}

template <int EPI, typename P>
cudaError_t run(const FfnArgs& a, const void* xp, int mcap, int num_sms, cudaStream_t s, int split,
                const CacheBlocks* cache = nullptr) {
  P p;
  memset(&p, 0, sizeof(p));
  const int stage = EPI == EPI_SWIGLU ? 1 : 2;
  if (!fill(p, a, xp, mcap, stage)) return cudaErrorInvalidValue;
  if constexpr (std::is_same_v<P, RowsLoraParams>) {
    if (!fill_lora(p, a, mcap, stage, split)) return cudaErrorInvalidValue;
  }
  if constexpr (std::is_same_v<P, RowsCacheParams>) {
    if (!fill_cache(p, a, *cache, stage)) return cudaErrorInvalidValue;
  }
  return launch_rows<EPI, P>(p, num_sms, s);
}

}  // namespace

cudaError_t launch_ffn_rows(const FfnArgs& a, const void* xp, int mcap, int num_sms, cudaStream_t s,
                            int stages, int split) {
  cudaError_t e = cudaSuccess;
  if (stages & 1)
    e = a.lrank > 0 ? run<EPI_SWIGLU, RowsLoraParams>(a, xp, mcap, num_sms, s, split)
                    : run<EPI_SWIGLU, RowsParams>(a, xp, mcap, num_sms, s, split);
  if (e != cudaSuccess || !(stages & 2)) return e;
  return a.lrank > 0 ? run<EPI_F32, RowsLoraParams>(a, xp, mcap, num_sms, s, split)
                     : run<EPI_F32, RowsParams>(a, xp, mcap, num_sms, s, split);
}

cudaError_t launch_ffn_rows_cached(const FfnArgs& a, const CacheBlocks& cache, const void* xp, int mcap,
                                   int num_sms, cudaStream_t s) {
  const cudaError_t e = run<EPI_SWIGLU, RowsCacheParams>(a, xp, mcap, num_sms, s, 1, &cache);
  return e != cudaSuccess ? e : run<EPI_F32, RowsCacheParams>(a, xp, mcap, num_sms, s, 1, &cache);
}

}  // namespace mcft
