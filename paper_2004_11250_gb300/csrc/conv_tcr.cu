// Pattern-pruned 3x3 convolution on CTA pairs of tensor cores, for layers with at
// most 64 filters (the inner layers of super-resolution stacks, the first blocks
// of VGG-like trunks) and 128-filter blocks on wide maps: the
// same dense 9-tap contraction and the same hi / lo splits as conv_tc.cu, with
// the whole weight set of a layer of at most 64 filters and 64 channels resident
// in shared memory.
//
// Method: Niu et al., IJCAI-20 demo, Sections 2 (pattern and connectivity
// pruning, here zeros of the dense 9-tap weights) and 3 (fused activation).
//
// What bounded the row-tiled kernel on these layers is the SM's shared memory
// (128 bytes per clock): per 8-channel chunk of a 2 x 128 pixel tile 252 KB of
// MMA operand reads, a 37 KB weight copy, and 68 KB of input box and operand
// staging.  Here two SMs form a pair (cta_group::2, M = 256 pixels, 128 of each
// CTA): each holds half of the weight rows, so that
//   * a tap's weights are read once for 256 pixels (198 KB per chunk instead of
//     252) and
//   * all chunks' weights fit (147 KB per CTA in tf32, 74 KB in f16) and are
//     copied once per launch instead of once per tile and chunk;
// and the loaders fetch x straight into registers, one chunk ahead, and write
// only the split operands to shared memory: no input box, and rows of any
// width and alignment take the same path.
//
// Weight rows.  For a tap the B operand of x_hi is [w_hi | w_lo] (N = 128), that
// of x_lo is w_hi (N = 64).  cta_group::2 takes the first half of B's columns
// from the even CTA and the second half from the odd one, at one shared-memory
// address in both.  With F0 / F1 the first / last 32 filters, the even CTA holds
// [w_hi F0 ; w_lo F1] and the odd one [w_hi F1 ; w_lo F0].  The first MMA's 128
// accumulator columns are then, by quarters, hi F0 | lo F1 | hi F1 | lo F0, and
// the second MMA (each CTA's first 32 rows) lands on two adjacent quarters:
//   tf32: on the first two, which are F0 and F1; F0 = q0 + q3, F1 = q1 + q2;
//   f16: on columns 128 .. 191 (the hi products need an accumulator of their
//     own), F0 = q0 + 2^-11 (q3 + c0), F1 = q2 + 2^-11 (q1 + c1).
//
// Input operands.  tf32: 8-channel chunks of a tile of 2 rows x 128 pixels (4 staged rows) in a ring of two
// stages; what is left of shared memory beside the weights holds no more.  f16: whole input rows, all channels, in a
// ring of four; a CTA walks down a strip of 128 columns, so a row is fetched and split once for its three output
// rows (the tiles' four staged rows per two output rows kept the loaders busy twice as long).
//
// Per CTA 24 warps, persistent: warps 10-23 load (a chunk or row is dealt to them in units of 128 pixels of one row
// and K half, plus one unit with the two halo columns past them; a warp fetches its next unit into registers before
// or right after it stores one); warps 8 and 9 of the even CTA issue the MMAs (warp 8 also owns the TMEM): in tf32 an
// output row of the tile each, in f16 a product each (x_hi [w_hi | w_lo], and x_lo w_hi into columns of its own); warps
// 0-7 are the epilogue.  Accumulators are handed over row by row.  Two issuing threads,
// because whatever one thread does between its MMAs (the wait for a stage, ~180 clocks, commits, loop control)
// leaves the tensor pipe idle: with one issuer a tf32 chunk's 36 MMAs took 2740 clocks, 1980 of them in the tensor
// pipe.  Arrivals on the even CTA's barriers have the default scope: what they hand over (operands behind a proxy
// fence, tensor memory) does not need the cluster-scope release, which waits for the thread's global stores.
//
// Measured, 64 -> 64 channels at 720 x 1280 (back to back): tf32 250 -> 219 us, f16 198 -> 143 us against the row-tiled
// kernel; 321 x 481 (rows not 16-byte aligned), tf32, 89 -> 44 us.  tf32 is bound by the tensor pipe (197 us with every
// load, store and epilogue left out: 110 clocks per tap and row, N = 64 MMAs taking 46 where 32 would be their rate);
// f16 by the epilogue and loader instructions beside the MMAs (117-126 us with them left out).  Tried and slower in f16:
// issuers on alternate rows, at once (170) or in turn (155 - 165), one issuer (197), releasing the accumulators before
// the stores (154), polling with test_wait (174), tiles as in tf32 (181).
//
// Streamed weights (tf32).  Layers of at most 64 filters with more input channels, and 128-filter blocks (one output row
// per CTA and tile, one issuer), take each chunk's weights with its input stage: one bulk copy per CTA and chunk, from a
// second copy of the weight tiles in the pairs' row order.  The odd CTA's idle MMA warp reports its copies to the even
// one.  Against the row-tiled kernel, whose 128-filter tile moves ~305 KB of a chunk through shared memory (2380 clocks)
// for 1728 clocks of MMAs, the pair moves ~214 KB: 128 -> 128 at 128 x 128 26.7 -> 23.5 us, 2 x 200 x 200 119 -> 100,
// 256 -> 256 at 120 x 160 150 -> 125; 64 filters: 100 -> 64 at 128 x 128 23.3 -> 19.0, 256 -> 48 at 100 x 130, batch 2
// (rows not 16-byte aligned), 141 -> 70, 512 -> 64 at 28 x 28 94 -> 69.
//
// Every wait on an mbarrier is bounded; on timeout the kernel records an error
// in the layer's device status word and skips the rest of its work.
#include <cuda_runtime.h>

#include <algorithm>

#include "internal.h"
#include "tc_ptx.cuh"

namespace {

using namespace ppc_ptx;

constexpr int NTAP = 9;
constexpr int TW = 128, BCOLS = TW + 2; // output columns of a tile, staged columns
constexpr int NLOADW = 14;              // loader warps (24 warps in all: 80 registers per thread)
constexpr int NEPIW = 8;                // warps 0-7: epilogue
constexpr int MMA_WARP = NEPIW;         // warps 8 and 9: MMA issuers
constexpr int LOAD_WARP0 = MMA_WARP + 2;
constexpr int NTHREADS = 32 * (LOAD_WARP0 + NLOADW);
constexpr long WAIT_LIMIT = PP_WAIT_POLLS;
constexpr int MAX_CI = 64;              // input channels whose weights stay resident (64 filters)
constexpr int KCH32 = 8, KCH16 = 16;    // input channels per chunk

// One instantiation: FB filters (64, or 128 in tf32); STREAM (tf32): each chunk's weights come with its input stage
// instead of staying resident.
template <bool F16, int FB, bool STREAM>
struct Geo {
  static_assert(!F16 || (FB == 64 && !STREAM), "f16: resident weights of 64 filters");
  static_assert(FB == 64 || STREAM, "128 filters' weights do not fit");
  static constexpr int R = FB == 64 ? 2 : 1;           // output rows of a tile (tf32)
  static constexpr int BROWS = R + 2, NPIX = BROWS * BCOLS;
  static constexpr int IN_HALF = NPIX * 16;            // one K half of the hi or lo input operand of a chunk
  static constexpr int IN_BYTES = 2 * IN_HALF;
  static constexpr int W_TAP = FB * 32;                // this CTA's FB weight rows of a tap, 32 bytes (K) each
  static constexpr int W_CHUNK = NTAP * W_TAP;
  static constexpr int UNITS = 2 * BROWS + 1;          // loader units of a chunk: each row and K half, the last 2 columns
  // tf32: chunks in a ring of stages (hi, lo; STREAM: weights first); f16: whole input rows in a ring of four
  static constexpr int ROW_HALF = BCOLS * 16;          // f16: one K half of a row's hi or lo operand in a chunk
  static constexpr int ROW_CHUNK = 4 * ROW_HALF;       // hi (2 halves), lo
  static constexpr int NRING = F16 ? 4 : !STREAM ? 2 : FB == 64 ? 4 : 3;
  static constexpr int ENTRY = F16 ? MAX_CI / KCH16 * ROW_CHUNK : 2 * IN_BYTES + (STREAM ? W_CHUNK : 0);
  static constexpr int X_OFF = STREAM ? W_CHUNK : MAX_CI / (F16 ? KCH16 : KCH32) * W_CHUNK;  // input of entry s at + s ENTRY
  static constexpr int SMEM = (STREAM ? 0 : X_OFF) + NRING * ENTRY + 1024;
  // accumulator slots, one output row each: tf32 of 2 FB columns, f16 of 192 (256 apart)
  static constexpr int NSLOT = F16 ? 2 : 512 / (2 * FB), SLOTC = F16 ? 256 : 2 * FB;
  static_assert(SMEM <= 232448 - 2304, "shared memory plan");
};

struct TcrParams {
  const float* rscale;      // f16: per reordered filter, 1 / (weight scale x input scale)
  float xscale;             // f16: power of two applied to x before the split
  const float* x;
  float* y;
  const float* skip;
  // resident: [nch][9][K half][128 rows][16 bytes], rows 0-63 hi, 64-127 lo; STREAM: [nfb][nch][rank][9][K half][FB rows]
  const unsigned char* wt;
  const int* perm;
  const float* bias;
  int* status;
  int N, Ci, Co, H, W, nch, flags;
  int tiles_x, nstrips;     // 128-column strips of an image row; strips in all
  int tiles_y, ntiles, nfb; // tf32: tiles of R rows; filter blocks
  int split, srows;         // f16: each strip is cut into `split` (1 or 2) pieces of srows rows
};

// f16: the output rows of one CTA pair.  Pieces of strips are numbered image by image, strip by strip, and taken
// two at a time (piece 2 k + rank belongs to the CTA of that rank), so the pieces in a row make npairs x srows
// rows of which every pair of CTAs walks an equal, contiguous range [pos, end).  A run is the part of the range
// within one pair of pieces; its input rows are the output rows and one more on either side.
struct Walk {
  int pos, end;       // first row of the run, end of the range
  int y, len;         // the run: rows y .. y + len - 1 of the piece
  int n, row0, c0;    // this CTA's image, first row of the piece, first column
  bool ok;            // this CTA has a piece here
  __device__ __forceinline__ void range(const TcrParams& p, int unit) {
    const int64_t units = (int64_t)((p.nstrips * p.split + 1) / 2) * (p.srows / unit);
    const int pair = (int)blockIdx.x >> 1, pairs = (int)gridDim.x >> 1;
    pos = (int)(units * pair / pairs) * unit;
    end = (int)(units * (pair + 1) / pairs) * unit;
    len = 0;
  }
  __device__ __forceinline__ bool run(const TcrParams& p, int rank) {  // the next run; false at the end
    pos += len;
    if (pos >= end) return false;
    const int k = pos / p.srows;
    y = pos - k * p.srows;
    len = min(p.srows - y, end - pos);
    int piece = 2 * k + rank;
    ok = piece < p.nstrips * p.split;
    row0 = p.split == 2 && (piece & 1) ? p.srows : 0;
    if (p.split == 2) piece >>= 1;
    n = ok ? piece / p.tiles_x : 0;
    c0 = (piece % p.tiles_x) * TW;
    return true;
  }
};

template <bool F16, bool POOL, int FB, bool STREAM>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(NTHREADS, 1) ppconv_tcr_kernel(const TcrParams p) {
  using G = Geo<F16, FB, STREAM>;
  static_assert(!POOL || G::R == 2, "pooling reads row pairs of a tile");
  constexpr int R = G::R, NSLOT = G::NSLOT, SLOTC = G::SLOTC, NRING = G::NRING, X_OFF = G::X_OFF, ENTRY = G::ENTRY;
  constexpr int NPIX = G::NPIX, IN_HALF = G::IN_HALF, IN_BYTES = G::IN_BYTES, UNITS = G::UNITS;
  constexpr int W_TAP = G::W_TAP, W_CHUNK = G::W_CHUNK, ROW_HALF = G::ROW_HALF, ROW_CHUNK = G::ROW_CHUNK;
  constexpr int NISS = F16 ? 2 : R;  // MMA issuers
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* smem = smem_raw + ((1024u - (su32(smem_raw) & 1023u)) & 1023u);
  // full (even CTA): both CTAs' loader warps have stored a ring entry; empty (tf32): the MMAs that read it are
  // complete; acc_full: a slot's row is accumulated (f16: and with it every earlier MMA is complete, which is what the
  // loaders wait for too); acc_empty (even CTA): both CTAs' epilogues have read it
  __shared__ __align__(8) uint64_t full[NRING], empty[NRING], acc_full[NSLOT], acc_empty[NSLOT], done_bar;
  __shared__ __align__(8) uint64_t wfull[NRING];  // STREAM, odd CTA: its weights of a stage have landed
  __shared__ volatile int wuse[NRING];            // STREAM: last use of a stage for which this CTA's copy was issued, or -1
  __shared__ uint32_t tmem_s;
  // per filter: output channel x plane size of y and of skip (0 past the last filter), bias, inverse scale
  // (64 filters; 128-filter layers may have several blocks and read them from memory)
  __shared__ __align__(16) int yoff[64], soff[64];
  __shared__ __align__(16) float bias_s[64], scale_s[64];
  __shared__ volatile int abort_s;

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t rank = cluster_rank();

  // Bounded wait that gives up early once another role has aborted.
  auto wait = [&](uint64_t* bar, uint32_t parity) -> bool {
    const uint32_t a = su32(bar);
    for (long i = 0; i < WAIT_LIMIT; ++i) {
      if (mbar_try(a, parity)) return true;
      if ((i & 255) == 255 && abort_s) return false;
    }
    abort_s = 1;
    atomicOr(p.status, ppc::kStatusTimeout);
    return false;
  };

  const int units = F16 ? 2 * p.nch + 1 : UNITS;  // loader units of a ring entry
  if (tid == 0) {
    for (int s = 0; s < NRING; ++s) {
      // STREAM: and one more for each CTA's weights (the even CTA's with its bytes)
      mbar_init(su32(&full[s]), 2 * units + (STREAM ? 2 : 0));
      mbar_init(su32(&empty[s]), NISS);
      mbar_init(su32(&wfull[s]), 1);
      wuse[s] = -1;
    }
    for (int s = 0; s < NSLOT; ++s) {
      mbar_init(su32(&acc_full[s]), F16 ? 2 : 1);
      mbar_init(su32(&acc_empty[s]), 2 * NEPIW);
    }
    mbar_init(su32(&done_bar), NISS);
    abort_s = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == MMA_WARP) {  // both CTAs of the pair allocate together
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(su32(&tmem_s)), "n"(512));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;");
  }
  if (FB == 64 && tid < FB) {
    const int o = tid < p.Co ? __ldg(p.perm + tid) : 0;
    yoff[tid] = o * (POOL ? (p.H / 2) * (p.W / 2) : p.H * p.W);
    soff[tid] = o * (p.H * p.W);
    bias_s[tid] = tid < p.Co && p.bias ? __ldg(p.bias + tid) : 0.f;
    scale_s[tid] = F16 ? __ldg(p.rscale + tid) : 1.f;
  }
  // This CTA's half of the weights (they do not depend on the previous kernel in the stream):
  // even CTA rows hi 0-31, lo 32-63; odd CTA rows hi 32-63, lo 0-31 of every tap.
  for (int i = tid; !STREAM && i < p.nch * NTAP * 128; i += NTHREADS) {
    const int r = i & 63, src = rank == 0 ? (r < 32 ? r : 64 + r) : 32 + r;
    reinterpret_cast<uint4*>(smem)[i] = __ldg(reinterpret_cast<const uint4*>(p.wt) + (i >> 6) * 128 + src);
  }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  tm_fence_before();
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
  tm_fence_after();
  const uint32_t tmem = tmem_s;

  // tf32: work item i of a pair is item u = pair + i pairs, the filter block u % nfb of the neighbouring tiles 2 v and 2 v
  // + 1, v = u / nfb; a tile past the last is loaded as zeros and not stored.
  const int pair = (int)blockIdx.x >> 1, npairs = (int)gridDim.x >> 1;
  const int items = (p.ntiles + 1) / 2 * p.nfb;
  const int nmine = items > pair ? (items - 1 - pair) / npairs + 1 : 0;
  auto tile_of = [&](int i, int& n, int& r0, int& c0, int& fb) -> bool {
    const int u = pair + i * npairs;
    fb = FB == 64 ? 0 : u % p.nfb;
    int t = 2 * (FB == 64 ? u : u / p.nfb) + (int)rank;
    if (t >= p.ntiles) return false;
    c0 = (t % p.tiles_x) * TW;
    t /= p.tiles_x;
    r0 = (t % p.tiles_y) * R;
    n = t / p.tiles_y;
    return true;
  };

  if (warp >= LOAD_WARP0) {
    // ------------------------------------------------------------ loaders
    const int HW = p.H * p.W;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    // v[j][k]: channel ch + k of pixel col + 32 j of a row (one: a single pixel per lane, v[0])
    auto fetch = [&](auto& v, int n, int ch, int row, int col, bool in, bool one) {
      constexpr int CPH = (int)(sizeof(v[0]) / 4);
      const bool rin = in && (unsigned)row < (unsigned)p.H;
      const float* src = p.x + ((size_t)n * p.Ci + ch) * HW + (row * p.W + col);
      if (__all_sync(0xffffffffu, rin && !one && col >= 0 && col + 96 < p.W && ch + CPH <= p.Ci)) {
#pragma unroll
        for (int k = 0; k < CPH; ++k) {
#pragma unroll
          for (int j = 0; j < 4; ++j) v[j][k] = __ldg(src + 32 * j);
          src += HW;
        }
        return;
      }
#pragma unroll
      for (int k = 0; k < CPH; ++k) {
        const bool kin = rin && ch + k < p.Ci;
#pragma unroll
        for (int j = 0; j < 4; ++j)
          v[j][k] = kin && (j == 0 || !one) && (unsigned)(col + 32 * j) < (unsigned)p.W ? __ldg(src + 32 * j) : 0.f;
        src += HW;
      }
    };
    // h and l of the four pixels to shared memory at dst (lo `lo` units further), then the unit is reported
    auto store = [&](uint4* dst, int lo, const uint4(&h)[4], const uint4(&l)[4], bool in, bool one, uint64_t* bar) {
      if (in) {
        dst[0] = h[0];
        dst[lo] = l[0];
      }
      if (!one) {
#pragma unroll
        for (int j = 1; j < 4; ++j) {
          dst[32 * j] = h[j];
          dst[32 * j + lo] = l[j];
        }
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive_pair(map_rank(su32(bar), 0));
    };
    if constexpr (F16) {
      __half2 hmax = __floats2half2_rn(0.f, 0.f);  // largest |x| after scaling: infinite or NaN out of fp16's range
      // A warp never skips two ring entries: it then knows, from its previous wait, that the phase before the one it
      // waits for is complete (a parity wait cannot tell a phase from the one two before it).
      const int nload = min(NLOADW, 2 * units);
      Walk w;
      w.range(p, POOL ? 2 : 1);
      bool more = warp - LOAD_WARP0 < nload && w.run(p, (int)rank);
      // ring entry sq (the k-th input row of the run), unit un of it: un < 2 nch is chunk un >> 1, K half un & 1 and
      // pixels 32 j + lane; the last holds pixels 128 and 129 (lane l: chunk l >> 2, K half (l >> 1) & 1, pixel l & 1)
      int un = warp - LOAD_WARP0, k = 0, sq = 0;
      // Input row k of a run is last read for its output row min(k, len - 1).  last[0]: the output row (counted over
      // all runs) after which the ring entry of row sq may be stored again, i.e. the last to read entry sq - NRING.
      int oc0 = 0, last[NRING] = {0, 0, 0, 0};
      auto settle = [&]() {
        while (more && un >= units) {
          un -= units;
          ++sq;
#pragma unroll
          for (int r = 0; r + 1 < NRING; ++r) last[r] = last[r + 1];
          last[NRING - 1] = oc0 + min(k, w.len - 1);
          if (++k == w.len + 2) {
            k = 0;
            oc0 += w.len;
            more = w.run(p, (int)rank);
          }
        }
      };
      settle();
      float v[4][8];
      auto load = [&]() {
        const bool one = un == units - 1;
        const int ch = one ? (lane >> 2) * 16 + ((lane >> 1) & 1) * 8 : un * 8;
        fetch(v, w.n, ch, w.row0 + w.y - 1 + k, w.c0 - 1 + (one ? 128 + (lane & 1) : lane), w.ok && (!one || lane < 4 * p.nch), one);
      };
      if (more) load();
      while (more) {
        uint4 h[4], l[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) split_f16x8_max(v[j], p.xscale, h[j], l[j], hmax);
        const int s = sq % NRING;
        const bool one = un == units - 1, in = !one || lane < 4 * p.nch;
        const int off = one ? (lane >> 2) * ROW_CHUNK + ((lane >> 1) & 1) * ROW_HALF + (128 + (lane & 1)) * 16
                            : (un >> 1) * ROW_CHUNK + (un & 1) * ROW_HALF + lane * 16;
        uint4* dst = reinterpret_cast<uint4*>(smem + X_OFF + s * ENTRY + (in ? off : 0));
        if (!__all_sync(0xffffffffu, sq < NRING || wait(&acc_full[last[0] & 1], (uint32_t)((last[0] >> 1) & 1)))) break;
        store(dst, 2 * ROW_HALF / 16, h, l, in, one, &full[s]);
        un += nload;
        settle();
        if (more) load();
      }
      if (f16_max_bad(hmax)) atomicOr(p.status, ppc::kStatusF16Range);
    } else {
      // (NLOADW < 2 UNITS: no warp skips two stages' entries, see above)
      static_assert(NLOADW <= 2 * UNITS, "a parity wait needs the phase before");
      // tile it, chunk c, unit un of the chunk in stage s: un < 2 BROWS is row un >> 1, K half un & 1 and pixels 32 j +
      // lane; the last holds pixels 128 and 129 (lane l: row l >> 2, K half (l >> 1) & 1, pixel l & 1)
      int it = 0, c = 0, un = warp - LOAD_WARP0, s = 0, use = 0, n = 0, r0 = 0, c0 = 0, fb = 0;
      bool ok = tile_of(0, n, r0, c0, fb);
      auto settle = [&]() {
        bool moved = false;
        while (un >= UNITS) {
          un -= UNITS;
          if (++s == NRING) {
            s = 0;
            ++use;
          }
          if (++c == p.nch) {
            c = 0;
            ++it;
            moved = true;
          }
        }
        if (moved) ok = tile_of(it, n, r0, c0, fb);
      };
      settle();
      float v[4][4];
      auto load = [&]() {
        const bool one = un == UNITS - 1;
        fetch(v, n, c * KCH32 + (one ? (lane >> 1) & 1 : un & 1) * 4, r0 - 1 + (one ? lane >> 2 : un >> 1),
              c0 - 1 + (one ? 128 + (lane & 1) : lane), ok && (!one || lane < 4 * G::BROWS), one);
      };
      if (it < nmine) load();
      while (it < nmine) {
        // split, and the next unit's loads, while the stage is still being read: only the stores wait for it
        uint4 h[4], l[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          h[j] = make_uint4(__float_as_uint(tf32_hi(v[j][0])), __float_as_uint(tf32_hi(v[j][1])),
                            __float_as_uint(tf32_hi(v[j][2])), __float_as_uint(tf32_hi(v[j][3])));
          l[j] = make_uint4(__float_as_uint(v[j][0] - __uint_as_float(h[j].x)),
                            __float_as_uint(v[j][1] - __uint_as_float(h[j].y)),
                            __float_as_uint(v[j][2] - __uint_as_float(h[j].z)),
                            __float_as_uint(v[j][3] - __uint_as_float(h[j].w)));
        }
        const int su = s, uu = use;
        const bool one = un == UNITS - 1, in = !one || lane < 4 * G::BROWS, head = un == 0;
        const unsigned char* wsrc = p.wt + ((size_t)(fb * p.nch + c) * 2 + rank) * W_CHUNK;
        uint4* dst = reinterpret_cast<uint4*>(smem + X_OFF + s * ENTRY) +
                     (one ? (in ? ((lane >> 1) & 1) * NPIX + (lane >> 2) * BCOLS + 128 + (lane & 1) : 0)
                          : (un & 1) * NPIX + (un >> 1) * BCOLS + lane);
        un += NLOADW;
        settle();
        if (it < nmine) load();
        if (!__all_sync(0xffffffffu, uu == 0 || wait(&empty[su], (uint32_t)((uu - 1) & 1)))) break;
        if (STREAM && head && lane == 0) {  // the warp with a stage's first unit copies its weights
          uint64_t* bar = rank == 0 ? &full[su] : &wfull[su];
          wuse[su] = uu;
          mbar_arrive_expect_tx(su32(bar), W_CHUNK);
          asm volatile(
              "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                  su32(smem + su * ENTRY)),
              "l"(wsrc), "r"(W_CHUNK), "r"(su32(bar))
              : "memory");
        }
        store(dst, IN_BYTES / 16, h, l, in, one, &full[su]);
      }
    }
    __syncwarp();
  } else if (warp >= MMA_WARP) {
    // ------------------------------------------------------------ MMA issuers (even CTA, for the pair)
    if (lane == 0 && rank == 0 && warp - MMA_WARP < NISS) {
      constexpr uint32_t ID1 = F16 ? idesc_f16(256, 2 * FB) : idesc_tf32(256, 2 * FB);
      constexpr uint32_t ID2 = F16 ? idesc_f16(256, FB) : idesc_tf32(256, FB);
      const int rr = warp - MMA_WARP;  // which issuer
      const uint32_t x_base = su32(smem) + X_OFF;
      if constexpr (F16) {
        // Issuer 0: x_hi [w_hi | w_lo]; issuer 1: x_lo w_hi, into columns of its own.
        const uint32_t id = rr == 0 ? ID1 : ID2;
        Walk w;
        w.range(p, POOL ? 2 : 1);
        int oc = 0, sq = 0;  // output rows so far, ring entry of the run's first input row
        bool ok = true;
        while (ok && w.run(p, 0)) {
          for (int y = 0; y < w.len && ok; ++y, ++oc) {
            const int slot = oc & 1;
            if (oc >= 2) ok = wait(&acc_empty[slot], (uint32_t)(((oc >> 1) - 1) & 1));
            const uint32_t d = tmem + (uint32_t)(slot * SLOTC + rr * 128);
            uint64_t xd[3], wd = smem_desc(su32(smem), FB * 16);
#pragma unroll
            for (int r = 0; r < 3; ++r) {  // the input rows' ring entries; the run's previous row waited for the first two
              const int q = sq + y + r;
              if (ok && (r == 2 || y == 0)) ok = wait(&full[q % NRING], (uint32_t)((q / NRING) & 1));
              xd[r] = smem_desc(x_base + (uint32_t)((q % NRING) * ENTRY + rr * 2 * ROW_HALF), ROW_HALF);
            }
            if (!ok) break;
            tm_fence_after();
            for (int c = 0; c < p.nch; ++c) {
#pragma unroll
              for (int t = 0; t < NTAP; ++t)  // pixels of 16 bytes
                mma_f16_pair(d, xd[t / 3] + (uint64_t)(t % 3), wd + (uint64_t)(t * W_TAP / 16), id,
                             t == 0 && c == 0 ? 0u : 1u);
              wd += W_CHUNK / 16;
#pragma unroll
              for (int r = 0; r < 3; ++r) xd[r] += ROW_CHUNK / 16;
            }
            mma_commit_pair(su32(&acc_full[slot]), (uint16_t)3);
          }
          sq += w.len + 2;
        }
      } else {
        // issuer rr: row rr of every tile
        int s = 0, ph = 0, slot = rr, sph = 0;
        bool ok = true;
        for (int i = 0; i < nmine && ok; ++i) {
          if (i >= NSLOT / R) ok = wait(&acc_empty[slot], (uint32_t)(sph ^ 1));
          const uint32_t d = tmem + (uint32_t)(slot * SLOTC);
          uint64_t w0 = smem_desc(su32(smem), FB * 16);
          for (int c = 0; c < p.nch && ok; ++c, w0 += STREAM ? 0 : W_CHUNK / 16) {
            ok = wait(&full[s], (uint32_t)ph);
            if (!ok) break;
            tm_fence_after();
            const uint64_t xh0 = smem_desc(x_base + (uint32_t)(s * ENTRY), IN_HALF) + (uint64_t)(rr * BCOLS);
            const uint64_t ws = w0 + (uint64_t)(STREAM ? s * (ENTRY / 16) : 0);
            const uint32_t acc0 = c == 0 ? 0u : 1u;
#pragma unroll
            for (int t = 0; t < NTAP; ++t) {
              const uint64_t xh = xh0 + (uint64_t)((t / 3) * BCOLS + t % 3);  // pixels of 16 bytes
              const uint64_t w = ws + (uint64_t)(t * W_TAP / 16);
              mma_tf32_pair(d, xh, w, ID1, t == 0 ? acc0 : 1u);
              mma_tf32_pair(d, xh + IN_BYTES / 16, w, ID2, 1u);
            }
            mma_commit_pair(su32(&empty[s]), (uint16_t)3);
            if (++s == NRING) {
              s = 0;
              ph ^= 1;
            }
          }
          if (!ok) break;
          mma_commit_pair(su32(&acc_full[slot]), (uint16_t)3);
          slot += R;
          if (slot >= NSLOT) {
            slot = rr;
            sph ^= 1;
          }
        }
      }
      // the next kernel in the stream may start its prologue (it waits for this
      // grid to complete before it reads anything this grid writes)
      asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
      mma_commit_pair(su32(&done_bar), (uint16_t)1);
      wait(&done_bar, 0u);
    } else if (lane == 0 && rank == 1 && warp == MMA_WARP) {
      if (STREAM) {  // reports the odd CTA's weights of each chunk to the even one
        int s = 0, ph = 0;
        for (int g = 0; g < nmine * p.nch; ++g) {
          if (!wait(&wfull[s], (uint32_t)ph)) break;
          mbar_arrive_remote(map_rank(su32(&full[s]), 0));
          if (++s == NRING) {
            s = 0;
            ph ^= 1;
          }
        }
      }
      asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    }
    __syncwarp();
  } else {
    // ------------------------------------------------------------ epilogue
    // lane = pixel 32 q + lane of the row; this warp's filters: F0 (half 0) or F1 (half 1)
    const int q = warp & 3, half = warp >> 2;
    const bool relu = p.flags & PP_RELU;
    constexpr int EB = POOL ? 8 : 16;  // filters handled together (pooling holds two rows of them)
    constexpr int Q = FB / 2;     // filters of a half, columns of a quarter
    const int f0 = Q * half;      // first filter of this half
    int fbase = 0, nf = p.Co - f0;  // the block's first filter; how many filters from f0 on exist
    const int HW = p.H * p.W, Wo = p.W / 2, HWo = (p.H / 2) * Wo;
    const uint32_t lanebase = tmem + ((uint32_t)(32 * q) << 16);
    // bias and output channel x plane of filters f0 + j .. + 3 (past the last filter: anything)
    auto bias4 = [&](int j) -> float4 {
      if (FB == 64) return *reinterpret_cast<const float4*>(&bias_s[f0 + j]);
      return p.bias && j < nf ? __ldg(reinterpret_cast<const float4*>(p.bias + fbase + f0 + j)) : make_float4(0.f, 0.f, 0.f, 0.f);
    };
    auto plane4 = [&](int j, bool y) -> int4 {
      if (FB == 64) return *reinterpret_cast<const int4*>(y ? &yoff[f0 + j] : &soff[f0 + j]);
      const int4 o = j < nf ? __ldg(reinterpret_cast<const int4*>(p.perm + fbase + f0 + j)) : make_int4(0, 0, 0, 0);
      // a vector's entries past the last filter are padding, not channels
      return make_int4(o.x * HW, j + 1 < nf ? o.y * HW : 0, j + 2 < nf ? o.z * HW : 0, j + 3 < nf ? o.w * HW : 0);
    };
    // filters f0 + jj .. + EB - 1, with their bias, from a slot's accumulators (warp-collective)
    auto get = [&](int slot, int jj, float(&a)[EB]) {
      const uint32_t b = lanebase + (uint32_t)(slot * SLOTC + jj);
      float a2[EB];
      tm_ld(b + (half ? 2 * Q : 0), a);
      tm_ld(b + (half ? Q : 3 * Q), a2);
      if constexpr (F16) {
        const uint64_t e = pack2(0x1p-11f, 0x1p-11f);
        float a3[EB];
        tm_ld(b + (half ? 160 : 128), a3);
        tm_wait_ld();
#pragma unroll
        for (int k = 0; k < EB; k += 4) {
          const float4 bv = *reinterpret_cast<const float4*>(&bias_s[f0 + jj + k]);
          const float4 rv = *reinterpret_cast<const float4*>(&scale_s[f0 + jj + k]);
          const uint64_t u0 = fma2(add2(pack2(a2[k], a2[k + 1]), pack2(a3[k], a3[k + 1])), e, pack2(a[k], a[k + 1]));
          const uint64_t u1 =
              fma2(add2(pack2(a2[k + 2], a2[k + 3]), pack2(a3[k + 2], a3[k + 3])), e, pack2(a[k + 2], a[k + 3]));
          unpack2(fma2(u0, pack2(rv.x, rv.y), pack2(bv.x, bv.y)), a[k], a[k + 1]);
          unpack2(fma2(u1, pack2(rv.z, rv.w), pack2(bv.z, bv.w)), a[k + 2], a[k + 3]);
        }
      } else {
        tm_wait_ld();
#pragma unroll
        for (int k = 0; k < EB; k += 4) {
          const float4 bv = bias4(jj + k);
          unpack2(add2(add2(pack2(a[k], a[k + 1]), pack2(a2[k], a2[k + 1])), pack2(bv.x, bv.y)), a[k], a[k + 1]);
          unpack2(add2(add2(pack2(a[k + 2], a[k + 3]), pack2(a2[k + 2], a2[k + 3])), pack2(bv.z, bv.w)), a[k + 2],
                  a[k + 3]);
        }
      }
    };
    // The r-th output row of this CTA (pooled: rows r and r + 1), row `row` of image n from column c0 on; valid: it
    // is stored.  False after a wait that gave up.
    auto emit = [&](int r, int n, int row, int c0, bool valid) -> bool {
      const int s0 = r % NSLOT, s1 = (r + 1) % NSLOT;
      const int col = c0 + 32 * q + lane;
      const bool in0 = valid && row < p.H && col < p.W;
      const int roff = row * p.W + col, poff = (row >> 1) * Wo + (col >> 1);
      const size_t nco = (size_t)n * p.Co;
      float* ybase = p.y + nco * (size_t)(POOL ? HWo : HW) + (POOL ? poff : roff);
      const float* sbase = (p.flags & PP_ADD_SKIP) ? p.skip + nco * (size_t)HW : nullptr;
      bool ok = wait(&acc_full[s0], (uint32_t)((r / NSLOT) & 1)) &&
                (!POOL || wait(&acc_full[s1], (uint32_t)(((r + 1) / NSLOT) & 1)));
      if (!__all_sync(0xffffffffu, ok)) return false;  // the whole warp leaves together
      tm_fence_after();
      auto release = [&]() {  // everything this warp needs of the slots is in registers
        tm_fence_before();
        __syncwarp();
        if (lane == 0) {
          mbar_arrive_pair(map_rank(su32(&acc_empty[s0]), 0));
          if (POOL) mbar_arrive_pair(map_rank(su32(&acc_empty[s1]), 0));
        }
      };
      // EB filters from f0 + jj on: residual, ReLU, pooling, stores
      auto finish = [&](int jj, float(&a)[EB], float* bb) {
        // residual: loads of their own before the stores, unconditional (lanes without an output
        // read the image's first element), so their latencies overlap
        if (sbase) {
#pragma unroll
          for (int k0 = 0; k0 < EB; k0 += 8) {
            const int4 so[2] = {plane4(jj + k0, false), plane4(jj + k0 + 4, false)};
            float sv[8], tv[POOL ? 8 : 1];
#pragma unroll
            for (int k = 0; k < 8; ++k) {
              const int o = (k & 3) == 0 ? so[k >> 2].x : (k & 3) == 1 ? so[k >> 2].y : (k & 3) == 2 ? so[k >> 2].z : so[k >> 2].w;
              sv[k] = __ldg(sbase + (in0 ? o + roff : 0));
              if constexpr (POOL) tv[k] = __ldg(sbase + (in0 ? o + roff + p.W : 0));
            }
#pragma unroll
            for (int k = 0; k < 8; ++k) {
              a[k0 + k] += sv[k];
              if constexpr (POOL) bb[k0 + k] += tv[k];
            }
          }
        }
        if (relu) {
#pragma unroll
          for (int k = 0; k < EB; ++k) {
            a[k] = fmaxf(a[k], 0.f);
            if constexpr (POOL) bb[k] = fmaxf(bb[k], 0.f);
          }
        }
#pragma unroll
        for (int k = 0; k < EB; k += 4) {
          const int4 o4 = plane4(jj + k, true);
          const int o[4] = {o4.x, o4.y, o4.z, o4.w};
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            if constexpr (!POOL) {
              if (in0 && jj + k + e < nf) ybase[o[e]] = a[k + e];
            } else {
              const float m = fmaxf(a[k + e], bb[k + e]);
              const float m2 = __shfl_down_sync(0xffffffffu, m, 1);
              if (((col & 1) == 0) && in0 && jj + k + e < nf) ybase[o[e]] = fmaxf(m, m2);
            }
          }
        }
      };
#pragma unroll(POOL ? 1 : 2)
      for (int jj = 0; jj < Q; jj += EB) {
        float a[EB], bb[POOL ? EB : 1];
        get(s0, jj, a);
        if constexpr (POOL) get(s1, jj, bb);
        if (jj == Q - EB) release();
        finish(jj, a, bb);
      }
      return true;
    };
    constexpr int STEP = POOL ? 2 : 1;
    bool ok = true;
    if constexpr (F16) {
      Walk w;
      w.range(p, STEP);
      int r = 0;
      while (ok && w.run(p, (int)rank))
        for (int y = 0; y < w.len && ok; y += STEP, r += STEP) ok = emit(r, w.n, w.row0 + w.y + y, w.c0, w.ok);
    } else {
      for (int i = 0; i < nmine && ok; ++i) {
        int n = 0, r0 = 0, c0 = 0, fb = 0;
        const bool valid = tile_of(i, n, r0, c0, fb);
        if (FB == 128) {
          fbase = fb * FB;
          nf = p.Co - fbase - f0;
        }
        for (int rr = 0; rr < R && ok; rr += STEP) ok = emit(i * R + rr, n, r0 + rr, c0, valid);
      }
    }
  }

  // neither CTA leaves (or frees its TMEM) while the pair's MMAs or arrivals may still reach it
  tm_fence_before();
  __syncwarp();
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
  tm_fence_after();
  if (warp == MMA_WARP)
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "n"(512));
  // After a wait that gave up, this CTA's weight copies may still be in flight: none may write shared memory once the
  // CTA has exited.  No more are issued (every loader has passed the barrier above); wait, bounded, for the last into
  // each stage.  (The even CTA's stage barriers may lack loader arrivals and never complete; the bounded wait then
  // outlasts any copy.)
  if (STREAM && abort_s && tid == 0) {
    long polls = 0;
    for (int s = 0; s < NRING; ++s)
      while (wuse[s] >= 0 && polls < WAIT_LIMIT && !mbar_try(su32(rank == 0 ? &full[s] : &wfull[s]), (uint32_t)(wuse[s] & 1)))
        ++polls;
  }
}

// Pairs that fit on the current device at once, per instantiation (0: pairs cannot be launched).
enum { K_TF32, K_TF32_POOL, K_F16, K_F16_POOL, K_STREAM64, K_STREAM64_POOL, K_STREAM128, K_COUNT };
int g_pairs[ppc::DeviceOnce::kMaxDevices][K_COUNT];
ppc::DeviceOnce g_once;

template <bool F16, bool POOL, int FB, bool STREAM>
cudaError_t setup(int dev, int k) {
  constexpr int SMEM = Geo<F16, FB, STREAM>::SMEM;
  const auto kernel = ppconv_tcr_kernel<F16, POOL, FB, STREAM>;
  const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = 2;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.gridDim = dim3(2);
  cfg.blockDim = dim3(NTHREADS);
  cfg.dynamicSmemBytes = SMEM;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) != cudaSuccess) {
    cudaGetLastError();
    n = 0;
  }
  g_pairs[dev][k] = n;
  return cudaSuccess;
}

cudaError_t prepare() {
  return g_once.run([](int dev) {
    cudaError_t e;
    if ((e = setup<false, false, 64, false>(dev, K_TF32)) != cudaSuccess) return e;
    if ((e = setup<false, true, 64, false>(dev, K_TF32_POOL)) != cudaSuccess) return e;
    if ((e = setup<true, false, 64, false>(dev, K_F16)) != cudaSuccess) return e;
    if ((e = setup<true, true, 64, false>(dev, K_F16_POOL)) != cudaSuccess) return e;
    if ((e = setup<false, false, 64, true>(dev, K_STREAM64)) != cudaSuccess) return e;
    if ((e = setup<false, true, 64, true>(dev, K_STREAM64_POOL)) != cudaSuccess) return e;
    return setup<false, false, 128, true>(dev, K_STREAM128);
  });
}

template <bool F16, bool POOL, int FB, bool STREAM>
cudaError_t launch(const TcrParams& p, int pairs, cudaStream_t stream) {
  cudaLaunchConfig_t cfg = {};
  // tf32: pairs of tiles and filter blocks; f16: pairs of strip pieces, row by row (pooled: row pair by row pair)
  const int64_t work = F16 ? (int64_t)((p.nstrips * p.split + 1) / 2) * (p.srows / (POOL ? 2 : 1))
                           : (int64_t)((p.ntiles + 1) / 2) * p.nfb;
  // No more pairs than the busiest one's share calls for, and in f16 at least two rows each (a row alone fetches three):
  // the SMs left over run what else is in flight (f16, three networks on streams of their own, a frame: 8 layers of 64
  // channels at 205 x 59 95 -> 75 us, 7 at 54 x 220 56 -> 39; alone a layer takes 12.8 -> 12.0 and 10.0 -> 11.0, the
  // row-tiled kernel 18.1 and 14.4).
  const int64_t share = std::max<int64_t>((work + pairs - 1) / pairs, F16 && !POOL ? 2 : 1);
  cfg.gridDim = dim3((unsigned)(2 * ((work + share - 1) / share)));
  cfg.blockDim = dim3(NTHREADS);
  cfg.dynamicSmemBytes = Geo<F16, FB, STREAM>::SMEM;
  cfg.stream = stream;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, ppconv_tcr_kernel<F16, POOL, FB, STREAM>, p);
}

// The tf32 weight tiles in the order that the pairs stream them: block (filter block, chunk, rank) of [9][K half][FB
// rows][16 bytes], rank 0 the rows [w_hi F0 ; w_lo F1], rank 1 [w_hi F1 ; w_lo F0] (F0 / F1: first / last FB / 2 filters).
__global__ void pair_layout_kernel(const uint4* a, uint4* ap, int64_t n, int FB) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const int r = (int)(i % FB);
    int64_t t = i / FB;
    const int th = (int)(t % (2 * NTAP));  // tap and K half
    t /= 2 * NTAP;
    const int rank = (int)(t & 1);
    const int src = rank == 0 ? (r < FB / 2 ? r : FB + r) : (r < FB / 2 ? FB / 2 + r : FB / 2 + r);
    ap[i] = a[((t >> 1) * (2 * NTAP) + th) * (2 * FB) + src];
  }
}

}  // namespace

namespace ppc {

// Every map wider than the flattened-row tiles take (62), where it measured 1.2 to 2 times as fast from one tile up to
// 720 x 1280.  Narrow maps leave half and more of its 128-pixel tiles empty and still win while every CTA has at most
// one tile (64 -> 64, tf32 / f16: 8 x 28 x 28, 112 tiles, 18.1 -> 15.2 / 14.3 -> 13.0 us; 8 x 40 x 40, 160 tiles,
// 17.5 -> 21.6 / 14.2 -> 15.7 us).
bool tcr_applicable(const TcLayout& T, int Ci, int N, int H, bool narrow) {
  if (T.FB == 128) return !T.f16 && T.ap && !narrow;
  if (Ci > MAX_CI && (T.f16 || !T.ap)) return false;
  return !narrow || (int64_t)N * ((H + 1) / 2) <= device_sms();
}

bool tcr_streams(const TcLayout& T, int Ci) { return T.FB == 128 || Ci > MAX_CI; }

pp_status tcr_pair_layout(TcLayout* T, cudaStream_t stream) {
  if (T->ap) return PP_OK;
  const int64_t bytes = (int64_t)T->nfb * T->nch * 2 * NTAP * 2 * T->FB * 16;
  void* d = nullptr;
  if (cudaMalloc(&d, (size_t)bytes) != cudaSuccess) {
    cudaGetLastError();
    return PP_ERR_OOM;
  }
  const int64_t n = bytes / 16;
  pair_layout_kernel<<<(unsigned)std::min<int64_t>((n + 255) / 256, 4096), 256, 0, stream>>>(
      reinterpret_cast<const uint4*>(T->a), static_cast<uint4*>(d), n, T->FB);
  if (cudaGetLastError() != cudaSuccess || cudaStreamSynchronize(stream) != cudaSuccess) {
    cudaFree(d);
    return PP_ERR_CUDA;
  }
  T->ap = static_cast<unsigned char*>(d);
  T->dbytesp = (size_t)bytes;
  return PP_OK;
}

void tcr_pair_free(TcLayout* T) {
  if (T->ap) cudaFree(T->ap);
  T->ap = nullptr;
  T->dbytesp = 0;
}

pp_status tcr_launch(const TcLayout& T, const LayerMeta& M, const float* x, float* y, const float* skip, int N, int H,
                     int W, int flags, cudaStream_t stream) {
  if (prepare() != cudaSuccess) return PP_ERR_CUDA;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return PP_ERR_CUDA;
  const bool f16 = T.f16;
  const bool pool = flags & PP_POOL2;
  const bool streams = tcr_streams(T, M.Ci);
  if (streams && (f16 || !T.ap || (pool && T.FB == 128))) return PP_ERR_UNSUPPORTED;
  const int k = f16 ? (pool ? K_F16_POOL : K_F16)
                    : T.FB == 128 ? K_STREAM128
                                  : streams ? (pool ? K_STREAM64_POOL : K_STREAM64) : (pool ? K_TF32_POOL : K_TF32);
  const int pairs = g_pairs[dev][k];
  const int R = T.FB == 128 ? 1 : 2;
  TcrParams p;
  p.rscale = T.rscale;
  p.xscale = T.xscale;
  p.x = x;
  p.y = y;
  p.skip = (flags & PP_ADD_SKIP) ? skip : nullptr;
  p.wt = streams ? T.ap : f16 ? T.a16 : T.a;
  p.perm = M.perm;
  p.bias = M.bias;
  p.status = T.status;
  p.N = N;
  p.Ci = M.Ci;
  p.Co = M.Co;
  p.H = H;
  p.W = W;
  p.nch = f16 ? T.nch16 : T.nch;
  p.flags = flags;
  p.tiles_x = (W + TW - 1) / TW;
  p.tiles_y = (H + R - 1) / R;
  const int64_t ns = (int64_t)p.tiles_x * N, nt = ns * p.tiles_y;
  if (pairs <= 0 || ns * (H + 2) * T.nfb > INT32_MAX / 2) return PP_ERR_UNSUPPORTED;
  p.nfb = T.nfb;
  p.ntiles = (int)nt;
  p.nstrips = (int)ns;
  // an odd number of strips is cut at half height, so that every pair of CTAs has two pieces
  p.split = ns & 1 ? 2 : 1;
  p.srows = p.split == 2 ? (pool ? (H / 2 + 1) / 2 * 2 : (H + 1) / 2) : H;
  cudaError_t e;
  switch (k) {
    case K_TF32: e = launch<false, false, 64, false>(p, pairs, stream); break;
    case K_TF32_POOL: e = launch<false, true, 64, false>(p, pairs, stream); break;
    case K_F16: e = launch<true, false, 64, false>(p, pairs, stream); break;
    case K_F16_POOL: e = launch<true, true, 64, false>(p, pairs, stream); break;
    case K_STREAM64: e = launch<false, false, 64, true>(p, pairs, stream); break;
    case K_STREAM64_POOL: e = launch<false, true, 64, true>(p, pairs, stream); break;
    default: e = launch<false, false, 128, true>(p, pairs, stream); break;
  }
  if (e != cudaSuccess) {
    cudaGetLastError();
    return PP_ERR_CUDA;
  }
  return PP_OK;
}

pp_status tcr_prepare() { return prepare() == cudaSuccess ? PP_OK : PP_ERR_CUDA; }

}  // namespace ppc
