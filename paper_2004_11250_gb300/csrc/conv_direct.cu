// Direct 3x3 convolution on the FP32 FMA pipes for layers with few input or
// few output channels (the first and last layers of the networks: VGG-16's
// 3 -> 64, the VDSR-shaped stack's 1 -> 64 and 64 -> 1 dense convolutions, the
// 16 -> 16 single layer) and for dense layers of any width.  For the former the
// tensor-core kernels cannot fill an MMA (K = 8 channels per chunk, M = 64 or
// 128 filters) and their per-tile start-up dominates; the latter have no
// pattern structure, and the register kernel's dispatch per entry ran them at
// 2 % of the FP32 rate.
//
// The weights are expanded to the dense 9 taps (pruned taps and kernels are
// exact zeros, so the sum is the one of Section 2 with zero terms added; where
// an input is not finite, layers that need it sum the kept taps alone again: redo).  Input
// channels are staged a few at a time (tile plus one-pixel zero halo) together
// with their weights, in a ring of stages.  Where a tensor map can describe x (W a
// multiple of 4, x 16-byte aligned) a stage's input is one box copy, issued by one
// thread; else every thread copies by cp.async, whose issue slots and load-store
// work then bound the kernels (64 -> 1 at 720 x 1280 52 us against 36 with boxes).
// Waits on the boxes' mbarriers are bounded; one that gives up is recorded in the
// layer's device status word.  Epilogue: + bias, + skip,
// ReLU, optional 2 x 2 max pool, stored in the original channel order.
//
// ppconv_direct_kernel: a CTA of 256 threads owns FBD filters of a tile; a
// thread owns a 2 x 2 pixel block and FBD x 4 accumulators.  What bounds it is
// instruction issue and, on large maps, the FMA pipe (64 -> 64 at 224 x 224,
// batch 4: 51 of 73 TFLOP/s, 45 with cp.async copies), so two filters share each packed FMA
// (fma.rn.f32x2): the weights lie as pairs of filters, 9 pairs per channel padded
// to 80 bytes, read as broadcasts; the thread's 4 x 4 window is duplicated once
// per channel.  Maps with few tiles split the staged channels over KS groups of
// threads on tiles of 1024 / KS pixels, whose sums meet in shared memory in group
// order: 64 -> 64 at 56 x 56 would otherwise have 4 tiles (register kernel 268
// us, here 13.5).  Each chunk of channels is summed by itself and then added,
// which halves the rounding error of one long sum (1.1e-7 against 2.2e-7 of the
// result at 64 channels).
//
// ppconv_direct_wide_kernel: at most 3 filters on maps that its rows of 128 pixels
// do not mostly miss (a network's last layer).  These read far more than they compute (64 -> 1 at 720 x 1280: 236 MB
// of input), and with 2 x 2 blocks the shared-memory reads of the windows (16
// for 36 FMAs) took longer than the copies.  A thread owns 4 x 4 pixels, a warp 4
// rows of 128, so a window row is one 16-byte read and two shuffles for 12 FMAs a
// row and filter.  A warp of its own copies, and the others free a stage each for
// itself: with a barrier over the CTA per chunk their reads and their FMAs came in
// turns.  Three stages of two channels keep 40 KB per CTA in flight; where the
// tiles leave SMs without three CTAs, groups of warps share a tile's channels.
// 64 -> 1 at 720 x 1280 with the residual, alone: 97 us (2 x 2 blocks), 61
// (cp.async), 43 (boxes), 42 (copying warp), 36 among other launches, 6.7 TB/s of
// input, residual and output, where HBM bounds it; at 360 x 640 27.2 -> 16.3.
//
// ppconv_direct_first_kernel: at most 4 input channels (a network's first
// layer) on maps wider than a tile's half whose columns its tiles do not miss too much of.  These write far more than they read:
// a CTA stages its tile's input once for up to 64 filters, 8 at a time, and a
// thread's 2 x 4 pixels leave in 16-byte stores.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>
#include <vector>

#include "internal.h"
#include "tc_ptx.cuh"

namespace {

using namespace ppc_ptx;

constexpr int DTHREADS = 256;
constexpr int FBMAX = 8;      // filters per CTA at most
constexpr int WPAIR = 20;     // floats of one channel of a filter pair: 9 taps x 2 filters, the 2 filters' kept taps (bits)

struct DirectParams {
  const float* x;
  float* y;
  const float* skip;
  // [Ci][npair][WPAIR]: tap t of filters 2 q, 2 q + 1 at 2 t, 2 t + 1, a bit per kept tap of each at 18, 19; original
  // filter order
  const float* w;
  const float* bias;  // [Co] or null
  int N, Ci, Co, H, W, flags;
  int npair;
  int tiles_x, tiles_y;
  const float* wdup;  // at most 3 filters: [Ci][Co][20], tap t twice at 2 t, 2 t + 1
  int* status;        // device status word
  int redo;           // sums that are not finite are computed again: see redo
  // x 16-byte aligned, W a multiple of 4 and offsets within a channel in 32 bits: rows staged in 16-byte copies
  int vec;
};

__device__ __forceinline__ bool nan2(uint64_t v) {
  float a, b;
  unpack2(v, a, b);
  return a != a || b != b;
}

// A pruned tap is no part of the sum, but the kernels multiply it as a zero weight, and zero times an infinity or a NaN is
// not zero.  Every such product makes its output NaN.  In the instantiations with REDO a thread that meets a sum which is
// not finite computes its block of outputs (filters o0 .., rows r0 .., columns c0 ..) again over the kept taps alone,
// straight from x, after its stores.  Layers whose choice without these kernels would be one over the kept taps alone take
// those: within 2 % of the others' time in the wide kernel (256 -> 1 at 720 x 1280 150.7 -> 153.4 us),
// at it in the 2 x 2 kernel (64 -> 16 at 224 x 224 31.1 -> 30.8).
__device__ __forceinline__ void redo(const DirectParams& p, int n, int o0, int no, int r0, int nr, int c0, int nc) {
  const size_t plane = (size_t)p.H * p.W;
  const auto output = [&](int o, int r, int c) -> float {
    const float* w = p.w + (size_t)(o >> 1) * WPAIR + (o & 1);
    const float* x = p.x + (size_t)n * p.Ci * plane;
    float sum = 0.f;
    for (int i = 0; i < p.Ci; ++i, w += (size_t)p.npair * WPAIR, x += plane) {
      const uint32_t kept = __float_as_uint(__ldg(w + 18));
      for (int t = 0; t < 9; ++t) {
        if (!(kept >> t & 1)) continue;
        const int row = r - 1 + t / 3, col = c - 1 + t % 3;
        const bool in = (unsigned)row < (unsigned)p.H && (unsigned)col < (unsigned)p.W;
        sum = fmaf(__ldg(w + 2 * t), in ? __ldg(x + (size_t)row * p.W + col) : 0.f, sum);
      }
    }
    if (p.bias) sum += __ldg(p.bias + o);
    if (p.flags & PP_ADD_SKIP) sum += __ldg(p.skip + ((size_t)n * p.Co + o) * plane + (size_t)r * p.W + c);
    return p.flags & PP_RELU ? fmaxf(sum, 0.f) : sum;
  };
  for (int o = o0; o < min(o0 + no, p.Co); ++o)
    for (int r = r0; r < min(r0 + nr, p.H); r += p.flags & PP_POOL2 ? 2 : 1)
      for (int c = c0; c < min(c0 + nc, p.W); c += p.flags & PP_POOL2 ? 2 : 1) {
        const size_t q = (size_t)n * p.Co + o;
        if (p.flags & PP_POOL2)
          p.y[(q * (p.H / 2) + r / 2) * (p.W / 2) + c / 2] =
              fmaxf(fmaxf(output(o, r, c), output(o, r, c + 1)), fmaxf(output(o, r + 1, c), output(o, r + 1, c + 1)));
        else
          p.y[(q * p.H + r) * p.W + c] = output(o, r, c);
      }
}

// The same as a call: inlined it costs the 2 x 2 kernel registers (70 -> 90 for two filters, a CTA less per SM), while
// a call costs the wide kernel 8 %.
__device__ __noinline__ void redo_call(const DirectParams p, int n, int o0, int no, int r0, int nr, int c0, int nc) {
  redo(p, n, o0, no, r0, nr, c0, nc);
}

__device__ __forceinline__ void cp_async4(float* dst, const float* src, bool valid) {
  const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(d), "l"(src), "r"(valid ? 4 : 0) : "memory");
}
__device__ __forceinline__ void cp_async16(float* dst, const float* src, bool valid) {
  const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(valid ? 16 : 0) : "memory");
}

// Stages rows r0 - 1 .. r0 + ROWS - 2 and columns c0 - 4 .. c0 + COLS - 5 of some channels of an image, zero outside it
// and beyond Ci, as [channel][ROWS][COLS].  With W a multiple of 4 every 16-byte group is wholly inside or outside;
// otherwise only the columns c0 - 1 .. c0 + COLS - 8 that are read are copied, one by one.  A thread copies the same
// places of every channel: their offsets are worked out once (vec), so a copy costs an add and the copy itself.
template <int ROWS, int COLS, int NT>
struct XStage {
  static constexpr int GROUPS = ROWS * (COLS / 4), NE = (GROUPS + NT - 1) / NT;
  int src[NE];  // offset within a channel of x, or -1 outside the image
  __device__ __forceinline__ void init(const DirectParams& p, int r0, int c0, int tid) {
#pragma unroll
    for (int i = 0; i < NE; ++i) {
      const int e = tid + i * NT, rr = e / (COLS / 4), g = e - rr * (COLS / 4);
      const int r = r0 - 1 + rr, col = c0 - 4 + 4 * g;
      src[i] = e < GROUPS && (unsigned)r < (unsigned)p.H && (unsigned)col < (unsigned)p.W ? r * p.W + col : -1;
    }
  }
  template <int CC>
  __device__ __forceinline__ void copy(float* dst, const DirectParams& p, const float* xb, int ch0, int r0, int c0,
                                       int tid) const {
    const size_t plane = (size_t)p.H * p.W;
    const float* xc = xb + (size_t)ch0 * plane;
    if (p.vec) {
#pragma unroll
      for (int k = 0; k < CC; ++k, xc += plane) {
        const bool have = ch0 + k < p.Ci;
#pragma unroll
        for (int i = 0; i < NE; ++i)
          if ((i + 1) * NT <= GROUPS || tid + i * NT < GROUPS) {
            const bool in = have && src[i] >= 0;
            cp_async16(dst + k * ROWS * COLS + 4 * (tid + i * NT), in ? xc + src[i] : p.x, in);
          }
      }
    } else {
      constexpr int USED = COLS - 6;
      for (int e = tid; e < ROWS * USED; e += NT) {
        const int rr = e / USED, cc = e - rr * USED;
        const int r = r0 - 1 + rr, col = c0 - 1 + cc;
        const bool inside = (unsigned)r < (unsigned)p.H && (unsigned)col < (unsigned)p.W;
        const float* sp = xc + (size_t)r * p.W + col;
#pragma unroll
        for (int k = 0; k < CC; ++k, sp += plane) {
          const bool in = inside && ch0 + k < p.Ci;
          cp_async4(dst + (k * ROWS + rr) * COLS + cc + 3, in ? sp : p.x, in);
        }
      }
    }
  }
};

// Where x can be box-copied (a tensor map: W a multiple of 4, x 16-byte aligned) a stage's input is one copy by one thread
// that completes on the stage's mbarrier, with its zeros outside the image; XStage's copies are the other maps' path.
// Channels ch0 .. of image n from row r0 - 1, column c0 - 4 into dst; `more` further bytes come by bulk_copy.
__device__ __forceinline__ void box_copy(const CUtensorMap* m, float* dst, int bytes, int more, int ch0, int r0, int c0,
                                         int n, uint64_t* full) {
  mbar_arrive_expect_tx(su32(full), bytes + more);
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, "
      "%5}], [%6];" ::"r"(su32(dst)),
      "l"(reinterpret_cast<uint64_t>(m)), "r"(c0 - 4), "r"(r0 - 1), "r"(ch0), "r"(n), "r"(su32(full))
      : "memory");
}
__device__ __forceinline__ void bulk_copy(float* dst, const float* src, int bytes, uint64_t* full) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(su32(dst)),
               "l"(src), "r"(bytes), "r"(su32(full))
               : "memory");
}
// A bounded wait: false when it gave up.
__device__ __forceinline__ bool mbar_poll(uint32_t bar, uint32_t parity) {
  for (long q = 0; q < PP_WAIT_POLLS; ++q)
    if (mbar_try(bar, parity)) return true;
  return false;
}

// The full barriers of a ring whose stages are freed by a barrier over the CTA: every thread calls wait for every chunk,
// in order; thread 0 copies.
template <int NS>
struct BoxRing {
  uint64_t* full;  // [NS] in shared memory
  int issued = 0;  // thread 0: chunks whose copy was issued
  bool dead = false;
  __device__ __forceinline__ void init(int tid) {
    if (tid == 0) {
      for (int s = 0; s < NS; ++s) mbar_init(su32(full + s), 1);
      asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
  }
  __device__ __forceinline__ bool poll(int ch) const {
    return mbar_poll(su32(full + ch % NS), (uint32_t)((ch / NS) & 1));
  }
  // A wait that gives up is recorded, and the thread waits (and thread 0 copies) no more.
  __device__ __forceinline__ void wait(int ch, int* status) {
    if (dead || poll(ch)) return;
    dead = true;
    atomicOr(status, ppc::kStatusTimeout);
  }
  // Thread 0, after the last chunk: no copy may be in flight when the CTA's shared memory is reused or given back.
  __device__ __forceinline__ void drain() const {
    if (!dead) return;
    for (int ch = issued > NS ? issued - NS : 0; ch < issued; ++ch) poll(ch);
  }
};

// The tensor map as a kernel argument, nothing where there is none.
template <bool BOX>
struct BoxMap {
  CUtensorMap m;
};
template <>
struct BoxMap<false> {};

template <int CC, int FBD, int KS>
struct DirectGeo {
  static constexpr int TH = KS == 1 ? 32 : 16, TW = KS == 4 ? 16 : 32;  // tile of 1024 / KS pixels
  static constexpr int ROWS = TH + 2, COLS = TW + 8;                    // staged; columns from c0 - 4
  static constexpr int XS = CC * ROWS * COLS, WS = CC * (FBD / 2) * WPAIR;
  static constexpr int RED = KS > 1 ? (KS - 1) * (DTHREADS / KS) * FBD * 4 : 0;  // sums of groups 1 ..
  // stages: one chunk's arithmetic does not cover the copies' latency (small tiles have less of it)
  static constexpr int NS = KS == 1 ? 3 : 4;
  static constexpr int FLOATS = NS * (XS + WS) > RED ? NS * (XS + WS) : RED;
  static_assert(CC != 4 || XS * 4 % 128 == 0, "box copies start at 128 bytes");
  static_assert(CC % KS == 0 && FBD % 2 == 0, "channels over the groups, filters in pairs");
};

// Fewer than 4 channels are one chunk: latency decides, and a third CTA per SM hides it (1 -> 64 at 446 x 56, batch 2, 8.4 us
// against 6.1, although 8 filters of 2 or 3 channels then spill some 100 bytes).
template <int CC, int FBD, int KS, bool BOX, bool REDO>
__global__ void __launch_bounds__(DTHREADS, CC < 4 ? 3 : 2) ppconv_direct_kernel(const DirectParams p, const __grid_constant__ BoxMap<BOX> xmap) {
  using G = DirectGeo<CC, FBD, KS>;
  constexpr int NP = FBD / 2, GT = DTHREADS / KS, TX = G::TW / 2;
  // boxes start at 128 bytes, so the weights lie after them all; else in their stage
  constexpr int XSTEP = BOX ? G::XS : G::XS + G::WS, WSTEP = BOX ? G::WS : XSTEP, W0 = BOX ? G::NS * G::XS : G::XS;
  // NS stages of [CC][ROWS][COLS] input and [CC][NP][WPAIR] weights; at the end the groups' sums
  extern __shared__ __align__(128) float dsm[];
  __shared__ uint64_t full[G::NS];
  const int tid = threadIdx.x, grp = tid / GT, gt = tid % GT, tx = gt % TX, ty = gt / TX;
  int t = (int)blockIdx.x;
  const int bx = t % p.tiles_x;
  t /= p.tiles_x;
  const int by = t % p.tiles_y;
  const int n = t / p.tiles_y;
  const int q0 = (int)(blockIdx.z * gridDim.y + blockIdx.y) * NP;  // first filter pair
  if (q0 >= p.npair) return;
  const int r0 = by * G::TH, c0 = bx * G::TW;
  const float* xb = p.x + (size_t)n * p.Ci * p.H * p.W;
  const int nchunks = (p.Ci + CC - 1) / CC;

  XStage<G::ROWS, G::COLS, DTHREADS> xst;
  BoxRing<G::NS> ring{full};
  if constexpr (BOX) ring.init(tid);
  else xst.init(p, r0, c0, tid);
  auto stage = [&](int ch) {
    float* xs = dsm + (ch % G::NS) * XSTEP;
    float* ws = dsm + W0 + (ch % G::NS) * WSTEP;
    if constexpr (BOX) {
      if (tid == 0 && ch < nchunks && !ring.dead) {
        const int have = min(CC, p.Ci - ch * CC);  // the weights of these channels, a bulk copy each
        uint64_t* bar = full + ch % G::NS;
        box_copy(&xmap.m, xs, G::XS * 4, have * NP * WPAIR * 4, ch * CC, r0, c0, n, bar);
        for (int k = 0; k < have; ++k)
          bulk_copy(ws + k * NP * WPAIR, p.w + ((size_t)(ch * CC + k) * p.npair + q0) * WPAIR, NP * WPAIR * 4, bar);
        ring.issued = ch + 1;
      }
      return;
    }
    if (ch < nchunks) {
      xst.template copy<CC>(xs, p, xb, ch * CC, r0, c0, tid);
      for (int e = tid; e < CC * NP * (WPAIR / 4); e += DTHREADS) {  // the layout is padded to FBMAX filters
        const int k = e / (NP * (WPAIR / 4)), rem = e - k * (NP * (WPAIR / 4));
        const bool in = ch * CC + k < p.Ci;
        cp_async16(ws + 4 * e, in ? p.w + ((size_t)(ch * CC + k) * p.npair + q0) * WPAIR + 4 * rem : p.w, in);
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");  // one group per step, empty past the last chunk
  };

  uint64_t acc[NP][4];
#pragma unroll
  for (int o = 0; o < NP; ++o)
#pragma unroll
    for (int q = 0; q < 4; ++q) acc[o][q] = 0;

  // programmatic dependent launch: nothing of the previous kernel in the
  // stream is read or overwritten before this wait
  asm volatile("griddepcontrol.wait;" ::: "memory");
#pragma unroll
  for (int st = 0; st < G::NS - 1; ++st) stage(st);
  for (int ch = 0; ch < nchunks; ++ch) {
    if constexpr (BOX) asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // reads, before the next copy
    else asm volatile("cp.async.wait_group %0;" ::"n"(G::NS - 2) : "memory");
    __syncthreads();  // chunk ch has landed (cp.async); every thread is done with the stage that is filled next
    stage(ch + G::NS - 1);
    if constexpr (BOX) ring.wait(ch, p.status);
    const float* xs = dsm + (ch % G::NS) * XSTEP;
    const float* ws = dsm + W0 + (ch % G::NS) * WSTEP;
    uint64_t part[NP][4];  // the chunk's sum: added to acc as one term, which keeps the rounding error of long sums low
#pragma unroll
    for (int o = 0; o < NP; ++o)
#pragma unroll
      for (int q = 0; q < 4; ++q) part[o][q] = 0;
#pragma unroll 1
    for (int kk = 0; kk < CC / KS; ++kk) {
      const int k = kk * KS + grp;
      if (ch * CC + k >= p.Ci) break;
      // the thread's 4 x 4 input window (staged rows 2 ty .., columns 2 tx + 3 .. 2 tx + 6), each value twice
      uint64_t xv[4][4];
#pragma unroll
      for (int a = 0; a < 4; ++a) {
        const float2* row = reinterpret_cast<const float2*>(xs + (k * G::ROWS + 2 * ty + a) * G::COLS + 2 * tx + 2);
        const float2 u = row[0], v = row[1], w = row[2];
        xv[a][0] = pack2(u.y, u.y);
        xv[a][1] = pack2(v.x, v.x);
        xv[a][2] = pack2(v.y, v.y);
        xv[a][3] = pack2(w.x, w.x);
      }
#pragma unroll
      for (int o = 0; o < NP; ++o) {
        const float* wp = ws + (k * NP + o) * WPAIR;
        uint64_t wt[9];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(wp + 4 * e);
          wt[2 * e] = v.x;
          wt[2 * e + 1] = v.y;
        }
        wt[8] = *reinterpret_cast<const uint64_t*>(wp + 16);
#pragma unroll
        for (int dy = 0; dy < 3; ++dy)
#pragma unroll
          for (int dx = 0; dx < 3; ++dx)
#pragma unroll
            for (int py = 0; py < 2; ++py)
#pragma unroll
              for (int px = 0; px < 2; ++px)
                part[o][py * 2 + px] = fma2(wt[dy * 3 + dx], xv[py + dy][px + dx], part[o][py * 2 + px]);
      }
    }
#pragma unroll
    for (int o = 0; o < NP; ++o)
#pragma unroll
      for (int q = 0; q < 4; ++q) acc[o][q] = add2(acc[o][q], part[o][q]);
  }

  if constexpr (BOX)
    if (tid == 0) ring.drain();
  // the next kernel may start its prologue (it waits for this grid to finish)
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if (KS > 1) {
    // groups 1 .. hand their sums to group 0, which adds them in order
    uint64_t* red = reinterpret_cast<uint64_t*>(dsm);
    __syncthreads();  // every thread is done with the stages (no copy is in flight: the last groups are empty)
    if (grp > 0) {
#pragma unroll
      for (int o = 0; o < NP; ++o)
#pragma unroll
        for (int q = 0; q < 4; ++q) red[((grp - 1) * NP * 4 + o * 4 + q) * GT + gt] = acc[o][q];
    }
    __syncthreads();
    if (grp > 0) return;
#pragma unroll
    for (int g = 0; g < KS - 1; ++g)
#pragma unroll
      for (int o = 0; o < NP; ++o)
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[o][q] = add2(acc[o][q], red[(g * NP * 4 + o * 4 + q) * GT + gt]);
  }
  const bool relu = p.flags & PP_RELU, pool = p.flags & PP_POOL2;
  const float* skip = (p.flags & PP_ADD_SKIP) ? p.skip : nullptr;
  const int r = r0 + 2 * ty, c = c0 + 2 * tx;
  uint64_t bad = 0;  // zero times every sum: NaN once one is not finite
  if constexpr (REDO) {
#pragma unroll
    for (int o = 0; o < NP; ++o)
#pragma unroll
      for (int q = 0; q < 4; ++q) bad = fma2(acc[o][q], 0, bad);
  }
#pragma unroll
  for (int o = 0; o < FBD; ++o) {
    const int oo = 2 * q0 + o;
    if (oo >= p.Co) break;
    const size_t plane = (size_t)n * p.Co + oo;
    const float bs = p.bias ? __ldg(p.bias + oo) : 0.f;
    float v[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int rq = r + (q >> 1), cq = c + (q & 1);
      float lo, hi;
      unpack2(acc[o / 2][q], lo, hi);
      v[q] = (o & 1 ? hi : lo) + bs;
      if (skip && rq < p.H && cq < p.W) v[q] += __ldg(skip + (plane * p.H + rq) * p.W + cq);
      if (relu) v[q] = fmaxf(v[q], 0.f);
    }
    if (pool) {
      // H and W are even, so a block inside the image is whole
      if (r < p.H && c < p.W)
        p.y[(plane * (p.H / 2) + r / 2) * (p.W / 2) + c / 2] = fmaxf(fmaxf(v[0], v[1]), fmaxf(v[2], v[3]));
    } else {
#pragma unroll
      for (int py = 0; py < 2; ++py) {
        const int rq = r + py;
        if (rq >= p.H) break;
        float* yr = p.y + (plane * p.H + rq) * p.W;
        if ((p.W & 1) == 0 && c + 1 < p.W) {
          *reinterpret_cast<float2*>(yr + c) = make_float2(v[py * 2], v[py * 2 + 1]);
        } else {
          if (c < p.W) yr[c] = v[py * 2];
          if (c + 1 < p.W) yr[c + 1] = v[py * 2 + 1];
        }
      }
    }
  }
  if (REDO && nan2(bad)) redo_call(p, n, 2 * q0, FBD, r, 2, c, 2);
}

constexpr int VH = 16, VW = 128;             // tile: 4 rows of 128 pixels per warp of a group
constexpr int VROWS = VH + 2, VCOLS = VW + 8;

// KS groups of 4 warps take the channels of a stage in turn; group 0 adds their sums.
template <int CO, int KS, bool BOX>
struct WideGeo {
  static constexpr int NT = 128 * KS, VCC = KS == 4 ? 4 : 2;          // computing threads, channels per stage
  static constexpr int VST = KS == 1 ? 3 : 5;                         // stages
  static constexpr int THREADS = NT + (BOX ? 32 : 0);                 // and the warp that issues the copies
  static constexpr int XS = VCC * VROWS * VCOLS, WS = VCC * CO * 20;  // floats of a stage
  static constexpr int BYTES = VST * (XS + WS) * 4;
  static_assert(XS * 4 % 128 == 0, "box copies start at 128 bytes");
  static_assert((KS - 1) * CO * 8 * 128 * 8 <= BYTES, "the groups' sums lie over the stages");
};

template <int CO, int KS, bool BOX, bool REDO>
__global__ void __launch_bounds__(WideGeo<CO, KS, BOX>::THREADS, KS == 1 ? 3 : 1)
    ppconv_direct_wide_kernel(const DirectParams p, const __grid_constant__ BoxMap<BOX> xmap) {
  using G = WideGeo<CO, KS, BOX>;
  constexpr int VCC = G::VCC, VST = G::VST;
  // VST stages of [VCC][VROWS][VCOLS] input, then of [VCC][CO][9][2] weights (each twice, for packed FMAs)
  extern __shared__ __align__(128) float dsm[];
  __shared__ uint64_t full[VST], empty[VST];
  float* const wsm = dsm + VST * G::XS;
  const int tid = threadIdx.x, grp = tid >> 7, gt = tid & 127, warp = gt >> 5, lane = tid & 31;
  int t = (int)blockIdx.x;
  const int bx = t % p.tiles_x;
  t /= p.tiles_x;
  const int by = t % p.tiles_y;
  const int n = t / p.tiles_y;
  const int r0 = by * VH, c0 = bx * VW;
  const int nchunks = (p.Ci + VCC - 1) / VCC;

  if constexpr (BOX) {
    if (tid == 0) {
      for (int s = 0; s < VST; ++s) {
        mbar_init(su32(full + s), 1);
        mbar_init(su32(empty + s), 4 * KS);  // one arrival per computing warp
      }
      asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
  }
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if constexpr (BOX) {
    if (tid >= G::NT) {
      // One thread copies a chunk's input box and weights into its stage once every warp is done with the chunk before.
      if (lane == 0) {
        int ch = 0;
        for (; ch < nchunks; ++ch) {
          const int st = ch % VST;
          if (ch >= VST && !mbar_poll(su32(empty + st), (uint32_t)((ch / VST - 1) & 1))) {
            atomicOr(p.status, ppc::kStatusTimeout);
            break;
          }
          const int wbytes = min(VCC, p.Ci - ch * VCC) * CO * 80;
          box_copy(&xmap.m, dsm + st * G::XS, G::XS * 4, wbytes, ch * VCC, r0, c0, n, full + st);
          bulk_copy(wsm + st * G::WS, p.wdup + (size_t)ch * VCC * CO * 20, wbytes, full + st);
        }
        // no copy may be in flight when the CTA exits (the computing warps waited for them unless a wait gave up)
        for (int c = ch > VST ? ch - VST : 0; c < ch; ++c) mbar_poll(su32(full + c % VST), (uint32_t)((c / VST) & 1));
      }
      asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
      return;
    }
  }

  uint64_t acc[CO][4][2];  // 4 rows x 4 columns as pairs of columns
#pragma unroll
  for (int o = 0; o < CO; ++o)
#pragma unroll
    for (int r = 0; r < 4; ++r) acc[o][r][0] = acc[o][r][1] = 0;

  auto compute = [&](int ch) {
    const float* xs = dsm + (ch % VST) * G::XS;
    const float* ws = wsm + (ch % VST) * G::WS;
#pragma unroll
    for (int kk = 0; kk < VCC / KS; ++kk) {
      const int k = kk * KS + grp;
      if (ch * VCC + k >= p.Ci) break;
      // window rows 0 .. 5, columns -1 .. 4 of the thread's block: pairs starting at each of the columns -1 .. 3
      uint64_t xp[6][5];
#pragma unroll
      for (int a = 0; a < 6; ++a) {
        const float* row = xs + (k * VROWS + 4 * warp + a) * VCOLS;
        const float4 v = *reinterpret_cast<const float4*>(row + 4 * lane + 4);
        const float edge = row[lane == 0 ? 3 : VW + 4];
        float l = __shfl_up_sync(0xffffffffu, v.w, 1), r = __shfl_down_sync(0xffffffffu, v.x, 1);
        l = lane == 0 ? edge : l;
        r = lane == 31 ? edge : r;
        xp[a][0] = pack2(l, v.x);
        xp[a][1] = pack2(v.x, v.y);
        xp[a][2] = pack2(v.y, v.z);
        xp[a][3] = pack2(v.z, v.w);
        xp[a][4] = pack2(v.w, r);
      }
#pragma unroll
      for (int o = 0; o < CO; ++o) {
        const float* wp = ws + (k * CO + o) * 20;
        uint64_t wt[9];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(wp + 4 * e);
          wt[2 * e] = v.x;
          wt[2 * e + 1] = v.y;
        }
        wt[8] = *reinterpret_cast<const uint64_t*>(wp + 16);
#pragma unroll
        for (int dy = 0; dy < 3; ++dy)
#pragma unroll
          for (int dx = 0; dx < 3; ++dx)
#pragma unroll
            for (int r = 0; r < 4; ++r)
#pragma unroll
              for (int h = 0; h < 2; ++h)
                acc[o][r][h] = fma2(wt[dy * 3 + dx], xp[r + dy][2 * h + dx], acc[o][r][h]);
      }
    }
  };

  if constexpr (BOX) {
    bool dead = false;  // after a wait that gave up the thread waits no more; the output is invalid
    for (int ch = 0; ch < nchunks; ++ch) {
      const int st = ch % VST;
      if (!dead && !mbar_poll(su32(full + st), (uint32_t)((ch / VST) & 1))) {
        dead = true;
        atomicOr(p.status, ppc::kStatusTimeout);
      }
      compute(ch);
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // these reads, before the next copy into the stage
      __syncwarp();
      if (lane == 0) mbar_arrive(su32(empty + st));
    }
  } else {
    const float* xb = p.x + (size_t)n * p.Ci * p.H * p.W;
    XStage<VROWS, VCOLS, G::NT> xst;
    xst.init(p, r0, c0, tid);
    auto stage = [&](int ch) {
      const int st = ch % VST;
      if (ch < nchunks) {
        xst.template copy<VCC>(dsm + st * G::XS, p, xb, ch * VCC, r0, c0, tid);
        const int have = min(VCC, p.Ci - ch * VCC) * CO * 5;
        for (int e = tid; e < have; e += G::NT)
          cp_async16(wsm + st * G::WS + 4 * e, p.wdup + (size_t)ch * VCC * CO * 20 + 4 * e, true);
      }
      asm volatile("cp.async.commit_group;" ::: "memory");  // one group per step, empty past the last chunk
    };
#pragma unroll
    for (int s = 0; s < VST - 1; ++s) stage(s);
    for (int ch = 0; ch < nchunks; ++ch) {
      asm volatile("cp.async.wait_group %0;" ::"n"(VST - 2) : "memory");
      __syncthreads();  // chunk ch has landed; every thread is done with the stage that is filled next
      stage(ch + VST - 1);
      compute(ch);
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
  }

  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if constexpr (KS > 1) {
    uint64_t* red = reinterpret_cast<uint64_t*>(dsm);
    group_sync<G::NT>();  // every thread is done with the stages
    if (grp > 0) {
#pragma unroll
      for (int o = 0; o < CO; ++o)
#pragma unroll
        for (int e = 0; e < 8; ++e) red[(((grp - 1) * CO + o) * 8 + e) * 128 + gt] = acc[o][e >> 1][e & 1];
    }
    group_sync<G::NT>();
    if (grp > 0) return;
#pragma unroll
    for (int g = 0; g < KS - 1; ++g)
#pragma unroll
      for (int o = 0; o < CO; ++o)
#pragma unroll
        for (int e = 0; e < 8; ++e)
          acc[o][e >> 1][e & 1] = add2(acc[o][e >> 1][e & 1], red[((g * CO + o) * 8 + e) * 128 + gt]);
  }
  const bool relu = p.flags & PP_RELU, pool = p.flags & PP_POOL2;
  const float* skip = (p.flags & PP_ADD_SKIP) ? p.skip : nullptr;
  const int row0 = r0 + 4 * warp, c = c0 + 4 * lane;
  const bool wide = (p.W & 3) == 0;
  uint64_t bad = 0;  // zero times every sum: NaN once one is not finite
  if constexpr (REDO) {
#pragma unroll
    for (int o = 0; o < CO; ++o)
#pragma unroll
      for (int e = 0; e < 8; ++e) bad = fma2(acc[o][e >> 1][e & 1], 0, bad);
  }
#pragma unroll
  for (int o = 0; o < CO; ++o) {
    const size_t plane = (size_t)n * p.Co + o;
    const float bs = p.bias ? __ldg(p.bias + o) : 0.f;
    float v[4][4];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      unpack2(acc[o][r][0], v[r][0], v[r][1]);
      unpack2(acc[o][r][1], v[r][2], v[r][3]);
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        v[r][k] += bs;
        if (skip && row0 + r < p.H && c + k < p.W) v[r][k] += __ldg(skip + (plane * p.H + row0 + r) * p.W + c + k);
        if (relu) v[r][k] = fmaxf(v[r][k], 0.f);
      }
    }
    if (pool) {  // H and W are even, so a 2 x 2 window inside the image is whole
#pragma unroll
      for (int r = 0; r < 4; r += 2)
#pragma unroll
        for (int k = 0; k < 4; k += 2)
          if (row0 + r < p.H && c + k < p.W)
            p.y[(plane * (p.H / 2) + (row0 + r) / 2) * (p.W / 2) + (c + k) / 2] =
                fmaxf(fmaxf(v[r][k], v[r][k + 1]), fmaxf(v[r + 1][k], v[r + 1][k + 1]));
    } else {
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        if (row0 + r >= p.H) break;
        float* yr = p.y + (plane * p.H + row0 + r) * p.W;
        if (wide) {
          if (c < p.W) *reinterpret_cast<float4*>(yr + c) = make_float4(v[r][0], v[r][1], v[r][2], v[r][3]);
        } else {
#pragma unroll
          for (int k = 0; k < 4; ++k)
            if (c + k < p.W) yr[c + k] = v[r][k];
        }
      }
    }
  }
  if (REDO && nan2(bad)) redo(p, n, 0, CO, row0, 4, c, 4);
}

constexpr int UTHREADS = 128;                // 4 warps
constexpr int UH = 8, UW = 128;              // tile: 2 rows of 128 pixels per warp
constexpr int UROWS = UH + 2, UCOLS = UW + 8;
constexpr int UFMAX = 64;                    // filters per CTA at most

template <int CI>
__global__ void __launch_bounds__(UTHREADS, 3) ppconv_direct_first_kernel(const DirectParams p, int fpc) {
  constexpr int NP = FBMAX / 2;
  __shared__ __align__(16) float xs[CI * UROWS * UCOLS];
  __shared__ __align__(16) float ws[CI * (UFMAX / 2) * WPAIR];  // [CI][fpc / 2][WPAIR]
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  int t = (int)blockIdx.x;
  const int bx = t % p.tiles_x;
  t /= p.tiles_x;
  const int by = t % p.tiles_y;
  const int n = t / p.tiles_y;
  const int r0 = by * UH, c0 = bx * UW;
  const int q0 = (int)blockIdx.y * (fpc / 2), nq = min(fpc / 2, p.npair - q0);  // filter pairs of this CTA
  // the weights do not depend on the previous kernel in the stream
  for (int e = tid; e < CI * nq * (WPAIR / 4); e += UTHREADS) {
    const int k = e / (nq * (WPAIR / 4)), rem = e - k * (nq * (WPAIR / 4));
    cp_async16(ws + 4 * e, p.w + ((size_t)k * p.npair + q0) * WPAIR + 4 * rem, true);
  }
  asm volatile("griddepcontrol.wait;" ::: "memory");
  XStage<UROWS, UCOLS, UTHREADS> xst;
  xst.init(p, r0, c0, tid);
  xst.template copy<CI>(xs, p, p.x + (size_t)n * p.Ci * p.H * p.W, 0, r0, c0, tid);
  asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 0;" ::: "memory");
  __syncthreads();
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

  const bool relu = p.flags & PP_RELU, pool = p.flags & PP_POOL2;
  const float* skip = (p.flags & PP_ADD_SKIP) ? p.skip : nullptr;
  const int row0 = r0 + 2 * warp, c = c0 + 4 * lane;
  const bool wide = (p.W & 3) == 0;
  for (int q = 0; q < nq; q += NP) {
    uint64_t acc[NP][2][4];  // filter pairs x 2 rows x 4 columns
#pragma unroll
    for (int o = 0; o < NP; ++o)
#pragma unroll
      for (int e = 0; e < 8; ++e) acc[o][e >> 2][e & 3] = 0;
#pragma unroll
    for (int k = 0; k < CI; ++k) {
      uint64_t xv[4][6];  // window rows, columns -1 .. 4 of the thread's block, each value twice
#pragma unroll
      for (int a = 0; a < 4; ++a) {
        const float* row = xs + (k * UROWS + 2 * warp + a) * UCOLS;
        const float4 v = *reinterpret_cast<const float4*>(row + 4 * lane + 4);
        const float edge = row[lane == 0 ? 3 : UW + 4];
        float l = __shfl_up_sync(0xffffffffu, v.w, 1), r = __shfl_down_sync(0xffffffffu, v.x, 1);
        l = lane == 0 ? edge : l;
        r = lane == 31 ? edge : r;
        xv[a][0] = pack2(l, l);
        xv[a][1] = pack2(v.x, v.x);
        xv[a][2] = pack2(v.y, v.y);
        xv[a][3] = pack2(v.z, v.z);
        xv[a][4] = pack2(v.w, v.w);
        xv[a][5] = pack2(r, r);
      }
#pragma unroll
      for (int o = 0; o < NP; ++o) {
        const float* wp = ws + (k * nq + q + o) * WPAIR;  // the layout is padded to whole groups of FBMAX filters
        uint64_t wt[9];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(wp + 4 * e);
          wt[2 * e] = v.x;
          wt[2 * e + 1] = v.y;
        }
        wt[8] = *reinterpret_cast<const uint64_t*>(wp + 16);
#pragma unroll
        for (int dy = 0; dy < 3; ++dy)
#pragma unroll
          for (int dx = 0; dx < 3; ++dx)
#pragma unroll
            for (int py = 0; py < 2; ++py)
#pragma unroll
              for (int px = 0; px < 4; ++px)
                acc[o][py][px] = fma2(wt[dy * 3 + dx], xv[py + dy][px + dx], acc[o][py][px]);
      }
    }
#pragma unroll
    for (int o = 0; o < FBMAX; ++o) {
      const int oo = 2 * (q0 + q) + o;
      if (oo >= p.Co) break;
      const size_t plane = (size_t)n * p.Co + oo;
      const float bs = p.bias ? __ldg(p.bias + oo) : 0.f;
      float v[2][4];
#pragma unroll
      for (int r = 0; r < 2; ++r)
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          float lo, hi;
          unpack2(acc[o / 2][r][k], lo, hi);
          v[r][k] = (o & 1 ? hi : lo) + bs;
          if (skip && row0 + r < p.H && c + k < p.W) v[r][k] += __ldg(skip + (plane * p.H + row0 + r) * p.W + c + k);
          if (relu) v[r][k] = fmaxf(v[r][k], 0.f);
        }
      if (pool) {  // H and W are even, so a 2 x 2 window inside the image is whole
#pragma unroll
        for (int k = 0; k < 4; k += 2)
          if (row0 < p.H && c + k < p.W)
            p.y[(plane * (p.H / 2) + row0 / 2) * (p.W / 2) + (c + k) / 2] =
                fmaxf(fmaxf(v[0][k], v[0][k + 1]), fmaxf(v[1][k], v[1][k + 1]));
      } else {
#pragma unroll
        for (int r = 0; r < 2; ++r) {
          if (row0 + r >= p.H) break;
          float* yr = p.y + (plane * p.H + row0 + r) * p.W;
          if (wide) {
            if (c < p.W) *reinterpret_cast<float4*>(yr + c) = make_float4(v[r][0], v[r][1], v[r][2], v[r][3]);
          } else {
#pragma unroll
            for (int k = 0; k < 4; ++k)
              if (c + k < p.W) yr[c + k] = v[r][k];
          }
        }
      }
    }
  }
}

// One launch of kernel K (its dynamic shared memory allowed once per device).
template <class K, class... A>
cudaError_t launch_kernel(K kernel, ppc::DeviceOnce& once, dim3 grid, int threads, int bytes, cudaStream_t stream,
                          const A&... args) {
  const cudaError_t ea =
      once.run([&](int) { return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes); });
  if (ea != cudaSuccess) return ea;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  cfg.gridDim = grid;
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = (size_t)bytes;
  cfg.stream = stream;
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}

template <int CC, int FBD, int KS>
cudaError_t launch_one(DirectParams p, cudaStream_t stream) {
  using G = DirectGeo<CC, FBD, KS>;
  static ppc::DeviceOnce once;  // one per instantiation
  p.tiles_x = (p.W + G::TW - 1) / G::TW;
  p.tiles_y = (p.H + G::TH - 1) / G::TH;
  const int64_t nt = (int64_t)p.N * p.tiles_x * p.tiles_y, nfb = (p.Co + FBD - 1) / FBD;
  if (nt > INT32_MAX) return cudaErrorInvalidConfiguration;
  const unsigned gy = (unsigned)std::min<int64_t>(nfb, 65535);  // the grid's y extent; the rest in z
  const dim3 grid((unsigned)nt, gy, (unsigned)((nfb + gy - 1) / gy));
  // Boxes where the grid is large (64 -> 64 at 224 x 224 94 -> 83 us, 96 -> 96 at 112 x 112 73.5 -> 70.5); with four
  // groups on small tiles a box's latency costs more than the copies it saves (64 -> 64 at 56 x 56 14.6 against 14.0).
  if constexpr (CC == 4 && KS <= 2) {
    BoxMap<true> xmap;
    if (p.Ci > CC && ppc::image_map(&xmap.m, p.x, p.N, p.Ci, p.H, p.W, G::COLS, G::ROWS, CC)) {
      static ppc::DeviceOnce box, box_redo;
      return p.redo ? launch_kernel(ppconv_direct_kernel<CC, FBD, KS, true, true>, box_redo, grid, DTHREADS, G::FLOATS * 4,
                                    stream, p, xmap)
                    : launch_kernel(ppconv_direct_kernel<CC, FBD, KS, true, false>, box, grid, DTHREADS, G::FLOATS * 4,
                                    stream, p, xmap);
    }
  }
  if constexpr (CC == 4) {  // with fewer channels no other kernel runs a layer by default
    static ppc::DeviceOnce once_redo;
    if (p.redo)
      return launch_kernel(ppconv_direct_kernel<CC, FBD, KS, false, true>, once_redo, grid, DTHREADS, G::FLOATS * 4, stream,
                           p, BoxMap<false>());
  }
  return launch_kernel(ppconv_direct_kernel<CC, FBD, KS, false, false>, once, grid, DTHREADS, G::FLOATS * 4, stream, p,
                       BoxMap<false>());
}

template <int CO, int KS, bool BOX>
cudaError_t launch_wide_one(const DirectParams& p, int64_t nt, const BoxMap<BOX>& xmap, cudaStream_t stream) {
  using G = WideGeo<CO, KS, BOX>;
  static ppc::DeviceOnce once, once_redo;  // one per instantiation
  return p.redo ? launch_kernel(ppconv_direct_wide_kernel<CO, KS, BOX, true>, once_redo, dim3((unsigned)nt), G::THREADS,
                                G::BYTES, stream, p, xmap)
                : launch_kernel(ppconv_direct_wide_kernel<CO, KS, BOX, false>, once, dim3((unsigned)nt), G::THREADS,
                                G::BYTES, stream, p, xmap);
}

template <int CO, int KS>
cudaError_t launch_wide(DirectParams p, cudaStream_t stream) {
  p.tiles_x = (p.W + VW - 1) / VW;
  p.tiles_y = (p.H + VH - 1) / VH;
  const int64_t nt = (int64_t)p.N * p.tiles_x * p.tiles_y;
  if (nt > INT32_MAX) return cudaErrorInvalidConfiguration;
  BoxMap<true> xmap;
  if (ppc::image_map(&xmap.m, p.x, p.N, p.Ci, p.H, p.W, VCOLS, VROWS, WideGeo<CO, KS, true>::VCC))
    return launch_wide_one<CO, KS, true>(p, nt, xmap, stream);
  return launch_wide_one<CO, KS, false>(p, nt, BoxMap<false>(), stream);
}

template <int CI>
cudaError_t launch_first(DirectParams p, int fpc, cudaStream_t stream) {
  static ppc::DeviceOnce once;
  p.tiles_x = (p.W + UW - 1) / UW;
  p.tiles_y = (p.H + UH - 1) / UH;
  const int64_t nt = (int64_t)p.N * p.tiles_x * p.tiles_y, nf = (2 * (int64_t)p.npair + fpc - 1) / fpc;
  if (nt > INT32_MAX || nf > 65535) return cudaErrorInvalidConfiguration;
  return launch_kernel(ppconv_direct_first_kernel<CI>, once, dim3((unsigned)nt, (unsigned)nf), UTHREADS, 0, stream, p,
                       fpc);
}

template <int CC, int KS>
cudaError_t launch_fbd(const DirectParams& p, int fbd, cudaStream_t stream) {
  switch (fbd) {
    case 2: return launch_one<CC, 2, KS>(p, stream);
    case 4: return launch_one<CC, 4, KS>(p, stream);
    default: return launch_one<CC, FBMAX, KS>(p, stream);
  }
}

}  // namespace

namespace ppc {

// Pruned layers get a direct layout when one side is small (dense ones always do).
bool direct_applicable(int Co, int Ci) {
  return (Ci <= kDirectMaxSmall || Co <= kDirectMaxSmall) && (int64_t)Co * Ci <= (int64_t(1) << 20);
}

// Weights (npair pairs of filters, padded to whole CTAs of FBMAX filters with zeros), the wide kernel's (each twice), bias.
static std::vector<float> direct_host(const float* w_dense, const uint16_t* kept, const float* bias, int Co, int Ci,
                                      int npair) {
  const size_t ndup = Co <= 3 ? (size_t)Ci * Co * WPAIR : 0;
  const size_t np = (size_t)Ci * npair * WPAIR, nw = np + ndup;
  std::vector<float> host(nw + (bias ? Co : 0), 0.f);
  for (int o = 0; o < Co; ++o)
    for (int i = 0; i < Ci; ++i) {
      float* dst = &host[((size_t)i * npair + (o >> 1)) * WPAIR + (o & 1)];
      const float* src = w_dense + ((size_t)o * Ci + i) * 9;
      for (int t = 0; t < 9; ++t) dst[2 * t] = src[t];
      const uint32_t bits = kept ? kept[(size_t)o * Ci + i] : 0x1ffu;
      std::memcpy(dst + 18, &bits, 4);
      if (ndup)
        for (int t = 0; t < 18; ++t) host[np + ((size_t)i * Co + o) * WPAIR + t] = src[t >> 1];
    }
  if (bias) std::copy_n(bias, Co, &host[nw]);
  return host;
}

pp_status direct_build(DirectLayout* D, const float* w_dense, const uint16_t* kept, const float* bias, int Co, int Ci,
                       cudaStream_t stream) {
  const int npair = (Co + FBMAX - 1) / FBMAX * (FBMAX / 2);
  const std::vector<float> host = direct_host(w_dense, kept, bias, Co, Ci, npair);
  void* d = nullptr;
  if (cudaMalloc(&d, (host.size() + 1) * 4) != cudaSuccess) {
    cudaGetLastError();
    return PP_ERR_OOM;
  }
  int* status = reinterpret_cast<int*>(static_cast<float*>(d) + host.size());
  if (cudaMemsetAsync(status, 0, sizeof(int), stream) != cudaSuccess ||
      cudaMemcpyAsync(d, host.data(), host.size() * 4, cudaMemcpyHostToDevice, stream) != cudaSuccess ||
      cudaStreamSynchronize(stream) != cudaSuccess) {
    cudaFree(d);
    return PP_ERR_CUDA;
  }
  D->dmem = d;
  D->dbytes = (host.size() + 1) * 4;
  D->status = status;
  D->w = static_cast<const float*>(d);
  D->bias = bias ? static_cast<const float*>(d) + host.size() - Co : nullptr;
  D->wdup = Co <= 3 ? static_cast<const float*>(d) + (size_t)Ci * npair * WPAIR : nullptr;
  D->npair = npair;
  D->redo = kept != nullptr;
  D->Co = Co;
  D->Ci = Ci;
  return PP_OK;
}

pp_status direct_update(const DirectLayout& D, const float* w_dense, const uint16_t* kept, const float* bias,
                        cudaStream_t stream) {
  const std::vector<float> host = direct_host(w_dense, kept, bias, D.Co, D.Ci, D.npair);
  if (cudaMemcpyAsync(D.dmem, host.data(), host.size() * 4, cudaMemcpyHostToDevice, stream) != cudaSuccess ||
      cudaStreamSynchronize(stream) != cudaSuccess) {
    cudaGetLastError();
    return PP_ERR_CUDA;
  }
  return PP_OK;
}

// CTAs of tiles of th x tw pixels and f filters.
static int64_t tiles(const DirectLayout& D, int N, int H, int W, int th, int tw, int f) {
  return (int64_t)N * ((H + th - 1) / th) * ((W + tw - 1) / tw) * ((D.Co + f - 1) / f);
}

// Which of the 2 x 2 and wide kernels a layer runs on a map, and in which form.
struct Plan {
  int fbd = 0, ks = 1;   // 2 x 2 kernel: filters per CTA, channel groups
  int64_t grid = 0;      // and its CTAs
  int64_t vt = 0;        // tiles of the wide kernel, 0 for layers that it does not run
  bool wide = false;
  double wide_us = 0;    // its time at 64 channels where it was considered
};
static Plan make_plan(const DirectLayout& D, int N, int H, int W, bool vec, int64_t sms) {
  Plan pl;
  const auto ctas = [&](int th, int tw, int f) { return tiles(D, N, H, W, th, tw, f); };
  // 2 x 2 kernel, filters per CTA: as many as there are, up to 8; channel groups while the grid would leave SMs without two
  // CTAs, and fewer filters (the input tile is then staged more often) only when even four groups leave a quarter of the
  // SMs idle (64 -> 64 at 56 x 56, 128 CTAs of 8 filters: 13.5 us, of 4 filters 19.7).
  int fbd = D.Co > 4 ? 8 : D.Co > 2 ? 4 : 2, ks = 1;
  const auto grid = [&]() { return ctas(ks == 1 ? 32 : 16, ks == 4 ? 16 : 32, fbd); };
  if (D.Ci > 4) {
    if (grid() < 2 * sms) ks = 2;
    if (grid() < 2 * sms) ks = 4;
  }
  while (fbd > 2 && grid() < (ks == 4 ? sms * 3 / 4 : 2 * sms)) fbd /= 2;

  // The wide kernel where it has tiles for two SMs in five (64 -> 1 at 128 x 128, batch 8, 64 tiles: 16.0 us against the 2 x
  // 2 kernel's 19.6), with more groups of warps the fewer there are (64 -> 1 at 360 x 640, 115 tiles: 1 / 2 / 4 groups 21.0
  // / 18.8 / 16.3, 2 x 2 kernel 27.2; 540 x 960, 272 tiles: 38.9 / 30.4 / 34.3, 42.9; 720 x 1280, 450 tiles: 40.6 / 46.3 /
  // 51.2, 70.5), and where its 128 columns are not spent on the map's edge: both kernels' time goes by the CTAs of the
  // busiest SM, and the wide kernel's take about as long as the 2 x 2 kernel's with half as many pixels.  The figures
  // below are us at 64 channels (they scale with the channels) on 252 maps of 8 .. 640 columns, where this choice is within
  // 9 % of the better kernel; by tiles alone narrow maps took up to 4.9 times as long (64 -> 3 at 781 x 16, batch 4, 68.9
  // against 13.9; 64 x 3125 157 against 96; 64 -> 1 at 6250 x 32 127 against 61).
  const int64_t vt = D.Ci >= 8 && D.Co <= 3 ? ctas(VH, VW, 4) : 0;
  const auto rounds = [&](int64_t n) { return (double)((n + sms - 1) / sms); };
  bool wide = vt && (D.Co == 1   ? vt * (vec ? 5 : 4) >= 2 * sms
                     : D.Co == 2 ? vt >= 2 * sms
                                 : vt >= sms || (vec && vt * 3 >= sms * 2));
  if (wide) {
    const double c = rounds(vt);
    const double tw = D.Co == 1 ? (vec ? (vt <= sms ? 16.2 : vt < 2 * sms ? 29.2 : 10.8 * c + 8.6)
                                         : (vt < sms ? 28.3 : 22.2 * c + 11.0))
                      : D.Co == 2 ? (vec ? 17.4 * c + 8.0 : 30.5 * c + 14.0)
                                  : (vec ? (vt < 2 * sms ? 34.7 * c : 24.6 * c + 9.8)
                                           : (vt < 2 * sms ? 53.4 * c : 39.2 * c + 13.0));
    // us of one CTA for each SM, by channel groups (1, 2, 4): rows of whole 16-byte groups or not, 2 or 4 filters
    static const double round_us[2][2][3] = {{{16.3, 9.6, 6.0}, {21.2, 12.5, 8.0}}, {{10.1, 6.6, 5.05}, {16.0, 10.4, 7.0}}};
    pl.wide_us = tw;
    wide = tw < round_us[vec ? 1 : 0][fbd > 2][ks == 4 ? 2 : ks - 1] * rounds(grid());
  }
  pl.fbd = fbd;
  pl.ks = ks;
  pl.grid = grid();
  pl.vt = vt;
  pl.wide = wide;
  return pl;
}

// us of a launch with more than 4 channels: within 12 % for nine in ten of 726 random pruned layers and maps that it was not
// fitted to (5 .. 512 channels, 1 .. 253 filters, 5 x 5 to 800 x 1300): a pass over the channels and a round of CTAs over
// the SMs, both in proportion to the channels.
double direct_estimate_us(const DirectLayout& D, int N, int H, int W) {
  const int64_t sms = device_sms();
  if (sms <= 0) return 0.0;
  const Plan pl = make_plan(D, N, H, W, (W & 3) == 0, sms);
  if (pl.wide) return 2.2 + D.Ci / 64.0 * pl.wide_us;
  static const double pass_us[3] = {0.7, 4.0, 3.0};  // 64 channels, by groups (1, 2, 4)
  // by filters (2, 4, 8), groups, rows of whole 16-byte groups or not
  static const double round_us[3][3][2] = {{{10.1, 16.3}, {4.6, 6.6}, {2.5, 3.6}},
                                           {{15.3, 20.6}, {8.3, 10.4}, {4.5, 5.7}},
                                           {{27.3, 32.0}, {14.2, 16.6}, {8.2, 9.6}}};
  const int f = pl.fbd == 2 ? 0 : pl.fbd == 4 ? 1 : 2, k = pl.ks == 4 ? 2 : pl.ks - 1;
  return 2.2 + ((D.Ci + 3) / 4) / 16.0 *
                   (pass_us[k] + (double)((pl.grid + sms - 1) / sms) * round_us[f][k][(W & 3) ? 1 : 0]);
}

pp_status direct_launch(const DirectLayout& D, const float* x, float* y, const float* skip, int N, int H, int W,
                        int flags, cudaStream_t stream) {
  if (!D.w) return PP_ERR_UNSUPPORTED;
  const int64_t sms = device_sms();
  if (sms <= 0) return PP_ERR_CUDA;
  DirectParams p;
  p.x = x;
  p.y = y;
  p.skip = (flags & PP_ADD_SKIP) ? skip : nullptr;
  p.w = D.w;
  p.bias = D.bias;
  p.wdup = D.wdup;
  p.status = D.status;
  p.redo = D.redo;
  p.N = N;
  p.Ci = D.Ci;
  p.Co = D.Co;
  p.H = H;
  p.W = W;
  p.flags = flags;
  p.npair = D.npair;
  p.tiles_x = p.tiles_y = 0;
  p.vec = (W & 3) == 0 && ((uintptr_t)x & 15) == 0 && (int64_t)H * W <= INT32_MAX;
  const Plan pl = make_plan(D, N, H, W, p.vec, sms);
  const int64_t vt = pl.vt;
  const bool wide = pl.wide;
  const int fbd = pl.fbd, ks = pl.ks;
  const auto ctas = [&](int th, int tw, int f) { return tiles(D, N, H, W, th, tw, f); };
  cudaError_t e;
  if (wide && D.Co == 1) {
    e = vt >= (p.vec ? 2 : 1) * sms ? launch_wide<1, 1>(p, stream)
                                    : vt > sms ? launch_wide<1, 2>(p, stream) : launch_wide<1, 4>(p, stream);
  } else if (wide && D.Co == 2) {
    e = launch_wide<2, 1>(p, stream);
  } else if (wide) {
    e = vt >= 2 * sms ? launch_wide<3, 1>(p, stream) : launch_wide<3, 2>(p, stream);
  } else if (D.Ci <= 4 && W > UW / 2 && D.Co > 4 && D.Co <= 65535 && ctas(UH, UW, FBMAX) >= sms / 2 &&
             10 * ((W + UW - 1) / UW * UW) < 13 * ((W + 31) / 32 * 32)) {
    // (1 -> 64 at 720 x 1280 48 us against 86 with the 32 x 32 tiles, 3 -> 64 at 224 x 224 7.2 against 9.1; below half
    // a CTA per SM the smaller tiles win: 1 -> 64 at 64 x 96, 64 CTAs, 3.0 against 2.7; where its rows of 128 pixels are
    // 1.3 times the columns that the others pad to, or more, these: 4 -> 64 at 625 x 160, batch 2, 52 against 33, 1 -> 16
    // at 666 x 150 8.7 against 6.7)
    int fpc = UFMAX;
    while (fpc > FBMAX && ctas(UH, UW, fpc) < 2 * sms) fpc /= 2;
    switch (D.Ci) {
      case 1: e = launch_first<1>(p, fpc, stream); break;
      case 2: e = launch_first<2>(p, fpc, stream); break;
      case 3: e = launch_first<3>(p, fpc, stream); break;
      default: e = launch_first<4>(p, fpc, stream); break;
    }
  } else {
    if (D.Ci <= 4) {
      switch (D.Ci) {
        case 1: e = launch_fbd<1, 1>(p, fbd, stream); break;
        case 2: e = launch_fbd<2, 1>(p, fbd, stream); break;
        case 3: e = launch_fbd<3, 1>(p, fbd, stream); break;
        default: e = launch_fbd<4, 1>(p, fbd, stream); break;
      }
    } else {
      e = ks == 1 ? launch_fbd<4, 1>(p, fbd, stream)
                  : ks == 2 ? launch_fbd<4, 2>(p, fbd, stream) : launch_fbd<4, 4>(p, fbd, stream);
    }
  }
  if (e == cudaErrorInvalidConfiguration) {
    cudaGetLastError();
    return PP_ERR_UNSUPPORTED;
  }
  if (e != cudaSuccess) {
    cudaGetLastError();
    return PP_ERR_CUDA;
  }
  return PP_OK;
}

void direct_free(DirectLayout* D) {
  if (D->dmem) cudaFree(D->dmem);
  *D = DirectLayout();
}

}  // namespace ppc
