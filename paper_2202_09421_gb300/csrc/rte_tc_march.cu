// Several AB4 steps of every group in one launch (tensor-core passes).
//
// The two passes of a step stay what they are (rte_tc.cu), but their slab
// tiles are items of one persistent launch instead of two grids: CTAs take
// items by a ticket, in an order that puts the y items of a group right
// behind the x items of the next group, step after step, and items wait for
// what they read on per-group counters in global memory:
//   x item (s, g)   u^s of the group: every y item (s - 1, g);
//   y item (s, g)   u^s before its main loop (as above), and R before its
//                   epilogue: every x item (s, g).
// A ticket is taken by a CTA that is running, its roles work their items off
// in ticket order, and an item waits only for items with smaller tickets: the
// unfinished item with the smallest ticket can always proceed, however many
// of the launch's CTAs run at a time.  Every wait is bounded.
//
// u^{s+1} goes where R was: the y epilogue reads an element of R and writes
// that element of u^{s+1} over it, so two buffers alternate, nothing is
// updated in place while other items read it, and a column tile can be split
// over its output rows.
//
// One CTA per SM; its roles run on separate warps and hand work over through
// mbarriers:
//   warp 13, one lane   takes the tickets and copies the operator units (128
//                       output positions x one K chunk, hi and lo) into a
//                       ring;
//   warps 8-11          convert the slab: a thread owns four neighbouring
//                       slab columns, loads their values two pieces ahead
//                       into registers, scales, splits and writes its part of
//                       the K-major operand chunk;
//   warp 12, one lane   issues the MMAs into one of two accumulators in
//                       tensor memory;
//   warps 0-7           the epilogue of the item before (x_epilogue,
//                       y_epilogue);
//   warp 14, one lane   counts an item as done once its writes are visible
//                       (the fence takes over a microsecond).
// So the tensor cores work on one item while the previous one is finished.
//
// What bounds it: at 16 groups of 256^2 (M = 32, 3xTF32) the memory traffic of
// the y epilogues (36 B an update measured, 24 needed) and the epilogue warps'
// issue slots together; with one or two groups the chain of an item, whose
// slowest are the tiles with an x-face column (every row of theirs waits for
// its reflected ordinates).  Time per step against the two launches per step
// of rte_tc.cu, 3xTF32 at 256^2: one group 81 -> 46 us, four 113 -> 94,
// sixteen 355 -> 278 (318 with the TMA-fed x-pass); bf16x3 at 512^2, M = 64,
// 359 -> 287; TF32 at 200 x 131, three groups, 50 -> 44.
#include <cstdint>

#include "rte_tc_common.cuh"

namespace rte_kern {

namespace {

using namespace tc;

constexpr int kEpiWarps = 8, kCvtWarps = 4;
constexpr int kWarpMMA = kEpiWarps + kCvtWarps, kWarpCopy = kWarpMMA + 1, kWarpSignal = kWarpCopy + 1;
constexpr int kMarchThreads = (kWarpSignal + 1) * 32;
// The copying warp is at most ten items ahead of the signal warp (items of a
// single unit: four in its ring, two accumulators, and two by the signals),
// so a slot of the item ring is read before it is written again.
constexpr int kItemRing = 16;
// Groups that the x items are ahead of the y items within a step (256^2, 16
// groups: 278 us a step with 5, 280 with 3, 295 with 1).
constexpr int kMarchLag = 5;

constexpr int kMaxM = 64;
constexpr int kMaxD = 4;                                       // ring slots, at most
// y-pass epilogue: per warp a ring of two pairs of rows of 5 arrays, per CTA
// a [16][128] accumulator tile and the boundary tables of BcTables.  The
// x-pass epilogue keeps its 8 KB of node values per warp at the warp's place
// of that ring, so that a warp may go on to another item on its own.
constexpr int kYPair = 2 * 5 * 512;                            // bytes of a warp's two rows
constexpr int kYWarpBytes = 2 * kYPair;                        // 10 KB
constexpr size_t kYRingBytes = static_cast<size_t>(kEpiWarps) * kYWarpBytes;
constexpr size_t kYTileBytes = 16 * kNC * 4;
constexpr size_t kBcTabBytes = kMaxM * (8 * 8 + 4 * 4);
constexpr size_t kEpiBytes = kYRingBytes + kYTileBytes + kBcTabBytes;

// Bounded wait (kWaitNs of wall clock); false, and the timeout word set,
// when the limit runs out.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, int* err) {
  const unsigned long long t0 = global_ns();
  while (!mbar_try(bar, parity))
    if (global_ns() - t0 > kWaitNs) {
      atomicExch(err, 1);
      return false;
    }
  return true;
}

// The MMAs of one operator unit (128 output positions x one K chunk of a
// 128-byte row) against the slab chunk, into the accumulator of its row tile.
// idesc: D = F32, A = B = TF32 (2) or BF16 (1), K-major, M = 128; N = 128
// slab columns (x-pass: A is the operator) or the unit's rows (y-pass: A is
// the slab).  One thread.
template <bool XPASS, bool BF, bool X3>
__device__ __forceinline__ void issue_unit_mmas(unsigned char* unit, uint64_t dSh, uint64_t dSl, uint32_t acc,
                                                int rows, bool first) {
  constexpr uint32_t kFmt = BF ? 1u : 2u;
  const uint32_t idesc = (1u << 4) | (kFmt << 7) | (kFmt << 10) | (static_cast<uint32_t>(kMT >> 4) << 24) |
                         (static_cast<uint32_t>((XPASS ? kNC : rows) >> 3) << 17);
  const uint64_t dDh = sw128_desc(smem_u32(unit)), dDl = sw128_desc(smem_u32(unit + kTileBytes));
#pragma unroll
  for (int kk = 0; kk < 4; ++kk) {
    const uint64_t o = static_cast<uint64_t>(kk * 2);   // 32 bytes per K step
    const uint32_t accumulate = (!first || kk > 0) ? 1u : 0u;
    if (XPASS) {
      mma<BF>(acc, dDh + o, dSh + o, idesc, accumulate);
      if (X3) {
        mma<BF>(acc, dDh + o, dSl + o, idesc, 1u);
        mma<BF>(acc, dDl + o, dSh + o, idesc, 1u);
      }
    } else {
      mma<BF>(acc, dSh + o, dDh + o, idesc, accumulate);
      if (X3) {
        mma<BF>(acc, dSh + o, dDl + o, idesc, 1u);
        mma<BF>(acc, dSl + o, dDh + o, idesc, 1u);
      }
    }
  }
}

// x-pass epilogue of an item, warps 0..7 (each on its own): R = b P~u -
// (a + b) u + acc on the nodes of grid rows t0 .. t0 + 128/M - 1 and output
// tiles row0/128 .. + nrt.  sm_epi: the epilogues' shared memory; released()
// is called by every lane after the warp's last tensor-memory load.
template <int MM, class Released>
__device__ __forceinline__ void x_epilogue(const StepArgs& a, const float* U, float* R, size_t goff, int t0, int row0,
                                           int nrt, const float* pcs, uint32_t tmem, unsigned char* sm_epi, int warp,
                                           int lane, Released&& released) {
  constexpr int M = MM;
  constexpr int per_tile = kNC / M;
  const int nx = a.nx, ny = a.ny;
  const int quarter = warp & 3, half = warp >> 2;
  const uint64_t pol_keep = policy_evict_last();
  // lane = output position i, columns = (row, m).  The (tile t, row rc)
  // pairs of the item, p = t * per_tile + rc, alternate between warps 0-3
  // and warps 4-7; warp w reads TMEM lanes 32 (w % 4) ...  A pair is 32
  // consecutive nodes of a grid row, one contiguous run of memory: it is
  // copied to and from shared memory in 16-byte pieces by consecutive lanes
  // (whole lines per request; a lane reading its own node's 128 B in place
  // takes a request of 32 lines per piece), and the lanes read and write
  // their nodes there, the pieces of node k rotated by k against bank
  // conflicts.
  constexpr int V = M / 4;                                     // 16-byte pieces per node
  constexpr int kXBuf = M == 64 ? 1 : 2;                       // pairs in shared memory per warp
  constexpr int kPairBytes = 32 * M * 4;
  unsigned char* xb = sm_epi + warp * kYWarpBytes;
  const int n_pairs = nrt * per_tile;
  const uint32_t tq = tmem + (static_cast<uint32_t>(32 * quarter) << 16);
  auto piece = [&](int node, int v) {
    const int key = M == 16 ? (node >> 1) & 3 : node & 7;
    return node * (M * 4) + ((v ^ key) << 4);
  };
  auto pair_base = [&](int p, int& i0, int& j) {
    const int t = p / per_tile, rc = p - t * per_tile;
    i0 = row0 + t * kMT + 32 * quarter;
    j = t0 + rc;
    return p < n_pairs && i0 < nx && j < ny;
  };
  auto fetch = [&](int p, int slot) {
    int i0, j;
    if (pair_base(p, i0, j)) {
      const float* src = U + goff + (static_cast<size_t>(j) * nx + i0) * M;
      const int nodes = min(32, nx - i0);
#pragma unroll
      for (int k = 0; k < V; ++k) {
        const int e = lane + 32 * k, node = e / V, v = e - node * V;
        if (node < nodes)
          asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                           smem_u32(xb + slot * kPairBytes + piece(node, v))),
                       "l"(src + 4 * e)
                       : "memory");
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  // b and a + b of the lane's node, one pair ahead like the node values
  auto fetch_ab = [&](int p, float& ab, float& bb) {
    int i0, j;
    ab = bb = 0.f;
    if (pair_base(p, i0, j) && i0 + lane < nx) {
      const size_t cell = static_cast<size_t>(j) * nx + i0 + lane;
      bb = __ldg(a.mus + cell);
      ab = __ldg(a.mua + cell);
    }
  };
  fetch(half, 0);
  float a_next, b_next;
  fetch_ab(half, a_next, b_next);
  int slot = 0;
  for (int p = half; p < n_pairs; p += 2) {
    int i0, j;
    const bool any = pair_base(p, i0, j);                      // warp-uniform
    const int t = p / per_tile, rc = p - t * per_tile;
    if (kXBuf == 2) fetch(p + 2, slot ^ 1);
    const int nodes = min(32, nx - i0);
    const float bb = b_next, ab = a_next + b_next;
    fetch_ab(p + 2, a_next, b_next);
    if (kXBuf == 2)
      asm volatile("cp.async.wait_group 1;" ::: "memory");
    else
      asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncwarp();
    unsigned char* nb = xb + slot * kPairBytes;
    float uu[M];
#pragma unroll
    for (int v = 0; v < V; ++v) {
      const float4 u4 = *reinterpret_cast<const float4*>(nb + piece(lane, v));
      uu[4 * v] = u4.x; uu[4 * v + 1] = u4.y; uu[4 * v + 2] = u4.z; uu[4 * v + 3] = u4.w;
    }
    if constexpr (M == 64) {
      // 64 ordinates: the outputs in halves of 32, P~[k][0] from shared
      // memory (one broadcast value per k)
#pragma unroll 1
      for (int h = 0; h < 2; ++h) {
        float sc[32];
#pragma unroll
        for (int m = 0; m < 32; ++m) sc[m] = 0.f;
#pragma unroll
        for (int k = 0; k < M; ++k) {
          const float pk = pcs[k];
#pragma unroll
          for (int m = 0; m < 32; ++m) sc[m] = fmaf(pk, uu[(m - k + M) % M], sc[m]);
        }
#pragma unroll
        for (int gq = 0; gq < 2; ++gq) {
          float acc[16];
          tmem_ld16(tq + t * kNC + rc * M + 32 * h + 16 * gq, acc);
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const int m = 16 * gq + 4 * e;
            *reinterpret_cast<float4*>(nb + piece(lane, 8 * h + m / 4)) =
                make_float4(fmaf(bb, sc[m], acc[4 * e] - ab * uu[m]),
                            fmaf(bb, sc[m + 1], acc[4 * e + 1] - ab * uu[m + 1]),
                            fmaf(bb, sc[m + 2], acc[4 * e + 2] - ab * uu[m + 2]),
                            fmaf(bb, sc[m + 3], acc[4 * e + 3] - ab * uu[m + 3]));
          }
        }
        // the second half works on the ordinates rotated by 32
#pragma unroll
        for (int m = 0; m < 32; ++m) {
          const float x = uu[m];
          uu[m] = uu[m + 32];
          uu[m + 32] = x;
        }
      }
    } else {
      float acc[M];
      tmem_ld16(tq + t * kNC + rc * M, acc);
      if (M > 16) tmem_ld16(tq + t * kNC + rc * M + 16, acc + (M > 16 ? 16 : 0));
      xpass_node_rhs<M, false>(acc, uu, pcs, ab, bb);
#pragma unroll
      for (int v = 0; v < V; ++v)
        *reinterpret_cast<float4*>(nb + piece(lane, v)) =
            make_float4(acc[4 * v], acc[4 * v + 1], acc[4 * v + 2], acc[4 * v + 3]);
    }
    __syncwarp();
    if (any) {
      float* dst = R + goff + (static_cast<size_t>(j) * nx + i0) * M;
#pragma unroll
      for (int k = 0; k < V; ++k) {
        const int e = lane + 32 * k, node = e / V, v = e - node * V;
        if (node < nodes)                                      // R is read by the y-pass that follows
          st_hint(dst + 4 * e, *reinterpret_cast<const float4*>(nb + piece(node, v)), pol_keep);
      }
    }
    __syncwarp();                                              // the slot may be refilled
    if (kXBuf == 2) slot ^= 1;
    else fetch(p + 2, 0);
  }
  released();
}

// Boundary tables of the y epilogue in shared memory: faces 0..3, corners
// 4..7.  An entry holds the factor and the reflected ordinate (its own, and
// the sign bit set, where nothing is imposed), so that an ordinate is one
// load and one dependent load, without a branch.
struct BcTables {
  int2* e;                   // [8][M]: factor's bits, reflected ordinate
  float* wexit;              // [4][M]
  __device__ __forceinline__ BcTables(unsigned char* sm_epi, int M) {
    e = reinterpret_cast<int2*>(sm_epi + kYRingBytes + kYTileBytes);
    wexit = reinterpret_cast<float*>(e + 8 * M);
  }
  // filled by n_thr threads; the caller synchronises
  __device__ __forceinline__ void fill(const BoundaryArgs& b, int M, int t, int n_thr) const {
    for (int k0 = t; k0 < 8 * M; k0 += n_thr) {
      const bool face = k0 < 4 * M;
      const int k = face ? k0 : k0 - 4 * M;
      const bool act = (face ? b.face_act[k] : b.corner_act[k]) != 0;
      e[k0] = make_int2(__float_as_int(face ? b.face_f[k] : b.corner_f[k]),
                        act ? (face ? b.face_refl[k] : b.corner_refl[k]) : static_cast<int>(0x80000000u | (k % M)));
      if (face) wexit[k0] = b.wexit[k];
    }
  }
};

// sum_m we_m x_m of a node whose M ordinates lie on M / 4 adjacent lanes, four
// each: every lane's four in order, then the lanes pairwise (all lanes of a
// converged warp; the sum in each lane of the node).
template <int M>
__device__ __forceinline__ float exitance_sum(const float* we, const float* x) {
  float ex = we[0] * x[0];
#pragma unroll
  for (int e = 1; e < 4; ++e) ex = fmaf(we[e], x[e], ex);
#pragma unroll
  for (int o = 1; o < M / 4; o <<= 1) ex += __shfl_xor_sync(0xffffffffu, ex, o);
  return ex;
}

// y-pass epilogue of an item, warps 0..7: L^k = R + acc, AB4, the boundary
// nodes.  u^{k+1} goes over R.  sync(): a barrier of the eight warps;
// released() as in x_epilogue.
template <int MM, class Sync, class Released>
__device__ __forceinline__ void y_epilogue(const StepArgs& a, const BoundaryArgs& b, const float* U, float* R,
                                           const float* L1, const float* L2, float* L3, size_t goff, int step, int g,
                                           int t0, int row0, int nrt, uint32_t tmem, unsigned char* sm_epi, int warp,
                                           int lane, Sync&& sync, Released&& released) {
  constexpr int M = MM;
  constexpr int per_tile = kNC / M;
  const int nx = a.nx, ny = a.ny;
  const int half = warp >> 2;
  const uint64_t pol_keep = policy_evict_last();
  // acc[lane = slab column c][column = output row j].  The rows are worked off
  // in blocks of sixteen, two rows per warp at a time (one hides the other's
  // latency): lane l has the 16-byte piece l of a row's 128 columns, so that a
  // request is 512 contiguous bytes (pieces of 128 B per row, with the four
  // column quarters on different warps, measured slower at the DRAM).  A warp
  // streams u, R, L1, L2, L3 of its rows through a private ring (cp.async, one
  // block ahead; a lane reads back what it copied).  The accumulator of a
  // block passes through a [16][128] tile: every warp loads its part of the
  // next block into registers before it works on this one and stores it
  // between two barriers.  The nodes of a row lie within its warp: the
  // boundary condition (eq. RTE third line) reads the reflected ordinates from
  // the row's place in the tile, and the exitance (eq. OpMed) is summed over
  // each lane's four ordinates, then over the node's lanes.
  unsigned char* ring = sm_epi + warp * kYWarpBytes;
  float* tile = reinterpret_cast<float*>(sm_epi + kYRingBytes);     // [16][128]
  const int ring_len = 2 * ny + 2 * nx;
  const int rows_item = min(nrt * kMT, ny - row0);
  const int nblk = (rows_item + 15) / 16;
  const int c = lane * 4, w = c / M, m0 = c - w * M, i = t0 + w;
  const bool col_ok = i < nx, lf = i == 0, rt = i == nx - 1;
  const bool x_tile = t0 == 0 || t0 + per_tile >= nx;          // the tile has an x-face column
  const uint32_t rs = static_cast<uint32_t>(nx) * M;           // row stride; a group's plane has under 2^25 values
  // this lane's place in the warp's first row (16 blk + 2 warp) of block 0
  const size_t base = goff + static_cast<size_t>(row0 + 2 * warp) * rs + static_cast<uint32_t>(t0) * M + c;
  const float *Ub = U + base, *L1b = L1 + base, *L2b = L2 + base;
  float *Rb = R + base, *L3b = L3 + base;
  const int rows_left = col_ok ? ny - row0 - 2 * warp : 0;     // valid: 16 blk + r < rows_left
  const uint64_t pol_once = policy_evict_first();
  const uint32_t ring_s = smem_u32(ring) + lane * 16;
  auto issue = [&](int blk) {
    if (blk < nblk) {
#pragma unroll
      for (int r = 0; r < 2; ++r)
        if (16 * blk + r < rows_left) {
          const uint32_t o = static_cast<uint32_t>(16 * blk + r) * rs;
          const uint32_t dst = ring_s + (blk & 1) * kYPair + r * 2560;
          const float* srcs[5] = {Ub, Rb, L1b, L2b, L3b};
#pragma unroll
          for (int arr = 0; arr < 5; ++arr)
            asm volatile("cp.async.cg.shared.global.L2::cache_hint [%0], [%1], 16, %2;" ::"r"(dst + arr * 512),
                         "l"(srcs[arr] + o), "l"(pol_once)
                         : "memory");
        }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  // warp w holds TMEM lanes 32 (w % 4) ..; warps 0-3 take the block's first
  // eight rows, warps 4-7 the others
  const uint32_t tbase = tmem + (static_cast<uint32_t>(32 * (warp & 3)) << 16) + 8 * half;
  float* tdst = tile + 8 * half * kNC + 32 * (warp & 3) + lane;
  uint32_t ar[8];
  auto tile_load = [&](int blk) {
    __syncwarp();
    tmem_ld8_async(tbase + blk * 16, ar);
  };
  auto tile_store = [&]() {
    __syncwarp();
    tmem_ld8_wait(ar);
#pragma unroll
    for (int t = 0; t < 8; ++t) tdst[t * kNC] = __uint_as_float(ar[t]);
  };
  const BcTables tab(sm_epi, M);
  issue(0);
  sync();                                                      // the tile's readers of an item before are done
  tile_load(0);
  tile_store();
  sync();
  for (int blk = 0; blk < nblk; ++blk) {
    issue(blk + 1);
    if (blk + 1 < nblk) tile_load(blk + 1);
    const int j0 = row0 + 16 * blk + 2 * warp;                 // the warp's first row of the block
    const bool bc_blk = x_tile || j0 == 0 || (j0 <= ny - 1 && j0 + 1 >= ny - 1);   // warp-uniform: boundary nodes
    asm volatile("cp.async.wait_group 1;" ::: "memory");
    const float* buf = reinterpret_cast<const float*>(ring + (blk & 1) * kYPair) + c;
    float* row = tile + 2 * warp * kNC;
    float4 v[2], hn[2];                                        // u^{k+1}, L^k
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const float4 u4 = *reinterpret_cast<const float4*>(buf + r * 640);
      const float4 r4 = *reinterpret_cast<const float4*>(buf + r * 640 + 128);
      const float4 p4 = *reinterpret_cast<const float4*>(buf + r * 640 + 256);
      const float4 q4 = *reinterpret_cast<const float4*>(buf + r * 640 + 384);
      const float4 s4 = *reinterpret_cast<const float4*>(buf + r * 640 + 512);
      const float4 ac = *reinterpret_cast<const float4*>(row + r * kNC + c);
      hn[r] = make_float4(r4.x + ac.x, r4.y + ac.y, r4.z + ac.z, r4.w + ac.w);
      v[r].x = ab4_node(a.cdt, hn[r].x, p4.x, q4.x, s4.x, u4.x);
      v[r].y = ab4_node(a.cdt, hn[r].y, p4.y, q4.y, s4.y, u4.y);
      v[r].z = ab4_node(a.cdt, hn[r].z, p4.z, q4.z, s4.z, u4.z);
      v[r].w = ab4_node(a.cdt, hn[r].w, p4.w, q4.w, s4.w, u4.w);
    }
    if (bc_blk) {
#pragma unroll
      for (int r = 0; r < 2; ++r) *reinterpret_cast<float4*>(row + r * kNC + c) = v[r];
      __syncwarp();
#pragma unroll 1
      for (int r = 0; r < 2; ++r) {
        const int jj = j0 + r;
        const bool bt = jj == 0, tp = jj == ny - 1;
        const bool bnd = col_ok && jj < ny && (lf || rt || bt || tp);
        const bool corner = (lf || rt) && (bt || tp);
        const int tb = corner ? 4 + (rt ? 1 : 0) + (tp ? 2 : 0) : (lf ? 0 : rt ? 1 : bt ? 2 : 3);
        const float* rw = row + r * kNC;
        const float4 h = r == 0 ? v[0] : v[1];
        float x[4] = {h.x, h.y, h.z, h.w};
        if (bnd) {
          const int node = lf ? jj : rt ? ny + jj : bt ? 2 * ny + i : 2 * ny + nx + i;
          float q[4] = {0.f, 0.f, 0.f, 0.f};
          for (int k = 0; k < b.kmax; ++k) {
            const size_t gk = static_cast<size_t>(g) * b.kmax + k;
            const float sk = __ldg(b.S + gk * ring_len + node), tk = __ldg(b.T + gk * b.T_len + step);
            const float4 ak = __ldg(reinterpret_cast<const float4*>(b.A + gk * M + m0));
            q[0] = fmaf(sk * ak.x, tk, q[0]);
            q[1] = fmaf(sk * ak.y, tk, q[1]);
            q[2] = fmaf(sk * ak.z, tk, q[2]);
            q[3] = fmaf(sk * ak.w, tk, q[3]);
          }
          const float rho =
              b.rho ? __ldg(b.rho + (static_cast<size_t>(g) * b.rho_len + step) * ring_len + node) : 0.f;
            const int4* te = reinterpret_cast<const int4*>(tab.e + tb * M + m0);
            const int4 t01 = te[0], t23 = te[1];
            const int fb[4] = {t01.x, t01.z, t23.x, t23.z}, rf[4] = {t01.y, t01.w, t23.y, t23.w};
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              const float fco = __int_as_float(fb[e]);
              if (b.rho) q[e] = fmaf(1.0f - fco, rho, q[e]);
              const float z = fmaf(fco, rw[w * M + (rf[e] & 0x7fffffff)], q[e]);
              x[e] = rf[e] >= 0 ? z : x[e];
            }
        }
        if (b.ring_out) {
          float* ro = b.ring_out + (static_cast<size_t>(g) * b.ring_steps + step) * ring_len;
          if (x_tile) {                                        // warp-uniform, as bt and tp are
            const float ex = exitance_sum<M>(tab.wexit + (lf ? 0 : 1) * M + m0, x);
            if (bnd && (lf || rt) && m0 == 0) ro[lf ? jj : ny + jj] = ex;
          }
          if (bt || tp) {
            const float ex = exitance_sum<M>(tab.wexit + (bt ? 2 : 3) * M + m0, x);
            if (bnd && m0 == 0) ro[bt ? 2 * ny + i : 2 * ny + nx + i] = ex;
          }
        }
        const float4 o = make_float4(x[0], x[1], x[2], x[3]);
        if (r == 0) v[0] = o;
        else v[1] = o;
      }
    }
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      if (16 * blk + r < rows_left) {
        const uint32_t o = static_cast<uint32_t>(16 * blk + r) * rs;
        *reinterpret_cast<float4*>(L3b + o) = hn[r];
        st_hint(Rb + o, v[r], pol_keep);                       // read by the next x-pass
      }
    }
    if (blk + 1 < nblk) {
      sync();                                                  // every warp is done with the tile
      tile_store();
      sync();                                                  // the next block's tile is there
    }
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  released();
}

// Item counts of a march step, and the item behind a ticket.
struct MarchItems {
  int G, rt, lag;                    // groups; 128-row output tiles per item; see Item
  int px, py;                        // row parts of a tile (x, y)
  int nxi, nyi;                      // items per group and step (x, y)
  __host__ __device__ MarchItems(const StepArgs& a, int rt_, int lag_) : G(a.G), rt(rt_) {
    const int per_tile = kNC / a.M;
    const int mtx = (a.nx + kMT - 1) / kMT, mty = (a.ny + kMT - 1) / kMT;
    px = (mtx + rt - 1) / rt;
    py = (mty + rt - 1) / rt;
    nxi = (a.ny + per_tile - 1) / per_tile * px;
    nyi = (a.nx + per_tile - 1) / per_tile * py;
    lag = lag_ < G ? lag_ : G;
  }
  __host__ __device__ int per_step() const { return G * (nxi + nyi); }
};

struct Item {
  bool xpass;
  int s, g, tile, rt0, nrt, n, n_kc;
  // step order: x(0), .., x(lag - 1); x(lag), y(0); ..; x(G - 1), y(G - 1 -
  // lag); y(G - lag), .., y(G - 1)
  __device__ __forceinline__ Item(const MarchItems& it, const StepArgs& a, int kc, int ticket) {
    s = ticket / it.per_step();
    int r = ticket - s * it.per_step(), idx;
    const int head = it.lag * it.nxi, body = (it.G - it.lag) * (it.nxi + it.nyi);
    if (r < head) {
      xpass = true;
      g = r / it.nxi;
      idx = r - g * it.nxi;
    } else if (r < head + body) {
      r -= head;
      const int pair = r / (it.nxi + it.nyi);
      r -= pair * (it.nxi + it.nyi);
      xpass = r < it.nxi;
      g = xpass ? it.lag + pair : pair;
      idx = xpass ? r : r - it.nxi;
    } else {
      r -= head + body;
      xpass = false;
      g = r / it.nyi;
      idx = r - g * it.nyi;
      g += it.G - it.lag;
    }

    const int parts = xpass ? it.px : it.py;
    tile = idx / parts;
    rt0 = (idx - tile * parts) * it.rt;
    n = xpass ? a.nx : a.ny;
    nrt = min(it.rt, (n + kMT - 1) / kMT - rt0);
    n_kc = (n + kc - 1) / kc;
  }
  // rows of operator unit t: rows past the line are not copied (they only
  // feed accumulator rows that nobody reads)
  __device__ __forceinline__ int unit_rows(int t) const { return min(kMT, (n - (rt0 + t) * kMT + 15) & ~15); }
};

struct MarchShared {
  uint64_t d_full[kMaxD], d_empty[kMaxD], s_full[kMaxD], s_empty[kMaxD], acc_full[2], acc_empty[2], mma_done, epi_done[2], sig_done[2];
  uint64_t item_full[kItemRing];
  int item[kItemRing];
  uint32_t tmem_slot;
  int abort_flag;
  float pcs[kMaxM];
  BoundaryArgs pb, pb2;              // DUAL: of the two marches
};

// Bounded wait on an mbarrier; false when it, or any other wait of the CTA,
// gave up.
__device__ __forceinline__ bool m_wait(uint64_t* bar, uint32_t parity, volatile int* abort_flag, int* err) {
  const uint32_t addr = smem_u32(bar);
  const unsigned long long t0 = global_ns();
  while (!mbar_try(addr, parity)) {
    if (*abort_flag) return false;
    if (global_ns() - t0 > kWaitNs) {
      atomicExch(err, 1);
      *abort_flag = 1;
      return false;
    }
  }
  return true;
}

// Bounded wait, by a converged warp, until *p >= v: lane 0 polls.  False when
// the timeout word is set meanwhile or a wait of the CTA gave up.
__device__ __forceinline__ bool dep_wait(const int* p, int v, int lane, volatile int* abort_flag, int* err) {
  int fine = 1;
  if (lane == 0) {
    const unsigned long long t0 = global_ns();
    for (;;) {
      int c;
      asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(c) : "l"(p) : "memory");
      if (c >= v) break;
      if (*abort_flag || *static_cast<volatile int*>(err)) {
        *abort_flag = 1;
        fine = 0;
        break;
      }
      if (global_ns() - t0 > kWaitNs) {
        atomicExch(err, 1);
        *abort_flag = 1;
        fine = 0;
        break;
      }
      __nanosleep(20);
    }
  }
  fine = __shfl_sync(0xffffffffu, fine, 0);
  __syncwarp();
  return fine != 0;
}

// True in all of the eight epilogue warps if x is true in every thread of them.
__device__ __forceinline__ bool epi_all(bool x) {
  uint32_t r;
  asm volatile(
      "{\n.reg .pred p, q;\nsetp.ne.u32 p, %1, 0;\nbarrier.cta.red.and.pred q, 1, 256, p;\nselp.u32 %0, 1, 0, q;\n}\n"
      : "=r"(r)
      : "r"(x ? 1u : 0u)
      : "memory");
  return r != 0;
}

__device__ __forceinline__ void m_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

// Ring depths: units of 32 KB in the split forms, 16 KB in the others.
template <bool X3>
struct MarchRing {
  static constexpr int ND = X3 ? 2 : 4, NS = X3 ? 2 : 4;
  static constexpr int kUnit = (X3 ? 2 : 1) * kTileBytes;
  static constexpr int kStage = (ND + NS) * kUnit;            // 128 KB
};

// DUAL: two marches of one medium, a.G counting the groups of both, which
// alternate.
template <int PREC, int MM, bool DUAL>
__global__ void __launch_bounds__(kMarchThreads, 1) tc_march_kernel(MarchArgs ma) {
  using K = Kind<PREC>;
  constexpr bool X3 = K::X3, BF = K::BF;
  constexpr int KC = K::KC, GV = K::GV, M = MM;
  constexpr int per_tile = kNC / M;
  using Ring = MarchRing<X3>;
  constexpr int ND = Ring::ND, NS = Ring::NS, kUnit = Ring::kUnit;
  extern __shared__ __align__(1024) unsigned char smraw[];
  __shared__ __align__(8) MarchShared sh;
  const StepArgs& a = ma.a;
  // A launch after a timed-out one does nothing (the march reports the error).
  if (cta_timed_out(a.err)) return;
  const MarchItems it(a, ma.rt, ma.lag);         // (DUAL: a.G is doubled by the launcher)
  const int total = it.per_step() * ma.n_steps;
  const int acc_cols = it.rt * kMT, tmem_cols = 2 * acc_cols;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  unsigned char* sm = smraw + ((1024 - (smem_u32(smraw) & 1023)) & 1023);
  unsigned char* sm_d = sm;
  unsigned char* sm_s = sm + ND * kUnit;
  unsigned char* sm_epi = sm + Ring::kStage;
  if (tid == 0) {
    for (int k = 0; k < ND; ++k) {
      mbar_init(smem_u32(&sh.d_full[k]), 1);
      mbar_init(smem_u32(&sh.d_empty[k]), 1);
    }
    for (int k = 0; k < NS; ++k) {
      mbar_init(smem_u32(&sh.s_full[k]), kCvtWarps * 32);
      mbar_init(smem_u32(&sh.s_empty[k]), 1);
    }
    for (int k = 0; k < 2; ++k) {
      mbar_init(smem_u32(&sh.acc_full[k]), 1);
      mbar_init(smem_u32(&sh.acc_empty[k]), kEpiWarps);
      mbar_init(smem_u32(&sh.epi_done[k]), kEpiWarps);
      mbar_init(smem_u32(&sh.sig_done[k]), 1);
    }
    mbar_init(smem_u32(&sh.mma_done), 1);
    for (int k = 0; k < kItemRing; ++k) mbar_init(smem_u32(&sh.item_full[k]), 1);
    sh.abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if constexpr (DUAL) {
    if (tid == 0) {
      sh.pb = ma.b;
      sh.pb2 = ma.two.b;
    }
  }
  for (int k = tid; k < M; k += kMarchThreads) sh.pcs[k] = __ldg(a.PT + k);
  BcTables(sm_epi, M).fill(ma.b, M, tid, kMarchThreads);
  if (warp == kWarpCopy) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&sh.tmem_slot)),
                 "r"(tmem_cols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = sh.tmem_slot;
  volatile int* abrt = &sh.abort_flag;
  int* xdone = ma.ctl + 32;                    // [G]
  int* ydone = xdone + it.G;
  // side and group of an item's group (DUAL)
  auto side_of = [&](int gg) { return DUAL ? gg & 1 : 0; };
  auto group_of = [&](int gg) { return DUAL ? gg >> 1 : gg; };
  auto ubuf = [&](int gg, int k) {
    if constexpr (DUAL) {
      if (side_of(gg)) {
        if (ma.two.slots) return k == 0 ? ma.two.u0 : ma.two.slots + static_cast<size_t>(k - 1) * ma.two.slot_floats;
        return (k & 1) ? ma.two.u1 : ma.two.u0;
      }
    }
    if (ma.slots) return k == 0 ? ma.u0 : ma.slots + static_cast<size_t>(k - 1) * ma.slot_floats;
    return (k & 1) ? ma.u1 : ma.u0;
  };
  // The k-th item of this CTA (every role walks them in order); -1: no more,
  // or a wait gave up.
  auto next_item = [&](int k) {
    if (!m_wait(&sh.item_full[k % kItemRing], (k / kItemRing) & 1, abrt, a.err)) return -1;
    return *static_cast<volatile int*>(&sh.item[k % kItemRing]);
  };

  if (warp == kWarpCopy) {
    // ---------------- tickets and operator copies ----------------
    if (lane == 0) {
      int n = 0;
      bool fine = true;
      for (int k = 0; fine; ++k) {
        const int t = atomicAdd(ma.ctl, 1);
        // Failure injection (tests): the CTA of the first item waits on a
        // barrier that nothing arrives on, before it has issued any copy or
        // MMA; the bounded wait runs out and every role of every CTA leaves.
        if (a.test_expire && t == 0 && !m_wait(&sh.d_full[0], 0, abrt, a.err)) break;
        sh.item[k % kItemRing] = t < total ? t : -1;
        m_arrive(&sh.item_full[k % kItemRing]);
        if (t >= total) break;
        const Item im = Item(it, a, KC, t);
        const unsigned char* Dimg = static_cast<const unsigned char*>(im.xpass ? a.DxImg : a.DyImg);
        const size_t lo_off = static_cast<size_t>((im.n + kMT - 1) / kMT) * kTileBytes;   // lo rows of a chunk
        for (int q = 0; q < im.n_kc && fine; ++q)
          for (int u = 0; u < im.nrt; ++u, ++n) {
            const int slot = n % ND;
            if (!m_wait(&sh.d_empty[slot], ((n / ND) & 1) ^ 1, abrt, a.err)) {
              fine = false;
              break;
            }
            const unsigned char* src = Dimg + q * (2 * lo_off) + static_cast<size_t>(im.rt0 + u) * kTileBytes;
            const uint32_t dst = smem_u32(sm_d + slot * kUnit);
            bulk_copy2(dst, src, X3 ? dst + kTileBytes : 0u, src + lo_off, im.unit_rows(u) * 128,
                       smem_u32(&sh.d_full[slot]));
          }
      }
      // every copy issued has landed before the CTA leaves
      for (int k = 0; k < ND && k < n; ++k) {
        const int j = n - 1 - k;
        mbar_wait(smem_u32(&sh.d_full[j % ND]), (j / ND) & 1, a.err);
      }
    }
  } else if (warp == kWarpMMA) {
    // ---------------- MMA issue ----------------
    if (lane == 0) {
      int nd = 0, ns = 0;
      bool fine = true;
      for (int k = 0; fine; ++k) {
        const int t = next_item(k);
        if (t < 0) break;
        const Item im = Item(it, a, KC, t);
        const int b2 = k & 1;
        if (!m_wait(&sh.acc_empty[b2], ((k >> 1) & 1) ^ 1, abrt, a.err)) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t acc = tmem + b2 * acc_cols;
        for (int q = 0; q < im.n_kc && fine; ++q, ++ns) {
          const int sb = ns % NS;
          if (!m_wait(&sh.s_full[sb], (ns / NS) & 1, abrt, a.err)) {
            fine = false;
            break;
          }
          const uint64_t dSh = sw128_desc(smem_u32(sm_s + sb * kUnit)),
                         dSl = sw128_desc(smem_u32(sm_s + sb * kUnit + kTileBytes));
          for (int u = 0; u < im.nrt; ++u, ++nd) {
            const int slot = nd % ND;
            if (!m_wait(&sh.d_full[slot], (nd / ND) & 1, abrt, a.err)) {
              fine = false;
              break;
            }
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            if (im.xpass)
              issue_unit_mmas<true, BF, X3>(sm_d + slot * kUnit, dSh, dSl, acc + u * kMT, kMT, q == 0);
            else
              issue_unit_mmas<false, BF, X3>(sm_d + slot * kUnit, dSh, dSl, acc + u * kMT, im.unit_rows(u), q == 0);
            mma_commit(smem_u32(&sh.d_empty[slot]));
          }
          mma_commit(smem_u32(&sh.s_empty[sb]));
        }
        if (fine) mma_commit(smem_u32(&sh.acc_full[b2]));
      }
      // every MMA issued has completed before the tensor memory is freed
      mma_commit(smem_u32(&sh.mma_done));
      mbar_wait(smem_u32(&sh.mma_done), 0, a.err);
    }
  } else if (warp == kWarpSignal) {
    // ---------------- completion counts ----------------
    // (two barriers in turn; the epilogue waits for the count of item k - 2
    // before it arrives for item k, see there)
    if (lane == 0)
      for (int k = 0;; ++k) {
        const int t = next_item(k);
        if (t < 0) break;
        const Item im = Item(it, a, KC, t);
        if (!m_wait(&sh.epi_done[k & 1], (k >> 1) & 1, abrt, a.err)) break;
        m_arrive(&sh.sig_done[k & 1]);
        __threadfence();
        atomicAdd((im.xpass ? xdone : ydone) + im.g, 1);
      }
  } else if (warp >= kEpiWarps) {
    // ---------------- slab conversion ----------------
    // A thread owns four neighbouring slab columns (quad ct / 4: the same
    // grid line, four ordinates) and every fourth 16-byte group of their
    // operand rows: it loads 16 bytes of one position at a time and the
    // registers of a group, read across, are its operand rows.  (Lanes in
    // this order read whole lines and write without bank conflicts.)  A
    // piece is 32 values, a TF32 chunk or half a BF16 chunk; two pieces are
    // in flight.
    const int ct = tid - kEpiWarps * 32;
    const int c0 = (ct >> 2) * 4, kg = ct & 3;
    const int m = c0 % M;
    float scx[4], scy[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      scx[j] = -__ldg(a.xi + m + j);
      scy[j] = -__ldg(a.eta + m + j);
    }
    constexpr int kPieces = BF ? 2 : 1;                  // pieces per chunk
    constexpr int kGrp = 8 / GV;                         // groups per piece: 2 of 4 positions, 1 of 8
    const uint64_t pol_keep = policy_evict_last();
    int ns = 0;
    for (int k = 0;; ++k) {
      const int t = __shfl_sync(0xffffffffu, next_item(k), 0);
      if (t < 0) break;
      const Item im = Item(it, a, KC, t);
      // u^s is complete once every y item of the step before is
      if (im.s > 0 && !dep_wait(ydone + im.g, im.s * it.nyi, lane, abrt, a.err)) break;
      const int line = im.tile * per_tile + c0 / M;
      const bool col_ok = line < (im.xpass ? a.ny : a.nx);
      const size_t kstride = im.xpass ? M : static_cast<size_t>(a.nx) * M;
      const float* src = ubuf(im.g, im.s) + static_cast<size_t>(group_of(im.g)) * a.plane +
                         static_cast<size_t>(line) * (im.xpass ? static_cast<size_t>(a.nx) * M : M) + m;
      float sc[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) sc[j] = im.xpass ? scx[j] : scy[j];
      const int np = im.n_kc * kPieces;
      // group h of piece p: positions GV (grp_of(p, h)) + e of chunk p / kPieces
      auto grp_of = [&](int p, int h) { return kg + 4 * (BF ? p % kPieces : h); };
      auto load = [&](float4 (&v)[8], int p) {
#pragma unroll
        for (int h = 0; h < kGrp; ++h) {
          const int k0 = p / kPieces * KC + grp_of(p, h) * GV;
          const float* s0 = src + k0 * kstride;
#pragma unroll
          for (int e = 0; e < GV; ++e) {
            v[h * GV + e] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (col_ok && k0 + e < im.n) v[h * GV + e] = ld4_hint(s0 + e * kstride, pol_keep);
          }
        }
      };
      bool fine = true;
      auto convert = [&](float4 (&v)[8], int p) {
        const int sb = ns % NS;
        if (p % kPieces == 0) fine = m_wait(&sh.s_empty[sb], ((ns / NS) & 1) ^ 1, abrt, a.err);
        unsigned char* Shi = sm_s + sb * kUnit;
        unsigned char* Slo = Shi + kTileBytes;
#pragma unroll
        for (int h = 0; h < kGrp; ++h)
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const int off = sw128_off(c0 + j, grp_of(p, h));
            auto comp = [&](int e) {
              const float4& w = v[h * GV + e];
              return j == 0 ? w.x : j == 1 ? w.y : j == 2 ? w.z : w.w;
            };
            if constexpr (BF) {
              float col[8];
#pragma unroll
              for (int e = 0; e < 8; ++e) col[e] = comp(e);
              uint4 hi, lo;
              split8_bf16(col, sc[j], hi, lo);
              *reinterpret_cast<uint4*>(Shi + off) = hi;
              if (X3) *reinterpret_cast<uint4*>(Slo + off) = lo;
            } else {
              float4 hi, lo;
              split4(make_float4(comp(0), comp(1), comp(2), comp(3)), sc[j], hi, lo);
              *reinterpret_cast<float4*>(Shi + off) = hi;
              if (X3) *reinterpret_cast<float4*>(Slo + off) = lo;
            }
          }
        if (p % kPieces == kPieces - 1) {
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
          m_arrive(&sh.s_full[sb]);
          ++ns;
        }
      };
      float4 va[8], vb[8];
      load(va, 0);
      if (np > 1) load(vb, 1);
      for (int p = 0; p < np && fine; p += 2) {
        convert(va, p);
        if (p + 2 < np) load(va, p + 2);
        if (p + 1 < np && fine) {
          convert(vb, p + 1);
          if (p + 3 < np) load(vb, p + 3);
        }
      }
      if (!__all_sync(0xffffffffu, fine)) break;
    }
  } else {
    // ---------------- epilogue ----------------
    // The eight warps decide together (epi_all) whether to go on, so that
    // none is left waiting at the barriers of the y epilogue.
    auto epi_bargs = [&](int side) -> const BoundaryArgs& {
      if constexpr (DUAL) return side ? sh.pb2 : sh.pb;
      else return ma.b;
    };
    bool ok = true;
    for (int k = 0;; ++k) {
      const int t = __shfl_sync(0xffffffffu, next_item(k), 0);
      if (!epi_all(t >= 0 && ok)) break;
      const Item im = Item(it, a, KC, t);
      const int b2 = k & 1;
      const int side = side_of(im.g), lg = group_of(im.g);
      const size_t goff = static_cast<size_t>(lg) * a.plane;
      const float* U = ubuf(im.g, im.s);
      float* R = ubuf(im.g, im.s + 1);
      const uint32_t acc = tmem + b2 * acc_cols;
      const int t0 = im.tile * per_tile, row0 = im.rt0 * kMT;
      const int hl = ((DUAL && side ? ma.two.hl : ma.hl) + 2 * im.s) % 3;
      auto hist = [&](int q) {
        if constexpr (DUAL) return side ? ma.two.L[q] : ma.L[q];
        else return ma.L[q];
      };
      const float *L1 = hist(hl), *L2 = hist((hl + 1) % 3);
      float* L3 = hist((hl + 2) % 3);
      ok = m_wait(&sh.acc_full[b2], (k >> 1) & 1, abrt, a.err);
      __syncwarp();
      // y: R of this step is complete once every x item of the group is
      if (!im.xpass) ok = dep_wait(xdone + im.g, (im.s + 1) * it.nxi, lane, abrt, a.err) && ok;
      if (!epi_all(ok)) break;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      auto released = [&] {
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncwarp();
        if (lane == 0) m_arrive(&sh.acc_empty[b2]);
      };
      if (im.xpass) {
        x_epilogue<MM>(a, U, R, goff, t0, row0, im.nrt, sh.pcs, acc, sm_epi, warp, lane, released);
      } else {
        const int step = DUAL && side ? ma.two.step0 + im.s * ma.two.dstep : ma.step0 + im.s * ma.dstep;
        y_epilogue<MM>(a, epi_bargs(side), U, R, L1, L2, L3, goff, step, lg, t0, row0, im.nrt, acc,
                       sm_epi, warp, lane, [] { asm volatile("bar.sync 1, 256;" ::: "memory"); }, released);
      }
      // handed to the signal warp, which has taken item k - 2's phase
      if (k >= 2) ok = m_wait(&sh.sig_done[b2], ((k >> 1) - 1) & 1, abrt, a.err);
      ok = __all_sync(0xffffffffu, ok);                        // false: the next epi_all ends the loop
      if (ok && lane == 0) m_arrive(&sh.epi_done[b2]);
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == kWarpCopy)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(tmem_cols));
}

template <int PREC, int MM, bool DUAL>
cudaError_t launch_march_t(const MarchArgs& ma, int sms, cudaStream_t s) {
  constexpr size_t smem = 1024 + MarchRing<Kind<PREC>::X3>::kStage + kEpiBytes;
  static const cudaError_t attr = cudaFuncSetAttribute(
      tc_march_kernel<PREC, MM, DUAL>, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
  if (attr != cudaSuccess) return attr;
  const long long items = static_cast<long long>(MarchItems(ma.a, ma.rt, ma.lag).per_step()) * ma.n_steps;
  const int grid = items < sms ? static_cast<int>(items) : sms;
  tc_march_kernel<PREC, MM, DUAL><<<grid, kMarchThreads, smem, s>>>(ma);
  return cudaGetLastError();
}

template <int PREC, bool DUAL>
cudaError_t launch_march_m(const MarchArgs& ma, int sms, cudaStream_t s) {
  switch (ma.a.M) {
    case 16: return launch_march_t<PREC, 16, DUAL>(ma, sms, s);
    case 32: return launch_march_t<PREC, 32, DUAL>(ma, sms, s);
    default: return launch_march_t<PREC, 64, DUAL>(ma, sms, s);
  }
}

template <bool DUAL>
cudaError_t launch_march_p(const MarchArgs& ma, int sms, cudaStream_t s) {
  switch (ma.a.tc_mode) {
    case 1: return launch_march_m<1, DUAL>(ma, sms, s);
    case 2: return launch_march_m<2, DUAL>(ma, sms, s);
    case 3: return launch_march_m<3, DUAL>(ma, sms, s);
    default: return launch_march_m<4, DUAL>(ma, sms, s);
  }
}

// What a pass of all groups has to work off.
struct PassTiles {
  long long most, shorter;           // slab tiles: of either pass at most, of the pass along the shorter axis
  int lo, hi;                        // positions of the shorter and the longer axis
  bool pairs;                        // the one-tile passes hold two CTAs on an SM
  explicit PassTiles(const StepArgs& a) {
    const int per_tile = kNC / a.M;
    const long long tx = static_cast<long long>(a.G) * ((a.ny + per_tile - 1) / per_tile),
                    ty = static_cast<long long>(a.G) * ((a.nx + per_tile - 1) / per_tile);
    most = tx > ty ? tx : ty;
    shorter = a.nx < a.ny ? tx : ty;
    lo = a.nx < a.ny ? a.nx : a.ny;
    hi = a.nx < a.ny ? a.ny : a.nx;
    pairs = a.M < 64 && hi <= 256;
  }
};

// Whether the multi-step launches are faster than two one-tile passes a step.
// They gain where a pass is a chain (few tiles, many K chunks: the split
// products of 3xTF32) or holds one CTA per SM; they lose where the passes fill
// every SM with two CTAs and have little to do per tile: a short axis (its
// items are mostly latency, here one at a time per SM), a second row tile of a
// few rows, tiles that fit one wave of two per SM but not one of one.  The
// lines are drawn through times at 1010 random sizes (16 to 512 positions, 1
// to 24 groups, every precision and M), 40 steps in one run; the speed of the
// passes is 1:
//   taken: 696 sizes, geometric mean 1.25, 4 below 0.97 (the worst 0.94);
//   left:  0.41 to 1.36 (206 x 21, M = 32, 22 groups, BF16 66 us a step in the
//   passes, 130 here; 24 x 256, M = 16, 40 groups, 3xTF32 88 against 150;
//   260 x 24, M = 32, 16 groups, TF32 60 against 113; 130 x 130, M = 16, 16
//   groups, TF32 51 against 69), geometric mean 0.94.
bool march_pays(const StepArgs& a) {
  const PassTiles t(a);
  const int sms = device_sms();
  const bool x3tf32 = a.tc_mode == 1, bf16 = a.tc_mode == 4;
  const bool x_short = a.nx < a.ny;
  if (a.M == 16 && t.pairs && t.most > 2 * sms) return x3tf32 && t.lo >= 160;
  if (a.M == 64 && t.lo >= 96 && t.most > sms) return true;
  if (!bf16 && 4 * t.most <= sms) return true;
  if (x3tf32) {
    if (a.M == 64 && (t.hi > 256 || (t.lo >= 32 && t.most > sms))) return true;
    if (t.hi > 400) return t.shorter <= 8 * sms || t.lo >= 40;
    if (t.lo >= 64 || (t.lo >= 40 && t.shorter <= 8 * sms)) return t.hi >= 152 || 2 * t.most <= sms;
    return (t.shorter <= sms && t.hi >= 160) || (t.shorter <= (x_short ? 6 : 4) * sms && t.hi > 300);
  }
  if (t.hi < 152) return false;
  if (!bf16) {
    if (a.M == 64 && (t.hi > 300 || t.lo >= 40)) return true;
    if ((x_short && t.hi > 300) || (2 * t.most <= sms && (t.lo > 64 || t.hi > 256))) return true;
    if (t.hi > 360 && t.shorter <= sms) return true;
  }
  if (a.M == 32 && t.lo > kMT && t.most > 2 * sms) return true;
  if (t.lo >= 152) {
    const bool one_wave = t.pairs && t.most > sms && t.most <= 2 * sms && (a.M == 16 || bf16);
    return !one_wave && !(bf16 && a.M < 64 && t.hi > 256 && t.hi <= 300);
  }
  if (t.hi > 432 && t.lo >= 32 && (!bf16 || x_short)) return true;
  if (x_short && t.hi > 256) return t.lo >= 56 || t.shorter <= sms;
  return a.tc_mode == 2 && t.lo > kMT && t.hi >= 160 && t.most <= sms;
}

}  // namespace

bool tc_march_supported(const StepArgs& a) {
  if (a.tc_mode == 0 || a.tc_scatter != 0 || a.x_variant != 1 || (a.nx <= kMT && a.ny <= kMT)) return false;
  return a.march_all || march_pays(a);
}

int tc_march_min_run(const StepArgs& a) {
  // A launch's ramp is 6 to 40 us (its first x items and last y items by
  // themselves).  A run of one step pays where a pass leaves half of the SMs
  // idle anyway (256^2, one group, a snapshot at every step: 58 us a step
  // against 90 in the passes) or the passes hold one CTA per SM (512^2, M =
  // 64: 329 against 458); runs of two do in 3xTF32 (120 sizes: 1.23 of the
  // passes' speed on average), in the other precisions those of four (of two
  // beside passes with one CTA per SM, but not with BF16 operands: 257 x 206, M
  // = 64, ten groups, the balance of every step 574 us in the passes, 630 in
  // launches of two steps).
  if (a.march_all) return 1;
  const PassTiles t(a);
  if (2 * t.most <= device_sms()) return 1;
  if (a.tc_mode == 1) return t.pairs ? 2 : 1;
  return t.pairs || a.tc_mode == 4 ? 4 : 2;
}

bool tc_march_shares(const StepArgs& a) {
  // Three waves of 3xTF32 items: two and four solves on streams of their own,
  // us for a step of all, in the passes and in multi-step launches, 256^2, M =
  // 32: four groups 168, 306 and 189, 374; six 250, 457 and 238, 472; eight
  // 324, 607 and 284, 564; sixteen 605, 1205 and 553, 1101; 512^2, M = 32, two
  // groups 502, 982 and 442, 879; but 300^2, M = 64, four groups, bf16x3 654,
  // 1321 and 776, 1546, and 160^2, M = 32, sixteen groups 276, 515 and 285, 564.
  const PassTiles t(a);
  return a.tc_mode == 1 && a.M < 64 && t.lo > 192 && 2 * t.most >= (t.pairs ? 6 : 3) * device_sms();
}

bool tc_march_dual(const StepArgs& a) {
  // Where one march leaves SMs without an item now and then, fewer than two
  // items of a pass for each.  256^2, M = 32, a gradient's step (forward,
  // recompute and adjoint) side by side against in turn: one group 125 us
  // against 134, two 188 against 208, four 302 against 316, eight 472 against
  // 448, sixteen 925 against 878 (twice the state between two uses in L2).
  const MarchItems it(a, 2, 0);
  return a.G * static_cast<long long>(it.nxi > it.nyi ? it.nxi : it.nyi) < 2 * device_sms();
}

size_t tc_march_ctl_bytes(int G) { return (32 + 2 * static_cast<size_t>(G)) * sizeof(int); }

cudaError_t launch_march_tc(MarchArgs ma, cudaStream_t s, long long* launches) {
  const int sms = device_sms();
  if (ma.dual) ma.a.G *= 2;
  // Row tiles per item: two output tiles share a conversion of the slab, one
  // makes twice the items.  One where a pass has no more items than SMs that
  // way (256^2, M = 32, 3xTF32: one group 46 us a step against 60; four
  // groups 95 against 94, sixteen 415 against 278).
  ma.lag = kMarchLag;
  ma.rt = 1;
  const MarchItems one(ma.a, 1, ma.lag);
  if (ma.a.G * static_cast<long long>(one.nxi > one.nyi ? one.nxi : one.nyi) > sms) ma.rt = 2;
  cudaError_t e = cudaMemsetAsync(ma.ctl, 0, tc_march_ctl_bytes(ma.a.G), s);
  if (e != cudaSuccess) return e;
  e = ma.dual ? launch_march_p<true>(ma, sms, s) : launch_march_p<false>(ma, sms, s);
  if (launches) *launches += 1;
  return e;
}

}  // namespace rte_kern
