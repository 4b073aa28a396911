// Plain FP32 SIMT kernels of the FC-DOM step (Algorithm 1 loop body).
//
// Layout: U[g][j][i][m] (group, y, x, ordinate), FP32, ordinate innermost so
// that one grid node's M intensities are contiguous (the scattering sum and
// the boundary reflections are node-local) and both line directions are
// dense: an x-line tile is rows (j) x all i x all m; a y-line tile is all j x
// a few columns (i) x all m, contiguous per row.
//
// x-pass: for a block of rows, R = b P~u - (a + b) u - xi_m (D_x u)  [one GEMM
//         D_x (nx x nx) times the rows' (nx x rows*M) slab, plus the node-local
//         M x M scattering]
// y-pass: for a block of columns, L^k = R - eta_m (D_y u); AB4 update of
//         eq. (RTEAB4); boundary condition of eq. (RTE) on Gamma_-; exitance
//         of eq. (OpMed) on the boundary ring.  U is updated in place; the
//         new L^k overwrites the oldest history slot.
// The same passes take the transposed step of the exact discrete adjoint
// (BoundaryArgs::bct_src set): transposed D operators in the GEMMs and the
// transposed AB4 / boundary / readout bookkeeping in the y-pass epilogue.
#include <algorithm>
#include <cstdint>

#include "rte_kernels.cuh"

namespace rte_kern {

namespace {

constexpr float kAB0 = 55.0f / 24.0f, kAB1 = -59.0f / 24.0f, kAB2 = 37.0f / 24.0f,
                kAB3 = -9.0f / 24.0f;

__device__ inline float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// ---------------------------------------------------------------- passes
//
// A pass is a GEMM of the n x n operator with the slab of a tile of lines,
// n x BN (BN = lines per tile x M).  A CTA computes every row of its tile, so
// that the y-pass may update U in place: its slab sits in shared memory from
// the first read to the epilogue.  A thread has T x T outputs: blocks of four
// rows, T / 4 of them, by T neighbouring columns of one node, so that the
// epilogues move 16-byte pieces of whole lines.  The products are packed in
// pairs of rows (fma.rn.f32x2: the same fused multiply-adds, two an
// instruction, which leaves the issue slots for the shared-memory loads).
//
// Operator and slab arrive in chunks of kKC positions by cp.async, the
// operator through a ring of kRing chunks; the operator array is padded with
// zeros (simt_ld, simt_rows), so that a chunk is one contiguous run without
// bounds checks.
//
// What bounds it: shared-memory reads (a 16-byte load returns 512 bytes a
// warp; with 8 x 8 outputs the loads of a position take as long as its
// multiply-adds) and the FP32 pipe (36.7 TFMA/s measured for independent
// FFMA) together on large problems; on small ones the latency of the chunks,
// the epilogue's loads and the launch.  Time per step before (one warp per
// node in the y epilogue, a 64-column tile, bounds-checked operator loads)
// and now: 256^2, M = 32, four groups 498 -> 215 us; 203 x 131, M = 24, three
// groups 159 -> 62; 64^2, M = 16, one group 94 -> 12.
struct TileShape {
  int ntx, nty;                      // threads over columns and rows
  int BN, per_tile;                  // columns and grid lines of the tile
};

constexpr int kSlabPad = 4;          // floats after a slab row (conflict-free column reads in the scattering)
constexpr int kMaxThreads = 512;
constexpr int kRing = 2;             // operator chunks in shared memory (four measured no faster and cost occupancy)

// Column block tx and row block ty of a thread.  Eight neighbouring lanes
// take four column blocks of two row blocks where the tile has them, so that
// their 16-byte pieces of a slab row (T = 8: every other one) lie in
// different banks.
__device__ __forceinline__ void thread_place(const TileShape& ts, int& tx, int& ty) {
  const int tid = threadIdx.x;
  if ((ts.ntx & 3) == 0 && (ts.nty & 1) == 0) {
    const int n4 = ts.ntx >> 2, q = tid >> 3;
    tx = (tid & 3) + 4 * (q % n4);
    ty = ((tid >> 2) & 1) + 2 * (q / n4);
  } else {
    tx = tid % ts.ntx;
    ty = tid / ts.ntx;
  }
}

// Boundary nodes of a y tile, at most: both x-faces and two y-face rows.
__host__ __device__ inline int tile_nodes(int n, int M, int BN) { return (BN > M ? 2 : 1) * n + 2 * (BN / M); }

size_t tile_smem(int n, int M, int BN, bool xpass) {
  const size_t ld = simt_ld(n), rows = simt_rows(n);
  size_t f = rows * (BN + kSlabPad) + static_cast<size_t>(kRing) * kKC * ld;
  // P~, or the boundary tables and the boundary nodes' sources
  f += xpass ? static_cast<size_t>(M) : static_cast<size_t>(8 * M) * 2 + 4 * M + 2 * tile_nodes(n, M, BN);
  return f * sizeof(float);
}

__device__ __forceinline__ void cp_async16(float* dst, const float* src, bool valid) {
  const uint32_t d = static_cast<uint32_t>(__cvta_generic_to_shared(dst));
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(valid ? 16 : 0) : "memory");
}

// 16 bytes that the launch before may still be writing when this one begins
// (dependent launches): a plain load, behind the wait.  A const __restrict__
// pointer would allow read-only loads, which hold only for memory that nobody
// writes while the kernel lives, and would let them move above the wait.
__device__ __forceinline__ float4 ld_plain4(const float* p) {
  float4 v;
  asm volatile("ld.global.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p));
  return v;
}

// acc[r][c] = sum_k AT[k][row(r)] slab[k][col(c)], k ascending.  copy_slab(k0)
// starts the copies of slab rows k0 .. k0 + kKC - 1 (zeros past the line).
template <int T, class CopySlab>
__device__ __forceinline__ void tile_gemm(const float* __restrict__ AT, int n, const TileShape& ts, const float* Bs,
                                          float* As, int tx, int ty, CopySlab&& copy_slab, float (&acc)[T][T]) {
  const int tid = threadIdx.x, nthr = blockDim.x;
  const int ld = simt_ld(n), n_chunks = simt_rows(n) / kKC, ldb = ts.BN + kSlabPad;
  const int chunk = kKC * ld;
  auto fetch = [&](int c) {
    if (c < n_chunks) {
      const float* src = AT + static_cast<size_t>(c) * chunk;
      float* dst = As + (c % kRing) * chunk;
      for (int e = tid * 4; e < chunk; e += nthr * 4) cp_async16(dst + e, src + e, true);
      copy_slab(c * kKC);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
#pragma unroll
  for (int c = 0; c < kRing - 1; ++c) fetch(c);
  unsigned long long acc2[T / 2][T];                 // two rows each (fma.rn.f32x2)
#pragma unroll
  for (int r = 0; r < T / 2; ++r)
#pragma unroll
    for (int c = 0; c < T; ++c) acc2[r][c] = 0ull;
  for (int c = 0; c < n_chunks; ++c) {
    asm volatile("cp.async.wait_group %0;" ::"n"(kRing - 2) : "memory");
    __syncthreads();                                 // chunk c is there; every thread is done with chunk c - 1
    fetch(c + kRing - 1);
    const float* ap = As + (c % kRing) * chunk + ty * 4;
    const float* bp = Bs + c * kKC * ldb + tx * T;
#pragma unroll
    for (int k = 0; k < kKC; ++k) {
      unsigned long long a2[T / 2];
      float b[T];
#pragma unroll
      for (int v = 0; v < T / 4; ++v) {
        const ulonglong2 x = *reinterpret_cast<const ulonglong2*>(ap + k * ld + v * 4 * ts.nty);
        a2[2 * v] = x.x; a2[2 * v + 1] = x.y;
      }
#pragma unroll
      for (int v = 0; v < T / 4; ++v) {
        const float4 y = *reinterpret_cast<const float4*>(bp + k * ldb + v * 4);
        b[4 * v] = y.x; b[4 * v + 1] = y.y; b[4 * v + 2] = y.z; b[4 * v + 3] = y.w;
      }
#pragma unroll
      for (int q = 0; q < T; ++q) {
        unsigned long long b2;
        asm("mov.b64 %0, {%1, %1};" : "=l"(b2) : "f"(b[q]));
#pragma unroll
        for (int r = 0; r < T / 2; ++r)
          asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc2[r][q]) : "l"(a2[r]), "l"(b2));
      }
    }
  }
#pragma unroll
  for (int r = 0; r < T / 2; ++r)
#pragma unroll
    for (int q = 0; q < T; ++q)
      asm("mov.b64 {%0, %1}, %2;" : "=f"(acc[2 * r][q]), "=f"(acc[2 * r + 1][q]) : "l"(acc2[r][q]));
}

template <int T>
__global__ void __launch_bounds__(kMaxThreads) xpass_kernel(StepArgs a, TileShape ts, const float* U,
                                                            float* __restrict__ R) {
  extern __shared__ __align__(16) float smem[];
  const int n = a.nx, M = a.M, ldb = ts.BN + kSlabPad;
  float* Bs = smem;                                   // [rows][ldb]
  float* As = Bs + simt_rows(n) * ldb;                // [kRing][kKC][ld]
  float* Ps = As + kRing * kKC * simt_ld(n);              // [M]: p_d = P~[d][0], the circulant's first column
  const int g = blockIdx.z, j0 = blockIdx.x * ts.per_tile;
  const int tid = threadIdx.x, nthr = blockDim.x;
  int tx, ty;
  thread_place(ts, tx, ty);
  const float* Ug = U + static_cast<size_t>(g) * a.plane;
  for (int e = tid; e < M; e += nthr) Ps[e] = __ldg(a.PT + e);
  asm volatile("griddepcontrol.wait;" ::: "memory");
  // slab row k: u[j0 + r][k][m] at column r M + m.  A thread copies the same
  // 16 bytes of every nrow-th row.
  const int cw = ts.BN / 4, ck = tid / cw, cc = (tid - ck * cw) * 4, nrow = nthr / cw;
  const int cr = cc / M;
  const bool c_ok = ck < nrow && j0 + cr < a.ny;
  const float* csrc = Ug + static_cast<size_t>(c_ok ? j0 + cr : 0) * n * M + (cc - cr * M);
  auto copy_slab = [&](int k0) {
    if (ck < nrow)
      for (int k = ck; k < kKC; k += nrow) {
        const bool ok = c_ok && k0 + k < n;
        cp_async16(Bs + (k0 + k) * ldb + cc, csrc + (ok ? static_cast<size_t>(k0 + k) * M : 0), ok);
      }
  };
  float acc[T][T];
  tile_gemm<T>(a.DxT, n, ts, Bs, As, tx, ty, copy_slab, acc);
  asm volatile("griddepcontrol.launch_dependents;");

  // Epilogue: node-local scattering and absorption, minus xi * d_x u.  The
  // thread's columns lie in one node per row.  P~[m][q] = p_{(m - q) mod M}:
  // the T weights of ordinate q are those of q - 1 moved by one, so that T
  // ordinates take 2 T weights, half of them from the T before; kHR rows at
  // a time (registers).
  constexpr int kHR = T == 4 ? 4 : 2;
  const int c0 = tx * T, r = c0 / M, mb = c0 - r * M, j = j0 + r;
#pragma unroll
  for (int h = 0; h < T / kHR; ++h) {
    auto row_of = [&](int ii) { return ((h * kHR + ii) / 4) * 4 * ts.nty + ty * 4 + (h * kHR + ii) % 4; };
    float s[kHR][T], w[2 * T];
#pragma unroll
    for (int ii = 0; ii < kHR; ++ii)
#pragma unroll
      for (int t = 0; t < T; ++t) s[ii][t] = 0.f;
    // w[T + d] = p_{mb - q + d}, d in [-T, T)
    auto load_w = [&](int k, float* dst) {             // p_k .. p_{k + T - 1}
      k = k < 0 ? k + M : k;
#pragma unroll
      for (int v = 0; v < T / 4; ++v) {
        const float4 p4 = *reinterpret_cast<const float4*>(Ps + k + 4 * v);
        dst[4 * v] = p4.x; dst[4 * v + 1] = p4.y; dst[4 * v + 2] = p4.z; dst[4 * v + 3] = p4.w;
      }
    };
    load_w(mb, w + T);
    const float* ub[kHR];
#pragma unroll
    for (int ii = 0; ii < kHR; ++ii) ub[ii] = Bs + row_of(ii) * ldb + r * M;
    for (int q = 0; q < M; q += T) {
      load_w(mb - q - T, w);
#pragma unroll
      for (int q4 = 0; q4 < T / 4; ++q4) {
        float u[kHR][4];
#pragma unroll
        for (int ii = 0; ii < kHR; ++ii) {
          const float4 u4 = *reinterpret_cast<const float4*>(ub[ii] + q + 4 * q4);
          u[ii][0] = u4.x; u[ii][1] = u4.y; u[ii][2] = u4.z; u[ii][3] = u4.w;
        }
#pragma unroll
        for (int t = 0; t < 4; ++t)
#pragma unroll
          for (int ii = 0; ii < kHR; ++ii)
#pragma unroll
            for (int e = 0; e < T; ++e) s[ii][e] = fmaf(w[T - (4 * q4 + t) + e], u[ii][t], s[ii][e]);
      }
#pragma unroll
      for (int e = 0; e < T; ++e) w[T + e] = w[e];
    }
#pragma unroll
    for (int ii = 0; ii < kHR; ++ii) {
      const int i = row_of(ii);
      if (i < n && j < a.ny) {
        const size_t cell = static_cast<size_t>(j) * n + i;
        const float av = __ldg(a.mua + cell), bv = __ldg(a.mus + cell);
        float* dst = R + static_cast<size_t>(g) * a.plane + cell * M + mb;
#pragma unroll
        for (int v = 0; v < T / 4; ++v) {
          const float4 u4 = *reinterpret_cast<const float4*>(Bs + i * ldb + c0 + 4 * v);
          const float4 xi = __ldg(reinterpret_cast<const float4*>(a.xi + mb + 4 * v));
          const float* ac = &acc[h * kHR + ii][4 * v];
          const float* sv = &s[ii][4 * v];
          *reinterpret_cast<float4*>(dst + 4 * v) =
              make_float4(bv * sv[0] - (av + bv) * u4.x - xi.x * ac[0], bv * sv[1] - (av + bv) * u4.y - xi.y * ac[1],
                          bv * sv[2] - (av + bv) * u4.z - xi.z * ac[2], bv * sv[3] - (av + bv) * u4.w - xi.w * ac[3]);
        }
      }
    }
  }
}

// TR: the transposed step of the discrete adjoint (BoundaryArgs::bct_src);
// a separate instance, so that the forward step compiles without it.
template <int T, bool TR>
__global__ void __launch_bounds__(kMaxThreads) ypass_kernel(StepArgs a, BoundaryArgs b, TileShape ts,
                                                            float* __restrict__ U, const float* R,
                                                            const float* __restrict__ L1,
                                                            const float* __restrict__ L2, float* __restrict__ L3,
                                                            int src_step, int ring_step) {
  extern __shared__ __align__(16) float smem[];
  const int nx = a.nx, n = a.ny, M = a.M, ldb = ts.BN + kSlabPad;
  float* Bs = smem;                                   // [rows][ldb]
  float* As = Bs + simt_rows(n) * ldb;                // [kRing][kKC][ld]
  // boundary tables: faces 0..3, corners 4..7; the factor and the reflected
  // ordinate (its own with the sign bit set where nothing is imposed)
  int2* bct = reinterpret_cast<int2*>(As + kRing * kKC * simt_ld(n));   // [8][M]
  float* wexit = reinterpret_cast<float*>(bct + 8 * M);             // [4][M]
  float* src0 = wexit + 4 * M;       // [node of the tile]: the first beam's S
  float* srho = src0 + tile_nodes(n, M, ts.BN);                     // [node of the tile]: rho
  // the tiles with an x-face, whose epilogue takes longest, start first
  const int g = blockIdx.z;
  const int tile = blockIdx.x == 0 ? 0 : blockIdx.x == 1 ? gridDim.x - 1 : blockIdx.x - 1;
  const int i0 = tile * ts.per_tile;
  const int tid = threadIdx.x, nthr = blockDim.x;
  int tx, ty;
  thread_place(ts, tx, ty);
  const size_t goff = static_cast<size_t>(g) * a.plane;
  float* Ug = U + goff;
  for (int e = tid; e < 8 * M; e += nthr) {
    const bool face = e < 4 * M;
    const int k = face ? e : e - 4 * M;
    const bool act = (face ? b.face_act[k] : b.corner_act[k]) != 0;
    bct[e] = make_int2(__float_as_int(face ? b.face_f[k] : b.corner_f[k]),
                       act ? (face ? b.face_refl[k] : b.corner_refl[k]) : static_cast<int>(0x80000000u | (k % M)));
    if (face) wexit[e] = b.wexit[k];
  }
  // Boundary nodes of the tile: the left face's, the right one's, the y-faces'
  // (those that are not corners; false past the grid).  Their S and rho are
  // asked for before the GEMM.
  const int ring_len = 2 * n + 2 * nx;
  const int n_l = i0 == 0 ? n : 0, n_r = i0 + ts.per_tile >= nx ? n : 0, n_nodes = n_l + n_r + 2 * ts.per_tile;
  auto node_at = [&](int q, int& i, int& j) {
    if (q < n_l + n_r) {
      i = q < n_l ? 0 : nx - 1;
      j = q < n_l ? q : q - n_l;
      return true;
    }
    q -= n_l + n_r;
    j = q < ts.per_tile ? 0 : n - 1;
    i = i0 + (q < ts.per_tile ? q : q - ts.per_tile);
    return i > 0 && i < nx - 1;
  };
  // ring node of the source data (x-face index at corners)
  auto ring_node = [&](int i, int j) {
    return i == 0 ? j : i == nx - 1 ? n + j : j == 0 ? 2 * n + i : 2 * n + nx + i;
  };
  if constexpr (!TR)
    for (int q = tid; q < n_nodes; q += nthr) {
      int i, j;
      if (!node_at(q, i, j)) continue;
      if (b.kmax > 0) src0[q] = __ldg(b.S + static_cast<size_t>(g) * b.kmax * ring_len + ring_node(i, j));
      if (b.rho) srho[q] = __ldg(b.rho + (static_cast<size_t>(g) * b.rho_len + src_step) * ring_len + ring_node(i, j));
    }
  asm volatile("griddepcontrol.wait;" ::: "memory");
  // slab row k: u[k][i0 + w][m] at column w M + m (contiguous)
  const int cw = ts.BN / 4, ck = tid / cw, cc = (tid - ck * cw) * 4, nrow = nthr / cw;
  const bool c_ok = ck < nrow && i0 + cc / M < nx;
  const float* csrc = Ug + (c_ok ? static_cast<size_t>(i0) * M + cc : 0);
  auto copy_slab = [&](int k0) {
    if (ck < nrow)
      for (int k = ck; k < kKC; k += nrow) {
        const bool ok = c_ok && k0 + k < n;
        cp_async16(Bs + (k0 + k) * ldb + cc, csrc + (ok ? static_cast<size_t>(k0 + k) * nx * M : 0), ok);
      }
  };
  float acc[T][T];
  tile_gemm<T>(a.DyT, n, ts, Bs, As, tx, ty, copy_slab, acc);
  asm volatile("griddepcontrol.launch_dependents;");

  // AB4 update (eq. RTEAB4); interior nodes are finished here, boundary nodes
  // keep u^{k+1} before the boundary condition (TR: ubar) in acc.
  auto row_of = [&](int jj) { return (jj / 4) * 4 * ts.nty + ty * 4 + jj % 4; };
  auto is_bnd = [&](int i, int j) { return i == 0 || i == nx - 1 || j == 0 || j == n - 1; };
  auto ld4 = [](const float* p) { return *reinterpret_cast<const float4*>(p); };
#pragma unroll
  for (int v = 0; v < T / 4; ++v) {
    const int c0 = tx * T + 4 * v, w = c0 / M, mb = c0 - w * M, i = i0 + w;
    const float4 eta = __ldg(reinterpret_cast<const float4*>(a.eta + mb));
    const size_t base0 = goff + static_cast<size_t>(i) * M + mb;
#pragma unroll
    for (int jj = 0; jj < T; ++jj) {
      const int j = row_of(jj);
      if (i >= nx || j >= n) continue;
      float* ac = &acc[jj][4 * v];
      const size_t base = base0 + static_cast<size_t>(j) * nx * M;
      const float4 r4 = ld_plain4(R + base), p4 = ld4(L1 + base), q4 = ld4(L2 + base), s4 = ld4(L3 + base);
      if constexpr (TR) {
        // transposed step: ubar = w^{k+1} + L^T v
        ac[0] = r4.x - eta.x * ac[0] + p4.x;
        ac[1] = r4.y - eta.y * ac[1] + p4.y;
        ac[2] = r4.z - eta.z * ac[2] + p4.z;
        ac[3] = r4.w - eta.w * ac[3] + p4.w;
        if (!is_bnd(i, j)) {
          *reinterpret_cast<float4*>(U + base) =
              make_float4(a.cdt * (kAB0 * ac[0] + kAB1 * p4.x + kAB2 * q4.x + kAB3 * s4.x),
                          a.cdt * (kAB0 * ac[1] + kAB1 * p4.y + kAB2 * q4.y + kAB3 * s4.y),
                          a.cdt * (kAB0 * ac[2] + kAB1 * p4.z + kAB2 * q4.z + kAB3 * s4.z),
                          a.cdt * (kAB0 * ac[3] + kAB1 * p4.w + kAB2 * q4.w + kAB3 * s4.w));
          *reinterpret_cast<float4*>(L3 + base) = make_float4(ac[0], ac[1], ac[2], ac[3]);
        }
      } else {
        const float4 u4 = ld4(Bs + j * ldb + c0);
        float4 lk;
        lk.x = r4.x - eta.x * ac[0];
        lk.y = r4.y - eta.y * ac[1];
        lk.z = r4.z - eta.z * ac[2];
        lk.w = r4.w - eta.w * ac[3];
        ac[0] = fmaf(a.cdt, kAB0 * lk.x + kAB1 * p4.x + kAB2 * q4.x + kAB3 * s4.x, u4.x);
        ac[1] = fmaf(a.cdt, kAB0 * lk.y + kAB1 * p4.y + kAB2 * q4.y + kAB3 * s4.y, u4.y);
        ac[2] = fmaf(a.cdt, kAB0 * lk.z + kAB1 * p4.z + kAB2 * q4.z + kAB3 * s4.z, u4.z);
        ac[3] = fmaf(a.cdt, kAB0 * lk.w + kAB1 * p4.w + kAB2 * q4.w + kAB3 * s4.w, u4.w);
        *reinterpret_cast<float4*>(L3 + base) = lk;
        if (!is_bnd(i, j)) *reinterpret_cast<float4*>(U + base) = make_float4(ac[0], ac[1], ac[2], ac[3]);
      }
    }
  }

  // Boundary nodes: the values before the boundary condition go to the slab's
  // place, and all threads share the nodes, four ordinates each, in a rolled
  // loop (unrolled over a thread's own outputs the code of this part did not
  // fit the instruction cache).
  __syncthreads();                                    // every thread has read u^k and the operator
#pragma unroll
  for (int v = 0; v < T / 4; ++v) {
    const int c0 = tx * T + 4 * v, i = i0 + c0 / M;
#pragma unroll
    for (int jj = 0; jj < T; ++jj) {
      const int j = row_of(jj);
      const float* ac = &acc[jj][4 * v];
      if (i < nx && j < n && is_bnd(i, j))
        *reinterpret_cast<float4*>(Bs + j * ldb + c0) = make_float4(ac[0], ac[1], ac[2], ac[3]);
    }
  }
  __syncthreads();
  const int V = M / 4, n_items = n_nodes * V;         // four ordinates each
  auto item = [&](int e, int& q, int& i, int& j, int& m) {
    q = e / V;
    m = (e - q * V) * 4;
    return node_at(q, i, j);
  };
  if constexpr (TR) {                                 // the readout transpose on every face the node lies on
    const float* eb = b.ebar + (static_cast<size_t>(g) * b.ebar_len + src_step) * ring_len;
    for (int e = tid; e < n_items; e += nthr) {
      int q, i, j, m;
      if (!item(e, q, i, j, m)) continue;
      float* pre = Bs + j * ldb + (i - i0) * M + m;
      const float ex = i == 0 || i == nx - 1 ? __ldg(eb + (i == 0 ? j : n + j)) : 0.f;
      const float ey = j == 0 || j == n - 1 ? __ldg(eb + (j == 0 ? 2 * n + i : 2 * n + nx + i)) : 0.f;
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        float x = pre[t];
        if (i == 0 || i == nx - 1) x = fmaf(wexit[(i == 0 ? 0 : 1) * M + m + t], ex, x);
        if (j == 0 || j == n - 1) x = fmaf(wexit[(j == 0 ? 2 : 3) * M + m + t], ey, x);
        pre[t] = x;
      }
    }
    __syncthreads();
  }
  // Boundary condition (eq. RTE third line), and the four ordinates' part of
  // the exitance of eq. (OpMed): x-faces in px[j][column / 4], y-faces in
  // py[face][column / 4], in the operator's place, which is large enough for
  // tiles of up to 64 columns (kRing kKC ld >= ld BN / 4 + BN / 2).
  const int cq = ts.BN / 4;
  float* px = As;
  float* py = As + simt_ld(n) * cq;
  for (int e = tid; e < n_items; e += nthr) {
    int nd, i, j, m;
    if (!item(e, nd, i, j, m)) continue;
    const int c0 = (i - i0) * M + m;
    const bool lf = i == 0, rt = i == nx - 1, bt = j == 0, tp = j == n - 1;
    const float* pre = Bs + j * ldb + (i - i0) * M;
    const int tb = ((lf || rt) && (bt || tp)) ? 4 + (rt ? 1 : 0) + (tp ? 2 : 0) : (lf ? 0 : rt ? 1 : bt ? 2 : 3);
    const size_t base = goff + (static_cast<size_t>(j) * nx + i) * M + m;
    if constexpr (TR) {
      // w = BC^T ubar, then v' = c dt (chi0 w + chi1 w^{k+1} + chi2 w^{k+2} + chi3 w^{k+3})
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        const int* src = b.bct_src + (tb * M + m + t) * 4;
        const float* cf = b.bct_f + (tb * M + m + t) * 4;
        float wv = 0.f;
#pragma unroll
        for (int q = 0; q < 4; ++q) wv = fmaf(__ldg(cf + q), pre[__ldg(src + q)], wv);
        U[base + t] = a.cdt * (kAB0 * wv + kAB1 * L1[base + t] + kAB2 * L2[base + t] + kAB3 * L3[base + t]);
        L3[base + t] = wv;
      }
    } else {
      float q[4] = {0.f, 0.f, 0.f, 0.f};
      for (int k = 0; k < b.kmax; ++k) {
        const size_t gk = static_cast<size_t>(g) * b.kmax + k;
        const float sk = k == 0 ? src0[nd] : __ldg(b.S + gk * ring_len + ring_node(i, j));
        const float tk = __ldg(b.T + gk * b.T_len + src_step);
        const float4 ak = __ldg(reinterpret_cast<const float4*>(b.A + gk * M + m));
        q[0] = fmaf(sk * ak.x, tk, q[0]);
        q[1] = fmaf(sk * ak.y, tk, q[1]);
        q[2] = fmaf(sk * ak.z, tk, q[2]);
        q[3] = fmaf(sk * ak.w, tk, q[3]);
      }
      const float rho = b.rho ? srho[nd] : 0.f;
      float x[4];
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        const int2 en = bct[tb * M + m + t];
        const float fco = __int_as_float(en.x);
        if (b.rho) q[t] = fmaf(1.0f - fco, rho, q[t]);
        const float z = fmaf(fco, pre[en.y & 0x7fffffff], q[t]);
        x[t] = en.y >= 0 ? z : pre[m + t];
      }
      *reinterpret_cast<float4*>(U + base) = make_float4(x[0], x[1], x[2], x[3]);
      auto part = [&](int face) {
        const float* we = wexit + face * M + m;
        return fmaf(we[3], x[3], fmaf(we[2], x[2], fmaf(we[1], x[1], we[0] * x[0])));
      };
      if (lf || rt) px[j * cq + c0 / 4] = part(lf ? 0 : 1);
      if (bt || tp) py[(bt ? 0 : cq) + c0 / 4] = part(bt ? 2 : 3);
    }
  }
  if (TR || ring_step < 0) return;
  __syncthreads();
  // exitance of a boundary node: its M / 4 parts in order
  float* ro = b.ring_out + (static_cast<size_t>(g) * b.ring_steps + ring_step) * ring_len;
  auto node_sum = [&](const float* q) {
    float e = q[0];
    for (int k = 1; k < M / 4; ++k) e += q[k];
    return e;
  };
  if (i0 == 0)
    for (int j = tid; j < n; j += nthr) ro[j] = node_sum(px + j * cq);
  if (i0 + ts.per_tile >= nx)
    for (int j = tid; j < n; j += nthr) ro[n + j] = node_sum(px + j * cq + (nx - 1 - i0) * (M / 4));
  for (int k = tid; k < 2 * ts.per_tile; k += nthr) {
    const int face = k / ts.per_tile, w = k - face * ts.per_tile;
    if (i0 + w < nx) ro[2 * n + face * nx + i0 + w] = node_sum(py + face * cq + w * (M / 4));
  }
}

__global__ void fluence_kernel(const float* __restrict__ U, float* __restrict__ out,
                               size_t out_gs, int ncell, int M, size_t plane, float w) {
  const int lane = threadIdx.x & 31;
  const long long warp = (static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
  const int g = blockIdx.y;
  if (warp >= ncell) return;
  const float* u = U + static_cast<size_t>(g) * plane + static_cast<size_t>(warp) * M;
  float s = 0.f;
  for (int m = lane; m < M; m += 32) s += u[m];
  s = warp_sum(s);
  if (lane == 0) out[static_cast<size_t>(g) * out_gs + warp] = w * s;
}

__global__ void readout_kernel(const float* __restrict__ ring, int ring_len, int n_steps, int G,
                               const float* __restrict__ Wd, const int* __restrict__ lo,
                               const int* __restrict__ hi, int n_det, float* curves,
                               double* curves64) {
  const long long idx = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x;
  const long long total = static_cast<long long>(G) * n_det * n_steps;
  if (idx >= total) return;
  const int s = static_cast<int>(idx % n_steps);
  const int d = static_cast<int>((idx / n_steps) % n_det);
  const int g = static_cast<int>(idx / (static_cast<long long>(n_steps) * n_det));
  const float* r = ring + (static_cast<size_t>(g) * n_steps + s) * ring_len;
  double acc = 0.0;
  for (int k = lo[d]; k < hi[d]; ++k) {
    const float wv = Wd[static_cast<size_t>(d) * ring_len + k];
    if (wv != 0.f) acc += static_cast<double>(wv) * static_cast<double>(r[k]);
  }
  if (curves) curves[idx] = static_cast<float>(acc);
  if (curves64) curves64[idx] = acc;
}

__global__ void objective_partial(const double* __restrict__ c64, const float* __restrict__ meas,
                                  size_t n, float* __restrict__ resid, double* __restrict__ partial) {
  __shared__ double sh[256];
  double s = 0.0;
  for (size_t k = static_cast<size_t>(blockIdx.x) * blockDim.x + threadIdx.x; k < n;
       k += static_cast<size_t>(gridDim.x) * blockDim.x) {
    const double r = c64[k] - static_cast<double>(meas[k]);
    resid[k] = static_cast<float>(r);
    s += r * r;
  }
  sh[threadIdx.x] = s;
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if (threadIdx.x < o) sh[threadIdx.x] += sh[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) partial[blockIdx.x] = sh[0];
}

__global__ void objective_final(const double* __restrict__ partial, int nb, double scale,
                                double* J) {
  __shared__ double sh[256];
  double s = 0.0;
  for (int k = threadIdx.x; k < nb; k += blockDim.x) s += partial[k];
  sh[threadIdx.x] = s;
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if (threadIdx.x < o) sh[threadIdx.x] += sh[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) *J = scale * sh[0];
}

__global__ void rho_kernel(const float* __restrict__ resid, const float* __restrict__ Wn, int n_det,
                           int ring_len, int n_steps, int G, float scale, float* __restrict__ rho) {
  const long long idx = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x;
  const long long total = static_cast<long long>(G) * n_steps * ring_len;
  if (idx >= total) return;
  const int node = static_cast<int>(idx % ring_len);
  const int s = static_cast<int>((idx / ring_len) % n_steps);
  const int g = static_cast<int>(idx / (static_cast<long long>(ring_len) * n_steps));
  float acc = 0.f;
  for (int d = 0; d < n_det; ++d)
    acc = fmaf(Wn[static_cast<size_t>(d) * ring_len + node],
               resid[(static_cast<size_t>(g) * n_det + d) * n_steps + s], acc);
  rho[idx] = scale * acc;
}

// The gradient terms of eq. (FDwin22) at one grid cell, summed over the
// groups and the ordinates (see launch_grad):
//   sa = sum_g sum_m lam_m u_m,  sb = sum_g sum_m lam_m (u_m - (P~u)_m),
// lam the adjoint field (its ordinates flipped by M/2 in the continuous form).
// One thread per cell for M in {16, 32}: the node's M values of u and lam
// arrive as 32-byte loads, and P~u uses the circulant's first column p_d =
// P~[d][0] (P~[m][q] = p_{(m - q) mod M}) from registers, summed over q in
// order for every m.
// 32 bytes of read-only data into 8 registers (32-byte aligned address).
__device__ __forceinline__ void ld32b(const float* ptr, float* v) {
  asm volatile("ld.global.nc.v8.f32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7])
               : "l"(ptr));
}

// A cell's groups are shared by `split` neighbouring lanes (a power of two; the
// FP32 sums of a lane's groups are added in FP64), so that small grids with
// many groups fill the chip: 64^2, 16 groups, M = 32: 33 us with one lane per
// cell, whose groups come one after another, 9 us with sixteen.
constexpr long long kGradThreads = 152 * 256;

template <int MM>
__device__ __forceinline__ void grad_node(const float* __restrict__ MU, const float* __restrict__ Useg,
                                          const float* __restrict__ PT, const float* __restrict__ area,
                                          long long t, int ncell, int G, int split, size_t plane, size_t useg_gs,
                                          double scale, int flip, const GradLevels lv, double* __restrict__ grad_a,
                                          double* __restrict__ grad_b) {
  const int lane = static_cast<int>(t) & (split - 1);
  const long long cell = t / split;
  const bool valid = cell < ncell;
  float p[MM];
#pragma unroll
  for (int d = 0; d < MM; ++d) p[d] = __ldg(PT + d);            // P~[0][d] = p_d (symmetric circulant)
  const double k = area && valid ? scale * static_cast<double>(area[cell]) : scale;
  double ga = valid && grad_a ? grad_a[cell] : 0.0, gb = valid && grad_b ? grad_b[cell] : 0.0;
  for (int l = 0; l < lv.n; ++l) {
    float sa = 0.f, sb = 0.f;
    for (int g = valid ? lane : G; g < G; g += split) {
      const float* u = Useg + l * lv.u_step + static_cast<size_t>(g) * useg_gs + static_cast<size_t>(cell) * MM;
      const float* mu = MU + l * lv.mu_step + static_cast<size_t>(g) * plane + static_cast<size_t>(cell) * MM;
      float uu[MM], lam[MM];
#pragma unroll
      for (int q = 0; q < MM / 8; ++q) {
        ld32b(u + 8 * q, uu + 8 * q);
        ld32b(mu + 8 * q, lam + 8 * q);
      }
#pragma unroll
      for (int m = 0; m < MM; ++m) {
        float pu = 0.f;
#pragma unroll
        for (int q = 0; q < MM; ++q) pu = fmaf(p[(m - q + MM) % MM], uu[q], pu);
        const float x = flip ? lam[(m + MM / 2) % MM] : lam[m];
        sa = fmaf(x, uu[m], sa);
        sb = fmaf(x, uu[m] - pu, sb);
      }
    }
    double da = static_cast<double>(sa), db = static_cast<double>(sb);
    for (int o = 1; o < split; o <<= 1) {
      da += __shfl_xor_sync(0xffffffffu, da, o);
      db += __shfl_xor_sync(0xffffffffu, db, o);
    }
    ga -= k * da;
    gb -= k * db;
  }
  if (!valid || lane != 0) return;
  if (grad_a) grad_a[cell] = ga;
  if (grad_b) grad_b[cell] = gb;
}

// Lanes per cell, until every SM has eight warps.
__host__ __device__ inline int grad_split(long long ncell, int G) {
  int split = 1;
  while (2 * split <= G && split < 16 && ncell * split < kGradThreads) split *= 2;
  return split;
}

// Any M: one warp per cell, the lanes over the ordinates, the row of P~ from
// memory.
__device__ __forceinline__ void grad_cell(const float* __restrict__ MU, const float* __restrict__ Useg,
                                          const float* __restrict__ PT, const float* __restrict__ area,
                                          long long cell, int M, int G, size_t plane, size_t useg_gs,
                                          double scale, int flip, const GradLevels lv,
                                          double* __restrict__ grad_a, double* __restrict__ grad_b) {
  __shared__ float ubuf[8][64];
  const int lane = threadIdx.x & 31, wl = threadIdx.x >> 5;
  const double k = area ? scale * static_cast<double>(area[cell]) : scale;
  double da = grad_a ? grad_a[cell] : 0.0, db = grad_b ? grad_b[cell] : 0.0;
  for (int l = 0; l < lv.n; ++l) {
    float sa = 0.f, sb = 0.f;
    for (int g = 0; g < G; ++g) {
      const float* u = Useg + l * lv.u_step + static_cast<size_t>(g) * useg_gs + static_cast<size_t>(cell) * M;
      const float* mu = MU + l * lv.mu_step + static_cast<size_t>(g) * plane + static_cast<size_t>(cell) * M;
      for (int m = lane; m < M; m += 32) ubuf[wl][m] = u[m];
      __syncwarp();
      for (int m = lane; m < M; m += 32) {
        float pu = 0.f;
        for (int q = 0; q < M; ++q) pu = fmaf(PT[q * M + m], ubuf[wl][q], pu);
        const float lam = flip ? mu[(m + M / 2) % M] : mu[m];
        sa = fmaf(lam, ubuf[wl][m], sa);
        sb = fmaf(lam, ubuf[wl][m] - pu, sb);
      }
      __syncwarp();
    }
    da -= k * static_cast<double>(warp_sum(sa));
    db -= k * static_cast<double>(warp_sum(sb));
  }
  if (lane == 0) {
    if (grad_a) grad_a[cell] = da;
    if (grad_b) grad_b[cell] = db;
  }
}

// M in {16, 32}: one thread per cell; other M: one warp per cell.
__device__ __forceinline__ bool grad_by_thread(int M) { return M == 16 || M == 32; }

__global__ void grad_kernel(const float* __restrict__ MU, const float* __restrict__ Useg,
                            const float* __restrict__ PT, const float* __restrict__ area, int ncell,
                            int M, int G, int split, size_t plane, size_t useg_gs, double scale, int flip,
                            GradLevels lv,
                            double* __restrict__ grad_a, double* __restrict__ grad_b) {
  const long long t = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (grad_by_thread(M)) {
    if (M == 32) grad_node<32>(MU, Useg, PT, area, t, ncell, G, split, plane, useg_gs, scale, flip, lv, grad_a, grad_b);
    else grad_node<16>(MU, Useg, PT, area, t, ncell, G, split, plane, useg_gs, scale, flip, lv, grad_a, grad_b);
    return;
  }
  const long long cell = t >> 5;
  if (cell >= ncell) return;   // whole warp exits together
  grad_cell(MU, Useg, PT, area, cell, M, G, plane, useg_gs, scale, flip, lv, grad_a, grad_b);
}

// Batched forms for media that march in lockstep: blockIdx.y picks the
// medium; its forward state of the level sits in slot `slot` of its segment
// buffer.
__global__ void grad_batch_kernel(const GradJob* __restrict__ jobs, int slot, int flip) {
  const GradJob& j = jobs[blockIdx.y];
  const long long t = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x;
  const float* useg = j.seg + static_cast<size_t>(slot) * j.slot_floats;
  const GradLevels one{1, 0, 0};
  if (grad_by_thread(j.M)) {
    const int nc = static_cast<int>(j.ncell);
    if (j.M == 32)
      grad_node<32>(j.MU, useg, j.PT, j.area, t, nc, j.G, grad_split(nc, j.G), j.plane, j.plane, j.scale, flip, one, j.grad_a, j.grad_b);
    else
      grad_node<16>(j.MU, useg, j.PT, j.area, t, nc, j.G, grad_split(nc, j.G), j.plane, j.plane, j.scale, flip, one, j.grad_a, j.grad_b);
    return;
  }
  const long long cell = t >> 5;
  if (cell >= j.ncell) return;
  grad_cell(j.MU, useg, j.PT, j.area, cell, j.M, j.G, j.plane, j.plane, j.scale, flip, one, j.grad_a, j.grad_b);
}

__global__ void save_batch_kernel(const SaveJob* __restrict__ jobs, int slot) {
  const SaveJob& j = jobs[blockIdx.y];
  const size_t n4 = j.n_floats / 4;
  const float4* src = reinterpret_cast<const float4*>(j.src);
  float4* dst = reinterpret_cast<float4*>(j.seg + static_cast<size_t>(slot) * j.n_floats);
  // four independent 16-byte loads in flight per thread and pass
  const size_t stride = static_cast<size_t>(gridDim.x) * blockDim.x;
  size_t k = static_cast<size_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  for (; k + 3 * stride < n4; k += 4 * stride) {
    const float4 v0 = __ldg(src + k), v1 = __ldg(src + k + stride), v2 = __ldg(src + k + 2 * stride),
                 v3 = __ldg(src + k + 3 * stride);
    dst[k] = v0;
    dst[k + stride] = v1;
    dst[k + 2 * stride] = v2;
    dst[k + 3 * stride] = v3;
  }
  for (; k < n4; k += stride) dst[k] = __ldg(src + k);
}

__global__ void to_float_kernel(const double* in, float* out, size_t n) {
  const size_t k = static_cast<size_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (k < n) out[k] = static_cast<float>(in[k]);
}

// Photon balance of one post-BC state (eq. RTE integrated over theta and
// Omega; the scattering term integrates to zero): per group,
//   S0 = sum_nodes A_node sum_m u_m,   S1 = sum_nodes A_node a sum_m u_m,
//   S2 = sum_faces sum_face nodes w_face sum_m (theta_m . nu) u_m,
// with the trapezoid node areas A_node and face weights w_face (half at the
// face ends).  One thread per float4 of the state: the M/4 lanes of a node
// add its ordinates in FP32 (a pairwise tree of M terms) and the node's first
// lane adds A_node sum_m u_m and a A_node sum_m u_m to its own compensated
// (Kahan) FP32 sums, at most kBalItems nodes a thread (32); the boundary fluxes
// are formed in FP64 from a double table of cos and sin of the ordinates.
// GB300's FP64 pipe issues a warp instruction in tens of clocks, so FP64
// work runs once per thread and per boundary node, not per node.  From the
// threads up everything is FP64: warp and block sums in a fixed order, then
// the last block of a group to finish (ticket counter) adds the block
// partials in block order, so the sums do not depend on the schedule.
// out[(g n_steps + step) 3 + k] = (w S0 / c, w S1, w S2).
constexpr int kBalThreads = 256, kBalItems = 32;

__device__ __forceinline__ void kahan_add(float& sum, float& comp, float x) {
  const float y = x - comp;
  const float t = sum + y;
  comp = (t - sum) - y;
  sum = t;
}

__global__ void __launch_bounds__(kBalThreads)
    balance_kernel(const float* __restrict__ U, size_t plane, int nx, int ny, int M,
                   const float* __restrict__ mua, const double* __restrict__ trig, double dx, double dy,
                   double w, double inv_c, double* __restrict__ partial, unsigned* __restrict__ ticket,
                   double* __restrict__ out, int step, int n_steps) {
  __shared__ double red[3][kBalThreads / 32];
  __shared__ int last;
  const int g = blockIdx.y, b = blockIdx.x, nb = gridDim.x;
  const int V = M / 4;                                  // lanes per node: 2, 4, 8 or 16
  const int lv = __ffs(V) - 1;                          // log2 V
  // at most 512 x 512 nodes x 16 float4: 32-bit indices
  const int n4 = nx * ny * V;
  const float4* u4 = reinterpret_cast<const float4*>(U + static_cast<size_t>(g) * plane);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const float fdx = static_cast<float>(dx), fdy = static_cast<float>(dy);
  float a0 = 0.f, c0 = 0.f, a1 = 0.f, c1 = 0.f;        // Kahan sums of A sum_m u and a A sum_m u
  double s2 = 0.0;
  const int base = b * kBalItems * kBalThreads;
  for (int k = 0; k < kBalItems; ++k) {
    const int q = base + k * kBalThreads + static_cast<int>(threadIdx.x);
    const bool valid = q < n4;                          // node groups never straddle the end
    const float4 v = valid ? __ldcs(u4 + q) : make_float4(0.f, 0.f, 0.f, 0.f);
    float su = (v.x + v.y) + (v.z + v.w);
    for (int o = 1; o < V; o <<= 1) su += __shfl_xor_sync(0xffffffffu, su, o);
    if (!valid) continue;
    const int node = q >> lv;
    const int r = q & (V - 1);
    const int j = node / nx, i = node - j * nx;
    const bool xe = i == 0 || i == nx - 1, ye = j == 0 || j == ny - 1;
    if (r == 0) {
      // trapezoid node area: dx dy, halved on each face the node lies on
      const float area = (xe ? 0.5f * fdx : fdx) * (ye ? 0.5f * fdy : fdy);
      const float t = area * su;
      kahan_add(a0, c0, t);
      kahan_add(a1, c1, t * __ldg(mua + node));
    }
    if (xe || ye) {
      const double wx = (i == 0 || i == nx - 1) ? 0.5 * dx : dx;
      const double wy = (j == 0 || j == ny - 1) ? 0.5 * dy : dy;
      const int m0 = 4 * r;
      const double e[4] = {v.x, v.y, v.z, v.w};
      double fx = 0.0, fy = 0.0;
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        fx += __ldg(trig + m0 + t) * e[t];
        fy += __ldg(trig + M + m0 + t) * e[t];
      }
      if (i == 0) s2 -= wy * fx;
      if (i == nx - 1) s2 += wy * fx;
      if (j == 0) s2 -= wx * fy;
      if (j == ny - 1) s2 += wx * fy;
    }
  }
  double s0 = static_cast<double>(a0) - static_cast<double>(c0);
  double s1 = static_cast<double>(a1) - static_cast<double>(c1);
  for (int o = 16; o > 0; o >>= 1) {
    s0 += __shfl_xor_sync(0xffffffffu, s0, o);
    s1 += __shfl_xor_sync(0xffffffffu, s1, o);
    s2 += __shfl_xor_sync(0xffffffffu, s2, o);
  }
  if (lane == 0) {
    red[0][warp] = s0;
    red[1][warp] = s1;
    red[2][warp] = s2;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double t[3] = {0.0, 0.0, 0.0};
    for (int k = 0; k < 3; ++k)
      for (int wv = 0; wv < kBalThreads / 32; ++wv) t[k] += red[k][wv];
    double* pp = partial + (static_cast<size_t>(g) * nb + b) * 3;
    pp[0] = t[0];
    pp[1] = t[1];
    pp[2] = t[2];
    __threadfence();
    last = atomicAdd(ticket + g, 1u) == static_cast<unsigned>(nb - 1);
  }
  __syncthreads();
  if (!last || warp != 0) return;
  // the group's last block: lane l adds blocks l, l + 32, ... in order, then
  // a fixed butterfly combines the lanes
  __threadfence();
  const volatile double* pg = partial + static_cast<size_t>(g) * nb * 3;
  double t0 = 0.0, t1 = 0.0, t2 = 0.0;
  for (int bb = lane; bb < nb; bb += 32) {
    t0 += pg[3 * bb];
    t1 += pg[3 * bb + 1];
    t2 += pg[3 * bb + 2];
  }
  for (int o = 16; o > 0; o >>= 1) {
    t0 += __shfl_xor_sync(0xffffffffu, t0, o);
    t1 += __shfl_xor_sync(0xffffffffu, t1, o);
    t2 += __shfl_xor_sync(0xffffffffu, t2, o);
  }
  if (lane == 0) {
    double* o = out + (static_cast<size_t>(g) * n_steps + step) * 3;
    o[0] = w * inv_c * t0;
    o[1] = w * t1;
    o[2] = w * t2;
    ticket[g] = 0u;
  }
}

}  // namespace

int device_sms() {
  static const int n = [] {
    int dev = 0, v = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev);
    return v > 0 ? v : 1;
  }();
  return n;
}

namespace {

struct TilePlan {
  TileShape ts;
  int T, tiles;                      // outputs per thread T x T; tiles per group
  size_t smem;
};

// Tile of a pass: n positions per line, `lines` lines per group.
//
// Eight by eight outputs a thread where that leaves every SM eight warps, in
// tiles of 32 columns (256^2, M = 32, four groups: 215 us a step; 64 columns
// 242; four by four 266).  Otherwise four by four, whose threads are four
// times as many (64^2, M = 16, one group: 12 us against 26; 203 x 131, M =
// 24, three groups: 62 against 85), in the widest tile of up to 64 columns
// that still makes 128 CTAs (64^2, M = 32, four groups: 17 us with 64 columns
// and 128 CTAs, 22 with 32 and 256), and otherwise in the narrowest of at
// least four warps (64^2, M = 16, one group: 12.2 with 32, 13.3 with 64).
TilePlan plan_tile(int n, int lines, int M, int G, bool xpass) {
  TilePlan p{};
  const long long outputs = static_cast<long long>(n) * lines * M * G;
  auto tiles = [&](int per) { return (lines + per - 1) / per; };
  auto threads4 = [&](int per) { return simt_ld(n) / 4 * (per * M / 4); };
  int per = 1;
  if (outputs >= 64LL * 256 * device_sms() || threads4(1) > kMaxThreads) {
    p.T = 8;
    per = M < 32 ? 32 / M : 1;
  } else {
    p.T = 4;
    const int last = M < 64 ? 64 / M : 1;
    while (per < last && threads4(per) < 128) ++per;
    for (int k = per + 1; k <= last && threads4(k) <= kMaxThreads && static_cast<long long>(tiles(k)) * G >= 128; ++k)
      per = k;
  }
  p.ts.per_tile = per;
  p.ts.BN = per * M;
  p.ts.ntx = p.ts.BN / p.T;
  p.ts.nty = simt_ld(n) / p.T;
  p.tiles = tiles(per);
  p.smem = tile_smem(n, M, p.ts.BN, xpass);
  return p;
}

// Launches a pass with programmatic serialisation: the passes wait for the
// launch before them (griddepcontrol.wait) after their prologue and let the
// one behind them in after their GEMM, so that launch and prologue of a pass
// overlap the epilogue of the pass before (64^2, M = 16: 16.6 us a step
// without, 13.2 when let in at the start, 12 after the GEMM; let in at the
// start, a grid that leaves SMs free is followed by CTAs that crowd on those).
template <auto Kernel, class... A>
cudaError_t launch_tile(const TilePlan& p, int G, cudaStream_t s, const A&... args) {
  static const cudaError_t attr =
      cudaFuncSetAttribute(Kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 232448);
  if (attr != cudaSuccess) return attr;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(p.tiles, 1, G);
  cfg.blockDim = dim3(p.ts.ntx * p.ts.nty);
  cfg.dynamicSmemBytes = p.smem;
  cfg.stream = s;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, Kernel, args...);
}

template <int T>
cudaError_t launch_x(const TilePlan& p, const StepArgs& a, const float* U, float* R, cudaStream_t s) {
  return launch_tile<xpass_kernel<T>>(p, a.G, s, a, p.ts, U, R);
}

template <int T, bool XT>
cudaError_t launch_y(const TilePlan& p, const StepArgs& a, const BoundaryArgs& b, float* U, const float* R,
                     const float* L1, const float* L2, float* L3, int step, cudaStream_t s) {
  return launch_tile<ypass_kernel<T, XT>>(p, a.G, s, a, b, p.ts, U, R, L1, L2, L3, step, b.ring_out ? step : -1);
}

}  // namespace

cudaError_t launch_step(const StepArgs& a, const BoundaryArgs& b, float* U, float* R,
                        const float* L1, const float* L2, float* L3, int step,
                        cudaStream_t s, long long* launches, cudaEvent_t* ev) {
  if (a.tc_mode != 0) return launch_step_tc(a, b, U, R, L1, L2, L3, step, s, launches, ev);
  const TilePlan px = plan_tile(a.nx, a.ny, a.M, a.G, true), py = plan_tile(a.ny, a.nx, a.M, a.G, false);
  if (ev) cudaEventRecord(ev[0], s);
  cudaError_t e = px.T == 8 ? launch_x<8>(px, a, U, R, s) : launch_x<4>(px, a, U, R, s);
  if (ev) cudaEventRecord(ev[1], s);
  if (e == cudaSuccess) {
    if (b.bct_src)
      e = py.T == 8 ? launch_y<8, true>(py, a, b, U, R, L1, L2, L3, step, s)
                    : launch_y<4, true>(py, a, b, U, R, L1, L2, L3, step, s);
    else
      e = py.T == 8 ? launch_y<8, false>(py, a, b, U, R, L1, L2, L3, step, s)
                    : launch_y<4, false>(py, a, b, U, R, L1, L2, L3, step, s);
  }
  if (ev) cudaEventRecord(ev[2], s);
  if (launches) *launches += 2;
  return e;
}

cudaError_t launch_fluence(const float* U, float* out, size_t out_group_stride, int nx, int ny,
                           int M, int G, size_t plane, float w, cudaStream_t s,
                           long long* launches) {
  const int ncell = nx * ny;
  dim3 grid((ncell * 32 + 255) / 256, G);
  fluence_kernel<<<grid, 256, 0, s>>>(U, out, out_group_stride, ncell, M, plane, w);
  if (launches) *launches += 1;
  return cudaGetLastError();
}

cudaError_t launch_readout(const float* ring, int ring_len, int n_steps, int G,
                           const float* Wd, const int* lo, const int* hi, int n_det,
                           float* curves, double* curves64, cudaStream_t s,
                           long long* launches) {
  const long long total = static_cast<long long>(G) * n_det * n_steps;
  if (total == 0) return cudaSuccess;
  readout_kernel<<<static_cast<unsigned>((total + 255) / 256), 256, 0, s>>>(
      ring, ring_len, n_steps, G, Wd, lo, hi, n_det, curves, curves64);
  if (launches) *launches += 1;
  return cudaGetLastError();
}

cudaError_t launch_objective(const double* curves64, const float* measured, size_t n,
                             double dt, float* resid, double* partial, double* J_dev,
                             cudaStream_t s, long long* launches) {
  const int nb = 256;
  objective_partial<<<nb, 256, 0, s>>>(curves64, measured, n, resid, partial);
  objective_final<<<1, 256, 0, s>>>(partial, nb, 0.5 * dt, J_dev);
  if (launches) *launches += 2;
  return cudaGetLastError();
}

cudaError_t launch_rho(const float* resid, const float* Wn, int n_det, int ring_len,
                       int n_steps, int G, float scale, float* rho, cudaStream_t s,
                       long long* launches) {
  const long long total = static_cast<long long>(G) * n_steps * ring_len;
  if (total == 0) return cudaSuccess;
  rho_kernel<<<static_cast<unsigned>((total + 255) / 256), 256, 0, s>>>(resid, Wn, n_det, ring_len,
                                                                         n_steps, G, scale, rho);
  if (launches) *launches += 1;
  return cudaGetLastError();
}

cudaError_t launch_grad_batch(const GradJob* jobs_dev, int n_jobs, int max_ncell, int m_common, int slot,
                              int flip, cudaStream_t s, long long* launches) {
  dim3 grid((max_ncell * 32 + 255) / 256, n_jobs);
  // M in {16, 32} (every medium of a batch shares M): grad_split lanes per
  // cell, fewer than 2 kGradThreads where that is more than one
  if (m_common == 16 || m_common == 32)
    grid.x = static_cast<unsigned>((std::max<long long>(max_ncell, 2 * kGradThreads) + 255) / 256);
  grad_batch_kernel<<<grid, 256, 0, s>>>(jobs_dev, slot, flip);
  if (launches) *launches += 1;
  return cudaGetLastError();
}

cudaError_t launch_save_batch(const SaveJob* jobs_dev, int n_jobs, int slot, cudaStream_t s, long long* launches) {
  dim3 grid(4 * device_sms(), n_jobs);
  save_batch_kernel<<<grid, 256, 0, s>>>(jobs_dev, slot);
  if (launches) *launches += 1;
  return cudaGetLastError();
}

int balance_blocks(int nx, int ny, int M) {
  const long long n4 = static_cast<long long>(nx) * ny * (M / 4);
  return static_cast<int>((n4 + kBalItems * kBalThreads - 1) / (kBalItems * kBalThreads));
}

cudaError_t launch_balance(const float* U, size_t plane, int nx, int ny, int M, int G, const float* mua,
                           const double* trig, double dx, double dy, double w, double c, double* partial,
                           unsigned* ticket, double* out, int step, int n_steps, cudaStream_t s,
                           long long* launches) {
  dim3 grid(balance_blocks(nx, ny, M), G);
  balance_kernel<<<grid, kBalThreads, 0, s>>>(U, plane, nx, ny, M, mua, trig, dx, dy, w, 1.0 / c, partial,
                                              ticket, out, step, n_steps);
  if (launches) *launches += 1;
  return cudaGetLastError();
}

cudaError_t launch_grad(const float* MU, const float* Useg, const float* PT, const float* area,
                        int nx, int ny, int M, int G, size_t plane, size_t useg_group_stride,
                        double scale, int flip, GradLevels lv, double* grad_a, double* grad_b,
                        cudaStream_t s, long long* launches) {
  const int ncell = nx * ny;
  const int split = grad_split(ncell, G);
  const long long threads = (M == 16 || M == 32) ? static_cast<long long>(ncell) * split : 32LL * ncell;
  grad_kernel<<<static_cast<int>((threads + 127) / 128), 128, 0, s>>>(MU, Useg, PT, area, ncell, M, G, split, plane,
                                                                      useg_group_stride, scale, flip, lv, grad_a,
                                                                      grad_b);
  if (launches) *launches += 1;
  return cudaGetLastError();
}

cudaError_t launch_to_float(const double* in, float* out, size_t n, cudaStream_t s,
                            long long* launches) {
  to_float_kernel<<<static_cast<unsigned>((n + 255) / 256), 256, 0, s>>>(in, out, n);
  if (launches) *launches += 1;
  return cudaGetLastError();
}

}  // namespace rte_kern
