// Tile-local fused FC-DOM step for the decomposed FC operator of Sec. 4.4
// (Algorithm 1's subdomains): one CTA owns one subdomain of one group, all M
// ordinates, and does the whole step of eq. (RTEAB4) in shared memory.
//
// Subdomain (kx, ky) owns x in [x_lo, x_hi), y in [y_lo, y_hi); its FC
// segments add two fringe points on interior sides.  The derivative at an
// owned point is the row of the owner's segment operator (ox x sx, dense, a
// few KB), so the x- and y-derivatives of the whole subdomain need only the
// owned block plus a two-point halo: the "box".  Per step the CTA
//   1. copies the box of u^k (owned + halo, from the input state buffer)
//      into shared memory (cp.async);
//   2. x- and y-derivatives, side by side: half of the threads take x-lines
//      (row, four ordinates), the other half y-lines (column, four
//      ordinates); lbuf = -xi_m D_x,seg u, then lbuf += -eta_m D_y,seg u;
//   3. per node and eight ordinates, a thread: L^k = lbuf + b P~u - (a + b) u,
//      the AB4 update, the Fresnel boundary condition with beam or adjoint
//      injection on physical boundary nodes (eq. RTE), the exitance ring (eq.
//      OpMed); writes u^{k+1} to the output state buffer and L^k over the
//      oldest history slot.
// Neighbouring CTAs read this CTA's owned values as their halo during the
// same step, so input and output states are different buffers.
//
// Per update: 4 B of u (plus the halo share) + 12 B of history read, 8 B
// written: about 25 B against the two-pass form's 36 B, and 2 (s_x + s_y) +
// 2 M flops of operator and scattering work instead of 2 (n_x + n_y) + 2 M.
// The history is not staged in shared memory (that would leave one CTA per
// SM): a thread loads a node's while it works on the one before.
//
// What bounds it: shared-memory reads.  A 16-byte load returns 512 bytes a
// warp, four cycles of the SM however few distinct words it asks for.  With
// one ordinate per lane in the scattering (eight such loads for 32
// multiply-adds a lane) and two lines per thread in the derivatives (4.5 for
// 64) the loads took 16 k cycles of the SM per CTA against 4.6 k of FP32
// multiply-adds.  Eight ordinates per thread share the node's u, with the
// whole circulant in registers, and four lines share the operator: 6 k.
// 256^2, M = 32, 16 groups, 16 x 16 parts: 279 -> 192 us a step.
#include <cstdint>

#include "rte_kernels.cuh"

namespace rte_kern {

namespace {

constexpr float kAB0 = 55.0f / 24.0f, kAB1 = -59.0f / 24.0f, kAB2 = 37.0f / 24.0f,
                kAB3 = -9.0f / 24.0f;
constexpr int kFThreads = 256;
constexpr int kHalo = 2;

__device__ __forceinline__ uint32_t smem_addr(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void cp16(float* dst, const float* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_addr(dst)), "l"(src) : "memory");
}

// Shared-memory layout (floats) of one CTA for MM ordinates and at most OM
// owned points per axis; every region starts on a 16-byte boundary.  About
// 99 KB at M = 32: two CTAs per SM.
template <int MM, int OM>
struct FusedSmem {
  static constexpr int kBox = OM + 2 * kHalo;                      // box side (nodes)
  static constexpr int kN = MM + 4;                                // node stride: neighbours in different banks
  static constexpr int kRow = kBox * kN;                           // box row stride
  static constexpr int kOwn = OM * OM * kN;                        // owned values
  static constexpr int kBoxF = kBox * kRow;
  static constexpr int kOpF = (OM + 2 * kHalo) * OM;               // [k < seg][i < OM]
  static constexpr int kTotal = kBoxF + kOwn + 2 * kOpF + 2 * OM * OM;
  static constexpr size_t kBytes = static_cast<size_t>(kTotal) * sizeof(float);
};

// Two FP32 fused multiply-adds in one instruction (each rounded as fmaf).
__device__ __forceinline__ float2 fma2(float2 x, float2 y, float2 z) { return __ffma2_rn(x, y, z); }

__device__ __forceinline__ float group_sum(float v, int width) {
  for (int o = width / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// 32 bytes of global memory (32-byte aligned: eight ordinates of a node).
__device__ __forceinline__ void ld32(const float* p, float (&v)[8]) {
  asm volatile("ld.global.v8.f32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7])
               : "l"(p)
               : "memory");
}
__device__ __forceinline__ void st32(float* p, const float (&v)[8]) {
  asm volatile("st.global.v8.f32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"l"(p), "f"(v[0]), "f"(v[1]), "f"(v[2]),
               "f"(v[3]), "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7])
               : "memory");
}

// Derivative of four lines (neighbouring ordinates, u at line + k stride) at
// kOut owned points: acc[q][t] holds points 2 q and 2 q + 1 of line t.  op:
// [k][OM], the points in question first.
template <int OM, int kOut>
__device__ __forceinline__ void derive(const float* line, int stride, const float* op, int n_k,
                                       float2 (&acc)[kOut / 2][4]) {
#pragma unroll
  for (int q = 0; q < kOut / 2; ++q)
#pragma unroll
    for (int t = 0; t < 4; ++t) acc[q][t] = make_float2(0.f, 0.f);
#pragma unroll 4
  for (int k = 0; k < n_k; ++k) {
    const float4 u4 = *reinterpret_cast<const float4*>(line + k * stride);
    const float2 uu[4] = {make_float2(u4.x, u4.x), make_float2(u4.y, u4.y), make_float2(u4.z, u4.z),
                          make_float2(u4.w, u4.w)};
    const float4* dk = reinterpret_cast<const float4*>(op + k * OM);
#pragma unroll
    for (int q = 0; q < kOut / 4; ++q) {
      const float4 c = dk[q];
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        acc[2 * q][t] = fma2(make_float2(c.x, c.y), uu[t], acc[2 * q][t]);
        acc[2 * q + 1][t] = fma2(make_float2(c.z, c.w), uu[t], acc[2 * q + 1][t]);
      }
    }
  }
}

template <int MM, int OM, bool EXACT>
__global__ void __launch_bounds__(kFThreads, 2)
    fused_step_kernel(StepArgs a, BoundaryArgs b, const float* __restrict__ Uin, float* __restrict__ Uout,
                      const float* __restrict__ L1, const float* __restrict__ L2, float* __restrict__ L3,
                      int src_step, int ring_step) {
  using S = FusedSmem<MM, OM>;
  extern __shared__ __align__(16) float sm[];
  float* box = sm;                                  // [kBox][kRow]: node (x_lo-2+ib, y_lo-2+jb)
  float* lbuf = box + S::kBoxF;                     // [ny_own][nx_own][kN]
  float* dxs = lbuf + S::kOwn;                      // [k < sx][i < OM]
  float* dys = dxs + S::kOpF;                       // [k < sy][j < OM]
  float* abs_ = dys + S::kOpF;                      // [2][ny_own][nx_own]: a, b

  const int nx = a.nx, ny = a.ny, M = MM;
  const int part = blockIdx.x, g = blockIdx.y;
  const int kx = part % a.px, ky = part / a.px;
  const int x_lo = a.fxp[4 * kx], x_hi = a.fxp[4 * kx + 1], x_slo = a.fxp[4 * kx + 2], x_shi = a.fxp[4 * kx + 3];
  const int y_lo = a.fyp[4 * ky], y_hi = a.fyp[4 * ky + 1], y_slo = a.fyp[4 * ky + 2], y_shi = a.fyp[4 * ky + 3];
  // EXACT: every part owns OM x OM points (compile-time loop bounds)
  const int ox = EXACT ? OM : x_hi - x_lo, oy = EXACT ? OM : y_hi - y_lo;
  const int sx = x_shi - x_slo, sy = y_shi - y_slo;
  const int own = ox * oy;
  const int tid = threadIdx.x;
  const size_t goff = static_cast<size_t>(g) * a.plane;
  const float* Ug = Uin + goff;

  // The part's history is asked for from L2 at once (lines of 32 floats): its
  // loads come when the derivatives are done (256^2, 16 groups: 203 us a step
  // without, 194 with; loaded into registers here instead, 245: spills).
  {
    const int per_row = ox * MM / 32;
    for (int q = tid; q < oy * per_row; q += kFThreads) {
      const int row = q / per_row, c = q - row * per_row;
      const size_t at = goff + (static_cast<size_t>(y_lo + row) * nx + x_lo) * M + c * 32;
      asm volatile("prefetch.global.L2 [%0];" ::"l"(L1 + at));
      asm volatile("prefetch.global.L2 [%0];" ::"l"(L2 + at));
      asm volatile("prefetch.global.L2 [%0];" ::"l"(L3 + at));
    }
  }
  // Dependent launches: a step waits here for the step before it, and lets
  // the next one in when its derivatives are done (two groups: 33.5 us a step
  // without, 31 with).
  asm volatile("griddepcontrol.wait;" ::: "memory");
  // 1. The box of u^k by cp.async: rows of the y-segment; owned rows span the
  //    x-segment, fringe rows the owned columns.
  {
    constexpr int V = MM / 4;                       // float4 per node
    for (int r = 0; r < sy; ++r) {
      const int gj = y_slo + r;
      const bool owned_row = gj >= y_lo && gj < y_hi;
      const int c0 = owned_row ? x_slo : x_lo, c1 = owned_row ? x_shi : x_hi;
      const int items = (c1 - c0) * V;
      const float* src = Ug + (static_cast<size_t>(gj) * nx + c0) * M;
      float* dst = box + (gj - y_lo + kHalo) * S::kRow + (c0 - x_lo + kHalo) * S::kN;
      for (int e = tid; e < items; e += kFThreads) cp16(dst + e / V * S::kN + e % V * 4, src + 4 * e);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  }
  // Segment operators of this part (transposed: [k][i]), the phase matrix,
  // and the owned block of a and b.
  {
    const float* fx = a.FxT + static_cast<size_t>(kx) * S::kOpF;
    const float* fy = a.FyT + static_cast<size_t>(ky) * S::kOpF;
    for (int e = tid; e < S::kOpF; e += kFThreads) {
      dxs[e] = __ldg(fx + e);
      dys[e] = __ldg(fy + e);
    }
    for (int e = tid; e < own; e += kFThreads) {
      const int jl = e / ox, il = e - jl * ox;
      const size_t cell = static_cast<size_t>(y_lo + jl) * nx + x_lo + il;
      abs_[e] = __ldg(a.mua + cell);
      abs_[OM * OM + e] = __ldg(a.mus + cell);
    }
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();

  // 2. The derivatives: threads 0 .. 127 the x-lines of (row, ordinates 4 mq
  //    ..), the others the y-lines of (column, ...); with 16 ordinates two
  //    threads share a line's owned points.
  {
    constexpr int kHalf = kFThreads / 2, MQ = MM / 4;
    constexpr int kSplit = kHalf / (OM * MQ), kOut = OM / kSplit;
    static_assert(kSplit * OM * MQ == kHalf, "one item per thread");
    const bool xhalf = tid < kHalf;
    const int ht = xhalf ? tid : tid - kHalf;
    const int m0 = (ht % MQ) * 4, rest = ht / MQ, p0 = (rest % kSplit) * kOut, l = rest / kSplit;
    const bool on = l < (xhalf ? oy : ox);
    // interior parts have the full segment (owned range + two fringe points
    // on each side): a fixed trip count
    const int n_seg = xhalf ? sx : sy;
    const int n_k = !on ? 0 : (EXACT && n_seg == OM + 2 * kHalo) ? OM + 2 * kHalo : n_seg;
    const float* line = xhalf ? box + (l + kHalo) * S::kRow + (x_slo - x_lo + kHalo) * S::kN + m0
                              : box + (y_slo - y_lo + kHalo) * S::kRow + (l + kHalo) * S::kN + m0;
    float2 acc[kOut / 2][4];
    derive<OM, kOut>(line, xhalf ? S::kN : S::kRow, (xhalf ? dxs : dys) + p0, n_k, acc);
    const float4 w4 = __ldg(reinterpret_cast<const float4*>((xhalf ? a.xi : a.eta) + m0));
    // point p of the line: node (row l, column p) or (row p, column l)
    auto at = [&](int p) { return lbuf + (xhalf ? l * ox + p : p * ox + l) * S::kN + m0; };
    if (on && xhalf) {
#pragma unroll
      for (int i = 0; i < kOut; ++i) {
        if (p0 + i >= ox) continue;
        auto v = [&](int t) { return (i & 1) ? acc[i / 2][t].y : acc[i / 2][t].x; };
        *reinterpret_cast<float4*>(at(p0 + i)) = make_float4(-w4.x * v(0), -w4.y * v(1), -w4.z * v(2), -w4.w * v(3));
      }
    }
    __syncthreads();
    if (on && !xhalf) {
#pragma unroll
      for (int i = 0; i < kOut; ++i) {
        if (p0 + i >= oy) continue;
        auto v = [&](int t) { return (i & 1) ? acc[i / 2][t].y : acc[i / 2][t].x; };
        float4* d = reinterpret_cast<float4*>(at(p0 + i));
        const float4 x = *d;
        *d = make_float4(fmaf(-w4.x, v(0), x.x), fmaf(-w4.y, v(1), x.y), fmaf(-w4.z, v(2), x.z),
                         fmaf(-w4.w, v(3), x.w));
      }
    }
    __syncthreads();
  }

  asm volatile("griddepcontrol.launch_dependents;");
  // 3. Per node and eight ordinates mb .. mb + 7: scattering, L^k, AB4,
  //    boundary condition, exitance.  P~[m][q] = p_{(m - q) mod M}: a thread
  //    keeps p_{mb + k}, k = 0 .. M - 1.
  constexpr int NB = MM / 8, kNodes = kFThreads / NB;          // threads per node, nodes per sweep
  const int mb = (tid % NB) * 8;
  float p[MM];
#pragma unroll
  for (int k = 0; k < MM; ++k) p[k] = __ldg(a.PT + (mb + k) % MM);
  const int ring_len = 2 * ny + 2 * nx;
  const bool interior = x_lo > 0 && x_hi < nx && y_lo > 0 && y_hi < ny;   // CTA-uniform: no boundary node
  auto place = [&](int n, int& jl, int& il) {
    const int nn = n < own ? n : 0;
    jl = nn / ox;
    il = nn - jl * ox;
    return goff + (static_cast<size_t>(y_lo + jl) * nx + x_lo + il) * M + mb;
  };
  float h1[8], h2[8], h3[8];
  int jl, il;
  size_t e = place(tid / NB, jl, il);
  ld32(L1 + e, h1);
  ld32(L2 + e, h2);
  ld32(L3 + e, h3);
  for (int n0 = 0; n0 < own; n0 += kNodes) {
    const int n = n0 + tid / NB;
    const bool valid = n < own;
    float g1[8], g2[8], g3[8];
    int jn, in;
    const size_t en = place(n + kNodes, jn, in);
    const bool more = n + kNodes < own;
#pragma unroll
    for (int t = 0; t < 8; ++t) g1[t] = g2[t] = g3[t] = 0.f;
    if (more) {
      ld32(L1 + en, g1);
      ld32(L2 + en, g2);
      ld32(L3 + en, g3);
    }
    const float* un = box + (jl + kHalo) * S::kRow + (il + kHalo) * S::kN;
    float s0[8], s1[8];                                        // even and odd q
#pragma unroll
    for (int t = 0; t < 8; ++t) s0[t] = s1[t] = 0.f;
#pragma unroll
    for (int q = 0; q < MM; q += 4) {
      const float4 v = *reinterpret_cast<const float4*>(un + q);
#pragma unroll
      for (int t = 0; t < 8; ++t) {
        s0[t] = fmaf(p[(t - q + 2 * MM) % MM], v.x, s0[t]);
        s1[t] = fmaf(p[(t - q - 1 + 2 * MM) % MM], v.y, s1[t]);
        s0[t] = fmaf(p[(t - q - 2 + 2 * MM) % MM], v.z, s0[t]);
        s1[t] = fmaf(p[(t - q - 3 + 2 * MM) % MM], v.w, s1[t]);
      }
    }
    float* lb = lbuf + (jl * ox + il) * S::kN;
    const float av = abs_[jl * ox + il], bv = abs_[OM * OM + jl * ox + il];
    float lk[8], v[8];
#pragma unroll
    for (int w = 0; w < 2; ++w) {
      const float4 l4 = *reinterpret_cast<const float4*>(lb + mb + 4 * w);
      const float4 u4 = *reinterpret_cast<const float4*>(un + mb + 4 * w);
      const float ll[4] = {l4.x, l4.y, l4.z, l4.w}, uu[4] = {u4.x, u4.y, u4.z, u4.w};
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const int t = 4 * w + r;
        lk[t] = fmaf(bv, s0[t] + s1[t], ll[r] - (av + bv) * uu[r]);
        v[t] = fmaf(a.cdt, kAB0 * lk[t] + kAB1 * h1[t] + kAB2 * h2[t] + kAB3 * h3[t], uu[r]);
      }
    }
    if (valid) st32(L3 + e, lk);
    if (!interior) {
      const int gj = y_lo + jl, gi = x_lo + il;
      const bool lf = gi == 0, rt = gi == nx - 1, bt = gj == 0, tp = gj == ny - 1;
      const bool bnd = valid && (lf || rt || bt || tp);
      if (__any_sync(0xffffffffu, bnd)) {
        // pre-BC values through shared memory (this node's lbuf entries are
        // no longer needed)
        if (bnd) {
          *reinterpret_cast<float4*>(lb + mb) = make_float4(v[0], v[1], v[2], v[3]);
          *reinterpret_cast<float4*>(lb + mb + 4) = make_float4(v[4], v[5], v[6], v[7]);
        }
        __syncwarp();
        float ex = 0.f, ey = 0.f;
        if (bnd) {
          const int* refl;
          const float* fco;
          const unsigned char* act;
          if ((lf || rt) && (bt || tp)) {
            const int c = (rt ? 1 : 0) + (tp ? 2 : 0);
            refl = b.corner_refl + c * M; fco = b.corner_f + c * M; act = b.corner_act + c * M;
          } else {
            const int F = lf ? 0 : rt ? 1 : bt ? 2 : 3;
            refl = b.face_refl + F * M; fco = b.face_f + F * M; act = b.face_act + F * M;
          }
          const int node = lf ? gj : rt ? ny + gj : bt ? 2 * ny + gi : 2 * ny + nx + gi;
          float q[8];
#pragma unroll
          for (int t = 0; t < 8; ++t) q[t] = 0.f;
          for (int k = 0; k < b.kmax; ++k) {
            const size_t gk = static_cast<size_t>(g) * b.kmax + k;
            const float sk = __ldg(b.S + gk * ring_len + node), tk = __ldg(b.T + gk * b.T_len + src_step);
#pragma unroll
            for (int t = 0; t < 8; ++t) q[t] = fmaf(sk * __ldg(b.A + gk * M + mb + t), tk, q[t]);
          }
          const float rho =
              b.rho ? __ldg(b.rho + (static_cast<size_t>(g) * b.rho_len + src_step) * ring_len + node) : 0.f;
#pragma unroll
          for (int t = 0; t < 8; ++t) {
            if (act[mb + t]) {
              const float fc = __ldg(fco + mb + t);
              if (b.rho) q[t] = fmaf(1.0f - fc, rho, q[t]);
              v[t] = fmaf(fc, lb[__ldg(refl + mb + t)], q[t]);
            }
            // exitance of the node's faces (eq. OpMed)
            if (lf || rt) ex = fmaf(__ldg(b.wexit + (lf ? 0 : 1) * M + mb + t), v[t], ex);
            if (bt || tp) ey = fmaf(__ldg(b.wexit + (bt ? 2 : 3) * M + mb + t), v[t], ey);
          }
        }
        ex = group_sum(ex, NB);
        ey = group_sum(ey, NB);
        if (bnd && mb == 0 && b.ring_out && ring_step >= 0) {
          float* ro = b.ring_out + (static_cast<size_t>(g) * b.ring_steps + ring_step) * ring_len;
          if (lf || rt) ro[lf ? gj : ny + gj] = ex;
          if (bt || tp) ro[bt ? 2 * ny + gi : 2 * ny + nx + gi] = ey;
        }
      }
    }
    if (valid) st32(Uout + e, v);
    e = en;
    jl = jn;
    il = in;
#pragma unroll
    for (int t = 0; t < 8; ++t) {
      h1[t] = g1[t];
      h2[t] = g2[t];
      h3[t] = g3[t];
    }
  }
}

template <int MM, int OM, bool EXACT>
cudaError_t launch_fused_t(const StepArgs& a, const BoundaryArgs& b, const float* Uin, float* Uout,
                           const float* L1, const float* L2, float* L3, int src_step, int ring_step,
                           cudaStream_t s) {
  using S = FusedSmem<MM, OM>;
  static bool attr_done = false;
  if (!attr_done) {
    cudaError_t e = cudaFuncSetAttribute(fused_step_kernel<MM, OM, EXACT>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(S::kBytes));
    if (e != cudaSuccess) return e;
    attr_done = true;
  }
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(a.px * a.py, a.G);
  cfg.blockDim = dim3(kFThreads);
  cfg.dynamicSmemBytes = S::kBytes;
  cfg.stream = s;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, fused_step_kernel<MM, OM, EXACT>, a, b, Uin, Uout, L1, L2, L3, src_step, ring_step);
}

template <int MM>
cudaError_t launch_fused_m(const StepArgs& a, const BoundaryArgs& b, const float* Uin, float* Uout,
                           const float* L1, const float* L2, float* L3, int src_step, int ring_step,
                           cudaStream_t s) {
  return a.fused_exact ? launch_fused_t<MM, kFusedOwnMax, true>(a, b, Uin, Uout, L1, L2, L3, src_step, ring_step, s)
                       : launch_fused_t<MM, kFusedOwnMax, false>(a, b, Uin, Uout, L1, L2, L3, src_step, ring_step, s);
}

}  // namespace

bool fused_supported(const StepArgs& a) {
  if (a.px < 2 || a.py < 2 || !a.FxT || !a.FyT || !a.fxp || !a.fyp) return false;
  return (a.M == 16 || a.M == 32) && a.fused_own_max <= kFusedOwnMax;
}

cudaError_t launch_step_fused(const StepArgs& a, const BoundaryArgs& b, const float* Uin, float* Uout,
                              const float* L1, const float* L2, float* L3, int step, cudaStream_t s,
                              long long* launches, cudaEvent_t* ev) {
  const int ring_step = b.ring_out ? step : -1;
  if (ev) {
    cudaEventRecord(ev[0], s);
    cudaEventRecord(ev[1], s);
  }
  const cudaError_t e = a.M == 16 ? launch_fused_m<16>(a, b, Uin, Uout, L1, L2, L3, step, ring_step, s)
                                  : launch_fused_m<32>(a, b, Uin, Uout, L1, L2, L3, step, ring_step, s);
  if (ev) cudaEventRecord(ev[2], s);
  if (launches) *launches += 1;
  return e;
}

}  // namespace rte_kern
