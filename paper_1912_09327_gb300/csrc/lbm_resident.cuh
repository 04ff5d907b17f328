// Several LBMTau1 steps per launch on regions held in registers.
//
// What bounds one launch per step: small domains pay a launch and the serial
// chain of a warp's marched rows (10 to 14 us a step from 64 x 32 to 1024^2,
// where the arithmetic of all nodes is below 3 us), large ones the two trips
// through memory (24 B a node).  Here a block loads a region of 64 columns x
// (kR * warps) rows once, takes up to `steps` steps on it in registers and
// stores the nodes that no missing neighbour has reached: a region's rim goes
// stale by one node per step, so regions overlap by that much.  The inner
// steps of lbm_step run this way, and its reduced last one as a launch of one
// step (below).
//
// Layout: a lane holds two adjacent columns (one packed pair) of kR rows, a
// warp all 64 columns.  Two columns and eight rows keep the same 16 nodes in a
// lane as four columns and four rows, with half the temporaries per row: the
// march over the rows fits 128 registers, so 16 warps are resident (the
// single-step kernel holds 12).  Left and right neighbours come by shuffle;
// what a warp's first and last row add to the warps below and above goes
// through shared memory (double-buffered: one barrier a step), as sums, so no
// row is computed twice.  No more than the node types' 9-bit wall codes and
// those sums are in shared memory.  The time loop exists twice: a block with no
// wall and no kept node in or around its rows takes the copy without the wall
// terms' tests and branches (4096^2 box: 62 -> 52.6 us a step; the tests cost
// issue slots, and their code instruction fetches: 1.07 no-instruction stalls
// per issue before, 0.24 after).
//
// The multiphase step runs here too, in two passes a step with a barrier each:
// the potentials and their horizontal terms give every row its force, which is
// added to the momentum in its registers; then the single-phase step.  Its
// result reaches two nodes to each side, so a region's rim goes stale by two
// nodes a step (drop 2048^2: 61.8 us a step launched one by one, 21.1 here in
// launches of two).
//
// A call's reduced last step runs here as a launch of one step (us per
// lbm_step(ctx, 1), single-step kernel -> this, with the finalize: 64^2
// 24.6 -> 6.5, 1024^2 26.6 -> 15.2, 2048^2 59 -> 36, 4096^2 156 -> 121), except
// where a large domain's tiles are mostly clean (choose_reduce).
//
// Every node's arithmetic is that of step_tile (lbm_kernels.cuh), operation by
// operation, and 16-bit formats round to storage after every step with the
// random bits of the node's own place: the states are equal bit for bit.
//
// Measured (us per step in runs of 200, one launch per step -> this, FP32
// periodic boxes): 256^2 12.0 -> 0.96, 512^2 12.1 -> 1.45, 1024^2 14.2 -> 4.5,
// 2048^2 40.7 -> 13.5, 4096^2 114 -> 49.1, 8192^2 312 -> 188, 16384^2 1062 ->
// 737 (364 k MLUPS: more than one trip through memory per step allows).  The
// next launch's early start is worth 14 % at 1024^2 (5.1 -> 4.4 us a step) and
// 1.6 % at 4096^2.  A step on full SMs runs at 500 k MLUPS before the overlap
// and the loads are paid for; the FMA pipe, which a packed operation holds for
// two cycles, is 68 % busy then.
#pragma once

#include "lbm_kernels.cuh"

namespace lbmtau1 {
namespace {

constexpr int kResCols = 2;                     // columns per lane
constexpr int kResWidth = kLanes * kResCols;    // columns of a region
constexpr int kResMaxWarps = 16;

// What a warp hands its neighbours each step, one slot per lane: the sums a
// boundary row adds to the row beyond it, and that row's momentum.
struct alignas(16) EdgeA {
  float2 dd, mx;
};
struct alignas(16) EdgeB {
  float2 my, zx;
};
struct Edge {
  EdgeA a[kLanes];
  EdgeB b[kLanes];
  float2 zy[kLanes];
};

// The multiphase step's boundary rows: their potential and its horizontal
// difference and sum.
struct PsiEdge {
  float2 c[kLanes], a[kLanes], s[kLanes];
};
static_assert(sizeof(PsiEdge) <= sizeof(Edge), "shares the edges' buffer");

template <int kR, bool kSC>
__host__ __device__ constexpr int resident_smem(int warps) {
  return 512 * static_cast<int>(sizeof(SolidSums)) +
         warps * (4 * static_cast<int>(sizeof(Edge)) +
                  kR * kLanes * (kSC ? 4 + 16 : 4));
}

// 1 / x as __fdividef(1, x) rounds it, without the product by one.
__device__ __forceinline__ float rcp(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

// One step's values of a column pair, rounded to the storage format and back
// (exactly what a store and a load do).  (c0, c1): the domain's columns of
// the pair, whose random bits are those of the pair they are stored in; whole:
// every lane of the warp holds a stored pair.
template <typename T, bool kSr>
__device__ __forceinline__ void round_pair(float2 &d, float2 &x, float2 &y,
                                           uint32_t key, uint32_t c0,
                                           uint32_t c1, bool whole) {
  using S = Storage<T>;
  if constexpr (!std::is_same<T, float>::value) {
    const float2 sd = bc(S::kD), sj = bc(S::kJ);
    const float2 id = bc(1.0f / S::kD), ij = bc(1.0f / S::kJ);
    union {
      uint32_t w;
      T e[2];
    } u[3];
    auto times = [](float2 v, float2 by, bool one) {
      return one ? v : __fmul2_rn(v, by);
    };
    const float2 v[3] = {times(d, sd, S::kD == 1.0f),
                         times(x, sj, S::kJ == 1.0f),
                         times(y, sj, S::kJ == 1.0f)};
    if constexpr (kSr) {
      const uint32_t h0 = fmix32(key + (c0 & ~1u) * 0x9e3779b1u);
#pragma unroll
      for (int f = 0; f < 3; ++f)
        u[f].w = pack_sr(T(), v[f].x, v[f].y,
                         __funnelshift_l(h0, h0, 11 * f));
      if (!whole) {  // a wrapped pair of an odd width: column by column
        const uint32_t h1 = fmix32(key + (c1 & ~1u) * 0x9e3779b1u);
#pragma unroll
        for (int f = 0; f < 3; ++f) {
          union {
            uint32_t w;
            T e[2];
          } p, q;
          p.w = pack_sr(T(), v[f].x, v[f].x, __funnelshift_l(h0, h0, 11 * f));
          q.w = pack_sr(T(), v[f].y, v[f].y, __funnelshift_l(h1, h1, 11 * f));
          u[f].e[0] = (c0 & 1u) ? p.e[1] : p.e[0];
          u[f].e[1] = (c1 & 1u) ? q.e[1] : q.e[0];
        }
      }
    } else {
#pragma unroll
      for (int f = 0; f < 3; ++f) {
        u[f].e[0] = S::encode(v[f].x);
        u[f].e[1] = S::encode(v[f].y);
      }
    }
    d = times(make_float2(S::decode(u[0].e[0]), S::decode(u[0].e[1])), id,
              S::kD == 1.0f);
    x = times(make_float2(S::decode(u[1].e[0]), S::decode(u[1].e[1])), ij,
              S::kJ == 1.0f);
    y = times(make_float2(S::decode(u[2].e[0]), S::decode(u[2].e[1])), ij,
              S::kJ == 1.0f);
  }
}

// Takes nsteps steps on region (bx, by) (kSC: Shan-Chen multiphase steps;
// kReduce: one step, whose residual and mass terms become the region's partial
// triple; kForce: the body force is not zero, whose sums are left out
// otherwise: 5 of the 51 packed operations of a pair); every thread of the
// block calls it.
template <typename T, int kR, bool kSr, bool kSC, bool kReduce, bool kForce>
__device__ __forceinline__ void resident_region(const StepLaunch &a,
                                                const ResidentTiles &g, int bx,
                                                int by, int nsteps,
                                                unsigned char *smem) {
  using S = Storage<T>;
  constexpr bool kF32 = std::is_same<T, float>::value;
  // In blocks with walls every row takes the wall terms and the kept nodes'
  // selects without a test (rows of porous samples and of small domains mostly
  // need them, and three tests a row cost their branches' instruction fetches:
  // porous 2048^2 20.0 -> 17.4 us a step, 48 batched domains 37 -> 33.6, cavity
  // 256^2 1.04 -> 0.97).  Not where that lost: with 8 rows and no force the
  // registers it takes spill in the wall-free loop as well (ptxas: 48 bytes of
  // spill stores instead of 16; box 4096^2 49 -> 51), and with 2 rows and a
  // force (channel 64 x 32, the one domain it was measured on, +5 %).
  constexpr bool kFlat = kR == 4 || (kR == 8) == kForce;
  SolidSums *lut = reinterpret_cast<SolidSums *>(smem);
  const int warps = blockDim.x / kLanes;
  Edge *edges = reinterpret_cast<Edge *>(smem + 512 * sizeof(SolidSums));
  unsigned *codes = reinterpret_cast<unsigned *>(edges + 4 * warps);
  // kSC: the momentum of kept nodes, which the force does not change (a
  // node's register holds its momentum with the force while a step goes on)
  float4 *kept = reinterpret_cast<float4 *>(codes + warps * kR * kLanes);
  const int lane = threadIdx.x & (kLanes - 1), w = threadIdx.x / kLanes;

  // The region: its first column and row, and the outputs it owns.
  const int nx = static_cast<int>(a.nx), ny = static_cast<int>(a.ny);
  const int64_t pitch = a.pitch;
  const int x0 = bx * g.ox - g.lead_x, y0 = by * g.oy - g.lead_y;
  const int xb = x0 + kResCols * lane, yb = y0 + w * kR;
  const int xlo = a.periodic_x || bx > 0 ? x0 + g.hx : 0;
  const int xhi = a.periodic_x || bx + 1 < g.gx
                      ? min(x0 + kResWidth - g.hx, nx) : nx;
  const int ylo = a.periodic_y || by > 0 ? y0 + g.hy : 0;
  const int yhi = a.periodic_y || by + 1 < g.gy
                      ? min(y0 + warps * kR - g.hy, ny) : ny;

  // columns of this lane in the domain (-1: outside)
  auto wrap = [](int v, int n, int periodic) -> int {
    if (v >= 0 && v < n) return v;
    return periodic ? static_cast<int>(wrap_index(v, n)) : -1;
  };
  const int c0 = wrap(xb, nx, a.periodic_x), c1 = wrap(xb + 1, nx, a.periodic_x);
  const bool vec =
      __all_sync(kFull, (c0 & 1) == 0 && c1 == c0 + 1 && c0 >= 0);
  // the row whose random bits lane r < kR keeps (16-bit formats)
  const int key_row = a.periodic_y ? wrap(yb + lane % kR, ny, 1)
                                   : yb + lane % kR;
  const float fx = a.fx, fy = a.fy;

  // Node types and fields of the region's rows: all loads first, then what is
  // derived from them.  A region that lies in the domain with the rows around
  // it needs no index of its own per row and column: one 32-bit offset per row
  // serves the four planes (a 64-bit index per row, column and plane took 8 %
  // of the instructions of a three-step launch: box 4096^2 52.6 -> 50.7 us a
  // step, 64 x 32 regions 69 -> 59).
  unsigned m0[kR + 2], m1[kR + 2];  // rows yb - 1 .. yb + kR
  unsigned inside = (1u << (kR + 2)) - 1u;
  float2 d[kR], zx[kR], zy[kR];
  const T *sd = static_cast<const T *>(a.src.d);
  const T *sx = static_cast<const T *>(a.src.jx);
  const T *sy = static_cast<const T *>(a.src.jy);
  // (its blocks with walls build their table below)
  const bool inner = x0 >= 0 && x0 + kResWidth <= nx && y0 >= 1 &&
                     y0 + warps * kR < ny;
  const int64_t corner = static_cast<int64_t>(y0) * pitch + x0;
  const unsigned step_y = static_cast<unsigned>(pitch);
  const unsigned mine0 = static_cast<unsigned>(w * kR) * step_y +
                         static_cast<unsigned>(kResCols * lane);
  if (inner) {
    const uint8_t *pm = a.mask + (corner - pitch);
#pragma unroll
    for (int r = 0; r < kR + 2; ++r)
      m0[r] = *reinterpret_cast<const unsigned short *>(
          pm + (mine0 + r * step_y));
    pdl_wait();  // the fields: written by the launch before this one
    sd += corner;
    sx += corner;
    sy += corner;
#pragma unroll
    for (int r = 0; r < kR; ++r) {
      const unsigned o = mine0 + r * step_y;
      float2 t[1];
      load_pairs<2, T>(sd + o, t, 1.0f / S::kD);
      d[r] = t[0];
      load_pairs<2, T>(sx + o, t, 1.0f / S::kJ);
      zx[r] = t[0];
      load_pairs<2, T>(sy + o, t, 1.0f / S::kJ);
      zy[r] = t[0];
    }
#pragma unroll
    for (int r = 0; r < kR + 2; ++r) {
      m1[r] = m0[r] >> 8;
      m0[r] &= 0xffu;
    }
  } else {
    // rows and columns outside the domain read some inside node and count as
    // solid
    build_solid_lut(lut);
    const int q0 = max(c0, 0), q1 = max(c1, 0);
    int64_t off[kR + 2];
    inside = 0u;
#pragma unroll
    for (int r = 0; r < kR + 2; ++r) {
      const int row = wrap(yb + r - 1, ny, a.periodic_y);
      inside |= (row >= 0 ? 1u : 0u) << r;
      off[r] = static_cast<int64_t>(max(row, 0)) * pitch;
    }
    if (vec) {
#pragma unroll
      for (int r = 0; r < kR + 2; ++r)
        m0[r] = *reinterpret_cast<const unsigned short *>(a.mask + off[r] + q0);
#pragma unroll
      for (int r = 0; r < kR + 2; ++r) {
        m1[r] = m0[r] >> 8;
        m0[r] &= 0xffu;
      }
    } else {
#pragma unroll
      for (int r = 0; r < kR + 2; ++r) {
        m0[r] = a.mask[off[r] + q0];
        m1[r] = a.mask[off[r] + q1];
      }
    }
    pdl_wait();  // the fields: written by the launch before this one
    if (vec) {
#pragma unroll
      for (int r = 0; r < kR; ++r) {
        float2 t[1];
        load_pairs<2, T>(sd + off[r + 1] + q0, t, 1.0f / S::kD);
        d[r] = t[0];
        load_pairs<2, T>(sx + off[r + 1] + q0, t, 1.0f / S::kJ);
        zx[r] = t[0];
        load_pairs<2, T>(sy + off[r + 1] + q0, t, 1.0f / S::kJ);
        zy[r] = t[0];
      }
    } else {
#pragma unroll
      for (int r = 0; r < kR; ++r) {
        const int64_t o = off[r + 1];
        d[r] = make_float2(S::decode(sd[o + q0]) * (1.0f / S::kD),
                           S::decode(sd[o + q1]) * (1.0f / S::kD));
        zx[r] = make_float2(S::decode(sx[o + q0]) * (1.0f / S::kJ),
                            S::decode(sx[o + q1]) * (1.0f / S::kJ));
        zy[r] = make_float2(S::decode(sy[o + q0]) * (1.0f / S::kJ),
                            S::decode(sy[o + q1]) * (1.0f / S::kJ));
      }
    }
  }
  unsigned walls = 0u, keep = 0u;  // rows with solid neighbours / kept nodes
  unsigned any = 0u;
#pragma unroll
  for (int r = 0; r < kR + 2; ++r) any |= m0[r] | m1[r];
  any |= (c0 < 0 || c1 < 0 || inside != (1u << (kR + 2)) - 1u) ? 1u : 0u;
  bool any_walls = false;
  if constexpr (kFlat) any_walls = __syncthreads_or(any != 0u);
  if (kFlat ? any_walls : __any_sync(kFull, any != 0u) != 0) {
    // solid bits of a row's columns -1 .. 2, and its fluid bits
    auto types = [&](int r, unsigned &fluid) -> unsigned {
      const bool in = (inside >> r) & 1u;
      const unsigned t0 = in && c0 >= 0 ? m0[r] : 1u;
      const unsigned t1 = in && c1 >= 0 ? m1[r] : 1u;
      fluid = (t0 == 0u ? 1u : 0u) | (t1 == 0u ? 2u : 0u);
      const unsigned s = (t0 == 1u ? 1u : 0u) | (t1 == 1u ? 2u : 0u);
      const unsigned l = __shfl_up_sync(kFull, s, 1);
      const unsigned p = __shfl_down_sync(kFull, s, 1);
      return (l >> 1) | (s << 1) | ((p & 1u) << 3);
    };
    unsigned fl, fc, fn;
    unsigned lo = types(0, fl), own = types(1, fc);
#pragma unroll
    for (int r = 0; r < kR; ++r) {
      const unsigned hi = types(r + 2, fn);
      const unsigned i0 = (lo & 7u) | ((own & 7u) << 3) | ((hi & 7u) << 6);
      const unsigned i1 = (lo >> 1) | ((own >> 1) << 3) | ((hi >> 1) << 6);
      codes[(w * kR + r) * kLanes + lane] = i0 | (i1 << 9) | (fc << 18);
      if (__any_sync(kFull, (lo | own | hi) != 0u)) walls |= 1u << r;
      if (__any_sync(kFull, fc != 3u)) keep |= 1u << r;
      // a solid node's momentum as a source: -F (zero momentum j + F)
      if (own & 2u) { d[r].x = 0.f; zx[r].x = -fx; zy[r].x = -fy; }
      if (own & 4u) { d[r].y = 0.f; zx[r].y = -fx; zy[r].y = -fy; }
      if constexpr (kSC)
        kept[(w * kR + r) * kLanes + lane] =
            make_float4(zx[r].x, zx[r].y, zy[r].x, zy[r].y);
      lo = own;
      own = hi;
      fc = fn;
    }
  }
  if constexpr (!kFlat) any_walls = __syncthreads_or((walls | keep) != 0u);
  pdl_release();
  if (any_walls && inner) {
    build_solid_lut(lut);
    __syncthreads();
  }

  const float2 F2x = bc(fx), F2y = bc(fy), F22y = bc(2.0f * fy);
  const float2 one = bc(1.0f), c3 = bc(3.0f), cm15 = bc(-1.5f);
  const float2 w1_9 = bc(k1_9), w1_36 = bc(k1_36), w1_12 = bc(k1_12),
               w1_3 = bc(k1_3), w4_9 = bc(k4_9), w1_6 = bc(k1_6),
               wm1_6 = bc(-k1_6), half = bc(0.5f), mhalf = bc(-0.5f),
               quarter = bc(0.25f);

  auto with_force = [](float2 v, float2 f) { return kForce ? add(v, f) : v; };

  // The residual's and the mass's sums, as step_tile takes them: FP32 per lane
  // (the mass compensated over the rows), FP64 from the warps' sums on.
  float2 rs_num = bc(0.f), rs_den = bc(0.f);
  float rs_mass = 0.f, rs_comp = 0.f, rmin = 1.0f;
  const bool own_cols = xb >= xlo && xb < xhi;
  auto add_terms = [&](float2 dO, float2 xO, float2 yO, float2 dn, float2 xn,
                       float2 yn, bool v0, bool v1) {
    const float2 rn = add(dn, bc(1.0f));
    const float2 irn = make_float2(rcp(rn.x), rcp(rn.y));
    const float2 irn2 = mul(irn, irn);
    const float2 t = mul(sub(dO, dn), irn);
    const float2 ex = fma2(xO, t, sub(xn, xO));
    const float2 ey = fma2(yO, t, sub(yn, yO));
    const float2 nn = fma2(ex, ex, mul(ey, ey));
    const float2 dd = fma2(xn, xn, mul(yn, yn));
    float m = 0.f;
    if (v0) {
      rs_num.x = fmaf(nn.x, irn2.x, rs_num.x);
      rs_den.x = fmaf(dd.x, irn2.x, rs_den.x);
      m += dn.x;
      rmin = fminf(rmin, rn.x);
    }
    if (v1) {
      rs_num.y = fmaf(nn.y, irn2.y, rs_num.y);
      rs_den.y = fmaf(dd.y, irn2.y, rs_den.y);
      m += dn.y;
      rmin = fminf(rmin, rn.y);
    }
    const float y = __fsub_rn(m, rs_comp);
    const float u = __fadd_rn(rs_mass, y);
    rs_comp = __fsub_rn(__fsub_rn(u, rs_mass), y);
    rs_mass = u;
  };

  // kWalls: some row of the block has solid neighbours or kept nodes
  auto march = [&](auto with_walls) {
    constexpr bool kWalls = decltype(with_walls)::value;
    for (int t = 0; t < nsteps; ++t) {
      const float2 dither = bc(kF32 && kSr ? fp32_dither(a.step + t) : 0.0f);
      // stochastic rounding: lane r holds the key of row r and this step (all
      // lanes hashing every row's took 8 of a pair's 48 integer operations;
      // with it, and no test per lane for a wrapped pair: FP16 4096^2
      // 74.3 -> 62.5 us a step, 1024^2 7.0 -> 5.7)
      uint32_t row_keys = 0u;
      if constexpr (!kF32 && kSr)
        row_keys = fmix32(fmix32(a.step + t) ^
                          (static_cast<uint32_t>(key_row) * 0x85ebca77u));
      // [0] down, [1] up (kSC: two barriers a step, so one buffer; the other
      // holds the potentials)
      Edge *mine = edges + ((kSC ? 0 : t & 1) * warps + w) * 2;
      if constexpr (kSC) {
        // The force of every row (Eq. f_sc; the terms and their order are
        // step_tile's), added to its momentum.
        struct Psi {
          float2 c, a, s;
        };
        const float2 mg = bc(-a.g_sc), one = bc(1.0f);
        const float2 w1_9 = bc(k1_9), w1_36 = bc(k1_36);
        auto terms = [&](int r) -> Psi {
          const float2 rho = add(d[r], one);
          float2 c = make_float2(1.0f - __expf(-rho.x), 1.0f - __expf(-rho.y));
          if (kWalls && (kFlat || ((walls >> r) & 1u))) {
            const unsigned code = codes[(w * kR + r) * kLanes + lane];
            if (code & (1u << 4)) c.x = 0.f;   // the node's own solid bit
            if (code & (1u << 13)) c.y = 0.f;
          }
          const float l = __shfl_up_sync(kFull, c.y, 1);
          const float p = __shfl_down_sync(kFull, c.x, 1);
          return {c, make_float2(__fsub_rn(c.y, l), __fsub_rn(p, c.x)),
                  make_float2(__fadd_rn(c.y, l), __fadd_rn(p, c.x))};
        };
        auto force = [&](int r, const Psi &lo, const Psi &own, const Psi &hi) {
          const float2 k = mul(own.c, mg);
          const float2 sx = fma2(w1_36, add(lo.a, hi.a), mul(w1_9, own.a));
          const float2 sy =
              fma2(w1_9, sub(hi.c, lo.c), mul(w1_36, sub(hi.s, lo.s)));
          zx[r] = add(zx[r], mul(k, sx));
          zy[r] = add(zy[r], mul(k, sy));
        };
        PsiEdge *psi = reinterpret_cast<PsiEdge *>(edges + 2 * warps) + 2 * w;
        Psi lo, own, r0, r1;
#pragma unroll
        for (int r = 0; r < kR; ++r) {
          const Psi now = terms(r);
          if (r == 0 || r == kR - 1) {
            PsiEdge &e = psi[r == 0 ? 0 : 1];
            e.c[lane] = now.c;
            e.a[lane] = now.a;
            e.s[lane] = now.s;
          }
          if (r == 0) r0 = now;
          if (r == 1) r1 = now;
          if (r > 1) force(r - 1, lo, own, now);
          if (r > 0) lo = own;
          own = now;
        }
        __syncthreads();
        auto edge = [&](bool there, const PsiEdge *e) -> Psi {
          if (!there) return {bc(0.f), bc(0.f), bc(0.f)};
          return {e->c[lane], e->a[lane], e->s[lane]};
        };
        force(0, edge(w > 0, psi - 1), r0, r1);
        force(kR - 1, lo, own, edge(w + 1 < warps, psi + 2));
      }

      // completes row r: acc holds South(r - 1) + Same(r) with the vertical
      // difference to row r - 1, (nd, nx_, ny_) the row above's contribution
      // and (ex, ey) its momentum less the row's own
      auto finish = [&](int r, float2 ad, float2 ax, float2 ay, float2 nd,
                        float2 nmx, float2 nmy, float2 ex, float2 ey) {
        const float2 dO = d[r], zxO = zx[r], zyO = zy[r];
        float2 dn = add(ad, nd);
        float2 incx = fma2(w1_6, ex, with_force(add(ax, nmx), F2x));
        float2 incy = fma2(half, ey, with_force(add(ay, nmy), F2y));
        unsigned code = 0u;
        if (kWalls && (kFlat || (((walls | keep) >> r) & 1u)))
          code = codes[(w * kR + r) * kLanes + lane];
        if (kWalls && (kFlat || ((walls >> r) & 1u))) {
          const SolidSums E0 = lut[code & 511u], E1 = lut[(code >> 9) & 511u];
          dn.x = fmaf(dO.x, E0.s0, dn.x);
          incx.x = fmaf(dO.x, E0.sx, incx.x);
          incy.x = fmaf(dO.x, E0.sy, incy.x);
          dn.y = fmaf(dO.y, E1.s0, dn.y);
          incx.y = fmaf(dO.y, E1.sx, incx.y);
          incy.y = fmaf(dO.y, E1.sy, incy.y);
        }
        if constexpr (kF32 && kSr) {
          incx = fma2(lead_pow2(zxO), dither, incx);
          incy = fma2(lead_pow2(zyO), dither, incy);
        }
        float2 xn = add(zxO, incx), yn = add(zyO, incy);
        if constexpr (kReduce) {
          const bool own = own_cols && yb + r >= ylo && yb + r < yhi;
          const unsigned fluid =
              kWalls && (kFlat || ((keep >> r) & 1u)) ? code >> 18 : 3u;
          add_terms(dO, zxO, zyO, dn, xn, yn, own && (fluid & 1u),
                    own && (fluid & 2u) && xb + 1 < nx);
        }
        if constexpr (!kF32)
          round_pair<T, kSr>(dn, xn, yn,
                             kSr ? __shfl_sync(kFull, row_keys, r) : 0u,
                             static_cast<uint32_t>(c0),
                             static_cast<uint32_t>(c1), vec);
        if (kWalls && (kFlat || ((keep >> r) & 1u))) {
          const bool f0 = (code >> 18) & 1u, f1 = (code >> 19) & 1u;
          float2 xk = zxO, yk = zyO;
          if constexpr (kSC) {
            const float4 k = kept[(w * kR + r) * kLanes + lane];
            xk = make_float2(k.x, k.y);
            yk = make_float2(k.z, k.w);
          }
          dn = make_float2(f0 ? dn.x : dO.x, f1 ? dn.y : dO.y);
          xn = make_float2(f0 ? xn.x : xk.x, f1 ? xn.y : xk.y);
          yn = make_float2(f0 ? yn.x : yk.x, f1 ? yn.y : yk.y);
        }
        d[r] = dn;
        zx[r] = xn;
        zy[r] = yn;
      };

      float2 acd, acx, acy;              // South(r - 1) + Same(r)
      float2 td, tx, ty;                 // South(r)
      float2 s0d, s0x;                   // Same(0)
      float2 n1d, n1x, n1y, e1x, e1y;    // North(1) and z(1) - z(0)
#pragma unroll
      for (int r = 0; r < kR; ++r) {
        const float2 dc = d[r], zxC = zx[r], zyC = zy[r];
        const float2 mx = with_force(zxC, F2x), my = with_force(zyC, F2y);
        const float2 rho = add(dc, one);
        const float2 ir = make_float2(rcp(rho.x), rcp(rho.y));
        const float2 q = mul(mx, ir);
        const float2 pxx = mul(q, mx), pxy = mul(q, my);
        const float2 pyy = mul(mul(my, my), ir);
        const float2 tr = add(pxx, pyy);
        const float2 K = fma2(w1_9, dc, fma2(w1_3, pxx, mul(wm1_6, pyy)));
        const float2 P = fma2(c3, pyy, fma2(cm15, pxx, dc));
        const float2 G = fma2(w1_12, tr, mul(w1_36, dc));
        const float2 X = mul(quarter, pxy);
        const float2 R0 = fma2(cm15, tr, dc);
        struct Halo {
          float m, p;
        };
        auto halo = [&](float2 v) -> Halo {
          return {__shfl_up_sync(kFull, v.y, 1),
                  __shfl_down_sync(kFull, v.x, 1)};
        };
        const Halo hK = halo(K), hG = halo(G), hX = halo(X);
        const Halo hZx = halo(zxC), hZy = halo(zyC);
        auto lpr = [](float2 v, Halo h) {
          return make_float2(__fadd_rn(h.m, v.y), __fadd_rn(v.x, h.p));
        };
        auto lmr = [](float2 v, Halo h) {
          return make_float2(__fsub_rn(h.m, v.y), __fsub_rn(v.x, h.p));
        };
        // (left - own) + (right - own), both differences exact
        auto second = [](float2 v, Halo h) {
          const float e = __fsub_rn(v.y, v.x);
          return make_float2(__fadd_rn(__fsub_rn(h.m, v.x), e),
                             __fsub_rn(__fsub_rn(h.p, v.y), e));
        };
        const float2 Ks = lpr(K, hK), Kd = lmr(K, hK);
        const float2 Gs = lpr(G, hG), Gd = lmr(G, hG);
        const float2 Xs = lpr(X, hX), Xd = lmr(X, hX);
        const float2 mxd = lmr(zxC, hZx), myd = lmr(zyC, hZy);
        const float2 mys = with_force(lpr(zyC, hZy), F22y);
        const float2 hx = second(zxC, hZx), hy = second(zyC, hZy);
        const float2 U = fma2(w1_9, P, fma2(w1_12, mxd, Gs));
        const float2 V = fma2(w1_3, my, fma2(w1_12, mys, Xd));
        const float2 Y = fma2(w1_12, hy, Xd);
        const float2 Up = fma2(w1_12, hx, Gd), Vp = fma2(w1_12, myd, Xs);
        const float2 Sdd = fma2(w4_9, R0, fma2(w1_3, mxd, Ks));
        const float2 Smx = fma2(w1_3, hx, Kd);
        const float2 nd = sub(U, V), nmx = sub(Up, Vp), nmy = sub(Y, U);
        if (r == 0) {
          mine[0].a[lane] = {nd, nmx};
          mine[0].b[lane] = {nmy, zxC};
          mine[0].zy[lane] = zyC;
          s0d = Sdd;
          s0x = Smx;
        } else {
          const float2 ex = sub(zxC, zx[r - 1]), ey = sub(zyC, zy[r - 1]);
          const float2 bd = add(td, Sdd);
          const float2 bx_ = fma2(wm1_6, ex, add(tx, Smx));
          const float2 by_ = fma2(mhalf, ey, ty);
          if (r == 1) {
            n1d = nd;
            n1x = nmx;
            n1y = nmy;
            e1x = ex;
            e1y = ey;
          } else {
            finish(r - 1, acd, acx, acy, nd, nmx, nmy, ex, ey);
          }
          acd = bd;
          acx = bx_;
          acy = by_;
        }
        td = add(U, V);
        tx = add(Up, Vp);
        ty = add(Y, U);
        if (r == kR - 1) {
          mine[1].a[lane] = {td, tx};
          mine[1].b[lane] = {ty, zxC};
          mine[1].zy[lane] = zyC;
        }
      }
      __syncthreads();
      {  // the first row, with the row below's contribution (none: solid)
        EdgeA ea = {bc(0.f), bc(0.f)};
        EdgeB eb = {bc(0.f), bc(-fx)};
        float2 ez = bc(-fy);
        if (w > 0) {
          const Edge *e = mine - 1;
          ea = e->a[lane];
          eb = e->b[lane];
          ez = e->zy[lane];
        }
        finish(0, add(ea.dd, s0d),
               fma2(w1_6, sub(eb.zx, zx[0]), add(ea.mx, s0x)),
               fma2(half, sub(ez, zy[0]), eb.my), n1d, n1x, n1y, e1x, e1y);
      }
      {  // the last row, with the row above's contribution
        EdgeA ea = {bc(0.f), bc(0.f)};
        EdgeB eb = {bc(0.f), bc(-fx)};
        float2 ez = bc(-fy);
        if (w + 1 < warps) {
          const Edge *e = mine + 2;
          ea = e->a[lane];
          eb = e->b[lane];
          ez = e->zy[lane];
        }
        finish(kR - 1, acd, acx, acy, ea.dd, ea.mx, eb.my,
               sub(eb.zx, zx[kR - 1]), sub(ez, zy[kR - 1]));
      }
    }
  };
  if (any_walls)
    march(std::true_type{});
  else
    march(std::false_type{});

  if constexpr (kReduce) {
    const bool finite = isfinite(rs_num.x) && isfinite(rs_num.y) &&
                        isfinite(rs_den.x) && isfinite(rs_den.y) &&
                        isfinite(rs_mass) && isfinite(rs_comp);
    if (__any_sync(kFull, !(rmin > 0.f) || !finite) && lane == 0)
      atomicOr(a.flag, kFlagUnstable);
    // The lanes' sums, as pairs of addends, to shared memory; one warp per sum
    // adds each lane's over the warps in two-float arithmetic (exact to about
    // 2^-46, where the lanes' FP32 sums are to 2^-24) and only then goes to
    // FP64: the FP64 pipe takes 16 cycles or more per warp instruction, and a
    // butterfly of three sums in every warp kept it busy for 2 us per region.
    // With FP64 from the lanes on, lbm_step(1) at 4096^2 takes 130 us instead
    // of 120, with three floats 123.  FP64 does serve where the floats overflow,
    // as lanes' sums within FP32's range may together.
    __syncthreads();  // the edges' buffer is free
    float2 *terms = reinterpret_cast<float2 *>(edges);
    const int n = warps * kLanes;
    terms[threadIdx.x] = rs_num;
    terms[n + threadIdx.x] = rs_den;
    terms[2 * n + threadIdx.x] = make_float2(rs_mass, -rs_comp);
    __syncthreads();
    const int region = by * g.gx + bx, last = g.gx * g.gy - 1;
    for (int k = w; k < 3; k += warps) {
      float hi = 0.f, lo = 0.f;
      for (int i = 0; i < warps; ++i) {
        const float2 v = terms[k * n + i * kLanes + lane];
#pragma unroll
        for (int e = 0; e < 2; ++e) {  // hi + lo += v, the rounding kept
          const float x = e ? v.y : v.x;
          const float s = __fadd_rn(hi, x);
          const float t = __fsub_rn(s, hi);
          lo = __fadd_rn(lo, __fadd_rn(__fsub_rn(hi, __fsub_rn(s, t)),
                                       __fsub_rn(x, t)));
          hi = s;
        }
      }
      double total = static_cast<double>(hi) + lo;
      if (!isfinite(hi)) {
        total = 0.0;
        for (int i = 0; i < warps; ++i) {
          const float2 v = terms[k * n + i * kLanes + lane];
          total += static_cast<double>(v.x) + v.y;
        }
      }
#pragma unroll
      for (int o = kLanes / 2; o > 0; o >>= 1)
        total += __shfl_xor_sync(kFull, total, o);
      if (lane == 0) {
        a.partials[3 * static_cast<int64_t>(region) + k] = total;
        // the finalize kernel takes triples by fours
        if (region == last)
          for (int i = last + 1; i % kTileWarps; ++i)
            a.partials[3 * static_cast<int64_t>(i) + k] = 0.0;
      }
    }
  }

  // the owned outputs
  if (xb < xlo || xb >= xhi) return;
  const int64_t first = static_cast<int64_t>(y0) * pitch + x0;
  T *dd = static_cast<T *>(a.dst.d) + first;
  T *dx = static_cast<T *>(a.dst.jx) + first;
  T *dy = static_cast<T *>(a.dst.jy) + first;
#pragma unroll
  for (int r = 0; r < kR; ++r) {
    const int row = yb + r;
    if (row < ylo || row >= yhi) continue;
    const int64_t o = static_cast<int64_t>(mine0 + r * step_y);
    const float2 vd[1] = {d[r]}, vx[1] = {zx[r]}, vy[1] = {zy[r]};
    store_pairs<2, T>(dd + o, vd, S::kD);
    store_pairs<2, T>(dx + o, vx, S::kJ);
    store_pairs<2, T>(dy + o, vy, S::kJ);
  }
}

template <typename T, int kR, bool kSr, bool kSC, bool kReduce, bool kForce>
__global__ void __launch_bounds__(kResMaxWarps *kLanes, 1)
    lbm_resident_kernel(const StepLaunch a, const ResidentTiles g, int nsteps) {
  extern __shared__ __align__(128) unsigned char smem[];
  resident_region<T, kR, kSr, kSC, kReduce, kForce>(
      a, g, blockIdx.x, blockIdx.y, nsteps, smem);
}

// A batch's regions: one block per region of the work list.  The launch state
// stays in shared memory, read where the region needs it.
template <typename T, int kR, bool kSr>
__global__ void __launch_bounds__(kResMaxWarps *kLanes, 1)
    lbm_resident_batch_kernel(const ResidentBatch b, int nsteps) {
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ __align__(16) unsigned char raw_a[sizeof(StepLaunch)];
  __shared__ __align__(16) unsigned char raw_g[sizeof(ResidentTiles)];
  StepLaunch &a = *reinterpret_cast<StepLaunch *>(raw_a);
  ResidentTiles &g = *reinterpret_cast<ResidentTiles *>(raw_g);
  const int4 item = b.items[blockIdx.x];  // member, region x, region y
  if (threadIdx.x == 0) {
    const BatchMember &m = b.members[item.x];
    // (read before the launches before this one have ended: none of them
    // changes the clock, and the call's first launch follows a copy)
    const unsigned clock = *b.clock + b.taken;
    fill_launch(a, m, (m.cur ^ b.parity) & 1, b.storage, clock);
    g = m.tiles;
    // The clock for the step that follows the region launches, set by the last
    // block to have read it (the launches before this one have: their blocks
    // read it before they let this one start).  At the end of the block a fence
    // and this took 3 % of a launch.
    if (b.advance && atomicAdd(b.done, 1u) == gridDim.x - 1) {
      *b.done = 0u;
      *b.clock = clock + nsteps;
    }
  }
  __syncthreads();
  resident_region<T, kR, kSr, false, false, true>(a, g, item.y, item.z, nsteps,
                                                  smem);
}

// Launches a region kernel; `early`: it may start while the launch before it
// ends (its node types are settled).
template <auto kKern, typename... A>
cudaError_t launch_regions(dim3 grid, int warps, int smem, int most_smem,
                           bool early, cudaStream_t s, const A &...args) {
  static cudaError_t attr = cudaFuncSetAttribute(
      kKern, cudaFuncAttributeMaxDynamicSharedMemorySize, most_smem);
  if (attr != cudaSuccess) return attr;
  (void)cudaGetLastError();
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(warps * kLanes);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = early ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kKern, args...);
}

template <typename T, int kR, bool kSr, bool kSC, bool kReduce>
cudaError_t launch_resident_k(const StepLaunch &a, const ResidentTiles &g,
                              int nsteps, cudaStream_t s) {
  // Without a body force its sums are left out (us a step: cavity 1024^2 5.5 ->
  // 5.3, FP16 4096x2500 50.5 -> 48.7, drop 2048^2 22.3 -> 21.6).
  auto go = [&](auto force) {
    // (a reduced step, one per call, has the one kernel)
    return launch_regions<lbm_resident_kernel<
        T, kR, kSr, kSC, kReduce, decltype(force)::value || kReduce>>(
        dim3(g.gx, g.gy), g.warps, resident_smem<kR, kSC>(g.warps),
        resident_smem<kR, kSC>(kResMaxWarps), a.mask_settled, s, a, g, nsteps);
  };
  return a.fx != 0.f || a.fy != 0.f ? go(std::true_type{})
                                    : go(std::false_type{});
}

template <typename T, int kR, bool kSr>
cudaError_t launch_resident_batch_k(const ResidentBatch &b, int nsteps,
                                    cudaStream_t s) {
  return launch_regions<lbm_resident_batch_kernel<T, kR, kSr>>(
      dim3(static_cast<unsigned>(b.nitems)), b.warps,
      resident_smem<kR, false>(b.warps),
      resident_smem<kR, false>(kResMaxWarps), true, s, b, nsteps);
}

// f(rows per warp, stochastic rounding) as compile-time constants
template <typename F>
cudaError_t with_rows(int rows, bool sr, F &&f) {
  auto go = [&](auto r) {
    return sr ? f(r, std::true_type{}) : f(r, std::false_type{});
  };
  switch (rows) {
    case 2: return go(std::integral_constant<int, 2>{});
    case 4: return go(std::integral_constant<int, 4>{});
    default: return go(std::integral_constant<int, 8>{});
  }
}

template <typename T>
cudaError_t launch_resident_t(const StepLaunch &a, const ResidentTiles &g,
                              int nsteps, bool reduce, cudaStream_t s) {
  if (a.g_sc != 0.0f) {
    if constexpr (std::is_same<T, float>::value)
      if (!reduce)
        return with_rows(g.rows, false, [&](auto r, auto) {
          return launch_resident_k<T, decltype(r)::value, false, true, false>(
              a, g, nsteps, s);
        });
    return cudaErrorInvalidValue;
  }
  if (reduce && nsteps != 1) return cudaErrorInvalidValue;
  return with_rows(g.rows, a.sr != 0, [&](auto r, auto sr) {
    constexpr int kR = decltype(r)::value;
    constexpr bool kSr = decltype(sr)::value;
    return reduce
               ? launch_resident_k<T, kR, kSr, false, true>(a, g, 1, s)
               : launch_resident_k<T, kR, kSr, false, false>(a, g, nsteps, s);
  });
}

template <typename T>
cudaError_t launch_resident_batch_t(const ResidentBatch &b, int nsteps,
                                    cudaStream_t s) {
  return with_rows(b.rows, b.sr != 0, [&](auto r, auto sr) {
    return launch_resident_batch_k<T, decltype(r)::value,
                                   decltype(sr)::value>(b, nsteps, s);
  });
}

// The launchers of storage type T, as the table lbm_step.cu dispatches on.
template <typename T>
constexpr StorageOps make_ops() {
  return StorageOps{&launch_step_t<T>, &launch_batch_t<T>, &choose_variant_t<T>,
                    &launch_resident_t<T>, &launch_resident_batch_t<T>,
                    &pack_t<T>,        &unpack_t<T>,       &solid_t<T>,
                    &change_t<T>};
}

}  // namespace
}  // namespace lbmtau1
