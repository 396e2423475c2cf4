// hs_quad.cuh -- the FP32 tile engine with four nodes per lane (3-D grids whose
// x-lines are whole 16-byte quads, n_x a multiple of 4).
//
// The FP32 passes move 32 to 56 bytes per node and are not FP64-bound, so
// what holds them back is instruction issue and the number of bytes in flight
// (the one-node engine: 150 instructions per node and CG iteration on stored
// coefficients, 62 % of the issue slots, 3.4 TB/s).  Here a lane owns four
// consecutive nodes: every vector is copied in 16-byte pieces by cp.async
// into a ring of QNS steps in shared memory, zero-filled outside the grid,
// and address and control instructions are shared by four nodes.  A block of
// 256 lanes covers 64 x 16 nodes of a plane and marches along z as
// zmarch_item does: the plane's source values sit in a double-buffered slab
// for the x and y neighbours, the planes below and above in registers, one
// block barrier per plane.
//
// Stored face couplings are read once: the upper x face is the next node's
// lower one in the staged row (one more scalar per row), the upper y face the
// staged row above (one more row), the upper z face the next plane's.
// Staged data of a step are read by other lanes, so each step ends by waiting
// for the next step's group in front of the barrier.
//
// Measured at 256^3: FP32 CG on stored coefficients 213 -> 171 us per
// iteration (140 us of traffic), FP32 Jacobi 63 -> 38 us per sweep (30 us).
// Three steps in the ring: two give Jacobi 48, four give CG 183 (one block per
// SM).
#pragma once
#include "hs_stencil.cuh"

namespace hs {

constexpr int QLR = 16, QR = 256 / QLR, QTW = 4 * QLR;   // lanes per row, rows, tile width
constexpr int QNS = 3;                                    // steps in the ring
constexpr int QSW = QTW + 8;                              // slab row: data from element 4

template <class Src, class Sink>
__host__ __device__ constexpr int quad_stage() {
  return Src::NA * (1024 + 8 * QLR + 2 * QR) + Sink::NQ * 1024 +
         (Sink::kOp == OP_VARK ? 2 * 1024 + QR * (QTW + 4) + (QR + 1) * QTW : 0);
}
template <class Src, class Sink>
__host__ __device__ constexpr size_t quad_bytes() {
  return 4 * (size_t)(2 * (QR + 2) * QSW + QNS * quad_stage<Src, Sink>());
}

__device__ __forceinline__ void cp_async16(unsigned dst, const float* src, unsigned bytes) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void cp_async4(unsigned dst, const float* src, unsigned bytes) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}

template <class Src, class Sink>
__device__ __forceinline__ void zmarch_quad(const Geom& g, const Tiling& tl, int item, float* sm, const Src& src,
                                            Sink& sink) {
  constexpr int NA = Src::NA, NQ = Sink::NQ;
  constexpr bool VK = Sink::kOp == OP_VARK;
  constexpr int STG = quad_stage<Src, Sink>();
  // offsets inside a stage (floats)
  constexpr int OH = NA * 1024, OS = OH + NA * 8 * QLR, OQ = OS + NA * 2 * QR, OD = OQ + NQ * 1024, OZ = OD + 1024,
                OX = OZ + 1024, OY = OX + QR * (QTW + 4);
  int i0, j0, z0, z1;
  decode_item(tl, g, item, i0, j0, z0, z1);
  const int tid = threadIdx.x;
  const int qx = tid % QLR, row = tid / QLR;
  const int i = i0 + 4 * qx, j = j0 + row;
  const bool inside = i < g.nx && j < g.ny;
  const unsigned P = (unsigned)g.plane, nx = (unsigned)g.nx;
  // halo producers: lanes 0 .. 2 QLR - 1 a quad of the row below / above the
  // tile, lanes 64 .. 64 + 2 QR - 1 a node of the side columns
  const bool hq = tid < 2 * QLR, side = tid >= 64 && tid < 64 + 2 * QR;
  int hi = 0, hj = -1, hslab = 0;
  if (hq) {
    hi = i0 + 4 * (tid % QLR);
    hj = tid < QLR ? j0 - 1 : j0 + QR;
    hslab = (tid < QLR ? 0 : QR + 1) * QSW + 4 + 4 * (tid % QLR);
  } else if (side) {
    const int s = tid - 64;
    hi = s < QR ? i0 - 1 : i0 + QTW;
    hj = j0 + s % QR;
    hslab = (s % QR + 1) * QSW + (s < QR ? 3 : 4 + QTW);
  }
  const bool hin = hi >= 0 && hi < g.nx && hj >= 0 && hj < g.ny;
  const unsigned oc = inside ? (unsigned)j * nx + (unsigned)i : 0u;
  const unsigned hcol = hin ? (unsigned)hj * nx + (unsigned)hi : 0u;
  const unsigned in16 = inside ? 16u : 0u;
  // the extra face operands: the row above the tile (ay), the node right of it (ax)
  const bool ey = VK && tid < QLR && i < g.nx && j0 + QR < g.ny;
  const bool ex = VK && qx == QLR - 1 && i + 4 < g.nx && j < g.ny;
  const unsigned eyo = ey ? (unsigned)(j0 + QR) * nx + (unsigned)i : 0u;

  float* const ring = sm + 2 * (QR + 2) * QSW;
  const unsigned ring_s = (unsigned)__cvta_generic_to_shared(ring);
  auto issue = [&](int k) {
    const unsigned at = ring_s + 4u * (unsigned)(((k - z0) % QNS) * STG);
    const unsigned up = (unsigned)min(k + 1, g.nz - 1) * P;
    const bool a_up = k + 1 <= z1 && k + 1 < g.nz;
    const unsigned sz = a_up ? in16 : 0u;
#pragma unroll
    for (int a = 0; a < NA; a++)
      if (HS_IN_BOUNDS(oc + up + 3, g.N)) cp_async16(at + 4u * (a * 1024 + 4 * tid), src.arr(a) + (oc + up), sz);
    if (hq) {
      const unsigned hsz = hin && k + 1 < z1 ? 16u : 0u;
#pragma unroll
      for (int a = 0; a < NA; a++)
        if (HS_IN_BOUNDS(hcol + up + 3, g.N))
          cp_async16(at + 4u * (OH + a * 8 * QLR + 4 * tid), src.arr(a) + (hcol + up), hsz);
    } else if (side) {
      const unsigned hsz = hin && k + 1 < z1 ? 4u : 0u;
#pragma unroll
      for (int a = 0; a < NA; a++)
        if (HS_IN_BOUNDS(hcol + up, g.N))
          cp_async4(at + 4u * (OS + a * 2 * QR + tid - 64), src.arr(a) + (hcol + up), hsz);
    }
    const unsigned here = (unsigned)min(k, g.nz - 1) * P;
    const unsigned ksz = k < z1 ? in16 : 0u;
#pragma unroll
    for (int b = 0; b < NQ; b++)
      if (HS_IN_BOUNDS(oc + here + 3, g.N)) cp_async16(at + 4u * (OQ + b * 1024 + 4 * tid), sink.opnd(b) + (oc + here), ksz);
    if constexpr (VK) {
      if (HS_IN_BOUNDS(oc + here + 3, g.N)) {
        cp_async16(at + 4u * (OD + 4 * tid), sink.cf.D + (oc + here), ksz);
        cp_async16(at + 4u * (OX + row * (QTW + 4) + 4 * qx), sink.cf.ax + (oc + here), ksz);
        cp_async16(at + 4u * (OY + row * QTW + 4 * qx), sink.cf.ay + (oc + here), ksz);
      }
      if (HS_IN_BOUNDS(oc + up + 3, g.N)) cp_async16(at + 4u * (OZ + 4 * tid), sink.cf.az + (oc + up), sz);
      if (qx == QLR - 1 && HS_IN_BOUNDS((ex ? oc + 4 : 0u) + here, g.N))
        cp_async4(at + 4u * (OX + row * (QTW + 4) + QTW), sink.cf.ax + ((ex ? oc + 4 : 0u) + here),
                  ex && k < z1 ? 4u : 0u);
      if (tid < QLR && HS_IN_BOUNDS(eyo + here + 3, g.N))
        cp_async16(at + 4u * (OY + QR * QTW + 4 * tid), sink.cf.ay + (eyo + here), ey && k < z1 ? 16u : 0u);
    }
    cp_async_commit();
  };
  auto make4 = [&](const float4 (&q)[NA]) -> float4 {
    float v[4];
#pragma unroll
    for (int c = 0; c < 4; c++) {
      float w[NA];
#pragma unroll
      for (int a = 0; a < NA; a++) w[a] = c == 0 ? q[a].x : c == 1 ? q[a].y : c == 2 ? q[a].z : q[a].w;
      v[c] = src.make(src.pack(w), 0, false);
    }
    return make_float4(v[0], v[1], v[2], v[3]);
  };
  auto quad = [&](const float* p) -> float4 { return *reinterpret_cast<const float4*>(p); };

#pragma unroll
  for (int n = 0; n < QNS - 1; n++) issue(z0 + n);
  const float4 zero4 = make_float4(0.f, 0.f, 0.f, 0.f);
  float4 vb = zero4, vc = zero4, zl = zero4;
  unsigned o = oc + (unsigned)z0 * P;
  const int slab0 = (row + 1) * QSW + 4 + 4 * qx;
  if (inside && HS_IN_BOUNDS(o + 3, g.N)) {
    float4 rc[NA], rb[NA];
    const bool low = z0 > 0;
#pragma unroll
    for (int a = 0; a < NA; a++) {
      rc[a] = __ldcg(reinterpret_cast<const float4*>(src.arr(a) + o));
      rb[a] = low ? __ldcg(reinterpret_cast<const float4*>(src.arr(a) + (o - P))) : zero4;
    }
    if constexpr (VK) zl = __ldcg(reinterpret_cast<const float4*>(sink.cf.az + o));
    vc = make4(rc);
    src.put4(o, vc);
    if (low) vb = make4(rb);
  }
  *reinterpret_cast<float4*>(sm + slab0) = vc;
  if (hq) {
    float4 h = zero4;
    if (hin) {
      float4 rh[NA];
#pragma unroll
      for (int a = 0; a < NA; a++)
        rh[a] = __ldcg(reinterpret_cast<const float4*>(src.arr(a) + (hcol + (unsigned)z0 * P)));
      h = make4(rh);
    }
    *reinterpret_cast<float4*>(sm + hslab) = h;
  } else if (side) {
    float h = 0.f;
    if (hin) {
      float rh[NA];
#pragma unroll
      for (int a = 0; a < NA; a++) rh[a] = __ldcg(src.arr(a) + (hcol + (unsigned)z0 * P));
      h = src.make(src.pack(rh), 0, false);
    }
    sm[hslab] = h;
  }
  cp_async_wait<QNS - 2>();
  __syncthreads();

#pragma unroll 1
  for (int k = z0; k < z1; k++) {
    issue(k + QNS - 1);
    const float* const st = ring + ((k - z0) % QNS) * STG;
    const int cur = ((k - z0) & 1) * (QR + 2) * QSW, next = (QR + 2) * QSW - cur;
    // plane k + 1: source values, slab
    float4 rt[NA];
#pragma unroll
    for (int a = 0; a < NA; a++) rt[a] = quad(st + a * 1024 + 4 * tid);
    const float4 vt = make4(rt);
    if (k + 1 < z1 && inside) src.put4(o + P, vt);
    *reinterpret_cast<float4*>(sm + next + slab0) = vt;
    if (hq) {
      float4 rh[NA];
#pragma unroll
      for (int a = 0; a < NA; a++) rh[a] = quad(st + OH + a * 8 * QLR + 4 * tid);
      *reinterpret_cast<float4*>(sm + next + hslab) = make4(rh);
    } else if (side) {
      float rh[NA];
#pragma unroll
      for (int a = 0; a < NA; a++) rh[a] = st[OS + a * 2 * QR + tid - 64];
      sm[next + hslab] = src.make(src.pack(rh), 0, false);
    }
    // plane k
    float4 zu = zero4;
    if constexpr (VK) zu = quad(st + OZ + 4 * tid);
    if (inside) {
      const float* const c0 = sm + cur + slab0;
      const float4 s4 = quad(c0 - QSW), n4 = quad(c0 + QSW);
      const float cc[6] = {c0[-1], vc.x, vc.y, vc.z, vc.w, c0[4]};
      const float ss[4] = {s4.x, s4.y, s4.z, s4.w}, nn[4] = {n4.x, n4.y, n4.z, n4.w};
      const float bb[4] = {vb.x, vb.y, vb.z, vb.w}, tt[4] = {vt.x, vt.y, vt.z, vt.w};
      float dd[4] = {}, xx[5] = {}, yy[4] = {}, yu[4] = {}, ex4[NQ > 0 ? NQ : 1][4] = {};
      const float zz[4] = {zl.x, zl.y, zl.z, zl.w}, zv[4] = {zu.x, zu.y, zu.z, zu.w};
      if constexpr (VK) {
        const float4 d4 = quad(st + OD + 4 * tid), x4 = quad(st + OX + row * (QTW + 4) + 4 * qx),
                     y4 = quad(st + OY + row * QTW + 4 * qx), u4 = quad(st + OY + (row + 1) * QTW + 4 * qx);
        dd[0] = d4.x; dd[1] = d4.y; dd[2] = d4.z; dd[3] = d4.w;
        xx[0] = x4.x; xx[1] = x4.y; xx[2] = x4.z; xx[3] = x4.w;
        xx[4] = st[OX + row * (QTW + 4) + 4 * qx + 4];
        yy[0] = y4.x; yy[1] = y4.y; yy[2] = y4.z; yy[3] = y4.w;
        yu[0] = u4.x; yu[1] = u4.y; yu[2] = u4.z; yu[3] = u4.w;
      }
#pragma unroll
      for (int b = 0; b < NQ; b++) {
        const float4 e4 = quad(st + OQ + b * 1024 + 4 * tid);
        ex4[b][0] = e4.x; ex4[b][1] = e4.y; ex4[b][2] = e4.z; ex4[b][3] = e4.w;
      }
      float out[4];
#pragma unroll
      for (int c = 0; c < 4; c++) {
        Nbr<float> nb;
        nb.c = cc[c + 1];
        nb.w = cc[c];
        nb.e = cc[c + 2];
        nb.s = ss[c];
        nb.n = nn[c];
        nb.b = bb[c];
        nb.t = tt[c];
        nb.box = 0.f;
        OpRaw<float, Sink::kOp> q{};
        if constexpr (VK) {
          q.d = dd[c];
          q.xl = xx[c];
          q.xu = xx[c + 1];
          q.yl = yy[c];
          q.yu = yu[c];
          q.zl = zz[c];
          q.zu = zv[c];
        }
        out[c] = sink.value(nb, q, ex4[0][c]);
      }
      if (HS_IN_BOUNDS(o + 3, g.N))
        *reinterpret_cast<float4*>(sink.out() + o) = make_float4(out[0], out[1], out[2], out[3]);
    }
    o += P;
    vb = vc;
    vc = vt;
    zl = zu;
    cp_async_wait<QNS - 2>();
    __syncthreads();
  }
  cp_async_wait<0>();
  __syncthreads();   // the next item refills the ring
}

}  // namespace hs
