// Warp-packet traversal of the transfer rays (Sec. 4.4-4.5).
//
// Every receiver traces the same S world-space directions, so the rays that 32 receivers
// adjacent in Morton order cast along one direction are parallel and start from a small patch
// of the scene. One warp takes such a packet: the lanes walk the LBVH together, testing up to
// 32 nodes per step against the packet's beam (the rectangle the packet's origins span in the
// plane orthogonal to the direction, and the depth range along it that the lanes still need),
// and collect the leaves the beam meets in a shared-memory chunk. The leaves of a chunk are staged 32
// at a time, those whose own ellipse misses the beam are dropped, every lane takes a cheap conservative
// test of the rest, and only what passes it is tested exactly; every hit decision, product and
// index-matrix rule is that of a single ray, only the traversal is shared.
//
// What bounds it: issue slots and the latency of the node steps (about 40 % of the time), with L2 serving
// the tree; a walk of surface-100k meets 1,300 nodes and 820 boxes of leaves, of which 560 leaves are
// tested and 270 are hit by one of the 30 rays (9 of them each). Measured against testing every leaf
// exactly, in step: surface-100k with bounces 77.4 -> 60.2 ms, a 60k volume 30.2 -> 24.1 ms, six tilings of a
// million splats with bounces and glossy matrices 0.973-1.041 -> 0.840-0.956 s. Tried and left out: the tree
// projected once per direction (surface-100k 62.8 -> 62.8 ms before the search had its own kernel, but the
// million splats 1.17 s: a direction's tree no longer fits the L2, and a launch per few directions ends with
// a millisecond of few busy warps).
//
//  k_packet<B>    visibility V_is of every (receiver, direction) of a receiver batch into
//                 V[s][i] (Eq. 4 along a ray, Eq. 27 read as the Gaussian's maximum); with B
//                 (bounce) also the horizon, the nearest front-facing hit and, where that settles
//                 it, the index matrix of Sec. 4.4.
//  k_search       the rest of the index matrix: rounds over the hits in key order until the argmax
//                 of W_j (Eq. 26) is settled.
//  k_project      P_i = sum_s (4 pi / S) V_is max(0, n_i.w_s) Y(w_s) (Eq. 29 with Eq. 9),
//                 one lane per receiver, compensated sums; also copies V of glossy receivers.
#include "trace.cuh"

namespace prtgs {

constexpr int kPacketWarps = 4;
constexpr int kPacketThreads = 32 * kPacketWarps;
constexpr int kPStack = 384;     // node stack of a warp (ints)
#ifndef PRTGS_PACKET_ROUND_HITS
// k_search at 4 blocks per SM: surface-100k transfer 60.3 ms at 14 hits, 58.1 at 18, 57.3 at 20, 61.2 at 24
#define PRTGS_PACKET_ROUND_HITS 20
#endif
constexpr int kPacketRoundHits = PRTGS_PACKET_ROUND_HITS;  // hits per index-matrix search round
#ifndef PRTGS_PACKET_LEAVES
#define PRTGS_PACKET_LEAVES 224
#endif
#ifndef PRTGS_PACKET_MIN_BLOCKS
#define PRTGS_PACKET_MIN_BLOCKS 5  // visibility only: a 60k volume at 128 directions 24.6 ms at 4, 24.1 at 5, 24.7 at 6
#endif
// leaf chunk of a warp (> 64: a step appends up to 64 leaves; flushed past kPLeaves - 64). Longer
// chunks flush less often: 1M bounce transfer 1.085 s at 96, 0.988 s at 128, 0.957 s at 224 (as measured
// when the index search still ran in the same kernel; now surface-100k 57.8 ms at 160, 57.3 at 224).
// The chunk also sets when the beam shrinks, and with it the order in which hits are met.
constexpr int kPLeaves = PRTGS_PACKET_LEAVES;
// wide pops (32 nodes) only while the stack keeps room for their pushes plus a full one-node-
// at-a-time descent of the deepest possible tree (64 levels)
constexpr int kPHeadroom = 64 + 64 + 4;
// directions per work item by default: one, so that the warps running at a time work on few
// windows and share the BVH nodes around them in L1/L2 (surface-100k visibility 47 ms against 72
// at 16 directions; the 1M tiled transfer 1.69 s against 1.97 s)
constexpr int kPacketDirs = 1;
// Receivers of a backward window (64 to 256): the wider, the fewer packets are left with a few lanes (isotropic
// normals: half of a window faces a direction). 100k volume at 128 directions: 83.5 ms at 64, 78.7 at 128, 76.4 at 256.
// The forward keeps 64: its hit decisions depend on a packet's reference point to the last bit.
constexpr int kBwdWindow = 256;

struct PacketSmem {
  int stack[kPStack];
  int lpos[kPLeaves];      // the chunk's leaves (sorted positions)
  float4 stage[4][32];     // a group of leaves, staged: the exact-test terms of stage_leaf, term-major (the
                           // lanes of a drain read different leaves: 16-byte stride, few bank conflicts)
  float4 quick[2][32];     // ... and the terms of the quick test
  // the window slots of the receivers that face the direction
  unsigned char rlist[kBwdWindow];
};

// k_search, per warp after the PacketSmem array: the search round's nearest hits of each lane,
// t*, position, and alpha with the sign bit set for a front-facing hit (m > 0; m itself is formed
// again from the record by the few hits that need it: 12 bytes a hit leave room for 20 of them).
struct RoundHits {
  float t[kPacketRoundHits][32];
  int pos[kPacketRoundHits][32];
  float sal[kPacketRoundHits][32];
};

// Orthonormal frame (e1, e2, w) around a unit direction w (Duff et al. 2017, "Building an
// orthonormal basis, revisited": the branchless form).
struct Frame {
  float e1x, e1y, e1z, e2x, e2y, e2z, wx, wy, wz;
};

__device__ __forceinline__ Frame make_frame(float x, float y, float z) {
  const float sgn = copysignf(1.0f, z);
  const float a = -1.0f / (sgn + z);
  const float b = x * y * a;
  Frame f;
  f.e1x = 1.0f + sgn * x * x * a;
  f.e1y = sgn * b;
  f.e1z = -sgn * x;
  f.e2x = b;
  f.e2y = sgn + y * y * a;
  f.e2z = -y;
  f.wx = x;
  f.wy = y;
  f.wz = z;
  return f;
}

// The packet's beam: the projected origins' rectangle and the depth range along w that the
// lanes still need.
struct Beam {
  float xlo, xhi, ylo, yhi, zlo, zhi;
};

// Over the full warp, one instruction each (NaN inputs are ignored).
__device__ __forceinline__ float warp_min(float v) {
  float r;
  asm volatile("redux.sync.min.f32 %0, %1, 0xffffffff;" : "=f"(r) : "f"(v));
  return r;
}
__device__ __forceinline__ float warp_max(float v) {
  float r;
  asm volatile("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(r) : "f"(v));
  return r;
}

__device__ __forceinline__ Beam make_beam(bool need, float xl, float yl, float zlo, float zhi) {
  Beam b;
  b.xlo = warp_min(need ? xl : FLT_MAX);
  b.xhi = warp_max(need ? xl : -FLT_MAX);
  b.ylo = warp_min(need ? yl : FLT_MAX);
  b.yhi = warp_max(need ? yl : -FLT_MAX);
  b.zlo = warp_min(need ? zlo : FLT_MAX);
  b.zhi = warp_max(need ? zhi : -FLT_MAX);
  return b;
}

// The exact ray / Gaussian test of a packet. Every ray of the packet has the direction w, so the
// whitened closest-approach distance depends only on the ray origin's offset from the Gaussian in
// the plane (e1, e2): with u = o - mu = dx e1 + dy e2 + uz w and the rows of A = diag(1/s) R^T,
//   D^2 = |A u x A w|^2 / |A w|^2 = |dx (A e1 x a) + dy (A e2 x a)|^2,  a = A w / |A w|,
//   t*  = -(u^T A^T A w) / |A w|^2 = -uz - dx m1 - dy m2,  m_k = (A e_k . A w) / |A w|^2
// (the component of u along w drops out exactly). The per-Gaussian terms are formed once per
// staged leaf; a lane then needs two additions, six FMAs for the vector and three for its norm.
// Offsets are taken against a reference point R of the packet (one of its ray origins). A leaf's
// R - mu is moved along w to p, the reference ray's point nearest to the Gaussian (D^2 does not
// change along w; the move keeps the frame's own rounding, w.e1 of a few ulp, from mixing the
// distance along w into dx and dy), and p and the lane's o - R are projected on e1, e2 in twice the
// working precision (exact products and sums, hi + lo), so dx = (o - R).e1 + p.e1 carries about one
// rounding of itself: the role that the error-free o - mu and the refinement at the closest point
// play in the per-ray test.
struct Rel {
  float Rx, Ry, Rz;        // reference point (warp-uniform)
  float Rxl, Ryl, Rzl;     // ... and its place on the frame
  float xr, xr_lo, yr, yr_lo;  // this lane's origin minus R on e1, e2, each as an unevaluated sum hi + lo
  float zr;                // ... and on w
};

// a . b of three terms as an unevaluated sum hi + lo (error-free products by FMA, error-free sums
// by TwoSum, their errors gathered in lo): twice the working precision.
__device__ __forceinline__ void dot3_pair(float ax, float ay, float az, float bx, float by, float bz, float& hi,
                                          float& lo) {
  const float p = ax * bx, ep = fmaf(ax, bx, -p);
  const float q = ay * by, eq = fmaf(ay, by, -q);
  const float r = az * bz, er = fmaf(az, bz, -r);
  float s, t, s2, t2;
  two_sum(p, q, s, t);
  two_sum(s, r, s2, t2);
  hi = s2;
  lo = ((ep + eq) + er) + (t + t2);
}

// The lane's offset o - R from the reference point R on the frame, e1 and e2 parts as hi + lo.
// The frame is orthonormal only to a few ulp: its e1.w and e2.w (taken in twice the working
// precision) times the offset along w are taken off, so that dx e1 + dy e2 is the part of o - R
// across w (up to a multiple of w, which D^2 does not see) and not a few ulp of the packet's depth
// off it, which 1/s_min of a thin Gaussian would magnify.
__device__ __forceinline__ Rel make_rel(const Frame& f, float ox0, float oy0, float oz0, float Rx, float Ry,
                                        float Rz) {
  Rel rel;
  rel.Rx = Rx;
  rel.Ry = Ry;
  rel.Rz = Rz;
  rel.Rxl = fmaf(f.e1x, Rx, fmaf(f.e1y, Ry, f.e1z * Rz));
  rel.Ryl = fmaf(f.e2x, Rx, fmaf(f.e2y, Ry, f.e2z * Rz));
  rel.Rzl = fmaf(f.wx, Rx, fmaf(f.wy, Ry, f.wz * Rz));
  float ox, oy, oz, lox, loy, loz;
  two_sum(ox0, -Rx, ox, lox);
  two_sum(oy0, -Ry, oy, loy);
  two_sum(oz0, -Rz, oz, loz);
  dot3_pair(f.e1x, f.e1y, f.e1z, ox, oy, oz, rel.xr, rel.xr_lo);
  dot3_pair(f.e2x, f.e2y, f.e2z, ox, oy, oz, rel.yr, rel.yr_lo);
  rel.zr = fmaf(f.wx, ox, fmaf(f.wy, oy, f.wz * oz)) + fmaf(f.wx, lox, fmaf(f.wy, loy, f.wz * loz));
  float d1, d1l, d2, d2l;
  dot3_pair(f.e1x, f.e1y, f.e1z, f.wx, f.wy, f.wz, d1, d1l);
  dot3_pair(f.e2x, f.e2y, f.e2z, f.wx, f.wy, f.wz, d2, d2l);
  rel.xr_lo += fmaf(f.e1x, lox, fmaf(f.e1y, loy, f.e1z * loz)) - rel.zr * (d1 + d1l);
  rel.yr_lo += fmaf(f.e2x, lox, fmaf(f.e2y, loy, f.e2z * loz)) - rel.zr * (d2 + d2l);
  return rel;
}

__device__ __forceinline__ float facing(const Frame& f, const float4& q3) {
  return fmaxf(-fmaf(f.wx, q3.y, fmaf(f.wy, q3.z, f.wz * q3.w)), 0.0f);
}

// Stage 32 leaves for the packet, one per lane (pos < 0: none), and return how many were kept: a leaf
// whose own 3-sigma ellipse misses the beam is dropped (of the leaves whose box meets it, two in five).
// Per leaf: (p on e1, e2 (high parts), R - mu on w; opacity), (A e1 x a; m1), (A e2 x a; m2), (facing term
// max(-w.n_j, 0); sorted position; p on e1, e2 (low parts)), and the quick test's terms (quick_mask), for
// which X, Y bound the lanes' |xr|, |yr|. et: the largest error bound of the quick t.
__device__ __forceinline__ int stage_leaves(const float4* __restrict__ recs, int pos, const Frame& f, const Rel& rel,
                                            const Beam& bm, float X, float Y, PacketSmem& sm, float& et) {
  const float4* rec = recs + 4 * (int64_t)max(pos, 0);
  const float4 q0 = __ldg(rec), q1 = __ldg(rec + 1), q2 = __ldg(rec + 2), q3 = __ldg(rec + 3);
  // R - mu = h + l exactly; p = R - mu + t_ref w, the offset of mu from the point of the reference
  // ray nearest to it, formed with one rounding per component (the product t_ref w is exact inside
  // the FMA): D^2 does not change along w, so the lanes use p in place of R - mu, and its projections
  // on e1, e2 are small numbers, unaffected by the frame's own rounding (w.e1 of a few ulp times the
  // distance to the Gaussian); uz keeps the distance along w as w.p - t_ref.
  float hx, lx, hy, ly, hz, lz;
  two_sum(rel.Rx, -q0.x, hx, lx);
  two_sum(rel.Ry, -q0.y, hy, ly);
  two_sum(rel.Rz, -q0.z, hz, lz);
  const float t_ref = -fmaf(f.wx, hx, fmaf(f.wy, hy, f.wz * hz));
  // p = h + l + t_ref w per component as hi + lo: the product exactly (FMA), the sum by TwoSum
  float px, pxl, py, pyl, pz, pzl;
  {
    const float ax = t_ref * f.wx, ay = t_ref * f.wy, az = t_ref * f.wz;
    const float eax = fmaf(t_ref, f.wx, -ax), eay = fmaf(t_ref, f.wy, -ay), eaz = fmaf(t_ref, f.wz, -az);
    float e;
    two_sum(hx, ax, px, e);
    pxl = e + eax + lx;
    two_sum(hy, ay, py, e);
    pyl = e + eay + ly;
    two_sum(hz, az, pz, e);
    pzl = e + eaz + lz;
  }
  float cx, cxl, cy, cyl;
  dot3_pair(f.e1x, f.e1y, f.e1z, px, py, pz, cx, cxl);
  dot3_pair(f.e2x, f.e2y, f.e2z, px, py, pz, cy, cyl);
  cxl += fmaf(f.e1x, pxl, fmaf(f.e1y, pyl, f.e1z * pzl));
  cyl += fmaf(f.e2x, pxl, fmaf(f.e2y, pyl, f.e2z * pzl));
  const float cz = fmaf(f.wx, hx, fmaf(f.wy, hy, f.wz * hz)) + fmaf(f.wx, lx, fmaf(f.wy, ly, f.wz * lz));
  // rows of A: (q1.x q1.y q1.z), (q1.w q2.x q2.y), (q2.z q2.w q3.x)
  const float b1x = fmaf(q1.x, f.e1x, fmaf(q1.y, f.e1y, q1.z * f.e1z));
  const float b1y = fmaf(q1.w, f.e1x, fmaf(q2.x, f.e1y, q2.y * f.e1z));
  const float b1z = fmaf(q2.z, f.e1x, fmaf(q2.w, f.e1y, q3.x * f.e1z));
  const float b2x = fmaf(q1.x, f.e2x, fmaf(q1.y, f.e2y, q1.z * f.e2z));
  const float b2y = fmaf(q1.w, f.e2x, fmaf(q2.x, f.e2y, q2.y * f.e2z));
  const float b2z = fmaf(q2.z, f.e2x, fmaf(q2.w, f.e2y, q3.x * f.e2z));
  const float adx = fmaf(q1.x, f.wx, fmaf(q1.y, f.wy, q1.z * f.wz));
  const float ady = fmaf(q1.w, f.wx, fmaf(q2.x, f.wy, q2.y * f.wz));
  const float adz = fmaf(q2.z, f.wx, fmaf(q2.w, f.wy, q3.x * f.wz));
  const float dd = fmaf(adx, adx, fmaf(ady, ady, adz * adz));
  const float id = 1.0f / sqrtf(dd);
  const float ax = adx * id, ay = ady * id, az = adz * id;
  const float idd = 1.0f / dd;
  const float4 s1 = make_float4(diff_prod(b1y, az, b1z, ay), diff_prod(b1z, ax, b1x, az), diff_prod(b1x, ay, b1y, ax),
                                fmaf(b1x, adx, fmaf(b1y, ady, b1z * adz)) * idd);
  const float4 s2 = make_float4(diff_prod(b2y, az, b2z, ay), diff_prod(b2z, ax, b2x, az), diff_prod(b2x, ay, b2y, ax),
                                fmaf(b2x, adx, fmaf(b2y, ady, b2z * adz)) * idd);
  // quick test: D^2 = |dx B1 + dy B2|^2 = u^2 + v^2, u = l11 dx + l21 dy, v = l22 dy (Cholesky of the
  // Gram matrix of B1, B2; both are orthogonal to a, so l22 |B1| = |(B1 x B2) . a|). Every coefficient
  // is off by a few ulp of |B1| or |B2|, so u and v are off by at most e below; a leaf that meets
  // D^2 <= 9 then has u^2 + v^2 <= 9 + 12 e + 2 e^2. All are scaled so that this bound is 1.
  const float g11 = fmaf(s1.x, s1.x, fmaf(s1.y, s1.y, s1.z * s1.z));
  const float g12 = fmaf(s1.x, s2.x, fmaf(s1.y, s2.y, s1.z * s2.z));
  const float cr = fmaf(s1.y * s2.z - s1.z * s2.y, ax, fmaf(s1.z * s2.x - s1.x * s2.z, ay, (s1.x * s2.y - s1.y * s2.x) * az));
  const float rl = rsqrtf(g11);
  const float c11 = g11 * rl, c21 = g12 * rl, c22 = fabsf(cr) * rl;
  const float Xc = X + fabsf(cx), Yc = Y + fabsf(cy);
  const float e = 2e-6f * fmaf(c11, Xc, (fabsf(c21) + c22) * Yc);
  const float sc = rsqrtf(9.01f + fmaf(12.0f, e, 2.0f * e * e));
  const float l11 = c11 * sc, l21 = c21 * sc, l22 = c22 * sc;
  // t* + zr = -cz - dx m1 - dy m2, off by at most et (widened by it: a hit ahead of the origin stays so)
  const float ter = 2e-6f * (fabsf(cz) + fmaf(fabsf(s1.w), Xc, fabsf(s2.w) * Yc));
  // the ellipse u^2 + v^2 <= 1 holds |dy| <= 1 / l22, |dx| <= |(l21, l22)| / (l11 l22) and
  // |dx m1 + dy m2| <= |L^-1 m|; its centre is at (-cx, -cy, -cz) from R. A NaN keeps the leaf.
  bool keep = pos >= 0;
  {
    const float i11 = __fdividef(1.0f, l11), i22 = __fdividef(1.0f, l22);
    const float k21 = l21 * i22, w1 = s1.w * i11, w2 = (s2.w - l21 * w1) * i22;
    const float m = 3e-5f * (1.0f + fabsf(rel.Rx) + fabsf(rel.Ry) + fabsf(rel.Rz) + fabsf(cx) + fabsf(cy) + fabsf(cz));
    const float rx = 1.001f * i11 * sqrtf(fmaf(k21, k21, 1.0f)) + m, ry = 1.001f * i22 + m;
    const float rz = 1.001f * sqrtf(fmaf(w1, w1, w2 * w2)) + 1e-3f * (fabsf(s1.w) * rx + fabsf(s2.w) * ry) + m;
    const float ox = rel.Rxl - cx, oy = rel.Ryl - cy, oz = rel.Rzl - cz;  // the centre on the frame
    keep = keep && !(ox + rx < bm.xlo) && !(ox - rx > bm.xhi) && !(oy + ry < bm.ylo) && !(oy - ry > bm.yhi) &&
           !(oz + rz < bm.zlo) && !(oz - rz > bm.zhi);
  }
  const unsigned m = __ballot_sync(0xffffffffu, keep);
  const int slot = __popc(m & ((1u << (threadIdx.x & 31)) - 1u));
  if (keep) {
    sm.stage[0][slot] = make_float4(cx, cy, cz, q0.w);
    sm.stage[1][slot] = s1;
    sm.stage[2][slot] = s2;
    sm.stage[3][slot] = make_float4(facing(f, q3), __int_as_float(pos), cxl, cyl);
    sm.quick[0][slot] = make_float4(l11, l21, fmaf(l11, cx, l21 * cy), ter - cz - fmaf(cx, s1.w, cy * s2.w));
    sm.quick[1][slot] = make_float4(l22, l22 * cy, s1.w, s2.w);
  }
  et = warp_max(keep ? ter : 0.0f);
  __syncwarp();
  return __popc(m);
}

// Projection of a box [lo, hi] on the frame: centre and half-width along e1, e2 and w, widened
// by a margin above the FP32 error of these sums and of a ray's drift off its projected origin
// (|w.e1| of a few ulp times the distance travelled). Any point of the box -- in particular the
// closest approach of a ray that hits a Gaussian inside it -- projects inside these intervals.
__device__ __forceinline__ void project_box(const Frame& f, float lx, float ly, float lz, float hx, float hy,
                                            float hz, float4& A, float2& Z) {
  const float cx = 0.5f * (lx + hx), cy = 0.5f * (ly + hy), cz = 0.5f * (lz + hz);
  const float hxx = 0.5f * (hx - lx), hyy = 0.5f * (hy - ly), hzz = 0.5f * (hz - lz);
  const float px = f.e1x * cx + f.e1y * cy + f.e1z * cz;
  const float py = f.e2x * cx + f.e2y * cy + f.e2z * cz;
  const float pz = f.wx * cx + f.wy * cy + f.wz * cz;
  const float rx = fabsf(f.e1x) * hxx + fabsf(f.e1y) * hyy + fabsf(f.e1z) * hzz;
  const float ry = fabsf(f.e2x) * hxx + fabsf(f.e2y) * hyy + fabsf(f.e2z) * hzz;
  const float rz = fabsf(f.wx) * hxx + fabsf(f.wy) * hyy + fabsf(f.wz) * hzz;
  const float m = 3e-5f * (1.0f + fabsf(cx) + fabsf(cy) + fabsf(cz) + hxx + hyy + hzz);
  A = make_float4(px, py, rx + m, ry + m);
  Z = make_float2(pz - rz - m, pz + rz + m);
}

__device__ __forceinline__ bool beam_meets(const Beam& b, const float4& A, const float2& Z) {
  return A.x + A.z >= b.xlo && A.x - A.z <= b.xhi && A.y + A.w >= b.ylo && A.y - A.w <= b.yhi && Z.y >= b.zlo &&
         Z.x <= b.zhi;
}

// The exact test of one staged leaf for the lane: D^2 and t* (see Rel). The high parts of dx
// cancel without rounding error of their own beyond eps |dx| (exactly where they nearly cancel);
// the low parts carry the roundings of both.
__device__ __forceinline__ void leaf_offset(const Rel& rel, const PacketSmem& sm, int j, float& wx, float& wy, float& wz,
                                            float& t) {
  const float4 s0 = sm.stage[0][j], s1 = sm.stage[1][j], s2 = sm.stage[2][j], s3 = sm.stage[3][j];
  const float dx = (rel.xr + s0.x) + (rel.xr_lo + s3.z), dy = (rel.yr + s0.y) + (rel.yr_lo + s3.w);
  wx = fmaf(dx, s1.x, dy * s2.x);
  wy = fmaf(dx, s1.y, dy * s2.y);
  wz = fmaf(dx, s1.z, dy * s2.z);
  t = -(rel.zr + s0.z) - fmaf(dx, s1.w, dy * s2.w);
}

__device__ __forceinline__ void leaf_test(const Rel& rel, const PacketSmem& sm, int j, float& d2, float& t) {
  float wx, wy, wz;
  leaf_offset(rel, sm, j, wx, wy, wz, t);
  d2 = fmaf(wx, wx, fmaf(wy, wy, wz * wz));
}

// Hit decision of a leaf by the single ray's own test (the transfer backward decides as the per-ray
// walk does): only where the planar test is near a boundary, D^2 = 9 or t* = 0, can the two differ.
// The band is some ten times the largest difference of their roundings.
__device__ __noinline__ bool ray_hit(const float4* __restrict__ recs, int pos, float ox, float oy, float oz, float dx,
                                     float dy, float dz) {
  Ray r{};
  r.ox = ox;
  r.oy = oy;
  r.oz = oz;
  r.dx = dx;
  r.dy = dy;
  r.dz = dz;
  float t, al, m;
  return gauss_hit(recs, pos, r, t, al, m);
}

__device__ __forceinline__ bool ray_decides(const float4* __restrict__ recs, const Frame& f, float ox, float oy, float oz,
                                            const Rel& rel, const PacketSmem& sm, int j, int pos, float d2, float t,
                                            bool planar) {
  const float4 s0 = sm.stage[0][j];
  const float dx = rel.xr + s0.x, dy = rel.yr + s0.y;
  const float band = 1e-4f * (fabsf(rel.zr) + fabsf(s0.z) + fabsf(dx) * (1.0f + fabsf(sm.stage[1][j].w)) +
                              fabsf(dy) * (1.0f + fabsf(sm.stage[2][j].w)));
  if (!(d2 > 9.02f) && !(t < -band) && (!(d2 < 8.98f) || !(t > band)))
    return ray_hit(recs, pos, ox, oy, oz, f.wx, f.wy, f.wz);
  return planar;
}

// Quick test of the staged leaves for the lane: bit j of the result is set for every leaf j < cnt whose
// exact test can pass (and for a few more). Two 16-byte loads, seven FMAs and three comparisons per
// leaf, no branch; a NaN passes on to the exact test. zlo: tlo + zr, zhi: thn + zr, both widened.
__device__ __forceinline__ unsigned quick_mask(const PacketSmem& sm, int cnt, float x, float y, float zlo, float zhi) {
  unsigned pass = 0u;
#pragma unroll 1
  for (int j0 = 0; j0 < cnt; j0 += 8) {
    unsigned m = 0u;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const float4 a = sm.quick[0][j0 + k], b = sm.quick[1][j0 + k];
      const float u = fmaf(a.x, x, fmaf(a.y, y, a.z));
      const float v = fmaf(b.x, y, b.y);
      const float d = fmaf(u, u, v * v);
      const float t = fmaf(-b.z, x, fmaf(-b.w, y, a.w));
      if (!(d > 1.0f) && !(t <= zlo) && !(t > zhi)) m |= 1u << k;
    }
    pass |= m << j0;
  }
  return cnt < 32 ? pass & ((1u << cnt) - 1u) : pass;
}

// One packet walk. Lane state: `active` (this lane's ray takes part), its projected origin
// (xl, yl) and depth zl (for the beam), its offset from the packet's reference point (rel, for the
// exact test), the lower bound t_lo of the hits it wants (0: all hits ahead) and its visitor, whose
// t_hi() bounds the hits it still wants and stop() ends its ray. The leaves of a chunk are staged
// 32 at a time (one record load and the per-Gaussian terms of the tests per lane). Every lane then
// takes the quick test of all of them into a 32-bit mask, without a branch, and drains its mask: the
// exact test (of Rel above) and, for the hits, vis.hit(), in chunk order. A leaf is hit by about a
// tenth of the lanes, so walking the leaves in step and branching to the visitor would run it with
// three lanes of 32; in the drain every lane is at a hit of its own.
template <class Vis>
__device__ void packet_walk(const TraceArgs& a, const Frame& f, const Rel& rel, int self, int root,
                            bool active, float xl, float yl, float zl, float t_lo, Vis& vis, PacketSmem& sm,
                            RayStats& st, unsigned& node_count) {
  const int lane = threadIdx.x & 31;
  const float prune_lo = t_lo > 0.f ? t_lo * (1.0f - 1e-5f) - 1e-6f : -FLT_MAX;
  // t > 0 && t >= prune_lo as one strict test against the float below prune_lo (or 0)
  const float tlo = prune_lo > 0.f ? nextafterf(prune_lo, 0.0f) : 0.0f;
  const unsigned above = lane == 31 ? 0u : (0xffffffffu << (lane + 1));  // lanes > lane
  const unsigned below = (1u << lane) - 1u;                                // lanes < lane
  const float zlo_l = t_lo > 0.f ? zl + (t_lo * (1.0f - 1e-5f) - 1e-6f) : zl;
  bool need = active && !vis.stop();
  if (!__any_sync(0xffffffffu, need) || root == INT32_MIN) return;
  if (root < 0) return;  // a one-Gaussian scene: the receiver alone
  float th = vis.t_hi();
  Beam bm = make_beam(need, xl, yl, zlo_l, th == FLT_MAX ? FLT_MAX : zl + th);
  const float X = warp_max(need ? fabsf(rel.xr) : 0.0f), Y = warp_max(need ? fabsf(rel.yr) : 0.0f);
  const float zlo_q = (tlo + rel.zr) - 2e-6f * (tlo + fabsf(rel.zr));
  int sp = 1, nl = 0;
  if (lane == 0) sm.stack[0] = root;
  __syncwarp();
  const int64_t max_steps = 4 * a.n + 64;
  for (int64_t step = 0;; ++step) {
    if (step > max_steps) {
      set_status(a.status, PRTGS_STATUS_BAD_INDEX);
      break;
    }
    if (sp > 0) {
      const int npop = sp + kPHeadroom <= kPStack ? min(32, sp) : 1;
      int node = -1;
      if (lane < npop) node = sm.stack[sp - 1 - lane];
      sp -= npop;
      if (lane == 0) node_count += npop;
      bool push0 = false, push1 = false, leaf0 = false, leaf1 = false;
      int c0 = 0, c1 = 0;
      bool near0 = true;
      if (node >= 0) {
        float4 n0, n1, n2, A0, A1;
        float2 Z0, Z1;
        load_node(a.nodes, node, n0, n1, n2, c0, c1);
        project_box(f, n0.x, n0.y, n0.z, n0.w, n1.x, n1.y, A0, Z0);
        project_box(f, n1.z, n1.w, n2.x, n2.y, n2.z, n2.w, A1, Z1);
        const bool h0 = beam_meets(bm, A0, Z0) && child_ok(c0, a.n, a.status);
        const bool h1 = beam_meets(bm, A1, Z1) && child_ok(c1, a.n, a.status);
        push0 = h0 && c0 >= 0;
        push1 = h1 && c1 >= 0;
        leaf0 = h0 && c0 < 0;
        leaf1 = h1 && c1 < 0;
        near0 = Z0.x + Z0.y <= Z1.x + Z1.y;  // nearer box centre along w
      }
      // pushes: far child first, near child on top; lane 0's pushes end on top of the stack
      const int np = (int)push0 + (int)push1;
      const unsigned b1 = __ballot_sync(0xffffffffu, np >= 1), b2 = __ballot_sync(0xffffffffu, np == 2);
      int pos = sp + __popc(b1 & above) + __popc(b2 & above);
      if (pos + np > kPStack) {  // only a malformed tree gets here: report, drop the pushes
        set_status(a.status, PRTGS_STATUS_STACK_OVERFLOW);
      } else if (np == 2) {
        sm.stack[pos] = near0 ? c1 : c0;
        sm.stack[pos + 1] = near0 ? c0 : c1;
      } else if (np == 1) {
        sm.stack[pos] = push0 ? c0 : c1;
      }
      sp = min(sp + __popc(b1) + __popc(b2), kPStack);
      // leaves: appended to the chunk (every lane tests its own ray against them)
      const int nlf = (int)leaf0 + (int)leaf1;
      const unsigned l1 = __ballot_sync(0xffffffffu, nlf >= 1), l2 = __ballot_sync(0xffffffffu, nlf == 2);
      int lp = nl + __popc(l1 & below) + __popc(l2 & below);
      if (leaf0) sm.lpos[lp++] = ~c0;
      if (leaf1) sm.lpos[lp] = ~c1;
      nl += __popc(l1) + __popc(l2);
      __syncwarp();
    }
    if (nl > kPLeaves - 64 || (sp == 0 && nl > 0)) {
      for (int g = 0; g < nl; g += 32) {
        float et;
        const int cnt = stage_leaves(a.recs, g + lane < nl ? sm.lpos[g + lane] : -1, f, rel, bm, X, Y, sm, et);
        if (lane == 0) st.entries += cnt;
        if (need) st.leaves += cnt;  // leaf tests of the lane (its own Gaussian included)
        float thn = need ? th : -FLT_MAX;  // a lane that wants no hits passes no test
        const float zhi_q = need ? (thn + rel.zr) + (2.0f * et + 2e-6f * (fabsf(thn) + fabsf(rel.zr))) : -FLT_MAX;
        // ray_decides' band about t* = 0, but for its terms of the lane's own depth (zlo_q has 2e-6 of it) and offset
        const float zlo_g = Vis::kRayDecides ? zlo_q - 50.0f * et : zlo_q;
        unsigned pass = need ? quick_mask(sm, cnt, rel.xr, rel.yr, zlo_g, zhi_q) : 0u;
        if constexpr (Vis::kInStep) {
          unsigned any = __reduce_or_sync(0xffffffffu, pass);
          while (any) {
            const int j = __ffs(any) - 1;
            any &= any - 1u;
            float d2, t;
            leaf_test(rel, sm, j, d2, t);
            const int pos = __float_as_int(sm.stage[3][j].y);
            bool h = d2 <= 9.0f && t > tlo && t <= thn && pos != self;
            if constexpr (Vis::kRayDecides) {
              if (need && pos != self) h = ray_decides(a.recs, f, vis.ox, vis.oy, vis.oz, rel, sm, j, pos, d2, t, h);
            }
            if (vis.step(h, pos, t, sm.stage[0][j].w * expf(-0.5f * d2), sm.stage[3][j].x)) ++st.hits;
          }
          need = need && !vis.stop();
          th = vis.t_hi();
          pass = 0u;
        }
        while (pass) {
          const int j = __ffs(pass) - 1;
          pass &= pass - 1u;
          float d2, t;
          leaf_test(rel, sm, j, d2, t);
          const float4 s3 = sm.stage[3][j];
          const int pos = __float_as_int(s3.y);
          if (d2 <= 9.0f && t > tlo && t <= thn && pos != self) {
            ++st.hits;
            vis.hit(pos, t, sm.stage[0][j].w * expf(-0.5f * d2), s3.x);
            th = vis.t_hi();  // th only falls
            need = !vis.stop();
            thn = th;
            if (!need) pass = 0u;
          }
        }
        __syncwarp();
      }
      nl = 0;
      if (!__any_sync(0xffffffffu, need)) break;
      th = vis.t_hi();
      bm = make_beam(need, xl, yl, zlo_l, th == FLT_MAX ? FLT_MAX : zl + th);
      __syncwarp();
    }
    if (sp == 0 && nl == 0) break;
  }
  __syncwarp();
}

// Visibility: product of (1 - alpha) over every hit, in any order; stops below t_min. Its code is short
// and the hits of a leaf fall on neighbouring rays (9 lanes of 30 per leaf that is hit at all), so the
// lanes take the leaves in step, each factor a select: no divergence, and the staged terms are
// broadcast reads.
struct VisibilityVis {
  static constexpr bool kRayDecides = false;
  static constexpr bool kInStep = true;
  float t_min, T;
  __device__ float t_hi() const { return FLT_MAX; }
  __device__ bool stop() const { return T < t_min; }
  __device__ bool step(bool h, int, float, float al, float) {
    h = h && !(T < t_min);
    T = h ? T * (1.0f - al) : T;
    return h;
  }
  __device__ void hit(int, float, float, float) {}
};

// Visibility walk of the bounce mode. Until T < t_min it multiplies every hit into T (in any
// order, as ShadowVis), records the largest alpha m of the front-facing hits and, at the cut-off,
// the horizon: the largest t* met so far (a hit past it has prefix transmittance below t_min and
// is no index-matrix candidate). It keeps the nearest front-facing hit (by key). After the cut-off
// the walk goes on pruned to the nearer of the horizon and that hit, so that it ends as the
// nearest front-facing hit of the whole ray within the horizon: the first index-matrix candidate.
// It also sums log(1 - alpha) over the hits in front of the current candidate (lpre). That sum
// stays exact while no hit it holds lies behind a nearer candidate found later (checked with the
// largest key summed); when it holds, the index search needs no walk in front of the candidate.
struct BounceVis {
  static constexpr bool kRayDecides = false;
  static constexpr bool kInStep = false;  // surface-100k transfer 60.3 ms drained, 61.8 in step
  float t_min;
  float T;
  float t_seen;
  float t_hor;
  float tf;  // nearest front-facing hit: t*, position, alpha
  int pf;
  float af;
  float amax;  // largest alpha m of the front-facing hits multiplied into T
  float lpre;  // sum of log(1 - alpha) of the hits with key below (tf, pf)
  float ts;    // largest key summed into lpre: t*, position
  int ps;
  bool pre_ok;  // lpre is the prefix of (tf, pf)
  __device__ float t_hi() const { return T < t_min ? fminf(slack_hi(t_hor), slack_hi(tf)) : FLT_MAX; }
  __device__ bool stop() const { return false; }
  __device__ bool step(bool, int, float, float, float) { return false; }
  // (a hit past t_hi() changes nothing here)
  __device__ void hit(int pos, float t, float al, float m) {
    const bool live = !(T < t_min);
    if (live) {
      T *= 1.0f - al;
      t_seen = fmaxf(t_seen, t);
      if (T < t_min) t_hor = t_seen;
      if (m > 0.f) amax = fmaxf(amax, al * m);
    }
    const bool closer = (live || !(t > t_hor)) && key_less(t, pos, tf, pf);
    if (m > 0.f) {
      if (closer) {
        if (ps != INT32_MIN && !key_less(ts, ps, t, pos)) pre_ok = false;  // a summed hit lies behind it
        tf = t;
        pf = pos;
        af = al;
      }
    } else if (closer) {
      lpre += log1pf(-al);
      if (ps == INT32_MIN || key_less(ts, ps, t, pos)) {
        ts = t;
        ps = pos;
      }
    }
  }
};

// One search round of the index matrix: the KR nearest hits of any kind with key past the last
// one processed (and t* within the horizon), kept sorted by key in the lane's column of a shared-
// memory buffer, for processing in key order. In the first round (no hit processed yet) the hits
// in front of the first candidate (key below (tf, pf)) are not kept but summed into lbase = log of
// the prefix transmittance in front of that candidate.
template <int KR>
struct SearchVis {
  static constexpr bool kRayDecides = false;
  static constexpr bool kInStep = false;
  __device__ bool step(bool, int, float, float, float) { return false; }
  float t_last;
  int p_last;
  float t_hor;
  float tf;
  int pf;
  float lbase;
  RoundHits& buf;
  int lane;
  int count;
  float t_max;  // key of the last kept hit once the buffer is full
  int p_max;
  __device__ float t_hi() const { return fminf(count == KR ? slack_hi(t_max) : FLT_MAX, slack_hi(t_hor)); }
  __device__ bool stop() const { return false; }
  __device__ void hit(int pos, float t, float al, float m) {
    if (!key_less(t_last, p_last, t, pos)) return;
    if (key_less(t, pos, tf, pf)) {
      lbase += log1pf(-al);
      return;
    }
    if (count == KR && !key_less(t, pos, t_max, p_max)) return;
    // sorted insertion: shift the larger keys up by one (the last falls out when full)
    int k = count < KR ? count : KR - 1;
    while (k > 0) {
      const float te = buf.t[k - 1][lane];
      const int pe = buf.pos[k - 1][lane];
      if (!key_less(t, pos, te, pe)) break;
      buf.t[k][lane] = te;
      buf.pos[k][lane] = pe;
      buf.sal[k][lane] = buf.sal[k - 1][lane];
      --k;
    }
    buf.t[k][lane] = t;
    buf.pos[k][lane] = pos;
    buf.sal[k][lane] = m > 0.f ? -al : al;
    if (count < KR) ++count;
    if (count == KR) {
      t_max = buf.t[KR - 1][lane];
      p_max = buf.pos[KR - 1][lane];
    }
  }
};

// A ray handed from the visibility walk to the index-matrix search (self < 0: none).
struct __align__(16) SearchRec {
  int self;
  int ref;  // receiver whose origin is the reference point of the exact tests; sign bit: lpre is exact
  float t_hor;
  float tf;  // the nearest front-facing hit: t*, position, alpha
  int pf;
  float af;
  float lamax;  // every later candidate has log W_j <= lamax + log T_j
  float lpre;
};

// Index matrix (Sec. 4.4): argmax of W_j = alpha_j T_j m_j over the hits in key order, T_j the prefix
// transmittance; candidates need T_j >= t_min and T_j <= filter_t. Every later candidate has
// W_j <= amax T_j (amax covers every front-facing hit when no cut-off happened, else the trivial bound
// 1). With an exact prefix of the first candidate, the candidate is taken here, as the rounds would
// take it (same arithmetic), and the rounds start behind it, if they are still needed: often its
// weight already settles the argmax.
struct FirstCandidate {
  bool searching;
  float t_last, lt, lw_best;
  int p_last, best;
};

__device__ __forceinline__ FirstCandidate first_candidate(const TraceArgs& a, const Frame& f, const SearchRec& r) {
  FirstCandidate c{true, -FLT_MAX, 0.0f, -FLT_MAX, INT32_MIN, -1};
  if (r.ref >= 0) return c;
  const float lmin = a.t_min > 0.f ? logf(a.t_min) : -FLT_MAX;
  c.lt = r.lpre;
  if (c.lt < lmin) {
    c.searching = false;
    return c;
  }
  if (c.lt <= logf(a.filter_t)) {
    const float lw = logf(r.af * facing(f, __ldg(a.recs + 4 * (int64_t)r.pf + 3))) + c.lt;
    if (lw > c.lw_best) {
      c.lw_best = lw;
      c.best = r.pf;
    }
  }
  c.lt += log1pf(-r.af);
  if (c.lt < lmin || c.lt + r.lamax <= c.lw_best) c.searching = false;
  c.t_last = r.tf;
  c.p_last = r.pf;
  return c;
}

// Visibility (and with BOUNCE the first index-matrix candidates) of the rays of receiver batch [r0, r1):
// V[s * batch + (i - r0)] (0 where n.w <= 0), idx[gid * S + s].
#ifndef PRTGS_PACKET_BOUNCE_MIN_BLOCKS
#define PRTGS_PACKET_BOUNCE_MIN_BLOCKS 4  // surface-100k transfer 60.3 ms at 4, 61.8 at 5
#endif
template <bool BOUNCE>
__global__ void __launch_bounds__(kPacketThreads, BOUNCE ? PRTGS_PACKET_BOUNCE_MIN_BLOCKS : PRTGS_PACKET_MIN_BLOCKS)
    k_packet(TraceArgs a, float* __restrict__ V, int dpi) {
  extern __shared__ float4 psmem4[];
  PacketSmem* wsm = reinterpret_cast<PacketSmem*>(psmem4);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  PacketSmem& sm = wsm[warp];
  __shared__ unsigned int s_item[kPacketWarps];
  const int64_t batch = a.r1 - a.r0;
  const int64_t n_windows = (batch + 63) / 64;
  const int dblocks = (a.S + dpi - 1) / dpi;  // dpi directions per work item
  const unsigned below = (1u << lane) - 1u;
  RayStats rs{0u, 0u, 0u, 0u, 0u, 0u};
  unsigned traced = 0, walks = 0;
  for (;;) {
    if (lane == 0) s_item[warp] = atomicAdd(a.work, 1u);
    __syncwarp();
    const unsigned item = s_item[warp];
    __syncwarp();
    if ((int64_t)item >= 2 * n_windows * dblocks) break;
    // a window of 64 receivers adjacent in Morton order, in up to two packets of 32 lanes, an item each (one
    // after the other in one item, 1,024 splats at 64 directions took 143 us, now 114: few items, long walks);
    // each lane stages two of them
    const int pass = (int)(item & 1u);
    const int64_t base = a.r0 + 64 * ((item >> 1) / dblocks);
    const int s0 = (int)((item >> 1) % dblocks) * dpi;
    float4 nq[2];  // record row 3 of the lane's two receivers (its .yzw: the normal)
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int j = lane + 32 * h;
      nq[h] = __ldg(a.recs + 4 * (base + j < a.r1 ? base + j : a.r0) + 3);
    }
    const int s1 = min(a.S, s0 + dpi);
    for (int s = s0; s < s1; ++s) {
      const float d[3] = {__ldg(a.dirs + 3 * s), __ldg(a.dirs + 3 * s + 1), __ldg(a.dirs + 3 * s + 2)};
      // the receivers of the window that face direction s, compacted into packets of 32 lanes
      // (a window whose receivers all face it gives the two packets of its halves)
      bool upj[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int j = lane + 32 * h;
        const bool vj = base + j < a.r1;
        upj[h] = vj && ray_cos(nq[h].y, nq[h].z, nq[h].w, d) > 0.0f;
        if (vj && !upj[h] && pass == 0) {  // untraced ray: no visibility, no index-matrix entry
          V[(int64_t)s * batch + (base + j - a.r0)] = 0.0f;
          if (BOUNCE) a.idx[(int64_t)__ldg(a.order + base + j) * a.S + s] = -1;
        }
      }
      const unsigned m0 = __ballot_sync(0xffffffffu, upj[0]), m1 = __ballot_sync(0xffffffffu, upj[1]);
      const int total = __popc(m0) + __popc(m1);
      if (pass * 32 >= total) continue;
      if (upj[0]) sm.rlist[__popc(m0 & below)] = (unsigned char)lane;
      if (upj[1]) sm.rlist[__popc(m0) + __popc(m1 & below)] = (unsigned char)(lane + 32);
      __syncwarp();
      const bool up = pass * 32 + lane < total;
      const int jw = up ? sm.rlist[pass * 32 + lane] : 0;
      const int self = (int)(base + jw);
      const float4 q0 = __ldg(a.recs + 4 * (int64_t)self);
      const int gid = __ldg(a.order + self);
      int root = INT32_MIN;
      if (up) {
        root = a.roots[find_scene(a.offsets, a.n_scenes, gid)];
        if (root != INT32_MIN && !child_ok(root, a.n, a.status)) root = INT32_MIN;
      }
      float vis = up ? 1.0f : 0.0f;
      int best = -1;  // index-matrix entry (sorted position of the chosen hit)
      SearchRec rec;
      rec.self = -1;
      if ((a.flags & PRTGS_SHADOW) && __any_sync(0xffffffffu, up)) {
        const Frame f = make_frame(d[0], d[1], d[2]);
        const float xl = f.e1x * q0.x + f.e1y * q0.y + f.e1z * q0.z;
        const float yl = f.e2x * q0.x + f.e2y * q0.y + f.e2z * q0.z;
        const float zl = f.wx * q0.x + f.wy * q0.y + f.wz * q0.z;
        traced += up ? 1u : 0u;
        // lanes of different scenes walk their own subtrees, one group at a time
        unsigned todo = __ballot_sync(0xffffffffu, up);
        while (todo) {
          const int leader = __ffs(todo) - 1;
          const int groot = __shfl_sync(0xffffffffu, root, leader);
          const unsigned grp = __ballot_sync(0xffffffffu, up && root == groot) & todo;
          const bool mine = (grp >> lane) & 1u;
          if (lane == 0) ++walks;
          const int leader_self = __shfl_sync(0xffffffffu, self, leader);
          // reference point of the group's exact tests: its leader's ray origin
          const Rel rel = make_rel(f, q0.x, q0.y, q0.z, __shfl_sync(0xffffffffu, q0.x, leader),
                                   __shfl_sync(0xffffffffu, q0.y, leader), __shfl_sync(0xffffffffu, q0.z, leader));
          if (!BOUNCE) {
            VisibilityVis sv{a.t_min, 1.0f};
            packet_walk(a, f, rel, self, groot, mine, xl, yl, zl, 0.0f, sv, sm, rs, rs.nodes);
            if (mine) vis = sv.T;
          } else {
            BounceVis bv{a.t_min, 1.0f, 0.0f, FLT_MAX, FLT_MAX, INT32_MAX, 0.0f, 0.0f, 0.0f, 0.0f, INT32_MIN, true};
            packet_walk(a, f, rel, self, groot, mine, xl, yl, zl, 0.0f, bv, sm, rs, rs.nodes);
            if (mine) vis = bv.T;
            // the index-matrix search goes on in k_search, for the rays whose first candidate does not
            // already settle the argmax
            FirstCandidate fc;
            if (mine && bv.tf != FLT_MAX) {
              const float lamax = bv.T < a.t_min ? 0.0f : logf(bv.amax);
              rec = SearchRec{self, leader_self | (bv.pre_ok ? INT32_MIN : 0), bv.t_hor, bv.tf, bv.pf, bv.af, lamax, bv.lpre};
              fc = first_candidate(a, f, rec);
              best = fc.best;
              if (!fc.searching) rec.self = -1;
            }
          }
          todo &= ~grp;
        }
      }
      if (up) {
        V[(int64_t)s * batch + (self - a.r0)] = vis;
        if (BOUNCE) a.idx[(int64_t)gid * a.S + s] = best >= 0 ? a.order[best] : -1;
      }
      if (BOUNCE && __any_sync(0xffffffffu, rec.self >= 0)) {  // a search item: the packet's rays that go on
        unsigned e = 0;
        if (lane == 0) e = atomicAdd(a.queue_count, 1u);
        e = __shfl_sync(0xffffffffu, e, 0);
        if (lane == 0) a.pending[e] = (uint32_t)s;
        static_cast<SearchRec*>(a.queue)[(int64_t)e * 32 + lane] = rec;
      }
      __syncwarp();  // the compacted list is rewritten for the next direction
    }
    __syncwarp();  // the window is restaged by the next work item
  }
  if (a.stats) {
    unsigned long long c0 = warp_sum_u64(rs.nodes), c1 = warp_sum_u64(rs.search_nodes),
                       c2 = warp_sum_u64(rs.leaves), c3 = warp_sum_u64(rs.hits), c4 = warp_sum_u64(rs.rounds),
                       c5 = warp_sum_u64(traced), c8 = warp_sum_u64(walks), c9 = warp_sum_u64(rs.entries);
    if (lane == 0) {
      atomicAdd(a.stats + 0, c0);
      atomicAdd(a.stats + 1, c1);
      atomicAdd(a.stats + 4, c4);
      atomicAdd(a.stats + 2, c2);
      atomicAdd(a.stats + 3, c3);
      atomicAdd(a.stats + 5, c5);
      atomicAdd(a.stats + 8, c8);
      atomicAdd(a.stats + 9, c9);
    }
  }
}

// The index-matrix search of the packets that k_packet<true> left: one warp per item, rounds of kPacketRoundHits hits
// in key order until every ray's argmax is settled. A kernel of its own: only a third of the packets
// get here, and beside the visibility walk's code and registers both ran slower.
#ifndef PRTGS_SEARCH_MIN_BLOCKS
#define PRTGS_SEARCH_MIN_BLOCKS 4
#endif
__global__ void __launch_bounds__(kPacketThreads, PRTGS_SEARCH_MIN_BLOCKS) k_search(TraceArgs a) {
  extern __shared__ float4 psmem4[];
  PacketSmem* wsm = reinterpret_cast<PacketSmem*>(psmem4);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  PacketSmem& sm = wsm[warp];
  RoundHits& hbuf = reinterpret_cast<RoundHits*>(wsm + kPacketWarps)[warp];
  RayStats rs{0u, 0u, 0u, 0u, 0u, 0u};
  const unsigned items = *a.queue_count;
  for (;;) {
    unsigned item = 0;
    if (lane == 0) item = atomicAdd(a.work, 1u);
    item = __shfl_sync(0xffffffffu, item, 0);
    if (item >= items) break;
    const int s = (int)a.pending[item];
    const SearchRec rec = static_cast<const SearchRec*>(a.queue)[(int64_t)item * 32 + lane];
    const bool mine = rec.self >= 0;
    const int self = mine ? rec.self : (int)a.r0;
    const float d[3] = {__ldg(a.dirs + 3 * s), __ldg(a.dirs + 3 * s + 1), __ldg(a.dirs + 3 * s + 2)};
    const Frame f = make_frame(d[0], d[1], d[2]);
    const float4 q0 = __ldg(a.recs + 4 * (int64_t)self);
    const int gid = __ldg(a.order + self);
    const int ref = rec.ref & INT32_MAX;
    const int root = mine ? a.roots[find_scene(a.offsets, a.n_scenes, gid)] : INT32_MIN;
    const float xl = f.e1x * q0.x + f.e1y * q0.y + f.e1z * q0.z;
    const float yl = f.e2x * q0.x + f.e2y * q0.y + f.e2z * q0.z;
    const float zl = f.wx * q0.x + f.wy * q0.y + f.wz * q0.z;
    const float lfilter = logf(a.filter_t);
    const float lmin = a.t_min > 0.f ? logf(a.t_min) : -FLT_MAX;
    const bool pre = rec.ref < 0;
    FirstCandidate c{false, -FLT_MAX, 0.0f, -FLT_MAX, INT32_MIN, -1};
    if (mine) c = first_candidate(a, f, rec);
    unsigned todo = __ballot_sync(0xffffffffu, mine);
    while (todo) {  // rays of different scenes one group at a time
      const int leader = __ffs(todo) - 1;
      const int groot = __shfl_sync(0xffffffffu, root, leader);
      const unsigned grp = __ballot_sync(0xffffffffu, mine && root == groot) & todo;
      const int gref = __shfl_sync(0xffffffffu, ref, leader);
      const float4 R = __ldg(a.recs + 4 * (int64_t)gref);
      const Rel rel = make_rel(f, q0.x, q0.y, q0.z, R.x, R.y, R.z);
      bool searching = ((grp >> lane) & 1u) && c.searching;
      for (int64_t round = 0; __any_sync(0xffffffffu, searching); ++round) {
        if (round > a.n / kPacketRoundHits + 1) {
          if (searching) set_status(a.status, PRTGS_STATUS_BAD_INDEX);
          break;
        }
        SearchVis<kPacketRoundHits> sv{c.t_last, c.p_last, rec.t_hor, rec.tf, rec.pf, 0.0f, hbuf, lane, 0, FLT_MAX, INT32_MAX};
        if (searching) ++rs.rounds;
        packet_walk(a, f, rel, self, groot, searching, xl, yl, zl, c.t_last > 0.f ? c.t_last : 0.0f, sv, sm, rs,
                    rs.search_nodes);
        if (searching) {
          if (round == 0 && !pre) c.lt = sv.lbase;
          const int nh = sv.count;
          bool decided = false;
          for (int k = 0; k < nh && !decided; ++k) {
            if (c.lt < lmin || c.lt + rec.lamax <= c.lw_best) {
              decided = true;
            } else {
              const float sal = hbuf.sal[k][lane], al = fabsf(sal);
              if (signbit(sal) && c.lt <= lfilter) {  // front-facing
                const int pos = hbuf.pos[k][lane];
                const float lw = logf(al * facing(f, __ldg(a.recs + 4 * (int64_t)pos + 3))) + c.lt;
                if (lw > c.lw_best) {
                  c.lw_best = lw;
                  c.best = pos;
                }
              }
              c.lt += log1pf(-al);
            }
          }
          if (decided || nh < kPacketRoundHits || c.lt < lmin || c.lt + rec.lamax <= c.lw_best) {
            searching = false;
          } else {
            c.t_last = sv.t_max;
            c.p_last = sv.p_max;
          }
        }
        __syncwarp();
      }
      todo &= ~grp;
    }
    if (mine) a.idx[(int64_t)gid * a.S + s] = c.best >= 0 ? a.order[c.best] : -1;
    __syncwarp();
  }
  if (a.stats) {
    const unsigned long long c1 = warp_sum_u64(rs.search_nodes), c2 = warp_sum_u64(rs.leaves), c3 = warp_sum_u64(rs.hits),
                             c4 = warp_sum_u64(rs.rounds), c9 = warp_sum_u64(rs.entries);
    if (lane == 0) {
      atomicAdd(a.stats + 1, c1);
      atomicAdd(a.stats + 2, c2);
      atomicAdd(a.stats + 3, c3);
      atomicAdd(a.stats + 4, c4);
      atomicAdd(a.stats + 9, c9);
    }
  }
}

// ---- backward of the shadowed transfer ---------------------------------------------------------------
// Per ray V = prod (1 - alpha_j); with g_V its gradient, dL/dalpha_j = -g_V V / (1 - alpha_j), and with
// x the whitened offset at the closest approach (D^2 = |x|^2), g = dL/dD^2 = -alpha/2 dL/dalpha:
//   d opacity_j += dL/dalpha exp(-D^2/2),  d mu_j -= 2 g A^T x,  d o += 2 g A^T x,
//   d s_k -= 2 g x_k^2 / s_k,  d R_jk += 2 g x_k w_j / s_k with w = R diag(s) x.
// So a Gaussian needs only sum g_alpha exp(-D^2/2), sum g x and sum g x x^T over its hits, ten numbers
// that do not depend on the direction. k_packet_bwd walks each packet once for V, noting the leaves that
// any of its rays hit, then goes through that list: every lane forms its g and the offset w' = x cross a
// (two coordinates in a plane of the leaf), the six moments are summed over the packet's rays through
// shared memory, and one lane per leaf turns them into the ten sums and adds them with three vector
// reductions. k_bwd_finish forms the gradients, once per Gaussian.
// Walking each ray alone and twice, with twelve atomics per hit, took 843 ms for a 100k volume at 128
// directions and 147 ms for 40k surface splats at 256; this takes 77 and 14 ms, bound by issue slots.
// Hits are decided as by the ray's own test (ray_decides, a tenth of that time): on a surface, splats in
// the receiver's own plane have t* = 0 up to rounding and a large alpha.

// Hits of the packet's rays, as VisibilityVis, and the list of the leaves hit by any of them from the
// skip-th on (a list that overflows is continued by another walk: the same leaves in the same order).
struct HitListVis {
  static constexpr bool kInStep = true, kRayDecides = true;
  float t_min, T;
  float ox, oy, oz;  // the ray's origin
  int* list;
  int skip, cap, total;
  __device__ float t_hi() const { return FLT_MAX; }
  __device__ bool stop() const { return T < t_min; }
  __device__ bool step(bool h, int pos, float, float al, float) {
    h = h && !(T < t_min);
    T = h ? T * (1.0f - al) : T;
    if (__any_sync(0xffffffffu, h)) {
      const int k = total - skip;
      if ((threadIdx.x & 31) == 0 && k >= 0 && k < cap) list[k] = pos;
      ++total;
    }
    return h;
  }
  __device__ void hit(int, float, float, float) {}
};

constexpr int kBwdBlocks = 4;      // per SM
constexpr int kBwdMaxBlocks = 152 * kBwdBlocks;  // of a launch: the workspace depends on the arguments, not on a device
constexpr int kBwdList = 2048;     // hit leaves of a packet kept at a time
constexpr int kBwdBatch = 5;       // leaves whose six moments are summed together (30 lanes, one sum each)
constexpr int kBwdRow = 36;        // 32 lanes' values and padding: 16-byte reads of 30 rows without conflicts

struct BwdSmem {
  float row[6 * kBwdBatch][kBwdRow];
  float sum[32][8];
};

// G, GV: [S][batch] gradients of each ray's c V (for the normal) and of its V; acc: [n][12] sums per
// Gaussian, rayacc: [n][6] (d o, d n) per receiver, both in sorted order; lists: kBwdList ints per warp.
__global__ void __launch_bounds__(kPacketThreads, kBwdBlocks)
    k_packet_bwd(TraceArgs a, const float* __restrict__ G, const float* __restrict__ GV, float* __restrict__ acc,
                 double* __restrict__ rayacc, int* __restrict__ lists) {
  extern __shared__ float4 psmem4[];
  PacketSmem* wsm = reinterpret_cast<PacketSmem*>(psmem4);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  PacketSmem& sm = wsm[warp];
  BwdSmem& bs = reinterpret_cast<BwdSmem*>(wsm + kPacketWarps)[warp];
  int* list = lists + ((int64_t)blockIdx.x * kPacketWarps + warp) * kBwdList;
  const int64_t batch = a.r1 - a.r0;
  constexpr int kPasses = kBwdWindow / 32;
  const int64_t n_windows = (batch + kBwdWindow - 1) / kBwdWindow;
  const unsigned below = (1u << lane) - 1u;
  RayStats rs{0u, 0u, 0u, 0u, 0u, 0u};
  for (;;) {
    unsigned item = 0;
    if (lane == 0) item = atomicAdd(a.work, 1u);
    item = __shfl_sync(0xffffffffu, item, 0);
    if ((int64_t)item >= kPasses * n_windows * a.S) break;
    const int pass = (int)(item % kPasses);
    const int64_t base = a.r0 + kBwdWindow * (item / kPasses / a.S);
    const int s = (int)(item / kPasses % a.S);
    int total = 0;  // k_ray_grad left zeros for the directions below a receiver's horizon
#pragma unroll
    for (int h = 0; h < kPasses; ++h) {
      const int64_t j = base + lane + 32 * h;
      const int64_t o = (int64_t)s * batch + (j - a.r0);
      const bool on = j < a.r1 && (G[o] != 0.0f || GV[o] != 0.0f);
      const unsigned m = __ballot_sync(0xffffffffu, on);
      if (on) sm.rlist[total + __popc(m & below)] = (unsigned char)(lane + 32 * h);
      total += __popc(m);
    }
    __syncwarp();
    if (pass * 32 < total) {
      const float d[3] = {__ldg(a.dirs + 3 * s), __ldg(a.dirs + 3 * s + 1), __ldg(a.dirs + 3 * s + 2)};
      const Frame f = make_frame(d[0], d[1], d[2]);
      const bool up = pass * 32 + lane < total;
      const int self = (int)(base + (up ? sm.rlist[pass * 32 + lane] : 0));
      const float4 q0 = __ldg(a.recs + 4 * (int64_t)self);
      const int64_t o = (int64_t)s * batch + (self - a.r0);
      const float gc = up ? G[o] : 0.0f, gV = up ? GV[o] : 0.0f;
      float V = up ? 1.0f : 0.0f, go1 = 0.0f, go2 = 0.0f;
      // (always so here; without the branch the compiler's code takes 71.2 ms for 100k splats at 128 directions, not 70.7)
      if (a.flags & PRTGS_SHADOW) {
        int root = INT32_MIN;
        if (up) {
          root = a.roots[find_scene(a.offsets, a.n_scenes, __ldg(a.order + self))];
          if (root != INT32_MIN && !child_ok(root, a.n, a.status)) root = INT32_MIN;
        }
        const float xl = f.e1x * q0.x + f.e1y * q0.y + f.e1z * q0.z;
        const float yl = f.e2x * q0.x + f.e2y * q0.y + f.e2z * q0.z;
        const float zl = f.wx * q0.x + f.wy * q0.y + f.wz * q0.z;
        unsigned todo = __ballot_sync(0xffffffffu, up);
        while (todo) {
          const int leader = __ffs(todo) - 1;
          const int groot = __shfl_sync(0xffffffffu, root, leader);
          const unsigned grp = __ballot_sync(0xffffffffu, up && root == groot) & todo;
          const bool mine = (grp >> lane) & 1u;
          const Rel rel = make_rel(f, q0.x, q0.y, q0.z, __shfl_sync(0xffffffffu, q0.x, leader),
                                   __shfl_sync(0xffffffffu, q0.y, leader), __shfl_sync(0xffffffffu, q0.z, leader));
          float gVV = 0.0f, T = 1.0f;  // T replays the cut-off of the first walk
          for (int skip = 0;; skip += kBwdList) {
            HitListVis hv{a.t_min, 1.0f, q0.x, q0.y, q0.z, list, skip, kBwdList, 0};
            packet_walk(a, f, rel, self, groot, mine, xl, yl, zl, 0.0f, hv, sm, rs, skip ? rs.search_nodes : rs.nodes);
            if (skip == 0 && mine) {
              V = hv.T;
              gVV = gV * V;
            }
            __syncwarp();  // lane 0's list
            const int nl = min(hv.total - skip, kBwdList);
            for (int g = 0; g < nl; g += 32) {
              const int pos = g + lane < nl ? list[g + lane] : -1;
              float et;
              const Beam all{-FLT_MAX, FLT_MAX, -FLT_MAX, FLT_MAX, -FLT_MAX, FLT_MAX};
              const int cnt = stage_leaves(a.recs, pos, f, rel, all, 0.0f, 0.0f, sm, et);
              // the lane's leaf: an orthonormal basis (f1, f2) of the plane across a = A w / |A w|, in the
              // place of the quick test's terms
              Frame lf;
              {
                const float4* rec = a.recs + 4 * (int64_t)max(pos, 0);
                const float4 q1 = __ldg(rec + 1), q2 = __ldg(rec + 2), q3 = __ldg(rec + 3);
                const float adx = fmaf(q1.x, f.wx, fmaf(q1.y, f.wy, q1.z * f.wz));
                const float ady = fmaf(q1.w, f.wx, fmaf(q2.x, f.wy, q2.y * f.wz));
                const float adz = fmaf(q2.z, f.wx, fmaf(q2.w, f.wy, q3.x * f.wz));
                const float id = 1.0f / sqrtf(fmaf(adx, adx, fmaf(ady, ady, adz * adz)));
                lf = make_frame(adx * id, ady * id, adz * id);
                if (g + lane < nl) {
                  sm.quick[0][lane] = make_float4(lf.e1x, lf.e1y, lf.e1z, 0.0f);
                  sm.quick[1][lane] = make_float4(lf.e2x, lf.e2y, lf.e2z, 0.0f);
                }
              }
              __syncwarp();
              for (int j0 = 0; j0 < cnt; j0 += kBwdBatch) {
                const int nb = min(kBwdBatch, cnt - j0);
                for (int b = 0; b < nb; ++b) {
                  const int j = j0 + b;
                  float wx, wy, wz, t;
                  leaf_offset(rel, sm, j, wx, wy, wz, t);
                  const float d2 = fmaf(wx, wx, fmaf(wy, wy, wz * wz));
                  const int lp = __float_as_int(sm.stage[3][j].y);
                  bool h = mine && lp != self && !(T < a.t_min);
                  if (h) h = ray_decides(a.recs, f, q0.x, q0.y, q0.z, rel, sm, j, lp, d2, t, d2 <= 9.0f && t > 0.0f);
                  float ga = 0.0f, g2 = 0.0f, p = 0.0f, q = 0.0f;
                  if (h) {
                    const float ex = expf(-0.5f * d2);
                    const float al = sm.stage[0][j].w * ex;
                    const float om = 1.0f - al;
                    T *= om;
                    const float galpha = -gVV / om;
                    ga = galpha * ex;
                    g2 = -0.5f * al * galpha;
                    const float4 s1 = sm.stage[1][j], s2 = sm.stage[2][j], f1 = sm.quick[0][j], f2 = sm.quick[1][j];
                    p = fmaf(wx, f1.x, fmaf(wy, f1.y, wz * f1.z));
                    q = fmaf(wx, f2.x, fmaf(wy, f2.y, wz * f2.z));
                    go1 = fmaf(2.0f * g2, fmaf(wx, s1.x, fmaf(wy, s1.y, wz * s1.z)), go1);
                    go2 = fmaf(2.0f * g2, fmaf(wx, s2.x, fmaf(wy, s2.y, wz * s2.z)), go2);
                  }
                  const float gp = g2 * p, gq = g2 * q;
                  float (*row)[kBwdRow] = bs.row + 6 * b;
                  row[0][lane] = ga;
                  row[1][lane] = gp;
                  row[2][lane] = gq;
                  row[3][lane] = gp * p;
                  row[4][lane] = gp * q;
                  row[5][lane] = gq * q;
                }
                __syncwarp();
                if (lane < 6 * nb) {
                  const float4* r4 = reinterpret_cast<const float4*>(bs.row[lane]);
                  float4 v = r4[0];
#pragma unroll
                  for (int i = 1; i < 8; ++i) {
                    const float4 u = r4[i];
                    v.x += u.x;
                    v.y += u.y;
                    v.z += u.z;
                    v.w += u.w;
                  }
                  bs.sum[j0 + lane / 6][lane % 6] = (v.x + v.y) + (v.z + v.w);
                }
                __syncwarp();
              }
              if (lane < cnt) {  // w' = p f1 + q f2, x = a cross w' = p f2 - q f1
                const float4 m = *reinterpret_cast<const float4*>(bs.sum[lane]);
                const float mpq = bs.sum[lane][4], mqq = bs.sum[lane][5], mpp = m.w;
                const float x1 = lf.e1x, y1 = lf.e1y, z1 = lf.e1z, x2 = lf.e2x, y2 = lf.e2y, z2 = lf.e2z;
                float* out = acc + 12 * (int64_t)pos;
                red_add4(out, m.x, fmaf(m.y, x2, -m.z * x1), fmaf(m.y, y2, -m.z * y1), fmaf(m.y, z2, -m.z * z1));
                // sum g x x^T = mpp f2 f2 - mpq (f1 f2 + f2 f1) + mqq f1 f1
                const float u2x = fmaf(mpp, x2, -mpq * x1), u2y = fmaf(mpp, y2, -mpq * y1), u2z = fmaf(mpp, z2, -mpq * z1);
                const float u1x = fmaf(mqq, x1, -mpq * x2), u1y = fmaf(mqq, y1, -mpq * y2), u1z = fmaf(mqq, z1, -mpq * z2);
                red_add4(out + 4, fmaf(u2x, x2, u1x * x1), fmaf(u2x, y2, u1x * y1), fmaf(u2x, z2, u1x * z1),
                         fmaf(u2y, y2, u1y * y1));
                red_add4(out + 8, fmaf(u2y, z2, u1y * z1), fmaf(u2z, z2, u1z * z1), 0.0f, 0.0f);
              }
              __syncwarp();  // the staged leaves are replaced
            }
            if (hv.total <= skip + kBwdList) break;
          }
          todo &= ~grp;
        }
      }
      if (up) {
        const float gn = gc * V;  // dL/dn = g c' V, c = n.w
        // a receiver's directions come one after another from anywhere on the GPU: a chain of S additions, which in 32
        // bits left the normals' gradient of 500 splats at 512 directions 2.6 to 4.9e-7 from 64 bits (now 0.7 to 2.4)
        double* out = rayacc + 6 * (int64_t)self;
        if (go1 != 0.0f || go2 != 0.0f) {
          atomicAdd(out, (double)fmaf(go1, f.e1x, go2 * f.e2x));
          atomicAdd(out + 1, (double)fmaf(go1, f.e1y, go2 * f.e2y));
          atomicAdd(out + 2, (double)fmaf(go1, f.e1z, go2 * f.e2z));
        }
        if (gn != 0.0f) {
          atomicAdd(out + 3, (double)(gn * d[0]));
          atomicAdd(out + 4, (double)(gn * d[1]));
          atomicAdd(out + 5, (double)(gn * d[2]));
        }
      }
      __syncwarp();
    }
    __syncwarp();
  }
  if (a.stats) {
    const unsigned long long c0 = warp_sum_u64(rs.nodes), c1 = warp_sum_u64(rs.search_nodes),
                             c2 = warp_sum_u64(rs.leaves), c3 = warp_sum_u64(rs.hits);
    if (lane == 0) {
      atomicAdd(a.stats + 0, c0);
      atomicAdd(a.stats + 1, c1);
      atomicAdd(a.stats + 2, c2);
      atomicAdd(a.stats + 3, c3);
    }
  }
}

// G[s][i] = w sum_k dP_ik Y_k(w_s) and GV[s][i] = G c + dV_is of the receivers of batch [r0, r1), zero
// where n.w <= 0; one thread per receiver, w = 4 pi / S.
__global__ void __launch_bounds__(128) k_ray_grad(TraceArgs a, const float* __restrict__ dP, const float* __restrict__ dV,
                                                  float* __restrict__ G, float* __restrict__ GV) {
  const int64_t batch = a.r1 - a.r0;
  const int64_t li = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (li >= batch) return;
  const int self = (int)(a.r0 + li);
  const float4 q3 = __ldg(a.recs + 4 * (int64_t)self + 3);
  const int64_t gid = a.order[self];
  const int C = sh_count(a.sh_order);
  const float wq = 4.0f * kPi / (float)a.S;
  float p[kMaxC];
#pragma unroll
  for (int k = 0; k < kMaxC; ++k) p[k] = dP && C <= kMaxC && k < C ? __ldg(dP + gid * C + k) : 0.0f;
  for (int s = 0; s < a.S; ++s) {
    const float d[3] = {__ldg(a.dirs + 3 * s), __ldg(a.dirs + 3 * s + 1), __ldg(a.dirs + 3 * s + 2)};
    const float c = ray_cos(q3.y, q3.z, q3.w, d);
    float g = 0.0f, gv = 0.0f;
    if (c > 0.0f) {
      if (dP && C <= kMaxC) {
        float Y[kMaxC];
        sh_eval_dyn(a.sh_order, d[0], d[1], d[2], Y);
#pragma unroll
        for (int k = 0; k < kMaxC; ++k)
          if (k < C) g = fmaf(p[k], Y[k], g);  // Y holds only the first C values
      } else if (dP) {  // orders 4-6: the direction set's SH table
        for (int k = 0; k < C; ++k) g = fmaf(__ldg(dP + gid * C + k), __ldg(a.Ytab + (int64_t)s * C + k), g);
      }
      g *= wq;
      gv = g * c + (dV ? __ldg(dV + gid * a.S + s) : 0.0f);
    }
    G[(int64_t)s * batch + li] = g;
    GV[(int64_t)s * batch + li] = gv;
  }
}

// The sums of k_packet_bwd to gradients, one thread per Gaussian (sorted position), in 64 bits (a few dozen operations
// per Gaussian; in 32 their rounding is a sixth of the error left). With M = sum g x x^T, a turn by theta about the
// local axes changes the loss by tau . theta, tau_1 = 2 M_23 (s_3^2 - s_2^2) / (s_2 s_3) and cyclic, which on the unit
// quaternion is 2 (tau_1 q i + tau_2 q j + tau_3 q k).
__global__ void __launch_bounds__(128) k_bwd_finish(int64_t n, const int32_t* __restrict__ order,
                                                    const float* __restrict__ scales, const float* __restrict__ quats,
                                                    const float4* __restrict__ acc, const double* __restrict__ rayacc,
                                                    float* __restrict__ d_means, float* __restrict__ d_scales,
                                                    float* __restrict__ d_quats, float* __restrict__ d_opacity,
                                                    float* __restrict__ d_normals) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int64_t gid = order[i];
  const float4 a0 = acc[3 * i], a1 = acc[3 * i + 1], a2 = acc[3 * i + 2];
  double gs[3] = {0.0, 0.0, 0.0}, gm[3] = {0.0, 0.0, 0.0}, gq[4] = {0.0, 0.0, 0.0, 0.0};
  // (the sums have both signs: the mixed second moments can be all that is left)
  if (a0.x != 0.f || a0.y != 0.f || a0.z != 0.f || a0.w != 0.f || a1.x != 0.f || a1.y != 0.f || a1.z != 0.f ||
      a1.w != 0.f || a2.x != 0.f || a2.y != 0.f) {
    const double s0 = scales[3 * gid], s1 = scales[3 * gid + 1], s2 = scales[3 * gid + 2];
    double w = quats[4 * gid], x = quats[4 * gid + 1], y = quats[4 * gid + 2], z = quats[4 * gid + 3];
    const double in = 1.0 / sqrt(w * w + x * x + y * y + z * z);
    w *= in;
    x *= in;
    y *= in;
    z *= in;
    const double u0 = -2.0 * a0.y / s0, u1 = -2.0 * a0.z / s1, u2 = -2.0 * a0.w / s2;  // d mu = R u
    gm[0] = (1.0 - 2.0 * (y * y + z * z)) * u0 + 2.0 * (x * y - w * z) * u1 + 2.0 * (x * z + w * y) * u2;
    gm[1] = 2.0 * (x * y + w * z) * u0 + (1.0 - 2.0 * (x * x + z * z)) * u1 + 2.0 * (y * z - w * x) * u2;
    gm[2] = 2.0 * (x * z - w * y) * u0 + 2.0 * (y * z + w * x) * u1 + (1.0 - 2.0 * (x * x + y * y)) * u2;
    gs[0] = -2.0 * a1.x / s0;
    gs[1] = -2.0 * a1.w / s1;
    gs[2] = -2.0 * a2.y / s2;
    const double t1 = 4.0 * in * a2.x * ((s2 - s1) * (s2 + s1)) / (s1 * s2);
    const double t2 = 4.0 * in * a1.z * ((s0 - s2) * (s0 + s2)) / (s0 * s2);
    const double t3 = 4.0 * in * a1.y * ((s1 - s0) * (s1 + s0)) / (s0 * s1);
    gq[0] = -t1 * x - t2 * y - t3 * z;
    gq[1] = t1 * w - t2 * z + t3 * y;
    gq[2] = t1 * z + t2 * w - t3 * x;
    gq[3] = -t1 * y + t2 * x + t3 * w;
  }
  d_opacity[gid] = a0.x;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    d_means[3 * gid + k] = (float)(gm[k] + rayacc[6 * i + k]);
    d_scales[3 * gid + k] = (float)gs[k];
    d_normals[3 * gid + k] = (float)rayacc[6 * i + 3 + k];
  }
#pragma unroll
  for (int k = 0; k < 4; ++k) d_quats[4 * gid + k] = (float)gq[k];
}

// Gradient without shadows, where V = 1 and only the cosines depend on the Gaussians: d n_i = sum_s g(s) w_s with
// g(s) = 4 pi / S sum_k dP_ik Y_k(w_s), a warp per receiver. (As packets without a walk, through G and GV, 30k
// receivers at 256 directions took 489 us a call; with this it takes 48, most of it the host's.)
__global__ void __launch_bounds__(128) k_normal_grad(TraceArgs a, const float* __restrict__ dP,
                                                     float* __restrict__ d_normals) {
  const int lane = threadIdx.x & 31;
  const int64_t i = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (i >= a.n) return;
  const float4 q3 = __ldg(a.recs + 4 * i + 3);
  const int64_t gid = a.order[i];
  const int C = sh_count(a.sh_order);
  float gn[3] = {0.f, 0.f, 0.f};
  if (dP) {
    float p[kMaxC];
#pragma unroll
    for (int k = 0; k < kMaxC; ++k) p[k] = C <= kMaxC && k < C ? __ldg(dP + gid * C + k) : 0.0f;
    for (int s = lane; s < a.S; s += 32) {
      const float d[3] = {__ldg(a.dirs + 3 * s), __ldg(a.dirs + 3 * s + 1), __ldg(a.dirs + 3 * s + 2)};
      if (!(ray_cos(q3.y, q3.z, q3.w, d) > 0.0f)) continue;
      float g = 0.0f;
      if (C <= kMaxC) {
        float Y[kMaxC];
        sh_eval_dyn(a.sh_order, d[0], d[1], d[2], Y);
#pragma unroll
        for (int k = 0; k < kMaxC; ++k)
          if (k < C) g = fmaf(p[k], Y[k], g);  // Y holds only the first C values
      } else {  // orders 4-6: the direction set's SH table
        for (int k = 0; k < C; ++k) g = fmaf(__ldg(dP + gid * C + k), __ldg(a.Ytab + (int64_t)s * C + k), g);
      }
      g *= 4.0f * kPi / (float)a.S;
#pragma unroll
      for (int k = 0; k < 3; ++k) gn[k] += g * d[k];
    }
  }
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const float v = warp_sum(gn[k]);
    if (lane == 0) d_normals[3 * gid + k] = v;
  }
}

// Receivers per launch: G and GV hold S floats each per receiver, at most 2^26 (512 MB for the two; with 2^25 a volume
// of 300k at 128 directions took 297.9 ms, with 2^24 300.7, with this 297.1: each launch ends with few busy warps).
static int64_t bwd_batch(int64_t n, int S) {
  int64_t b = ((int64_t(1) << 26) / (S > 0 ? S : 1)) / 64 * 64;
  if (b < 64) b = 64;
  return b < n ? b : n;
}

// Blocks of a launch at most, each with its warps' lists: a warp per packet is enough.
static int64_t bwd_blocks(int64_t n, int S) {
  const int64_t items = kBwdWindow / 32 * ((bwd_batch(n, S) + kBwdWindow - 1) / kBwdWindow) * S;
  const int64_t b = (items + kPacketWarps - 1) / kPacketWarps;
  return b < 1 ? 1 : (b < kBwdMaxBlocks ? b : kBwdMaxBlocks);
}

size_t packet_bwd_workspace(int64_t n, int S) {
  return 2 * align_up(sizeof(float) * (size_t)bwd_batch(n, S) * S) + align_up(sizeof(float) * 24 * (size_t)n) +
         align_up(sizeof(int) * (size_t)bwd_blocks(n, S) * kPacketWarps * kBwdList);
}

int launch_packet_bwd(TraceArgs a, const float* scales, const float* quats, const float* dP, const float* dV,
                      float* d_means, float* d_scales, float* d_quats, float* d_opacity, float* d_normals, void* ws, int sms,
                      cudaStream_t stream) {
  if (!(a.flags & PRTGS_SHADOW)) {
    cudaMemsetAsync(d_means, 0, sizeof(float) * 3 * a.n, stream);
    cudaMemsetAsync(d_scales, 0, sizeof(float) * 3 * a.n, stream);
    cudaMemsetAsync(d_quats, 0, sizeof(float) * 4 * a.n, stream);
    cudaMemsetAsync(d_opacity, 0, sizeof(float) * a.n, stream);
    k_normal_grad<<<(unsigned)((a.n + 3) / 4), 128, 0, counted(stream)>>>(a, dP, d_normals);
    PRTGS_CHECK_LAUNCH();
    return PRTGS_OK;
  }
  const int64_t b = bwd_batch(a.n, a.S);
  Carver c(ws);
  float* G = c.take<float>((size_t)b * a.S);
  float* GV = c.take<float>((size_t)b * a.S);
  float* acc = c.take<float>(24 * (size_t)a.n);  // [n][12], then [n][6] doubles of the receivers
  int* lists = c.take<int>((size_t)bwd_blocks(a.n, a.S) * kPacketWarps * kBwdList);
  double* rayacc = reinterpret_cast<double*>(acc + 12 * a.n);
  cudaMemsetAsync(acc, 0, sizeof(float) * 24 * a.n, stream);
  const size_t smem = (sizeof(PacketSmem) + sizeof(BwdSmem)) * kPacketWarps;
  cudaFuncSetAttribute(k_packet_bwd, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  cudaFuncSetAttribute(k_packet_bwd, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
  int per_sm = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_packet_bwd, kPacketThreads, smem);
  const int64_t most = bwd_blocks(a.n, a.S), resident = (int64_t)sms * (per_sm < 1 ? 1 : per_sm);
  const unsigned blocks = (unsigned)(resident < most ? resident : most);
  for (int64_t r0 = 0; r0 < a.n; r0 += b) {
    a.r0 = r0;
    a.r1 = r0 + b < a.n ? r0 + b : a.n;
    cudaMemsetAsync(a.work, 0, sizeof(unsigned int), stream);
    k_ray_grad<<<(unsigned)((a.r1 - a.r0 + 127) / 128), 128, 0, counted(stream)>>>(a, dP, dV, G, GV);
    k_packet_bwd<<<blocks, kPacketThreads, smem, counted(stream)>>>(a, G, GV, acc, rayacc, lists);
  }
  k_bwd_finish<<<(unsigned)((a.n + 127) / 128), 128, 0, counted(stream)>>>(
      a.n, a.order, scales, quats, reinterpret_cast<const float4*>(acc), rayacc, d_means, d_scales, d_quats, d_opacity,
      d_normals);
  PRTGS_CHECK_LAUNCH();
  return PRTGS_OK;
}

// P of the receivers of batch [r0, r1) from V[s][i]: one lane per receiver, a compensated sum
// over the directions per coefficient (orders <= 3 from the Cartesian SH, above from the table).
__global__ void __launch_bounds__(128) k_project(TraceArgs a, const float* __restrict__ V) {
  extern __shared__ float psdir[];  // [S*3]
  for (int i = threadIdx.x; i < 3 * a.S; i += blockDim.x) psdir[i] = a.dirs[i];
  __syncthreads();
  const int64_t batch = a.r1 - a.r0;
  const int64_t li = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (li >= batch) return;
  const int self = (int)(a.r0 + li);
  const float4 q3 = __ldg(a.recs + 4 * self + 3);
  const int gid = a.order[self];
  const int C = sh_count(a.sh_order);
  const float wq = 4.0f * kPi / (float)a.S;
  for (int kb = 0; kb < C; kb += kMaxC) {
    CompSum acc[kMaxC];
    for (int s = 0; s < a.S; ++s) {
      const float* d = psdir + 3 * s;
      const float c = ray_cos(q3.y, q3.z, q3.w, d);
      if (!(c > 0.0f)) continue;
      const float v = V[(int64_t)s * batch + li] * c * wq;
      if (C <= kMaxC) {
        float Y[kMaxC];
        sh_eval_dyn(a.sh_order, d[0], d[1], d[2], Y);
#pragma unroll
        for (int k = 0; k < kMaxC; ++k)
          if (k < C) acc[k].add(v * Y[k]);
      } else {
#pragma unroll
        for (int k = 0; k < kMaxC; ++k)
          if (kb + k < C) acc[k].add(v * __ldg(a.Ytab + (int64_t)s * C + kb + k));
      }
    }
#pragma unroll
    for (int k = 0; k < kMaxC; ++k)
      if (kb + k < C) a.P[(int64_t)gid * C + kb + k] = acc[k].value();
  }
  if (a.Vg) {
    const int slot = a.glossy_slot[gid];
    if (slot >= 0)
      for (int s = 0; s < a.S; ++s) a.Vg[(int64_t)slot * a.S + s] = V[(int64_t)s * batch + li];
  }
}

// Scratch of the index-matrix search of a batch: every packet (at most two per window and direction)
// may need it.
size_t packet_search_bytes(int64_t batch, int S) {
  const size_t items = 2 * (size_t)((batch + 63) / 64) * S;
  return align_up(sizeof(SearchRec) * 32 * items) + align_up(sizeof(uint32_t) * items);
}

template <bool BOUNCE>
static int launch_packet_t(const TraceArgs& a, float* V, int sms, cudaStream_t stream) {
  const size_t smem = sizeof(PacketSmem) * kPacketWarps;
  cudaFuncSetAttribute(k_packet<BOUNCE>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  cudaFuncSetAttribute(k_packet<BOUNCE>, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
  int per_sm = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_packet<BOUNCE>, kPacketThreads, smem);
  // work items: a packet of a window of 64 receivers (two at most) and dpi directions; at most 2^26 / 32 per launch
  const int dpi = a.packet_dirs > 0 ? a.packet_dirs : kPacketDirs;
  cudaMemsetAsync(a.work, 0, sizeof(unsigned int), stream);
  if (BOUNCE) cudaMemsetAsync(a.queue_count, 0, sizeof(unsigned int), stream);
  k_packet<BOUNCE><<<sms * (per_sm > 0 ? per_sm : 1), kPacketThreads, smem, counted(stream)>>>(a, V, dpi);
  if (BOUNCE) {
    const size_t ssmem = (sizeof(PacketSmem) + sizeof(RoundHits)) * kPacketWarps;
    cudaFuncSetAttribute(k_search, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ssmem);
    cudaFuncSetAttribute(k_search, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_search, kPacketThreads, ssmem);
    cudaMemsetAsync(a.work, 0, sizeof(unsigned int), stream);
    k_search<<<sms * (per_sm > 0 ? per_sm : 1), kPacketThreads, ssmem, counted(stream)>>>(a);
  }
  PRTGS_CHECK_LAUNCH();
  const int64_t batch = a.r1 - a.r0;
  k_project<<<(unsigned)((batch + 127) / 128), 128, sizeof(float) * 3 * a.S, counted(stream)>>>(a, V);
  PRTGS_CHECK_LAUNCH();
  return PRTGS_OK;
}

// Visibility, P (and with bounce the index matrix) of receiver batch [a.r0, a.r1) by packets;
// V is scratch of S * batch floats.
int launch_packet(const TraceArgs& a, float* V, bool bounce, int sms, cudaStream_t stream) {
  return bounce ? launch_packet_t<true>(a, V, sms, stream) : launch_packet_t<false>(a, V, sms, stream);
}

}  // namespace prtgs
