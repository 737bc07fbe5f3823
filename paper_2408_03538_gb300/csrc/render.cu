// Tile-binned splat rasteriser (Sec. 3.1: Eq. 2 covariance, Eq. 3 EWA projection, Eq. 4
// front-to-back alpha blending) with the 3DGS conventions the paper builds on, and its
// backward pass.
//
// Forward: k_preprocess (one thread per Gaussian) -> the Gaussians in depth order (radix sort of the depth
// bits) -> inclusive scan of the touched-tile counts in that order -> k_duplicate writes (tile, Gaussian)
// pairs -> stable radix sort by tile, on the device-side pair count -> k_ranges -> k_composite (two blocks per
// 16x16-pixel tile, a warp per 8x4 pixels that stages the splats that reach them, evaluated once for a group of up to
// 16 light colour sets).
// Backward: k_composite_bwd walks each pixel's list back to front from its last contributor and sums
// every splat's moments and colour gradients over a warp's pixels before a few vector reductions;
// k_preprocess_bwd maps the sums to opacities, colours, means, scales and rotations.
#include "blend.cuh"
#include "common.cuh"
#include "internal.h"

namespace prtgs {

constexpr int kTile = 16;
constexpr int kTileThreads = kTile * kTile;
// Blocks of a tile's eight warps: its warps end at different times, and a block keeps its place until the last
// has. Composite of 300k splats at 1080p, forward and backward, at 1, 2, 4 and 8: 228, 221, 224, 239 and 463, 449, 457,
// 466 us; of 8 scenes x 4 lights 596, 570, 579, 594 and 2,150, 1,244, 1,535, 1,612 (the backward's register bounds being
// those for two).
constexpr int kSplit = 2;
constexpr int kCompThreads = kTileThreads / kSplit;
constexpr float kNear = 0.2f;
constexpr float kDilation = 0.3f;
constexpr float kAlphaMax = 0.99f;
constexpr float kAlphaMin = 1.0f / 255.0f;
constexpr float kTStop = 1e-4f;

struct Cam {
  float r[9], t[3];
  float fx, fy, cx, cy;
  int W, H, gx, gy;
  float near_plane;
  float limx, limy;
};

static Cam make_cam(const prtgs_camera* c) {
  Cam k;
  for (int i = 0; i < 9; ++i) k.r[i] = c->rot[i];
  for (int i = 0; i < 3; ++i) k.t[i] = c->trans[i];
  k.fx = c->fx; k.fy = c->fy; k.cx = c->cx; k.cy = c->cy;
  k.W = c->width; k.H = c->height;
  k.gx = (c->width + kTile - 1) / kTile;
  k.gy = (c->height + kTile - 1) / kTile;
  k.near_plane = c->near_plane > 0.f ? c->near_plane : kNear;
  k.limx = 1.3f * (0.5f * (float)c->width / c->fx);
  k.limy = 1.3f * (0.5f * (float)c->height / c->fy);
  return k;
}

// Where each Gaussian's camera, colours and image live. OneView: a single scene (colours
// [k][n][3], image [k][3][H][W]). ManyViews: scene b holds Gaussians offs[b] .. offs[b+1], has its
// own camera (every camera has the same image size), its colours are the [k][n_b][3] block at
// 3 k offs[b] (the layout of prtgs_relight_batched) and its images the [k][3][H][W] block b. The
// cameras travel by value in the kernel parameters (no device copy, graph-capturable).
struct OneView {
  static constexpr bool kRows = false;
  Cam c;
  __device__ __forceinline__ int scene_of(int64_t) const { return 0; }
  __device__ __forceinline__ const Cam& cam(int) const { return c; }
  __device__ __forceinline__ int64_t first(int) const { return 0; }
  __device__ __forceinline__ int64_t count(int, int64_t n) const { return n; }
};

struct ManyViews {
  static constexpr bool kRows = false;
  Cam c[kMaxScenes];
  const int64_t* offs;
  int B;
  __device__ __forceinline__ int scene_of(int64_t i) const { return find_scene(offs, B, i); }
  __device__ __forceinline__ const Cam& cam(int b) const { return c[b]; }
  __device__ __forceinline__ int64_t first(int b) const { return offs[b]; }
  __device__ __forceinline__ int64_t count(int b, int64_t) const { return offs[b + 1] - offs[b]; }
};

// A view with the colours as rows [n][color_floats(k)]: one splat's sets side by side.
template <class V>
struct Rows : V {
  static constexpr bool kRows = true;
};

// Colour of light l, channel ch of Gaussian g (in scene b).
template <class V>
__device__ __forceinline__ int64_t color_at(const V& v, int b, int64_t g, int l, int k, int64_t n) {
  const int64_t o = v.first(b);
  return 3 * (int64_t)k * o + ((int64_t)l * v.count(b, n) + (g - o)) * 3;
}

size_t render_state_bytes(int64_t n, int32_t width, int32_t height, int64_t max_pairs) {
  return render_state_bytes_batched(n, 1, width, height, max_pairs);
}

int render_state_layout(void* buffer, int64_t n, int32_t width, int32_t height, int64_t max_pairs,
                        prtgs_render_state* out) {
  return render_state_layout_batched(buffer, n, 1, width, height, max_pairs, out);
}

// B scenes of one image size: tile ranges, final transmittance and contributor counts per scene.
size_t render_state_bytes_batched(int64_t n, int32_t B, int32_t width, int32_t height, int64_t max_pairs) {
  int64_t tiles = (int64_t)((width + kTile - 1) / kTile) * ((height + kTile - 1) / kTile) * B;
  int64_t px = (int64_t)width * height * B;
  return align_up(sizeof(float) * 2 * n) + align_up(sizeof(float) * 4 * n) + align_up(sizeof(float) * n) +
         align_up(sizeof(int32_t) * n) + align_up(sizeof(uint32_t) * n) + align_up(sizeof(uint64_t) * max_pairs) +
         align_up(sizeof(int32_t) * max_pairs) + align_up(sizeof(uint32_t) * 2 * tiles) +
         align_up(sizeof(float) * px) + align_up(sizeof(int32_t) * px) + align_up(sizeof(uint32_t));
}

int render_state_layout_batched(void* buffer, int64_t n, int32_t B, int32_t width, int32_t height,
                                int64_t max_pairs, prtgs_render_state* out) {
  int64_t tiles = (int64_t)((width + kTile - 1) / kTile) * ((height + kTile - 1) / kTile) * B;
  int64_t px = (int64_t)width * height * B;
  Carver c(buffer);
  out->n_scenes = B;
  out->n = n;
  out->max_pairs = max_pairs;
  out->width = width;
  out->height = height;
  out->tiles_x = (width + kTile - 1) / kTile;
  out->tiles_y = (height + kTile - 1) / kTile;
  out->mean2d = c.take<float>(2 * n);
  out->conic_op = c.take<float>(4 * n);
  out->depth = c.take<float>(n);
  out->radius = c.take<int32_t>(n);
  out->tiles_touched = c.take<uint32_t>(n);
  out->pair_keys = c.take<uint64_t>(max_pairs);
  out->pair_ids = c.take<int32_t>(max_pairs);
  out->ranges = c.take<uint32_t>(2 * tiles);
  out->final_T = c.take<float>(px);
  out->n_contrib = c.take<int32_t>(px);
  out->n_pairs = c.take<uint32_t>(1);
  return PRTGS_OK;
}

size_t render_workspace(int64_t n, int32_t, int32_t, int64_t max_pairs) {
  return scan_workspace(n) + 6 * align_up(sizeof(uint32_t) * n) + 5 * align_up(sizeof(uint32_t) * max_pairs) +
         radix_sort_workspace(max_pairs > n ? max_pairs : n);
}

__device__ __forceinline__ void quat_rot(float qw, float qx, float qy, float qz, float R[3][3]) {
  float n = rsqrtf(qw * qw + qx * qx + qy * qy + qz * qz);
  qw *= n; qx *= n; qy *= n; qz *= n;
  R[0][0] = 1.f - 2.f * (qy * qy + qz * qz); R[0][1] = 2.f * (qx * qy - qw * qz); R[0][2] = 2.f * (qx * qz + qw * qy);
  R[1][0] = 2.f * (qx * qy + qw * qz); R[1][1] = 1.f - 2.f * (qx * qx + qz * qz); R[1][2] = 2.f * (qy * qz - qw * qx);
  R[2][0] = 2.f * (qx * qz - qw * qy); R[2][1] = 2.f * (qy * qz + qw * qx); R[2][2] = 1.f - 2.f * (qx * qx + qy * qy);
}

// Sigma = R diag(s^2) R^T (Eq. 2), upper triangle (00, 01, 02, 11, 12, 22).
__device__ __forceinline__ void covariance3d(const float R[3][3], float s0, float s1, float s2, float S[6]) {
  float d[3] = {s0 * s0, s1 * s1, s2 * s2};
  S[0] = R[0][0] * R[0][0] * d[0] + R[0][1] * R[0][1] * d[1] + R[0][2] * R[0][2] * d[2];
  S[1] = R[0][0] * R[1][0] * d[0] + R[0][1] * R[1][1] * d[1] + R[0][2] * R[1][2] * d[2];
  S[2] = R[0][0] * R[2][0] * d[0] + R[0][1] * R[2][1] * d[1] + R[0][2] * R[2][2] * d[2];
  S[3] = R[1][0] * R[1][0] * d[0] + R[1][1] * R[1][1] * d[1] + R[1][2] * R[1][2] * d[2];
  S[4] = R[1][0] * R[2][0] * d[0] + R[1][1] * R[2][1] * d[1] + R[1][2] * R[2][2] * d[2];
  S[5] = R[2][0] * R[2][0] * d[0] + R[2][1] * R[2][1] * d[1] + R[2][2] * R[2][2] * d[2];
}

__device__ __forceinline__ void tile_rect(float mx, float my, int r, const Cam& c, int& x0, int& y0, int& x1,
                                          int& y1) {
  const float fr = (float)r;
  x0 = min(max((int)floorf((mx - fr) / kTile), 0), c.gx);
  x1 = min(max((int)floorf((mx + fr) / kTile) + 1, 0), c.gx);
  y0 = min(max((int)floorf((my - fr) / kTile), 0), c.gy);
  y1 = min(max((int)floorf((my + fr) / kTile) + 1, 0), c.gy);
}

template <class V>
__global__ void k_preprocess(int64_t n, const float* __restrict__ means, const float* __restrict__ scales,
                             const float* __restrict__ quats, const float* __restrict__ opacity, V v,
                             float* __restrict__ mean2d, float4* __restrict__ conic_op, float* __restrict__ depth,
                             int32_t* __restrict__ radius, uint32_t* __restrict__ touched,
                             uint32_t* __restrict__ depth_key) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const Cam& c = v.cam(v.scene_of(i));
  radius[i] = 0;
  touched[i] = 0;
  depth_key[i] = 0xffffffffu;  // behind every visible splat
  const float mx = means[3 * i], my = means[3 * i + 1], mz = means[3 * i + 2];
  const float x = c.r[0] * mx + c.r[1] * my + c.r[2] * mz + c.t[0];
  const float y = c.r[3] * mx + c.r[4] * my + c.r[5] * mz + c.t[1];
  const float z = c.r[6] * mx + c.r[7] * my + c.r[8] * mz + c.t[2];
  depth[i] = z;
  if (!(z > c.near_plane)) return;
  float R[3][3];
  quat_rot(quats[4 * i], quats[4 * i + 1], quats[4 * i + 2], quats[4 * i + 3], R);
  float S[6];
  covariance3d(R, scales[3 * i], scales[3 * i + 1], scales[3 * i + 2], S);
  const float iz = 1.0f / z;
  const float tx = fminf(c.limx, fmaxf(-c.limx, x * iz)) * z;
  const float ty = fminf(c.limy, fmaxf(-c.limy, y * iz)) * z;
  // J (2x3) = [[fx/z, 0, -fx tx/z^2], [0, fy/z, -fy ty/z^2]]; M = J W
  const float j00 = c.fx * iz, j02 = -c.fx * tx * iz * iz, j11 = c.fy * iz, j12 = -c.fy * ty * iz * iz;
  float m0[3], m1[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    m0[k] = j00 * c.r[k] + j02 * c.r[6 + k];
    m1[k] = j11 * c.r[3 + k] + j12 * c.r[6 + k];
  }
  // cov2 = M Sigma M^T
  float s0[3] = {S[0] * m0[0] + S[1] * m0[1] + S[2] * m0[2], S[1] * m0[0] + S[3] * m0[1] + S[4] * m0[2],
                 S[2] * m0[0] + S[4] * m0[1] + S[5] * m0[2]};
  float s1[3] = {S[0] * m1[0] + S[1] * m1[1] + S[2] * m1[2], S[1] * m1[0] + S[3] * m1[1] + S[4] * m1[2],
                 S[2] * m1[0] + S[4] * m1[1] + S[5] * m1[2]};
  const float a = m0[0] * s0[0] + m0[1] * s0[1] + m0[2] * s0[2] + kDilation;
  const float b = m0[0] * s1[0] + m0[1] * s1[1] + m0[2] * s1[2];
  const float cc = m1[0] * s1[0] + m1[1] * s1[1] + m1[2] * s1[2] + kDilation;
  const float det = a * cc - b * b;
  if (!(det > 0.f)) return;
  const float idet = 1.0f / det;
  const float mid = 0.5f * (a + cc);
  const float lam = mid + sqrtf(fmaxf(0.1f, mid * mid - det));
  const int r = (int)ceilf(3.0f * sqrtf(lam));
  const float px = c.fx * x * iz + c.cx, py = c.fy * y * iz + c.cy;
  int x0, y0, x1, y1;
  tile_rect(px, py, r, c, x0, y0, x1, y1);
  const uint32_t cnt = (uint32_t)((x1 - x0) * (y1 - y0));
  if (r <= 0 || cnt == 0) return;
  mean2d[2 * i] = px;
  mean2d[2 * i + 1] = py;
  conic_op[i] = make_float4(cc * idet, -b * idet, a * idet, opacity[i]);
  radius[i] = r;
  touched[i] = cnt;
  depth_key[i] = __float_as_uint(z);  // z > 0: the bits order as the depths
}

// (tile, Gaussian) pairs in depth order: a warp takes 32 splats of that order and writes their pairs, the
// lanes on consecutive pairs (each finds its splat in the warp's prefix sums), so that the writes coalesce and a
// splat of many tiles does not hold the others up. (A thread per splat took 0.54 ms for the 25 M pairs of 300k
// splats; this takes 0.075.)
template <class V>
__global__ void __launch_bounds__(256) k_duplicate(int64_t n, V v, const int32_t* __restrict__ by_depth,
                                                   const float* __restrict__ mean2d, const int32_t* __restrict__ radius,
                                                   const uint32_t* __restrict__ incl, int64_t max_pairs,
                                                   uint32_t* __restrict__ tiles, int32_t* __restrict__ ids,
                                                   int32_t* status) {
  const int lane = threadIdx.x & 31;
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  int g = 0, x0 = 0, y0 = 0, w = 1, count = 0;
  uint32_t tile0 = 0;
  if (i < n) {
    g = by_depth[i];
    const int r = radius[g];
    if (r > 0) {
      const int b = v.scene_of(g);
      const Cam& c = v.cam(b);
      int x1, y1;
      tile_rect(mean2d[2 * (int64_t)g], mean2d[2 * (int64_t)g + 1], r, c, x0, y0, x1, y1);
      w = x1 - x0;
      count = w * (y1 - y0);
      tile0 = (uint32_t)(b * (c.gx * c.gy) + y0 * c.gx + x0);  // the splat's first tile
      if ((int64_t)incl[i] > max_pairs) set_status(status, PRTGS_STATUS_CAPACITY);
    }
  }
  const int gx = v.cam(0).gx;
  int end = count;  // inclusive prefix sum over the warp
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, end, off);
    if (lane >= off) end += y;
  }
  const int total = __shfl_sync(0xffffffffu, end, 31);
  if (total == 0) return;
  const int64_t first = (int64_t)__shfl_sync(0xffffffffu, i < n ? incl[i] : 0u, 0) - __shfl_sync(0xffffffffu, count, 0);
  for (int base = 0; base < total; base += 32) {
    const int p = base + lane;
    int o = 0;  // the first lane whose prefix sum is above p
#pragma unroll
    for (int step = 16; step > 0; step >>= 1)
      if (__shfl_sync(0xffffffffu, end, o + step - 1) <= p) o += step;
    o = min(o, 31);
    const int og = __shfl_sync(0xffffffffu, g, o), ow = __shfl_sync(0xffffffffu, w, o);
    const uint32_t ot = __shfl_sync(0xffffffffu, tile0, o);
    const int k = p - __shfl_sync(0xffffffffu, end - count, o);
    if (p < total && first + p < max_pairs) {
      tiles[first + p] = ot + (uint32_t)((k / ow) * gx + k % ow);
      ids[first + p] = og;
    }
  }
}

// First of the n sorted pairs whose tile is at least `tile`, by a warp: each round cuts the range into 32.
__device__ __forceinline__ int64_t first_pair(const uint64_t* __restrict__ keys, int64_t n, uint64_t tile) {
  const int lane = threadIdx.x & 31;
  int64_t lo = 0, hi = n;
  while (lo < hi) {
    const int64_t step = (hi - lo + 31) / 32, at = lo + lane * step;
    const bool below = at < hi && (__ldg(keys + min(at + step, hi) - 1) >> 32) < tile;  // the whole part lies in front
    lo = min(hi, lo + __popc(__ballot_sync(0xffffffffu, below)) * step);
    hi = min(hi, lo + step - 1);
  }
  return lo;
}

// Tile ranges of the sorted pairs, a warp per tile (empty tiles: 0, 0). A pass over all pairs that compared
// neighbours and wrote their 64-bit keys took 165 us for 25 M pairs; the sort's last pass writes those now.
__global__ void __launch_bounds__(256) k_ranges(const uint64_t* __restrict__ keys, const uint32_t* __restrict__ count,
                                                int64_t tiles, uint32_t* __restrict__ ranges) {
  const int64_t tile = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (tile >= tiles) return;
  const int64_t n = *count;
  const int64_t lo = first_pair(keys, n, (uint64_t)tile);
  const int64_t hi = first_pair(keys, n, (uint64_t)tile + 1);
  if ((threadIdx.x & 31) == 0) {
    ranges[2 * tile] = lo < hi ? (uint32_t)lo : 0u;
    ranges[2 * tile + 1] = lo < hi ? (uint32_t)hi : 0u;
  }
}

// Whether a splat can have alpha >= 1/255 at any pixel centre of [x0, x1] x [y0, y1]: the smallest value of its
// form f = a dx^2 + 2 b dx dy + c dy^2 over that rectangle against K = 2 ln(255 opacity). f is convex, so the
// minimum is 0 at the centre if the rectangle holds it, else it lies on one of the sides that face the centre, where
// f is a parabola. The margins lie beyond the rounding of this test and of the alphas themselves (both some ulp of
// f's terms). NaNs and a form that is not positive beyond its rounding keep the splat. (Against the ellipse's
// bounding box, which keeps a quarter more: 8 lights of 100k splats 475 -> 423 us, the geometry maps 450 -> 392, the
// backward of 8 scenes 1,745 -> 1,644.)
__device__ __forceinline__ bool reaches(float mx, float my, const float4& co, float x0, float x1, float y0, float y1) {
  const float K = fmaf(2.002f, __logf(255.0f * co.w), 0.01f);
  if (K < 0.0f) return false;
  const float ac = co.x * co.z, bb = co.y * co.y;
  if (!((ac - bb) - 1e-6f * (ac + bb) > 0.0f)) return true;
  const float xl = x0 - mx, xh = x1 - mx, yl = y0 - my, yh = y1 - my;
  const float dx = fminf(fmaxf(0.0f, xl), xh), dy = fminf(fmaxf(0.0f, yl), yh);  // the point nearest to the centre
  const float ys = fminf(fmaxf(__fdividef(-co.y * dx, co.z), yl), yh);           // ... the smallest f on its column
  const float xs = fminf(fmaxf(__fdividef(-co.y * dy, co.x), xl), xh);           // ... and on its row
  const float ax = co.x * dx * dx, cx = co.z * ys * ys, bx = 2.0f * co.y * dx * ys;
  const float ay = co.x * xs * xs, cy = co.z * dy * dy, by = 2.0f * co.y * xs * dy;
  const float fx = (ax + cx + bx) - 1e-5f * (ax + cx), fy = (ay + cy + by) - 1e-5f * (ay + cy);
  return !(fx > K) || !(fy > K);
}

// The colours of k >= 2 sets as rows. A warp's 32 splats lie anywhere, so from [k][n][3] each of their sets is a
// sector of its own, read a word at a time; from rows it is 16-byte words of a few lines. 8 lights of 100k splats:
// composite 423 us from [k][n][3], 370 from rows, which take 7 to write; the backward of 8 scenes x 4 lights 1,644
// and 1,394 us.
template <class V>
__global__ void __launch_bounds__(256) k_color_rows(int64_t n, V v, const float* __restrict__ colors, int k,
                                                    float4* __restrict__ rows) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int b = v.scene_of(i);
  const int q = color_floats(k) / 4;
  for (int j = 0; j < q; ++j) {
    float f[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int l = (4 * j + e) / 3, ch = (4 * j + e) % 3;
      f[e] = l < k ? __ldg(colors + color_at(v, b, i, l, k, n) + ch) : 0.f;
    }
    rows[i * q + j] = make_float4(f[0], f[1], f[2], f[3]);
  }
}

template <class V>
static Rows<V> rows_of(const V& v) {
  Rows<V> r;
  static_cast<V&>(r) = v;
  return r;
}

// Per-warp staging of k_composite: 32 splats and their colours.
template <int KG>
struct FwdWarp {
  float4 co[32];
  float4 xy[32];  // mean2d, Gaussian, position in the tile's list (bits)
  float col[32][color_floats(KG)];
};

// The colour sets l0 .. l0 + KG of nk staged splats (xy.z: the Gaussian) from rows: consecutive lanes on a row's
// 16-byte words; past the row's end, zeros.
template <int KG>
__device__ __forceinline__ void stage_rows(float (*col)[color_floats(KG)], const float4* xy, int nk,
                                           const float* __restrict__ rows, int l0, int k) {
  constexpr int Q = color_floats(KG) / 4;
  const int stride = color_floats(k) / 4, q0 = 3 * l0 / 4;
  for (int e = threadIdx.x & 31; e < nk * Q; e += 32) {
    const int slot = e / Q, q = e % Q;
    reinterpret_cast<float4*>(col[slot])[q] =
        q0 + q < stride ? __ldg(reinterpret_cast<const float4*>(rows) + (int64_t)__float_as_int(xy[slot].z) * stride + q0 + q)
                        : make_float4(0.f, 0.f, 0.f, 0.f);
  }
}

// One warp per 8 x 4 pixels of a tile, on its own (no block barrier), for a group of KG colour sets: it takes its
// tile's list 32 splats at a time, one per lane, drops those that cannot reach its pixels (reaches; most of a
// tile's list, as a splat of a few pixels meets one or two of the eight warps), stages the rest with their colours
// in shared memory and blends them, lane = pixel; the next 32 are on their way meanwhile. It stops when its own
// pixels are opaque. Only splats that add nothing are dropped, so the results are those of the whole list. Bound
// by issue slots. (Staging the whole list by block and evaluating every splat at every pixel took 485 us for 300k
// splats at full HD, 875 us for the geometry maps of 300k surface splats and 2,320 us for the 48 channels of a million;
// this takes 221, 391 and 1,130 us.) The blocks per SM are what the registers of a group allow (a spill of 12 bytes in two forms).
template <int KG, class V>
__global__ void __launch_bounds__(kCompThreads, (KG <= 2 ? 5 : KG <= 4 ? 4 : KG <= 8 ? 3 : 2) * kSplit) k_composite(
    V v, const uint32_t* __restrict__ ranges, const int32_t* __restrict__ ids, const float* __restrict__ mean2d,
    const float4* __restrict__ conic_op, const float* __restrict__ colors, int64_t n, int k,
    const float* __restrict__ bg, float* __restrict__ image, float* __restrict__ final_T,
    int32_t* __restrict__ n_contrib) {
  extern __shared__ float4 fwd_smem[];
  const int lane = threadIdx.x & 31, warp = (blockIdx.x % kSplit) * (8 / kSplit) + (threadIdx.x >> 5);
  FwdWarp<KG>& sm = reinterpret_cast<FwdWarp<KG>*>(fwd_smem)[threadIdx.x >> 5];
  const int gtile = blockIdx.x / kSplit;  // scene-major tile index
  const Cam& c = v.cam(0);
  const int per_scene = c.gx * c.gy;
  const int b = gtile / per_scene, tile = gtile % per_scene;
  const int l0 = blockIdx.y * KG;
  const int nl = min(KG, k - l0);
  const int bx = (tile % c.gx) * kTile + (warp & 1) * 8, by = (tile / c.gx) * kTile + (warp >> 1) * 4;
  if (bx >= c.W || by >= c.H) return;  // the warp's pixels lie outside the image
  const int px = bx + (lane & 7), py = by + (lane >> 3);
  const bool inside = px < c.W && py < c.H;
  const uint32_t start = ranges[2 * gtile];
  const int len = (int)(ranges[2 * gtile + 1] - start);
  float T = 1.0f;
  float acc[3 * KG];
#pragma unroll
  for (int e = 0; e < 3 * KG; ++e) acc[e] = 0.f;
  bool done = !inside;
  int last = 0;
  const float fpx = (float)px, fpy = (float)py;
  int gid = 0;
  float2 xy = make_float2(0.f, 0.f);
  float4 co = make_float4(0.f, 0.f, 0.f, 0.f);
  auto fetch = [&](int p) {
    if (p < len) {
      gid = ids[start + p];
      xy = *reinterpret_cast<const float2*>(mean2d + 2 * (int64_t)gid);
      co = conic_op[gid];
    }
  };
  fetch(lane);
  for (int base = 0; base < len; base += 32) {
    const bool keep = base + lane < len && reaches(xy.x, xy.y, co, (float)bx, (float)(bx + 7), (float)by, (float)(by + 3));
    const unsigned m = __ballot_sync(0xffffffffu, keep);
    const int nk = __popc(m);
    if (keep) {
      const int slot = __popc(m & ((1u << lane) - 1u));
      sm.co[slot] = co;
      sm.xy[slot] = make_float4(xy.x, xy.y, __int_as_float(gid), __int_as_float(base + lane));
      if constexpr (!V::kRows) {
#pragma unroll
        for (int l = 0; l < KG; ++l) {
          const float* cp = colors + color_at(v, b, gid, l0 + (l < nl ? l : 0), k, n);
#pragma unroll
          for (int ch = 0; ch < 3; ++ch) sm.col[slot][3 * l + ch] = l < nl ? cp[ch] : 0.f;
        }
      }
    }
    fetch(base + 32 + lane);
    __syncwarp();
    if constexpr (V::kRows) {
      stage_rows<KG>(sm.col, sm.xy, nk, colors, l0, k);
      __syncwarp();
    }
    for (int j = 0; j < nk; ++j) {
      const float4 q = sm.xy[j], o = sm.co[j];
      const float dx = q.x - fpx, dy = q.y - fpy;
      const float power = -0.5f * (o.x * dx * dx + o.z * dy * dy) - o.y * dx * dy;
      const float alpha = fminf(kAlphaMax, o.w * __expf(power));
      if (done || power > 0.f || alpha < kAlphaMin) continue;
      const float test_T = T * (1.0f - alpha);
      if (test_T < kTStop) {
        done = true;
        continue;
      }
      const float wgt = alpha * T;
      blend_row<KG>(acc, sm.col[j], wgt);
      T = test_T;
      last = __float_as_int(q.w) + 1;
    }
    __syncwarp();  // the staged splats are replaced
    if (__all_sync(0xffffffffu, done)) break;
  }
  if (!inside) return;
  const int64_t HW = (int64_t)c.W * c.H;
  const int64_t pix = (int64_t)py * c.W + px;
  if (blockIdx.y == 0) {
    final_T[b * HW + pix] = T;
    n_contrib[b * HW + pix] = last;
  }
  float* img = image + (int64_t)b * k * 3 * HW;
#pragma unroll
  for (int e = 0; e < 3 * KG; ++e)
    if (e < 3 * nl) img[((int64_t)3 * l0 + e) * HW + pix] = acc[e] + T * bg[e % 3];
}

template <int KG, class V>
static void launch_composite_t(const V& v, unsigned tiles, const prtgs_render_state* st, const float* colors, int64_t n,
                               int k, const float* bg, float* image, cudaStream_t stream) {
  const size_t smem = sizeof(FwdWarp<KG>) * (kCompThreads / 32);
  if (smem > 48 * 1024) cudaFuncSetAttribute(k_composite<KG, V>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  k_composite<KG, V><<<dim3(tiles * kSplit, (unsigned)((k + KG - 1) / KG)), kCompThreads, smem, counted(stream)>>>(
      v, st->ranges, st->pair_ids, st->mean2d, reinterpret_cast<const float4*>(st->conic_op), colors, n, k, bg, image,
      st->final_T, st->n_contrib);
}

// Colour sets per block: the smallest group that holds k; above 8, groups of 16 where they leave no more sets
// empty than groups of 8 (every group evaluates the alphas again, and every set of a group costs its sums).
template <class V>
static void launch_composite(const V& v, unsigned tiles, const prtgs_render_state* st, const float* colors, int64_t n, int k,
                             const float* bg, float* image, cudaStream_t stream) {
  if constexpr (!V::kRows) {  // rows hold two sets or more
    if (k <= 1) return launch_composite_t<1>(v, tiles, st, colors, n, k, bg, image, stream);
  }
  if (k <= 2) launch_composite_t<2>(v, tiles, st, colors, n, k, bg, image, stream);
  else if (k <= 4) launch_composite_t<4>(v, tiles, st, colors, n, k, bg, image, stream);
  else if ((k + 7) / 8 % 2 == 0) launch_composite_t<16>(v, tiles, st, colors, n, k, bg, image, stream);
  else launch_composite_t<8>(v, tiles, st, colors, n, k, bg, image, stream);
}

// Forward pass for B scenes of one image size (B = 1 with OneView): tiles are numbered
// scene-major, so one sort and one composite launch cover every scene.
template <class V>
static int render_views(const prtgs_gaussians* g, const float* colors, int32_t k, const V& v, const Cam& c, int B,
                        const float* bg, float* image, prtgs_render_state* st, int32_t* status, void* ws,
                        cudaStream_t stream) {
  const int64_t n = g->n;
  const int64_t tiles = (int64_t)c.gx * c.gy * B;
  Carver cv(ws);
  void* scan_ws = cv.take<char>(scan_workspace(n));
  uint32_t* dkey[3];
  for (auto& p : dkey) p = cv.take<uint32_t>(n);
  int32_t* by_depth = cv.take<int32_t>(n);
  int32_t* by_depth_y = cv.take<int32_t>(n);
  uint32_t* incl = cv.take<uint32_t>(n);
  uint32_t* tkey[3];
  for (auto& p : tkey) p = cv.take<uint32_t>(st->max_pairs);
  int32_t* ids_x = cv.take<int32_t>(st->max_pairs);
  int32_t* ids_y = cv.take<int32_t>(st->max_pairs);
  void* sort_ws = cv.take<char>(radix_sort_workspace(st->max_pairs > n ? st->max_pairs : n));
  if (n == 0) {
    cudaMemsetAsync(st->ranges, 0, sizeof(uint32_t) * 2 * tiles, stream);
    cudaMemsetAsync(st->n_pairs, 0, sizeof(uint32_t), stream);
  } else {
    if (st->max_pairs <= 0) return PRTGS_ERR_CUDA;  // no room for any pair: nothing to launch the sort on
    const unsigned blocks = (unsigned)((n + 255) / 256);
    k_preprocess<V><<<blocks, 256, 0, counted(stream)>>>(
        n, g->means, g->scales, g->quats, g->opacity, v, st->mean2d, reinterpret_cast<float4*>(st->conic_op),
        st->depth, st->radius, st->tiles_touched, dkey[0]);
    PRTGS_CHECK_LAUNCH();
    // The (tile, depth) order as the splats' depth order followed by a stable sort of the pairs by tile: the
    // 32 depth bits are sorted once per splat instead of once per pair (25 M pairs of 300k splats: six
    // passes over 12-byte pairs, 1.57 ms, became two over 8-byte ones and four short ones, 0.44 ms).
    int rc = radix_sort_pairs(dkey[0], nullptr, dkey[2], by_depth, dkey[1], by_depth_y, n, nullptr, 0, 32, sort_ws, stream);
    if (rc != PRTGS_OK) return rc;
    const uint32_t cap = (uint32_t)(st->max_pairs < 0xffffffffll ? st->max_pairs : 0xffffffffll);
    rc = scan_u32(st->tiles_touched, incl, n, false, nullptr, scan_ws, stream, by_depth);
    if (rc != PRTGS_OK) return rc;
    rc = scan_u32(st->tiles_touched, st->tiles_touched, n, false, st->n_pairs, scan_ws, stream, nullptr, cap);
    if (rc != PRTGS_OK) return rc;
    k_duplicate<V><<<blocks, 256, 0, counted(stream)>>>(n, v, by_depth, st->mean2d, st->radius, incl, st->max_pairs, tkey[0],
                                                        ids_x, status);
    PRTGS_CHECK_LAUNCH();
    int tile_bits = 0;
    while ((int64_t(1) << tile_bits) < tiles) ++tile_bits;
    rc = radix_sort_pairs(tkey[0], ids_x, tkey[2], st->pair_ids, tkey[1], ids_y, st->max_pairs, st->n_pairs, 0, tile_bits,
                          sort_ws, stream, st->depth, st->pair_keys);
    if (rc != PRTGS_OK) return rc;
    k_ranges<<<(unsigned)((tiles + 7) / 8), 256, 0, counted(stream)>>>(st->pair_keys, st->n_pairs, tiles, st->ranges);
    PRTGS_CHECK_LAUNCH();
  }
  if constexpr (!V::kRows) {
    // rows for the colours, where the sort's buffers, which are free again, have the room
    const size_t room = reinterpret_cast<char*>(sort_ws) - reinterpret_cast<char*>(tkey[0]);
    if (k >= 2 && n > 0 && sizeof(float) * color_floats(k) * (size_t)n <= room) {
      k_color_rows<V><<<(unsigned)((n + 255) / 256), 256, 0, counted(stream)>>>(n, v, colors, k,
                                                                                reinterpret_cast<float4*>(tkey[0]));
      launch_composite(rows_of(v), (unsigned)tiles, st, reinterpret_cast<const float*>(tkey[0]), n, k, bg, image, stream);
      PRTGS_CHECK_LAUNCH();
      return PRTGS_OK;
    }
  }
  launch_composite(v, (unsigned)tiles, st, colors, n, k, bg, image, stream);
  PRTGS_CHECK_LAUNCH();
  return PRTGS_OK;
}

int render(const prtgs_gaussians* g, const float* colors, int32_t k, const prtgs_camera* cam, const float* bg,
           float* image, prtgs_render_state* st, int32_t* status, void* ws, cudaStream_t stream) {
  OneView v{make_cam(cam)};
  return render_views(g, colors, k, v, v.c, 1, bg, image, st, status, ws, stream);
}

int render_rows(const prtgs_gaussians* g, const float* rows, int32_t k, const prtgs_camera* cam, const float* bg,
                float* image, prtgs_render_state* st, int32_t* status, void* ws, cudaStream_t stream) {
  Rows<OneView> v;
  v.c = make_cam(cam);
  return render_views(g, rows, k, v, v.c, 1, bg, image, st, status, ws, stream);
}

size_t render_rows_floats(int32_t k) { return (size_t)color_floats(k); }

static int many_views(const prtgs_camera* cams, int32_t B, const int64_t* offsets, ManyViews& v) {
  if (B < 1 || B > kMaxScenes) return PRTGS_ERR_UNSUPPORTED;
  for (int b = 0; b < B; ++b) {
    v.c[b] = make_cam(cams + b);
    if (cams[b].width != cams[0].width || cams[b].height != cams[0].height) return PRTGS_ERR_SHAPE;
  }
  v.offs = offsets;
  v.B = B;
  return PRTGS_OK;
}

int render_batched(const prtgs_gaussians* g, const int64_t* offsets, int32_t B, const float* colors, int32_t k,
                   const prtgs_camera* cams, const float* bg, float* images, prtgs_render_state* st, int32_t* status,
                   void* ws, cudaStream_t stream) {
  static_assert(sizeof(ManyViews) < 30000, "the cameras must fit the kernel parameter space");
  ManyViews v;
  const int rc = many_views(cams, B, offsets, v);
  if (rc != PRTGS_OK) return rc;
  return render_views(g, colors, k, v, v.c[0], B, bg, images, st, status, ws, stream);
}

// ---- backward ------------------------------------------------------------------------------
// Sums of one splat, accumulated over the pixels and kept until k_preprocess_bwd: with g = dL/dpower, K the conic
// and (u, v) = K (mean2d - pixel), sum g, g u, g v, g u^2, g u v, g v^2, then sum alpha T dL/dpixel per colour
// channel, each group of KG colour sets on a 16-byte boundary. Power is -(K d).d / 2, so dL/dmean2d = -sum g (u, v)
// and dL/dcov = sum g (u, v)(u, v)^T / 2. Of sums of g d and g d d^T, in which a needle's long axis is large, both
// gradients would be what is left after it cancels: with scales that differ by e^1.4 at random (900 splats, 160 x 90,
// geometric mean of six scenes, one colour set) the errors against 64 bits of means, scales and rotations were 1.6e-3,
// 1.6e-3 and 3.0e-3 that way, 1.1e-3, 1.2e-3 and 2.2e-3 with K d and d d^T summed pixel by pixel, and are 8e-5, 1.2e-4
// and 1.4e-4 like this.
constexpr int kMoments = 8;  // six sums, padded
static int bwd_group(int k) { return k <= 1 ? 1 : (k <= 4 ? 4 : 8); }
static int bwd_stride(int k) { return kMoments + color_floats(bwd_group(k)) * ((k + bwd_group(k) - 1) / bwd_group(k)); }

// Per-warp staging of k_composite_bwd.
constexpr int kBwdChunk = 16;
template <int KG>
struct BwdWarp {
  float4 co[32];
  float4 xy[32];                       // mean2d, Gaussian, position in the tile's list (bits)
  float col[32][color_floats(KG)];
  float dpix[32][color_floats(KG)];    // dL/dimage of the warp's pixels
  float g[kBwdChunk][33], w[kBwdChunk][33];
};

// One warp per 8 x 4 pixels of a tile, on its own (no block barrier): it takes its tile's list from the
// last contributor of its pixels backwards, 32 splats at a time, drops those that cannot reach its pixels
// (reaches), and works on up to 16 of the rest in two phases. First lane = pixel: T, and per splat the two
// numbers that everything else follows from, g = dL/dpower and w = alpha T, go to shared memory. Then lane =
// (splat, half of the pixels): the moments of g and the colour sums of w are plain sums in registers, and a
// splat's sums leave the warp as a few vector reductions. (Reducing every value of every splat over the warp
// by shuffles and adding it to shared memory by one lane was 5.47 ms of the 8.4 ms of a 300k-splat full-HD
// frame; this takes 0.45 ms. 8 scenes x 4 lights at 720p: 14.8 -> 1.24 ms.) Bound by issue slots. The bounds
// leave 56 registers for one set (its own choice), 80 for groups of four and 96 of eight, which spill 12 and 28 bytes: 3 sets
// of 300k splats 688 us a call with 6 blocks, 708 with 5, 732 with 7; 8 sets 1,089 with 5, 1,245 with 6, 1,122 unbounded.
// The colours enter dL/dalpha through the scalar c . dL/dpixel only, whose blended remainder follows the same
// recursion as the colours'.
template <int KG, class V>
__global__ void __launch_bounds__(kCompThreads, KG == 1 ? 0 : KG == 4 ? 6 : 5) k_composite_bwd(
    V v, const uint32_t* __restrict__ ranges, const int32_t* __restrict__ ids, const float* __restrict__ mean2d,
    const float4* __restrict__ conic_op, const float* __restrict__ colors, int64_t n, int k,
    const float* __restrict__ bg, const float* __restrict__ final_T, const int32_t* __restrict__ n_contrib,
    const float* __restrict__ dimage, float* __restrict__ acc, int stride) {
  constexpr int CF = color_floats(KG);
  extern __shared__ float4 bwd_smem[];
  const int lane = threadIdx.x & 31, warp = (blockIdx.x % kSplit) * (8 / kSplit) + (threadIdx.x >> 5);
  BwdWarp<KG>& sm = reinterpret_cast<BwdWarp<KG>*>(bwd_smem)[threadIdx.x >> 5];
  const int gtile = blockIdx.x / kSplit;  // scene-major tile index
  const Cam& c = v.cam(0);
  const int per_scene = c.gx * c.gy;
  const int b = gtile / per_scene, tile = gtile % per_scene;
  const int l0 = blockIdx.y * KG;
  const int nl = min(KG, k - l0);
  const int bx = (tile % c.gx) * kTile + (warp & 1) * 8, by = (tile / c.gx) * kTile + (warp >> 1) * 4;
  const int px = bx + (lane & 7), py = by + (lane >> 3);
  const bool inside = px < c.W && py < c.H;
  const uint32_t start = ranges[2 * gtile], end = ranges[2 * gtile + 1];
  const int64_t HW = (int64_t)c.W * c.H;
  const int64_t pix = (int64_t)py * c.W + px;
  const float T_final = inside ? final_T[b * HW + pix] : 0.f;
  const uint32_t last = inside ? min((uint32_t)n_contrib[b * HW + pix], end - start) : 0u;
  const uint32_t wlast = __reduce_max_sync(0xffffffffu, last);
  if (wlast == 0) return;
  const float* dimg = dimage + (int64_t)b * k * 3 * HW;
  float dpix[CF];
  float bg_dot = 0.f;
#pragma unroll
  for (int e = 0; e < CF; ++e) {
    dpix[e] = (inside && e < 3 * nl) ? dimg[((int64_t)3 * l0 + e) * HW + pix] : 0.f;
    if (e < 3 * KG) bg_dot += bg[e % 3] * dpix[e];
  }
#pragma unroll
  for (int e = 0; e < CF; e += 4)
    *reinterpret_cast<float4*>(&sm.dpix[lane][e]) = make_float4(dpix[e], dpix[e + 1], dpix[e + 2], dpix[e + 3]);
  const float fpx = (float)px, fpy = (float)py;
  float T = T_final, behind = 0.f, last_alpha = 0.f, last_cd = 0.f;
  for (int hi = (int)wlast; hi > 0; hi -= 32) {
    const int p = hi - 1 - lane;  // lane 0 the farthest
    bool keep = false;
    float2 xy;
    float4 co;
    int gid = 0;
    if (p >= 0) {
      gid = ids[start + p];
      xy = *reinterpret_cast<const float2*>(mean2d + 2 * (int64_t)gid);
      co = conic_op[gid];
      keep = reaches(xy.x, xy.y, co, (float)bx, (float)(bx + 7), (float)by, (float)(by + 3));
    }
    const unsigned m = __ballot_sync(0xffffffffu, keep);
    const int nk = __popc(m);
    if (nk == 0) continue;
    if (keep) {
      const int slot = __popc(m & ((1u << lane) - 1u));
      sm.co[slot] = co;
      sm.xy[slot] = make_float4(xy.x, xy.y, __int_as_float(gid), __int_as_float(p));
      if constexpr (!V::kRows) {
#pragma unroll
        for (int l = 0; l < KG; ++l) {
          const float* cp = colors + color_at(v, b, gid, l0 + (l < nl ? l : 0), k, n);
#pragma unroll
          for (int ch = 0; ch < 3; ++ch) sm.col[slot][3 * l + ch] = l < nl ? cp[ch] : 0.f;
        }
      }
    }
    __syncwarp();
    if constexpr (V::kRows) {
      stage_rows<KG>(sm.col, sm.xy, nk, colors, l0, k);
      __syncwarp();
    }
    for (int c0 = 0; c0 < nk; c0 += kBwdChunk) {
      const int cnt = min(kBwdChunk, nk - c0);
      for (int i = 0; i < cnt; ++i) {
        const float4 q = sm.xy[c0 + i];
        const float4 o = sm.co[c0 + i];
        const float dx = q.x - fpx, dy = q.y - fpy;
        const float power = -0.5f * (o.x * dx * dx + o.z * dy * dy) - o.y * dx * dy;
        const float raw = o.w * __expf(power);
        const float alpha = fminf(kAlphaMax, raw);
        float g = 0.f, w = 0.f;
        if (__float_as_int(q.w) < (int)last && power <= 0.f && alpha >= kAlphaMin) {
          const float om = 1.0f - alpha;
          T = T / om;
          w = alpha * T;
          float cd = 0.f;
#pragma unroll
          for (int e = 0; e < 3 * KG; ++e) cd = fmaf(sm.col[c0 + i][e], dpix[e], cd);
          behind = last_alpha * last_cd + (1.0f - last_alpha) * behind;
          last_cd = cd;
          last_alpha = alpha;
          const float da = fmaf(cd - behind, T, (-T_final / om) * bg_dot);
          if (raw < kAlphaMax) g = da * raw;
        }
        sm.g[i][lane] = g;
        sm.w[i][lane] = w;
      }
      __syncwarp();
      const int i = lane & (kBwdChunk - 1), half = lane >> 4;
      float m0 = 0.f, mx = 0.f, my = 0.f, mxx = 0.f, mxy = 0.f, myy = 0.f;  // of u and v
      float cs[CF];
#pragma unroll
      for (int e = 0; e < CF; ++e) cs[e] = 0.f;
      if (i < cnt) {
        const float4 q = sm.xy[c0 + i], o = sm.co[c0 + i];
        const float x0 = q.x - (float)bx, y0 = q.y - (float)(by + 2 * half);
        // along a row v = rho u + tau, so that the sums with v follow from the row's sums with u
        const float rho = o.x > 0.f ? __fdividef(o.y, o.x) : 0.f, dv = fmaf(-rho, o.y, o.z);  // (0: a form that underflowed)
        float u0 = fmaf(o.x, x0, o.y * y0), tau = dv * y0;  // at the half's first pixel
#pragma unroll
        for (int row = 0; row < 2; ++row) {
          float s0 = 0.f, su = 0.f, suu = 0.f;
#pragma unroll
          for (int r = 0; r < 8; ++r) {
            const int at = 16 * half + 8 * row + r;
            const float g = sm.g[i][at], w = sm.w[i][at];
            const float u = fmaf(-(float)r, o.x, u0);
            const float gu = g * u;
            s0 += g;
            su += gu;
            suu = fmaf(gu, u, suu);
#pragma unroll
            for (int e = 0; e < CF; e += 4) {
              const float4 d = *reinterpret_cast<const float4*>(&sm.dpix[at][e]);
              cs[e] = fmaf(w, d.x, cs[e]);
              cs[e + 1] = fmaf(w, d.y, cs[e + 1]);
              cs[e + 2] = fmaf(w, d.z, cs[e + 2]);
              if (e + 3 < 3 * KG) cs[e + 3] = fmaf(w, d.w, cs[e + 3]);
            }
          }
          const float sv = fmaf(rho, su, tau * s0), suv = fmaf(rho, suu, tau * su);
          m0 += s0;
          mx += su;
          my += sv;
          mxx += suu;
          mxy += suv;
          myy += fmaf(rho, suv, tau * sv);
          u0 -= o.y;
          tau -= dv;
        }
      }
      m0 += __shfl_xor_sync(0xffffffffu, m0, 16);
      mx += __shfl_xor_sync(0xffffffffu, mx, 16);
      my += __shfl_xor_sync(0xffffffffu, my, 16);
      mxx += __shfl_xor_sync(0xffffffffu, mxx, 16);
      mxy += __shfl_xor_sync(0xffffffffu, mxy, 16);
      myy += __shfl_xor_sync(0xffffffffu, myy, 16);
#pragma unroll
      for (int e = 0; e < 3 * KG; ++e) cs[e] += __shfl_xor_sync(0xffffffffu, cs[e], 16);
      if (i < cnt) {
        float* out = acc + (int64_t)__float_as_int(sm.xy[c0 + i].z) * stride;
        if (half == 0) {
          // g has both signs: the second moments can be all that is left
          if (m0 != 0.f || mx != 0.f || my != 0.f || mxx != 0.f) red_add4(out, m0, mx, my, mxx);
          if (mxy != 0.f || myy != 0.f) red_add4(out + 4, mxy, myy, 0.f, 0.f);
        } else {
          out += kMoments + CF * (int)blockIdx.y;
#pragma unroll
          for (int e = 0; e < CF; e += 4)
            if (cs[e] != 0.f || cs[e + 1] != 0.f || cs[e + 2] != 0.f || cs[e + 3] != 0.f)
              red_add4(out + e, cs[e], cs[e + 1], cs[e + 2], cs[e + 3]);
        }
      }
      __syncwarp();
    }
  }
}

// 2D gradients -> means, scales, rotations (chain rule through Eq. 3 and Eq. 2).
template <class V>
__global__ void k_preprocess_bwd(int64_t n, const float* __restrict__ means, const float* __restrict__ scales,
                                 const float* __restrict__ quats, V v, const int32_t* __restrict__ radius,
                                 const float4* __restrict__ conic_op, const float* __restrict__ acc, int stride, int k,
                                 int kg, float* __restrict__ d_means, float* __restrict__ d_scales,
                                 float* __restrict__ d_quats, float* __restrict__ d_opacity,
                                 float* __restrict__ d_colors) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int scene = v.scene_of(i);
  const Cam& c = v.cam(scene);
  const float* sums = acc + i * stride;
  for (int l = 0; l < k; ++l) {
    const float* cs = sums + kMoments + color_floats(kg) * (l / kg) + 3 * (l % kg);
    float* out = d_colors + color_at(v, scene, i, l, k, n);
    out[0] = cs[0];
    out[1] = cs[1];
    out[2] = cs[2];
  }
  const float4 ma = *reinterpret_cast<const float4*>(sums), mb = *reinterpret_cast<const float4*>(sums + 4);
  const float gmx = -ma.y, gmy = -ma.z;
  const float gop = radius[i] > 0 && ma.x != 0.f ? ma.x / conic_op[i].w : 0.f;  // dL/dopacity = sum g / opacity
  d_opacity[i] = gop;
  float gm[3] = {0.f, 0.f, 0.f}, gs[3] = {0.f, 0.f, 0.f}, gq[4] = {0.f, 0.f, 0.f, 0.f};
  if (radius[i] > 0) {
    const float mx = means[3 * i], my = means[3 * i + 1], mz = means[3 * i + 2];
    const float x = c.r[0] * mx + c.r[1] * my + c.r[2] * mz + c.t[0];
    const float y = c.r[3] * mx + c.r[4] * my + c.r[5] * mz + c.t[1];
    const float z = c.r[6] * mx + c.r[7] * my + c.r[8] * mz + c.t[2];
    const float qw0 = quats[4 * i], qx0 = quats[4 * i + 1], qy0 = quats[4 * i + 2], qz0 = quats[4 * i + 3];
    const float qn = sqrtf(qw0 * qw0 + qx0 * qx0 + qy0 * qy0 + qz0 * qz0);
    const float qw = qw0 / qn, qx = qx0 / qn, qy = qy0 / qn, qz = qz0 / qn;
    float R[3][3];
    quat_rot(qw, qx, qy, qz, R);
    const float s[3] = {scales[3 * i], scales[3 * i + 1], scales[3 * i + 2]};
    float S[6];
    covariance3d(R, s[0], s[1], s[2], S);
    const float Sm[3][3] = {{S[0], S[1], S[2]}, {S[1], S[3], S[4]}, {S[2], S[4], S[5]}};
    const float iz = 1.0f / z;
    const float xz = x * iz, yz = y * iz;
    const bool clx = xz < -c.limx || xz > c.limx, cly = yz < -c.limy || yz > c.limy;
    const float cxz = fminf(c.limx, fmaxf(-c.limx, xz)), cyz = fminf(c.limy, fmaxf(-c.limy, yz));
    // J = [[fx/z, 0, -fx cxz / z], [0, fy/z, -fy cyz / z]]
    const float J[2][3] = {{c.fx * iz, 0.f, -c.fx * cxz * iz}, {0.f, c.fy * iz, -c.fy * cyz * iz}};
    const float W[3][3] = {{c.r[0], c.r[1], c.r[2]}, {c.r[3], c.r[4], c.r[5]}, {c.r[6], c.r[7], c.r[8]}};
    float M[2][3];
    for (int a = 0; a < 2; ++a)
      for (int k2 = 0; k2 < 3; ++k2) M[a][k2] = J[a][0] * W[0][k2] + J[a][1] * W[1][k2] + J[a][2] * W[2][k2];
    // dL/dcov2
    const float G2[2][2] = {{0.5f * ma.w, 0.5f * mb.x}, {0.5f * mb.x, 0.5f * mb.y}};
    // dM = 2 G2 M Sigma ; dJ = dM W^T
    float dM[2][3];
    for (int a = 0; a < 2; ++a)
      for (int q = 0; q < 3; ++q) {
        float acc = 0.f;
        for (int b = 0; b < 2; ++b)
          for (int p = 0; p < 3; ++p) acc += G2[a][b] * M[b][p] * Sm[p][q];
        dM[a][q] = 2.f * acc;
      }
    float dJ[2][3];
    for (int a = 0; a < 2; ++a)
      for (int k2 = 0; k2 < 3; ++k2) dJ[a][k2] = dM[a][0] * W[k2][0] + dM[a][1] * W[k2][1] + dM[a][2] * W[k2][2];
    // camera-space gradient from J(x,y,z) and from mean2d = (fx x/z + cx, fy y/z + cy)
    float gx = gmx * c.fx * iz;
    float gy = gmy * c.fy * iz;
    float gz = -gmx * c.fx * x * iz * iz - gmy * c.fy * y * iz * iz;
    gz += dJ[0][0] * (-c.fx * iz * iz) + dJ[1][1] * (-c.fy * iz * iz);
    // J02 = -fx cxz / z, cxz = clamp(x/z)
    if (!clx) {
      gx += dJ[0][2] * (-c.fx * iz * iz);
      gz += dJ[0][2] * (2.f * c.fx * x * iz * iz * iz);
    } else {
      gz += dJ[0][2] * (c.fx * cxz * iz * iz);
    }
    if (!cly) {
      gy += dJ[1][2] * (-c.fy * iz * iz);
      gz += dJ[1][2] * (2.f * c.fy * y * iz * iz * iz);
    } else {
      gz += dJ[1][2] * (c.fy * cyz * iz * iz);
    }
    // world-space: p = W mu + t
    for (int k2 = 0; k2 < 3; ++k2) gm[k2] = W[0][k2] * gx + W[1][k2] * gy + W[2][k2] * gz;
    // cov2 = N diag(s^2) N^T with N = M R. With G = N^T G2 N (= R^T dSigma R): dL/ds_k = 2 s_k G_kk, and a rotation by
    // theta about the local axes, R exp([theta]x), changes L by tau . theta, tau_1 = 2 G_23 (s_2^2 - s_3^2) and cyclic
    // (exactly 0 for equal scales, where the chain through dL/dR leaves its rounding). On the unit quaternion that is
    // 2 (tau_1 q i + tau_2 q j + tau_3 q k).
    float N[2][3], G[3][3];
    for (int a = 0; a < 2; ++a)
      for (int k2 = 0; k2 < 3; ++k2) N[a][k2] = M[a][0] * R[0][k2] + M[a][1] * R[1][k2] + M[a][2] * R[2][k2];
    for (int a = 0; a < 3; ++a)
      for (int k2 = 0; k2 < 3; ++k2)
        G[a][k2] = N[0][a] * (G2[0][0] * N[0][k2] + G2[0][1] * N[1][k2]) + N[1][a] * (G2[1][0] * N[0][k2] + G2[1][1] * N[1][k2]);
    for (int k2 = 0; k2 < 3; ++k2) gs[k2] = 2.f * s[k2] * G[k2][k2];
    const float t1 = 2.f * (G[1][2] + G[2][1]) * ((s[1] - s[2]) * (s[1] + s[2])) / qn;
    const float t2 = 2.f * (G[0][2] + G[2][0]) * ((s[2] - s[0]) * (s[2] + s[0])) / qn;
    const float t3 = 2.f * (G[0][1] + G[1][0]) * ((s[0] - s[1]) * (s[0] + s[1])) / qn;
    gq[0] = -t1 * qx - t2 * qy - t3 * qz;
    gq[1] = t1 * qw - t2 * qz + t3 * qy;
    gq[2] = t1 * qz + t2 * qw - t3 * qx;
    gq[3] = -t1 * qy + t2 * qx + t3 * qw;
  }
  for (int k2 = 0; k2 < 3; ++k2) {
    d_means[3 * i + k2] = gm[k2];
    d_scales[3 * i + k2] = gs[k2];
  }
  for (int k2 = 0; k2 < 4; ++k2) d_quats[4 * i + k2] = gq[k2];
}

// ---- depth and normal maps (Eq. 23, Eq. 25): the composite of d_i and n_i -------------------------
// Rows for render_rows() with two "lights": light 0 carries (d_i, 0, 0), d_i the view-space
// depth of the splat's mean; light 1 carries the raw normal n_i.
__global__ void k_geometry_features(int64_t n, Cam c, const float* __restrict__ means,
                                    const float* __restrict__ normals, float* __restrict__ F) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const float x = means[3 * i], y = means[3 * i + 1], z = means[3 * i + 2];
  const float d = fmaf(c.r[6], x, fmaf(c.r[7], y, fmaf(c.r[8], z, c.t[2])));
  float4* row = reinterpret_cast<float4*>(F) + 2 * i;
  row[0] = make_float4(d, 0.f, 0.f, normals[3 * i]);
  row[1] = make_float4(normals[3 * i + 1], normals[3 * i + 2], 0.f, 0.f);
}

size_t render_geometry_workspace(int64_t n, int32_t width, int32_t height, int64_t max_pairs) {
  return align_up(sizeof(float) * 8 * (size_t)n) + align_up(sizeof(float) * 6 * (size_t)width * height) +
         align_up(sizeof(float) * 4) + render_workspace(n, width, height, max_pairs);
}

int render_geometry(const prtgs_gaussians* g, const prtgs_camera* cam, float* depth, float* normal,
                    prtgs_render_state* st, int32_t* status, void* ws, cudaStream_t stream) {
  const int64_t n = g->n;
  const int64_t n_pix = (int64_t)cam->width * cam->height;
  Carver cv(ws);
  float* F = cv.take<float>(8 * (size_t)n);
  float* img = cv.take<float>(6 * (size_t)n_pix);
  float* zero = cv.take<float>(4);
  void* rws = static_cast<char*>(ws) + cv.off;
  cudaMemsetAsync(zero, 0, sizeof(float) * 4, stream);
  if (n > 0) {
    k_geometry_features<<<(unsigned)((n + 255) / 256), 256, 0, counted(stream)>>>(n, make_cam(cam), g->means, g->normals, F);
    PRTGS_CHECK_LAUNCH();
  }
  const int rc = render_rows(g, F, 2, cam, zero, img, st, status, rws, stream);
  if (rc != PRTGS_OK) return rc;
  // image [2][3][H][W]: depth is light 0's first channel, the normal light 1's three channels
  cudaMemcpyAsync(depth, img, sizeof(float) * n_pix, cudaMemcpyDeviceToDevice, stream);
  cudaMemcpyAsync(normal, img + 3 * n_pix, sizeof(float) * 3 * n_pix, cudaMemcpyDeviceToDevice, stream);
  PRTGS_CHECK_LAUNCH();
  return PRTGS_OK;
}

size_t render_backward_workspace(int64_t n, int32_t k) {
  return align_up(sizeof(float) * (size_t)bwd_stride(k) * n) + (k >= 2 ? align_up(sizeof(float) * color_floats(k) * (size_t)n) : 0);
}

template <int KG, class V>
static void launch_composite_bwd(dim3 grid, const V& v, const prtgs_render_state* st, const float* colors, int64_t n, int k,
                                 const float* bg, const float* dimage, float* acc, int stride, cudaStream_t stream) {
  const size_t smem = sizeof(BwdWarp<KG>) * (kCompThreads / 32);
  cudaFuncSetAttribute(k_composite_bwd<KG, V>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  k_composite_bwd<KG, V><<<grid, kCompThreads, smem, counted(stream)>>>(
      v, st->ranges, st->pair_ids, st->mean2d, reinterpret_cast<const float4*>(st->conic_op), colors, n, k, bg,
      st->final_T, st->n_contrib, dimage, acc, stride);
}

template <class V>
static int render_backward_views(const prtgs_gaussians* g, const float* colors, int32_t k, const V& v, const Cam& c,
                                 int B, const float* bg, const prtgs_render_state* st, const float* dimage,
                                 float* d_means, float* d_scales, float* d_quats, float* d_opacity, float* d_colors,
                                 void* ws, cudaStream_t stream) {
  const int64_t n = g->n;
  if (n == 0) return PRTGS_OK;
  const int64_t tiles = (int64_t)c.gx * c.gy * B;
  const int kg = bwd_group(k), stride = bwd_stride(k);
  Carver cv(ws);
  float* acc = cv.take<float>((size_t)stride * n);
  cudaMemsetAsync(acc, 0, sizeof(float) * stride * n, stream);
  // every light's colour sets in groups of up to 8 (shared memory bound)
  dim3 grid((unsigned)tiles * kSplit, (unsigned)((k + kg - 1) / kg));
  if (kg == 1) {
    launch_composite_bwd<1>(grid, v, st, colors, n, k, bg, dimage, acc, stride, stream);
  } else {
    float* rows = cv.take<float>((size_t)color_floats(k) * n);
    k_color_rows<V><<<(unsigned)((n + 255) / 256), 256, 0, counted(stream)>>>(n, v, colors, k,
                                                                              reinterpret_cast<float4*>(rows));
    if (kg == 4) launch_composite_bwd<4>(grid, rows_of(v), st, rows, n, k, bg, dimage, acc, stride, stream);
    else launch_composite_bwd<8>(grid, rows_of(v), st, rows, n, k, bg, dimage, acc, stride, stream);
  }
  PRTGS_CHECK_LAUNCH();
  k_preprocess_bwd<V><<<(unsigned)((n + 255) / 256), 256, 0, counted(stream)>>>(
      n, g->means, g->scales, g->quats, v, st->radius, reinterpret_cast<const float4*>(st->conic_op), acc, stride, k, kg,
      d_means, d_scales, d_quats, d_opacity, d_colors);
  PRTGS_CHECK_LAUNCH();
  return PRTGS_OK;
}

int render_backward(const prtgs_gaussians* g, const float* colors, int32_t k, const prtgs_camera* cam,
                    const float* bg, const prtgs_render_state* st, const float* dimage, float* d_means,
                    float* d_scales, float* d_quats, float* d_opacity, float* d_colors, void* ws,
                    cudaStream_t stream) {
  OneView v{make_cam(cam)};
  return render_backward_views(g, colors, k, v, v.c, 1, bg, st, dimage, d_means, d_scales, d_quats, d_opacity,
                               d_colors, ws, stream);
}

int render_backward_batched(const prtgs_gaussians* g, const int64_t* offsets, int32_t B, const float* colors,
                            int32_t k, const prtgs_camera* cams, const float* bg, const prtgs_render_state* st,
                            const float* dimages, float* d_means, float* d_scales, float* d_quats, float* d_opacity,
                            float* d_colors, void* ws, cudaStream_t stream) {
  ManyViews v;
  const int rc = many_views(cams, B, offsets, v);
  if (rc != PRTGS_OK) return rc;
  return render_backward_views(g, colors, k, v, v.c[0], B, bg, st, dimages, d_means, d_scales, d_quats, d_opacity,
                               d_colors, ws, stream);
}

// ---- L2 loss ---------------------------------------------------------------------------------
constexpr int kLossThreads = 256;
constexpr int kLossItems = 16;

__global__ void k_l2_partial(const float* __restrict__ a, const float* __restrict__ b, int64_t count, float scale,
                             float* __restrict__ grad, float* __restrict__ partial) {
  __shared__ float sw[kLossThreads / 32];
  const int64_t base = (int64_t)blockIdx.x * kLossThreads * kLossItems;
  float s = 0.f;
  for (int q = 0; q < kLossItems; ++q) {
    int64_t i = base + (int64_t)q * kLossThreads + threadIdx.x;
    if (i < count) {
      float d = a[i] - b[i];
      grad[i] = scale * d;
      s = fmaf(d, d, s);
    }
  }
  s = warp_sum(s);
  if ((threadIdx.x & 31) == 0) sw[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    float t = 0.f;
    for (int w = 0; w < kLossThreads / 32; ++w) t += sw[w];
    partial[blockIdx.x] = t;
  }
}

__global__ void k_l2_final(const float* __restrict__ partial, int64_t nb, float inv_count, float* __restrict__ loss) {
  __shared__ double sd[256];
  double s = 0.0;
  for (int64_t b = threadIdx.x; b < nb; b += blockDim.x) s += (double)partial[b];
  sd[threadIdx.x] = s;
  __syncthreads();
  for (int off = blockDim.x / 2; off > 0; off >>= 1) {
    if ((int)threadIdx.x < off) sd[threadIdx.x] += sd[threadIdx.x + off];
    __syncthreads();
  }
  if (threadIdx.x == 0) *loss = (float)(sd[0] * (double)inv_count);
}

// Per-scene losses of B images of `count` elements each: loss[b] = mean over scene b, dimage =
// 2 (image - target) / count. Blocks never straddle scenes (grid.y = scene).
__global__ void k_l2_partial_batched(const float* __restrict__ a, const float* __restrict__ t, int64_t count,
                                     float scale, float* __restrict__ grad, float* __restrict__ partial) {
  __shared__ float sw[kLossThreads / 32];
  const int64_t off = (int64_t)blockIdx.y * count;
  const int64_t base = (int64_t)blockIdx.x * kLossThreads * kLossItems;
  float s = 0.f;
  for (int q = 0; q < kLossItems; ++q) {
    const int64_t i = base + (int64_t)q * kLossThreads + threadIdx.x;
    if (i < count) {
      const float d = a[off + i] - t[off + i];
      grad[off + i] = scale * d;
      s = fmaf(d, d, s);
    }
  }
  s = warp_sum(s);
  if ((threadIdx.x & 31) == 0) sw[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    float u = 0.f;
    for (int w = 0; w < kLossThreads / 32; ++w) u += sw[w];
    partial[(int64_t)blockIdx.y * gridDim.x + blockIdx.x] = u;
  }
}

__global__ void k_l2_final_batched(const float* __restrict__ partial, int64_t nb, float inv_count,
                                   float* __restrict__ loss) {
  __shared__ double sd[256];
  const float* p = partial + (int64_t)blockIdx.x * nb;
  double s = 0.0;
  for (int64_t b = threadIdx.x; b < nb; b += blockDim.x) s += (double)p[b];
  sd[threadIdx.x] = s;
  __syncthreads();
  for (int off = blockDim.x / 2; off > 0; off >>= 1) {
    if ((int)threadIdx.x < off) sd[threadIdx.x] += sd[threadIdx.x + off];
    __syncthreads();
  }
  if (threadIdx.x == 0) loss[blockIdx.x] = (float)(sd[0] * (double)inv_count);
}

size_t l2_loss_batched_workspace(int64_t count, int32_t n_scenes) {
  const int64_t nb = (count + kLossThreads * kLossItems - 1) / (kLossThreads * kLossItems);
  return align_up(sizeof(float) * (size_t)(nb > 0 ? nb : 1) * (n_scenes > 0 ? n_scenes : 1));
}

int l2_loss_batched(const float* images, const float* targets, int64_t count, int32_t n_scenes, float* losses,
                    float* dimages, void* ws, cudaStream_t stream) {
  if (count <= 0 || n_scenes <= 0) return PRTGS_ERR_INVALID_ARG;
  const int64_t nb = (count + kLossThreads * kLossItems - 1) / (kLossThreads * kLossItems);
  float* partial = static_cast<float*>(ws);
  k_l2_partial_batched<<<dim3((unsigned)nb, (unsigned)n_scenes), kLossThreads, 0, counted(stream)>>>(
      images, targets, count, 2.0f / (float)count, dimages, partial);
  k_l2_final_batched<<<(unsigned)n_scenes, 256, 0, counted(stream)>>>(partial, nb, 1.0f / (float)count, losses);
  PRTGS_CHECK_LAUNCH();
  return PRTGS_OK;
}

size_t l2_loss_workspace(int64_t count) {
  int64_t nb = (count + kLossThreads * kLossItems - 1) / (kLossThreads * kLossItems);
  return align_up(sizeof(float) * (size_t)(nb > 0 ? nb : 1));
}

int l2_loss(const float* image, const float* target, int64_t count, float* loss, float* dimage, void* ws,
            cudaStream_t stream) {
  if (count <= 0) return PRTGS_ERR_INVALID_ARG;
  int64_t nb = (count + kLossThreads * kLossItems - 1) / (kLossThreads * kLossItems);
  float* partial = static_cast<float*>(ws);
  k_l2_partial<<<(unsigned)nb, kLossThreads, 0, counted(stream)>>>(image, target, count, 2.0f / (float)count, dimage, partial);
  k_l2_final<<<1, 256, 0, counted(stream)>>>(partial, nb, 1.0f / (float)count, loss);
  PRTGS_CHECK_LAUNCH();
  return PRTGS_OK;
}

}  // namespace prtgs
