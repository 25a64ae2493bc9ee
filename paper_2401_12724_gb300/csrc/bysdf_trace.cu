// The step upstream of the BYSDF: camera rays against explicit yarns (Sec. 3.3)
// and their ray differentials (Sec. 5.3), producing BYSDF hit records.
//
// Yarns are straight pieces of yarn curves staged in shared memory (a
// piece's rotation-minimising frame is constant, so it carries its reference
// normal).  One thread per ray; pieces carry a bounding sphere, and so do
// groups of kGroupPieces consecutive pieces (neighbours along a yarn, in the
// caller's order).  The rays of a warp are neighbouring pixels, so the warp
// culls against a bound on all 32 rays at once: it tests 32 groups at a time,
// one per lane, then the pieces of up to four kept groups at a time, one per
// lane, and keeps the ballot of the pieces some ray may reach.  A warp that
// keeps many groups holds the end of a row of pixels and the start of the next
// one, and goes on with two bounds, one for each part.  Each ray then tests
// the kept pieces in ascending order: where a round kept many, a conservative
// bounding-sphere distance test (a tight bundle's kept pieces are reached by
// most of its rays, and the test is a quarter of the work), then the lateral
// surface about the ray's point of closest
// approach to the axis, where the square root is taken of R^2 minus a small
// distance (no cancellation between terms of the camera distance squared).
// The culling only skips pieces that no ray of the warp can hit: the result
// is that of testing every piece.
#include <algorithm>
#include <mutex>
#include <type_traits>
#include <vector>

#include "bysdf_launch.h"

namespace bysdf {

namespace {

// one piece in shared memory: 4 x float4
//   a = (p0, length), b = (t, R), c = (n_ref, v0), d = (centre, r_sphere^2)
struct PieceS {
  float4 a, b, c, d;
};

__device__ __forceinline__ float dot3(float ax, float ay, float az, float bx, float by, float bz) {
  return fmaf(ax, bx, fmaf(ay, by, az * bz));
}

// signed distance of the line (o, d) from the piece's axis in its
// cross-section, over R (the azimuthal offset); +inf along the axis
__device__ __forceinline__ float line_offset(const PieceS& p, float bx, float by, float bz,
                                             float ox, float oy, float oz, float dx, float dy,
                                             float dz) {
  const float qx = ox - p.a.x, qy = oy - p.a.y, qz = oz - p.a.z;
  const float q_n = dot3(qx, qy, qz, p.c.x, p.c.y, p.c.z);
  const float q_b = dot3(qx, qy, qz, bx, by, bz);
  const float d_n = dot3(dx, dy, dz, p.c.x, p.c.y, p.c.z);
  const float d_b = dot3(dx, dy, dz, bx, by, bz);
  const float l = sqrtf(d_n * d_n + d_b * d_b);
  if (!(l > 0.f)) return __int_as_float(0x7f800000);
  return (q_n * d_b - q_b * d_n) / (l * p.b.w);
}

constexpr int kGroupPieces = 8;
// the piece rounds give each of four groups 8 lanes (lane >> 3, lane & 7)
static_assert(kGroupPieces == 8, "the piece rounds assume groups of 8 pieces");

// A bound on the rays of some lanes: origin o and unit direction u of their
// middle lane, ro >= |o_i - o| and del >= |u_i - u|.
struct Bundle {
  float ox, oy, oz, ux, uy, uz, ro, del;
};

__device__ __forceinline__ Bundle make_bundle(bool in, int middle, float ox, float oy, float oz,
                                              float ux, float uy, float uz) {
  Bundle q;
  q.ox = __shfl_sync(0xffffffffu, ox, middle);
  q.oy = __shfl_sync(0xffffffffu, oy, middle);
  q.oz = __shfl_sync(0xffffffffu, oz, middle);
  q.ux = __shfl_sync(0xffffffffu, ux, middle);
  q.uy = __shfl_sync(0xffffffffu, uy, middle);
  q.uz = __shfl_sync(0xffffffffu, uz, middle);
  float ro = 0.f, del = 0.f;
  if (in) {
    const float ex = ox - q.ox, ey = oy - q.oy, ez = oz - q.oz;
    const float fx = ux - q.ux, fy = uy - q.uy, fz = uz - q.uz;
    ro = sqrtf(dot3(ex, ey, ez, ex, ey, ez));
    del = sqrtf(dot3(fx, fy, fz, fx, fy, fz));
  }
  // non-negative floats order like their bit patterns
  q.ro = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(ro)));
  q.del = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(del)));
  return q;
}

// The line of a ray of the bundle lies at least
// dist(C, axis) - ro - (|C - o| + ro) * del from a point C: a sphere (C, r^2)
// farther than r plus that slack from the axis is missed by every ray of the
// bundle.  A bound that is not finite (a degenerate ray) keeps the sphere.
__device__ __forceinline__ bool bundle_reaches(float4 sph, const Bundle& q) {
  const float vx = sph.x - q.ox, vy = sph.y - q.oy, vz = sph.z - q.oz;
  const float tv = dot3(vx, vy, vz, q.ux, q.uy, q.uz);
  const float px = fmaf(-tv, q.ux, vx), py = fmaf(-tv, q.uy, vy), pz = fmaf(-tv, q.uz, vz);
  const float thr =
      fmaf(sqrtf(dot3(vx, vy, vz, vx, vy, vz)) + q.ro, q.del, sqrtf(sph.w) + q.ro) * 1.0001f +
      1e-4f;
  return !(dot3(px, py, pz, px, py, pz) > thr * thr);
}

// Kept groups of 32 above which a warp's rays are bounded as two bundles.  A
// warp over a row's end kept nearly all pieces, and a few of them were the
// kernel's time: 333 x 777 rays against 1798 pieces 204 us with one bundle, 46
// with two.  Rows of 2048 take the second bound at 12 groups as rarely as at
// 20 (162 us against 512 pieces); at 9 they begin to (174 us), at 6 194 us.
constexpr int kSplitGroups = 12;
// Kept pieces of a round above which each ray tests their spheres first (512
// pieces 175 us, 182 us with the test always; 4 or 16 the same).
constexpr int kSpherePieces = 8;

// A launch's planes, one pointer each, with 32-bit indices below them: an
// address is then one multiply-add; a call of more rays than a launch's index
// holds is several launches.
constexpr int64_t kMaxLaunch = (int64_t)1 << 30;
struct Planes {
  const float* in[18];  // o, d, o1, d1, o2, d2 by component
  uint32_t n;
  bool diff;
  float light[3];
  float *h, *u, *v, *wi[3], *wo[3], *ratio, *t_hit;
  int32_t *mat_id, *yarn_id;
};

}  // namespace

// Bound by instruction issue (1,110 warp instructions per 32 rays) and
// the latency of the culling chain.  One CTA of 768 threads (24 warps, up to 85
// registers) per SM shares one copy of the pieces: CTAs of 256 held up to three
// copies, and 2048 pieces (140 KB) left room for one of 8 warps.  2048 x 2048
// rays against 512 pieces 175 -> 157 us, against 2048 pieces 443 -> 226 us (and
// 5% of both for the second bundle's code); 512 threads 190 and 276 us.  Before
// this kernel's shape, short list and tests 192 and 461 us.  Fewer rays than
// one CTA per SM go in CTAs of 256, so that they spread over the SMs.
template <int BLOCK>
__global__ void __launch_bounds__(BLOCK, 1) k_trace_yarns(const bysdf_yarn* __restrict__ yarns,
                                                     int n_yarns, const Planes a) {
  extern __shared__ float4 smem_pieces[];
  PieceS* ps = reinterpret_cast<PieceS*>(smem_pieces);
  const int n_grp = (n_yarns + kGroupPieces - 1) / kGroupPieces;
  float4* grp = smem_pieces + 4 * n_yarns;  // (centre, squared radius) per group
  int32_t* smat = reinterpret_cast<int32_t*>(grp + n_grp);  // material per piece
  // stage the pieces with an orthonormal frame: t / |t|, then n_ref without
  // its t component, normalised; bounding sphere about the piece's centre
  for (int k = threadIdx.x; k < n_yarns; k += blockDim.x) {
    const bysdf_yarn y = yarns[k];
    float tx = y.tangent[0], ty = y.tangent[1], tz = y.tangent[2];
    const float it = rsqrtf(dot3(tx, ty, tz, tx, ty, tz));
    tx *= it;
    ty *= it;
    tz *= it;
    const float nt = dot3(y.n_ref[0], y.n_ref[1], y.n_ref[2], tx, ty, tz);
    float nx = y.n_ref[0] - nt * tx, ny = y.n_ref[1] - nt * ty, nz = y.n_ref[2] - nt * tz;
    const float in = rsqrtf(dot3(nx, ny, nz, nx, ny, nz));
    nx *= in;
    ny *= in;
    nz *= in;
    const float hl = 0.5f * y.length;
    const float rs = sqrtf(hl * hl + y.radius * y.radius);
    PieceS p;
    p.a = make_float4(y.p0[0], y.p0[1], y.p0[2], y.length);
    p.b = make_float4(tx, ty, tz, y.radius);
    p.c = make_float4(nx, ny, nz, y.v0);
    // margin: 1e-4 relative plus 1e-4 absolute covers the float rounding of
    // the distance test below
    const float rm = rs * 1.0001f + 1e-4f;
    p.d = make_float4(y.p0[0] + hl * tx, y.p0[1] + hl * ty, y.p0[2] + hl * tz, rm * rm);
    ps[k] = p;
    smat[k] = y.mat_id;
  }
  __syncthreads();
  // group spheres: the box around the pieces' spheres, then the largest
  // reach from its centre, widened like the piece spheres
  for (int c = threadIdx.x; c < n_grp; c += blockDim.x) {
    const int k0 = c * kGroupPieces, k1 = min(k0 + kGroupPieces, n_yarns);
    float lx = 3.4e38f, ly = 3.4e38f, lz = 3.4e38f, hx = -3.4e38f, hy = -3.4e38f, hz = -3.4e38f;
    for (int k = k0; k < k1; ++k) {
      const float4 d = ps[k].d;
      const float r = sqrtf(d.w);
      lx = fminf(lx, d.x - r);
      ly = fminf(ly, d.y - r);
      lz = fminf(lz, d.z - r);
      hx = fmaxf(hx, d.x + r);
      hy = fmaxf(hy, d.y + r);
      hz = fmaxf(hz, d.z + r);
    }
    const float cx = 0.5f * (lx + hx), cy = 0.5f * (ly + hy), cz = 0.5f * (lz + hz);
    float R = 0.f;
    for (int k = k0; k < k1; ++k) {
      const float4 d = ps[k].d;
      const float ex = d.x - cx, ey = d.y - cy, ez = d.z - cz;
      R = fmaxf(R, sqrtf(dot3(ex, ey, ez, ex, ey, ez)) + sqrtf(d.w));
    }
    R = R * 1.0001f + 1e-4f;
    grp[c] = make_float4(cx, cy, cz, R * R);
  }
  __syncthreads();
  const uint32_t n = a.n;
  const uint32_t lane = threadIdx.x & 31;
  const uint32_t stride = gridDim.x * blockDim.x;
  const uint32_t below = (1u << lane) - 1u;
  __shared__ uint32_t lists[BLOCK / 32][8];
  uint32_t* mine = lists[threadIdx.x >> 5];
  // whole warps step through the rays (lanes past the end take part in the
  // ballots with a dummy ray and write nothing); each lane loads its next ray
  // while the current one is culled
  uint32_t i0 = blockIdx.x * blockDim.x + (threadIdx.x & ~31u);
  float nox = 0.f, noy = 0.f, noz = 0.f, ndx = 0.f, ndy = 0.f, ndz = 1.f;
  if (i0 + lane < n) {
    const uint32_t j = i0 + lane;
    nox = __ldg(a.in[0] + j), noy = __ldg(a.in[1] + j), noz = __ldg(a.in[2] + j);
    ndx = __ldg(a.in[3] + j), ndy = __ldg(a.in[4] + j), ndz = __ldg(a.in[5] + j);
  }
  for (; i0 < n; i0 += stride) {
    const uint32_t i = i0 + lane;
    const bool act = i < n;
    const float ox = nox, oy = noy, oz = noz, dx = ndx, dy = ndy, dz = ndz;
    if (i + stride < n) {
      const uint32_t j = i + stride;
      nox = __ldg(a.in[0] + j), noy = __ldg(a.in[1] + j), noz = __ldg(a.in[2] + j);
      ndx = __ldg(a.in[3] + j), ndy = __ldg(a.in[4] + j), ndz = __ldg(a.in[5] + j);
    }
    // the differential rays, loaded while the warp culls
    const bool diff = a.diff;
    float o1x = 0.f, o1y = 0.f, o1z = 0.f, d1x = 0.f, d1y = 0.f, d1z = 0.f;
    float o2x = 0.f, o2y = 0.f, o2z = 0.f, d2x = 0.f, d2y = 0.f, d2z = 0.f;
    if (act && diff) {
      o1x = __ldg(a.in[6] + i), o1y = __ldg(a.in[7] + i), o1z = __ldg(a.in[8] + i);
      d1x = __ldg(a.in[9] + i), d1y = __ldg(a.in[10] + i), d1z = __ldg(a.in[11] + i);
      o2x = __ldg(a.in[12] + i), o2y = __ldg(a.in[13] + i), o2z = __ldg(a.in[14] + i);
      d2x = __ldg(a.in[15] + i), d2y = __ldg(a.in[16] + i), d2z = __ldg(a.in[17] + i);
    }
    const float idd = 1.0f / dot3(dx, dy, dz, dx, dy, dz);
    const float ild = sqrtf(idd);
    // the warp's rays as one bundle (active lanes are 0 .. popc - 1)
    const int n_act = __popc(__ballot_sync(0xffffffffu, act));
    const float ux = dx * ild, uy = dy * ild, uz = dz * ild;
    Bundle q1 = make_bundle(act, (n_act - 1) >> 1, ox, oy, oz, ux, uy, uz);
    Bundle q2;
    int best = -1;
    float sbest = 0.f;
    // tests the pieces from group c0 on; with one bundle, up to the groups
    // that call for two, whose first it returns
    auto scan = [&](auto with_two, int c0) {
      constexpr bool kTwo = decltype(with_two)::value;
      auto reaches = [&](float4 sph) {
        return bundle_reaches(sph, q1) || (kTwo && bundle_reaches(sph, q2));
      };
      for (; c0 < n_grp; c0 += 32) {
        const unsigned gm = __ballot_sync(
            0xffffffffu, c0 + (int)lane < n_grp && reaches(grp[c0 + lane]));
        if (!kTwo && __popc(gm) > kSplitGroups && n_act > 1) return c0;
        // the kept groups' offsets in c0, in ascending order, a byte each, read
        // four at a time, 8 lanes to a group
        const uint32_t kept = __popc(gm);
        if (gm >> lane & 1) reinterpret_cast<uint8_t*>(mine)[__popc(gm & below)] = (uint8_t)lane;
        __syncwarp();
        for (uint32_t g0 = 0; 4 * g0 < kept; ++g0) {
          const uint32_t four = mine[g0];
          const int kl = (c0 + (int)((four >> (lane & 24)) & 0xffu)) * kGroupPieces + (int)(lane & 7);
          unsigned pm = __ballot_sync(
              0xffffffffu, (uint32_t)(4 * g0) + (lane >> 3) < kept && kl < n_yarns &&
                               reaches(ps[kl].d));
          const bool many = __popc(pm) > kSpherePieces;
          while (pm) {
            const int b = __ffs(pm) - 1;
            pm &= pm - 1;
            const int k = (c0 + (int)((four >> (b & 24)) & 0xffu)) * kGroupPieces + (b & 7);
            if (many) {
              const float4 sd = ps[k].d;
              // bounding sphere: distance of the centre from the ray line
              const float mx = ox - sd.x, my = oy - sd.y, mz = oz - sd.z;
              const float mb = dot3(mx, my, mz, dx, dy, dz) * idd;
              const float px = fmaf(-mb, dx, mx), py = fmaf(-mb, dy, my), pz = fmaf(-mb, dz, mz);
              if (dot3(px, py, pz, px, py, pz) > sd.w) continue;
            }
            const float4 pa = ps[k].a, pb = ps[k].b;
            // lateral surface about the ray's closest approach to the axis
            const float qx = ox - pa.x, qy = oy - pa.y, qz = oz - pa.z;
            const float qt = dot3(qx, qy, qz, pb.x, pb.y, pb.z);
            const float dt = dot3(dx, dy, dz, pb.x, pb.y, pb.z);
            const float qpx = fmaf(-qt, pb.x, qx), qpy = fmaf(-qt, pb.y, qy), qpz = fmaf(-qt, pb.z, qz);
            const float dpx = fmaf(-dt, pb.x, dx), dpy = fmaf(-dt, pb.y, dy), dpz = fmaf(-dt, pb.z, dz);
            const float aa = dot3(dpx, dpy, dpz, dpx, dpy, dpz);
            if (!(aa > 1e-20f)) continue;
            const float R2 = pb.w * pb.w;
            if (!(dot3(qpx, qpy, qpz, qpx, qpy, qpz) > R2)) continue;  // starts inside
            const float sc = -dot3(qpx, qpy, qpz, dpx, dpy, dpz) / aa;
            const float mpx = fmaf(sc, dpx, qpx), mpy = fmaf(sc, dpy, qpy), mpz = fmaf(sc, dpz, qpz);
            const float e2 = R2 - dot3(mpx, mpy, mpz, mpx, mpy, mpz);
            if (e2 < 0.f) continue;
            const float s = sc - sqrtf(e2 / aa);
            if (!(s > 0.f) || (best >= 0 && !(s < sbest))) continue;
            const float w = fmaf(s, dt, qt);
            if (w < 0.f || w > pa.w) continue;
            best = k;
            sbest = s;
          }
        }
        __syncwarp();  // the list is rewritten for the next groups
      }
      return n_grp;
    };
    const int wide = scan(std::false_type{}, 0);
    if (wide < n_grp) {
      // the rays of a row's end and the next row's start: two bundles, split
      // where neighbouring lanes differ most
      const float hx = ox - __shfl_up_sync(0xffffffffu, ox, 1);
      const float hy = oy - __shfl_up_sync(0xffffffffu, oy, 1);
      const float hz = oz - __shfl_up_sync(0xffffffffu, oz, 1);
      const float gx = ux - __shfl_up_sync(0xffffffffu, ux, 1);
      const float gy = uy - __shfl_up_sync(0xffffffffu, uy, 1);
      const float gz = uz - __shfl_up_sync(0xffffffffu, uz, 1);
      const bool pair = act && lane > 0;
      const uint32_t gap = pair ? __float_as_uint(dot3(hx, hy, hz, hx, hy, hz) +
                                                  dot3(gx, gy, gz, gx, gy, gz))
                                : 0u;
      const uint32_t top = __reduce_max_sync(0xffffffffu, gap);
      const int cut = __ffs(__ballot_sync(0xffffffffu, pair && gap == top)) - 1;  // >= 1
      q1 = make_bundle((int)lane < cut, (cut - 1) >> 1, ox, oy, oz, ux, uy, uz);
      q2 = make_bundle(act && (int)lane >= cut, (cut + n_act - 1) >> 1, ox, oy, oz, ux, uy, uz);
      scan(std::true_type{}, wide);
    }
    if (!act) continue;
    if (a.yarn_id) a.yarn_id[i] = best;
    if (a.t_hit) a.t_hit[i] = best >= 0 ? sbest : 0.f;
    if (best < 0) {
      a.h[i] = a.u[i] = a.v[i] = 0.f;
      if (a.ratio) a.ratio[i] = 0.f;
      for (int c = 0; c < 3; ++c) a.wi[c][i] = a.wo[c][i] = 0.f;
      a.mat_id[i] = -1;
      continue;
    }
    const PieceS p = ps[best];
    const float bx = p.b.y * p.c.z - p.b.z * p.c.y;  // b_ref = t x n_ref
    const float by = p.b.z * p.c.x - p.b.x * p.c.z;
    const float bz = p.b.x * p.c.y - p.b.y * p.c.x;
    // hit relative to the root: the camera distance enters only through one
    // fused multiply-add per coordinate
    const float qx = ox - p.a.x, qy = oy - p.a.y, qz = oz - p.a.z;
    const float xx = fmaf(sbest, dx, qx), xy = fmaf(sbest, dy, qy), xz = fmaf(sbest, dz, qz);
    const float w = dot3(xx, xy, xz, p.b.x, p.b.y, p.b.z);
    const float x_n = dot3(xx, xy, xz, p.c.x, p.c.y, p.c.z);
    const float x_b = dot3(xx, xy, xz, bx, by, bz);
    float u = atan2f(x_b, x_n);
    if (u < 0.f) u += 2.0f * kPi;
    if (u >= 2.0f * kPi) u = 0.f;
    // the azimuthal offset: signed distance of the ray from the axis over R
    const float h0 = fminf(fmaxf(line_offset(p, bx, by, bz, ox, oy, oz, dx, dy, dz), -1.f), 1.f);
    a.h[i] = h0;
    a.u[i] = u;
    a.v[i] = p.c.w + w;
    a.wi[0][i] = -dot3(dx, dy, dz, p.c.x, p.c.y, p.c.z);
    a.wi[1][i] = -dot3(dx, dy, dz, bx, by, bz);
    a.wi[2][i] = -dot3(dx, dy, dz, p.b.x, p.b.y, p.b.z);
    a.wo[0][i] = dot3(a.light[0], a.light[1], a.light[2], p.c.x, p.c.y, p.c.z);
    a.wo[1][i] = dot3(a.light[0], a.light[1], a.light[2], bx, by, bz);
    a.wo[2][i] = dot3(a.light[0], a.light[1], a.light[2], p.b.x, p.b.y, p.b.z);
    a.mat_id[i] = smat[best];
    if (a.ratio) {
      // Sec. 5.3: the differential rays' offsets about the same axis bound
      // the footprint; the record carries its half-width in h
      float r = 0.f;
      if (diff) {
        const float h1 = line_offset(p, bx, by, bz, o1x, o1y, o1z, d1x, d1y, d1z);
        const float h2 = line_offset(p, bx, by, bz, o2x, o2y, o2z, d2x, d2y, d2z);
        const float w1 = fabsf(h1 - h0), w2 = fabsf(h2 - h0);
        r = (isfinite(w1) && isfinite(w2)) ? fmaxf(w1, w2) : 2.0f;
      }
      a.ratio[i] = r;
    }
  }
}

cudaError_t launch_trace_yarns(const bysdf_yarn* yarns, int n_yarns, const TraceArgs& a,
                               cudaStream_t st) {
  const int n_grp = (n_yarns + kGroupPieces - 1) / kGroupPieces;
  const size_t smem = sizeof(PieceS) * (size_t)n_yarns + sizeof(float4) * (size_t)n_grp +
                      sizeof(int32_t) * (size_t)n_yarns;
  // one resident wave: every CTA stages the pieces once.  What the device
  // holds is looked up once per device, shape and size (host time of every
  // call)
  struct Entry {
    int dev, block, per_sm;
    size_t smem;
  };
  static std::mutex mu;
  static std::vector<Entry> seen;
  int dev = 0, sms = 0, per_sm = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess)
    return e;
  const int block = a.n >= (int64_t)sms * 768 ? 768 : 256;
  const void* kernel =
      block == 768 ? (const void*)k_trace_yarns<768> : (const void*)k_trace_yarns<256>;
  {
    std::lock_guard<std::mutex> lock(mu);
    for (const Entry& x : seen)
      if (x.dev == dev && x.block == block && x.smem == smem) per_sm = x.per_sm;
    if (per_sm == 0) {
      int optin = 0;
      if ((e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev)) !=
              cudaSuccess ||
          (e = raise_smem_limit(kernel, smem, (size_t)optin)) != cudaSuccess ||
          (e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, block, smem)) !=
              cudaSuccess)
        return e;
      if (per_sm < 1) return cudaErrorInvalidConfiguration;
      if (seen.size() >= 256) seen.clear();  // sizes come from the caller
      seen.push_back({dev, block, per_sm, smem});
    }
  }
  const int64_t ctas = (std::min(a.n, kMaxLaunch) + block - 1) / block;
  const int grid = (int)std::min<int64_t>(ctas, (int64_t)sms * per_sm);
  for (int64_t at = 0; at < a.n; at += kMaxLaunch) {
    Planes p;
    const float* in[] = {a.o, a.d, a.o1, a.d1, a.o2, a.d2};
    for (int k = 0; k < 18; ++k)
      p.in[k] = in[k / 3] ? in[k / 3] + (k % 3) * a.n + at : nullptr;
    p.n = (uint32_t)std::min(a.n - at, kMaxLaunch);
    p.diff = a.ratio && a.o1 && a.d1 && a.o2 && a.d2;
    for (int c = 0; c < 3; ++c) {
      p.light[c] = a.light[c];
      p.wi[c] = a.wi + c * a.n + at;
      p.wo[c] = a.wo + c * a.n + at;
    }
    p.h = a.h + at;
    p.u = a.u + at;
    p.v = a.v + at;
    p.ratio = a.ratio ? a.ratio + at : nullptr;
    p.t_hit = a.t_hit ? a.t_hit + at : nullptr;
    p.mat_id = a.mat_id + at;
    p.yarn_id = a.yarn_id ? a.yarn_id + at : nullptr;
    void* args[] = {&yarns, &n_yarns, &p};
    if ((e = cudaLaunchKernel(kernel, dim3(grid), dim3(block), args, smem, st)) != cudaSuccess)
      return e;
  }
  return cudaSuccess;
}

}  // namespace bysdf
