// The paper's own box pipeline (Sec. 3.3.1 of arXiv:2401.10878): rough
// contact detection on the lattice, correction of the bounding box, and the
// final sweep of N_c points per direction over the corrected box.
//
//   1. rough detection: the lattice nodes where both signed distances are
//      below half the cell diagonal, sqrt(0.75) dx; their node-index bounds
//      form the rough box (none: no contact).  The node ranges of this mode
//      are widened by that threshold, so the pair box holds all such nodes.
//   2. correction: the rough box widened by sqrt(0.75) dx (every point inside
//      both shapes lies within that distance of such a node) is B0; on each of
//      its six faces an N_c x N_c grid of points (the face's cell centres)
//      casts lines along the inward normal; a line's entry into the overlap
//      (the line clipped exactly against both shapes) is its distance to the
//      contact, and the face moves inward by the smallest one (a face whose
//      lines all miss stays; an axis left empty keeps B0's extent).
//   3. the N_c^3 cell centres of the corrected box are the sample points of
//      the overlap volume, contact point, normal and depth (the lattice
//      path's estimators, each sample weighing its cell's volume), then the
//      force law of Eq. (contact_force_normal).
//
// Three kernels over the pairs the pair builder keeps (pairs whose regions at
// the rough threshold are apart have no rough-contact node and keep their zero
// outputs, and two boxes' node box is cut to the bounding box of their regions'
// intersection): k_box_rough finds the rough boxes and k_box_pairs corrects and
// samples them, one warp per pair; k_box_law runs the force law of the
// overlapping ones, eight per warp pass.  The node tests, the line clipping and
// the sample sweep run in FP32 relative to the particle centres (offsets formed
// in FP64); each face's nearest line is re-clipped in FP64, so the corrected box
// carries no FP32 error; the pair sums, the depth at the deepest sample and the
// force law are FP64.  Bound: instruction issue and, in the force law, the FP64
// pipe.  A warp instruction on that pipe costs ~64 cycles however few lanes are
// active; one warp per pair throughout spent ~600 of them a pair.  Lanes take
// (face, particle) and (component, particle) in the correction (~75), a pass of
// the force law eight pairs: 147 -> 87 us for the three on 1934 cubes at
// N_c = 8 with the contact law (4318 kept pairs, 2031 overlapping).  Blocks of
// four or eight pairs with the FP64 steps of all of them on one warp took 102 us
// (16 resident warps per SM, three of four idle in the FP64 steps); one kernel
// per step took 105 us.
#include <cfloat>
#include <climits>

#include "contact_dev.cuh"
#include "force_law.cuh"
#include "line_clip.cuh"

namespace gbc {

namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kBoxWarps = 8;

// One shape of the pair in FP32, lattice units: centre relative to the pair
// box origin, R^T rows, sizes (inflate included), world planes (polytope),
// plane value at the box origin (wall).
struct ShapeF {
  int kind;
  float c[3];
  float rt[9];
  float sz[3];
  const float4* pl;
  int nf;
};

__device__ __forceinline__ void load_shape(const PairRec& r, bool second, const Shapes& S, const Parts& D, int pid,
                                           float4* sm, ShapeF& s) {
  const int lane = threadIdx.x & 31;
  s.kind = second ? (r.kinds >> 8) : (r.kinds & 0xff);
  const int* ci = second ? r.bi : r.ai;
  const float* cf = second ? r.bf : r.af;
  const float* rt = second ? r.rtb : r.rta;
  const float* sz = second ? r.szb : r.sza;
  for (int k = 0; k < 3; ++k) {
    s.c[k] = static_cast<float>(ci[k]) + cf[k];
    s.sz[k] = sz[k];
  }
  for (int k = 0; k < 9; ++k) s.rt[k] = rt[k];
  s.nf = 0;
  s.pl = sm;
  if (s.kind == KIND_POLY) {
    const int f0 = S.face_off[pid];
    s.nf = S.face_off[pid + 1] - f0;
    if (lane < s.nf) sm[lane] = D.wplane[f0 + lane];
    __syncwarp();
  }
}

// Signed distance (lattice units) at q = point - centre, and the world
// gradient of the active branch (first maximal face).  SET is the context's
// kind set (2: cubes only, 1: spheres, cuboids and walls, 0: every kind): the
// kinds a set cannot hold are compiled out.
template <int SET>
__device__ __forceinline__ float phi_f(const ShapeF& s, const float q[3], float g[3]) {
  if (SET != 2 && s.kind == KIND_SPHERE) {
    const float n2 = fmaf(q[0], q[0], fmaf(q[1], q[1], q[2] * q[2]));
    const float nr = sqrtf(n2);
    const float inv = nr > 0.f ? 1.f / nr : 0.f;
    for (int k = 0; k < 3; ++k) g[k] = q[k] * inv;
    return nr - s.sz[0];
  }
  if (SET != 2 && s.kind == KIND_WALL) {   // q = box-relative point; sz[0] = value at the box origin
    for (int k = 0; k < 3; ++k) g[k] = s.rt[k];
    return fmaf(s.rt[0], q[0], fmaf(s.rt[1], q[1], fmaf(s.rt[2], q[2], s.sz[0])));
  }
  if (SET != 0 || s.kind == KIND_CUBOID || s.kind == KIND_CUBE) {
    float best = -FLT_MAX;
    int kk = 0;
    float sg = 1.f;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const float y = fmaf(s.rt[3 * k], q[0], fmaf(s.rt[3 * k + 1], q[1], s.rt[3 * k + 2] * q[2]));
      const float a = fabsf(y) - s.sz[k];
      if (a > best) { best = a; kk = k; sg = y < 0.f ? -1.f : 1.f; }
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) g[k] = sg * (kk == 0 ? s.rt[k] : (kk == 1 ? s.rt[3 + k] : s.rt[6 + k]));
    return best;
  }
  float best = -FLT_MAX;
  int kk = 0;
  for (int f = 0; f < s.nf; ++f) {
    const float4 e = s.pl[f];
    const float v = fmaf(e.x, q[0], fmaf(e.y, q[1], fmaf(e.z, q[2], -e.w)));
    if (v > best) { best = v; kk = f; }
  }
  const float4 e = s.pl[kk];
  g[0] = e.x; g[1] = e.y; g[2] = e.z;
  return best;
}

// The bounds of a line q + t e (e = +-axis k) inside shapes, FP32: the faces'
// bounds -a/b as the largest lower and the smallest upper one, found with
// reciprocals (b is the same for every line of a grid) and then divided; a
// rounded quotient is a monotone function of the exact one, so dividing only
// the winners gives the extreme of the rounded quotients (but where two faces
// lie within an ulp or two of one another).  Spheres give their bounds directly.
struct LineBounds {
  float lx = -FLT_MAX, la = 0.f, lb = 0.f;   // lower: approximate value, a, b (b = 0: none yet)
  float hx = FLT_MAX, ha = 0.f, hb = 0.f;    // upper
  float t0 = -FLT_MAX, t1 = FLT_MAX;         // spheres
  bool empty = false;
  // the half-line a + b t <= 0 of one face, ib = face_inv(b)
  __device__ __forceinline__ void face(float a, float b, float ib) {
    if (b == 0.f) {
      empty = empty || a > 0.f;
      return;
    }
    const float x = ib != 0.f ? -a * ib : -a / b;
    if (b > 0.f) {
      if (x < hx) { hx = x; ha = a; hb = b; }
    } else {
      if (x > lx) { lx = x; la = a; lb = b; }
    }
  }
  __device__ __forceinline__ float lower() const { return empty ? FLT_MAX : fmaxf(t0, lb != 0.f ? -la / lb : -FLT_MAX); }
  __device__ __forceinline__ float upper() const { return empty ? -FLT_MAX : fminf(t1, hb != 0.f ? -ha / hb : FLT_MAX); }
};
// 1 / b, or 0 where that would overflow (the face is then divided)
__device__ __forceinline__ float face_inv(float b) { return fabsf(b) > 1e-30f ? __fdividef(1.f, b) : 0.f; }

__device__ __forceinline__ float comp3(float a, float b, float c, int k) { return k == 0 ? a : (k == 1 ? b : c); }

// What a shape's faces share on every line along e = sgn axis k.  A box: its
// three axes turned so that face n bounds the line from above (slope b >= 0 along
// e) and face -n from below; a wall: its plane's slope.  flat: a slope too small
// for its reciprocal (then the general form of each face).
struct FaceDirs {
  float n[9], b[3], ib[3];
  bool flat;
};
template <int SET>
__device__ __forceinline__ FaceDirs face_dirs(const ShapeF& s, int k, float sgn) {
  FaceDirs d;
  d.flat = false;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const float b = sgn * comp3(s.rt[3 * a], s.rt[3 * a + 1], s.rt[3 * a + 2], k);
    const bool turn = b < 0.f && !(SET != 2 && s.kind == KIND_WALL);
    d.b[a] = turn ? -b : b;
#pragma unroll
    for (int c = 0; c < 3; ++c) d.n[3 * a + c] = turn ? -s.rt[3 * a + c] : s.rt[3 * a + c];
    d.ib[a] = face_inv(d.b[a]);
    d.flat = d.flat || d.ib[a] == 0.f;
  }
  return d;
}

// The line q + t e (q = start - centre) cut to the shape; SET as for phi_f.
template <int SET>
__device__ __forceinline__ void clip_f(const ShapeF& s, const FaceDirs& d, const float q[3], int k, float sgn,
                                       LineBounds& lb) {
  if (SET != 2 && s.kind == KIND_SPHERE) {
    const float b = sgn * comp3(q[0], q[1], q[2], k);
    const float c = fmaf(q[0], q[0], fmaf(q[1], q[1], q[2] * q[2])) - s.sz[0] * s.sz[0];
    const float disc = b * b - c;
    if (disc < 0.f) {
      lb.empty = true;
      return;
    }
    const float sq = sqrtf(disc);
    lb.t0 = fmaxf(lb.t0, -b - sq);
    lb.t1 = fminf(lb.t1, -b + sq);
    return;
  }
  if (SET != 2 && s.kind == KIND_WALL) {
    lb.face(fmaf(s.rt[0], q[0], fmaf(s.rt[1], q[1], fmaf(s.rt[2], q[2], s.sz[0]))), d.b[0], d.ib[0]);
    return;
  }
  if (SET != 0 || s.kind == KIND_CUBOID || s.kind == KIND_CUBE) {
    if (d.flat) {   // warp-uniform
#pragma unroll 1
      for (int x = 0; x < 6; ++x) {
        const int a = x >> 1;
        const float g = (x & 1) ? -1.f : 1.f;
        const float n0 = g * comp3(s.rt[0], s.rt[3], s.rt[6], a), n1 = g * comp3(s.rt[1], s.rt[4], s.rt[7], a),
                    n2 = g * comp3(s.rt[2], s.rt[5], s.rt[8], a);
        const float b = sgn * comp3(n0, n1, n2, k);
        lb.face(fmaf(n0, q[0], fmaf(n1, q[1], fmaf(n2, q[2], -comp3(s.sz[0], s.sz[1], s.sz[2], a)))), b, face_inv(b));
      }
      return;
    }
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const float n0 = d.n[3 * a], n1 = d.n[3 * a + 1], n2 = d.n[3 * a + 2], h = s.sz[a];
      const float up = fmaf(n0, q[0], fmaf(n1, q[1], fmaf(n2, q[2], -h)));
      const float dn = fmaf(-n0, q[0], fmaf(-n1, q[1], fmaf(-n2, q[2], -h)));
      const float xu = -up * d.ib[a], xl = dn * d.ib[a];
      if (xu < lb.hx) { lb.hx = xu; lb.ha = up; lb.hb = d.b[a]; }
      if (xl > lb.lx) { lb.lx = xl; lb.la = dn; lb.lb = -d.b[a]; }
    }
    return;
  }
  for (int f = 0; f < s.nf; ++f) {
    const float4 e = s.pl[f];
    const float b = sgn * comp3(e.x, e.y, e.z, k);
    lb.face(fmaf(e.x, q[0], fmaf(e.y, q[1], fmaf(e.z, q[2], -e.w))), b, face_inv(b));
  }
}

// [lo, hi] (nodes along the box axis u) cut to where the shape's distance lies
// below T on the line through box node (c with c[u] = 0); inv: clip_inv of a
// box's slopes along u.
template <int SET>
__device__ __forceinline__ void clip_nodes_f(const ShapeF& s, const float inv[3], int u, const float q[3], float T,
                                             float& lo, float& hi) {
  if (SET != 2 && s.kind == KIND_SPHERE) {
    const float qu = comp3(q[0], q[1], q[2], u);
    const float q2 = fmaf(q[0], q[0], fmaf(q[1], q[1], q[2] * q[2]));
    clip_ball(-qu, fmaxf(fmaf(-qu, qu, q2), 0.f), s.sz[0], T, lo, hi);
    return;
  }
  if (SET != 2 && s.kind == KIND_WALL) {
    const float m = comp3(s.rt[0], s.rt[1], s.rt[2], u);
    clip_half(m, inv[0], fmaf(s.rt[0], q[0], fmaf(s.rt[1], q[1], fmaf(s.rt[2], q[2], s.sz[0]))), T, lo, hi);
    return;
  }
  if (SET != 0 || s.kind == KIND_CUBOID || s.kind == KIND_CUBE) {
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const float t = comp3(s.rt[3 * a], s.rt[3 * a + 1], s.rt[3 * a + 2], u);
      const float p = fmaf(s.rt[3 * a], q[0], fmaf(s.rt[3 * a + 1], q[1], s.rt[3 * a + 2] * q[2]));
      clip_slab(t, inv[a], p, s.sz[a] + T, lo, hi);
    }
    return;
  }
  for (int f = 0; f < s.nf; ++f) {
    const float4 e = s.pl[f];
    const float m = comp3(e.x, e.y, e.z, u);
    clip_half(m, clip_inv(m), fmaf(e.x, q[0], fmaf(e.y, q[1], fmaf(e.z, q[2], -e.w))), T, lo, hi);
  }
}

// A bound -a/b of a line, compared with others by products (b < 0: from below,
// b > 0: from above, b = 0: none).
struct Frac {
  double a = 0.0, b = 0.0;
  // the larger of two lower bounds: -a/b < -a'/b'  <=>  a' b < a b' (b b' > 0)
  __device__ __forceinline__ void raise(const Frac& o) {
    if (o.b != 0.0 && (b == 0.0 || o.a * b < a * o.b)) *this = o;
  }
  // the smaller of two upper bounds: -a'/b' < -a/b  <=>  a' b > a b'
  __device__ __forceinline__ void lower(const Frac& o) {
    if (o.b != 0.0 && (b == 0.0 || o.a * b > a * o.b)) *this = o;
  }
};

// The world plane n . x <= e[3] of a body plane e = (n, d), of a particle at X.
__device__ __forceinline__ void world_plane_d(const Params& P, const double* e, const double* R, const double X[3],
                                              double o[4]) {
  const double n0 = (R[0] * e[0] + R[1] * e[1]) + R[2] * e[2];
  const double n1 = (R[3] * e[0] + R[4] * e[1]) + R[5] * e[2];
  const double n2 = (R[6] * e[0] + R[7] * e[1]) + R[8] * e[2];
  o[0] = n0;
  o[1] = n1;
  o[2] = n2;
  o[3] = ((n0 * X[0] + n1 * X[1]) + n2 * X[2]) + e[3] + P.inflate;
}

// The same of every face of polytope (or wall) `pid`, a face per lane (the
// caller syncs the warp).  Formed by the lane of each line and particle, one face
// after the other, they were ~22 of ~36 FP64 instructions per face of a pair's
// chain: 81 -> 72 us on 86 mixed particles between walls at N_c = 6 (the time
// of one pair), 250 -> 239 us on 241 mixed at N_c = 16.
__device__ __forceinline__ void stage_planes_d(const Params& P, const Shapes& S, const Parts& D, int pid,
                                               const double X[3], double (*pl)[4]) {
  const int lane = threadIdx.x & 31, type = S.type[pid];
  if (type == 0 || type == 1) return;
  const int f0 = S.face_off[pid], nf = S.face_off[pid + 1] - f0;
  if (lane < nf) world_plane_d(P, S.planes + 4 * (f0 + lane), D.R + 9 * static_cast<size_t>(pid), X, pl[lane]);
}

// FP64 bounds of the line p + t e (e = sgn axis k, physical units) inside
// particle / wall `pid`, the same clipping as the FP32 form; used for each
// face's nearest line.  Returns false when the line misses the shape.  SET as
// for phi_f; pl: a polytope's (or wall's) world planes (SET 0, stage_planes_d).
template <int SET>
__device__ __forceinline__ bool clip_d(const Params& P, const Shapes& S, const Parts& D, int pid, const double X[3],
                                       const double p[3], int k, double sgn, const double (*pl)[4], Frac& lo,
                                       Frac& hi) {
  const int type = SET == 2 ? 1 : S.type[pid];
  const double* R = D.R + 9 * static_cast<size_t>(pid);
  const double q0 = p[0] - X[0], q1 = p[1] - X[1], q2 = p[2] - X[2];
  bool empty = false;
  // the half-line a + b t <= 0 of one face along the line
  auto bound = [&](double a, double b) {
    const long long s = __double_as_longlong(b);
    if (s << 1 == 0) {
      empty = empty || a > 0.0;
    } else if (s > 0) {
      hi.lower(Frac{a, b});
    } else {
      lo.raise(Frac{a, b});
    }
  };
  if (SET != 2 && type == 0) {   // sphere
    const double r = S.param[3 * pid] + P.inflate;
    const double b = sgn * (k == 0 ? q0 : (k == 1 ? q1 : q2));
    const double c = (q0 * q0 + q1 * q1 + q2 * q2) - r * r;
    const double disc = b * b - c;
    if (disc < 0.0) return false;
    const double sq = sqrt(disc);
    lo = Frac{-b - sq, -1.0};
    hi = Frac{b - sq, 1.0};
    return true;
  }
  if (SET == 2 || type == 1) {   // cuboid: faces +-R e_a share n = R e_a and d = n . (p - X)
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const double n0 = R[a], n1 = R[3 + a], n2 = R[6 + a];
      const double d = (n0 * q0 + n1 * q1) + n2 * q2;
      const double h = S.param[3 * pid + a] + P.inflate;
      const double b = sgn * (k == 0 ? n0 : (k == 1 ? n1 : n2));
      bound(d - h, b);     // n . (x - X) <= h
      bound(-d - h, -b);   // -n . (x - X) <= h
    }
  } else {   // polytope, or a wall's single plane
    const int f0 = S.face_off[pid], nf = S.face_off[pid + 1] - f0;
    for (int f = 0; f < nf; ++f) {
      double e[4];
      if constexpr (SET == 0) {
#pragma unroll
        for (int x = 0; x < 4; ++x) e[x] = pl[f][x];
      } else {
        world_plane_d(P, S.planes + 4 * (f0 + f), R, X, e);
      }
      bound(((e[0] * p[0] + e[1] * p[1]) + e[2] * p[2]) - e[3], sgn * (k == 0 ? e[0] : (k == 1 ? e[1] : e[2])));
    }
  }
  return !empty;
}

// floor(x / d) for x < 2^18 and 1 <= d <= 64 from rcp = recip_u(d): the
// reciprocal is at most 2^-32 too large, and x times that is below 1 / d (d = 1:
// the reciprocal 2^32 is stored as 0).
__device__ __forceinline__ unsigned recip_u(int d) { return 0xffffffffu / static_cast<unsigned>(d) + 1u; }
__device__ __forceinline__ int div_u(int x, unsigned rcp) {
  return rcp != 0u ? static_cast<int>(__umulhi(static_cast<unsigned>(x), rcp)) : x;
}

__device__ __forceinline__ float warp_sum_f(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
  return v;
}

// Component c of the partner's position in the pair's image.
__device__ __forceinline__ double image_x(const Params& P, const Parts& D, const PairRec& r, int j, int c) {
  return D.X[3 * j + c] - (r.shift[c] == 0 ? 0.0 : (r.shift[c] > 0 ? P.L[c] : -P.L[c]));
}

// The warp stages the pair record of tile-list entry t.
__device__ __forceinline__ void stage_rec(const Lists& W, const Params& P, int t, PairRec* dst) {
  const int lane = threadIdx.x & 31;
  __syncwarp();
  if (lane < kPairRecWords / 4)
    reinterpret_cast<int4*>(dst)[lane] = reinterpret_cast<const int4*>(W.tiles + checked_index(W.err, t, P.max_tiles, 0))[lane];
  __syncwarp();
}

// The rough boxes (step 1): one warp per kept pair.  Each lane clips node lines
// along the box's longest axis to the nodes where both distances lie below the
// threshold (plus the clip margin, far above the FP32 rounding) and tests nodes
// from both ends inwards until one qualifies, with the distances of a walk over
// every node; the first and the last qualifying node of each line bound the
// box as all of them would.
template <int SET>
__global__ void __launch_bounds__(kBoxWarps * 32, 2) k_box_rough(Params P, Shapes S, Parts D, Lists W) {
  __shared__ float4 s_pl[SET == 0 ? kBoxWarps : 1][2][kMaxFaces];
  __shared__ __align__(16) PairRec s_rec[kBoxWarps];
  pdl_begin();
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int ntl = W.counters[1];
  if (ntl > P.max_tiles) return;   // capacity exceeded: the step reports ECAPACITY
  const float T = kRoughT + P.clip_margin;
  for (int t = blockIdx.x + gridDim.x * wid; t < ntl; t += gridDim.x * kBoxWarps) {
    stage_rec(W, P, t, &s_rec[wid]);
    const PairRec& r = s_rec[wid];
    if (!record_in_bounds(P, W.err, r, true)) continue;   // warp-uniform (checked build only)
    ShapeF A, B;
    load_shape(r, false, S, D, r.i, s_pl[SET == 0 ? wid : 0][0], A);
    load_shape(r, true, S, D, r.j, s_pl[SET == 0 ? wid : 0][1], B);
    const int u = r.axis, v = u == 2 ? 0 : u + 1;
    float ia[3], ib[3];   // a box's inverse slopes along u
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      ia[a] = clip_inv(comp3(A.rt[3 * a], A.rt[3 * a + 1], A.rt[3 * a + 2], u));
      ib[a] = clip_inv(comp3(B.rt[3 * a], B.rt[3 * a + 1], B.rt[3 * a + 2], u));
    }
    const int du = r.dim[u], dv = r.dim[v], nlines = r.nitems;
    const float inv_dv = __fdividef(1.f, static_cast<float>(dv));
    // node-relative offsets of a box node (as the walk of every node forms them)
    const int ai[3] = {r.ai[0], r.ai[1], r.ai[2]}, bi[3] = {r.bi[0], r.bi[1], r.bi[2]};
    const float af[3] = {r.af[0], r.af[1], r.af[2]}, bf[3] = {r.bf[0], r.bf[1], r.bf[2]};
    auto offsets = [&](int cu, int cv, int cw, float qa[3], float qb[3]) {
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const int c = k == u ? cu : (k == v ? cv : cw);
        qa[k] = static_cast<float>(c - ai[k]) - af[k];
        qb[k] = B.kind == KIND_WALL ? static_cast<float>(c) : static_cast<float>(c - bi[k]) - bf[k];
      }
    };
    int mn[3] = {INT_MAX, INT_MAX, INT_MAX}, mx[3] = {INT_MIN, INT_MIN, INT_MIN};   // along u, v, w
    for (int l0 = 0; l0 < nlines; l0 += 32) {
      const int l = l0 + lane;
      if (l >= nlines) break;   // (no warp-wide operation inside the loop)
      int cv;
      const int cw = div_small(l, dv, inv_dv, &cv);
      float qa[3], qb[3], g[3];
      offsets(0, cv, cw, qa, qb);
      float lo = 0.f, hi = static_cast<float>(du - 1);
      clip_nodes_f<SET>(A, ia, u, qa, T, lo, hi);
      clip_nodes_f<SET>(B, ib, u, qb, T, lo, hi);
      int s0;
      const int n = clip_nodes(lo, hi, 0, du, &s0);
      int s1 = s0 + n - 1;
      auto rough = [&](int cu) {
        offsets(cu, cv, cw, qa, qb);
        return phi_f<SET>(A, qa, g) < kRoughT && phi_f<SET>(B, qb, g) < kRoughT;
      };
      while (s0 <= s1 && !rough(s0)) ++s0;
      if (s0 > s1) continue;
      while (s1 > s0 && !rough(s1)) --s1;
      mn[0] = min(mn[0], s0);
      mx[0] = max(mx[0], s1);
      mn[1] = min(mn[1], cv);
      mx[1] = max(mx[1], cv);
      mn[2] = min(mn[2], cw);
      mx[2] = max(mx[2], cw);
    }
    __syncwarp();
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      mn[k] = __reduce_min_sync(kFull, mn[k]);
      mx[k] = __reduce_max_sync(kFull, mx[k]);
    }
    if (mn[0] > mx[0]) continue;   // no rough contact: the pair builder's zero outputs stay
    if (lane == 0) {
      const int slot = checked_index(W.err, atomicAdd(&W.counters[2], 1), P.max_pairs, 0);
      // from (u, v, w) to (x, y, z): axis k sits at (k - u) mod 3
      int lo3[3], hi3[3];
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const int c = k == u ? 0 : (k == v ? 1 : 2);
        lo3[k] = c == 0 ? mn[0] : (c == 1 ? mn[1] : mn[2]);
        hi3[k] = c == 0 ? mx[0] : (c == 1 ? mx[1] : mx[2]);
      }
      int4* o = reinterpret_cast<int4*>(W.box_work + slot);   // t, bounds
      o[0] = make_int4(t, lo3[0], lo3[1], lo3[2]);
      o[1] = make_int4(hi3[0], hi3[1], hi3[2], 0);
    }
  }
}

// The largest lower and smallest upper bound of a box line inside a shape from
// reciprocals alone (relative error below 1e-6 of the value), with the face
// values of clip_f.  Returns false where a face is too parallel to the line
// for its reciprocal (warp-uniform: the slopes are the same on every line).
template <int SET>
__device__ __forceinline__ bool approx_f(const ShapeF& s, const FaceDirs& d, const float q[3], int k, float sgn,
                                         float& lo, float& hi) {
  auto face = [&](float a, float b, float ib) {
    const float x = -a * ib;
    if (b > 0.f) hi = fminf(hi, x);
    else lo = fmaxf(lo, x);
    return ib != 0.f;
  };
  if (SET != 2 && s.kind == KIND_SPHERE) {
    LineBounds lb;
    clip_f<SET>(s, d, q, k, sgn, lb);
    lo = lb.empty ? FLT_MAX : fmaxf(lo, lb.t0);
    hi = lb.empty ? -FLT_MAX : fminf(hi, lb.t1);
    return true;
  }
  if (SET != 2 && s.kind == KIND_WALL)
    return face(fmaf(s.rt[0], q[0], fmaf(s.rt[1], q[1], fmaf(s.rt[2], q[2], s.sz[0]))), d.b[0], d.ib[0]);
  if (SET != 0 || s.kind == KIND_CUBOID || s.kind == KIND_CUBE) {
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const float n0 = d.n[3 * a], n1 = d.n[3 * a + 1], n2 = d.n[3 * a + 2], h = s.sz[a];
      hi = fminf(hi, -fmaf(n0, q[0], fmaf(n1, q[1], fmaf(n2, q[2], -h))) * d.ib[a]);
      lo = fmaxf(lo, fmaf(-n0, q[0], fmaf(-n1, q[1], fmaf(-n2, q[2], -h))) * d.ib[a]);
    }
    return !d.flat;
  }
  bool ok = true;
  for (int f = 0; f < s.nf; ++f) {
    const float4 e = s.pl[f];
    const float b = sgn * comp3(e.x, e.y, e.z, k);
    ok = face(fmaf(e.x, q[0], fmaf(e.y, q[1], fmaf(e.z, q[2], -e.w))), b, face_inv(b)) && ok;
  }
  return ok;
}

// Each face's nearest line of the warp's pair in FP32 (the first of equals): a
// sweep of all lines with reciprocals; the lines within its error of the
// smallest are then compared by the rounded quotients (clip_f), unless there is
// only one.  off: a corner component's offset on lane (component, upper corner,
// particle); spl, lnl: line spacing and length on lane (axis).  The lanes with
// ff = f keep face f's.  KS: the kinds of this pair (2: two boxes), as SET.
template <int KS>
__device__ __forceinline__ void nearest_lines(const ShapeF& A, const ShapeF& B, float off, float spl, float lnl, int Nc,
                                              unsigned rcp_nc, int ff, unsigned& my_key, int& my_line) {
  const int lane = threadIdx.x & 31, nl = Nc * Nc;
#pragma unroll 1
  for (int f = 0; f < 6; ++f) {
    const int k = f >> 1, side = f & 1;
    const float sgn = side == 0 ? 1.f : -1.f;
    float ca[3], cb[3];
#pragma unroll
    for (int x = 0; x < 3; ++x) {
      const int src = x + ((x == k && side == 1) ? 3 : 0);
      ca[x] = __shfl_sync(kFull, off, src);
      cb[x] = __shfl_sync(kFull, off, src + 6);
    }
    const int u = k == 0 ? 1 : 0, v = k == 2 ? 1 : 2;
    const float du = __shfl_sync(kFull, spl, u), dv = __shfl_sync(kFull, spl, v), lenl = __shfl_sync(kFull, lnl, k);
    const FaceDirs da = face_dirs<KS>(A, k, sgn), db = face_dirs<KS>(B, k, sgn);
    auto start = [&](int l, float qa[3], float qb[3]) {
      const int a = div_u(l, rcp_nc), b = l - a * Nc;
      const float ou = (static_cast<float>(a) + 0.5f) * du, ov = (static_cast<float>(b) + 0.5f) * dv;
      // (selects, not a runtime index: the arrays stay in registers)
      const float o0 = u == 0 ? ou : 0.f, o1 = u == 1 ? ou : (v == 1 ? ov : 0.f), o2 = v == 2 ? ov : 0.f;
      qa[0] = ca[0] + o0; qa[1] = ca[1] + o1; qa[2] = ca[2] + o2;
      qb[0] = cb[0] + o0; qb[1] = cb[1] + o1; qb[2] = cb[2] + o2;
    };
    float p1 = FLT_MAX, p2 = FLT_MAX, sure = FLT_MAX;   // smallest two possible entries, smallest certain one
    int l1 = 0x7fffffff;
    bool ok = true;
    for (int l = lane; l < nl; l += 32) {
      float qa[3], qb[3], lo = -FLT_MAX, hi = FLT_MAX;
      start(l, qa, qb);
      ok = approx_f<KS>(A, da, qa, k, sgn, lo, hi) && ok;
      ok = approx_f<KS>(B, db, qb, k, sgn, lo, hi) && ok;
      const float tin = fmaxf(lo, 0.f), tout = fminf(hi, lenl);
      const float m = 1e-6f * (tin + lenl + 1.f);
      if (tin - m <= tout) {
        if (tin < p1) {
          p2 = p1;
          p1 = tin;
          l1 = l;
        } else {
          p2 = fminf(p2, tin);
        }
        if (tin + m <= tout) sure = fminf(sure, tin);
      }
    }
    __syncwarp();
    const float smin = __uint_as_float(__reduce_min_sync(kFull, __float_as_uint(sure)));   // (>= 0: bits order as values)
    const float thr = smin + 2e-6f * (smin + lenl + 1.f);
    const bool near = p1 <= thr;
    const unsigned nears = __ballot_sync(kFull, near && p1 < FLT_MAX);
    const bool all = __any_sync(kFull, !ok || (p1 < FLT_MAX && smin == FLT_MAX) || (near && p2 < FLT_MAX && p2 <= thr));
    float best = FLT_MAX;
    int bestl = 0x7fffffff;
    if (!all && __popc(nears) <= 1) {
      if (near && p1 < FLT_MAX) {
        best = p1;
        bestl = l1;
      }
    } else {
      // every line of the face, or the lane's only candidate
      for (int l = all ? lane : (near ? l1 : nl); l < nl; l += all ? 32 : nl) {
        float qa[3], qb[3];
        start(l, qa, qb);
        LineBounds lb;
        clip_f<KS>(A, da, qa, k, sgn, lb);
        clip_f<KS>(B, db, qb, k, sgn, lb);
        const float tin = fmaxf(lb.lower(), 0.f), tout = fminf(lb.upper(), lenl);
        if (tin <= tout && tin < best) { best = tin; bestl = l; }
      }
      __syncwarp();
    }
    const unsigned key = best < FLT_MAX ? __float_as_uint(best) : 0xffffffffu;
    const unsigned kmin = __reduce_min_sync(kFull, key);
    const int lmin = __reduce_min_sync(kFull, key == kmin ? bestl : 0x7fffffff);
    if (ff == f) {
      my_key = kmin;
      my_line = lmin;
    }
  }
}

// Per-lane sums over the N_c^3 sample points of the warp's pair: weight, first
// moments of the sample indices (exact integers in sharp mode), band terms of
// the normal, deepest sample.
struct SampleSums {
  float cnt = 0.f, m0 = 0.f, m1 = 0.f, m2 = 0.f, g0 = 0.f, g1 = 0.f, g2 = 0.f, bestf = -FLT_MAX;
  int bestidx = 0x7fffffff;
};
template <int KS>
__device__ __forceinline__ SampleSums sweep_samples(const Params& P, const ShapeF& A, const ShapeF& B, const float oA[3],
                                                    const float oB[3], const float st[3], int Nc, unsigned rcp_nc) {
  const int lane = threadIdx.x & 31, ns = Nc * Nc * Nc;
  const float hw = 0.5f * P.wdx_l;
  const float inv_w = P.inv_w;
  float cnt = 0.f, m0 = 0.f, m1 = 0.f, m2 = 0.f, g0 = 0.f, g1 = 0.f, g2 = 0.f, bestf = -FLT_MAX;
  int bestidx = 0x7fffffff;
  for (int sidx = lane; sidx < ns; sidx += 32) {
    const int iyz = div_u(sidx, rcp_nc), ix = sidx - iyz * Nc;
    const int iz = div_u(iyz, rcp_nc), iy = iyz - iz * Nc;
    const float t[3] = {static_cast<float>(ix), static_cast<float>(iy), static_cast<float>(iz)};
    float qa[3], qb[3], ga[3], gb[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      qa[k] = fmaf(t[k], st[k], oA[k]);
      qb[k] = fmaf(t[k], st[k], oB[k]);
    }
    const float fa = phi_f<KS>(A, qa, ga), fb = phi_f<KS>(B, qb, gb);
    if (fmaxf(fa, fb) >= hw) continue;   // no weight and no band term
    const float ta = __saturatef(fmaf(fa, -inv_w, 0.5f)), tb = __saturatef(fmaf(fb, -inv_w, 0.5f));
    float ww, ma, mb;
    if (P.smooth) {
      const float ha = ta * ta * fmaf(-2.f, ta, 3.f), hb = tb * tb * fmaf(-2.f, tb, 3.f);
      ww = ha * hb;
      ma = fmaf(-ta, ta, ta) * hb;
      mb = ha * fmaf(-tb, tb, tb);
    } else {
      ww = (fa <= 0.f && fb <= 0.f) ? 1.f : 0.f;
      ma = fb <= 0.f ? fmaf(-ta, ta, ta) : 0.f;
      mb = fa <= 0.f ? fmaf(-tb, tb, tb) : 0.f;
    }
    cnt += ww;   // moments of the sample indices (exact integers in sharp mode)
    m0 = fmaf(ww, t[0], m0);
    m1 = fmaf(ww, t[1], m1);
    m2 = fmaf(ww, t[2], m2);
    g0 += ma * ga[0] - mb * gb[0];
    g1 += ma * ga[1] - mb * gb[1];
    g2 += ma * ga[2] - mb * gb[2];
    const float f = -(fa + fb);
    if (ww > 0.f && (f > bestf || (f == bestf && sidx < bestidx))) { bestf = f; bestidx = sidx; }
  }
  SampleSums s;
  s.cnt = cnt; s.m0 = m0; s.m1 = m1; s.m2 = m2; s.g0 = g0; s.g1 = g1; s.g2 = g2;
  s.bestf = bestf; s.bestidx = bestidx;
  return s;
}

// Steps 2 and 3, one warp per pair with a rough contact.  The FP64 steps have a
// lane per (corner component and particle) or per (face and particle); their
// ~75 warp instructions a pair run on the FP64 pipe beside the other warps'
// FP32 line and sample tests.
template <int SET, bool HIST>
__global__ void __launch_bounds__(kBoxWarps * 32, 2) k_box_pairs(Params P, Shapes S, Parts D, Lists W) {
  __shared__ float4 s_pl[SET == 0 ? kBoxWarps : 1][2][kMaxFaces];
  __shared__ __align__(16) PairRec s_rec[kBoxWarps];
  __shared__ double s_b0[kBoxWarps][6];   // B0: lower, upper
  __shared__ double s_x[kBoxWarps][6];    // both centres
  __shared__ double s_pd[SET == 0 ? kBoxWarps : 1][2][kMaxFaces][4];   // polytopes' world planes (re-clip)
  pdl_begin();
  if (W.counters[1] > P.max_tiles) return;   // capacity exceeded: the step reports ECAPACITY
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int nc = min(W.counters[2], P.max_pairs);
  const int Nc = P.box_res;
  const unsigned rcp_nc = recip_u(Nc);
  const double inv_nc = 1.0 / Nc, s64 = sqrt(0.75) * P.dx;
  // lanes 0 .. 11 as (component, upper corner, particle) and as (face, particle)
  const int l12 = min(lane, 11), kc = l12 % 3, up = (l12 / 3) & 1, second = l12 / 6;
  const int ff = l12 % 6, fk = ff >> 1, fside = ff & 1;
  // (consecutive contacts on different SMs: the last, partly filled round spreads over all of them)
  for (int c = blockIdx.x + gridDim.x * wid; c < nc; c += gridDim.x * kBoxWarps) {
    BoxWork& w = W.box_work[c];
    stage_rec(W, P, w.t, &s_rec[wid]);
    const PairRec& r = s_rec[wid];
    const int i = checked_index(W.err, r.i, P.n, 0), j = checked_index(W.err, r.j, P.n + P.nwall, 0);
    ShapeF A, B;
    load_shape(r, false, S, D, i, s_pl[SET == 0 ? wid : 0][0], A);
    load_shape(r, true, S, D, j, s_pl[SET == 0 ? wid : 0][1], B);
    const bool wallj = SET != 2 && B.kind == KIND_WALL;
    // 2. B0 (physical, the rough box's nodes +- sqrt(0.75) dx) and the offsets
    // of its corners from both centres, the line spacings and lengths as FP32
    const int rlo = kc == 0 ? r.lo[0] : (kc == 1 ? r.lo[1] : r.lo[2]);
    const double xa = D.X[3 * i + kc];
    const double xp = second ? image_x(P, D, r, j, kc) : xa;
    double b0 = fl::int_to_double(rlo + w.bounds[3 * up + kc]) * P.dx + (up ? s64 : -s64);
    if (HIST) {
      // contact history (Sec. 4.3.3): an ongoing contact's last corrected box
      // (relative to X_i) is the warm start: moved with particle i and widened
      // by sqrt(0.75) dx, it cuts B0 down per axis (unless the cut leaves nothing)
      const int rd = W.counters[kStepCounter] & 1;
      const size_t base = (static_cast<size_t>(rd) * P.n + i) * P.max_nbr;
      const int cnt = min(W.hist_n[static_cast<size_t>(rd) * P.n + i], P.max_nbr);
      int hit = -1;
      for (int m = lane; m < cnt; m += 32)
        if (W.hist_j[base + m] == j) hit = m;
      hit = __reduce_max_sync(kFull, hit);
      if (hit >= 0) {
        const double wv = __dadd_rn(__dadd_rn(xa, W.hist_box[6 * (base + hit) + 3 * up + kc]), up ? s64 : -s64);
        const double cand = (order_key(wv) < order_key(b0)) == (up != 0) ? wv : b0;
        const double other = __shfl_sync(kFull, cand, up ? l12 - 3 : l12 + 3);
        if ((order_key(cand) > order_key(other)) == (up != 0) && cand != other) b0 = cand;
      }
    }
    const double b0o = __shfl_sync(kFull, b0, up ? l12 - 3 : l12 + 3);
    const double len = up ? b0 - b0o : b0o - b0;
    const float off = wallj && second ? narrow(b0 * P.inv_dx - rlo) : narrow((b0 - xp) * P.inv_dx);
    const float lnl = narrow(len * P.inv_dx), spl = narrow(len * (P.inv_dx * inv_nc));
    if (lane < 12) {
      s_b0[wid][3 * up + kc] = b0;
      s_x[wid][3 * second + kc] = xp;
    }
    __syncwarp();
    // (two boxes, the usual pair, without the other kinds' branches)
    const bool boxes = SET == 2 || ((A.kind == KIND_CUBE || A.kind == KIND_CUBOID) && (B.kind == KIND_CUBE || B.kind == KIND_CUBOID));
    if constexpr (SET == 0) {
#pragma unroll
      for (int x = 0; x < 2; ++x) stage_planes_d(P, S, D, x == 0 ? i : j, s_x[wid] + 3 * x, s_pd[wid][x]);
      __syncwarp();
    }
    unsigned my_key = 0xffffffffu;
    int my_line = 0;
    if (boxes) nearest_lines<2>(A, B, off, spl, lnl, Nc, rcp_nc, ff, my_key, my_line);
    else if constexpr (SET != 2) nearest_lines<SET>(A, B, off, spl, lnl, Nc, rcp_nc, ff, my_key, my_line);
    // the nearest lines re-clipped in FP64, lane (face, particle): each
    // particle's bounds as fractions -a/b, the larger lower and the smaller
    // upper one of the two particles divided side by side
    double shift = 0.0;
    {
      const double blk = s_b0[wid][fk], bhk = s_b0[wid][3 + fk];
      const bool some = my_key != 0xffffffffu;
      Frac lo, hi;
      bool empty = false;
      if (some) {
        const int a = div_u(my_line, rcp_nc), b = my_line - a * Nc;
        const int u = fk == 0 ? 1 : 0;
        double p[3], X[3];
#pragma unroll
        for (int x = 0; x < 3; ++x) {
          const double l = s_b0[wid][x], h = s_b0[wid][3 + x];
          const double ic = fl::int_to_double(x == u ? a : b) + 0.5;
          p[x] = x == fk ? (fside == 0 ? l : h) : l + ic * (h - l) * inv_nc;
          X[x] = s_x[wid][3 * second + x];
        }
        empty = !clip_d<SET>(P, S, D, second ? j : i, X, p, fk, fside == 0 ? 1.0 : -1.0,
                                 s_pd[SET == 0 ? wid : 0][second], lo, hi);
      }
      // (lanes l and l + 6: the two particles of a face)
      const int o = lane < 6 ? lane + 6 : (lane < 12 ? lane - 6 : lane);
      const Frac olo{__shfl_sync(kFull, lo.a, o), __shfl_sync(kFull, lo.b, o)};
      const Frac ohi{__shfl_sync(kFull, hi.a, o), __shfl_sync(kFull, hi.b, o)};
      empty = __shfl_sync(kFull, empty ? 1 : 0, o) != 0 || empty;
      lo.raise(olo);
      hi.lower(ohi);
      // lanes 0 .. 5 divide the entry, lanes 6 .. 11 the exit
      const Frac fr = second ? hi : lo;
      const bool some_fr = fr.b != 0.0;
      const double t = some_fr ? -fr.a / fr.b : 0.0;
      const double t_in = !some_fr || order_key(t) < 0 ? 0.0 : t;         // max(entry, 0)
      const double ln = bhk - blk;
      const double t_out_own = !some_fr || order_key(t) > order_key(ln) ? ln : t;   // min(exit, length)
      const double t_out = __shfl_sync(kFull, t_out_own, o);
      if (some)
        shift = !empty && order_key(t_in) <= order_key(t_out) ? t_in
                                                              : static_cast<double>(__uint_as_float(my_key)) * P.dx;
    }
    // the corrected box and 3. the first sample's offsets from each centre (and
    // the box origin) in FP64, rounded once: component kc and particle `second`
    float smp, sst;
    {
      const double cut0 = __shfl_sync(kFull, shift, 2 * kc), cut1 = __shfl_sync(kFull, shift, 2 * kc + 1);
      const double bl = s_b0[wid][kc], bh = s_b0[wid][3 + kc];
      double l = bl + cut0, h = bh - cut1;
      if (!(order_key(l) <= order_key(h))) {
        l = bl;
        h = bh;
      }
      const double st = (h - l) * inv_nc, first = l + 0.5 * st;
      smp = wallj && second ? narrow(first * P.inv_dx - rlo) : narrow((first - xp) * P.inv_dx);
      sst = narrow(st * P.inv_dx);
      if (lane < 3) {
        w.box.lo[lane] = l;
        w.box.hi[lane] = h;
        w.box.step[lane] = st;
      }
    }
    float oA[3], oB[3], st[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      oA[k] = __shfl_sync(kFull, smp, k);
      oB[k] = __shfl_sync(kFull, smp, 6 + k);
      st[k] = __shfl_sync(kFull, sst, k);
    }
    SampleSums sm;
    if (boxes) sm = sweep_samples<2>(P, A, B, oA, oB, st, Nc, rcp_nc);
    else if constexpr (SET != 2) sm = sweep_samples<SET>(P, A, B, oA, oB, st, Nc, rcp_nc);
    __syncwarp();
    const float cnt = warp_sum_f(sm.cnt);
    if (lane == 0) W.oflag[c] = cnt > 0.f ? 1 : 0;   // (by contact here, not by pair)
    if (!(cnt > 0.f)) continue;   // the pair builder's zero outputs stay
    const float m0 = warp_sum_f(sm.m0), m1 = warp_sum_f(sm.m1), m2 = warp_sum_f(sm.m2);
    const float g0 = warp_sum_f(sm.g0), g1 = warp_sum_f(sm.g1), g2 = warp_sum_f(sm.g2);
    const int bk = __float_as_int(sm.bestf);   // order-preserving key (-FLT_MAX: no sample, the lowest)
    const int key = bk >= 0 ? bk : (bk ^ 0x7fffffff);
    const int kmax = __reduce_max_sync(kFull, key);
    const int bestidx = __reduce_min_sync(kFull, key == kmax ? sm.bestidx : 0x7fffffff);
    // the pair's sums, entry c of the overlap list (dim: the samples per axis)
    OvlRec& e = W.olist[c];
    if (lane < 7)
      e.s[lane] = widen(lane == 0 ? cnt : (lane == 1 ? m0 : (lane == 2 ? m1 : (lane == 3 ? m2 : (lane == 4 ? g0 : (lane == 5 ? g1 : g2))))));
    if (lane == 7) {
      e.q = r.pair;
      e.idx = bestidx;
      e.i = r.i;
      e.j = r.j;
    }
    if (lane >= 8 && lane < 11) {
      e.lo[lane - 8] = 0;
      e.dim[lane - 8] = Nc;
      e.shift[lane - 8] = r.shift[lane - 8];
    }
  }
}

// Step 4: FP64 pair results and the force law, four lanes per overlapping pair;
// each warp gathers the overlapping ones of its range of contacts first.
template <int SET, bool LAW>
__global__ void __launch_bounds__(32) k_box_law(Params P, Shapes S, Parts D, Lists W, const double* __restrict__ vel,
                                                double* __restrict__ pair_out) {
  __shared__ __align__(16) OvlRec s_ovl[kForcePairsPerPass];
  __shared__ BoxGeom s_box[kForcePairsPerPass];
  __shared__ int s_q[32 + kForcePairsPerPass];
  pdl_begin();
  if (W.counters[1] > P.max_tiles) return;   // capacity exceeded: the step reports ECAPACITY
  const int lane = threadIdx.x, nw = gridDim.x;
  const int nc = min(W.counters[2], P.max_pairs);
  const int per = max(kForcePairsPerPass, (nc + nw - 1) / nw);
  int qb = per * static_cast<int>(blockIdx.x);
  const int q1 = min(qb + per, nc);
  if (qb >= q1) return;
  ForceArgs a = force_args(P, S, D, W, vel, pair_out);
  a.gbox = 0.5 * 6.0 / P.wdx;
  if (LAW && P.history) a.hb_wr = W.hist_box + static_cast<size_t>((W.counters[kStepCounter] & 1) ^ 1) * P.n * P.max_nbr * 6;
  constexpr int kPieces = static_cast<int>(sizeof(OvlRec) / 16), kGeo = static_cast<int>(sizeof(BoxGeom) / 8);
  int nov = 0, n = 0;   // overlapping pairs, pairs waiting
  for (;;) {
    while (n < kForcePairsPerPass && qb < q1) {
      const bool flag = qb + lane < q1 && W.oflag[qb + lane] != 0;
      const unsigned m = __ballot_sync(kFull, flag);
      if (flag) s_q[n + __popc(m & ((1u << lane) - 1u))] = qb + lane;
      n += __popc(m);
      nov += __popc(m);
      qb += 32;
      __syncwarp();
    }
    if (n == 0) break;
    const int m = min(n, kForcePairsPerPass);
    n -= m;
    for (int e = lane; e < m * kPieces; e += 32)
      reinterpret_cast<int4*>(s_ovl)[e] = reinterpret_cast<const int4*>(W.olist + s_q[n + e / kPieces])[e % kPieces];
    for (int e = lane; e < m * kGeo; e += 32)
      reinterpret_cast<double*>(s_box)[e] = reinterpret_cast<const double*>(&W.box_work[s_q[n + e / kGeo]].box)[e % kGeo];
    __syncwarp();
#ifdef CONTACT_CHECKS
    if (lane < m) {   // the staged entries' pair and particles
      OvlRec& e = s_ovl[lane];
      e.q = checked_index(W.err, e.q, P.max_pairs, 0);
      e.i = checked_index(W.err, e.i, P.n, 0);
      e.j = checked_index(W.err, e.j, P.n + P.nwall, 0);
    }
    __syncwarp();
#endif
    pair_force_law<SET, LAW, true>(a, s_ovl, m, s_box);
    __syncwarp();
  }
  if (lane == 0 && nov > 0) atomicAdd(&W.counters[5], nov);
}

}  // namespace

void launch_box(const Params& P, const Shapes& S, const Parts& D, const Lists& W, const double* vel, double* pair_out,
                int grid, cudaStream_t st) {
  // the node sweep's kind set: 2 cubes only, 1 spheres / cuboids / walls, 0 every kind;
  // persistent: as many blocks as are resident (each kernel's own occupancy)
  const bool law = P.history || P.friction || (vel != nullptr && P.damping_c != 0.0);
  auto rough = P.kind_set == 2 ? k_box_rough<2> : (P.kind_set == 1 ? k_box_rough<1> : k_box_rough<0>);
  auto pairs = P.history ? (P.kind_set == 2 ? k_box_pairs<2, true> : (P.kind_set == 1 ? k_box_pairs<1, true> : k_box_pairs<0, true>))
                         : (P.kind_set == 2 ? k_box_pairs<2, false> : (P.kind_set == 1 ? k_box_pairs<1, false> : k_box_pairs<0, false>));
  auto flaw = P.kind_set == 2 ? (law ? k_box_law<2, true> : k_box_law<2, false>)
                              : (law ? k_box_law<0, true> : k_box_law<0, false>);
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (sms <= 0) sms = grid;
  auto resident = [sms](auto kern) {
    int per_sm = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kBoxWarps * 32, 0);
    return dim3(sms * (per_sm > 0 ? per_sm : 1));
  };
  launch_pdl(rough, resident(rough), dim3(kBoxWarps * 32), 0, st, P, S, D, W);
  launch_pdl(pairs, resident(pairs), dim3(kBoxWarps * 32), 0, st, P, S, D, W);
  // (one-warp blocks: one per sub-partition)
  launch_pdl(flaw, dim3(4 * sms), dim3(32), 0, st, P, S, D, W, vel, pair_out);
}

}  // namespace gbc
