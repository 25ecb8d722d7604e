// Narrow phase of the contact step: every lattice node of every candidate
// pair's box is tested against both particles' signed distance functions and
// reduced to the overlap volume, its first moments, the band sum behind the
// contact normal and the deepest node (Sec. 3.3.1 of arXiv:2401.10878: "iterate
// over the entire overlap region to determine the overlap volume, the contact
// point, the contact normal, the indentation depth").
//
// k_narrow32 (FP32 node tests, FP32 tile partials):
//   * persistent grid, one warp per tile; warp w takes tiles w, w + W, ...
//     of the tile list (W warps, numbered across the blocks; no queue atomics),
//     the next tile's record fetched while the current one runs; pairs whose
//     distance regions are apart never reach the list (the pair builder's test);
//   * a pair's box is cut into node lines along its longest axis; a tile is
//     32 lanes x 4 lines of one pair;
//   * each lane clips its line to the interval where both signed distances
//     lie below w/2 (line_clip.cuh: one bound per face plane, the sphere's
//     quadratic) and evaluates only the nodes inside it: every node outside
//     adds exact zeros to every sum, and ~99 % of a settling box's pair-box
//     nodes lie outside;
//   * the clipped nodes are spread one per lane (sweep_tile);
//   * node coordinates relative to each particle are exact integers minus an
//     FP32 remainder in [-1/2, 1/2] (no large-offset cancellation);
//   * polytope faces (and their bounds along the lines) are staged in shared
//     memory;
//   * warp reduction per tile (skipped when no lane met a node to
//     evaluate); a pair of one tile is finished from the warp's registers,
//     otherwise the partials go to HBM and the warp that completes the pair's
//     last tile sums them in FP64 in tile order (deterministic).
// k_narrow64: all-FP64 comparison form over the same tiles, lines clipped in FP32.
#include <cfloat>
#include <climits>
#include <type_traits>

#include "contact_dev.cuh"
#include "force_law.cuh"
#include "line_clip.cuh"

namespace gbc {

namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kWarps = 8;  // warps per block of the persistent kernel

// Local sweep axes (u = along the lines, v, w across) and the node-index
// stride of each (the node index is x-fastest over the pair box).
struct Local {
  int u, v, w;
  int su, sv, sw;
};

__device__ __forceinline__ Local make_local(const PairRec& r) {
  Local L;
  L.u = r.axis;
  L.v = L.u == 2 ? 0 : L.u + 1;
  L.w = L.v == 2 ? 0 : L.v + 1;
  const int s1 = r.dim[0], s2 = r.dim[0] * r.dim[1];
  L.su = L.u == 0 ? 1 : (L.u == 1 ? s1 : s2);
  L.sv = L.v == 0 ? 1 : (L.v == 1 ? s1 : s2);
  L.sw = L.w == 0 ? 1 : (L.w == 1 ? s1 : s2);
  return L;
}

// (a_u, a_v, a_w) in local axes -> component c of the world vector
__device__ __forceinline__ float world_comp(int c, const Local& L, float au, float av, float aw) {
  return c == L.u ? au : (c == L.v ? av : aw);
}


// ---------------------------------------------------------------- evaluators
// Each evaluator holds one particle's geometry for the current tile, in
// lattice units, relative to the pair box origin; it reads the pair record
// from shared memory (second = the record's particle j).

// Cube (equal half extents h): phi = max_k |y_k| - h.  Only what the node
// loop needs stays in registers; the cross-axis terms are re-read from the
// shared-memory pair record at each line start.  The line clip reads per-tile
// constants from shared memory (prep_clip): along the line, slab k of
// |y_k| < h + T is the node-counter interval centred at
// c_k = fu - (tv_k rv + tw_k rw) / tu_k with half-width (h + T) / |tu_k|.
struct CubeEval {
  int iu;
  float fu, tu0, tu1, tu2, h, itu0, itu1, itu2;
  bool flat;   // a slab parallel to the lines (|tu_k| <= kClipFlat): the general clip
  float cnt_u, p0, p1, p2, y0, y1, y2;
  float gb0, gb1, gb2;
  // (the geometry comes with the staged constants: prep_lanes, then fetch)
  __device__ __forceinline__ void clear() { gb0 = gb1 = gb2 = 0.f; }
  __device__ __forceinline__ int faces() const { return 0; }
  __device__ __forceinline__ void begin_line_rec(const PairRec& r, bool second, const Local& L, int cv, int cw,
                                                 int u0) {
    const int* ci = second ? r.bi : r.ai;
    const float* cf = second ? r.bf : r.af;
    const float* rt = second ? r.rtb : r.rta;
    const float rv = static_cast<float>(cv - ci[L.v]) - cf[L.v];
    const float rw = static_cast<float>(cw - ci[L.w]) - cf[L.w];
    p0 = fmaf(-tu0, fu, fmaf(rt[L.v], rv, rt[L.w] * rw));
    p1 = fmaf(-tu1, fu, fmaf(rt[3 + L.v], rv, rt[3 + L.w] * rw));
    p2 = fmaf(-tu2, fu, fmaf(rt[6 + L.v], rv, rt[6 + L.w] * rw));
    cnt_u = static_cast<float>(u0 - iu) - 1.f;
  }
  __device__ __forceinline__ void clip(float T, float& lo, float& hi) const {
    const float o = static_cast<float>(iu), ht = h + T;
    float l = lo - o, hh = hi - o;
    clip_slab(tu0, itu0, p0, ht, l, hh);
    clip_slab(tu1, itu1, p1, ht, l, hh);
    clip_slab(tu2, itu2, p2, ht, l, hh);
    lo = l + o;
    hi = hh + o;
  }
  // per-tile constants in cs[0 .. 8): (sv_k, hd_0), (sw_k, hd_1),
  // (hd_2, iv + fv, iw + fw, fu + iu), (iv, iw, iu, fu), (tv_k, fv),
  // (tw_k, fw), (tu_k, h), (1 / tu_k, -) with sv_k = tv_k / tu_k,
  // sw_k = tw_k / tu_k, hd_k = (h + T) / |tu_k| (the line clip reads the
  // first three, the node start the next three).  Lane k < 3 forms axis k's entries, lane 3 the
  // centre and size (two cubes: lanes 4 .. 7 form B's in the same pass); the
  // caller syncs the warp once for both evaluators and every lane then
  // fetches its registers.
  // the stores of lane q of the group that forms the constants (q < 3: axis
  // q's entries, q = 3: the centre and size, q > 3: none)
  static __device__ __forceinline__ void prep_lanes(const PairRec& r, bool second, const Local& L, float T,
                                                    float4* cs, int q) {
    const int* ci = second ? r.bi : r.ai;
    const float* cf = second ? r.bf : r.af;
    const float* rt = second ? r.rtb : r.rta;
    const float hh = second ? r.szb[0] : r.sza[0];
    const int k = q < 3 ? q : 0;
    const float tu = rt[3 * k + L.u], tv = rt[3 * k + L.v], tw = rt[3 * k + L.w];
    const float itu = clip_inv(tu);
    float* f = reinterpret_cast<float*>(cs);
    if (q < 3) {
      f[k] = tv * itu;
      f[4 + k] = tw * itu;
      f[k == 0 ? 3 : (k == 1 ? 7 : 8)] = (hh + T) * fabsf(itu);
      f[16 + k] = tv;
      f[20 + k] = tw;
      f[24 + k] = tu;
      f[28 + k] = itu;
    } else if (q == 3) {
      const int iu = ci[L.u], iv = ci[L.v], iw = ci[L.w];
      const float fu = cf[L.u], fv = cf[L.v], fw = cf[L.w];
      f[9] = static_cast<float>(iv) + fv;
      f[10] = static_cast<float>(iw) + fw;
      f[11] = fu + static_cast<float>(iu);
      cs[3] = make_float4(__int_as_float(iv), __int_as_float(iw), __int_as_float(iu), fu);
      f[19] = fv;
      f[23] = fw;
      f[27] = hh;
    }
  }
  __device__ __forceinline__ void fetch(const float4* cs) {
    const float4 a = cs[6], b = cs[7], d = cs[3];
    tu0 = a.x; tu1 = a.y; tu2 = a.z; h = a.w;
    itu0 = b.x; itu1 = b.y; itu2 = b.z;
    fu = d.w;
    iu = __float_as_int(d.z);
    flat = !(fabsf(tu0) > kClipFlat && fabsf(tu1) > kClipFlat && fabsf(tu2) > kClipFlat);
  }
  // begin_line_rec from the staged constants (the same operands, the same arithmetic)
  __device__ __forceinline__ void begin_node(const float4* cs, int cv, int cw, int u0) {
    const float4 d = cs[3], tv = cs[4], tw = cs[5];
    const float rv = static_cast<float>(cv - __float_as_int(d.x)) - tv.w;
    const float rw = static_cast<float>(cw - __float_as_int(d.y)) - tw.w;
    p0 = fmaf(-tu0, fu, fmaf(tv.x, rv, tw.x * rw));
    p1 = fmaf(-tu1, fu, fmaf(tv.y, rv, tw.y * rw));
    p2 = fmaf(-tu2, fu, fmaf(tv.z, rv, tw.z * rw));
    cnt_u = static_cast<float>(u0 - iu) - 1.f;
  }
  // [lo, hi] cut to the nodes of line (cv, cw) inside all three slabs
  __device__ __forceinline__ void clip_line(const PairRec& r, bool second, const Local& L, const float4* cs, int cv,
                                            int cw, float T, float& lo, float& hi) {
    const float4 a = cs[0], b = cs[1], c = cs[2];
    if (flat) {
      begin_line_rec(r, second, L, cv, cw, 0);
      clip(T, lo, hi);
      return;
    }
    // in box nodes: the centre's offsets (iv + fv, iw + fw) and fu + iu formed
    // once per tile (their rounding, ~1e-5 cells, stays far inside the margin)
    const float rv = static_cast<float>(cv) - c.y;
    const float rw = static_cast<float>(cw) - c.z;
    const float x0 = fmaf(-a.x, rv, fmaf(-b.x, rw, c.w));
    const float x1 = fmaf(-a.y, rv, fmaf(-b.y, rw, c.w));
    const float x2 = fmaf(-a.z, rv, fmaf(-b.z, rw, c.w));
    lo = fmaxf(lo, max3f(x0 - a.w, x1 - b.w, x2 - c.x));
    hi = fminf(hi, min3f(x0 + a.w, x1 + b.w, x2 + c.x));
  }
  __device__ __forceinline__ float phi() {
    cnt_u += 1.f;
    y0 = fmaf(tu0, cnt_u, p0);
    y1 = fmaf(tu1, cnt_u, p1);
    y2 = fmaf(tu2, cnt_u, p2);
    return fmaxf(fabsf(y0), fmaxf(fabsf(y1), fabsf(y2))) - h;
  }
  __device__ __forceinline__ void grad(float m) {
    const float a0 = fabsf(y0), a1 = fabsf(y1), a2 = fabsf(y2);
    const bool s0 = a0 >= a1 && a0 >= a2;
    const bool s1 = !s0 && a1 >= a2;
    gb0 += s0 ? copysignf(m, y0) : 0.f;
    gb1 += s1 ? copysignf(m, y1) : 0.f;
    gb2 += (!s0 && !s1) ? copysignf(m, y2) : 0.f;
  }
  // what grad(m) adds for the current node (shared tiles): a factor and three components
  __device__ __forceinline__ float4 record(float m) const {
    const float a0 = fabsf(y0), a1 = fabsf(y1), a2 = fabsf(y2);
    const bool s0 = a0 >= a1 && a0 >= a2;
    const bool s1 = !s0 && a1 >= a2;
    return make_float4(1.f, s0 ? copysignf(m, y0) : 0.f, s1 ? copysignf(m, y1) : 0.f,
                       (!s0 && !s1) ? copysignf(m, y2) : 0.f);
  }
  __device__ __forceinline__ void set_sums(float a, float b, float c) {
    gb0 = a;
    gb1 = b;
    gb2 = c;
  }
  __device__ float world(int c, const Local&, const PairRec& r, bool second) const {
    const float* rt = second ? r.rtb : r.rta;
    return rt[c] * gb0 + rt[3 + c] * gb1 + rt[6 + c] * gb2;
  }
};

// Stage a polytope's world planes in local axes (u, v, w, offset) into shared
// memory; faces beyond nf are padded so that they never win the maximum (and are
// constant along the line, below any threshold).
__device__ __forceinline__ void stage_planes(const Shapes& S, const Parts& D, int pid, const Local& L,
                                            float4* sm, int npad) {
  const int lane = threadIdx.x & 31;
  const int f0 = S.face_off[pid];
  const int nf = S.face_off[pid + 1] - f0;
  if (lane < npad) {
    float4 e = make_float4(0.f, 0.f, 0.f, 1e30f);
    if (lane < nf) {
      const float4 w = D.wplane[f0 + lane];
      e = make_float4(L.u == 0 ? w.x : (L.u == 1 ? w.y : w.z), L.v == 0 ? w.x : (L.v == 1 ? w.y : w.z),
                      L.w == 0 ? w.x : (L.w == 1 ? w.y : w.z), w.w);
    }
    sm[lane] = e;
  }
  __syncwarp();
}

// Any kind, chosen at run time (the variant with every kind): what the other
// evaluators keep in registers stays in the warp's shared memory, so one copy of
// the code serves every pair of kinds.  With a sweep compiled per kind pair the
// warps of an SM, each on its own pair, waited on instruction fetches for most
// of the time (16 of 23 stalled cycles per instruction: 82 us for 15472
// smoothed mixed particles, 10.8 us for 1934 sharp ones; 39.5 and 8.9 us with
// one copy; where few kinds meet in deep tiles, see kDeepNodes).  The arithmetic of a line and of a node is that of the evaluators
// above, operation for operation.
// cs: sphere (radius); cuboid (tu, tv, tw, h) per axis, then 1 / tu; wall
// (mu, mv, mw, p0), then 1 / mu (p0 = the wall's value at the box origin,
// inflate included, formed in FP64 by the pair builder: box-relative values
// stay small, so FP32 keeps them to ~1e-6); polytope its planes in local axes
// and, from kMaxFaces, the half-line bounds of its faces: along the line, face
// f of slope m = e.x bounds the node counter c - iu by C_f - sy_f rv - sz_f rw
// (above for m > 0, below for m < 0) with sy_f = e.y / m, sz_f = e.z / m, C_f =
// (T + e.w) / m + fu, sorted into upper, lower and parallel faces (|m| <=
// kClipFlat: the plane, which keeps or empties the whole line).  POLY: there
// are polytopes; CUBE: cubes are swept as CubeEval does (its constants in cs),
// else as cuboids.
constexpr int kAnyKind = -1;   // as a kind known at compile time: none, the evaluator's own
template <bool POLY, bool CUBE>
struct AnyEval {
  int kind, iu, iv, iw, nf, nup, ndn;
  float fu, fv, fw;
  const float4* cs;
  float g0, g1, g2;   // band sum: local axes (sphere, polytope), body axes (cuboid), along the normal (wall)
  __device__ __forceinline__ int faces() const { return POLY ? nf : 0; }
  // the registers, with the constants staged in sm (a shared tile: by the warp that clipped it)
  __device__ void attach(const PairRec& r, bool second, const Shapes& S, const Local& L, float4* sm) {
    kind = second ? r.kinds >> 8 : r.kinds & 0xff;
    const int* ci = second ? r.bi : r.ai;
    const float* cf = second ? r.bf : r.af;
    iu = ci[L.u]; iv = ci[L.v]; iw = ci[L.w];
    fu = cf[L.u]; fv = cf[L.v]; fw = cf[L.w];
    cs = sm;
    nf = nup = ndn = 0;
    if (POLY && kind == KIND_POLY) {
      const int pid = second ? r.j : r.i;
      nf = S.face_off[pid + 1] - S.face_off[pid];
    }
    g0 = g1 = g2 = 0.f;
  }
  __device__ void load(const PairRec& r, bool second, const Shapes& S, const Parts& D, const Local& L, float T,
                       float4* sm) {
    const int lane = threadIdx.x & 31;
    attach(r, second, S, L, sm);
    const float* rt = second ? r.rtb : r.rta;
    const float* sz = second ? r.szb : r.sza;
    if (CUBE && kind == KIND_CUBE) {
      CubeEval::prep_lanes(r, second, L, T, sm, lane);
    } else if (POLY && kind == KIND_POLY) {
      stage_planes(S, D, second ? r.j : r.i, L, sm, kMaxFaces);
      const bool act = lane < nf;
      const float4 e = sm[act ? lane : 0];
      const bool up = act && e.x > kClipFlat, dn = act && e.x < -kClipFlat, par = act && !up && !dn;
      const unsigned bu = __ballot_sync(kFull, up), bd = __ballot_sync(kFull, dn), bp = __ballot_sync(kFull, par);
      nup = __popc(bu);
      ndn = __popc(bd);
      const unsigned lt = (1u << lane) - 1u;
      const int pos = up ? __popc(bu & lt) : (dn ? nup + __popc(bd & lt) : nup + ndn + __popc(bp & lt));
      if (act) {
        float4 c = e;
        if (!par) {
          const float im = __fdividef(1.f, e.x);
          c = make_float4(e.y * im, e.z * im, fmaf(T + e.w, im, fu), 0.f);
        }
        sm[kMaxFaces + pos] = c;
      }
    } else if (kind == KIND_SPHERE) {
      if (lane == 0) sm[0] = make_float4(sz[0], 0.f, 0.f, 0.f);
    } else if (kind == KIND_WALL) {
      if (lane == 0) sm[0] = make_float4(rt[L.u], rt[L.v], rt[L.w], sz[0]);
      if (lane == 1) sm[1] = make_float4(clip_inv(rt[L.u]), 0.f, 0.f, 0.f);
    } else {   // cuboids and cubes
      if (lane < 3) {
        sm[lane] = make_float4(rt[3 * lane + L.u], rt[3 * lane + L.v], rt[3 * lane + L.w], sz[lane]);
        reinterpret_cast<float*>(sm + 3)[lane] = clip_inv(rt[3 * lane + L.u]);
      }
    }
  }
  // [lo, hi] (line coordinates) cut to where phi < T on the line (cv, cw)
  __device__ __forceinline__ void clip_line(const PairRec& r, bool second, const Local& L, const float4*, int cv, int cw,
                                            float T, float& lo, float& hi) const {
    if (CUBE && kind == KIND_CUBE) {
      CubeEval e;
      e.fetch(cs);
      e.clip_line(r, second, L, cs, cv, cw, T, lo, hi);
      return;
    }
    const float rv = static_cast<float>(cv - iv) - fv;
    const float rw = static_cast<float>(cw - iw) - fw;
    const float o = static_cast<float>(iu);
    if (kind == KIND_WALL) {
      const float4 m = cs[0];
      clip_half(m.x, cs[1].x, fmaf(m.y, static_cast<float>(cv), fmaf(m.z, static_cast<float>(cw), m.w)), T, lo, hi);
      return;
    }
    float l = lo - o, h = hi - o;
    if (kind == KIND_SPHERE) {
      clip_ball(fu, fmaf(rv, rv, rw * rw), cs[0].x, T, l, h);
    } else if (POLY && kind == KIND_POLY) {
      const float4* cl = cs + kMaxFaces;
      int f = 0;
      for (; f < nup; ++f) {
        const float4 c = cl[f];
        h = fminf(h, fmaf(-c.x, rv, fmaf(-c.y, rw, c.z)));
      }
      for (; f < nup + ndn; ++f) {
        const float4 c = cl[f];
        l = fmaxf(l, fmaf(-c.x, rv, fmaf(-c.y, rw, c.z)));
      }
      for (; f < nf; ++f) {
        const float4 e = cl[f];
        if (!(fmaf(-e.x, fu, fmaf(e.y, rv, fmaf(e.z, rw, -e.w))) < T)) l = kClipEmpty;
      }
    } else {
      const float4 it = cs[3];
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const float4 e = cs[k];
        const float p = fmaf(-e.x, fu, fmaf(e.y, rv, e.z * rw));
        clip_slab(e.x, k == 0 ? it.x : (k == 1 ? it.y : it.z), p, e.w + T, l, h);
      }
    }
    lo = l + o;
    hi = h + o;
  }
  // phi at node (u, cv, cw), and d: the direction that add(m, d) adds m times
  // (a sphere's d.w scales m).  K: the kind, or kAnyKind
  template <int K>
  __device__ __forceinline__ float phi(int u, int cv, int cw, float4& d) const {
    const int kind = K == kAnyKind ? this->kind : K;
    if (CUBE && kind == KIND_CUBE) {
      CubeEval e;
      e.fetch(cs);
      e.begin_node(cs, cv, cw, u);
      const float f = e.phi();
      d = e.record(1.f);
      d = make_float4(d.y, d.z, d.w, 1.f);
      return f;
    }
    if (kind == KIND_WALL) {
      const float4 m = cs[0];
      d = make_float4(1.f, 0.f, 0.f, 1.f);
      return fmaf(m.x, static_cast<float>(u), fmaf(m.y, static_cast<float>(cv), fmaf(m.z, static_cast<float>(cw), m.w)));
    }
    const float rv = static_cast<float>(cv - iv) - fv;
    const float rw = static_cast<float>(cw - iw) - fw;
    const float cnt_u = static_cast<float>(u - iu);
    if (kind == KIND_SPHERE) {
      const float ru = cnt_u - fu;
      const float q = fmaf(ru, ru, fmaf(rv, rv, rw * rw));
      d = make_float4(ru, rv, rw, q > 0.f ? rsqrtf(q) : 0.f);
      return sqrtf(q) - cs[0].x;
    }
    if (POLY && kind == KIND_POLY) {
      const float ru = cnt_u - fu;
      float4 e = cs[0];
      float best = fmaf(e.x, ru, fmaf(e.y, rv, fmaf(e.z, rw, -e.w)));
      int k = 0;
      for (int f = 1; f < nf; ++f) {
        e = cs[f];
        const float v = fmaf(e.x, ru, fmaf(e.y, rv, fmaf(e.z, rw, -e.w)));
        if (v > best) { best = v; k = f; }
      }
      e = cs[k];
      d = make_float4(e.x, e.y, e.z, 1.f);
      return best;
    }
    float y[3], a[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const float4 e = cs[k];
      y[k] = fmaf(e.x, cnt_u, fmaf(-e.x, fu, fmaf(e.y, rv, e.z * rw)));
      a[k] = fabsf(y[k]) - e.w;
    }
    // active face: first maximal axis; gradient sign(y_k) e_k (body frame)
    const bool s0 = a[0] >= a[1] && a[0] >= a[2];
    const bool s1 = !s0 && a[1] >= a[2];
    d = make_float4(s0 ? copysignf(1.f, y[0]) : 0.f, s1 ? copysignf(1.f, y[1]) : 0.f,
                    (!s0 && !s1) ? copysignf(1.f, y[2]) : 0.f, 1.f);
    return fmaxf(a[0], fmaxf(a[1], a[2]));
  }
  template <int K>
  __device__ __forceinline__ void add(float m, const float4& d) {
    if (K == KIND_WALL) {
      g0 += m;   // (all of its band sum)
      return;
    }
    const float4 e = record(m, d);
    g0 = fmaf(e.x, e.y, g0);
    g1 = fmaf(e.x, e.z, g1);
    g2 = fmaf(e.x, e.w, g2);
  }
  // what add(m, d) adds: a factor and three components
  static __device__ __forceinline__ float4 record(float m, const float4& d) {
    return make_float4(m * d.w, d.x, d.y, d.z);
  }
  __device__ __forceinline__ void set_sums(float a, float b, float c) {
    g0 = a;
    g1 = b;
    g2 = c;
  }
  // component c of the band sum in the world frame
  __device__ float world(int c, const Local& L, const PairRec& r, bool second) const {
    const float* rt = second ? r.rtb : r.rta;
    if (kind == KIND_WALL) return rt[c] * g0;
    if (kind == KIND_SPHERE || (POLY && kind == KIND_POLY)) return world_comp(c, L, g0, g1, g2);
    return rt[c] * g0 + rt[3 + c] * g1 + rt[6 + c] * g2;
  }
};

// Kernel variants: every kind of particle; spheres, cubes and cuboids (no
// polytopes: fewer registers, no spills) of several kinds or of one kind, with
// walls; cubes alone (chosen at init).
enum KindSet : int { SET_ALL = 0, SET_SC = 1, SET_CUBE = 2, SET_ONE = 3 };

// ---------------------------------------------------------------- tile sweep
// Per-lane partials of a tile: node count and first moments (exact integers
// in sharp mode), the band sum of the normal, and the deepest node.
struct Partial {
  float cnt, mx, my, mz, gx, gy, gz, bestf;
  int bestidx;
  bool touched;   // warp-uniform: some lane evaluated a node (else every sum is zero)
  bool deferred;  // warp-uniform: left for the whole block, nothing evaluated
};

// A tile shared by the block's warps (COOP), clipped by one of them (its record,
// staged constants and node table in shared memory; nown lanes with nodes,
// total nodes): warp w evaluates node passes w, w + 8, ... and leaves what each
// node adds in shared memory (term c of node l of the round at add[c][l]: both
// evaluators' band terms as a factor and three components, the weight and node
// (u, v, w), depth and node index).  Six warps make the additions, two sums or
// the deepest node each, pass by pass in the order of a tile swept by one warp,
// so the sums are the same bit for bit (in rolled loops: unrolled, the code made
// every step's fetches longer, 400 cubes 33.5 us against 32.1).
enum CoopTerm : int { TERM_A = 0, TERM_B = 4, TERM_W = 8, TERM_F = 12, TERM_IDX = 13, kCoopTerms = 14 };
struct Coop {
  float add[kCoopTerms][kWarps * 32];
  float sum[12][32];   // cnt, mu, mv, mw; A's three; B's three; depth, node index
};
template <int K>
using KindC = std::integral_constant<int, K>;
// f(kind of A, kind of B) as compile-time constants, for a wall (A) and a particle that is no polytope, or two
// particles of one such kind
template <class F>
__device__ __forceinline__ void with_wall(int b, const F& f) {
  if (b == KIND_SPHERE) f(KindC<KIND_WALL>{}, KindC<KIND_SPHERE>{});
  else if (b == KIND_CUBE) f(KindC<KIND_WALL>{}, KindC<KIND_CUBE>{});
  else f(KindC<KIND_WALL>{}, KindC<KIND_CUBOID>{});
}
template <class F>
__device__ __forceinline__ void with_kind(int b, const F& f) {
  if (b == KIND_SPHERE) f(KindC<KIND_SPHERE>{}, KindC<KIND_SPHERE>{});
  else if (b == KIND_CUBE) f(KindC<KIND_CUBE>{}, KindC<KIND_CUBE>{});
  else f(KindC<KIND_CUBOID>{}, KindC<KIND_CUBOID>{});
}
// Passes compiled for the pair's kinds keep the constants in registers: a quarter
// of the run-time evaluator's instructions fewer.  Every such loop that is in use
// at a time costs instruction fetches, so they serve particles of one kind (that
// kind with itself and with walls) and, with several kinds, wall contacts of more
// clipped nodes than this.  Step with a sweep compiled per kind pair, with the
// run-time evaluator alone, and so: 4000 cuboids of 26 cells pressed on a floor
// and a ceiling 338, 370, 301 us; 936 cuboids in a dense lattice 121, 133, 121;
// 2000 spheres and cuboids on walls 196, 206, 172; 7819 spheres and cuboids
// pressed into one another and on walls 550, 349, 311 (335 with a loop for every
// pair of kinds).  With polytopes the loops cost the other tiles more than they
// gave (6956 mixed particles, smoothed: 481 us without, 491 with them).
constexpr int kDeepNodes = 64;

// A block's deep tiles, those of more than kShareNodes clipped nodes when every
// warp has at most one tile, are shared by its warps one after the other when
// that is expected to end before the longest of them on its own warp (cycles:
// kPassCycles and kFaceCycles for each polytope face a node pass; eight passes at
// a time a quarter more and kRoundCycles for the barriers and the additions;
// kTileCycles more for a further tile, whose additions wait for the one before).
// One tile alone is always worth it, two equal ones of boxes or spheres hardly,
// polytopes' several.  Step by single warps, all shared,
// and so: 49 spheres and cuboids of 26 cells on walls 61.6, 53.4, 48.0 us; 1000
// smoothed cubes on walls 47.3, 70.9, 47.1; 240 polytopes deep in one another 147,
// 99, 86.
constexpr int kShareNodes = 128;
constexpr int kPassCycles = 300, kFaceCycles = 20, kRoundCycles = 150, kTileCycles = 3200, kShareCycles = 300;
struct DeepTiles {
  int n, alone, shared;   // tiles, cycles of the longest alone and of all of them shared
  int3 tile[kWarps];      // the warp that clipped it, lanes with nodes, clipped nodes
};
// Every warp of the block counts itself once: one with a deep tile waits for all
// the others' counts, one without goes on at once (waiting too cost 0.4 us of the
// 31 of a step of 1934 cubes).
__device__ __forceinline__ void no_deep_tile() { asm volatile("bar.arrive 1, %0;" ::"r"(blockDim.x) : "memory"); }
// Enters the warp's tile when it is deep; true when it is left to the block.
__device__ __forceinline__ bool leave_to_block(DeepTiles* deep, int total, int nown, int faces) {
  if (total <= kShareNodes) {   // warp-uniform
    no_deep_tile();
    return false;
  }
  if ((threadIdx.x & 31) == 0) {
    const int np = (total + 31) / 32, pass = kPassCycles + kFaceCycles * faces;
    deep->tile[atomicAdd_block(&deep->n, 1)] = make_int3(threadIdx.x >> 5, nown, total);
    atomicMax_block(&deep->alone, np * pass);
    atomicAdd_block(&deep->shared, (np + kWarps - 1) / kWarps * (pass * 5 / 4 + kRoundCycles) + kTileCycles);
  }
  __syncwarp();
  asm volatile("bar.sync 1, %0;" ::"r"(blockDim.x) : "memory");
  const volatile DeepTiles* d = deep;
  return d->shared < d->alone;
}

// Order-preserving map of FP32 values to signed ints (for integer max).
__device__ __forceinline__ int float_key(float f) {
  const int b = __float_as_int(f);
  return b >= 0 ? b : (b ^ 0x7fffffff);
}
__device__ __forceinline__ float key_float(int k) { return __int_as_float(k >= 0 ? k : (k ^ 0x7fffffff)); }

// Two phases per tile.  (A) Lane l clips its lines it0 + 32 s + l (s <
// kTileItemsPerLane) to the nodes where both distances lie below w/2 (+ the
// clip margin) and keeps each clipped range's first node and count.  (B) The
// tile's clipped nodes, typically a few dozen spread over a few lines, are
// numbered lane by lane (a scan of the lanes' counts), each lane's in slot
// order, and each lane evaluates one of them: the owning lane from a table
// of the lanes with nodes, the slot by the owner's counts, and the evaluators
// start that node's line at the node itself, so the node gets exactly the
// arithmetic of a node walk (the same FP32 distances, bit for bit).
// E: the evaluator of both particles.  With AnyEval the slot loop stays rolled,
// with the slots' clipped ranges in shared memory, to keep the kernel's code
// small (unrolled: 38.8 -> 61.8 us on 15472 mixed particles); for two cubes they
// are unrolled over registers.
template <bool SMOOTH, int SET, bool COOP, class E>
__device__ __forceinline__ Partial sweep_tile(const Params& P, const Shapes& S, const Parts& D, const PairRec& r,
                                              bool swap, int tl, float4* smA, float4* smB, unsigned* spk,
                                              int4* own, DeepTiles* deep, Coop* coop, int nown, int total_in) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
  const Local L = make_local(r);
  constexpr bool ROLL = !std::is_same<E, CubeEval>::value;
  E A, B;
  const int du = r.dim[L.u], dv = r.dim[L.v];
  const float inv_dv = __fdividef(1.f, static_cast<float>(dv));
  const float inv_w = P.inv_w, hw = 0.5f * P.wdx_l, T = hw + P.clip_margin;
  if constexpr (ROLL && COOP) {
    A.attach(r, swap, S, L, smA);
    B.attach(r, !swap, S, L, smB);
  } else if constexpr (ROLL) {
    A.load(r, swap, S, D, L, T, smA);
    B.load(r, !swap, S, D, L, T, smB);
    __syncwarp();
  } else {
    A.clear();
    B.clear();
    if constexpr (!COOP) {
      // two cubes in one pass: lanes 0 .. 3 form A's constants, lanes 4 .. 7 B's
      const bool isb = (lane & 4) != 0;
      CubeEval::prep_lanes(r, isb ? !swap : swap, L, T, isb ? smB : smA, lane < 8 ? (lane & 3) : 4);
    }
    __syncwarp();
    A.fetch(smA);
    B.fetch(smB);
  }
  const float4* csA = smA;
  const float4* csB = smB;
  float cnt = 0.f, mu = 0.f, mv = 0.f, mw = 0.f, bestf = -FLT_MAX;
  [[maybe_unused]] float part0 = 0.f, part1 = 0.f;   // (COOP) the warp's two sums
  int bestidx = 0x7fffffff;
  const int it0 = tl * 32 * kTileItemsPerLane;
  const int ns = min(kTileItemsPerLane, (r.nitems - it0 + 31) >> 5);   // slots of this tile (warp-uniform)
  int total = total_in, excl = 0;
  bool has = false;
  if constexpr (COOP) {   // (only counts of first nodes matter below: lane k stands for entry k of own)
    has = lane < nown;
    excl = has ? own[lane].y : 0;
  } else {
    // (A) per slot: first clipped node (low 16 bits) and count (high 16 bits);
    // a pair box is below 2^16 nodes along an axis
    unsigned pk[kTileItemsPerLane];
    int nl = 0;
    // line it0 + 32 s + lane as (cv, cw) = its remainder and quotient by dv:
    // unrolled, one division for slot 0, then steps of 32 = q32 dv + r32; the
    // rolled loop divides per slot (fewer live registers)
    int cv = 0, r32 = 0, q32 = 0;
    int cw = 0;
    if constexpr (!ROLL) {
      cw = div_small(it0 + lane, dv, inv_dv, &cv);
      q32 = div_small(32, dv, inv_dv, &r32);
    }
#pragma unroll(ROLL ? 1 : kTileItemsPerLane)
    for (int s = 0; s < kTileItemsPerLane; ++s) {
      if (!ROLL) pk[s] = 0u;
      if (s < ns) {
        const int it = it0 + s * 32 + lane;
        if constexpr (ROLL) cw = div_small(it, dv, inv_dv, &cv);
        const int len = it < r.nitems ? du : 0;
        float clo = 0.f, chi = static_cast<float>(len - 1);
        A.clip_line(r, swap, L, csA, cv, cw, T, clo, chi);
        B.clip_line(r, !swap, L, csB, cv, cw, T, clo, chi);
        int ub;
        const int nk = clip_nodes(clo, chi, 0, len, &ub);
        const unsigned v = static_cast<unsigned>(ub) | (static_cast<unsigned>(nk) << 16);
        if constexpr (ROLL) spk[s * 32 + lane] = v;
        else pk[s] = v;
        nl += nk;
      }
      if constexpr (!ROLL) {
        cv += r32;
        cw += q32;
        if (cv >= dv) {
          cv -= dv;
          ++cw;
        }
      }
    }
    if (ROLL) __syncwarp();
    int incl = nl;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int v = __shfl_up_sync(kFull, incl, d);
      if (lane >= d) incl += v;
    }
    total = __shfl_sync(kFull, incl, 31);
    excl = incl - nl;
    // the lanes with nodes, in lane order (their first nodes strictly
    // increase): entry k of own holds the k-th one's lane, first node and
    // clipped ranges
    has = nl > 0;
    if (total > 0) {
      const int rank = __popc(__ballot_sync(kFull, has) & ((1u << lane) - 1u));
      if (has) {
        static_assert(kTileItemsPerLane == 4, "own holds four clipped ranges per lane");
        if constexpr (ROLL) {
#pragma unroll
          for (int s = 0; s < kTileItemsPerLane; ++s) pk[s] = s < ns ? spk[s * 32 + lane] : 0u;
        }
        // and the lane's node counts before slots 2 and 3
        const int c2 = static_cast<int>(pk[0] >> 16) + static_cast<int>(pk[1] >> 16);
        own[rank] = make_int4(lane, excl, static_cast<int>(pk[0]), static_cast<int>(pk[1]));
        own[32 + rank] = make_int4(static_cast<int>(pk[2]), static_cast<int>(pk[3]), c2,
                                   c2 + static_cast<int>(pk[2] >> 16));
      }
      __syncwarp();
    }
    if (deep != nullptr && leave_to_block(deep, total, __popc(__ballot_sync(kFull, has)),
                                        A.faces() + B.faces())) {
      Partial o{};
      o.deferred = true;
      return o;
    }
  }
  // (B) node g of the tile's clipped nodes on lane g mod 32; its owner is the
  // last lane with nodes whose first node is <= g, i.e. entry (number of such
  // lanes) - 1 of own, counted from the lanes that start before the pass and
  // a mask of the first nodes inside it
  const int step = COOP ? 32 * nwarp : 32;
  // (KA, KB: the kinds of A and B where the caller knows them)
  auto passes = [&](auto ka, auto kb) {
    [[maybe_unused]] constexpr int KA = decltype(ka)::value, KB = decltype(kb)::value;
    for (int base0 = 0; base0 < total; base0 += step) {
      const int base = COOP ? base0 + 32 * wid : base0;
      const int g = base + lane;
      const unsigned before = __ballot_sync(kFull, has && excl < base);
      const unsigned inside =
          __reduce_or_sync(kFull, (has && excl >= base && excl - base < 32) ? 1u << (excl - base) : 0u);
      const int cnt_le = __popc(before) + __popc(inside & (lane == 31 ? 0xffffffffu : (2u << lane) - 1u));
      const int4 e = own[min(max(cnt_le - 1, 0), 31)];
      const int o = e.x;
      const int k = g - e.y;   // the node's rank among the owner's
      const int4 e2 = own[32 + min(max(cnt_le - 1, 0), 31)];
      // the slot: how many of the owner's slot boundaries (node counts before
      // slots 1, 2, 3; empty slots repeat a boundary) lie at or below k
      const int c1 = static_cast<int>(static_cast<unsigned>(e.z) >> 16), c2 = e2.z, c3 = e2.w;
      const int os = (k >= c1 ? 1 : 0) + (k >= c2 ? 1 : 0) + (k >= c3 ? 1 : 0);
      const unsigned q = static_cast<unsigned>(os == 0 ? e.z : (os == 1 ? e.w : (os == 2 ? e2.x : e2.y)));
      const int u = static_cast<int>(q & 0xffffu) + k - (os == 0 ? 0 : (os == 1 ? c1 : (os == 2 ? c2 : c3)));
      int ocv;
      const int ocw = div_small(it0 + os * 32 + o, dv, inv_dv, &ocv);
      float fa, fb;
      float4 da, db;
      if constexpr (ROLL) {
        fa = A.template phi<KA>(u, ocv, ocw, da);
        fb = B.template phi<KB>(u, ocv, ocw, db);
      } else {
        A.begin_node(csA, ocv, ocw, u);
        B.begin_node(csB, ocv, ocw, u);
        fa = A.phi();
        fb = B.phi();
      }
      // W > 0, or a band term of the normal: max < w/2 and (sharp) min <= 0
      const bool any = g < total && fmaxf(fa, fb) < hw && (SMOOTH || fminf(fa, fb) <= 0.f);
      const float ta = __saturatef(fmaf(fa, -inv_w, 0.5f));
      const float tb = __saturatef(fmaf(fb, -inv_w, 0.5f));
      float w, ma, mb;
      if (SMOOTH) {
        const float ha = ta * ta * fmaf(-2.f, ta, 3.f);
        const float hb = tb * tb * fmaf(-2.f, tb, 3.f);
        w = any ? ha * hb : 0.f;
        ma = any ? fmaf(-ta, ta, ta) * hb : 0.f;
        mb = any ? ha * fmaf(-tb, tb, tb) : 0.f;
      } else {
        w = (any && fmaxf(fa, fb) <= 0.f) ? 1.f : 0.f;
        ma = (any && fb <= 0.f) ? fmaf(-ta, ta, ta) : 0.f;
        mb = (any && fa <= 0.f) ? fmaf(-tb, tb, tb) : 0.f;
      }
      float f = -(fa + fb);
      int idx = u * L.su + ocv * L.sv + ocw * L.sw;
      if constexpr (COOP) {
        if (base < total) {   // warp-uniform
          const int at = 32 * wid + lane;
          float4 ga, gb;
          if constexpr (ROLL) {
            ga = E::record(ma, da);
            gb = E::record(mb, db);
          } else {
            ga = A.record(ma);
            gb = B.record(mb);
          }
          const float term[kCoopTerms] = {ga.x, ga.y, ga.z, ga.w, gb.x, gb.y, gb.z, gb.w,
                                          w, static_cast<float>(u), static_cast<float>(ocv), static_cast<float>(ocw),
                                          f, __int_as_float(idx)};
#pragma unroll
          for (int c = 0; c < kCoopTerms; ++c) coop->add[c][at] = term[c];
        }
        __syncthreads();
        const int nq = min(nwarp, (total - base0 + 31) / 32);
        if (wid == 2) {
#pragma unroll 1
          for (int q = 0; q < nq; ++q) {
            const int at = 32 * q + lane;
            f = coop->add[TERM_F][at];
            idx = __float_as_int(coop->add[TERM_IDX][at]);
            if (coop->add[TERM_W][at] > 0.f && (f > bestf || (f == bestf && idx < bestidx))) {
              bestf = f;
              bestidx = idx;
            }
          }
        } else if (wid < 6) {
          // the warp's sums k: of (1, u, v, w) times the weight, of A's and of B's components times their factor
          const int k0 = wid < 2 ? 2 * wid : 2 * wid - 2;
          const float* x0 = coop->add[k0 < 4 ? TERM_W : (k0 < 7 ? TERM_A : TERM_B)];
          const float* y0 = k0 < 4 ? coop->add[TERM_W + k0] : coop->add[k0 < 7 ? TERM_A + k0 - 3 : TERM_B + k0 - 6];
          const int k1 = k0 + 1;
          const float* x1 = coop->add[k1 < 4 ? TERM_W : (k1 < 7 ? TERM_A : TERM_B)];
          const float* y1 = k1 < 4 ? coop->add[TERM_W + k1] : coop->add[k1 < 7 ? TERM_A + k1 - 3 : TERM_B + k1 - 6];
#pragma unroll 1
          for (int q = 0; q < nq; ++q) {
            const int at = 32 * q + lane;
            part0 = fmaf(x0[at], k0 == 0 ? 1.f : y0[at], part0);
            part1 = fmaf(x1[at], y1[at], part1);
          }
        }
        __syncthreads();
      } else {
        cnt += w;
        mu = fmaf(w, static_cast<float>(u), mu);
        mv = fmaf(w, static_cast<float>(ocv), mv);
        mw = fmaf(w, static_cast<float>(ocw), mw);
        if (w > 0.f && (f > bestf || (f == bestf && idx < bestidx))) {
          bestf = f;
          bestidx = idx;
        }
        if constexpr (ROLL) {
          A.template add<KA>(ma, da);
          B.template add<KB>(mb, db);
        } else {
          A.grad(ma);
          B.grad(mb);
        }
      }
    }
  };
  if constexpr (SET == SET_ONE && !COOP) {
    if (A.kind == KIND_WALL) with_wall(B.kind, passes);
    else with_kind(B.kind, passes);
  } else if constexpr (SET == SET_SC && !COOP) {
    if (A.kind == KIND_WALL && total > kDeepNodes) with_wall(B.kind, passes);
    else passes(KindC<kAnyKind>{}, KindC<kAnyKind>{});
  } else {
    passes(KindC<kAnyKind>{}, KindC<kAnyKind>{});
  }
  if constexpr (COOP) {   // the sums to the block's first warp
    if (wid == 2) {
      coop->sum[10][lane] = bestf;
      coop->sum[11][lane] = __int_as_float(bestidx);
    } else if (wid < 6) {
      const int k0 = wid < 2 ? 2 * wid : 2 * wid - 2;
      coop->sum[k0][lane] = part0;
      coop->sum[k0 + 1][lane] = part1;
    }
    __syncthreads();
    cnt = coop->sum[0][lane];
    mu = coop->sum[1][lane];
    mv = coop->sum[2][lane];
    mw = coop->sum[3][lane];
    A.set_sums(coop->sum[4][lane], coop->sum[5][lane], coop->sum[6][lane]);
    B.set_sums(coop->sum[7][lane], coop->sum[8][lane], coop->sum[9][lane]);
    bestf = coop->sum[10][lane];
    bestidx = __float_as_int(coop->sum[11][lane]);
  }
  Partial o;
  o.cnt = cnt;
  o.mx = world_comp(0, L, mu, mv, mw);
  o.my = world_comp(1, L, mu, mv, mw);
  o.mz = world_comp(2, L, mu, mv, mw);
  o.gx = A.world(0, L, r, swap) - B.world(0, L, r, !swap);
  o.gy = A.world(1, L, r, swap) - B.world(1, L, r, !swap);
  o.gz = A.world(2, L, r, swap) - B.world(2, L, r, !swap);
  o.bestf = bestf;
  o.bestidx = bestidx;
  o.touched = total > 0;
  o.deferred = false;
  return o;
}

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(kFull, v, off);
  return v;
}

// Warp sums of (a, b, c) by halving exchanges (7 shuffles): lanes 4, 5, 6
// return the sums of a, b, c (other lanes: partial values).
__device__ __forceinline__ float warp_sum3_to_456(float a, float b, float c) {
  const int lane = threadIdx.x & 31;
  const bool b4 = (lane >> 4) & 1, b3 = (lane >> 3) & 1;
  // (a, b) on lanes with bit 4 clear, (c, 0) on the others
  const float h0 = (b4 ? c : a) + __shfl_xor_sync(kFull, b4 ? a : c, 16);
  const float h1 = (b4 ? 0.f : b) + __shfl_xor_sync(kFull, b4 ? b : 0.f, 16);
  // component 2 b4 + b3
  float h = (b3 ? h1 : h0) + __shfl_xor_sync(kFull, b3 ? h0 : h1, 8);
  h += __shfl_xor_sync(kFull, h, 4);
  h += __shfl_xor_sync(kFull, h, 2);
  h += __shfl_xor_sync(kFull, h, 1);
  // lane 4 + c reads the lane holding component c (c = 0: lane 0, 1: lane 8, 2: lane 16)
  const int c3 = lane - 4;
  return __shfl_sync(kFull, h, (c3 >= 0 && c3 < 3) ? 8 * c3 : 0);
}

// Tile reduction.  Sharp mode: counts and moments are exact integers, summed
// with integer warp reductions; the deepest node via an integer max of an
// order-preserving key and an integer min of the node index among the ties.
template <bool SMOOTH>
__device__ __forceinline__ float reduce_tile(const Partial& o) {
  const int lane = threadIdx.x & 31;
  float c, x, y, z;
  if (SMOOTH) {
    c = warp_sum(o.cnt); x = warp_sum(o.mx); y = warp_sum(o.my); z = warp_sum(o.mz);
  } else {
    c = static_cast<float>(__reduce_add_sync(kFull, __float2int_rn(o.cnt)));
    x = static_cast<float>(__reduce_add_sync(kFull, __float2int_rn(o.mx)));
    y = static_cast<float>(__reduce_add_sync(kFull, __float2int_rn(o.my)));
    z = static_cast<float>(__reduce_add_sync(kFull, __float2int_rn(o.mz)));
  }
  const float g = warp_sum3_to_456(o.gx, o.gy, o.gz);   // lanes 4, 5, 6
  const int key = __reduce_max_sync(kFull, float_key(o.bestf));
  const int idx = __reduce_min_sync(kFull, float_key(o.bestf) == key ? o.bestidx : 0x7fffffff);
  float v = c;
  v = lane == 1 ? x : v;
  v = lane == 2 ? y : v;
  v = lane == 3 ? z : v;
  v = (lane >= 4 && lane < 7) ? g : v;
  v = lane == 7 ? key_float(key) : v;
  v = lane == 8 ? __int_as_float(idx) : v;
  return v;   // lane c < 9: component c of the tile partial
}

// The partial of a tile in which no node was evaluated: zero sums, no deepest node.
__device__ __forceinline__ float empty_partial() {
  const int lane = threadIdx.x & 31;
  return lane == 7 ? -FLT_MAX : (lane == 8 ? __int_as_float(0x7fffffff) : 0.f);
}

// The force law of the n <= 8 overlapping pairs staged in ov (whole warp).
template <int SET, bool LAW>
__device__ __forceinline__ void flush_overlaps(const Params& P, const Shapes& S, const Parts& D, const Lists& W,
                                               const double* vel, double* pair_out, OvlRec* ov, int nov) {
  if (nov == 0) return;
  __syncwarp();
  const ForceArgs a = force_args(P, S, D, W, vel, pair_out);
  pair_force_law<SET, LAW>(a, ov, nov);
  __syncwarp();
}

// End of a pair (called by the whole warp once all its nodes are summed):
// lanes c < 7 hold the FP64 sum of component c, every lane the deepest node.
// A pair without overlap keeps the zero outputs of the pair builder; an
// overlapping pair's sums go to its entry of the overlap list, flagged for the
// force law (the next kernel gathers the flagged entries, eight pairs per warp
// pass).
__device__ __forceinline__ void pair_done(const Lists& W, const PairRec& r, double sv, int idx) {
  const int lane = threadIdx.x & 31;
  const int q = r.pair;
  const double s0 = __shfl_sync(kFull, sv, 0);
  const bool hit = __double_as_longlong(s0) > 0;   // V > 0
  if (hit) {
    if (lane == 31) W.oflag[q] = 1;
    OvlRec* e = W.olist + q;
    if (lane < 7) e->s[lane] = sv;
    if (lane == 7) e->q = q;
    if (lane == 8) e->idx = idx;
    if (lane >= 9 && lane < 20) (&e->i)[lane - 9] = reinterpret_cast<const int*>(&r)[lane - 9];   // i, j, lo, dim, shift
  }
}

// After a tile: a pair of one tile is finished at once from the warp's
// registers; otherwise the partial is stored, and the warp that completes the
// pair's last tile sums all of them in FP64 in a fixed order (4 tile slots x
// 8 components per lane pattern, slots combined pairwise), whichever warp
// that is.
__device__ __forceinline__ void tile_done(const Lists& W, const PairRec& r, float v) {
  const int lane = threadIdx.x & 31;
  if (r.ntiles == 1) {
    const int idx = __shfl_sync(kFull, __float_as_int(v), 8);
    // (the hardware conversion: one issue slot on the node sweep's otherwise idle FP64 pipe)
    pair_done(W, r, lane < 7 ? static_cast<double>(v) : 0.0, idx);
    return;
  }
  const size_t t0 = static_cast<size_t>(r.tile0);
  if (lane < 9) W.partial[(t0 + r.tile) * kPartialFloats + lane] = v;
  __threadfence();
  int prev = 0;
  if (lane == 0) prev = atomicAdd(&W.pdone[r.pair], 1);
  prev = __shfl_sync(kFull, prev, 0);
  if (prev != r.ntiles - 1) return;
  __threadfence();
  const int nt = r.ntiles, slot = lane >> 3, c = lane & 7;
  double acc = 0.0;
  float bf = -FLT_MAX;
  int bi = 0x7fffffff;
  for (int tb = 0; tb < nt; tb += 32) {   // batches of 32 tiles, all loads in flight at once
    float x[8];
    int ix[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int t = tb + slot + 4 * u;
      const float* q = W.partial + (t0 + (t < nt ? t : 0)) * kPartialFloats;
      x[u] = t < nt ? __ldcg(q + c) : 0.0f;
      ix[u] = (t < nt && c == 7) ? __float_as_int(__ldcg(q + 8)) : 0x7fffffff;
    }
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int t = tb + slot + 4 * u;
      if (t < nt) {
        if (c < 7) {
          const double w = static_cast<double>(x[u]);
          acc = t == slot ? w : acc + w;
        } else if (x[u] > bf || (x[u] == bf && ix[u] < bi)) {
          bf = x[u];
          bi = ix[u];
        }
      }
    }
  }
  acc += __shfl_xor_sync(kFull, acc, 8);    // (s0 + s1) + (s2 + s3): the same on every lane
  acc += __shfl_xor_sync(kFull, acc, 16);
  for (int o = 8; o <= 16; o <<= 1) {
    const float ob = __shfl_xor_sync(kFull, bf, o);
    const int oi = __shfl_xor_sync(kFull, bi, o);
    if (ob > bf || (ob == bf && oi < bi)) { bf = ob; bi = oi; }
  }
  if (lane == 0) W.pdone[r.pair] = 0;   // ready for a repeated sweep of the same tiles
  pair_done(W, r, acc, __shfl_sync(kFull, bi, 7));
}


template <bool SMOOTH, int SET, bool COOP>
__device__ __forceinline__ Partial dispatch(const Params& P, const Shapes& S, const Parts& D, const PairRec& r,
                                            int tl, float4* smA, float4* smB, unsigned* spk, int4* own, DeepTiles* deep,
                                            Coop* coop, int nown, int total) {
  // evaluate the cheaper kind as A (G's sign flips back below); two cubes keep the record's order
  const bool swap = SET == SET_CUBE ? false : sweep_swap(r.kinds & 0xff, r.kinds >> 8);
  using E = typename std::conditional<SET == SET_CUBE, CubeEval, AnyEval<SET == SET_ALL, SET != SET_ALL>>::type;
  Partial o = sweep_tile<SMOOTH, SET, COOP, E>(P, S, D, r, swap, tl, smA, smB, spk, own, deep, coop, nown, total);
  if (swap) {
    o.gx = -o.gx; o.gy = -o.gy; o.gz = -o.gz;
  }
  return o;
}

// The warp copies a 224-byte pair record with 14 lanes x 16 bytes.
__device__ __forceinline__ int4 load_rec_part(const PairRec* src, int lane) {
  return lane < kPairRecWords / 4 ? reinterpret_cast<const int4*>(src)[lane] : make_int4(0, 0, 0, 0);
}
__device__ __forceinline__ void store_rec_part(PairRec* dst, int lane, int4 v) {
  if (lane < kPairRecWords / 4) reinterpret_cast<int4*>(dst)[lane] = v;
}

// Blocks per SM: 3 for the sphere/cuboid/cube variants (<= 85 registers, so
// 24 warps per SM: about one tile per warp at a settling box's size), 2 for
// the variant with every kind (measured faster than 3, which spills more).
template <int SET>
constexpr int kNarrowBlocks = SET == SET_ALL ? 2 : 3;

template <bool SMOOTH, int SET>
__global__ void __launch_bounds__(kWarps * 32, kNarrowBlocks<SET>) k_narrow32(Params P, Shapes S, Parts D, Lists W) {
  constexpr int NW = kWarps;
  __shared__ __align__(16) PairRec s_rec[NW][2];
  // per evaluator: a polytope's planes, then its line clip's constants (a cube: the clip constants)
  __shared__ float4 s_planes[NW][2][SET == SET_ALL ? 2 * kMaxFaces : 8];
  __shared__ unsigned s_pk[SET == SET_CUBE ? 1 : NW][kTileItemsPerLane * 32];   // clipped ranges (rolled sweep)
  __shared__ int4 s_own[NW][64];   // the lanes with clipped nodes (sweep_tile)
  __shared__ Coop s_coop;   // a shared tile's nodes
  __shared__ DeepTiles s_deep;
  pdl_begin();
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int ntiles = W.counters[1];
  // tiles w, w + W, ... of the list (W warps, numbered across the blocks first:
  // consecutive tiles, often of one pair, run on different SMs); the first
  // record is fetched with the tile count, the next one while a tile runs
  const int nwarps = gridDim.x * NW;
  int t = blockIdx.x + gridDim.x * wid;
  const int4 first = t < P.max_tiles ? load_rec_part(W.tiles + t, lane) : make_int4(0, 0, 0, 0);
  if (ntiles > P.max_tiles) return;   // capacity exceeded: the step reports ECAPACITY
  // with at most one tile per warp a tile of many node passes would be the
  // kernel's tail: the block's other warps help (leave_to_block)
  const bool share = ntiles <= nwarps;
  if (share) {
    if (threadIdx.x == 0) {
      s_deep.n = s_deep.alone = 0;
      s_deep.shared = kShareCycles - kTileCycles;
    }
    __syncthreads();
  }
  if (t < ntiles) store_rec_part(&s_rec[wid][0], lane, first);
  __syncwarp();
  int buf = 0;
  bool counted = false;   // the warp's tile among the block's deep ones
  while (t < ntiles) {
    const int tn = t + nwarps;
    const int4 next = tn < ntiles ? load_rec_part(W.tiles + tn, lane) : make_int4(0, 0, 0, 0);
    const PairRec& r = s_rec[wid][buf];
    if (record_in_bounds(P, W.err, r, true)) {
      const Partial o = dispatch<SMOOTH, SET, false>(P, S, D, r, r.tile, s_planes[wid][0], s_planes[wid][1],
                                                     s_pk[SET == SET_CUBE ? 0 : wid], s_own[wid],
                                                     share ? &s_deep : nullptr, nullptr, 0, 0);
      counted = true;
      if (!o.deferred) tile_done(W, r, o.touched ? reduce_tile<SMOOTH>(o) : empty_partial());
    }
    if (share) break;   // (one tile per warp at most: what it staged stays for the block)
    __syncwarp();
    if (tn < ntiles) store_rec_part(&s_rec[wid][buf ^ 1], lane, next);
    __syncwarp();
    buf ^= 1;
    t = tn;
  }
  if (!share) return;
  if (!counted) no_deep_tile();   // (a warp without a tile)
  __syncthreads();
  const int nd = s_deep.shared < s_deep.alone ? s_deep.n : 0;
  for (int d = 0; d < nd; ++d) {
    const int3 e = s_deep.tile[d];
    const PairRec& r = s_rec[e.x][0];
    const Partial o = dispatch<SMOOTH, SET, true>(P, S, D, r, r.tile, s_planes[e.x][0], s_planes[e.x][1], nullptr,
                                                  s_own[e.x], nullptr, &s_coop, e.y, e.z);
    if (wid == 0) tile_done(W, r, reduce_tile<SMOOTH>(o));
  }
}

// The force law of the step's overlapping pairs, up to eight per warp pass
// (four lanes each).  Bound: the FP64 pipe (one warp instruction per ~64 cycles
// and sub-partition) and, with one pass per warp, the latency of its chain.
//   * GATHER = false (up to 4096 particles): chunks of 16 consecutive pairs,
//     chunk c = b + grid * w (then c + grid * 8, ...) for warp w of block b; the
//     pairs' overlap flags and, in the same round of loads, all 16 entries of
//     the overlap list (the flagged ones are kept, in pair order), so one memory
//     round trip precedes the pass.  With one block per SM the chunks land on
//     different sub-partitions, so the passes run side by side.
//   * GATHER = true: each block collects the flagged pairs of its range, and its
//     warps take passes of eight.  Chunks of 16 filled 2.7 of the eight slots of
//     a pass (one pair in six overlaps), the ranges of single warps 4.7: 44.5 ->
//     31.0 -> 19.9 us on 52218 cubes (29242 overlapping pairs of 175090), 22.8 ->
//     20.1 -> 13.9 us with the whole contact law on 15472 spheres and cuboids.  (A
//     list written by the node sweep gave 17.5 and 12.2 us but cost the sweep
//     4.5 us, one atomic per pair or per 32.)
// The count of overlapping pairs goes to counters[5] (reported by
// contact_stats).
constexpr int kForceChunk = 16;

template <int SET, bool LAW, bool GATHER>
__global__ void __launch_bounds__(kWarps * 32, GATHER ? 2 : 1) k_force(Params P, Shapes S, Parts D, Lists W,
                                                                       const double* vel, double* pair_out) {
  __shared__ __align__(16) OvlRec s_ovl[kWarps][GATHER ? kForcePairsPerPass : kForceChunk];
  __shared__ int s_q[GATHER ? kGatherPairs : 1], s_n;
  pdl_begin();
  if (W.counters[1] > P.max_tiles) return;   // the node sweep did not run (ECAPACITY)
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int np = min(W.counters[0], P.max_pairs);
  constexpr int kPieces = static_cast<int>(sizeof(OvlRec) / 16);          // 16-byte pieces per entry
  int4* dst = reinterpret_cast<int4*>(s_ovl[wid]);
  auto pass = [&](int n) {   // the n staged entries
    __syncwarp();
#ifdef CONTACT_CHECKS
    if (lane < n) {   // the staged entries' pair and particles
      OvlRec& e = s_ovl[wid][lane];
      e.q = checked_index(W.err, e.q, P.max_pairs, 0);
      e.i = checked_index(W.err, e.i, P.n, 0);
      e.j = checked_index(W.err, e.j, P.n + P.nwall, 0);
    }
    __syncwarp();
#endif
    flush_overlaps<SET, LAW>(P, S, D, W, vel, pair_out, s_ovl[wid], n);
  };
  int nov = 0;
  if constexpr (GATHER) {
    const int per = (np + gridDim.x - 1) / gridDim.x;
    const int q1 = min(per * static_cast<int>(blockIdx.x + 1), np);
    // (two blocks per SM, the second one's passes two sub-partitions on)
    const int w = (wid + (blockIdx.x >= gridDim.x / 2 ? 2 : 0)) % kWarps;
    for (int q0 = per * static_cast<int>(blockIdx.x); q0 < q1; q0 += kGatherPairs) {
      const int cnt = gather_pairs(W.oflag, q0, min(kGatherPairs, q1 - q0), s_q, &s_n);
      if (threadIdx.x == 0) nov += cnt;
      for (int e0 = kForcePairsPerPass * w; e0 < cnt; e0 += kForcePairsPerPass * kWarps) {
        const int n = min(kForcePairsPerPass, cnt - e0);
#pragma unroll
        for (int u = 0; u < kForcePairsPerPass * kPieces / 32; ++u) {   // entry e / kPieces, part e % kPieces
          const int e = lane + 32 * u, r = e / kPieces;
          if (r < n) dst[e] = reinterpret_cast<const int4*>(W.olist + s_q[e0 + r])[e % kPieces];
        }
        pass(n);
      }
    }
  } else {
    const int nchunk = (np + kForceChunk - 1) / kForceChunk;
    constexpr int kPerLane = kForceChunk * kPieces / 32;                    // pieces per lane
    for (int c = blockIdx.x + gridDim.x * wid; c < nchunk; c += gridDim.x * kWarps) {
      const int q0 = kForceChunk * c;
      const int q = q0 + lane;
      const bool flag = lane < kForceChunk && q < np && W.oflag[q] != 0;
      int4 piece[kPerLane];
#pragma unroll
      for (int u = 0; u < kPerLane; ++u) {   // entry e / kPieces, part e % kPieces of the chunk
        const int e = lane + 32 * u;
        const int qe = q0 + e / kPieces;
        piece[u] = qe < np ? reinterpret_cast<const int4*>(W.olist + qe)[e % kPieces] : make_int4(0, 0, 0, 0);
      }
      unsigned mask = __ballot_sync(kFull, flag);
      nov += __popc(mask);
      while (mask != 0u) {
        const int n = min(__popc(mask), kForcePairsPerPass);
        // keep the next n flagged entries, packed in pair order
        unsigned take = mask;   // the lowest n flagged entries (all of them but in a rare 9th+)
        if (n < __popc(mask)) take = mask & ((1u << __fns(mask, 0, n + 1)) - 1u);   // below the (n+1)-th
#pragma unroll
        for (int u = 0; u < kPerLane; ++u) {
          const int e = lane + 32 * u, r = e / kPieces;
          if ((take >> r) & 1u) dst[__popc(take & ((1u << r) - 1u)) * kPieces + e % kPieces] = piece[u];
        }
        mask &= ~take;
        pass(n);
      }
    }
  }
  if (lane == 0 && nov > 0) atomicAdd(&W.counters[5], nov);
}

// ---------------------------------------------------------------- FP64 form
// The all-FP64 form takes the FP32 form's tiles, one per warp or, when there are
// few, one per two to eight warps of a block; each lane clips its lines in FP32 to the nodes near both surfaces (the
// margin is above the FP32 rounding at every size (line_clip.cuh), so every node
// left out has a distance of at least w/2 in FP64 too and would add exact
// zeros), and the clipped nodes, one per lane, are evaluated in FP64.  Bound: the FP64 pipe,
// ~64 cycles a warp instruction on this GPU.  One block per pair walking every
// node of the pair box in FP64 spent 1006 us on 1934 cubes at 30 % (2.64e6
// nodes, 1 % of which add to the sums); the clipped sweep takes 31 us.

// Sums of v[0 .. 8) over the warp by halving exchanges (nine FP64 additions):
// lane c < 8 returns the sum of component c.
__device__ __forceinline__ double warp_sum8(const double v[8]) {
  const int lane = threadIdx.x & 31;
  const bool b4 = (lane >> 4) & 1, b3 = (lane >> 3) & 1, b2 = (lane >> 2) & 1;
  double h4[4], h2[2];
#pragma unroll
  for (int k = 0; k < 4; ++k) h4[k] = (b4 ? v[4 + k] : v[k]) + __shfl_xor_sync(kFull, b4 ? v[k] : v[4 + k], 16);
#pragma unroll
  for (int k = 0; k < 2; ++k) h2[k] = (b3 ? h4[2 + k] : h4[k]) + __shfl_xor_sync(kFull, b3 ? h4[k] : h4[2 + k], 8);
  double h = (b2 ? h2[1] : h2[0]) + __shfl_xor_sync(kFull, b2 ? h2[0] : h2[1], 4);
  h += __shfl_xor_sync(kFull, h, 2);
  h += __shfl_xor_sync(kFull, h, 1);
  const int c = lane & 7;   // component c sits on lanes 4 (4 b4 + 2 b3 + b2)
  return __shfl_sync(kFull, h, ((c >> 2) << 4) | (((c >> 1) & 1) << 3) | ((c & 1) << 2));
}

// After a tile of the FP64 form (lane c < 7: component c of its sums; key, idx:
// the deepest node on every lane): as tile_done, with FP64 partials.
__device__ __forceinline__ void tile_done64(const Lists& W, const PairRec& r, double v, long long key, int idx) {
  const int lane = threadIdx.x & 31;
  if (r.ntiles == 1) {
    pair_done(W, r, lane < 7 ? v : 0.0, idx);
    return;
  }
  const size_t t0 = static_cast<size_t>(r.tile0);
  double* q = W.partial64 + (t0 + r.tile) * kPartialDoubles;
  if (lane < 7) q[lane] = v;
  if (lane == 7) q[7] = __longlong_as_double(key);
  if (lane == 8) q[8] = __longlong_as_double(static_cast<long long>(idx));
  __threadfence();
  int prev = 0;
  if (lane == 0) prev = atomicAdd(&W.pdone[r.pair], 1);
  prev = __shfl_sync(kFull, prev, 0);
  if (prev != r.ntiles - 1) return;
  __threadfence();
  // component c of tiles slot, slot + 4, ..., then the four slots pairwise
  const int slot = lane >> 3, c = lane & 7;
  double acc = 0.0;
  long long bk = LLONG_MIN;
  int bi = 0x7fffffff;
  for (int t = slot; t < r.ntiles; t += 4) {
    const double* p = W.partial64 + (t0 + t) * kPartialDoubles;
    const double x = __ldcg(p + c);
    if (c < 7) {
      acc += x;
    } else {
      const long long k = __double_as_longlong(x);
      const int i = static_cast<int>(__double_as_longlong(__ldcg(p + 8)));
      if (k > bk || (k == bk && i < bi)) {
        bk = k;
        bi = i;
      }
    }
  }
  acc += __shfl_xor_sync(kFull, acc, 8);
  acc += __shfl_xor_sync(kFull, acc, 16);
  for (int o = 8; o <= 16; o <<= 1) {
    const long long ok = __shfl_xor_sync(kFull, bk, o);
    const int oi = __shfl_xor_sync(kFull, bi, o);
    if (ok > bk || (ok == bk && oi < bi)) {
      bk = ok;
      bi = oi;
    }
  }
  if (lane == 0) W.pdone[r.pair] = 0;   // ready for a repeated sweep of the same tiles
  pair_done(W, r, acc, __shfl_sync(kFull, bi, 7));
}

// What a node adds to the sums.
struct Node64 {
  double w, g[3];   // weight, band terms
  long long key;    // depth (order_key)
  int c[3], idx;    // node, linear index
};

// The sweep's shared memory, per warp of a block.
struct Shared64 {
  alignas(16) PairRec rec[kWarps];
  float4 planes[kWarps][2][2 * kMaxFaces];       // the clips' constants; then a shared tile's nodes (Node64)
  unsigned pk[kWarps][kTileItemsPerLane * 32];   // clipped ranges: first node | count << 16
  int excl[kWarps][32];                          // nodes before each lane's
};

// The tiles of the calling warp.  SHARE: G = 2, 4 or 8 warps of a block have one
// tile, warp gw of them its node passes gw, gw + G, ... (at most one tile a group).
template <bool SMOOTH, bool SHARE>
__device__ __forceinline__ void sweep64(const Params& P, const Shapes& S, const Parts& D, const Lists& W, Shared64& sm,
                                        int ntiles, int G) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const float hw = 0.5f * P.wdx_l, T = hw + P.clip_margin;
  const double inv_wdx = 1.0 / P.wdx;
  const int group = SHARE ? wid / G : wid, gw = SHARE ? wid % G : 0;
  auto group_sync = [&]() { asm volatile("bar.sync %0, %1;" ::"r"(group + 1), "r"(32 * G) : "memory"); };
  for (int t = blockIdx.x + gridDim.x * group; t < ntiles; t += SHARE ? ntiles : gridDim.x * kWarps) {
    __syncwarp();
    store_rec_part(&sm.rec[wid], lane, load_rec_part(W.tiles + t, lane));
    __syncwarp();
    const PairRec& r = sm.rec[wid];
    if (!record_in_bounds(P, W.err, r, true)) continue;   // warp-uniform (checked build only)
    const Local L = make_local(r);
    const int i = r.i, j = r.j;
    AnyEval<true, false> A, B;
    A.load(r, false, S, D, L, T, sm.planes[wid][0]);
    B.load(r, true, S, D, L, T, sm.planes[wid][1]);
    __syncwarp();
    // both particles in FP64 (the same address on every lane)
    double XA[3], XB[3], RA[9], RB[9];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      XA[k] = D.X[3 * i + k];
      XB[k] = D.X[3 * j + k] - r.shift[k] * P.L[k];
    }
#pragma unroll
    for (int k = 0; k < 9; ++k) {
      RA[k] = D.R[9 * i + k];
      RB[k] = D.R[9 * j + k];
    }
    const int ta = S.type[i], tb = S.type[j];
    const double* pla = S.planes + 4 * S.face_off[i];
    const double* plb = S.planes + 4 * S.face_off[j];
    const int nfa = S.face_off[i + 1] - S.face_off[i], nfb = S.face_off[j + 1] - S.face_off[j];
    // (A) the lane's lines clipped in FP32
    const int du = r.dim[L.u], dv = r.dim[L.v];
    const float inv_dv = __fdividef(1.f, static_cast<float>(dv));
    const int it0 = r.tile * 32 * kTileItemsPerLane;
    const int ns = min(kTileItemsPerLane, (r.nitems - it0 + 31) >> 5);
    int nl = 0;
    for (int s = 0; s < ns; ++s) {
      const int it = it0 + s * 32 + lane;
      int cv;
      const int cw = div_small(it, dv, inv_dv, &cv);
      const int len = it < r.nitems ? du : 0;
      float clo = 0.f, chi = static_cast<float>(len - 1);
      A.clip_line(r, false, L, nullptr, cv, cw, T, clo, chi);
      B.clip_line(r, true, L, nullptr, cv, cw, T, clo, chi);
      int ub;
      const int nk = clip_nodes(clo, chi, 0, len, &ub);
      sm.pk[wid][s * 32 + lane] = static_cast<unsigned>(ub) | (static_cast<unsigned>(nk) << 16);
      nl += nk;
    }
    int incl = nl;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int v = __shfl_up_sync(kFull, incl, d);
      if (lane >= d) incl += v;
    }
    const int total = __shfl_sync(kFull, incl, 31);
    sm.excl[wid][lane] = incl - nl;
    __syncwarp();
    // (B) node g of the clipped nodes on lane g mod 32
    double acc[8] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
    long long bk = LLONG_MIN;
    int bi = 0x7fffffff;
    auto node = [&](int g, Node64& e) {
      int o = 0;   // the owner: the last lane whose first node is <= g (lanes without nodes repeat the next one's)
#pragma unroll
      for (int d = 16; d > 0; d >>= 1)
        if (sm.excl[wid][o + d] <= g) o += d;
      int k = g - sm.excl[wid][o], s = 0, n;
      unsigned q = sm.pk[wid][o];
      while (k >= (n = static_cast<int>(q >> 16)) && s < ns - 1) {
        k -= n;
        q = sm.pk[wid][++s * 32 + o];
      }
      const int u = static_cast<int>(q & 0xffffu) + k;
      int cv;
      const int cw = div_small(it0 + s * 32 + o, dv, inv_dv, &cv);
      e.c[0] = L.u == 0 ? u : (L.u == 1 ? cw : cv);
      e.c[1] = L.u == 1 ? u : (L.u == 2 ? cw : cv);
      e.c[2] = L.u == 2 ? u : (L.u == 0 ? cw : cv);
      const double x[3] = {(r.lo[0] + e.c[0]) * P.dx, (r.lo[1] + e.c[1]) * P.dx, (r.lo[2] + e.c[2]) * P.dx};
      double gA[3], gB[3];
      const double pa = sdf64(ta, S.param + 3 * i, pla, nfa, XA, RA, x, P.inflate, gA);
      const double pb = sdf64(tb, S.param + 3 * j, plb, nfb, XB, RB, x, P.inflate, gB);
      const double tA = fmin(fmax(fma(-pa, inv_wdx, 0.5), 0.0), 1.0);
      const double tB = fmin(fmax(fma(-pb, inv_wdx, 0.5), 0.0), 1.0);
      double hA, hB;
      if (SMOOTH) {
        hA = tA * tA * (3.0 - 2.0 * tA);
        hB = tB * tB * (3.0 - 2.0 * tB);
      } else {
        hA = pa <= 0.0 ? 1.0 : 0.0;
        hB = pb <= 0.0 ? 1.0 : 0.0;
      }
      e.w = hA * hB;
      const double ma = tA * (1.0 - tA) * hB, mb = hA * tB * (1.0 - tB);
#pragma unroll
      for (int a = 0; a < 3; ++a) e.g[a] = ma * gA[a] - mb * gB[a];
      e.key = e.w > 0.0 ? order_key(-(pa + pb)) : LLONG_MIN;
      e.idx = e.c[0] + r.dim[0] * (e.c[1] + r.dim[1] * e.c[2]);
    };
    const bool one = !SHARE || total <= 32;   // a single pass: no partners
    if (one && gw != 0) return;
    // the warp's components of the sums, k mod G = gw or all (7: the deepest node)
    auto mine = [&](int k) { return !SHARE || one || (k & (G - 1)) == gw; };
    auto add = [&](const Node64& e) {
      if (mine(0)) acc[0] += e.w;
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        if (mine(1 + a)) acc[1 + a] = fma(e.w, fl::int_to_double(e.c[a]), acc[1 + a]);
        if (mine(4 + a)) acc[4 + a] += e.g[a];
      }
      if (mine(7) && e.w > 0.0 && (e.key > bk || (e.key == bk && e.idx < bi))) {
        bk = e.key;
        bi = e.idx;
      }
    };
    if constexpr (!SHARE) {
      for (int base = 0; base < total; base += 32) {
        if (base + lane < total) {
          Node64 e;
          node(base + lane, e);
          add(e);
        }
      }
    } else {
      // warp q's nodes, where its clips' constants were
      auto nodes = [&](int q) { return reinterpret_cast<Node64*>(sm.planes[group * G + q]); };
      static_assert(sizeof(sm.planes[0]) >= 32 * sizeof(Node64), "in the planes' place");
      for (int base0 = 0; base0 < total; base0 += 32 * G) {   // (total: the same in every warp of the group)
        const int g = base0 + 32 * gw + lane;
        if (g < total) node(g, nodes(gw)[lane]);
        __syncwarp();
        if (!one) group_sync();
        for (int q = 0; q < G && base0 + 32 * q + lane < total; ++q) add(nodes(q)[lane]);
        __syncwarp();
        if (!one) group_sync();
      }
      // the components to the group's first warp
      static_assert(2 * sizeof(sm.planes[0]) >= 8 * 32 * sizeof(double) + 32 * sizeof(int), "in the nodes' place");
      if (!one) {
        double* red = reinterpret_cast<double*>(nodes(0));
        int* red_idx = reinterpret_cast<int*>(red + 8 * 32);
#pragma unroll
        for (int k = 0; k < 8; ++k)
          if (mine(k)) red[32 * k + lane] = k < 7 ? acc[k] : __longlong_as_double(bk);
        if (mine(7)) red_idx[lane] = bi;
        group_sync();
        if (gw != 0) return;   // (one tile a group)
#pragma unroll
        for (int k = 0; k < 7; ++k) acc[k] = red[32 * k + lane];
        bk = __double_as_longlong(red[32 * 7 + lane]);
        bi = red_idx[lane];
      }
    }
    double v = 0.0;
    if (total > 0) {   // warp-uniform
      v = warp_sum8(acc);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const long long ok = __shfl_xor_sync(kFull, bk, o);
        const int oi = __shfl_xor_sync(kFull, bi, o);
        if (ok > bk || (ok == bk && oi < bi)) {
          bk = ok;
          bi = oi;
        }
      }
    }
    tile_done64(W, r, v, bk, bi);
  }
}

// Fewer tiles than warps: several warps of a block share a tile.  Each of them
// clips the lines; the sums' components are added by different warps, each in
// pass order, so they are the same bit for bit however many share.  One warp a
// tile left most sub-partitions' FP64 pipes idle: 4000 spheres, twelve pairs of
// them deep in one another, step 81 -> 46 us (one block per pair box over every
// node: 53); 100 spheres and cuboids of 26 cells between walls 495 -> 295 us,
// 400 spheres and cuboids in four layers 218 -> 106 us.
template <bool SMOOTH>
__global__ void __launch_bounds__(kWarps * 32, 2) k_narrow64(Params P, Shapes S, Parts D, Lists W) {
  __shared__ Shared64 sm;
  pdl_begin();
  const int ntiles = W.counters[1];
  if (ntiles > P.max_tiles) return;   // capacity exceeded: the step reports ECAPACITY
  const long long nwarps = static_cast<long long>(gridDim.x) * kWarps;
  int G = 1;
  while (G < kWarps && 2 * G * static_cast<long long>(ntiles) <= nwarps) G *= 2;
  if (G == 1) sweep64<SMOOTH, false>(P, S, D, W, sm, ntiles, 1);
  else sweep64<SMOOTH, true>(P, S, D, W, sm, ntiles, G);
}

}  // namespace

int kind_variant(const Params& P) {
  return P.kind_set == SET_SC && P.one_kind ? static_cast<int>(SET_ONE) : P.kind_set;
}

// f(the context's node-sweep kernel)
template <class F>
auto with_narrow32(const Params& P, const F& f) {
  switch (kind_variant(P)) {
    case SET_CUBE: return P.smooth ? f(k_narrow32<true, SET_CUBE>) : f(k_narrow32<false, SET_CUBE>);
    case SET_ONE: return P.smooth ? f(k_narrow32<true, SET_ONE>) : f(k_narrow32<false, SET_ONE>);
    case SET_SC: return P.smooth ? f(k_narrow32<true, SET_SC>) : f(k_narrow32<false, SET_SC>);
    default: return P.smooth ? f(k_narrow32<true, SET_ALL>) : f(k_narrow32<false, SET_ALL>);
  }
}

int narrow_grid(const Params& P) {
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (P.precision == 1) return sms * 2;   // k_narrow64: two resident blocks per SM
  const int per_sm = with_narrow32(P, [](auto kern) {
    int n = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kern, kWarps * 32, 0);
    return n > 0 ? n : 1;
  });
  return sms * per_sm;
}

void launch_force(const Params& P, const Shapes& S, const Parts& D, const Lists& W, const double* vel, double* pair_out,
                  cudaStream_t st) {
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  // compiled per kind set (cubes only, or any) and with or without the
  // velocity-dependent law (damping from velocities, contact history, friction)
  const bool law = P.history || P.friction || (vel != nullptr && P.damping_c != 0.0);
  const bool gather = gather_overlaps(P);
  auto kern = P.kind_set == 2 ? (law ? (gather ? k_force<2, true, true> : k_force<2, true, false>)
                                     : (gather ? k_force<2, false, true> : k_force<2, false, false>))
                              : (law ? (gather ? k_force<0, true, true> : k_force<0, true, false>)
                                     : (gather ? k_force<0, false, true> : k_force<0, false, false>));
  launch_pdl(kern, dim3((gather ? 2 : 1) * (sms > 0 ? sms : 1)), dim3(kWarps * 32), 0, st, P, S, D, W, vel, pair_out);
}

void launch_narrow(const Params& P, const Shapes& S, const Parts& D, const Lists& W, const double* vel,
                   double* pair_out, int grid, cudaStream_t st) {
  if (P.box_mode == 1) {   // the paper's box pipeline instead of every node of the pair box
    launch_box(P, S, D, W, vel, pair_out, grid, st);
    return;
  }
  if (P.precision == 1) {
    if (P.smooth)
      launch_pdl(k_narrow64<true>, dim3(grid), dim3(kWarps * 32), 0, st, P, S, D, W);
    else
      launch_pdl(k_narrow64<false>, dim3(grid), dim3(kWarps * 32), 0, st, P, S, D, W);
    return;
  }
  with_narrow32(P, [&](auto kern) { return launch_pdl(kern, dim3(grid), dim3(kWarps * 32), 0, st, P, S, D, W); });
}

}  // namespace gbc
