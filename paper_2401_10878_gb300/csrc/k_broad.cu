// Pose -> AABB, cell-list broad phase and pair planning of the contact step.
//
// Paper (arXiv:2401.10878): Sec. 3.3.1 (a contact is swept over the region
// where both particles may overlap), Sec. 3.3.2 (periodic boundaries: the
// higher-ID particle is moved to the side of the lower-ID one), Sec. 4.1
// (the neighbourhood radius is the largest circumradius).
#include <cfloat>

#include "contact_dev.cuh"
#include "line_clip.cuh"

namespace gbc {

namespace {

constexpr unsigned kFull = 0xffffffffu;

// Enter particle p with the given node range into its bin's row (one lane).
// bin: its coordinates, eight bits each.
__device__ __forceinline__ void bin_insert(const Params& P, const Lists& W, int p, int bin, const int lo[3],
                                           const int hi[3]) {
  const int b = checked_index(W.err, (bin & 0xff) + P.nbin[0] * (((bin >> 8) & 0xff) + P.nbin[1] * (bin >> 16)),
                              static_cast<long long>(P.nbin[0]) * P.nbin[1] * P.nbin[2], 0);
  const int slot = atomicAdd(&W.bin_count[b], 1);
  if (slot >= P.bin_cap) {
    set_error(W.err, kErrCapacity);
    return;
  }
  const size_t at = static_cast<size_t>(b) * P.bin_cap + slot;
  const bool empty = hi[0] < lo[0] || hi[1] < lo[1] || hi[2] < lo[2];
  unsigned len = 0;
#pragma unroll
  for (int k = 0; k < 3; ++k) len |= static_cast<unsigned>(min(hi[k] - lo[k] + 1, kMaxLen) & kMaxLen) << (10 * k);
  W.bin_items[at] = p;
  *reinterpret_cast<int4*>(W.bin_rec + at) = make_int4(empty ? kNoNodes : lo[0], lo[1], lo[2], static_cast<int>(len));
}

// ---------------------------------------------------------------------------
// K1: rotation, node range and FP32 sweep geometry of every particle, and its
// bin entry.  ROWS = 1: three lanes per particle (lane k: axis k), ten particles
// per warp; ROWS = 3: one lane per particle.  Bound: the FP64 pipe (64 cycles a
// warp instruction).  FP64 is kept to what the bit-exact node range needs, the
// same instruction for the three rows (a branch per row ran all three in turn),
// and conversions, roundings and comparisons are integer operations.  Three
// lanes give the shorter chain while every warp has a sub-partition to itself;
// above that (6080 particles) what is common to the three rows is done once for
// 32 particles instead of ten: 52218 cubes 29.8 -> 22.9 us with three lanes,
// 17.7 us with one.
template <int ROWS>
__global__ void k_pose(Params P, Shapes S, Parts D, Lists W, const double* __restrict__ pos,
                       const double* __restrict__ quat) {
  constexpr int kPer = ROWS == 1 ? 10 : 32;   // particles of one warp
  __shared__ __align__(16) int s_rec[kPer][4 * kPartRecParts];
  pdl_begin();
  const int lane = threadIdx.x;   // one-warp blocks
  const int t = blockIdx.x * 32 + lane;
  // the host's token of this step (mapped host memory: read here, stored at the end)
  const int token = (t == 0 && W.publish) ? *reinterpret_cast<const volatile int*>(W.err_host + 2) : 0;
  // the step's counters start at zero (the previous step has completed)
  if (t == 0) {
    W.counters[0] = 0;   // pairs (written by the pair builder)
    W.counters[1] = 0;   // tiles allocated
    W.counters[2] = 0;   // box pipeline: pairs with a rough contact
    W.counters[5] = 0;   // pairs with V > 0
    W.u64[0] = 0;        // node evaluations
    W.u64[1] = 0;        // nominal lane-ops
  }
  if (t < (P.n + kRowGroup - 1) / kRowGroup) W.grp_sum[t] = 0;
  // contact history: this step's lists (the buffer not read) start empty
  if (P.history && t < P.n) W.hist_n[static_cast<size_t>(((W.counters[kStepCounter] & 1) ^ 1)) * P.n + t] = 0;
  const int g = ROWS == 1 ? min(lane / 3, kPer - 1) : lane;   // the particle's place in the warp
  const int k0 = ROWS == 1 ? lane - 3 * g : 0;                // (lanes 30, 31: k = 3, 4, no stores)
  const int p_ = blockIdx.x * kPer + g;
  const bool act = k0 < 3 && p_ < P.n;
  const int p = min(p_, P.n - 1);
  double q[4];
#pragma unroll
  for (int c = 0; c < 4; ++c) q[c] = quat[4 * p + c];
  // position check by bit patterns: 0 <= X < L (NaN and negatives fail; -0.0 counts as 0)
  bool bad = false;
  double X[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const double v = pos[3 * p + c];
    long long b = __double_as_longlong(v);
    if (b == static_cast<long long>(0x8000000000000000ULL)) b = 0;
    const bool ok = b >= 0 && b < __double_as_longlong(P.L[c]);
    bad = bad || !ok;
    X[c] = ok ? __longlong_as_double(b) : 0.0;
  }
  const double nn = dadd(dadd(dadd(dmul(q[0], q[0]), dmul(q[1], q[1])), dmul(q[2], q[2])), dmul(q[3], q[3]));
  // 1e-24 < nn < 1e300 (nn >= 0 or NaN: its bits order as its values, a NaN's above every number's)
  if (!(__double_as_longlong(nn) > __double_as_longlong(1e-24)) || !(__double_as_longlong(nn) < __double_as_longlong(1e300))) {
    bad = true;
    q[0] = 1.0; q[1] = q[2] = q[3] = 0.0;
  }
  if (bad && act && k0 == 0) set_error(W.err, kErrInval);
  const double s = bad ? 2.0 : dmul(2.0, __drcp_rn(nn));
  if (act && k0 == 0)
#pragma unroll
    for (int c = 0; c < 4; ++c) D.qhat[4 * p + c] = q[c];   // raw quaternion of the step (adjoint tape)
  const int type = S.type[p];
  const double* e = S.ext + 3 * p;
  const double e0 = e[0], e1 = e[1], e2 = e[2];
  int los[3], his[3], bins[3];
#pragma unroll
  for (int row = 0; row < ROWS; ++row) {
    const int k = ROWS == 1 ? (k0 < 3 ? k0 : 0) : row;
    const int k1 = k == 2 ? 0 : k + 1;
    const double Xk = k == 0 ? X[0] : (k == 1 ? X[1] : X[2]);
    // row k of the rotation of q / |q|, body -> world, in homogeneous form (s = 2 / |q|^2;
    // 2 RN(1/nn) == RN(2/nn): scaling by 2 is exact), with the row's cyclic axes k, k1, k2:
    // 1 - s (q_k1^2 + q_k2^2), s (q_k q_k1 - w q_k2), s (q_k q_k2 + w q_k1)
    const double qk = k == 0 ? q[1] : (k == 1 ? q[2] : q[3]);
    const double qk1 = k == 0 ? q[2] : (k == 1 ? q[3] : q[1]);
    const double qk2 = k == 0 ? q[3] : (k == 1 ? q[1] : q[2]);
    const double rd = dsub(1.0, dmul(s, dadd(dmul(qk1, qk1), dmul(qk2, qk2))));
    const double r1 = dmul(s, dsub(dmul(qk, qk1), dmul(q[0], qk2)));
    const double r2 = dmul(s, dadd(dmul(qk, qk2), dmul(q[0], qk1)));
    double r[3];   // by world column c
#pragma unroll
    for (int c = 0; c < 3; ++c) r[c] = c == k ? rd : (c == k1 ? r1 : r2);
    // extent along k of the offset shape {phi <= delta} (explicit rounding: compared bit for bit);
    // a polytope's node range and bin entry come from its own warp (k_pose_poly)
    double ext = dadd(dadd(dmul(fabs(r[0]), e0), dmul(fabs(r[1]), e1)), dmul(fabs(r[2]), e2));
    if (type == 0) ext = e0;
    const double mn = dsub(Xk, ext), mx = dadd(Xk, ext);
    const int lo = ceil_node(P.dx_pow2 ? dmul(mn, P.inv_dx) : __ddiv_rn(mn, P.dx));
    const int hi = floor_node(P.dx_pow2 ? dmul(mx, P.inv_dx) : __ddiv_rn(mx, P.dx));
    // nearest node of X / dx (round to even) by the 1.5 2^52 shift, and the remainder
    const double xl = Xk * P.inv_dx;
    const double sh = __dadd_rn(xl, 6755399441055744.0);
    const int kx = __double2loint(sh);
    const float fx = narrow(__dsub_rn(xl, __dsub_rn(sh, 6755399441055744.0)));
    // cell-list bin
    const int b = min(max(static_cast<int>(narrow(Xk) * P.inv_binw_f[k]), 0), P.nbin[k] - 1);
    if (ROWS == 1) {
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        los[c] = __shfl_sync(kFull, lo, 3 * g + c);
        his[c] = __shfl_sync(kFull, hi, 3 * g + c);
        bins[c] = __shfl_sync(kFull, b, 3 * g + c);
      }
    } else {
      los[row] = lo;
      his[row] = hi;
      bins[row] = b;
    }
    if (act) {
      D.X[3 * p + k] = Xk;
#pragma unroll
      for (int c = 0; c < 3; ++c) D.R[9 * p + 3 * k + c] = r[c];
      // the particle's line, staged so that the warp stores whole 16-byte pieces
      int* w = s_rec[g];
      w[k] = lo;
      w[4 + k] = hi;
      w[8 + k] = kx;
      w[11 + 4 * k + (k == 2 ? 6 : 0)] = __float_as_int(S.size_l[3 * p + k]);   // words 11, 15, 25
      w[12 + k] = __float_as_int(fx);
#pragma unroll
      for (int c = 0; c < 3; ++c) w[16 + 3 * c + k] = __float_as_int(narrow(r[c]));   // R^T row c, column k
    }
  }
  if (act && k0 == 0) {
    const int bin = bins[0] | (bins[1] << 8) | (bins[2] << 16);   // (at most 256 bins per axis)
    int* w = s_rec[g];
    w[3] = W.kind[p] | (S.nomops[p] << 8);
    w[7] = bin;
    w[26] = w[27] = 0;
    if (type != 2) bin_insert(P, W, p, bin, los, his);
  }
  __syncwarp();
  const int np = min(kPer, P.n - static_cast<int>(blockIdx.x) * kPer);
  for (int u = lane; u < kPartRecParts * np; u += 32) {
    const int gp = u / kPartRecParts, part = u - gp * kPartRecParts;
    reinterpret_cast<int4*>(D.rec + static_cast<size_t>(blockIdx.x) * kPer + gp)[part] =
        reinterpret_cast<const int4*>(s_rec[gp])[part];
  }
  if (t == 0 && W.publish) W.counters[kTokenCounter] = token;
}

// K1b: one warp per polytope: its node range along each axis (the extreme
// projections of the offset-shape vertices: an FP32 prefilter over the
// vertices on all lanes, FP64 for the at most two candidates per side, all
// vertices in FP64 when more lie within the prefilter's window), the FP32 world
// planes (faces on lanes) and its bin entry, from the rotation k_pose wrote.
// The FP64 arithmetic is the oracle's, operation for operation, so the node
// range is the same bit for bit.  Bound: the FP64 pipe; with the candidates of
// the three axes side by side on twelve lanes and the rotation read instead of
// formed again it takes ~16 FP64 instructions a polytope (~100 before): 39.7 ->
// 15.9 us on 5157 polytopes.
__global__ void k_pose_poly(Params P, Shapes S, Parts D, Lists W) {
  pdl_begin();
  const int p = S.poly_ids[blockIdx.x];
  const int lane = threadIdx.x & 31;
  const double* Rg = D.R + 9 * static_cast<size_t>(p);
  PartRec* rec = D.rec + p;
  float R32[3][3];   // row k: world axis k
#pragma unroll
  for (int k = 0; k < 3; ++k)
#pragma unroll
    for (int c = 0; c < 3; ++c) R32[k][c] = rec->rt[3 * c + k];
  const int bin = rec->bin;
  const int v0 = S.vert_off[p], v1 = S.vert_off[p + 1];
  // FP32 prefilter: extremes per axis and the largest |w|_1
  float lo32[3] = {FLT_MAX, FLT_MAX, FLT_MAX}, hi32[3] = {-FLT_MAX, -FLT_MAX, -FLT_MAX}, wmax = 0.f;
  for (int vb = v0; vb < v1; vb += 32) {
    const int v = vb + lane;
    if (v < v1) {
      const float* w = S.verts32 + 3 * v;
      const float x0 = w[0], x1 = w[1], x2 = w[2];
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const float tv = fmaf(R32[k][0], x0, fmaf(R32[k][1], x1, R32[k][2] * x2));
        lo32[k] = fminf(lo32[k], tv);
        hi32[k] = fmaxf(hi32[k], tv);
      }
      wmax = fmaxf(wmax, fabsf(x0) + fabsf(x1) + fabsf(x2));
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      lo32[k] = fminf(lo32[k], __shfl_xor_sync(kFull, lo32[k], o));
      hi32[k] = fmaxf(hi32[k], __shfl_xor_sync(kFull, hi32[k], o));
    }
    wmax = fmaxf(wmax, __shfl_xor_sync(kFull, wmax, o));
  }
  const float tol = 1e-5f * wmax + 1e-30f;
  // candidates within tol of the FP32 extremes, the first two in vertex order;
  // lane 4 k + c keeps candidate c of axis k (0, 1: lowest; 2, 3: highest)
  const int ax = min(lane >> 2, 2), cd = lane & 3;
  int mine = v0;
  bool rare[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    int nlo = 0, nhi = 0, lc[2] = {v0, v0}, hc[2] = {v0, v0};
    for (int vb = v0; vb < v1; vb += 32) {
      const int v = vb + lane;
      float tv = 0.f;
      if (v < v1) {
        const float* w = S.verts32 + 3 * v;
        tv = fmaf(R32[k][0], w[0], fmaf(R32[k][1], w[1], R32[k][2] * w[2]));
      }
      const unsigned bl = __ballot_sync(kFull, v < v1 && tv <= lo32[k] + tol);
      const unsigned bh = __ballot_sync(kFull, v < v1 && tv >= hi32[k] - tol);
      auto take = [&](unsigned m, int* cand, int& n) {
        if (m == 0u) return;
        const int f0 = vb + __ffs(m) - 1;
        const unsigned m1 = m & (m - 1u);
        const int f1 = m1 != 0u ? vb + __ffs(m1) - 1 : f0;
        if (n == 0) {
          cand[0] = f0;
          cand[1] = f1;
        } else if (n == 1) {
          cand[1] = f0;
        }
        n += __popc(m);
      };
      take(bl, lc, nlo);
      take(bh, hc, nhi);
    }
    if (nlo < 2) lc[1] = lc[0];
    if (nhi < 2) hc[1] = hc[0];
    if (ax == k) mine = cd == 0 ? lc[0] : (cd == 1 ? lc[1] : (cd == 2 ? hc[0] : hc[1]));
    rare[k] = nlo > 2 || nhi > 2;
  }
  // exact FP64 projection of the lane's candidate; the pair's extreme by order-preserving keys
  auto proj3 = [&](double r0, double r1, double r2, int v) {
    const double* w = S.verts + 3 * v;
    return dadd(dadd(dmul(r0, w[0]), dmul(r1, w[1])), dmul(r2, w[2]));
  };
  const double ra0 = Rg[3 * ax], ra1 = Rg[3 * ax + 1], ra2 = Rg[3 * ax + 2];
  double ext = proj3(ra0, ra1, ra2, mine);
  const bool up = cd >= 2;   // lanes 0, 1 of an axis: the lower extent, lanes 2, 3: the upper
  auto better = [&](double a, double b) { return (order_key(a) > order_key(b)) == up ? a : b; };
  ext = better(ext, __shfl_xor_sync(kFull, ext, 1));
  // rare: more than two vertices at an extreme -> every vertex in FP64 (lanes over vertices)
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    if (rare[k]) {   // warp-uniform
      double l = DBL_MAX, h = -DBL_MAX;
      for (int v = v0 + lane; v < v1; v += 32) {
        const double tt = proj3(Rg[3 * k], Rg[3 * k + 1], Rg[3 * k + 2], v);
        l = fmin(l, tt);
        h = fmax(h, tt);
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        l = fmin(l, __shfl_xor_sync(kFull, l, o));
        h = fmax(h, __shfl_xor_sync(kFull, h, o));
      }
      if (ax == k) ext = better(ext, up ? h : l);
    }
  }
  {
    const double v = dadd(D.X[3 * p + ax], ext);
    const double a = P.dx_pow2 ? dmul(v, P.inv_dx) : __ddiv_rn(v, P.dx);
    const int node = up ? floor_node(a) : ceil_node(a);
    const int los[3] = {__shfl_sync(kFull, node, 0), __shfl_sync(kFull, node, 4), __shfl_sync(kFull, node, 8)};
    const int his[3] = {__shfl_sync(kFull, node, 2), __shfl_sync(kFull, node, 6), __shfl_sync(kFull, node, 10)};
    if (lane == 0) {
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        rec->lo[k] = los[k];
        rec->hi[k] = his[k];
      }
      bin_insert(P, W, p, bin, los, his);
    }
  }
  // world planes: face f on lane f (FP64 product per component, one rounding to FP32)
  const int f0 = S.face_off[p], f1 = S.face_off[p + 1];
  for (int f = f0 + lane; f < f1; f += 32) {
    const double2* e = reinterpret_cast<const double2*>(S.planes + 4 * f);
    const double2 e01 = e[0], e2x = e[1];
    float4 o;
    o.x = narrow(fma(Rg[0], e01.x, fma(Rg[1], e01.y, Rg[2] * e2x.x)));
    o.y = narrow(fma(Rg[3], e01.x, fma(Rg[4], e01.y, Rg[5] * e2x.x)));
    o.z = narrow(fma(Rg[6], e01.x, fma(Rg[7], e01.y, Rg[8] * e2x.x)));
    o.w = S.off32[f];
    D.wplane[f] = o;
  }
}

// Node range [lo_q - s n, hi_q - s n] of the partner in the image that can meet
// p's: the offset of the lower corners is brought into [-n/2, n/2].  Two ranges
// that share a node have corners less than a range's length apart, and with L >
// 4 R_max + 2 dx every range is shorter than n/2, so no other image can meet it.
__device__ __forceinline__ int image_shift(int d, int n) { return d > (n >> 1) ? 1 : (d < -(n >> 1) ? -1 : 0); }

// K3: LP lanes per particle p (a warp, or half of one).  The lanes share out
// the 27 neighbour bins of the fixed-capacity cell list (only its own one along
// an axis of one bin), number the bins' entries by a scan of the counts and
// write the entries' places to a list in shared memory; then LP entries at a
// time (node range and particle, one 16-byte and one 4-byte word) are tested
// against p's node range.  The hits are collected with warp ballots and each
// goes to its rank among the partners above (j > p) or below (j < p).  Bound:
// instruction issue on large boxes, load latency on small ones.  A lane that
// walks its own bin makes as many rounds as the fullest of the 27 has entries,
// with 58 candidates in 160 lanes, each in a line of its own, and the set-up and
// the ranks of one particle's 7 hits leave most of a warp idle: on 52218 cubes
// 48 us with a bin per lane, 37 with four lanes per bin and two particles a warp,
// 38 with the list, 29.4 with the list and two particles a warp (32 with four);
// 15472 mixed particles 20.0 -> 13.4 us, 1934 cubes 6.05 -> 5.4 us (a warp each).
constexpr int kBroadWarps = 4;   // warps of a block
constexpr int kBroadList = 96;   // candidates of one particle listed at a time
static_assert(kRowGroup % (2 * kBroadWarps) == 0, "the particles of a block share one row group");
static_assert(kBroadList % 32 == 0, "the list is read by whole warps");
// Two particles per warp from where warps of one particle each fill every SM
// sub-partition with eight: fewer leave latency and not issue as the bound (a
// warp each against half a warp: 5.4 and 6.0 us at 1934 cubes, 13.9 and 11.7 us
// at 15472 spheres and cuboids).
inline bool broad_halves(const Params& P) { return P.n > 8 * 4 * kSms; }

template <int LP>
__global__ void __launch_bounds__(kBroadWarps * 32, 8) k_broad(Params P, Parts D, Lists W) {
  constexpr int PW = 32 / LP;                // particles of a warp
  constexpr int BPL = (27 + LP - 1) / LP;    // bins of a lane
  constexpr unsigned kGroup = LP == 32 ? kFull : (1u << (LP & 31)) - 1u;
  extern __shared__ int s_buf[];
  // the block's partner count (its particles share one row group), added
  // to the group sum by the block's last warp to finish: one global atomic per block
  __shared__ int s_gsum, s_gdone;
  if (threadIdx.x == 0) {
    s_gsum = 0;
    s_gdone = 0;
  }
  __syncthreads();
  pdl_begin();
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int grp = lane / LP, hl = lane % LP, g0 = lane - hl;
  const int slot = PW * wid + grp;   // the particle's place in the block
  const int p = blockIdx.x * PW * kBroadWarps + slot;
  auto group_sum = [&](int nup) {
    if (lane == 0) {
      if (nup > 0) atomicAdd_block(&s_gsum, nup);
      __threadfence_block();
      if (atomicAdd_block(&s_gdone, 1) == kBroadWarps - 1) {   // every warp's count is in
        __threadfence_block();
        const int tot = atomicAdd_block(&s_gsum, 0);
        if (tot > 0) atomicAdd(&W.grp_sum[(blockIdx.x * PW * kBroadWarps) / kRowGroup], tot);
      }
    }
  };
  if (p - grp >= P.n) {   // (uniform) none of the warp's particles
    group_sum(0);
    return;
  }
  const int cap = P.max_nbr;
  unsigned* list = reinterpret_cast<unsigned*>(s_buf) + slot * kBroadList;   // bin entries to test
  int* hits = s_buf + PW * kBroadWarps * kBroadList + slot * 2 * cap;   // at most cap partners on either side, else ECAPACITY
  const bool own = p < P.n;
  const int4* own_rec = reinterpret_cast<const int4*>(D.rec + (own ? p : P.n - 1));
  const int4 own_lo = own_rec[0], own_hi = own_rec[1];
  const int bin = own_hi.w;
  const int plo[3] = {own_lo.x, own_lo.y, own_lo.z}, phi[3] = {own_hi.x, own_hi.y, own_hi.z};
  const bool nodes = own && plo[0] <= phi[0] && plo[1] <= phi[1] && plo[2] <= phi[2];
  // the lane's bins: first entry and count
  unsigned row[BPL];
  int num[BPL];
  bool wrapped = false;   // a bin beyond the boundary: its particles lie one period away
#pragma unroll
  for (int s = 0; s < BPL; ++s) {
    const int b = hl + LP * s;
    const int off[3] = {b % 3, (b / 3) % 3, b / 9};
    int c[3];
    bool use = b < 27 && nodes;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const int nb = P.nbin[k];
      c[k] = ((bin >> (8 * k)) & 0xff) + off[k] - 1;
      use = use && (nb >= 3 || off[k] == 1);
      if (c[k] < 0 || c[k] >= nb) {
        c[k] += c[k] < 0 ? nb : -nb;
        wrapped = true;
      }
    }
    row[s] = 0;
    num[s] = 0;
    if (use) {
      const int q = checked_index(W.err, c[0] + P.nbin[0] * (c[1] + P.nbin[1] * c[2]),
                                  static_cast<long long>(P.nbin[0]) * P.nbin[1] * P.nbin[2], 0);
      row[s] = static_cast<unsigned>(q) * static_cast<unsigned>(P.bin_cap);
      num[s] = min(W.bin_count[q], P.bin_cap);
    }
  }
  // their entries numbered lane by lane
  int total = 0;
#pragma unroll
  for (int s = 0; s < BPL; ++s) total += num[s];
  int start = total;
#pragma unroll
  for (int d = 1; d < LP; d <<= 1) {
    const int up = __shfl_up_sync(kFull, start, d, LP);
    if (hl >= d) start += up;
  }
  start -= total;
  total = __shfl_sync(kFull, start + total, LP - 1, LP);
  const int most = PW == 1 ? total : __reduce_max_sync(kFull, total);
  const bool image = __any_sync(kFull, wrapped) || P.nbin[0] < 3 || P.nbin[1] < 3 || P.nbin[2] < 3;
  const int reach[3] = {phi[0] - plo[0], phi[1] - plo[1], phi[2] - plo[2]};
  const unsigned mine = kGroup << g0, below = ((1u << lane) - 1u) & mine;
  const int4* bin_rec = reinterpret_cast<const int4*>(W.bin_rec);
  int nhit = 0;
  for (int w0 = 0; w0 < most; w0 += kBroadList) {   // (one window but for crowded bins)
    int at = start - w0;
#pragma unroll
    for (int s = 0; s < BPL; ++s) {
      const int e1 = min(num[s], kBroadList - at);
#pragma unroll 1
      for (int e = max(0, -at); e < e1; ++e) list[at + e] = row[s] + static_cast<unsigned>(e);
      at += num[s];
    }
    __syncwarp();
    const int end = min(total - w0, kBroadList), last = min(most - w0, kBroadList);
    int4 rec = make_int4(0, 0, 0, 0);
    int id = -1;
    auto fetch = [&](int c) {
      if (c < end) {
        const unsigned e = list[c];
        rec = bin_rec[e];
        id = W.bin_items[e];
      }
    };
    fetch(hl);
    for (int c = hl; c - hl < last; c += LP) {
      const int j = c < end ? checked_index(W.err, id, P.n, p) : p;
      int d[3] = {rec.x - plo[0], rec.y - plo[1], rec.z - plo[2]};
      int len[3] = {rec.w & kMaxLen, (rec.w >> 10) & kMaxLen, rec.w >> 20};
      fetch(c + LP);   // (the next round's entry, under way during this one)
      if (image) {   // (uniform) the candidate's nearest image
#pragma unroll
        for (int k = 0; k < 3; ++k) d[k] -= image_shift(d[k], P.ncell[k]) * P.ncell[k];
      }
      if (P.wide && j != p) {   // (uniform) ranges beyond kMaxLen nodes
#pragma unroll
        for (int k = 0; k < 3; ++k) len[k] = D.rec[j].hi[k] - D.rec[j].lo[k] + 1;
      }
      // the ranges share a node: the partner's corner lies above p's by at most
      // p's reach and below it by less than its own length, -len < d <= reach
      bool hit = j != p;
#pragma unroll
      for (int k = 0; k < 3; ++k)
        hit = hit && static_cast<unsigned>(d[k] + len[k] - 1) < static_cast<unsigned>(reach[k] + len[k]);
      const unsigned bh = __ballot_sync(kFull, hit);
      if (hit) {
        const int to = nhit + __popc(bh & below);
        if (to < 2 * cap) hits[to] = j;
      }
      nhit += __popc(bh & mine);
    }
    __syncwarp();
  }
  // walls (partners n + w, after every particle): lane w tests wall w with an
  // FP32 prefilter, then exactly in FP64 (the node box must be non-empty)
  for (int w0 = 0; w0 < P.nwall; w0 += LP) {
    const int w = w0 + hl;
    bool hit = false;
    if (own && w < P.nwall) {
      const double* e = P.wall + 4 * w;
      const float m0 = static_cast<float>(e[0]), m1 = static_cast<float>(e[1]), m2 = static_cast<float>(e[2]);
      const float dxf = static_cast<float>(P.dx);
      const float t0 = m0 * static_cast<float>(m0 > 0.f ? plo[0] : phi[0]);
      const float t1 = m1 * static_cast<float>(m1 > 0.f ? plo[1] : phi[1]);
      const float t2 = m2 * static_cast<float>(m2 > 0.f ? plo[2] : phi[2]);
      const float lowest = (t0 + t1 + t2) * dxf;
      const float H = static_cast<float>(e[3] + P.delta);
      // the FP32 error of `lowest` is below 1e-6 of its terms' magnitudes:
      // walls beyond 1e-4 of them skip the exact FP64 test
      const float mag = (fabsf(t0) + fabsf(t1) + fabsf(t2)) * dxf + fabsf(H) + dxf;
      if (lowest <= H + 1e-4f * mag) {
        int lo[3], hi[3];
        hit = wall_box(e, P.delta, P.dx, plo, phi, lo, hi);
      }
    }
    const unsigned bw = __ballot_sync(kFull, hit);
    if (hit) {
      const int at = nhit + __popc(bw & below);
      if (at < 2 * cap) hits[at] = P.n + w;
    }
    nhit += __popc(bw & mine);
  }
  const bool over = nhit > 2 * cap;   // (then one side has more than cap)
  nhit = min(nhit, 2 * cap);
  __syncwarp();
  // each hit to its rank on its side (unique keys): above, the hits in (p, v);
  // below, those in [0, v)
  const int longest = PW == 1 ? nhit : __reduce_max_sync(kFull, nhit);
  int nup = 0;
  for (int e0 = 0; e0 < longest; e0 += LP) {
    const int e = e0 + hl;
    const int v = e < nhit ? hits[e] : -1;
    const bool up = v > p;
    const int from = up ? p + 1 : 0;
    const unsigned key = static_cast<unsigned>(v - from);
    int r = 0;
    for (int x = 0; x < nhit; ++x) r += static_cast<unsigned>(hits[x] - from) < key ? 1 : 0;
    if (e < nhit && r < cap) (up ? W.up_list : W.dn_list)[static_cast<size_t>(p) * cap + r] = v;
    __syncwarp();
    nup += __popc(__ballot_sync(kFull, e < nhit && up) & mine);
  }
  int ndn = nhit - nup;
  if (over || nup > cap || ndn > cap) {
    if (hl == 0) set_error(W.err, kErrCapacity);
    nup = min(nup, cap);
    ndn = min(ndn, cap);
  }
  if (hl == 0 && own) {
    W.up_count[p] = nup;
    W.dn_count[p] = ndn;
  }
  group_sum(PW == 1 ? nup : nup + __shfl_xor_sync(kFull, nup, 16));
}


// K4: the candidate pairs of `rows` consecutive particles per one-warp block,
// one lane per pair (their (row, partner) found in the rows' prefix sums): the
// pair record of pair row_off[i] + r, its sweep layout and its node tiles.
// Tiles are allocated with one atomic per round; a pair's tiles are contiguous,
// and its partial sums do not depend on where they land, so the results are
// deterministic.  No FP64 but for walls: centres come as integer node + FP32
// remainder from the pose kernel.  Bound: instruction issue and load
// wavefronts on large boxes, load latency on small ones.  One warp per row left
// 28 of 32 lanes idle (3.4 partners a particle): 120 -> 27 us on 52218 cubes
// with the lanes filled, the zero outputs stored by consecutive lanes and no
// record kept of pairs without tiles.
constexpr int kBuildRows = 8;   // most rows of a block
constexpr int kUpAhead = 8;     // partners of a row fetched before its count is known
// Rows per block: eight fill a warp at 3-4 partners a row (four in the box
// pipeline, whose wider ranges give six); half as many while that leaves the
// step with fewer than two blocks per SM sub-partition, where a block's latency
// counts and not its lanes (1934 cubes: 6.4 us against
// 9.6 us with sixteen rows on two warps).
inline int build_rows(const Params& P) {
  const int rows = P.box_mode == 1 ? 4 : 8;
  return P.n < 2 * 4 * kSms * rows ? rows / 2 : rows;
}

// Store a pair record (with its tile index) as fourteen 16-byte stores from
// registers, field by field (an aggregate copy would stage it in local memory).
__device__ __forceinline__ void store_pair_rec(PairRec* dst, const PairRec& r, int tile) {
  int4* d = reinterpret_cast<int4*>(dst);
  const auto f = [](float x) { return __float_as_int(x); };
  d[0] = make_int4(r.i, r.j, r.lo[0], r.lo[1]);
  d[1] = make_int4(r.lo[2], r.dim[0], r.dim[1], r.dim[2]);
  d[2] = make_int4(r.shift[0], r.shift[1], r.shift[2], r.axis);
  d[3] = make_int4(0, 0, r.nitems, r.tile0);
  d[4] = make_int4(r.ntiles, r.kinds, r.ai[0], r.ai[1]);
  d[5] = make_int4(r.ai[2], r.bi[0], r.bi[1], r.bi[2]);
  d[6] = make_int4(f(r.af[0]), f(r.af[1]), f(r.af[2]), f(r.bf[0]));
  d[7] = make_int4(f(r.bf[1]), f(r.bf[2]), f(r.rta[0]), f(r.rta[1]));
  d[8] = make_int4(f(r.rta[2]), f(r.rta[3]), f(r.rta[4]), f(r.rta[5]));
  d[9] = make_int4(f(r.rta[6]), f(r.rta[7]), f(r.rta[8]), f(r.rtb[0]));
  d[10] = make_int4(f(r.rtb[1]), f(r.rtb[2]), f(r.rtb[3]), f(r.rtb[4]));
  d[11] = make_int4(f(r.rtb[5]), f(r.rtb[6]), f(r.rtb[7]), f(r.rtb[8]));
  d[12] = make_int4(f(r.sza[0]), f(r.sza[1]), f(r.sza[2]), f(r.szb[0]));
  d[13] = make_int4(f(r.szb[1]), f(r.szb[2]), tile, r.pair);
}
static_assert(offsetof(PairRec, rta) == 30 * 4 && offsetof(PairRec, szb) == 51 * 4 &&
                  offsetof(PairRec, pair) == 55 * 4 && sizeof(PairRec) == 14 * 16,
              "store_pair_rec follows the PairRec layout");

// Whether the regions {phi_A < Ta} and {phi_B < Tb} of the pair are
// disjoint (by more than `margin` cells, the clip margin).  A node adds to the node sweep's
// sums only when both distances lie below w/2 and, with the sharp indicator,
// one of them is <= 0; so with T = w/2 (+ the clip margin) a pair apart for
// (T, T) (smoothed), or for both (0, T) and (T, 0) (sharp), has zero
// outputs and is not queued.  Spheres, cubes, cuboids and polytopes (their
// regions are balls and boxes of half extents size + T; a polytope is bounded
// by a ball, its circumradius at each threshold from the shape tables):
// box-box by the 15 separating axes (faces of either box, edge cross
// products), ball-box by the box's closest point, ball-ball by the centre
// distance; walls are never skipped.  FP32 in lattice units: the centres
// differ by an exact integer plus the FP32 difference of two remainders, and
// every rounding is far below the margin.

__device__ __forceinline__ float dot3(const float* a, const float* b) { return fmaf(a[0], b[0], fmaf(a[1], b[1], a[2] * b[2])); }

// The three threshold pairs of the test, from one set of projections: bit 0
// (T, T), bit 1 (0, T), bit 2 (T, 0) set when the regions are apart.  On an
// axis the reach of a box's region is R0 + T S (R0 its reach at 0, S the sum
// of its axes' projections), of a ball r + T or its tabulated radius.
struct Apart {
  float margin;
  unsigned bits = 0;
  __device__ __forceinline__ void axis(float proj, float ra0, float sa, float rb0, float sb, float T) {
    const float base = proj - margin - ra0 - rb0;
    bits |= (base > T * (sa + sb) ? 1u : 0u) | (base > T * sb ? 2u : 0u) | (base > T * sa ? 4u : 0u);
  }
};

__device__ unsigned pair_apart(const PairRec& r, float T, float margin) {
  const int ka = r.kinds & 0xff, kb = r.kinds >> 8;
  const bool pa = ka == KIND_POLY, pb = kb == KIND_POLY;
  const bool sa = ka == KIND_SPHERE || pa, sb = kb == KIND_SPHERE || pb;   // balls
  const bool ba = ka == KIND_CUBOID || ka == KIND_CUBE, bb = kb == KIND_CUBOID || kb == KIND_CUBE;
  if (!((sa || ba) && (sb || bb))) return 0u;
  float d[3];   // centre of B minus centre of A (lattice units)
#pragma unroll
  for (int k = 0; k < 3; ++k) d[k] = static_cast<float>(r.bi[k] - r.ai[k]) + (r.bf[k] - r.af[k]);
  Apart ap{margin};
  if (sa && sb) {
    // ball radii at 0 and at T: a sphere's r and r + T, a polytope's two tabulated radii
    const float a0 = r.sza[0], aT = pa ? r.sza[1] : r.sza[0] + T;
    const float b0 = r.szb[0], bT = pb ? r.szb[1] : r.szb[0] + T;
    const float dist = sqrtf(dot3(d, d));
    ap.axis(dist, a0, (aT - a0) / T, b0, (bT - b0) / T, T);
    return ap.bits;
  }
  if (sa || sb) {   // a ball and a box: the distance from the ball's centre to the box at each threshold
    // (element-wise selects: a runtime-chosen pointer into the record would put it in local memory)
    const bool pol = sa ? pa : pb;
    const float r0 = sa ? r.sza[0] : r.szb[0];
    const float rT = pol ? (sa ? r.sza[1] : r.szb[1]) : r0 + T;
    float y[3], sz[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {   // |ball centre - box centre| in the box frame
      const float t0 = sa ? r.rtb[3 * k] : r.rta[3 * k], t1 = sa ? r.rtb[3 * k + 1] : r.rta[3 * k + 1],
                  t2 = sa ? r.rtb[3 * k + 2] : r.rta[3 * k + 2];
      y[k] = fabsf(fmaf(t0, d[0], fmaf(t1, d[1], t2 * d[2])));
      sz[k] = sa ? r.szb[k] : r.sza[k];
    }
    // the box at 0 and at T, the ball at 0 and at T: bits as (A, B) thresholds
    float dist[2];
#pragma unroll
    for (int t = 0; t < 2; ++t) {
      float d2 = 0.f;
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const float o = fmaxf(y[k] - (sz[k] + (t ? T : 0.f)), 0.f);
        d2 = fmaf(o, o, d2);
      }
      dist[t] = sqrtf(d2) - margin;
    }
    // (T, T): box T, ball T; (0, T) and (T, 0) with the ball on side A or B
    const bool tt = dist[1] > rT, box0_ballT = dist[0] > rT, boxT_ball0 = dist[1] > r0;
    ap.bits = (tt ? 1u : 0u) | ((sa ? boxT_ball0 : box0_ballT) ? 2u : 0u) | ((sa ? box0_ballT : boxT_ball0) ? 4u : 0u);
    return ap.bits;
  }
  // two boxes: R[i][j] = a_i . b_j, t = d in A's frame; 15 axes
  float R[3][3], AR[3][3], t[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    t[i] = dot3(r.rta + 3 * i, d);
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      R[i][j] = dot3(r.rta + 3 * i, r.rtb + 3 * j);
      AR[i][j] = fabsf(R[i][j]) + 1e-6f;
    }
  }
  const float ea[3] = {r.sza[0], r.sza[1], r.sza[2]}, eb[3] = {r.szb[0], r.szb[1], r.szb[2]};
#pragma unroll
  for (int i = 0; i < 3; ++i) {   // A's faces
    const float sbi = AR[i][0] + AR[i][1] + AR[i][2];
    ap.axis(fabsf(t[i]), ea[i], 1.f, fmaf(eb[0], AR[i][0], fmaf(eb[1], AR[i][1], eb[2] * AR[i][2])), sbi, T);
  }
#pragma unroll
  for (int j = 0; j < 3; ++j) {   // B's faces
    const float tb = fmaf(t[0], R[0][j], fmaf(t[1], R[1][j], t[2] * R[2][j]));
    const float saj = AR[0][j] + AR[1][j] + AR[2][j];
    ap.axis(fabsf(tb), fmaf(ea[0], AR[0][j], fmaf(ea[1], AR[1][j], ea[2] * AR[2][j])), saj, eb[j], 1.f, T);
  }
#pragma unroll
  for (int i = 0; i < 3; ++i) {   // edge pairs a_i x b_j
    const int i1 = i == 2 ? 0 : i + 1, i2 = i1 == 2 ? 0 : i1 + 1;
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      const int j1 = j == 2 ? 0 : j + 1, j2 = j1 == 2 ? 0 : j1 + 1;
      const float ra0 = fmaf(ea[i1], AR[i2][j], ea[i2] * AR[i1][j]);
      const float rb0 = fmaf(eb[j1], AR[i][j2], eb[j2] * AR[i][j1]);
      ap.axis(fabsf(fmaf(t[i2], R[i1][j], -t[i1] * R[i2][j])), ra0, AR[i2][j] + AR[i1][j], rb0,
              AR[i][j2] + AR[i][j1], T);
    }
  }
  return ap.bits;
}

// The node range of a pair of boxes (cubes, cuboids) where both distances lie
// below T (the box pipeline's rough-detection threshold).  A node outside
// {phi_A < T} or {phi_B < T} is no rough-contact node, so the pair's node box
// shrinks to the bounding box of the intersection of the two boxes grown by T
// (half extents size + T).  The vertices of that intersection are end points
// of the edges of either box clipped to the other one, so each of the 24 edges
// (A's twelve, then B's) is clipped to the other box, grown by kCutSlack more,
// and the bounds of the end points are widened by kCutSlack.  FP32 in
// box-relative lattice units: the rounding (~1e-5 cells) stays far inside the
// slack, so every node with both distances below T is kept.  One lane per pair
// (a warp per pair with the edges on its lanes took a pair after the other:
// the kernel 26.3 -> 18.2 us on 1934 cubes).  Returns false when the
// intersection is empty.
constexpr float kCutSlack = 1e-2f;

__device__ __forceinline__ bool cut_box(const PairRec& r, float T, int nlo[3], int nhi[3]) {
  // M[a][b] = (A's body axis a) . (B's body axis b); d = centre of B - centre of A
  float M[3][3], ca[3], cb[3], d[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    ca[c] = static_cast<float>(r.ai[c]) + r.af[c];
    cb[c] = static_cast<float>(r.bi[c]) + r.bf[c];
    d[c] = cb[c] - ca[c];
  }
#pragma unroll
  for (int a = 0; a < 3; ++a)
#pragma unroll
    for (int b = 0; b < 3; ++b) M[a][b] = dot3(r.rta + 3 * a, r.rtb + 3 * b);
  float flo[3] = {FLT_MAX, FLT_MAX, FLT_MAX}, fhi[3] = {-FLT_MAX, -FLT_MAX, -FLT_MAX};
#pragma unroll
  for (int side = 0; side < 2; ++side) {   // A's edges against B's slabs, then B's against A's
    const float* ro = side ? r.rtb : r.rta;
    const float* rx = side ? r.rta : r.rtb;
    const float* eo = side ? r.szb : r.sza;
    const float* ex = side ? r.sza : r.szb;
    const float* co = side ? cb : ca;
    float base[3];   // the box's centre in the other's frame
#pragma unroll
    for (int k = 0; k < 3; ++k) base[k] = side ? dot3(rx + 3 * k, d) : -dot3(rx + 3 * k, d);
#pragma unroll
    for (int m = 0; m < 3; ++m) {   // edges along body axis m
      const int m1 = m == 2 ? 0 : m + 1, m2 = m1 == 2 ? 0 : m1 + 1;
      const float e0 = eo[m] + T, e1 = eo[m1] + T, e2 = eo[m2] + T;
      float sl[3], is[3], b1[3], b2[3];
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        sl[k] = e0 * (side ? M[k][m] : M[m][k]);
        is[k] = __fdividef(1.f, sl[k]);
        b1[k] = e1 * (side ? M[k][m1] : M[m1][k]);
        b2[k] = e2 * (side ? M[k][m2] : M[m2][k]);
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const float s1 = (q & 1) ? 1.f : -1.f, s2 = (q & 2) ? 1.f : -1.f;
        float t0 = -1.f, t1 = 1.f;   // p0 + t dv, t in [-1, 1]
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          const float p = fmaf(s2, b2[k], fmaf(s1, b1[k], base[k]));
          const float E = ex[k] + T + kCutSlack;
          if (fabsf(sl[k]) > 1e-6f) {
            const float x = (-E - p) * is[k], y = (E - p) * is[k];
            t0 = fmaxf(t0, fminf(x, y));
            t1 = fminf(t1, fmaxf(x, y));
          } else if (!(fabsf(p) <= E)) {
            t1 = -2.f;
          }
        }
        if (t0 <= t1) {
#pragma unroll
          for (int c = 0; c < 3; ++c) {
            const float p0 = fmaf(s2 * e2, ro[3 * m2 + c], fmaf(s1 * e1, ro[3 * m1 + c], co[c]));
            const float x = fmaf(t0 * e0, ro[3 * m + c], p0), y = fmaf(t1 * e0, ro[3 * m + c], p0);
            flo[c] = fminf(flo[c], fminf(x, y));
            fhi[c] = fmaxf(fhi[c], fmaxf(x, y));
          }
        }
      }
    }
  }
  bool any = true;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    any = any && flo[c] <= fhi[c];
    nlo[c] = any ? static_cast<int>(ceilf(flo[c] - kCutSlack)) : 1;
    nhi[c] = any ? static_cast<int>(floorf(fhi[c] + kCutSlack)) : 0;
    any = any && nlo[c] <= nhi[c];
  }
  return any;
}

// BOXM: the box pipeline's variant (its separation test at the rough threshold,
// the cut node boxes of two boxes, one list entry per kept pair).
template <bool BOXM>
__global__ void __launch_bounds__(32) k_build_pairs(Params P, Parts D, Lists W, int rows,
                                                               int32_t* __restrict__ pair_ij,
                                                               int32_t* __restrict__ n_pairs_out,
                                                               double* __restrict__ pair_out) {
  __shared__ int s_off[kBuildRows + 1];             // pairs before each row of the block
  __shared__ int s_up[kBuildRows][kUpAhead];        // the rows' first partners, fetched with their counts
  pdl_begin();
  const int lane = threadIdx.x;
  const int row0 = blockIdx.x * rows;
  const int nrow = min(rows, P.n - row0);
  const int cap = P.max_nbr;
#pragma unroll
  for (int u = 0; u < kBuildRows * kUpAhead / 32; ++u) {   // (entries past a row's count are stale and unused)
    const int x = lane + u * 32, rr = x / kUpAhead, k = x % kUpAhead;
    if (rr < nrow && k < cap) s_up[rr][k] = W.up_list[static_cast<size_t>(row0 + rr) * cap + k];
  }
  // the rows' partner counts and their prefix; the first pair of row0: the group sums before its
  // group plus the counts of the earlier particles of its group
  int incl = lane < nrow ? W.up_count[row0 + lane] : 0;
  const int g = row0 / kRowGroup;
  int acc = 0;
  for (int base = 0; base < g; base += 8 * 32) {
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int e = base + 32 * u + lane;
      acc += e < g ? W.grp_sum[e] : 0;
    }
  }
#pragma unroll
  for (int u = 0; u < kRowGroup / 32; ++u) {
    const int e = g * kRowGroup + 32 * u + lane;
    acc += e < row0 ? W.up_count[e] : 0;
  }
#pragma unroll
  for (int d = 1; d < kBuildRows; d <<= 1) {
    const int v = __shfl_up_sync(kFull, incl, d);
    if (lane >= d) incl += v;
  }
  if (lane < kBuildRows) s_off[lane + 1] = incl;
  if (lane == 0) s_off[0] = 0;
  const int row_base = __reduce_add_sync(kFull, acc);
  __syncwarp();
  const int total = s_off[nrow];
  if (lane < nrow) W.row_off[row0 + lane] = row_base + s_off[lane];
  if (lane == 0 && row0 + nrow == P.n) {   // the pair count: the last row's offset plus its partners
    const int all = row_base + total;
    W.counters[0] = all;
    W.row_off[P.n] = all;
    *n_pairs_out = all;
    if (all > P.max_pairs) set_error(W.err, kErrCapacity);
  }
  unsigned long long vol_sum = 0, ops_sum = 0;
  for (int base = 0; base < total; base += 32) {   // warp-uniform rounds of 32 pairs
    const int e = base + lane;
    const int pi = row_base + e;
    const bool active = e < total && pi < P.max_pairs;
    PairRec pr;
    int ntiles = 0;
    bool skip = false, cut = false;
    if (active) {
      int rr = 0;   // the last row that starts at or before the pair
#pragma unroll
      for (int d = kBuildRows / 2; d > 0; d >>= 1)
        if (rr + d < nrow && s_off[rr + d] <= e) rr += d;
      const int i = row0 + rr;
      const int k_ = e - s_off[rr];
      const int j = checked_index(W.err, k_ < kUpAhead ? s_up[rr][k_] : W.up_list[static_cast<size_t>(i) * cap + k_],
                                  P.n + P.nwall, i);
      // j's lower-partner list, fetched with j's line (slot of this pair below); a wall (j >= n) has none
      const bool wall = j >= P.n;
      const int* dl = W.dn_list + static_cast<size_t>(wall ? 0 : j) * cap;
      const int dc = wall ? 0 : checked_index(W.err, W.dn_count[j], cap + 1, 0);
      int dpre[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) dpre[u] = u < cap ? dl[u] : 0;
      // both particles' lines, 16 bytes at a time
      const int4* la = reinterpret_cast<const int4*>(D.rec + i);
      const int4* lb = reinterpret_cast<const int4*>(D.rec + j);
      const int4 a0 = la[0], a1 = la[1], a2 = la[2], a3 = la[3], a4 = la[4], a5 = la[5], a6 = la[6];
      const int4 b0 = lb[0], b1 = lb[1], b2 = lb[2], b3 = lb[3], b4 = lb[4], b5 = lb[5], b6 = lb[6];
      const int alo[3] = {a0.x, a0.y, a0.z}, ahi[3] = {a1.x, a1.y, a1.z};
      const int blo[3] = {b0.x, b0.y, b0.z}, bhi[3] = {b1.x, b1.y, b1.z};
      const int akx[3] = {a2.x, a2.y, a2.z}, bkx[3] = {b2.x, b2.y, b2.z};
      const auto f = [](int x) { return __int_as_float(x); };
      int lo[3], hi[3], shift[3] = {0, 0, 0};
      if (wall) {
        wall_box(P.wall + 4 * (j - P.n), P.delta, P.dx, alo, ahi, lo, hi);   // non-empty (tested by the broad phase)
      } else {
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          shift[k] = image_shift(blo[k] - alo[k], P.ncell[k]);
          lo[k] = max(alo[k], blo[k] - shift[k] * P.ncell[k]);
          hi[k] = min(ahi[k], bhi[k] - shift[k] * P.ncell[k]);
        }
      }
      pr.i = i;
      pr.j = j;
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        pr.shift[k] = shift[k];
        pr.lo[k] = lo[k];
        pr.dim[k] = hi[k] - lo[k] + 1;
        // X_i / dx - lo and X_j' / dx - lo = (X_j / dx - s n) - lo
        pr.ai[k] = akx[k] - lo[k];
        pr.bi[k] = bkx[k] - shift[k] * P.ncell[k] - lo[k];
      }
      // the candidate box's nodes (the cell evaluations and nominal lane-ops
      // of the step), whatever the node sweep later skips
      const unsigned long long vol =
          static_cast<unsigned long long>(static_cast<long long>(pr.dim[0]) * pr.dim[1] * pr.dim[2]);
      vol_sum += vol;
      ops_sum += vol * static_cast<unsigned long long>((a0.w >> 8) + (b0.w >> 8));
      pr.kinds = (a0.w & 0xff) | ((b0.w & 0xff) << 8);
      pr.af[0] = f(a3.x); pr.af[1] = f(a3.y); pr.af[2] = f(a3.z);
      pr.bf[0] = f(b3.x); pr.bf[1] = f(b3.y); pr.bf[2] = f(b3.z);
      pr.rta[0] = f(a4.x); pr.rta[1] = f(a4.y); pr.rta[2] = f(a4.z); pr.rta[3] = f(a4.w);
      pr.rta[4] = f(a5.x); pr.rta[5] = f(a5.y); pr.rta[6] = f(a5.z); pr.rta[7] = f(a5.w); pr.rta[8] = f(a6.x);
      pr.rtb[0] = f(b4.x); pr.rtb[1] = f(b4.y); pr.rtb[2] = f(b4.z); pr.rtb[3] = f(b4.w);
      pr.rtb[4] = f(b5.x); pr.rtb[5] = f(b5.y); pr.rtb[6] = f(b5.z); pr.rtb[7] = f(b5.w); pr.rtb[8] = f(b6.x);
      pr.sza[0] = f(a2.w); pr.sza[1] = f(a3.w); pr.sza[2] = f(a6.y);
      pr.szb[0] = f(b2.w); pr.szb[1] = f(b3.w); pr.szb[2] = f(b6.y);
      if (wall) {   // the wall's value at the box origin, m . lo - (h + inflate) / dx (lattice
                    // units), and its origin at the box origin (node offsets are box-relative)
        const double* w = P.wall + 4 * (j - P.n);
        const double p0 = ((w[0] * lo[0] + w[1] * lo[1]) + w[2] * lo[2]) - (w[3] + P.inflate) * P.inv_dx;
        pr.szb[0] = static_cast<float>(p0);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          pr.bi[k] = 0;
          pr.bf[k] = 0.f;
        }
      }
      // the node sweeps skip pairs whose distance regions are apart, and
      // so does the box pipeline (regions at its rough-detection threshold;
      // a polytope's tabulated radii belong to the node sweep's threshold, so
      // pairs with one are kept there); the skipped pairs keep their zero
      // outputs.  In the box pipeline two boxes' node box is also cut to
      // their regions' intersection (after the record is complete).
      const int ka = pr.kinds & 0xff, kb = pr.kinds >> 8;
      constexpr bool boxm = BOXM;
      const bool test = !boxm || (boxm && ka != KIND_POLY && kb != KIND_POLY);
      const unsigned apart = test ? pair_apart(pr, boxm ? kRoughT : 0.5f * P.wdx_l + P.clip_margin, P.clip_margin) : 0u;
      skip = (P.smooth || boxm) ? (apart & 1u) != 0u : (apart & 6u) == 6u;
      cut = boxm && !skip && (ka == KIND_CUBE || ka == KIND_CUBOID) && (kb == KIND_CUBE || kb == KIND_CUBOID);
      pr.tile = 0;
      pr.pair = pi;
      pair_ij[2 * static_cast<size_t>(pi)] = i;   // (the caller's array: 4-byte alignment)
      pair_ij[2 * static_cast<size_t>(pi) + 1] = j;
      // slot of this pair in j's (sorted) list of lower partners: the number of entries below i
      int s0 = 0;
#pragma unroll
      for (int u = 0; u < 8; ++u) s0 += (u < dc && dpre[u] < i) ? 1 : 0;
      for (int u = 8; u < dc; ++u) s0 += dl[u] < i ? 1 : 0;
      if (!wall) W.dn_pair[static_cast<size_t>(j) * cap + checked_index(W.err, s0, cap, 0)] = pi;
    }
    // the box pipeline's cut node boxes: the box, the centres' integer parts
    // and nothing else change, so every node keeps its FP32 distances
    if (BOXM && cut) {
      int nlo[3], nhi[3];
      bool keep = cut_box(pr, kRoughT, nlo, nhi);
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        nlo[k] = max(nlo[k], 0);
        nhi[k] = min(nhi[k], pr.dim[k] - 1);
        keep = keep && nlo[k] <= nhi[k];
      }
      if (keep) {
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          pr.lo[k] += nlo[k];
          pr.dim[k] = nhi[k] - nlo[k] + 1;
          pr.ai[k] -= nlo[k];
          pr.bi[k] -= nlo[k];
        }
      } else {
        skip = true;   // no rough-contact node: zero outputs
      }
    }
    if (active) {
      // sweep layout: whole node lines along the box's longest axis (the
      // fewest lines).  The node sweeps clip every line to the few nodes near
      // both surfaces, so a line costs about the same whatever its length
      // (selects, not a runtime index into pr.dim: that would put pr in local memory).
      const int lines_of[3] = {pr.dim[1] * pr.dim[2], pr.dim[0] * pr.dim[2], pr.dim[0] * pr.dim[1]};
      {
        const int a = pr.dim[1] > pr.dim[0] ? (pr.dim[2] > pr.dim[1] ? 2 : 1) : (pr.dim[2] > pr.dim[0] ? 2 : 0);
        pr.axis = a;
      }
      pr.nitems = pr.axis == 0 ? lines_of[0] : (pr.axis == 1 ? lines_of[1] : lines_of[2]);
      // the box pipeline takes each kept pair as one entry of the tile list
      ntiles = skip ? 0 : (BOXM ? 1 : (pr.nitems + 32 * kTileItemsPerLane - 1) / (32 * kTileItemsPerLane));
      pr.ntiles = ntiles;
    }
    // allocation aggregated over the warp (one atomic per round): the pairs'
    // tiles, contiguous per pair; tile k of a pair is entry tile0 + k of the
    // node sweep's tile list
    int tincl = ntiles;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int v = __shfl_up_sync(kFull, tincl, d);
      if (lane >= d) tincl += v;
    }
    const int wtiles = __shfl_sync(kFull, tincl, 31);
    int tbase = 0;
    if (lane == 0 && wtiles > 0) tbase = atomicAdd(&W.counters[1], wtiles);
    // while the atomic is under way: the round's pairs' outputs start as zeros (what a pair without
    // overlap keeps), consecutive lanes storing consecutive words
    {
      const size_t q0 = static_cast<size_t>(row_base) + base;
      const int np = max(0, min(min(32, total - base), P.max_pairs - (row_base + base)));
      double* po = pair_out + q0 * 11;
      for (int x = lane; x < 11 * np; x += 32) po[x] = 0.0;
      if constexpr (BOXM) {   // (the node sweep's pairs are read by their flag)
        double* pf = W.ft + q0 * kFtDoubles;
        for (int x = lane; x < kFtDoubles * np; x += 32) pf[x] = 0.0;
      }
      if (lane < np) {
        W.oflag[q0 + lane] = 0;
        W.pdone[q0 + lane] = 0;
      }
    }
    tbase = __shfl_sync(kFull, tbase, 0);
    if (ntiles > 0) {
      pr.tile0 = tbase + tincl - ntiles;
      // the tile records (beyond the tile capacity the step fails with
      // ECAPACITY and the node sweep does not run)
      for (int k = 0; k < ntiles; ++k) {
        if (pr.tile0 + k < P.max_tiles) {
          store_pair_rec(W.tiles + pr.tile0 + k, pr, k);
        } else {
          set_error(W.err, kErrCapacity);
        }
      }
    }
  }
  // the step's node evaluations and nominal lane-ops, one atomic each per block
  // (warp sums in 32 bits where they fit)
  if (__all_sync(kFull, vol_sum < (1u << 26) && ops_sum < (1u << 26))) {
    vol_sum = __reduce_add_sync(kFull, static_cast<unsigned>(vol_sum));
    ops_sum = __reduce_add_sync(kFull, static_cast<unsigned>(ops_sum));
  } else {
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) {
      vol_sum += __shfl_xor_sync(kFull, vol_sum, d);
      ops_sum += __shfl_xor_sync(kFull, ops_sum, d);
    }
  }
  if (lane == 0 && vol_sum > 0) {
    atomicAdd(&W.u64[0], vol_sum);
    atomicAdd(&W.u64[1], ops_sum);
  }
}

}  // namespace

void launch_pose(const Params& P, const Shapes& S, const Parts& D, const Lists& W, const double* pos,
                 const double* quat, cudaStream_t st) {
  // one-warp blocks: the FP64 chains of different warps land on different sub-partitions
  // (then one block per polytope for its vertices and faces)
  if (P.n > 10 * 4 * kSms) launch_pdl(k_pose<3>, dim3((P.n + 31) / 32), dim3(32), 0, st, P, S, D, W, pos, quat);
  else launch_pdl(k_pose<1>, dim3((P.n + 9) / 10), dim3(32), 0, st, P, S, D, W, pos, quat);
  if (P.npoly > 0) launch_pdl(k_pose_poly, dim3(P.npoly), dim3(32), 0, st, P, S, D, W);
}


void launch_broad(const Params& P, const Parts& D, const Lists& W, cudaStream_t st) {
  const bool halves = broad_halves(P);
  const int pw = halves ? 2 : 1;   // particles of a warp
  const size_t each = (kBroadList + 2 * static_cast<size_t>(P.max_nbr)) * sizeof(int);
  const int per = kBroadWarps * pw;   // particles of a block (at most 512 partners each: 36 KB)
  const int nb = (P.n + per - 1) / per;
  if (nb > 0)
    launch_pdl(halves ? k_broad<16> : k_broad<32>, dim3(nb), dim3(kBroadWarps * 32), per * each, st, P, D, W);
}

void launch_plan(const Params& P, const Parts& D, const Lists& W, int32_t* pair_ij, int32_t* n_pairs,
                 double* pair_out, cudaStream_t st) {
  const int rows = build_rows(P);
  const int nb = (P.n + rows - 1) / rows;
  launch_pdl(P.box_mode == 1 ? k_build_pairs<true> : k_build_pairs<false>, dim3(nb > 0 ? nb : 1), dim3(32), 0, st, P, D,
             W, rows, pair_ij, n_pairs, pair_out);
}

}  // namespace gbc
