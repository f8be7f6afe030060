// paths.cu -- duplicate-path removal, image-method validation, field, and
// the per-link reduction (a link is a transmitter-receiver pair: t * nrx + r;
// with one transmitter, the receiver index).
//
// Sec. III "Backward ray tracing":
//   step 2  a table of visited propagation paths per reflection depth: every
//           capture is keyed by (link, depth, triangle sequence); a
//           device hash table keeps one representative per distinct key
//           (the capture of the lowest ray index), and every other capture
//           is checked against it key by key (a 64-bit collision between
//           distinct keys is reported, never merged);
//   step 3  image receivers: the transmitter is mirrored in the plane of each
//           triangle of the sequence;
//   step 4  path validation: the back-trace from the receiver through the
//           images must cross each plane inside its triangle, and every
//           sub-segment must be unoccluded (FP32 any-hit over the trees);
//   step 6  per valid path: total length, delay, and the complex amplitude
//           of the ray field (Eq. 1) with the free-space spreading of Eq. 3
//           (exponent 2) and one Fresnel TE/TM reflection per bounce, with
//           vector polarisation (FP64).
// The per-link sums of amplitudes are formed in a fixed order (paths sorted
// by key), so the received power is reproducible bit for bit.
#include "paths.cuh"

#include <algorithm>

namespace dcem {

// ---------------------------------------------------------------------------
// keys
// ---------------------------------------------------------------------------
// 64-bit hash of (rx, depth, triangle sequence id_at(0..k-1)).
template <class F>
__device__ __forceinline__ unsigned long long seq_key(int rx, int k, F id_at) {
  unsigned long long h = mix64(0x9e3779b97f4a7c15ull + (unsigned long long)(unsigned)rx);
  h = mix64(h + 0x100000001b3ull * (unsigned long long)(k + 1));
  for (int j = 0; j < k; ++j)
    h = mix64(h + ((unsigned long long)(unsigned)id_at(j) | ((unsigned long long)(j + 1) << 40)));
  return h ? h : 1ull;
}

// Hit id of segment j of slot `ray` in the log ((N + T + 1) x R).
__device__ __forceinline__ int log_id_at(const PathArgs& a, int j, int ray) {
  return a.log_id[(size_t)DCEM_IDX(j, a.N + a.max_trans + 1) * a.R + DCEM_IDX(ray, a.R)];
}

// ... of `ray`'s first k logged segments.
__device__ __forceinline__ unsigned long long path_key_of(const PathArgs& a, int ray, int rx, int k) {
  return seq_key(rx, k, [&](int j) { return log_id_at(a, j, ray); });
}

// Hash-table key of a capture: its link (transmitter * nrx + receiver),
// depth and sequence, so that transmitters never share an entry.
__device__ __forceinline__ unsigned long long path_key(const PathArgs& a, Cand c) {
  return path_key_of(a, c.ray, cand_rx(c), cand_seg(c));
}

__device__ __forceinline__ bool same_key(const PathArgs& a, Cand x, Cand y) {
  if (cand_rx(x) != cand_rx(y) || cand_seg(x) != cand_seg(y)) return false;
  for (int j = 0; j < cand_seg(x); ++j)
    if (log_id_at(a, j, x.ray) != log_id_at(a, j, y.ray)) return false;
  return true;
}

__global__ void k_dedupe_insert(PathArgs a) {
  unsigned n = min(a.ctr->n_cand, a.cand_cap);
  unsigned mask = a.hcap - 1u;
  for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    Cand c = a.cand[i];
    unsigned long long h = path_key(a, c);
    unsigned slot = (unsigned)(h & mask);
    bool ok = false;
    for (unsigned p = 0; p < a.hcap; ++p) {
      unsigned long long prev = atomicCAS(&a.hkey[slot], 0ull, h);
      if (prev == 0ull || prev == h) { ok = true; break; }
      slot = (slot + 1u) & mask;
    }
    if (!ok) {
      atomicOr(&a.ctr->err, ERR_HASH_FULL);
      a.cand_slot[i] = -1;
      continue;
    }
    a.cand_slot[i] = (int)slot;
    // representative: the capture of the lowest primary ray (a transmission
    // child counts as its primary; one primary reaches a key at most once)
    int root = c.ray < a.R0 ? c.ray : a.inst_root[DCEM_IDX(c.ray - a.R0, a.R - a.R0)];
    atomicMin(&a.hrep[slot], ((unsigned long long)(unsigned)root << 32) | i);
  }
}

__global__ void k_dedupe_unique(PathArgs a) {
  unsigned n = min(a.ctr->n_cand, a.cand_cap);
  for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    int slot = a.cand_slot[i];
    if (slot < 0) continue;
    unsigned rep = (unsigned)(a.hrep[slot] & 0xffffffffull);
    if (rep == i) {
      unsigned u = atomicAdd(&a.ctr->n_unique, 1u);
      if (u < a.ucap) a.uniq[u] = (int)i;
      else atomicOr(&a.ctr->err, ERR_UNIQUE_OVERFLOW);
    } else if (!same_key(a, a.cand[i], a.cand[DCEM_IDX(rep, a.cand_cap)])) {
      atomicOr(&a.ctr->err, ERR_HASH_COLLISION);
    }
  }
}

// Sticky mode (Sec. III "Propagation path caching", paths kept until they are
// removed): each of the previous frame's valid paths is looked up in this
// frame's table; one that no capture has joins the distinct keys as entry ~i.
__global__ void k_sticky_probe(PathArgs a) {
  unsigned n = min(*a.sticky_prev_n, a.sticky_cap);
  unsigned mask = a.hcap - 1u;
  for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const StickyKey& sk = a.sticky_prev[i];
    unsigned long long h = seq_key(sk.link, sk.depth, [&](int j) { return sk.tri[j]; });
    unsigned slot = (unsigned)(h & mask);
    bool found = false;
    for (unsigned p = 0; p < a.hcap; ++p) {
      unsigned long long kk = a.hkey[slot];
      if (kk == 0ull) break;
      if (kk == h) {
        // the same key must be the same path: compare with the representative
        Cand c = a.cand[DCEM_IDX((unsigned)(a.hrep[slot] & 0xffffffffull), a.cand_cap)];
        bool same = cand_rx(c) == sk.link && cand_seg(c) == sk.depth;
        for (int j = 0; same && j < sk.depth; ++j) same = log_id_at(a, j, c.ray) == sk.tri[j];
        if (!same) atomicOr(&a.ctr->err, ERR_HASH_COLLISION);
        found = true;
        break;
      }
      slot = (slot + 1u) & mask;
    }
    if (found) continue;
    unsigned u = atomicAdd(&a.ctr->n_unique, 1u);
    if (u < a.ucap) a.uniq[u] = ~(int)i;
    else atomicOr(&a.ctr->err, ERR_UNIQUE_OVERFLOW);
  }
}

// ---------------------------------------------------------------------------
// FP64 geometry and complex arithmetic
// ---------------------------------------------------------------------------
struct d3 {
  double x, y, z;
};
__device__ __forceinline__ d3 mk3(double x, double y, double z) { return d3{x, y, z}; }
__device__ __forceinline__ d3 operator+(d3 a, d3 b) { return mk3(a.x + b.x, a.y + b.y, a.z + b.z); }
__device__ __forceinline__ d3 operator-(d3 a, d3 b) { return mk3(a.x - b.x, a.y - b.y, a.z - b.z); }
__device__ __forceinline__ d3 operator*(d3 a, double s) { return mk3(a.x * s, a.y * s, a.z * s); }
// Dot products and complex products use explicit fused operations (half the
// FP64 instructions); cross products do not, so that those of parallel
// vectors with equal rounded products stay exactly zero.
__device__ __forceinline__ double dd(d3 a, d3 b) { return fma(a.z, b.z, fma(a.y, b.y, a.x * b.x)); }
__device__ __forceinline__ d3 dx(d3 a, d3 b) {
  return mk3(a.y * b.z - a.z * b.y, a.z * b.x - a.x * b.z, a.x * b.y - a.y * b.x);
}
__device__ __forceinline__ double dn(d3 a) { return sqrt(dd(a, a)); }
// (a reciprocal square root is one chain of dependent operations, a square
// root and a division are two; both are within an ulp or two)
__device__ __forceinline__ d3 du(d3 a) { return a * rsqrt(dd(a, a)); }

// Double-float numbers (hi + lo, two FP32 values, about 44 significant
// bits): the validation geometry in this precision runs on the FP32 pipe.
// Sums and products are formed with the error-free transformations
// (Knuth's two-sum, the FMA two-product); quotients and square roots add
// correction steps from the remainder.
struct df {
  float hi, lo;
};
__device__ __forceinline__ df two_sum(float a, float b) {
  float s = __fadd_rn(a, b), bb = __fsub_rn(s, a);
  return df{s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb))};
}
__device__ __forceinline__ df quick_two_sum(float a, float b) {
  float s = __fadd_rn(a, b);
  return df{s, __fsub_rn(b, __fsub_rn(s, a))};
}
__device__ __forceinline__ df operator+(df a, df b) {
  df s = two_sum(a.hi, b.hi), t = two_sum(a.lo, b.lo);
  df r = quick_two_sum(s.hi, __fadd_rn(s.lo, t.hi));
  return quick_two_sum(r.hi, __fadd_rn(r.lo, t.lo));
}
__device__ __forceinline__ df operator-(df a) { return df{-a.hi, -a.lo}; }
__device__ __forceinline__ df operator-(df a, df b) { return a + (-b); }
__device__ __forceinline__ df operator*(df a, df b) {
  float p = __fmul_rn(a.hi, b.hi);
  float e = __fmaf_rn(a.hi, b.hi, -p);
  e = __fmaf_rn(a.hi, b.lo, __fmaf_rn(a.lo, b.hi, e));
  return quick_two_sum(p, e);
}
__device__ __forceinline__ df operator/(df a, df b) {
  float q1 = __fdiv_rn(a.hi, b.hi);
  df r = a - b * df{q1, 0.0f};
  float q2 = __fdiv_rn(r.hi, b.hi);
  r = r - b * df{q2, 0.0f};
  float q3 = __fdiv_rn(r.hi, b.hi);
  return quick_two_sum(q1, q2) + df{q3, 0.0f};
}
__device__ __forceinline__ double root(double a) { return ::sqrt(a); }
__device__ __forceinline__ df root(df a) {
  if (!(a.hi > 0.0f)) return df{0.0f, 0.0f};
  float s = __fsqrt_rn(a.hi);
  float p = __fmul_rn(s, s), pe = __fmaf_rn(s, s, -p);
  float e = __fdiv_rn(__fadd_rn(__fsub_rn(__fsub_rn(a.hi, p), pe), a.lo), __fmul_rn(2.0f, s));
  return quick_two_sum(s, e);
}

// Scalars of the validation geometry: FP64 (default) or double-float.
template <class T> __device__ __forceinline__ T sc_of(float v);
template <> __device__ __forceinline__ double sc_of<double>(float v) { return (double)v; }
template <> __device__ __forceinline__ df sc_of<df>(float v) { return df{v, 0.0f}; }
__device__ __forceinline__ double to_d(double v) { return v; }
__device__ __forceinline__ double to_d(df v) { return (double)v.hi + (double)v.lo; }
__device__ __forceinline__ bool pos(double v) { return v > 0.0; }
__device__ __forceinline__ bool pos(df v) { return v.hi > 0.0f || (v.hi == 0.0f && v.lo > 0.0f); }
__device__ __forceinline__ bool neg(double v) { return v < 0.0; }
__device__ __forceinline__ bool neg(df v) { return v.hi < 0.0f || (v.hi == 0.0f && v.lo < 0.0f); }
__device__ __forceinline__ bool zero(double v) { return v == 0.0; }
__device__ __forceinline__ bool zero(df v) { return v.hi == 0.0f && v.lo == 0.0f; }

template <class T>
struct v3 {
  T x, y, z;
};
template <class T> __device__ __forceinline__ v3<T> operator+(v3<T> a, v3<T> b) { return {a.x + b.x, a.y + b.y, a.z + b.z}; }
template <class T> __device__ __forceinline__ v3<T> operator-(v3<T> a, v3<T> b) { return {a.x - b.x, a.y - b.y, a.z - b.z}; }
template <class T> __device__ __forceinline__ v3<T> scale(v3<T> a, T s) { return {a.x * s, a.y * s, a.z * s}; }
// (not fused: path lengths stay equal to those of a plain FP64 evaluation)
template <class T> __device__ __forceinline__ T vdot(v3<T> a, v3<T> b) { return a.x * b.x + a.y * b.y + a.z * b.z; }
template <class T> __device__ __forceinline__ v3<T> vcross(v3<T> a, v3<T> b) {
  return {a.y * b.z - a.z * b.y, a.z * b.x - a.x * b.z, a.x * b.y - a.y * b.x};
}
template <class T> __device__ __forceinline__ v3<T> vof(float x, float y, float z) {
  return {sc_of<T>(x), sc_of<T>(y), sc_of<T>(z)};
}

// Complex FP64 arithmetic: reflection coefficients, polarisation and the
// diffraction coefficient.
struct zd {
  double re, im;
};
__device__ __forceinline__ zd Z(double r, double i = 0.0) { return zd{r, i}; }
__device__ __forceinline__ zd operator+(zd a, zd b) { return Z(a.re + b.re, a.im + b.im); }
__device__ __forceinline__ zd operator-(zd a, zd b) { return Z(a.re - b.re, a.im - b.im); }
__device__ __forceinline__ zd operator*(zd a, zd b) {
  return Z(fma(a.re, b.re, -(a.im * b.im)), fma(a.re, b.im, a.im * b.re));
}
__device__ __forceinline__ zd operator*(zd a, double s) { return Z(a.re * s, a.im * s); }
__device__ __forceinline__ zd zdiv(zd a, zd b) {
  const double r = 1.0 / fma(b.re, b.re, b.im * b.im);
  return Z(fma(a.re, b.re, a.im * b.im) * r, fma(a.im, b.re, -(a.re * b.im)) * r);
}
__device__ __forceinline__ zd zexp(zd a) {
  double m = exp(a.re), sn, cs;
  sincos(a.im, &sn, &cs);
  return Z(m * cs, m * sn);
}
// principal branch (the squares cannot overflow: a permittivity from FP32
// material constants)
__device__ __forceinline__ zd zsqrt(zd a) {
  double r = sqrt(fma(a.re, a.re, a.im * a.im));
  double x = sqrt(0.5 * (r + fabs(a.re)));
  if (x == 0.0) return Z(0.0, 0.0);
  double y = a.im / (2.0 * x);
  return a.re >= 0.0 ? Z(x, y) : Z(fabs(y), a.im >= 0.0 ? x : -x);
}

__device__ __forceinline__ float fdot3(float3 a, float3 b) { return a.x * b.x + a.y * b.y + a.z * b.z; }

struct z3 {
  zd x, y, z;
};
__device__ __forceinline__ zd zdot(z3 e, d3 v) {
  return Z(fma(e.z.re, v.z, fma(e.y.re, v.y, e.x.re * v.x)), fma(e.z.im, v.z, fma(e.y.im, v.y, e.x.im * v.x)));
}
__device__ __forceinline__ d3 dir_of(d3 a, d3 b) { return du(b - a); }  // unit vector a -> b
// Polarisation of an isotropic antenna along unit d: u - (u.d) d, normalised
// (a fixed axis instead when u is along d; the path is then flagged).
__device__ __forceinline__ d3 pol_of(d3 u, d3 d, unsigned& flags) {
  d3 p = u - d * dd(u, d);
  double n2 = dd(p, p);
  if (n2 < 1e-18) {
    flags |= DCEM_PATH_POL_DEGENERATE;
    d3 ax = fabs(d.x) < 0.9 ? mk3(1, 0, 0) : mk3(0, 1, 0);
    p = ax - d * dd(ax, d);
    n2 = dd(p, p);
  }
  return p * rsqrt(n2);
}

// ---------------------------------------------------------------------------
// validation + field, with many links in three kernels (k_validate: with few,
// in one):
//   k_val_geom   one thread per distinct key: image sources, back-trace,
//                reflection points inside their triangles (FP64)
//   k_val_occ    one thread per (key, sub-segment): FP32 any-hit occlusion
//   k_val_field  one thread per distinct key: length, Fresnel, polarisation,
//                complex amplitude (FP64); valid paths go to their link's
//                bucket
// ---------------------------------------------------------------------------
// Distinct keys are few (a thousand) in most frames and tens of thousands
// with many transmitters. Few: thread t of block b takes keys b + gridDim * t,
// so that every SM gets a share.
__device__ __forceinline__ unsigned spread_index(unsigned i) { return blockIdx.x + gridDim.x * i; }
// The FP64 kernels are launched with four times the blocks that the few-keys
// case wants (there, more warps with fewer lanes each only add FP64 warp
// instructions); all of them work when there are many keys.
constexpr unsigned kManyKeys = 16384;
__device__ __forceinline__ unsigned key_blocks(unsigned nu) { return nu > kManyKeys ? gridDim.x : gridDim.x / 4; }

// Validation reuse (Sec. III "Propagation path caching": the cached paths
// are re-checked each frame; here a check is skipped when its result cannot
// have changed). The previous frame's record of the same link key is copied
// bit for bit when the receiver did not move (a coherent frame has the same
// transmitter and parameters), no triangle of the sequence belongs to an
// object that moved (so the image geometry is the same), and, for a record
// whose geometry was valid, no sub-segment meets a moved object's old or new
// box (so its occlusion test is the same).
__device__ __forceinline__ int vc_find(const PathArgs& a, unsigned long long key) {
  const unsigned mask = a.vc_cap - 1u;
  unsigned slot = (unsigned)(key & mask);
  for (unsigned p = 0; p < a.vc_cap; ++p) {
    unsigned long long k = a.vc_prev_key[slot];
    if (k == 0ull) return -1;
    if (k == key) return (int)a.vc_prev_u[slot];
    slot = (slot + 1u) & mask;
  }
  return -1;
}

__device__ __forceinline__ bool vc_reusable(const PathArgs& a, int pu, int rxi, int k, const int* ids, TStack& st) {
  if (a.rx_moved[rxi % a.nrx]) return false;
  for (int j = 0; j < k; ++j) {
    int o = a.tri_obj[ids[j] & ~(kTransBit | kDiffBit)];
    if (o >= 0 && a.obj_moved[o]) return false;
  }
  if (a.prev_vstate[pu] == 0) return true;  // invalid geometry: depends on nothing else
  const d3* xs = reinterpret_cast<const d3*>(a.prev_vpts) + (size_t)pu * (kMaxRefl + 2);
  for (int j = 0; j <= k; ++j) {
    d3 p0 = xs[j], p1 = xs[j + 1];
    d3 dv = p1 - p0;
    RayPre rp = ray_pre(f3((float)p0.x, (float)p0.y, (float)p0.z), f3((float)dv.x, (float)dv.y, (float)dv.z));
    if (seg_hits_tree(a.mvt, rp, 1.0f, st)) return false;
  }
  return true;
}

// The steps of the geometry, T = double (FP64) or df (double-float); path
// points and length are stored in FP64 either way. Both validation kernels
// below run these same operations, so a key's result does not depend on which
// of them took it.
// An interaction's triangle and its (unnormalised) normal: false when it has
// none, or is a transmission (ids with kTransBit) through an opaque material.
template <class T>
__device__ __forceinline__ bool val_triangle(const PathArgs& a, int id, v3<T>& v0, v3<T>& v1, v3<T>& v2, v3<T>& n) {
  const float4* tp = a.tris + 3 * (size_t)DCEM_IDX(a.slot_of_id[DCEM_IDX(id & ~kTransBit, a.bvh.ntris)], a.bvh.ntris);
  const float4 p0 = tp[0], p1 = tp[1], p2 = tp[2];
  v0 = vof<T>(p0.x, p0.y, p0.z);
  v1 = vof<T>(p1.x, p1.y, p1.z);
  v2 = vof<T>(p2.x, p2.y, p2.z);
  n = vcross(v1 - v0, v2 - v0);
  const bool opaque = (id & kTransBit) && !(a.mats[__float_as_int(p1.w)].w >= 0.0f);
  return !opaque && pos(vdot(n, n));
}
// step 3: the image of I in the plane of (v0, n), nn = n.n (2 / nn formed
// beside the normals would take the division off the chain of images, but its
// rounding reaches the path length: three times the phase error)
template <class T>
__device__ __forceinline__ v3<T> val_image(v3<T> I, v3<T> v0, v3<T> n, T nn) {
  return I - scale(n, sc_of<T>(2.0f) * vdot(I - v0, n) / nn);
}
// step 4: where the leg from X toward Y crosses the plane, the parameter
// within (lo, 1); false when it does not
template <class T>
__device__ __forceinline__ bool val_cross(v3<T> X, v3<T> Y, v3<T> v0, v3<T> n, T lo, T& s, v3<T>& P) {
  const v3<T> dir = Y - X;
  const T den = vdot(dir, n);
  if (zero(den)) return false;
  s = vdot(v0 - X, n) / den;
  P = X + scale(dir, s);
  return pos(s - lo) && neg(s - sc_of<T>(1.0f));
}
template <class T>
__device__ __forceinline__ bool val_inside(v3<T> v0, v3<T> v1, v3<T> v2, v3<T> n, v3<T> x) {
  return !(neg(vdot(vcross(v1 - v0, x - v0), n)) || neg(vdot(vcross(v2 - v1, x - v1), n)) ||
           neg(vdot(vcross(v0 - v2, x - v2), n)));
}

template <class T>
__global__ void __launch_bounds__(64) k_val_geom(PathArgs a) {
  extern __shared__ int sstk[];
  TStack st;
  bind_stack(st, sstk, kStackSmall);
  unsigned nu = min(a.ctr->n_unique, a.ucap);
  const bool reuse = a.reuse && a.ctr->n_moved_boxes <= a.mv_cap;
  const unsigned nb = key_blocks(nu);
  if (blockIdx.x >= nb) return;
  for (unsigned t = threadIdx.x;; t += blockDim.x) {
    unsigned u = blockIdx.x + nb * t;
    if (u >= nu) break;
    int ci = a.uniq[u];
    PathRec rec;
    int k, rxi, ray;
    int ids[kMaxRefl];
    unsigned fl0 = 0u;
    unsigned long long lkey = 0ull;  // the link key (0: a sticky record)
    if (ci >= 0) {
      Cand c = a.cand[DCEM_IDX(ci, a.cand_cap)];
      int slot = DCEM_IDX(a.cand_slot[DCEM_IDX(ci, a.cand_cap)], a.hcap);
      rec.key = a.hkey[slot];
      lkey = rec.key;
      // this slot is no longer needed: leave the table empty for the next frame
      a.hkey[slot] = 0ull;
      a.hrep[slot] = ~0ull;
      k = cand_seg(c);
      rxi = cand_rx(c);
      ray = c.ray;
      // the record's key (the output order within a link) leaves the
      // transmitter out: (receiver, depth, sequence), as a single-transmitter
      // frame has it
      if (rxi >= a.nrx) rec.key = path_key_of(a, ray, rxi % a.nrx, k);
      for (int j = 0; j < kMaxRefl; ++j) ids[j] = j < k ? log_id_at(a, j, ray) : -1;
      if (ray >= a.R0) ray = a.inst_root[DCEM_IDX(ray - a.R0, a.R - a.R0)];  // reported as its primary ray
    } else {  // sticky mode: a kept path that no capture of this frame has
      const StickyKey& sk = a.sticky_prev[~ci];
      k = sk.depth;
      rxi = sk.link;
      ray = -1;
      for (int j = 0; j < kMaxRefl; ++j) ids[j] = j < k ? sk.tri[j] : -1;
      rec.key = seq_key(rxi % a.nrx, k, [&](int j) { return ids[j]; });
      fl0 = DCEM_PATH_STICKY;
    }
    if (a.ckey) a.ckey[u] = lkey;
    if (reuse && lkey) {
      int pu = vc_find(a, lkey);
      if (pu >= 0 && vc_reusable(a, pu, rxi, k, ids, st)) {
        PathRec pr = a.prev_prec[pu];
        pr.ray = ray;  // this frame's representative
        const int ps = a.prev_vstate[pu];
        const bool valid = ps == 1 || ps == 3;
        if (ps != 0) {
          const d3* src = reinterpret_cast<const d3*>(a.prev_vpts) + (size_t)pu * (kMaxRefl + 2);
          d3* dst = reinterpret_cast<d3*>(a.vpts) + (size_t)u * (kMaxRefl + 2);
          for (int j = 0; j <= k + 1; ++j) dst[j] = src[j];
        }
        a.prec[u] = pr;
        a.vstate[u] = valid ? 3 : ps;  // 3: valid, reused (occlusion and field skip it)
        if (valid) {
          unsigned pos = atomicAdd(&a.bucket_cnt[rxi], 1u);
          if (pos < (unsigned)a.bucket_cap) a.bucket[(size_t)rxi * a.bucket_cap + pos] = (int)u;
          else atomicOr(&a.ctr->err, ERR_BUCKET_OVERFLOW);
          atomicAdd(&a.ctr->n_valid, 1u);
        }
        atomicAdd(&a.ctr->n_val_reused, 1u);
        continue;
      }
    }
    rec.rx = rxi;
    rec.depth = k;
    rec.ray = ray;
    rec.flags = fl0;
    rec.valid = 0;
    rec.pad = 0;
    rec.len = 0.0;
    rec.amp_re = rec.amp_im = 0.0;
    for (int j = 0; j < kMaxRefl; ++j) {
      rec.tri[j] = ids[j];
      rec.pts[j][0] = rec.pts[j][1] = rec.pts[j][2] = 0.0f;
    }
    // link -> transmitter and receiver
    float4 rxv = a.rx[rxi % a.nrx], txv = a.txs[rxi / a.nrx];
    v3<T> X[kMaxRefl + 2], V0[kMaxRefl], V1[kMaxRefl], V2[kMaxRefl], Nn[kMaxRefl];
    v3<T> tx = vof<T>(txv.x, txv.y, txv.z), rx = vof<T>(rxv.x, rxv.y, rxv.z);
    bool ok = true;
    // interactions: reflections (rj lists them), and transmissions straight
    // through a transmitting triangle
    int rj[kMaxRefl], m = 0;
    for (int j = 0; j < k && ok; ++j) {
      ok = val_triangle(a, ids[j], V0[j], V1[j], V2[j], Nn[j]);
      if (!(ids[j] & kTransBit)) rj[m++] = j;
    }
    // image sources I_1..I_m in the planes of the reflecting triangles
    v3<T> img[kMaxRefl + 1];
    img[0] = tx;
    for (int q = 0; q < m && ok; ++q) {
      int j = rj[q];
      img[q + 1] = val_image(img[q], V0[j], Nn[j], vdot(Nn[j], Nn[j]));
    }
    // back-trace from the receiver; XR = reflection points
    v3<T> XR[kMaxRefl + 2];
    XR[0] = tx;
    XR[m + 1] = rx;
    for (int q = m; q >= 1 && ok; --q) {
      int j = rj[q - 1];
      T sp;
      ok = val_cross(XR[q + 1], img[q], V0[j], Nn[j], sc_of<T>(0.0f), sp, XR[q]);
    }
    // the interaction points in order: a transmission crosses its plane on
    // the straight piece between the surrounding reflection points, after
    // the previous interaction of that piece; every point inside its triangle
    X[0] = tx;
    X[k + 1] = rx;
    {
      int q = 0;
      T s_prev = sc_of<T>(0.0f);
      for (int j = 0; j < k && ok; ++j) {
        if (!(ids[j] & kTransBit)) {
          X[j + 1] = XR[++q];
          s_prev = sc_of<T>(0.0f);
        } else {
          T sp;
          ok = val_cross(XR[q], XR[q + 1], V0[j], Nn[j], s_prev, sp, X[j + 1]);
          if (!ok) break;
          s_prev = sp;
        }
        ok = val_inside(V0[j], V1[j], V2[j], Nn[j], X[j + 1]);
      }
    }
    T L = sc_of<T>(0.0f);
    if (ok) {
      for (int j = 0; j <= k; ++j) {
        v3<T> e = X[j + 1] - X[j];
        L = L + root(vdot(e, e));
      }
      if (!pos(L)) ok = false;
    }
    d3* xs = reinterpret_cast<d3*>(a.vpts) + (size_t)u * (kMaxRefl + 2);
    if (ok) {
      for (int j = 0; j <= k + 1; ++j) xs[j] = mk3(to_d(X[j].x), to_d(X[j].y), to_d(X[j].z));
      rec.len = to_d(L);
    }
    a.vstate[u] = ok ? 1 : 0;   // 1 = geometry valid, occlusion pending
    a.prec[u] = rec;
  }
}

__global__ void __launch_bounds__(64) k_val_occ(PathArgs a) {
  extern __shared__ int sstk[];
  TStack st;
  bind_stack(st, sstk, kStackTrace);
  unsigned nu = min(a.ctr->n_unique, a.ucap);
  unsigned W = (unsigned)(a.N + a.max_trans) + 1u;
  unsigned total = nu * W;
  unsigned ovf = 0;
  for (unsigned t = threadIdx.x;; t += blockDim.x) {
    unsigned q = spread_index(t);
    if (q >= total) break;
    unsigned u = q / W;
    int j = (int)(q - u * W);
    if (a.vstate[u] != 1) continue;
    const PathRec& rec = a.prec[u];
    int k = rec.depth;
    if (j > k) continue;
    const d3* xs = reinterpret_cast<const d3*>(a.vpts) + (size_t)u * (kMaxRefl + 2);
    d3 p0 = xs[j], p1 = xs[j + 1];
    d3 dv = p1 - p0;
    float3 o = f3((float)p0.x, (float)p0.y, (float)p0.z);
    float3 dvf = f3((float)dv.x, (float)dv.y, (float)dv.z);
    RayPre rp = ray_pre(o, dvf);
    int ex0 = j >= 1 ? rec.tri[j - 1] & ~kTransBit : -1;
    int ex1 = j < k ? rec.tri[j] & ~kTransBit : -1;
    if (any_hit(a.bvh, rp, a.eps_occ, 1.0f - a.eps_occ, ex0, ex1, ovf, st)) a.vstate[u] = 2;  // occluded
  }
  if (ovf) {
    atomicAdd(&a.ctr->stack_overflow, 1u);
    atomicOr(&a.ctr->err, ERR_STACK);
  }
}

// Field of a valid path, in FP64 throughout (Sec. III step 6, Eq. 1): the
// directions of the sub-segments, the polarisation basis of each bounce, the
// Fresnel coefficients and the phase k L (reduced modulo 2 pi in FP64 before
// the sincos). FP64 runs at a small fraction of the FP32 rate on this GPU, so
// a key is taken by a group of kFieldLanes lanes: each lane forms the
// coefficients of its own bounces (they depend only on the path points), and
// the group's first lane then carries the field through them in order.
constexpr int kFieldLanes = 8;
constexpr int kFieldThreads = 64;
struct BounceCoef {
  double sv[3], pin[3], pout[3];  // polarisation basis: s, p before and after the bounce
  double te_re, te_im, tm_re, tm_im;  // Gamma_TE, Gamma_TM (a transmission: te_re = field factor)
  int trans;
  int pad;
};
struct FieldEnds {
  double e0[3], prx[3];  // Tx and Rx polarisation along the first and last sub-segment
  double sn, cs;          // sin, cos of the reduced phase
  unsigned fl0, fl1;
};

// The coefficients of bounce j (1..k) of path X: incoming X[j-1] -> X[j],
// outgoing X[j] -> X[j+1].
__device__ __forceinline__ void bounce_coef(const PathArgs& a, const d3* X, int id, int j, double wfac, BounceCoef& c) {
  const float4* tp = a.tris + 3 * (size_t)DCEM_IDX(a.slot_of_id[DCEM_IDX(id & ~kTransBit, a.bvh.ntris)], a.bvh.ntris);
  float4 p0 = tp[0], p1 = tp[1], p2 = tp[2];
  const float4 mt = a.mats[__float_as_int(p1.w)];
  if (id & kTransBit) {  // penetration loss L dB: field times 10^(-L/20)
    c.trans = 1;
    c.te_re = pow(10.0, -(double)mt.w / 20.0);
    return;
  }
  c.trans = 0;
  d3 din = dir_of(X[j - 1], X[j]), dout = dir_of(X[j], X[j + 1]);
  d3 q0 = mk3(p0.x, p0.y, p0.z);
  d3 nh = du(dx(mk3(p1.x, p1.y, p1.z) - q0, mk3(p2.x, p2.y, p2.z) - q0));
  double ct = fabs(dd(din, nh));
  d3 sv = dx(din, nh);
  double sn2 = dd(sv, sv);
  if (sn2 < 1e-24) {  // normal incidence: any unit vector perpendicular to n
    d3 ax = fabs(nh.x) < 0.9 ? mk3(1, 0, 0) : mk3(0, 1, 0);
    sv = du(dx(nh, ax));
  } else {
    sv = sv * rsqrt(sn2);
  }
  d3 pin = dx(sv, din), pout = dx(sv, dout);
  zd gte, gtm;
  if (mt.z != 0.0f) {
    gte = Z(-1.0);
    gtm = Z(1.0);
  } else {
    zd ec = Z((double)mt.x, (double)mt.y * wfac);
    zd root = zsqrt(ec - Z(1.0 - ct * ct));
    gte = zdiv(Z(ct) - root, Z(ct) + root);
    gtm = zdiv(ec * ct - root, ec * ct + root);
  }
  c.sv[0] = sv.x; c.sv[1] = sv.y; c.sv[2] = sv.z;
  c.pin[0] = pin.x; c.pin[1] = pin.y; c.pin[2] = pin.z;
  c.pout[0] = pout.x; c.pout[1] = pout.y; c.pout[2] = pout.z;
  c.te_re = gte.re; c.te_im = gte.im;
  c.tm_re = gtm.re; c.tm_im = gtm.im;
}
__device__ __forceinline__ void bounce_field(const BounceCoef& c, z3& E) {
  if (c.trans) {
    E.x = E.x * c.te_re;
    E.y = E.y * c.te_re;
    E.z = E.z * c.te_re;
    return;
  }
  const d3 sv = mk3(c.sv[0], c.sv[1], c.sv[2]), pin = mk3(c.pin[0], c.pin[1], c.pin[2]),
           pout = mk3(c.pout[0], c.pout[1], c.pout[2]);
  zd ts = Z(c.te_re, c.te_im) * zdot(E, sv), tpp = Z(c.tm_re, c.tm_im) * zdot(E, pin);
  E.x = ts * sv.x + tpp * pout.x;
  E.y = ts * sv.y + tpp * pout.y;
  E.z = ts * sv.z + tpp * pout.z;
}
// Phase k L reduced modulo 2 pi: subtract the nearest multiple of 2 pi, the
// product n * 2 pi taken exactly by an FMA against a two-part 2 pi.
__device__ __forceinline__ void path_phase(double freq, double L, double* sn, double* cs) {
  double kl = 2.0 * M_PI * freq / 299792458.0 * L;
  double nq = rint(kl * (0.5 / M_PI));
  double ph = fma(-nq, 6.283185307179586, kl);
  ph = fma(-nq, 2.4492935982947064e-16, ph);
  sincos(ph, sn, cs);
}
// The amplitude from the field at the receiver, the record completed and its
// place in the link's bucket.
__device__ __forceinline__ void field_done(const PathArgs& a, PathRec& rec, const d3* X, unsigned u, const z3& E, d3 prx,
                                           double sn, double cs, unsigned fl) {
  const int k = rec.depth;
  zd proj = zdot(E, prx);
  double lam = 299792458.0 / a.freq;
  double g = lam / (4.0 * M_PI) / rec.len;
  double re = proj.re * cs + proj.im * sn, im = proj.im * cs - proj.re * sn;
  rec.valid = 1;
  rec.flags |= fl;
  rec.amp_re = re * g;
  rec.amp_im = im * g;
  for (int j = 0; j < k; ++j) {
    rec.pts[j][0] = (float)X[j + 1].x;
    rec.pts[j][1] = (float)X[j + 1].y;
    rec.pts[j][2] = (float)X[j + 1].z;
  }
  int rxi = rec.rx;
  unsigned pos = atomicAdd(&a.bucket_cnt[rxi], 1u);
  if (pos < (unsigned)a.bucket_cap) a.bucket[(size_t)rxi * a.bucket_cap + pos] = (int)u;
  else atomicOr(&a.ctr->err, ERR_BUCKET_OVERFLOW);
  atomicAdd(&a.ctr->n_valid, 1u);
  if (a.sticky_next) {  // kept for the next frame
    if (rec.flags & DCEM_PATH_STICKY) atomicAdd(&a.ctr->n_sticky_valid, 1u);
    unsigned q = atomicAdd(&a.ctr->n_sticky_next, 1u);
    if (q < a.sticky_cap) {
      StickyKey sk;
      sk.link = rxi;
      sk.depth = k;
      for (int j = 0; j < kMaxRefl; ++j) sk.tri[j] = rec.tri[j];
      a.sticky_next[q] = sk;
    }
  }
}

// With many keys the FP64 pipe's throughput binds, not one key's latency: a
// lane takes a whole key (the same operations in the same order), and the
// valid keys (a third of an urban frame's) wait in a per-warp queue so that
// the warp's FP64 instructions run on full lanes.
__device__ __noinline__ void field_many(const PathArgs& a, unsigned nu, unsigned* queue) {
  const int lane = threadIdx.x & 31;
  const d3 upol = mk3(a.pol.x, a.pol.y, a.pol.z);
  const double wfac = -1.0 / (2.0 * M_PI * a.freq * 8.8541878128e-12);
  const unsigned nwarp = gridDim.x * (blockDim.x >> 5);
  int n = 0;  // waiting (warp-uniform)
  auto take = [&](int m) {
    if (lane < m) {
      const unsigned u = queue[n - m + lane];
      PathRec& rec = a.prec[u];
      const int k = rec.depth;
      const d3* X = reinterpret_cast<const d3*>(a.vpts) + (size_t)u * (kMaxRefl + 2);
      unsigned fl = 0;
      const d3 e0 = pol_of(upol, dir_of(X[0], X[1]), fl);
      z3 E = {Z(e0.x), Z(e0.y), Z(e0.z)};
      for (int j = 1; j <= k; ++j) {
        BounceCoef c;
        bounce_coef(a, X, rec.tri[j - 1], j, wfac, c);
        bounce_field(c, E);
      }
      const d3 prx = pol_of(upol, dir_of(X[k + 1], X[k]), fl);
      double sn, cs;
      path_phase(a.freq, rec.len, &sn, &cs);
      field_done(a, rec, X, u, E, prx, sn, cs, fl);
    }
    n -= m;
    __syncwarp();
  };
  for (unsigned u0 = (blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) * 32; u0 < nu; u0 += 32 * nwarp) {
    const unsigned u = u0 + lane;
    const bool valid = u < nu && a.vstate[u] == 1;
    const unsigned m = __ballot_sync(0xffffffffu, valid);
    if (valid) queue[n + __popc(m & ((1u << lane) - 1u))] = u;
    n += __popc(m);
    __syncwarp();
    if (n >= 32) take(32);
  }
  if (n > 0) take(n);
}

__global__ void __launch_bounds__(kFieldThreads) k_val_field(PathArgs a) {
  constexpr int kGroups = kFieldThreads / kFieldLanes;
  __shared__ BounceCoef scoef[kGroups][kMaxRefl];
  __shared__ FieldEnds sends[kGroups];
  __shared__ unsigned squeue[kFieldThreads / 32][64];
  const unsigned nu = min(a.ctr->n_unique, a.ucap);
  if (nu > kManyKeys) {
    field_many(a, nu, squeue[threadIdx.x >> 5]);
    return;
  }
  const unsigned nb = key_blocks(nu);
  if (blockIdx.x >= nb) return;
  const int grp = threadIdx.x / kFieldLanes, gl = threadIdx.x % kFieldLanes;
  const unsigned gmask = ((1u << kFieldLanes) - 1u) << ((threadIdx.x & 31) & ~(kFieldLanes - 1));
  const d3 upol = mk3(a.pol.x, a.pol.y, a.pol.z);
  const double wfac = -1.0 / (2.0 * M_PI * a.freq * 8.8541878128e-12);
  BounceCoef* C = scoef[grp];
  FieldEnds& ends = sends[grp];
  for (unsigned it = 0;; ++it) {
    unsigned u = blockIdx.x + nb * (grp + kGroups * it);
    if (u >= nu) break;
    if (a.vstate[u] != 1) continue;
    PathRec& rec = a.prec[u];
    const int k = rec.depth;
    const d3* X = reinterpret_cast<const d3*>(a.vpts) + (size_t)u * (kMaxRefl + 2);
    for (int j = 1 + gl; j <= k; j += kFieldLanes) bounce_coef(a, X, rec.tri[j - 1], j, wfac, C[j - 1]);
    // the ends, on lanes that hold no bounce of a path of up to 5 bounces
    if (gl == kFieldLanes - 1) {
      unsigned f = 0;
      d3 e0 = pol_of(upol, dir_of(X[0], X[1]), f);
      ends.e0[0] = e0.x; ends.e0[1] = e0.y; ends.e0[2] = e0.z;
      ends.fl0 = f;
    } else if (gl == kFieldLanes - 2) {
      unsigned f = 0;
      d3 prx = pol_of(upol, dir_of(X[k + 1], X[k]), f);
      ends.prx[0] = prx.x; ends.prx[1] = prx.y; ends.prx[2] = prx.z;
      ends.fl1 = f;
    } else if (gl == kFieldLanes - 3) {
      path_phase(a.freq, rec.len, &ends.sn, &ends.cs);
    }
    __syncwarp(gmask);
    if (gl == 0) {
      z3 E = {Z(ends.e0[0]), Z(ends.e0[1]), Z(ends.e0[2])};
      for (int j = 0; j < k; ++j) bounce_field(C[j], E);
      field_done(a, rec, X, u, E, mk3(ends.prx[0], ends.prx[1], ends.prx[2]), ends.sn, ends.cs, ends.fl0 | ends.fl1);
    }
    __syncwarp(gmask);  // the group's shared records are free again
  }
}

// ---------------------------------------------------------------------------
// few links: the three steps in one kernel, a group of lanes per key
// ---------------------------------------------------------------------------
// With few links a frame has a few hundred keys, and validation is the time
// of one key's chain of dependent FP64 operations and loads, three times over
// (the highway: geometry 33, occlusion 21, field 27 us). Here a group of
// kFieldLanes lanes takes a key through all three: each lane its own
// interaction's triangle, normal and inside test, its own leg's length and
// occlusion, its own bounce's coefficients; only the images, the back-trace
// and the field's last step run in one lane. The key's state waits in shared
// memory.
template <class T>
struct ValKey {
  v3<T> v0[kMaxRefl], v1[kMaxRefl], v2[kMaxRefl], n[kMaxRefl], img[kMaxRefl + 1], X[kMaxRefl + 2];
  T nn[kMaxRefl], leg[kMaxRefl + 1];
  d3 P[kMaxRefl + 2];
  BounceCoef coef[kMaxRefl];
  FieldEnds ends;
  int ids[kMaxRefl];
};

template <class T>
__global__ void __launch_bounds__(kFieldThreads) k_validate(PathArgs a) {
  constexpr int kGroups = kFieldThreads / kFieldLanes;
  extern __shared__ int sstk[];
  __shared__ ValKey<T> skeys[kGroups];
  TStack st;
  bind_stack(st, sstk, kStackTrace);
  const int grp = threadIdx.x / kFieldLanes, gl = threadIdx.x % kFieldLanes;
  const unsigned gmask = ((1u << kFieldLanes) - 1u) << ((threadIdx.x & 31) & ~(kFieldLanes - 1));
  ValKey<T>& S = skeys[grp];
  const unsigned nu = min(a.ctr->n_unique, a.ucap);
  const bool reuse = a.reuse && a.ctr->n_moved_boxes <= a.mv_cap;
  const d3 upol = mk3(a.pol.x, a.pol.y, a.pol.z);
  const double wfac = -1.0 / (2.0 * M_PI * a.freq * 8.8541878128e-12);
  unsigned ovf = 0;
  for (unsigned it = 0;; ++it) {
    const unsigned u = blockIdx.x + gridDim.x * (grp + kGroups * it);
    if (u >= nu) break;
    __syncwarp(gmask);  // the group's record is free again
    // ---- the key
    const int ci = a.uniq[u];
    int k, rxi, ray;
    unsigned fl0 = 0u;
    unsigned long long lkey = 0ull, key;  // the link key (0: a sticky record) and the record's
    if (ci >= 0) {
      const Cand c = a.cand[DCEM_IDX(ci, a.cand_cap)];
      const int slot = DCEM_IDX(a.cand_slot[DCEM_IDX(ci, a.cand_cap)], a.hcap);
      key = lkey = a.hkey[slot];
      k = cand_seg(c);
      rxi = cand_rx(c);
      ray = c.ray;
      for (int j = gl; j < kMaxRefl; j += kFieldLanes) S.ids[j] = j < k ? log_id_at(a, j, ray) : -1;
      __syncwarp(gmask);
      if (gl == 0) {  // the slot is no longer needed: the table stays empty for the next frame
        a.hkey[slot] = 0ull;
        a.hrep[slot] = ~0ull;
      }
      // the record's key leaves the transmitter out: (receiver, depth,
      // sequence), as a single-transmitter frame has it
      if (rxi >= a.nrx) key = seq_key(rxi % a.nrx, k, [&](int j) { return S.ids[j]; });
      if (ray >= a.R0) ray = a.inst_root[DCEM_IDX(ray - a.R0, a.R - a.R0)];  // reported as its primary ray
    } else {  // sticky mode: a kept path that no capture of this frame has
      const StickyKey& sk = a.sticky_prev[~ci];
      k = sk.depth;
      rxi = sk.link;
      ray = -1;
      for (int j = gl; j < kMaxRefl; j += kFieldLanes) S.ids[j] = j < k ? sk.tri[j] : -1;
      __syncwarp(gmask);
      key = seq_key(rxi % a.nrx, k, [&](int j) { return S.ids[j]; });
      fl0 = DCEM_PATH_STICKY;
    }
    if (a.ckey && gl == 0) a.ckey[u] = lkey;
    PathRec& rec = a.prec[u];
    d3* xs = reinterpret_cast<d3*>(a.vpts) + (size_t)u * (kMaxRefl + 2);
    // ---- the previous frame's record, when nothing it depends on moved (vc_reusable, shared out)
    if (reuse && lkey) {
      const int pu = vc_find(a, lkey);
      if (pu >= 0) {
        const int ps = a.prev_vstate[pu];
        const d3* src = reinterpret_cast<const d3*>(a.prev_vpts) + (size_t)pu * (kMaxRefl + 2);
        bool same = !a.rx_moved[rxi % a.nrx];
        for (int j = gl; j < k && same; j += kFieldLanes) {
          const int o = a.tri_obj[S.ids[j] & ~(kTransBit | kDiffBit)];
          same = !(o >= 0 && a.obj_moved[o]);
        }
        if (ps != 0)  // (invalid geometry depends on nothing else)
          for (int j = gl; j <= k && same; j += kFieldLanes) {
            const d3 p0 = src[j], dv = src[j + 1] - p0;
            const RayPre rp =
                ray_pre(f3((float)p0.x, (float)p0.y, (float)p0.z), f3((float)dv.x, (float)dv.y, (float)dv.z));
            same = !seg_hits_tree(a.mvt, rp, 1.0f, st);
          }
        if (__all_sync(gmask, same)) {
          const bool valid = ps == 1 || ps == 3;
          if (ps != 0)
            for (int j = gl; j <= k + 1; j += kFieldLanes) xs[j] = src[j];
          const int* from = reinterpret_cast<const int*>(&a.prev_prec[pu]);
          int* to = reinterpret_cast<int*>(&rec);
          static_assert(sizeof(PathRec) % sizeof(int) == 0, "record copied by words");
          for (int w = gl; w < (int)(sizeof(PathRec) / sizeof(int)); w += kFieldLanes) to[w] = from[w];
          __syncwarp(gmask);
          if (gl == 0) {
            rec.ray = ray;  // this frame's representative
            a.vstate[u] = valid ? 3 : ps;  // 3: valid, reused
            if (valid) {
              unsigned pos = atomicAdd(&a.bucket_cnt[rxi], 1u);
              if (pos < (unsigned)a.bucket_cap) a.bucket[(size_t)rxi * a.bucket_cap + pos] = (int)u;
              else atomicOr(&a.ctr->err, ERR_BUCKET_OVERFLOW);
              atomicAdd(&a.ctr->n_valid, 1u);
            }
            atomicAdd(&a.ctr->n_val_reused, 1u);
          }
          continue;
        }
      }
    }
    // ---- geometry
    const float4 rxv = a.rx[rxi % a.nrx], txv = a.txs[rxi / a.nrx];
    bool ok = true;
    for (int j = gl; j < k; j += kFieldLanes) {
      v3<T> v0, v1, v2, n;
      ok = val_triangle(a, S.ids[j], v0, v1, v2, n) && ok;
      S.v0[j] = v0;
      S.v1[j] = v1;
      S.v2[j] = v2;
      S.n[j] = n;
      S.nn[j] = vdot(n, n);
    }
    ok = __all_sync(gmask, ok);
    if (ok && gl == 0) {
      S.X[0] = vof<T>(txv.x, txv.y, txv.z);
      S.X[k + 1] = vof<T>(rxv.x, rxv.y, rxv.z);
      // images of the transmitter, by interaction (a transmission keeps the last)
      v3<T> I = S.X[0];
      for (int j = 0; j < k; ++j) {
        if (!(S.ids[j] & kTransBit)) I = val_image(I, S.v0[j], S.n[j], S.nn[j]);
        S.img[j + 1] = I;
      }
      // reflection points, from the receiver back
      v3<T> Y = S.X[k + 1];
      T sp;
      for (int j = k - 1; j >= 0 && ok; --j) {
        if (S.ids[j] & kTransBit) continue;
        v3<T> P;
        ok = val_cross(Y, S.img[j + 1], S.v0[j], S.n[j], sc_of<T>(0.0f), sp, P);
        S.X[j + 1] = Y = P;
      }
      // transmissions cross the straight piece between the surrounding
      // reflection points, each after the previous one of its piece
      v3<T> A = S.X[0];
      T s_prev = sc_of<T>(0.0f);
      for (int j = 0; j < k && ok; ++j) {
        if (!(S.ids[j] & kTransBit)) {
          A = S.X[j + 1];
          s_prev = sc_of<T>(0.0f);
          continue;
        }
        int e = j + 1;  // the piece's end: the next reflection, or the receiver
        while (e < k && (S.ids[e] & kTransBit)) ++e;
        ok = val_cross(A, S.X[e + 1], S.v0[j], S.n[j], s_prev, sp, S.X[j + 1]);
        s_prev = sp;
      }
    }
    ok = __shfl_sync(gmask, (int)ok, 0, kFieldLanes) != 0;
    T L = sc_of<T>(0.0f);
    if (ok) {
      __syncwarp(gmask);
      for (int j = gl; j < k; j += kFieldLanes) ok = val_inside(S.v0[j], S.v1[j], S.v2[j], S.n[j], S.X[j + 1]) && ok;
      for (int j = gl; j <= k; j += kFieldLanes) {
        const v3<T> e = S.X[j + 1] - S.X[j];
        S.leg[j] = root(vdot(e, e));
      }
      for (int j = gl; j <= k + 1; j += kFieldLanes)
        S.P[j] = mk3(to_d(S.X[j].x), to_d(S.X[j].y), to_d(S.X[j].z));
      ok = __all_sync(gmask, ok);
      __syncwarp(gmask);
      for (int j = 0; j <= k; ++j) L = L + S.leg[j];
      ok = ok && pos(L);
    }
    int state = ok ? 1 : 0;  // 0: no geometry, 1: valid, 2: occluded
    if (ok) {
      for (int j = gl; j <= k + 1; j += kFieldLanes) xs[j] = S.P[j];
      // ---- occlusion: the legs
      bool hit = false;
      for (int j = gl; j <= k; j += kFieldLanes) {
        const d3 p0 = S.P[j], dv = S.P[j + 1] - p0;
        const RayPre rp = ray_pre(f3((float)p0.x, (float)p0.y, (float)p0.z), f3((float)dv.x, (float)dv.y, (float)dv.z));
        const int ex0 = j >= 1 ? S.ids[j - 1] & ~kTransBit : -1, ex1 = j < k ? S.ids[j] & ~kTransBit : -1;
        hit = any_hit(a.bvh, rp, a.eps_occ, 1.0f - a.eps_occ, ex0, ex1, ovf, st) || hit;
      }
      if (__any_sync(gmask, hit)) state = 2;
    }
    // ---- the record, and the field of a valid path
    const double len = ok ? to_d(L) : 0.0;
    for (int j = gl; j < kMaxRefl; j += kFieldLanes) {
      rec.tri[j] = S.ids[j];
      rec.pts[j][0] = rec.pts[j][1] = rec.pts[j][2] = 0.0f;
    }
    if (gl == 0) {
      rec.key = key;
      rec.rx = rxi;
      rec.depth = k;
      rec.ray = ray;
      rec.flags = fl0;
      rec.valid = 0;
      rec.pad = 0;
      rec.len = len;
      rec.amp_re = rec.amp_im = 0.0;
      a.vstate[u] = state;
    }
    if (state != 1) continue;
    for (int j = 1 + gl; j <= k; j += kFieldLanes) bounce_coef(a, S.P, S.ids[j - 1], j, wfac, S.coef[j - 1]);
    // the ends, on lanes that hold no bounce of a path of up to 5 bounces
    if (gl == kFieldLanes - 1) {
      unsigned f = 0;
      d3 e0 = pol_of(upol, dir_of(S.P[0], S.P[1]), f);
      S.ends.e0[0] = e0.x; S.ends.e0[1] = e0.y; S.ends.e0[2] = e0.z;
      S.ends.fl0 = f;
    } else if (gl == kFieldLanes - 2) {
      unsigned f = 0;
      d3 prx = pol_of(upol, dir_of(S.P[k + 1], S.P[k]), f);
      S.ends.prx[0] = prx.x; S.ends.prx[1] = prx.y; S.ends.prx[2] = prx.z;
      S.ends.fl1 = f;
    } else if (gl == kFieldLanes - 3) {
      path_phase(a.freq, len, &S.ends.sn, &S.ends.cs);
    }
    __syncwarp(gmask);
    if (gl == 0) {
      z3 E = {Z(S.ends.e0[0]), Z(S.ends.e0[1]), Z(S.ends.e0[2])};
      for (int j = 0; j < k; ++j) bounce_field(S.coef[j], E);
      field_done(a, rec, S.P, u, E, mk3(S.ends.prx[0], S.ends.prx[1], S.ends.prx[2]), S.ends.sn, S.ends.cs,
                 S.ends.fl0 | S.ends.fl1);
    }
  }
  if (ovf) {
    atomicAdd(&a.ctr->stack_overflow, 1u);
    atomicOr(&a.ctr->err, ERR_STACK);
  }
}

// ---------------------------------------------------------------------------
// first-order edge diffraction (Sec. III step 5) with the UTD
// ---------------------------------------------------------------------------
// -1/n and 1/(2n + 1) for the erf series below (a division costs about ten
// dependent FP64 operations, the rest of a term six).
struct ErfTab {
  double a[200], b[200];
  constexpr ErfTab() : a(), b() {
    for (int n = 1; n < 200; ++n) {
      a[n] = -1.0 / n;
      b[n] = 1.0 / (2 * n + 1);
    }
  }
};
__constant__ ErfTab kErfTab = ErfTab();

// erfc(z) for Re z > 0: the Maclaurin series of erf (Abramowitz & Stegun
// 7.1.5) for |z| < 3, else the continued fraction of A&S 7.1.14, truncated
// after 40, 30 or 20 terms for |z| from 3, 3.5 or 4.5 on (relative error
// below 3e-15 against a Faddeeva-function reference). Only |z| < 5.5 comes
// here: transition_fn takes its large-argument series from x = 30 on.
__device__ zd erfc_z(zd z) {
  const double rsqpi = 0.56418958354775628695;  // 1/sqrt(pi)
  double az = hypot(z.re, z.im);
  if (az < 3.0) {
    zd z2 = z * z, term = z, sum = z;
    for (int n = 1; n < 200; ++n) {
      term = term * z2 * kErfTab.a[n];
      zd t = term * kErfTab.b[n];
      sum = sum + t;
      if (fabs(t.re) + fabs(t.im) < 1e-17 * (fabs(sum.re) + fabs(sum.im))) break;
    }
    return Z(1.0) - sum * (2.0 * rsqpi);
  }
  // erfc z = e^{-z^2}/sqrt(pi) * 1/(z + (1/2)/(z + 1/(z + (3/2)/(z + ...)))),
  // the truncated fraction evaluated forward as A_n / B_n (A_k = z A_{k-1} +
  // (k/2) A_{k-2}, B likewise) with one division at the end; for |z| < 5.5
  // and 40 terms |A|, |B| stay below 1e40
  zd A0 = Z(1.0), A1 = z, B0 = Z(0.0), B1 = Z(1.0);
  const int nt = az < 3.5 ? 40 : az < 4.5 ? 30 : 20;
  for (int k = 1; k <= nt; ++k) {
    const double h = 0.5 * k;
    const zd za = z * A1, zb = z * B1;
    zd A2 = Z(fma(A0.re, h, za.re), fma(A0.im, h, za.im)), B2 = Z(fma(B0.re, h, zb.re), fma(B0.im, h, zb.im));
    A0 = A1;
    A1 = A2;
    B0 = B1;
    B1 = B2;
  }
  zd ez = zexp(Z(-(z.re * z.re - z.im * z.im), -2.0 * z.re * z.im));
  return zdiv(ez * rsqpi * B1, A1);
}

// UTD transition function F(x) = 2j sqrt(x) e^{jx} int_{sqrt x}^inf e^{-j t^2} dt,
// the tail integral being (sqrt(pi)/2) e^{-j pi/4} erfc(e^{j pi/4} sqrt x).
// For x >= 30 its large-argument expansion (repeated integration by parts of
// the tail integral, as Kouyoumjian & Pathak give it): F(x) = sum_m t_m with
// t_0 = 1, t_m = t_{m-1} j (2m - 1) / (2x), i.e. 1 + j/(2x) - 3/(4x^2) - ...;
// its terms shrink while 2m - 1 < 2x, and the sum stops there or at 1e-17;
// the error is below 1e-13 for x >= 30. Away from shadow and reflection
// boundaries x = 2kL cos^2(.) is in the thousands, so this is the usual case.
__device__ zd transition_fn(double x) {
  if (!(x > 0.0)) return Z(0.0);
  if (x >= 30.0) {
    const double r = 1.0 / (2.0 * x);
    zd t = Z(1.0), sum = Z(1.0);
    for (int m = 1; m <= 40; ++m) {
      double c = (2.0 * m - 1.0) * r;
      if (c >= 1.0) break;  // the terms grow from here on
      t = Z(-t.im * c, t.re * c);  // times j (2m - 1) / (2x)
      sum = sum + t;
      if (fabs(t.re) + fabs(t.im) < 1e-17 * (fabs(sum.re) + fabs(sum.im))) break;
    }
    return sum;
  }
  double a = sqrt(x);
  const double h = 0.70710678118654752440;
  zd G = Z(h, -h) * erfc_z(Z(h * a, h * a)) * 0.88622692545275801365;  // sqrt(pi)/2
  double sn, cs;
  sincos(x, &sn, &cs);
  return Z(0.0, 2.0 * a) * Z(cs, sn) * G;
}

__device__ zd utd_term(double n, double beta, double s, double kL, unsigned& fl) {
  double N = rint((beta + s * M_PI) / (2.0 * M_PI * n));
  double c = cos((2.0 * n * M_PI * N - beta) / 2.0);
  double arg = (M_PI + s * beta) / (2.0 * n);
  double sn = sin(arg);
  if (fabs(sn) < 1e-9) return Z(0.0);
  return transition_fn(kL * 2.0 * c * c) * (cos(arg) / sn);
}

// Kouyoumjian-Pathak wedge coefficient D = pre (t1 + t2 + r0 t3 + rn t4)
// with face reflection factors r0, rn. The prefactor and the four terms do
// not depend on r0 and rn, so the soft and hard coefficients share them
// (utd_parts once, utd_coeff per polarisation).
// The exact stage takes a survivor with a group of kDiffLanes lanes (or, with
// many survivors, one) that run the same code on the same values and split
// what is independent: the four terms here, the two faces' Fresnel factors,
// the legs' occlusion. The values are the same either way.
constexpr int kDiffLanes = 4;
__shared__ int diff_lanes;  // lanes per survivor, set by k_diffract
__device__ __forceinline__ int diff_lane() { return threadIdx.x & (diff_lanes - 1); }
__device__ __forceinline__ unsigned diff_mask() {
  return ((1u << diff_lanes) - 1u) << ((threadIdx.x & 31) & ~(diff_lanes - 1));
}
__device__ __forceinline__ zd diff_from(zd v, int lane) {  // the value of a lane of the group
  const unsigned m = diff_mask();
  return Z(__shfl_sync(m, v.re, lane, diff_lanes), __shfl_sync(m, v.im, lane, diff_lanes));
}
struct UtdParts {
  zd pre, t[4];
};
__device__ UtdParts utd_parts(double n, double phi, double phip, double beta0, double L, double k, unsigned& fl) {
  const double h = 0.70710678118654752440;
  UtdParts u;
  u.pre = Z(-h, h) * (1.0 / (2.0 * n * sqrt(2.0 * M_PI * k) * sin(beta0)));  // -e^{-j pi/4} / (...)
  // terms: (phi - phi', +), (phi - phi', -), (phi + phi', -), (phi + phi', +)
#pragma unroll 1
  for (int j0 = 0; j0 < 4; j0 += diff_lanes) {
    const int q = j0 + diff_lane();
    const zd t = utd_term(n, q < 2 ? phi - phip : phi + phip, q == 0 || q == 3 ? 1.0 : -1.0, k * L, fl);
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (j >= j0 && j < j0 + diff_lanes) u.t[j] = diff_from(t, j - j0);
  }
  return u;
}
__device__ zd utd_coeff(const UtdParts& u, zd r0, zd rn) {
  return u.pre * (u.t[0] + u.t[1] + r0 * u.t[2] + rn * u.t[3]);
}

// Fresnel TE / TM coefficients in FP64 (eps_c = eps_r - j sigma/(w eps0)).
__device__ void fresnel_d(float4 mt, double freq, double ct, zd& te, zd& tm) {
  if (mt.z != 0.0f) {
    te = Z(-1.0);
    tm = Z(1.0);
    return;
  }
  zd ec = Z((double)mt.x, -(double)mt.y / (2.0 * M_PI * freq * 8.8541878128e-12));
  zd root = zsqrt(ec - Z(1.0 - ct * ct));
  te = zdiv(Z(ct) - root, Z(ct) + root);
  tm = zdiv(ec * ct - root, ec * ct + root);
}

// ... of a wedge's two faces at once (te, tm of face 0, then of face n).
__device__ __forceinline__ void fresnel_faces(float4 ma, double cta, float4 mb, double ctb, double freq, zd& r0s,
                                              zd& r0h, zd& rns, zd& rnh) {
#pragma unroll 1
  for (int j = 0; j < 2; j += diff_lanes) {
    const bool second = (j + diff_lane()) & 1;
    zd te, tm;
    fresnel_d(second ? mb : ma, freq, second ? ctb : cta, te, tm);
    if (j == 0) {
      r0s = diff_from(te, 0);
      r0h = diff_from(tm, 0);
    }
    if (j == 1 || diff_lanes > 1) {
      rns = diff_from(te, 1 - j);
      rnh = diff_from(tm, 1 - j);
    }
  }
}

struct d3w {
  double x, y, z;
};
__device__ __forceinline__ d3w D3(double x, double y, double z) { return d3w{x, y, z}; }
__device__ __forceinline__ d3w operator-(d3w a, d3w b) { return D3(a.x - b.x, a.y - b.y, a.z - b.z); }
__device__ __forceinline__ d3w operator+(d3w a, d3w b) { return D3(a.x + b.x, a.y + b.y, a.z + b.z); }
__device__ __forceinline__ d3w operator*(d3w a, double s) { return D3(a.x * s, a.y * s, a.z * s); }
__device__ __forceinline__ double dotw(d3w a, d3w b) { return fma(a.z, b.z, fma(a.y, b.y, a.x * b.x)); }
__device__ __forceinline__ d3w crossw(d3w a, d3w b) {
  return D3(a.y * b.z - a.z * b.y, a.z * b.x - a.x * b.z, a.x * b.y - a.y * b.x);
}
__device__ __forceinline__ d3w unitw(d3w a) { return a * rsqrt(dotw(a, a)); }
__device__ __forceinline__ d3w polw(d3w u, d3w d, unsigned& fl) {
  d3w p = u - d * dotw(u, d);
  double n = sqrt(dotw(p, p));
  if (n < 1e-9) {
    fl |= DCEM_PATH_POL_DEGENERATE;
    d3w a = fabs(d.x) < 0.9 ? D3(1, 0, 0) : D3(0, 1, 0);
    p = a - d * dotw(a, d);
    n = sqrt(dotw(p, p));
  }
  return p * (1.0 / n);
}

// Angle of X about the wedge, from face 0 through the exterior.
__device__ __forceinline__ double wedge_angle(const Wedge& W, d3w X) {
  d3w e = D3(W.e[0], W.e[1], W.e[2]);
  d3w d = X - D3(W.p0[0], W.p0[1], W.p0[2]);
  d = d - e * dotw(d, e);
  double a = atan2(dotw(d, D3(W.y0[0], W.y0[1], W.y0[2])), dotw(d, D3(W.t0[0], W.t0[1], W.t0[2])));
  return a < 0.0 ? a + 2.0 * M_PI : a;
}

// FP32 pre-test of a (transmitter, receiver, wedge) triple: false only when
// the FP64 test below rejects the triple too, so that most triples (far from
// the Keller cone of a short vehicle edge, or on the lit side) cost no FP64
// work. Rejections keep margins above the FP32 rounding of the geometry: the
// Keller point off the edge by more than 5 cm (plus 1e-5 of the distances),
// an angle beyond the wedge or the shadow-boundary rule missed by more than
// ten times the angle's rounding bound (at least 1e-3 rad). Angles near the
// 0 / 2 pi cut, or of points near the edge line, reject nothing.
__device__ __forceinline__ float wedge_angle32(float3 d, float3 t0, float3 y0, float r, float dist, bool& sure,
                                               float& tol) {
  float a = atan2f(fdot3(d, y0), fdot3(d, t0));
  if (a < 0.0f) a += 6.2831853f;
  float err = 4e-6f * (dist + 1.0f) / r + 1e-5f;  // rounding of the in-plane direction, radians
  tol = fmaxf(1e-3f, 10.0f * err);
  sure = r > 0.0f && err < 1e-3f && a > tol && a < 6.2831853f - tol;
  return a;
}

__device__ __forceinline__ bool diffract_candidate(const WedgeF& W, float4 txv, float4 rxv) {
  const float3 e = W.e, p0 = W.p0;
  float3 dt = f3(txv.x - p0.x, txv.y - p0.y, txv.z - p0.z), dr = f3(rxv.x - p0.x, rxv.y - p0.y, rxv.z - p0.z);
  float zt = fdot3(dt, e), zr = fdot3(dr, e);
  float3 pt = f3(dt.x - e.x * zt, dt.y - e.y * zt, dt.z - e.z * zt);
  float3 pr = f3(dr.x - e.x * zr, dr.y - e.y * zr, dr.z - e.z * zr);
  float rt = sqrtf(fdot3(pt, pt)), rr = sqrtf(fdot3(pr, pr));
  float lt = sqrtf(fdot3(dt, dt)), lr = sqrtf(fdot3(dr, dr));
  if (!(rt > 1e-3f && rr > 1e-3f)) return true;
  float zq = zt + (zr - zt) * rt / (rt + rr);
  float mz = 0.05f + 1e-5f * (lt + lr);
  if (zq < -mz || zq > W.len + mz) return false;
  bool st, sr;
  float tt, tr;
  float phip = wedge_angle32(pt, W.t0, W.y0, rt, lt, st, tt), phi = wedge_angle32(pr, W.t0, W.y0, rr, lr, sr, tr);
  const float npi = W.npi;
  if ((st && phip > npi + tt) || (sr && phi > npi + tr)) return false;
  if (st && sr && fabsf(phi - phip) < 3.14159265f - (tt + tr)) return false;
  return true;
}

// Triangle slot geometry: vertices and the (unnormalised) normal.
__device__ __forceinline__ void tri64(const PathArgs& a, int id, d3w& v0, d3w& v1, d3w& v2, float4& mat) {
  const float4* tp = a.tris + 3 * (size_t)DCEM_IDX(a.slot_of_id[DCEM_IDX(id, a.bvh.ntris)], a.bvh.ntris);
  float4 p0 = tp[0], p1 = tp[1], p2 = tp[2];
  v0 = D3(p0.x, p0.y, p0.z);
  v1 = D3(p1.x, p1.y, p1.z);
  v2 = D3(p2.x, p2.y, p2.z);
  mat = a.mats[__float_as_int(p1.w)];
}

// The triangles (other than ex0 .. ex3) that the open segment p -> q crosses
// with parameter in (eps_occ, 1 - eps_occ) (FP32 traversal of the scene, as
// any_hit), in order along it: their ids in ids[0 .. n-1]. Returns n, or -1
// when one of them is opaque (a material without penetration loss, loss <
// 0) or there are more than cap (the transmissions a path has left).
__device__ __noinline__ int leg_crossings(const PathArgs& a, d3w p, d3w q, int ex0, int ex1, int ex2, int ex3,
                                          int* ids, int cap, unsigned& ovf, TStack& st) {
  const Bvh& bvh = a.bvh;
  const d3w dv = q - p;
  const RayPre r = ray_pre(f3((float)p.x, (float)p.y, (float)p.z), f3((float)dv.x, (float)dv.y, (float)dv.z));
  const float t0 = a.eps_occ, t1 = 1.0f - a.eps_occ;
  float ts[kMaxRefl];
  int n = 0;
  st.reset();
  if (bvh.root1 != kEmpty) st.push(bvh.root1);
  int cur = bvh.root0;
  for (int visits = 0;; ++visits) {
    if (visits > bvh.max_visits) {
      ovf = 1u;
      break;
    }
    if (cur == kEmpty) {
      if (st.empty()) break;
      cur = st.pop();
      continue;
    }
    if (cur >= 0) {
      const float4* nd = bvh.nodes + 4 * (size_t)DCEM_IDX(cur, bvh.nnodes);
      float4 n0 = __ldg(nd), n1 = __ldg(nd + 1), n2 = __ldg(nd + 2), n3 = __ldg(nd + 3);
      float tn0, tn1;
      bool h0 = slab(r, n0.x, n0.y, n0.z, n0.w, n2.x, n2.y, t1, tn0);
      bool h1 = slab(r, n1.x, n1.y, n1.z, n1.w, n2.z, n2.w, t1, tn1);
      int c0 = __float_as_int(n3.x), c1 = __float_as_int(n3.y);
      if (h0 && h1) {
        if (!st.push(c1)) ovf = 1u;
        cur = c0;
      } else if (h0) {
        cur = c0;
      } else if (h1) {
        cur = c1;
      } else {
        cur = kEmpty;
      }
    } else {
      const int slot = DCEM_IDX(~cur, bvh.ntris);
      float3 v0, v1, v2;
      int id;
      load_tri(bvh.tris, slot, v0, v1, v2, id);
      float t;
      cur = kEmpty;
      if (id == ex0 || id == ex1 || id == ex2 || id == ex3 || !tri_hit(r, v0, v1, v2, t) || !(t > t0 && t < t1))
        continue;
      const float loss = a.mats[__float_as_int(__ldg(&bvh.tris[3 * slot + 1]).w)].w;
      if (!(loss >= 0.0f) || n >= cap || n >= kMaxRefl) return -1;
      int k = n++;  // insertion in order along the segment
      while (k > 0 && ts[k - 1] > t) {
        ts[k] = ts[k - 1];
        ids[k] = ids[k - 1];
        --k;
      }
      ts[k] = t;
      ids[k] = id;
    }
  }
  return n;
}

// FP32 any-hit of the legs between the n points P of a path, two triangles
// excluded at each point; the legs are shared out over the group's lanes.
__device__ __noinline__ bool legs_occluded(const PathArgs& a, const d3w* P, const int (*ex)[2], int n, unsigned& ovf,
                                           TStack& st) {
  bool hit = false;
  for (int q = diff_lane(); q + 1 < n && !hit; q += diff_lanes) {
    const d3w dv = P[q + 1] - P[q];
    const RayPre rp = ray_pre(f3((float)P[q].x, (float)P[q].y, (float)P[q].z),
                              f3((float)dv.x, (float)dv.y, (float)dv.z));
    hit = any_hit(a.bvh, rp, a.eps_occ, 1.0f - a.eps_occ, ex[q][0], ex[q][1], ovf, st, ex[q + 1][0], ex[q + 1][1]);
  }
  return __any_sync(diff_mask(), hit);
}

// Wedge geometry from the current world triangles (moving objects' wedges
// follow their objects): the edge from its lexicographically lower vertex,
// the faces' directions normal to it, and n = exterior angle / pi.
__device__ __forceinline__ bool vless(float4 a, float4 b) {
  if (a.x != b.x) return a.x < b.x;
  if (a.y != b.y) return a.y < b.y;
  return a.z < b.z;
}

__global__ void k_wedge_geom(const float4* __restrict__ tris, const int* __restrict__ slot_of_id,
                             const WedgeTopo* __restrict__ topo, int nw, Wedge* out, WedgeF* outf) {
  for (int w = blockIdx.x * blockDim.x + threadIdx.x; w < nw; w += gridDim.x * blockDim.x) {
    WedgeTopo t = topo[w];
    const float4* A = tris + 3 * (size_t)slot_of_id[t.ta];
    const float4* B = tris + 3 * (size_t)slot_of_id[t.tb];
    float4 va = A[t.ka0], vb = A[t.ka1], vt = A[t.kat], vu = B[t.kbt];
    if (vless(vb, va)) {
      float4 x = va;
      va = vb;
      vb = x;
    }
    Wedge W;
    d3w p0 = D3(va.x, va.y, va.z), e = D3((double)vb.x - va.x, (double)vb.y - va.y, (double)vb.z - va.z);
    double len = sqrt(dotw(e, e));
    e = e * (1.0 / len);
    d3w da = D3((double)vt.x - va.x, (double)vt.y - va.y, (double)vt.z - va.z);
    d3w db = D3((double)vu.x - va.x, (double)vu.y - va.y, (double)vu.z - va.z);
    da = da - e * dotw(da, e);
    db = db - e * dotw(db, e);
    d3w t0 = da * (1.0 / sqrt(dotw(da, da))), tB = db * (1.0 / sqrt(dotw(db, db)));
    d3w y0 = crossw(e, t0);
    double alpha = atan2(dotw(tB, y0), dotw(tB, t0));
    if (alpha < 0.0) {
      y0 = y0 * -1.0;
      alpha = -alpha;
    }
    y0 = y0 * -1.0;  // the exterior runs away from face n
    W.p0[0] = p0.x; W.p0[1] = p0.y; W.p0[2] = p0.z;
    W.p1[0] = vb.x; W.p1[1] = vb.y; W.p1[2] = vb.z;
    W.e[0] = e.x; W.e[1] = e.y; W.e[2] = e.z;
    W.t0[0] = t0.x; W.t0[1] = t0.y; W.t0[2] = t0.z;
    W.tB[0] = tB.x; W.tB[1] = tB.y; W.tB[2] = tB.z;
    W.y0[0] = y0.x; W.y0[1] = y0.y; W.y0[2] = y0.z;
    W.len = len;
    W.n = 2.0 - alpha / M_PI;
    W.ta = t.ta;
    W.tb = t.tb;
    out[w] = W;
    WedgeF f;
    f.p0 = make_float3((float)W.p0[0], (float)W.p0[1], (float)W.p0[2]);
    f.e = make_float3((float)W.e[0], (float)W.e[1], (float)W.e[2]);
    f.t0 = make_float3((float)W.t0[0], (float)W.t0[1], (float)W.t0[2]);
    f.y0 = make_float3((float)W.y0[0], (float)W.y0[1], (float)W.y0[2]);
    f.len = (float)W.len;
    f.npi = (float)(W.n * M_PI);
    outf[w] = f;
  }
}

// Each wedge group's box (kWedgeGroup wedges in the order perm, one lane
// each): the min and max over its edges' two ends in FP32.
__global__ void k_wedge_boxes(const WedgeF* __restrict__ wf, const int* __restrict__ perm, int nw,
                              float* __restrict__ box) {
  const int lane = threadIdx.x & (kWedgeGroup - 1), ng = (nw + kWedgeGroup - 1) / kWedgeGroup;
  // whole warps walk the groups (kWedgeGroup divides 32), so the shuffles below are complete
  const int nwarp = (gridDim.x * blockDim.x) >> 5, per = 32 / kWedgeGroup;
  for (int w0 = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; w0 * per < ng; w0 += nwarp) {
    const int g = w0 * per + (threadIdx.x & 31) / kWedgeGroup, i = g * kWedgeGroup + lane;
    float lo[3] = {3e38f, 3e38f, 3e38f}, hi[3] = {-3e38f, -3e38f, -3e38f};
    if (i < nw) {
      const WedgeF f = wf[perm[i]];
      const float q[3] = {f.p0.x + f.e.x * f.len, f.p0.y + f.e.y * f.len, f.p0.z + f.e.z * f.len};
      const float p[3] = {f.p0.x, f.p0.y, f.p0.z};
      for (int k = 0; k < 3; ++k) {
        lo[k] = fminf(p[k], q[k]);
        hi[k] = fmaxf(p[k], q[k]);
      }
    }
    for (int o = kWedgeGroup / 2; o > 0; o >>= 1)
      for (int k = 0; k < 3; ++k) {
        lo[k] = fminf(lo[k], __shfl_xor_sync(0xffffffffu, lo[k], o));
        hi[k] = fmaxf(hi[k], __shfl_xor_sync(0xffffffffu, hi[k], o));
      }
    if (g < ng && lane < 6) box[6 * (size_t)g + lane] = lane < 3 ? lo[lane] : hi[lane - 3];
  }
}

// One thread per (link, wedge): the Keller point on the edge (unfolding the
// path about the edge line), the paper's shadow rule (the receiver beyond the
// incident shadow boundary), both legs unoccluded, then the UTD field; a
// valid path joins its link's bucket like a validated path.
// One (link, wedge) pair that passed the FP32 pre-test: the exact FP64
// test, the legs' occlusion, the UTD field and the path record.
__device__ __forceinline__ void diffract_pair(const PathArgs& a, long idx, double k, double lam, unsigned& ovf,
                                              TStack& st) {
  int link = (int)(idx / a.nw), w = (int)(idx - (long)link * a.nw);
  const Wedge W = a.wedges[w];
  float4 rxv = a.rx[link % a.nrx], txv = a.txs[link / a.nrx];
  d3w T = D3(txv.x, txv.y, txv.z), R = D3(rxv.x, rxv.y, rxv.z);
  d3w e = D3(W.e[0], W.e[1], W.e[2]), p0 = D3(W.p0[0], W.p0[1], W.p0[2]);
  d3w dt = T - p0, dr = R - p0;
  double zt = dotw(dt, e), zr = dotw(dr, e);
  d3w pt = dt - e * zt, pr = dr - e * zr;
  double rt = sqrt(dotw(pt, pt)), rr = sqrt(dotw(pr, pr));
  if (!(rt > 0.0 && rr > 0.0)) return;
  double zq = zt + (zr - zt) * rt / (rt + rr);
  double uq = zq / W.len;
  if (!(uq > 0.0 && uq < 1.0)) return;
  d3w Q = p0 + e * zq;
  double phip = wedge_angle(W, T), phi = wedge_angle(W, R), n = W.n;
  if (phip > n * M_PI || phi > n * M_PI) return;
  if (!(fabs(phi - phip) > M_PI)) return;
  // the legs: unoccluded, or with transmission on, crossing penetrable
  // triangles only, at most max_trans in all (Table II losses)
  int c1[kMaxRefl], c2[kMaxRefl], n1 = 0, n2 = 0;
  if (a.max_trans > 0) {
    const int mt = min(a.max_trans, kMaxRefl - 1);  // the wedge takes one of the record's slots
    n1 = leg_crossings(a, T, Q, W.ta, W.tb, W.tb, W.tb, c1, mt, ovf, st);
    if (n1 < 0) return;
    n2 = leg_crossings(a, Q, R, W.ta, W.tb, W.tb, W.tb, c2, mt - n1, ovf, st);
    if (n2 < 0) return;
  } else {
    const d3w P[3] = {T, Q, R};
    const int ex[3][2] = {{-1, -1}, {W.ta, W.tb}, {-1, -1}};
    if (legs_occluded(a, P, ex, 3, ovf, st)) return;
  }
  unsigned fl = 0;
  d3w qt = Q - T, rq = R - Q;
  double sp = sqrt(dotw(qt, qt)), s = sqrt(dotw(rq, rq));
  d3w ip = qt * (1.0 / sp), dd = rq * (1.0 / s);
  double beta0 = acos(fmax(-1.0, fmin(1.0, dotw(ip, e))));
  double sb = sin(beta0);
  double L = s * sp * sb * sb / (s + sp);
  d3w php = unitw(crossw(e, ip)) * -1.0, ph = unitw(crossw(e, dd));
  d3w bp = crossw(ip, php), bd = crossw(dd, ph);
  // Luebbers: the faces' Fresnel factors at the grazing angles phi' and n pi - phi
  const float4 ma =
      a.mats[__float_as_int(a.tris[3 * (size_t)DCEM_IDX(a.slot_of_id[DCEM_IDX(W.ta, a.bvh.ntris)], a.bvh.ntris) + 1].w)];
  const float4 mb =
      a.mats[__float_as_int(a.tris[3 * (size_t)DCEM_IDX(a.slot_of_id[DCEM_IDX(W.tb, a.bvh.ntris)], a.bvh.ntris) + 1].w)];
  zd r0s, r0h, rns, rnh;
  fresnel_faces(ma, fabs(sin(phip)), mb, fabs(sin(n * M_PI - phi)), a.freq, r0s, r0h, rns, rnh);
  const UtdParts up = utd_parts(n, phi, phip, beta0, L, k, fl);
  zd Ds = utd_coeff(up, r0s, rns);
  zd Dh = utd_coeff(up, r0h, rnh);
  d3w u = D3(a.pol.x, a.pol.y, a.pol.z);
  d3w e0 = polw(u, ip, fl), prx = polw(u, dd * -1.0, fl);
  double sn, cs;
  sincos(-k * sp, &sn, &cs);
  zd Ei = Z(cs / sp, sn / sp);
  zd Eb = Ei * dotw(e0, bp), Ep = Ei * dotw(e0, php);
  sincos(-k * s, &sn, &cs);
  zd A = Z(cs, sn) * sqrt(sp / (s * (s + sp)));
  zd proj = (Ds * Eb) * (-dotw(bd, prx)) + (Dh * Ep) * (-dotw(ph, prx));
  // each crossing's penetration loss (power dB): the field times 10^(-L/20)
  double g = 1.0;
  for (int i = 0; i < n1 + n2; ++i) {
    d3w v0, v1, v2;
    float4 mt;
    tri64(a, i < n1 ? c1[i] : c2[i - n1], v0, v1, v2, mt);
    g *= pow(10.0, -(double)mt.w / 20.0);
  }
  zd amp = proj * A * (lam / (4.0 * M_PI) * g);
  if (diff_lane() != 0) return;  // one lane of the group writes the record
  unsigned uu = atomicAdd(&a.ctr->n_unique, 1u);
  if (uu >= a.ucap) {
    atomicOr(&a.ctr->err, ERR_UNIQUE_OVERFLOW);
    return;
  }
  PathRec rec;
  // interactions in path order: the first leg's crossings, the wedge, the second leg's
  const int depth = n1 + 1 + n2;
  auto id_at = [&](int q) {
    return q < n1 ? (c1[q] | kTransBit) : q == n1 ? (w | kDiffBit) : (c2[q - n1 - 1] | kTransBit);
  };
  rec.key = seq_key(link % a.nrx, depth, id_at);
  rec.rx = link;
  rec.depth = depth;
  rec.ray = -1;
  rec.flags = fl;
  rec.valid = 1;
  rec.pad = 0;
  rec.len = sp + s;
  rec.amp_re = amp.re;
  rec.amp_im = amp.im;
  for (int j = 0; j < kMaxRefl; ++j) {
    rec.tri[j] = j < depth ? id_at(j) : -1;
    rec.pts[j][0] = rec.pts[j][1] = rec.pts[j][2] = 0.0f;
  }
  for (int j = 0; j < depth; ++j) {  // the crossings where the legs meet their triangles' planes, and Q
    d3w X = Q;
    if (j != n1) {
      const bool first = j < n1;
      const d3w o = first ? T : Q, dl = first ? qt : rq;
      d3w v0, v1, v2;
      float4 mt;
      tri64(a, first ? c1[j] : c2[j - n1 - 1], v0, v1, v2, mt);
      const d3w nv = crossw(v1 - v0, v2 - v0);
      X = o + dl * (dotw(v0 - o, nv) / dotw(dl, nv));
    }
    rec.pts[j][0] = (float)X.x;
    rec.pts[j][1] = (float)X.y;
    rec.pts[j][2] = (float)X.z;
  }
  a.prec[uu] = rec;
  unsigned pos = atomicAdd(&a.bucket_cnt[link], 1u);
  if (pos < (unsigned)a.bucket_cap) a.bucket[(size_t)link * a.bucket_cap + pos] = (int)uu;
  else atomicOr(&a.ctr->err, ERR_BUCKET_OVERFLOW);
  atomicAdd(&a.ctr->n_valid, 1u);
}

// ---------------------------------------------------------------------------
// one reflection before or after a diffraction (Sec. III steps 3-5)
// ---------------------------------------------------------------------------
// By image theory a reflection on plane (n, c) before the wedge is the
// diffraction of the transmitter's image, a reflection after it the
// diffraction toward the receiver's image; the reflection point is where the
// unfolded leg (image -> Q, or Q -> image) crosses the plane. Candidates are
// (link, wedge, reflector plane, order); survivors of the FP32 pre-test carry
// bit 63 in the survivor list: ((link * nw + wedge) * nrp + plane) * 2 + first.
constexpr unsigned long long kReflTag = 1ull << 63;

__device__ __forceinline__ float3 mirror32(float3 x, float3 n, float c) {
  float h = 2.0f * (fdot3(n, x) - c);
  return f3(x.x - h * n.x, x.y - h * n.y, x.z - h * n.z);
}

// FP32 pre-test: false only when the FP64 test rejects the candidate too
// (Keller point and angles as diffract_candidate with the image; the
// reflection point off the plane's box by more than 5 cm + 1e-4 of the
// distances, or off the unfolded leg).
__device__ __forceinline__ bool diffract_refl_candidate(const WedgeF& W, const RPlane& P, float4 txv, float4 rxv,
                                                        bool first) {
  const float3 n = f3(P.nf[0], P.nf[1], P.nf[2]);
  const float c = P.cf;
  float3 T = f3(txv.x, txv.y, txv.z), R = f3(rxv.x, rxv.y, rxv.z);
  float3 S = first ? mirror32(T, n, c) : T, O = first ? R : mirror32(R, n, c);
  if (!diffract_candidate(W, make_float4(S.x, S.y, S.z, 0.0f), make_float4(O.x, O.y, O.z, 0.0f))) return false;
  const float3 e = W.e, p0 = W.p0;
  float3 dt = f3(S.x - p0.x, S.y - p0.y, S.z - p0.z), dr = f3(O.x - p0.x, O.y - p0.y, O.z - p0.z);
  float zt = fdot3(dt, e), zr = fdot3(dr, e);
  float3 pt = f3(dt.x - e.x * zt, dt.y - e.y * zt, dt.z - e.z * zt);
  float3 pr = f3(dr.x - e.x * zr, dr.y - e.y * zr, dr.z - e.z * zr);
  float rt = sqrtf(fdot3(pt, pt)), rr = sqrtf(fdot3(pr, pr));
  if (!(rt > 1e-3f && rr > 1e-3f)) return true;
  float zq = zt + (zr - zt) * rt / (rt + rr);
  float3 Q = f3(p0.x + e.x * zq, p0.y + e.y * zq, p0.z + e.z * zq);
  float3 a0 = first ? S : Q, a1 = first ? Q : O;
  float3 dv = f3(a1.x - a0.x, a1.y - a0.y, a1.z - a0.z);
  float den = fdot3(n, dv), len = sqrtf(fdot3(dv, dv));
  if (!(fabsf(den) > 1e-6f * len)) return true;
  float t = (c - fdot3(n, a0)) / den;
  float mt = (0.05f + 1e-4f * (len + sqrtf(fdot3(a0, a0)))) / len;
  if (t < -mt || t > 1.0f + mt) return false;
  float3 X = f3(a0.x + t * dv.x, a0.y + t * dv.y, a0.z + t * dv.z);
  float mb = 0.05f + 1e-4f * (len + sqrtf(fdot3(X, X)));
  if (X.x < P.box[0] - mb || X.y < P.box[1] - mb || X.z < P.box[2] - mb || X.x > P.box[3] + mb ||
      X.y > P.box[4] + mb || X.z > P.box[5] + mb)
    return false;
  return true;
}

// Image, Keller point and reflection point for plane (n, c): false when the
// Keller point leaves the edge, an angle falls inside the wedge, the shadow
// rule fails or the reflection point leaves the unfolded leg.
struct ReflGeom {
  d3w S, O, Q, P;  // source (or image), observer (or image), diffraction and reflection points
  double phip, phi;
};
__device__ __forceinline__ bool refl_geometry(const Wedge& W, d3w n, double c, d3w T, d3w R, bool first,
                                              ReflGeom& g) {
  g.S = first ? T - n * (2.0 * (dotw(n, T) - c)) : T;
  g.O = first ? R : R - n * (2.0 * (dotw(n, R) - c));
  d3w e = D3(W.e[0], W.e[1], W.e[2]), p0 = D3(W.p0[0], W.p0[1], W.p0[2]);
  d3w dt = g.S - p0, dr = g.O - p0;
  double zt = dotw(dt, e), zr = dotw(dr, e);
  d3w pt = dt - e * zt, pr = dr - e * zr;
  double rt = sqrt(dotw(pt, pt)), rr = sqrt(dotw(pr, pr));
  if (!(rt > 0.0 && rr > 0.0)) return false;
  double zq = zt + (zr - zt) * rt / (rt + rr);
  double uq = zq / W.len;
  if (!(uq > 0.0 && uq < 1.0)) return false;
  g.Q = p0 + e * zq;
  g.phip = wedge_angle(W, g.S);
  g.phi = wedge_angle(W, g.O);
  if (g.phip > W.n * M_PI || g.phi > W.n * M_PI) return false;
  if (!(fabs(g.phi - g.phip) > M_PI)) return false;
  d3w a0 = first ? g.S : g.Q, a1 = first ? g.Q : g.O;
  double den = dotw(n, a1 - a0);
  if (den == 0.0) return false;
  double t = (c - dotw(n, a0)) / den;
  if (!(t > 0.0 && t < 1.0)) return false;
  g.P = a0 + (a1 - a0) * t;
  return true;
}


// Can triangle id hold point x (on its plane group's plane, within 1e-4 m of
// the triangle's own)? x must lie in the triangle's FP32 box widened by 1 mm +
// 1e-6 of the coordinates; the FP64 test (inside_tri64) follows for those
// that do.
__device__ __forceinline__ bool tri_box_near(const PathArgs& a, int id, d3w x) {
  const float4* tp = a.tris + 3 * (size_t)DCEM_IDX(a.slot_of_id[DCEM_IDX(id, a.bvh.ntris)], a.bvh.ntris);
  const float4 p0 = tp[0], p1 = tp[1], p2 = tp[2];
  const float X = (float)x.x, Y = (float)x.y, Zc = (float)x.z;
  const float m = 1e-3f + 1e-6f * (fabsf(X) + fabsf(Y) + fabsf(Zc));
  return !(X < fminf(p0.x, fminf(p1.x, p2.x)) - m || X > fmaxf(p0.x, fmaxf(p1.x, p2.x)) + m ||
           Y < fminf(p0.y, fminf(p1.y, p2.y)) - m || Y > fmaxf(p0.y, fmaxf(p1.y, p2.y)) + m ||
           Zc < fminf(p0.z, fminf(p1.z, p2.z)) - m || Zc > fmaxf(p0.z, fmaxf(p1.z, p2.z)) + m);
}

__device__ __forceinline__ bool inside_tri64(d3w v0, d3w v1, d3w v2, d3w x) {
  d3w n = crossw(v1 - v0, v2 - v0);
  return !(dotw(crossw(v1 - v0, x - v0), n) < 0.0 || dotw(crossw(v2 - v1, x - v1), n) < 0.0 ||
           dotw(crossw(v0 - v2, x - v2), n) < 0.0);
}

// The member triangle of plane G holding point x (on G's plane), none of the
// nex ids in ex: the lowest id among the members whose box holds x
// (tri_box_near) and that contain it (inside_tri64) -- the one a scan of the
// members in id order finds first -- with its vertices and material; -1 when
// there is none. The members are sorted by their lowest coordinate along G's
// axis, so only those with that coordinate in [u - 2 m - ext, u + 2 m] can
// pass the box test (u: x's coordinate, m: the test's margin, ext: the
// members' largest extent along the axis): a binary search, then a scan of
// that range.
__device__ int member_at(const PathArgs& a, const RPlane& G, d3w x, const int* ex, int nex, d3w& v0, d3w& v1,
                         d3w& v2, float4& mat) {
  const float X = (float)x.x, Y = (float)x.y, Z = (float)x.z;
  const float m = 1e-3f + 1e-6f * (fabsf(X) + fabsf(Y) + fabsf(Z));
  const float u = G.axis == 0 ? X : (G.axis == 1 ? Y : Z);
  const float hi = u + 2.0f * m, lo = u - 2.0f * m - G.ext * (1.0f + 1e-6f);
  int l = G.first, r = G.first + G.count;  // the first member whose key exceeds hi
  while (l < r) {
    const int mid = (l + r) >> 1;
    if (a.rkeys[mid] <= hi) l = mid + 1;
    else r = mid;
  }
  int best = -1;
  for (int k = l - 1; k >= G.first && a.rkeys[k] >= lo; --k) {
    const int id = a.rmembers[k];
    if (best >= 0 && id > best) continue;
    bool skip = false;
    for (int i = 0; i < nex; ++i) skip = skip || id == ex[i];
    if (skip || !tri_box_near(a, id, x)) continue;
    d3w w0, w1, w2;
    float4 mt;
    tri64(a, id, w0, w1, w2, mt);
    if (inside_tri64(w0, w1, w2, x)) {
      best = id;
      v0 = w0;
      v1 = w1;
      v2 = w2;
      mat = mt;
    }
  }
  return best;
}

struct zv3 {
  zd x, y, z;
};
__device__ __forceinline__ zd zvdot(zv3 e, d3w v) {
  return Z(fma(e.z.re, v.z, fma(e.y.re, v.y, e.x.re * v.x)), fma(e.z.im, v.z, fma(e.y.im, v.y, e.x.im * v.x)));
}

// One survivor: exact geometry on the plane, the member triangle holding the
// reflection point, the geometry again on that triangle's own plane, the
// three legs, then the UTD field with the Fresnel reflection at P (bounce
// basis as in k_val_field) and the path record (depth 2).
__device__ __forceinline__ void diffract_refl_pair(const PathArgs& a, unsigned long long code, double k,
                                                   double lam, unsigned& ovf, TStack& st) {
  const bool first = (code & 1ull) != 0;
  code >>= 1;
  const int p = (int)(code % (unsigned long long)a.nrp);
  code /= (unsigned long long)a.nrp;
  const int w = (int)(code % (unsigned long long)a.nw), link = (int)(code / (unsigned long long)a.nw);
  const Wedge W = a.wedges[w];
  const RPlane Pl = a.rplanes[p];
  float4 rxv = a.rx[link % a.nrx], txv = a.txs[link / a.nrx];
  d3w T = D3(txv.x, txv.y, txv.z), R = D3(rxv.x, rxv.y, rxv.z);
  ReflGeom g;
  if (!refl_geometry(W, D3(Pl.n[0], Pl.n[1], Pl.n[2]), Pl.c, T, R, first, g)) return;
  d3w v0, v1, v2;
  float4 mj;
  const int exw[2] = {W.ta, W.tb};
  const int j = member_at(a, Pl, g.P, exw, 2, v0, v1, v2, mj);
  if (j < 0) return;
  // the member's own plane
  d3w nj = unitw(crossw(v1 - v0, v2 - v0));
  if (!refl_geometry(W, nj, dotw(nj, v0), T, R, first, g)) return;
  if (!inside_tri64(v0, v1, v2, g.P)) return;
  const d3w Q = g.Q, Pp = g.P;
  const d3w P[4] = {T, first ? Pp : Q, first ? Q : Pp, R};
  const int e0 = first ? j : W.ta, e1 = first ? j : W.tb, e2 = first ? W.ta : j, e3 = first ? W.tb : j;
  const int ex[4][2] = {{-1, -1}, {e0, e1}, {e2, e3}, {-1, -1}};
  if (legs_occluded(a, P, ex, 4, ovf, st)) return;
  unsigned fl = 0;
  const double n = W.n, phip = g.phip, phi = g.phi;
  d3w e = D3(W.e[0], W.e[1], W.e[2]);
  d3w qs = Q - g.S, oq = g.O - Q;
  double sp = sqrt(dotw(qs, qs)), s = sqrt(dotw(oq, oq));
  d3w ip = qs * (1.0 / sp), dd = oq * (1.0 / s);
  double beta0 = acos(fmax(-1.0, fmin(1.0, dotw(ip, e))));
  double sb = sin(beta0);
  double L = s * sp * sb * sb / (s + sp);
  d3w php = unitw(crossw(e, ip)) * -1.0, ph = unitw(crossw(e, dd));
  d3w bp = crossw(ip, php), bd = crossw(dd, ph);
  float4 ma, mb;
  {
    d3w x0, x1, x2;
    tri64(a, W.ta, x0, x1, x2, ma);
    tri64(a, W.tb, x0, x1, x2, mb);
  }
  zd r0s, r0h, rns, rnh;
  fresnel_faces(ma, fabs(sin(phip)), mb, fabs(sin(n * M_PI - phi)), a.freq, r0s, r0h, rns, rnh);
  const UtdParts up = utd_parts(n, phi, phip, beta0, L, k, fl);
  zd Ds = utd_coeff(up, r0s, rns);
  zd Dh = utd_coeff(up, r0h, rnh);
  // the reflection at P: directions and bounce basis
  d3w din = first ? unitw(Pp - T) : dd;
  d3w dout = first ? ip : unitw(R - Pp);
  double ct = fabs(dotw(din, nj));
  d3w sv = crossw(din, nj);
  double sn_ = sqrt(dotw(sv, sv));
  if (sn_ < 1e-12) {
    d3w ax = fabs(nj.x) < 0.9 ? D3(1, 0, 0) : D3(0, 1, 0);
    sv = unitw(crossw(nj, ax));
  } else {
    sv = sv * (1.0 / sn_);
  }
  d3w pin = crossw(sv, din), pout = crossw(sv, dout);
  zd gte, gtm;
  fresnel_d(mj, a.freq, ct, gte, gtm);
  d3w u = D3(a.pol.x, a.pol.y, a.pol.z);
  double sn, cs;
  sincos(-k * sp, &sn, &cs);
  zd Ei = Z(cs / sp, sn / sp);
  sincos(-k * s, &sn, &cs);
  zd A = Z(cs, sn) * sqrt(sp / (s * (s + sp)));
  zd proj;
  if (first) {
    d3w e0 = polw(u, din, fl);
    zd es = Z(dotw(e0, sv)), ep = Z(dotw(e0, pin));
    zd ts = gte * es, tp = gtm * ep;
    zv3 E1 = {ts * sv.x + tp * pout.x, ts * sv.y + tp * pout.y, ts * sv.z + tp * pout.z};
    zd Eb = Ei * zvdot(E1, bp), Ep = Ei * zvdot(E1, php);
    d3w prx = polw(u, dd * -1.0, fl);
    proj = (Ds * Eb) * (-dotw(bd, prx)) + (Dh * Ep) * (-dotw(ph, prx));
  } else {
    d3w e0 = polw(u, ip, fl);
    zd Eb = Ei * dotw(e0, bp), Ep = Ei * dotw(e0, php);
    zd cb = (Ds * Eb) * -1.0, cp = (Dh * Ep) * -1.0;
    zv3 Ed = {cb * bd.x + cp * ph.x, cb * bd.y + cp * ph.y, cb * bd.z + cp * ph.z};
    zd ts = gte * zvdot(Ed, sv), tp = gtm * zvdot(Ed, pin);
    zv3 E2 = {ts * sv.x + tp * pout.x, ts * sv.y + tp * pout.y, ts * sv.z + tp * pout.z};
    d3w prx = polw(u, dout * -1.0, fl);
    proj = zvdot(E2, prx);
  }
  zd amp = proj * A * (lam / (4.0 * M_PI));
  if (diff_lane() != 0) return;  // one lane of the group writes the record
  unsigned uu = atomicAdd(&a.ctr->n_unique, 1u);
  if (uu >= a.ucap) {
    atomicOr(&a.ctr->err, ERR_UNIQUE_OVERFLOW);
    return;
  }
  PathRec rec;
  const int id0 = first ? j : (w | kDiffBit), id1 = first ? (w | kDiffBit) : j;
  rec.key = seq_key(link % a.nrx, 2, [&](int q) { return q == 0 ? id0 : id1; });
  rec.rx = link;
  rec.depth = 2;
  rec.ray = -1;
  rec.flags = fl;
  rec.valid = 1;
  rec.pad = 0;
  rec.len = sp + s;
  rec.amp_re = amp.re;
  rec.amp_im = amp.im;
  for (int q = 0; q < kMaxRefl; ++q) {
    rec.tri[q] = q == 0 ? id0 : q == 1 ? id1 : -1;
    rec.pts[q][0] = rec.pts[q][1] = rec.pts[q][2] = 0.0f;
  }
  const d3w x0 = first ? Pp : Q, x1 = first ? Q : Pp;
  rec.pts[0][0] = (float)x0.x;
  rec.pts[0][1] = (float)x0.y;
  rec.pts[0][2] = (float)x0.z;
  rec.pts[1][0] = (float)x1.x;
  rec.pts[1][1] = (float)x1.y;
  rec.pts[1][2] = (float)x1.z;
  a.prec[uu] = rec;
  unsigned pos = atomicAdd(&a.bucket_cnt[link], 1u);
  if (pos < (unsigned)a.bucket_cap) a.bucket[(size_t)link * a.bucket_cap + pos] = (int)uu;
  else atomicOr(&a.ctr->err, ERR_BUCKET_OVERFLOW);
  atomicAdd(&a.ctr->n_valid, 1u);
}

// ---------------------------------------------------------------------------
// diffraction of order 2 and 3 (Sec. III step 5; the paper's bound is 3)
// ---------------------------------------------------------------------------
// Paths Tx -> Q_1 -> .. -> Q_m -> Rx over m pairwise distinct wedges,
// consecutive ones sharing no vertex, not on one line, neither edge in a
// face plane of the other. Per frame: the
// ordered wedge pairs that can start a path from a transmitter
// (k_diff_pairs), for m = 3 the triples built from them (k_diff_triples),
// then every (sequence, receiver) through an FP32 pre-test
// (k_diff_multi_pre). The pre-tests only reject what the FP64 test rejects
// too (margins above FP32 rounding); the
// survivors go to the diffraction survivor list with their order in the top
// bits: 01 order 2, 11 order 3 (10 is a reflection pair, 00 first order).
constexpr unsigned long long kKindShift = 62;
constexpr unsigned long long kMulti2 = 1ull << kKindShift, kMulti3 = 3ull << kKindShift;

__device__ __forceinline__ WedgeF wedge_f(const Wedge& W) {
  WedgeF f;
  f.p0 = f3((float)W.p0[0], (float)W.p0[1], (float)W.p0[2]);
  f.e = f3((float)W.e[0], (float)W.e[1], (float)W.e[2]);
  f.t0 = f3((float)W.t0[0], (float)W.t0[1], (float)W.t0[2]);
  f.y0 = f3((float)W.y0[0], (float)W.y0[1], (float)W.y0[2]);
  f.len = (float)W.len;
  f.npi = (float)(W.n * M_PI);
  return f;
}
// X in the wedge's normal plane: (along t0, along y0), its distance from the
// edge line and from the wedge's start.
__device__ __forceinline__ float2 wedge_plane(const WedgeF& W, float3 X, float& r, float& dist) {
  float3 d = f3(X.x - W.p0.x, X.y - W.p0.y, X.z - W.p0.z);
  float z = fdot3(d, W.e);
  float3 q = f3(d.x - W.e.x * z, d.y - W.e.y * z, d.z - W.e.z * z);
  r = sqrtf(fdot3(q, q));
  dist = sqrtf(fdot3(d, d));
  return make_float2(fdot3(q, W.t0), fdot3(q, W.y0));
}
// The point at parameter t along the edge.
__device__ __forceinline__ float3 edge_point(const WedgeF& W, float t) {
  return f3(W.p0.x + W.e.x * t, W.p0.y + W.e.y * t, W.p0.z + W.e.z * t);
}
// The edge's end points.
__device__ __forceinline__ void edge_ends(const WedgeF& W, float3& A, float3& B) {
  A = W.p0;
  B = f3(W.p0.x + W.e.x * W.len, W.p0.y + W.e.y * W.len, W.p0.z + W.e.z * W.len);
}
// Could some point of segment A-B lie strictly inside the angular sector
// (lo, hi) about wedge W (angles from face 0 through the exterior, hi - lo
// below pi)? The sector is the intersection of two half-spaces bounded by
// planes through the edge line, so the test clips the segment's parameter
// range against both; each plane is moved outward by `m` (metres) and the
// sector widened by `ta` (radians) first, so the answer is "no" only when
// the exact sector misses the segment by more than the margins.
__device__ __forceinline__ bool sector_meets(const WedgeF& W, float lo, float hi, float ta, float m, float3 A,
                                             float3 B) {
  lo -= ta;
  hi += ta;
  if (hi - lo >= 3.14f) return true;
  float ra, rb, da, db;
  float2 pa = wedge_plane(W, A, ra, da), pb = wedge_plane(W, B, rb, db);
  float u0 = 0.0f, u1 = 1.0f;
  for (int q = 0; q < 2; ++q) {
    float ang = q == 0 ? lo : hi, sg = q == 0 ? 1.0f : -1.0f;
    float c = cosf(ang), s = sinf(ang);
    // signed distance beyond the plane at angle `ang` toward the sector's inside
    float fa = sg * (c * pa.y - s * pa.x) + m, fb = sg * (c * pb.y - s * pb.x) + m;
    if (fa < 0.0f && fb < 0.0f) return false;
    if (fa < 0.0f) u0 = fmaxf(u0, fa / (fa - fb));
    else if (fb < 0.0f) u1 = fminf(u1, fa / (fa - fb));
  }
  return u0 <= u1 + 1e-3f;
}
// Margins of the pre-tests: angles by ten times their rounding bound (at
// least 1e-3 rad), positions by 5 cm plus 1e-5 of the coordinates' size.
__device__ __forceinline__ float pre_margin_m(float3 X) {
  return 0.05f + 1e-5f * (fabsf(X.x) + fabsf(X.y) + fabsf(X.z));
}
// Is X certainly inside wedge W (beyond its exterior [0, n pi])?
__device__ __forceinline__ bool surely_inside(const WedgeF& W, float3 X) {
  float r, dist;
  float2 p = wedge_plane(W, X, r, dist);
  bool sure;
  float tol;
  float a = wedge_angle32(f3(p.x * W.t0.x + p.y * W.y0.x, p.x * W.t0.y + p.y * W.y0.y, p.x * W.t0.z + p.y * W.y0.z),
                          W.t0, W.y0, r, dist, sure, tol);
  return sure && r > pre_margin_m(X) && a > W.npi + tol;
}
// Could some point of edge B's segment be in wedge A's exterior [0, n pi]?
__device__ __forceinline__ bool edge_sees(const WedgeF& A, const WedgeF& B, float m) {
  float3 P, Q;
  edge_ends(B, P, Q);
  // n >= 1: the interior (n pi, 2 pi) is a convex sector, so the segment is
  // inside it only when both ends are; n < 1: the exterior is the convex one
  if (A.npi >= 3.14159265f) return !(surely_inside(A, P) && surely_inside(A, Q));
  return sector_meets(A, 0.0f, A.npi, 1e-3f, m, P, Q);
}
// Could a point of segment P-Q be beyond the incident shadow boundary of a
// source X at wedge W (|phi - phi'| > pi, phi <= n pi)? The rule is
// symmetric in the two points, so this also tests a receiver X against the
// previous edge.
__device__ __forceinline__ bool shadow_meets(const WedgeF& W, float3 X, float3 P, float3 Q) {
  float r, dist;
  float2 p = wedge_plane(W, X, r, dist);
  float m = fmaxf(pre_margin_m(X), fmaxf(pre_margin_m(P), pre_margin_m(Q)));
  if (!(r > m)) return true;
  bool sure;
  float tol;
  float a = wedge_angle32(f3(p.x * W.t0.x + p.y * W.y0.x, p.x * W.t0.y + p.y * W.y0.y, p.x * W.t0.z + p.y * W.y0.z),
                          W.t0, W.y0, r, dist, sure, tol);
  if (!sure) return true;
  if (a > W.npi + tol) return false;  // X inside the wedge
  const float pi = 3.14159265f;
  if (fabsf(a - pi) <= tol) return true;
  float lo = a < pi ? a + pi : 0.0f, hi = a < pi ? W.npi : a - pi;
  if (hi < lo - tol) return false;
  return sector_meets(W, lo, hi, tol, m, P, Q);
}

// Keller points from the convexity of the unfolded length. The length of a
// chain is a sum of distances between affine functions of the edge
// parameters, so it is convex in them jointly and its derivative along one
// edge, e.(Q - A)/|Q - A| + e.(Q - B)/|Q - B| for Q's neighbours A and B,
// does not decrease as Q moves along the edge. When that derivative is
// positive at the edge's start (less a margin) for every position of the
// neighbours on their edges, or negative at its end, the minimum -- the
// Keller points -- has Q, or a neighbour, off its edge, and the exact stage
// rejects the chain. The tests below bound the derivative's two terms.

// Extremes of e.(Q - Y)/|Q - Y| for Y on wedge S's edge with parameter in
// [lo, hi], and a lower bound of |Q - Y| there. The directions from Q to the
// segment's points sweep an arc of a great circle (below pi), along which
// the cosine is |e_p| cos(angle to e_p), e_p the projection of e onto the
// arc's plane: the extremes are at the arc's ends, or +-|e_p| where e_p (or
// -e_p) points into the arc.
__device__ __forceinline__ void cos_over_edge(float3 e, float3 Q, const WedgeF& S, float lo, float hi, float& cmin,
                                              float& cmax, float& dmin) {
  const float3 d0 = f3(Q.x - S.p0.x - S.e.x * lo, Q.y - S.p0.y - S.e.y * lo, Q.z - S.p0.z - S.e.z * lo);
  const float3 d1 = f3(Q.x - S.p0.x - S.e.x * hi, Q.y - S.p0.y - S.e.y * hi, Q.z - S.p0.z - S.e.z * hi);
  const float l0 = sqrtf(fdot3(d0, d0)), l1 = sqrtf(fdot3(d1, d1));
  const float c0 = fdot3(e, d0) / l0, c1 = fdot3(e, d1) / l1;
  cmin = fminf(c0, c1);
  cmax = fmaxf(c0, c1);
  const float3 n = cross3(d0, d1);
  const float nn = sqrtf(fdot3(n, n));
  dmin = fminf(fminf(l0, l1), nn / (hi - lo));  // the distance to the segment's line at most
  if (nn > 1e-3f * l0 * l1) {
    const float3 u = f3(n.x / nn, n.y / nn, n.z / nn);
    const float en = fdot3(e, u), pn = sqrtf(fmaxf(0.0f, 1.0f - en * en));
    const float3 ep = f3(e.x - en * u.x, e.y - en * u.y, e.z - en * u.z);
    // e_p between the arc's ends (with a tolerance that only widens the range)
    const float s0 = fdot3(ep, cross3(u, d0)), s1 = fdot3(ep, cross3(d1, u));
    const float g0 = 1e-3f * l0, g1 = 1e-3f * l1;
    if (s0 >= -g0 && s1 >= -g1) cmax = fmaxf(cmax, pn);
    if (s0 <= g0 && s1 <= g1) cmin = fminf(cmin, -pn);
  } else {  // an arc shorter than 1e-3 rad (or Q on the segment: dmin tells)
    cmin -= 2e-3f;
    cmax += 2e-3f;
  }
}
// Could the Keller point on wedge W's edge lie within m of the edge, its
// neighbours being point F (has_f) or a point of wedge S1's edge, and a
// point of wedge S2's edge, both edges widened by m? False only when the
// derivative's bound keeps its sign at both ends by more than its FP32
// rounding (1e-6 of the coordinates' size over the distance, per term).
__device__ bool keller_on_edge(const WedgeF& W, bool has_f, float3 F, const WedgeF& S1, const WedgeF& S2, float m) {
  for (int q = 0; q < 2; ++q) {
    const float t = q ? W.len + m : -m;
    const float3 Q = edge_point(W, t);
    const float sq = fabsf(Q.x) + fabsf(Q.y) + fabsf(Q.z);
    float lo1, hi1, d1, lo2, hi2, d2, s1;
    if (has_f) {
      const float3 d = f3(Q.x - F.x, Q.y - F.y, Q.z - F.z);
      d1 = sqrtf(fdot3(d, d));
      lo1 = hi1 = fdot3(W.e, d) / d1;
      s1 = fabsf(F.x) + fabsf(F.y) + fabsf(F.z);
    } else {
      cos_over_edge(W.e, Q, S1, -m, S1.len + m, lo1, hi1, d1);
      s1 = fabsf(S1.p0.x) + fabsf(S1.p0.y) + fabsf(S1.p0.z) + S1.len;
    }
    cos_over_edge(W.e, Q, S2, -m, S2.len + m, lo2, hi2, d2);
    const float s2 = fabsf(S2.p0.x) + fabsf(S2.p0.y) + fabsf(S2.p0.z) + S2.len;
    if (!(d1 > 4.0f * m && d2 > 4.0f * m)) return true;
    const float err = 4e-5f + 2e-6f * ((sq + s1) / d1 + (sq + s2) / d2);
    if (q == 0 && lo1 + lo2 > err) return false;
    if (q == 1 && hi1 + hi2 < -err) return false;
  }
  return true;
}
// The margin of these tests: 5 cm plus 1e-5 of the coordinates' size.
__device__ __forceinline__ float keller_margin(const WedgeF& W, float3 F) {
  return 0.05f + 1e-5f * (fabsf(W.p0.x) + fabsf(W.p0.y) + fabsf(W.p0.z) + W.len + fabsf(F.x) + fabsf(F.y) + fabsf(F.z));
}

// Do two edges share an end vertex (identical coordinates)? Consecutive
// wedges of a chain may not (which includes sharing a face): the length's
// minimum then tends to the common corner, or the leg between them runs
// along a face they bound.
__device__ __forceinline__ bool share_vertex(const Wedge& A, const Wedge& B) {
  const double* a[2] = {A.p0, A.p1};
  const double* b[2] = {B.p0, B.p1};
  for (int i = 0; i < 2; ++i)
    for (int j = 0; j < 2; ++j)
      if (a[i][0] == b[j][0] && a[i][1] == b[j][1] && a[i][2] == b[j][2]) return true;
  return false;
}

// Do two edges lie on one line (directions parallel to 1e-9, the second's
// start within 1e-9 m, relative to the coordinates' size, of the first's
// line)? Consecutive wedges of a chain may not: the leg between them would
// run along both edges (no Keller points: the length's minimum is where it
// vanishes). Decided in FP64 from the wedges' frames.
__device__ __forceinline__ bool collinear_edges(const Wedge& A, const Wedge& B) {
  d3w ea = D3(A.e[0], A.e[1], A.e[2]), eb = D3(B.e[0], B.e[1], B.e[2]);
  d3w c = crossw(ea, eb);
  if (sqrt(dotw(c, c)) > 1e-9) return false;
  d3w pa = D3(A.p0[0], A.p0[1], A.p0[2]), pb = D3(B.p0[0], B.p0[1], B.p0[2]);
  d3w q = crossw(pb - pa, ea);
  double sa = fmax(fabs(pa.x), fmax(fabs(pa.y), fabs(pa.z))), sb = fmax(fabs(pb.x), fmax(fabs(pb.y), fabs(pb.z)));
  return sqrt(dotw(q, q)) <= 1e-9 * (1.0 + sa + sb);
}

// Does edge B lie in the plane of a face of wedge A (both ends within 1e-9 m,
// relative to the coordinates' size)? Then so does the leg between them,
// along that face (grazing) or its extension beyond A's edge, where no source
// in A's exterior has its shadow boundary crossed: no chain passes.
__device__ __forceinline__ bool in_face_plane(const Wedge& A, const Wedge& B) {
  d3w e = D3(A.e[0], A.e[1], A.e[2]), pa = D3(A.p0[0], A.p0[1], A.p0[2]);
  d3w b0 = D3(B.p0[0], B.p0[1], B.p0[2]) - pa, b1 = D3(B.p1[0], B.p1[1], B.p1[2]) - pa;
  double sa = fmax(fabs(pa.x), fmax(fabs(pa.y), fabs(pa.z)));
  double sb = fmax(fabs(B.p0[0]), fmax(fabs(B.p0[1]), fabs(B.p0[2])));
  double tol = 1e-9 * (1.0 + sa + sb);
  d3w f[2] = {crossw(e, D3(A.t0[0], A.t0[1], A.t0[2])), crossw(e, D3(A.tB[0], A.tB[1], A.tB[2]))};
  for (int q = 0; q < 2; ++q)
    if (fabs(dotw(f[q], b0)) <= tol && fabs(dotw(f[q], b1)) <= tol) return true;
  return false;
}

// Source v of a chain (a transmitter, or its image in a reflector plane) and
// observer rho (a receiver, or its image), in FP32 for the pre-tests.
__device__ __forceinline__ float3 chain_source32(const PathArgs& a, int v) {
  if (v < a.dntx) {
    float4 t = a.txs[v];
    return f3(t.x, t.y, t.z);
  }
  int i = v - a.dntx;
  float4 t = a.txs[i / a.nrpr];
  const RPlane& P = a.rplanes[i % a.nrpr];
  return mirror32(f3(t.x, t.y, t.z), f3(P.nf[0], P.nf[1], P.nf[2]), P.cf);
}
__device__ __forceinline__ float3 chain_observer32(const PathArgs& a, int rho) {
  if (rho < a.nrx) {
    float4 r = a.rx[rho];
    return f3(r.x, r.y, r.z);
  }
  int i = rho - a.nrx;
  float4 r = a.rx[i / a.nrpr];
  const RPlane& P = a.rplanes[i % a.nrpr];
  return mirror32(f3(r.x, r.y, r.z), f3(P.nf[0], P.nf[1], P.nf[2]), P.cf);
}

// Can a leg from S to some point of segment A-B cross reflector plane Pl
// inside its box? The legs fill the triangle S, A, B; its section by the
// plane lies within the box of the crossings of its three sides, so the
// answer is "no" when S, A and B lie on one side of the plane (by more than
// the margin m), or when that box, widened by m, misses the plane's box;
// else [lo, hi] is the part of it (widened by m) that holds the crossings.
__device__ __forceinline__ bool leg_window(const RPlane& Pl, float3 S, float3 A, float3 B, float m, float* lo,
                                           float* hi) {
  const float3 n = f3(Pl.nf[0], Pl.nf[1], Pl.nf[2]);
  const float c = Pl.cf;
  const float ds = fdot3(n, S) - c, da = fdot3(n, A) - c, db = fdot3(n, B) - c;
  if ((ds > m && da > m && db > m) || (ds < -m && da < -m && db < -m)) return false;
  for (int k = 0; k < 3; ++k) {
    lo[k] = 3e38f;
    hi[k] = -3e38f;
  }
  bool any = false;
  const float3 P0[3] = {S, S, A}, P1[3] = {A, B, B};
  const float d0[3] = {ds, ds, da}, d1[3] = {da, db, db};
  for (int e = 0; e < 3; ++e) {
    if ((d0[e] > m && d1[e] > m) || (d0[e] < -m && d1[e] < -m)) continue;
    // the part of this side within m of the plane
    float den = d0[e] - d1[e];
    float ta = 0.0f, tb = 1.0f;
    if (fabsf(den) > 1e-30f) {
      float t1 = (d0[e] - m) / den, t2 = (d0[e] + m) / den;
      ta = fmaxf(0.0f, fminf(t1, t2));
      tb = fminf(1.0f, fmaxf(t1, t2));
    }
    if (ta > tb) continue;
    for (int q = 0; q < 2; ++q) {
      float t = q ? tb : ta;
      float x = P0[e].x + t * (P1[e].x - P0[e].x), y = P0[e].y + t * (P1[e].y - P0[e].y),
            z = P0[e].z + t * (P1[e].z - P0[e].z);
      lo[0] = fminf(lo[0], x); lo[1] = fminf(lo[1], y); lo[2] = fminf(lo[2], z);
      hi[0] = fmaxf(hi[0], x); hi[1] = fmaxf(hi[1], y); hi[2] = fmaxf(hi[2], z);
    }
    any = true;
  }
  if (!any) return false;
  bool meet = true;
  for (int k = 0; k < 3; ++k) {
    lo[k] = fmaxf(lo[k], Pl.box[k]) - m;
    hi[k] = fminf(hi[k], Pl.box[3 + k]) + m;
    meet = meet && lo[k] <= hi[k];
  }
  return meet;
}
__device__ __forceinline__ bool plane_reachable(const RPlane& Pl, float3 S, float3 A, float3 B, float m) {
  float lo[3], hi[3];
  return leg_window(Pl, S, A, B, m, lo, hi);
}

// ---- what an end point can see ----
// In built-up scenes most reflector planes and wedges are hidden from a given
// end point (and from one another) behind one wall, and every real leg must
// be free: so the planes and wedges that are certainly hidden from an end
// point as a whole take no part as its first reflection or as the wedge it
// sees directly, and two wedges hidden from each other are no chain's
// neighbours. A target is hidden when one convex wall quad -- two static coplanar
// triangles that share an edge -- is crossed strictly inside, by the margins
// of leg_surely_blocked, by the legs to every corner of the target: the
// crossings of the legs to the points between the corners lie between
// theirs. The quads tried are those the leg to the target's middle crosses.

__device__ __forceinline__ float3 end_point(const PathArgs& a, int ntx, int x) {
  const float4 v = x < ntx ? a.txs[x] : a.rx[x - ntx];
  return f3(v.x, v.y, v.z);
}

// Does quad q (q[0].w != 0) cut off point X from E with margin?
__device__ __forceinline__ bool quad_between(const float4* __restrict__ q, float3 E, float3 X, float eps_occ) {
  const float4 q0 = q[0], q1 = q[1], q2 = q[2], q3 = q[3];
  if (q0.w == 0.0f) return false;
  const float3 c[4] = {f3(q0.x, q0.y, q0.z), f3(q1.x, q1.y, q1.z), f3(q2.x, q2.y, q2.z), f3(q3.x, q3.y, q3.z)};
  const float3 dv = f3(X.x - E.x, X.y - E.y, X.z - E.z);
  const float dl = sqrtf(fdot3(dv, dv));
  const float3 nv = cross3(f3(c[1].x - c[0].x, c[1].y - c[0].y, c[1].z - c[0].z),
                           f3(c[2].x - c[0].x, c[2].y - c[0].y, c[2].z - c[0].z));
  const float nn = sqrtf(fdot3(nv, nv)), dn = fdot3(dv, nv);
  if (!(dl > 0.0f && fabsf(dn) > 1e-3f * dl * nn)) return false;
  const float u = fdot3(f3(c[0].x - E.x, c[0].y - E.y, c[0].z - E.z), nv) / dn;
  const float slack = 2e-3f + 1e-6f * (fabsf(E.x) + fabsf(E.y) + fabsf(E.z) + dl);
  const float mu = 0.01f * (1.0f + dl * nn / fabsf(dn)) + slack, nu = mu / dl;
  if (!(u > eps_occ + nu && u < 1.0f - eps_occ - nu)) return false;
  const float3 H = f3(E.x + dv.x * u, E.y + dv.y * u, E.z + dv.z * u);
  for (int k = 0; k < 4; ++k) {
    const float3 a = c[k], b = c[(k + 1) & 3];
    const float3 e = f3(b.x - a.x, b.y - a.y, b.z - a.z);
    const float el = sqrtf(fdot3(e, e));
    if (el > 0.0f && !(fdot3(cross3(e, f3(H.x - a.x, H.y - a.y, H.z - a.z)), nv) > mu * el * nn)) return false;
  }
  return true;
}

// What is to be hidden: from E0 the box lo..hi (kind 0) or the segment lo-hi
// (1), or from the segment E0-E1 the segment lo-hi (2: the crossings of the
// legs between two segments on either side of a plane are convex
// combinations of those of the four legs between their ends).
struct HiddenCase {
  int kind;
  float3 E0, E1, lo, hi;
};
// Is it certainly hidden behind one quad?
__device__ __noinline__ bool surely_hidden(const PathArgs& a, const HiddenCase& h, TStack& st) {
  const float3 lo = h.lo, hi = h.hi;
  const float3 mid = f3(0.5f * (lo.x + hi.x), 0.5f * (lo.y + hi.y), 0.5f * (lo.z + hi.z));
  const float3 E = h.kind < 2 ? h.E0 : f3(0.5f * (h.E0.x + h.E1.x), 0.5f * (h.E0.y + h.E1.y), 0.5f * (h.E0.z + h.E1.z));
  const RayPre rp = ray_pre(E, f3(mid.x - E.x, mid.y - E.y, mid.z - E.z));
  st.reset();
  int cur = a.bvh.root0;  // static triangles only
  for (int visits = 0; visits <= a.bvh.max_visits; ++visits) {
    if (cur == kEmpty) {
      if (st.empty()) break;
      cur = st.pop();
      continue;
    }
    if (cur >= 0) {
      const float4* n = a.bvh.nodes + 4 * (size_t)DCEM_IDX(cur, a.bvh.nnodes);
      float4 n0 = __ldg(n), n1 = __ldg(n + 1), n2 = __ldg(n + 2), n3 = __ldg(n + 3);
      float tn0, tn1;
      const bool h0 = slab(rp, n0.x, n0.y, n0.z, n0.w, n2.x, n2.y, 1.0f, tn0);
      const bool h1 = slab(rp, n1.x, n1.y, n1.z, n1.w, n2.z, n2.w, 1.0f, tn1);
      const int c0 = __float_as_int(n3.x), c1 = __float_as_int(n3.y);
      if (h0 && h1) {
        if (!st.push(c1)) return false;
        cur = c0;
      } else {
        cur = h0 ? c0 : h1 ? c1 : kEmpty;
      }
      continue;
    }
    const int id = __float_as_int(__ldg(&a.bvh.tris[3 * (size_t)DCEM_IDX(~cur, a.bvh.ntris)]).w);
    cur = kEmpty;
    const float4* q = a.quads + 4 * (size_t)DCEM_IDX(id, a.bvh.ntris);
    bool all = quad_between(q, E, mid, a.eps_occ);
    for (int k = 0; all && k < (h.kind == 0 ? 8 : 2 * h.kind); ++k) {
      const float3 X = h.kind ? ((k & 1) ? hi : lo)
                              : f3((k & 1) ? hi.x : lo.x, (k & 2) ? hi.y : lo.y, (k & 4) ? hi.z : lo.z);
      all = quad_between(q, h.kind == 2 ? ((k & 2) ? h.E1 : h.E0) : E, X, a.eps_occ);
    }
    if (all) return true;
  }
  return false;
}

// Per end point the planes, then the wedges (in the order wperm) it may see,
// one warp per word. A wedge the end point is inside of is not seen. Both
// orders are spatial, so that a warp's legs run close together. Without
// `test` everything else counts as seen: a road and its barriers are open, and
// a highway's 480,000 legs of up to 2 km cost 240 us a frame and hid nothing.
// Neither do they pay for one reflection without chains, whose candidates are
// cheap to form: 8 x 8 city blocks with 10, 30 and 60 receivers 542, 587 and
// 648 us a frame with the tests, 365, 453 and 531 without.
__global__ void __launch_bounds__(64) k_diff_visible(PathArgs a, int ntx, bool test) {
  extern __shared__ int sstk[];
  TStack st;
  bind_stack(st, sstk, kStackTrace);
  const int npw = (a.nrp + 31) / 32, row = npw + a.nwc, lane = threadIdx.x & 31;
  const long nitem = (long)(ntx + a.nrx) * row, nwarp = (long)gridDim.x * (blockDim.x >> 5);
  for (long it = (long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); it < nitem; it += nwarp) {
    const int x = (int)(it / row), c = (int)(it - (long)x * row);
    const float3 E = end_point(a, ntx, x);
    bool see = false;
    if (c < npw) {
      const int p = c * 32 + lane;
      if (p < a.nrp) {
        const float* b = a.rplanes[p].box;
        see = !test || !surely_hidden(a, HiddenCase{0, E, E, f3(b[0], b[1], b[2]), f3(b[3], b[4], b[5])}, st);
      }
    } else {
      const int i = (c - npw) * kWedgeCluster + lane;
      if (i < a.nw) {
        const WedgeF W = a.wf[a.wperm[i]];
        float3 A, B;
        edge_ends(W, A, B);
        see = !surely_inside(W, E) && !(test && surely_hidden(a, HiddenCase{1, E, E, A, B}, st));
      }
    }
    const unsigned m = __ballot_sync(0xffffffffu, see);
    if (lane == 0) a.vis[it] = m;
  }
}
// Pairs of up to kHiddenSample planes: is the one's box hidden from the
// other's middle? Once per scene (the static triangles do not move). One
// thread a block: the time is that of one warp's traversals (8 x 8 city: the
// set-up of the planes takes 321 us without, 436 with this, 495 with four pairs
// a warp, 718 with 64 planes and 32 pairs a warp).
constexpr int kHiddenSample = 32;
__global__ void __launch_bounds__(1) k_hidden_planes(PathArgs a, unsigned* cnt) {
  extern __shared__ int sstk[];
  TStack st;
  bind_stack(st, sstk, kStackTrace);
  const int n = gridDim.y;
  if (blockIdx.x == blockIdx.y) return;
  const float* b = a.rplanes[(int)((long)blockIdx.x * a.nrp / n)].box;
  const float* c = a.rplanes[(int)((long)blockIdx.y * a.nrp / n)].box;
  const float3 E = f3(0.5f * (b[0] + b[3]), 0.5f * (b[1] + b[4]), 0.5f * (b[2] + b[5]));
  if (surely_hidden(a, HiddenCase{0, E, E, f3(c[0], c[1], c[2]), f3(c[3], c[4], c[5])}, st)) atomicAdd(&cnt[0], 1u);
  atomicAdd(&cnt[1], 1u);
}

// The wedges some transmitter (words 0 .. nwc - 1) or some receiver sees, and
// lists of the groups that hold any (per side a count, then the groups).
__global__ void __launch_bounds__(256) k_diff_visible_any(PathArgs a, int ntx) {
  __shared__ unsigned cnt;
  const int npw = (a.nrp + 31) / 32, row = npw + a.nwc, side = blockIdx.x;
  const int ng = (a.nw + kWedgeGroup - 1) / kWedgeGroup;
  int* list = a.vis_grp + (size_t)side * (ng + 1);
  if (threadIdx.x == 0) cnt = 0u;
  __syncthreads();
  for (int c0 = 0; c0 < a.nwc; c0 += 32) {  // lanes: words, warps: end points
    __shared__ unsigned part[32];
    const int c = c0 + (threadIdx.x & 31);
    if (threadIdx.x < 32) part[threadIdx.x] = 0u;
    __syncthreads();
    if (c < a.nwc) {
      unsigned m = 0;
      const int x1 = side ? ntx + a.nrx : ntx;
      for (int x = (side ? ntx : 0) + (threadIdx.x >> 5); x < x1; x += 8) m |= a.vis[(long)x * row + npw + c];
      atomicOr(&part[threadIdx.x & 31], m);
    }
    __syncthreads();
    if (threadIdx.x < 32 && c < a.nwc) {
      const unsigned m = part[threadIdx.x];
      a.vis_any[side * a.nwc + c] = m;
      for (int k = 0; k < 4; ++k)
        if ((m >> (8 * k)) & 0xffu) list[1 + atomicAdd(&cnt, 1u)] = 4 * c + k;
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) list[0] = (int)cnt;
}
__device__ __forceinline__ bool sees_plane(const PathArgs& a, int x, int p) {
  const int npw = (a.nrp + 31) / 32;
  return (a.vis[(long)x * (npw + a.nwc) + p / 32] >> (p & 31)) & 1u;
}
// (i: the wedge's place in the order wperm)
__device__ __forceinline__ bool sees_wedge(const PathArgs& a, int x, int i) {
  const int npw = (a.nrp + 31) / 32;
  return (a.vis[(long)x * (npw + a.nwc) + npw + i / kWedgeCluster] >> (i % kWedgeCluster)) & 1u;
}

// (as sees_wedge, for wedge w; true when the rows are not built)
__device__ __forceinline__ bool end_sees(const PathArgs& a, int x, int w) { return !a.vis || sees_wedge(a, x, a.wplace[w]); }
__device__ __forceinline__ bool wedges_hidden(const PathArgs& a, const WedgeF& A, const WedgeF& B, TStack& st) {
  HiddenCase h;
  h.kind = 2;
  edge_ends(A, h.E0, h.E1);
  edge_ends(B, h.lo, h.hi);
  return surely_hidden(a, h, st);
}

// The relation of consecutive wedges in a chain, once per frame (moving
// wedges change it): distinct, no shared vertex, not on one line, neither
// edge in a face plane of the other, each edge partly in the other's
// exterior; one bit per ordered pair (w1, w2) in a.drel. It is symmetric: a
// warp takes 32 pairs w1 < w2 of one w1 and sets both bits. With chains of
// three wedges the pairs hidden from each other are dropped here (every
// triple holds two; 8 x 8 city: 335k triples become a tenth). With chains of
// two that costs more than it saves: 8 x 8, 5 x 5 and 3 x 3 city blocks with
// one reflection 2910, 991 and 694 us a frame with it, 2703, 860 and 642 without.
__global__ void __launch_bounds__(256) k_diff_rel(PathArgs a) {
  extern __shared__ int sstk[];
  TStack st;
  bind_stack(st, sstk, kStackTrace);
  const long nw = a.nw, nch = (nw + 31) / 32, nitem = nw * nch;
  const int lane = threadIdx.x & 31;
  const long nwarp = (long)gridDim.x * (blockDim.x >> 5);
  for (long it = (long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); it < nitem; it += nwarp) {
    const int w1 = (int)(it / nch), w2 = (int)(it - (long)w1 * nch) * 32 + lane;
    bool rel = w1 < w2 && w2 < nw;
    if (!__any_sync(0xffffffffu, rel)) continue;
    if (rel) {  // the FP32 exterior tests first: they reject most pairs
      const WedgeF fa = a.wf[w1], fb = a.wf[w2];
      float3 pa, qa, pb, qb;
      edge_ends(fa, pa, qa);
      edge_ends(fb, pb, qb);
      const float m = fmaxf(fmaxf(pre_margin_m(pa), pre_margin_m(qa)), fmaxf(pre_margin_m(pb), pre_margin_m(qb)));
      rel = edge_sees(fa, fb, m) && edge_sees(fb, fa, m);
      if (rel && a.diff_order >= 3) rel = !wedges_hidden(a, fa, fb, st);
    }
    if (rel) {
      const Wedge &A = a.wedges[w1], &B = a.wedges[w2];
      rel = !share_vertex(A, B) && !collinear_edges(A, B) && !in_face_plane(A, B) && !in_face_plane(B, A);
    }
    if (rel) {
      const long x = (long)w1 * nw + w2, y = (long)w2 * nw + w1;
      atomicOr(&a.drel[x >> 5], 1u << (x & 31));
      atomicOr(&a.drel[y >> 5], 1u << (y & 31));
    }
  }
}

// Ordered pairs (w1, w2) per source (transmitter or transmitter image) that
// can start a path of order >= 2: in the relation (k_diff_rel), the
// transmitter outside w1, some point of edge 2 beyond the incident shadow
// boundary of the transmitter at w1, a Keller point on w1 possible between
// the transmitter and edge 2 (keller_on_edge), and w1 (an image's plane) not
// hidden from the transmitter. (No test here of whether w2 is hidden from w1:
// the traversal took the kernel from 63 to 89 registers and 296 B of stack,
// for every pair; without it 8 x 8 city blocks took 559 us a frame instead of
// 682 at order 2, 2890 instead of 3283 with one reflection, and this kernel on
// a 200-vehicle highway 810 us instead of 1190.)
__global__ void __launch_bounds__(256) k_diff_pairs(PathArgs a, int nsrc) {
  const long nw = a.nw, total = (long)nsrc * nw * nw;
  const int lane = threadIdx.x & 31;
  const long stride = (long)gridDim.x * blockDim.x;
  for (long base = (long)blockIdx.x * blockDim.x + (threadIdx.x & ~31); base < total; base += stride) {
    long idx = base + lane;
    bool keep = false;
    int t = 0, w1 = 0, w2 = 0;
    if (idx < total) {
      t = (int)(idx / (nw * nw));
      long r = idx - (long)t * nw * nw;
      w1 = (int)(r / nw);
      w2 = (int)(r - (long)w1 * nw);
      const bool seen = t < a.dntx ? end_sees(a, t, w1)
                                   : !a.vis || sees_plane(a, (t - a.dntx) / a.nrpr, (t - a.dntx) % a.nrpr);
      if (seen && ((a.drel[r >> 5] >> (r & 31)) & 1u)) {
        const WedgeF fa = a.wf[w1], fb = a.wf[w2];
        float3 T = chain_source32(a, t), P, Q;
        edge_ends(fb, P, Q);
        keep = !surely_inside(fa, T) && shadow_meets(fa, T, P, Q) && keller_on_edge(fa, true, T, fb, fb, keller_margin(fa, T));
        if (keep && t >= a.dntx) {  // the image's leg to edge 1 crosses its plane inside the box
          float3 A1, B1;
          edge_ends(fa, A1, B1);
          float mg = 0.1f + 1e-4f * (fabsf(T.x) + fabsf(T.y) + fabsf(T.z) + fa.len);
          keep = plane_reachable(a.rplanes[(t - a.dntx) % a.nrpr], T, A1, B1, mg);
        }
      }
    }
    unsigned mk = __ballot_sync(0xffffffffu, keep);
    if (!mk) continue;
    unsigned at = 0;
    if (lane == 0) at = atomicAdd(&a.ctr->n_dpair, (unsigned)__popc(mk));
    at = __shfl_sync(0xffffffffu, at, 0) + __popc(mk & ((1u << lane) - 1u));
    if (keep) {
      if (at < a.dseq2_cap) a.dseq2[at] = make_int4(t, w1, w2, -1);
      else atomicOr(&a.ctr->err, ERR_DIFF_OVERFLOW);
      if (a.dobs1) atomicOr(&a.dsecond[w2 >> 5], 1u << (w2 & 31));
    }
  }
}

// A wedge's FP32 frame mirrored in plane (n, c): the point and directions
// mirrored, the length and exterior angle kept (the angle of a mirrored
// point about the mirrored edge is that of the point about the edge).
__device__ __forceinline__ WedgeF wedge_mirror32(const WedgeF& W, float3 n, float c) {
  auto dir = [&](float3 v) {
    const float h = 2.0f * fdot3(n, v);
    return f3(v.x - h * n.x, v.y - h * n.y, v.z - h * n.z);
  };
  WedgeF M = W;
  M.p0 = mirror32(W.p0, n, c);
  M.e = dir(W.e);
  M.t0 = dir(W.t0);
  M.y0 = dir(W.y0);
  return M;
}

// A wedge mirrored in plane (n, c) in FP64 (as wedge_mirror32).
__device__ __forceinline__ Wedge wedge_mirror64(const Wedge& W, d3w n, double c) {
  auto put = [](double* dst, d3w v) {
    dst[0] = v.x;
    dst[1] = v.y;
    dst[2] = v.z;
  };
  auto pt = [&](const double* x) {
    const d3w v = D3(x[0], x[1], x[2]);
    return v - n * (2.0 * (dotw(n, v) - c));
  };
  auto dir = [&](const double* x) {
    const d3w v = D3(x[0], x[1], x[2]);
    return v - n * (2.0 * dotw(n, v));
  };
  Wedge M = W;
  put(M.p0, pt(W.p0));
  put(M.p1, pt(W.p1));
  put(M.e, dir(W.e));
  put(M.t0, dir(W.t0));
  put(M.y0, dir(W.y0));
  put(M.tB, dir(W.tB));
  return M;
}

// Does the edge of W lie in plane (n, c) up to rounding (both ends within
// 1e-12 m, relative to the coordinates' size)? A reflection in that plane
// next to the edge would sit at the diffraction point itself (the oracle
// flags such a reflection point at its leg's end).
__device__ __forceinline__ bool edge_in_plane(const Wedge& W, d3w n, double c) {
  const double tol = 1e-12 * (1.0 + fmax(fabs(W.p0[0]), fmax(fabs(W.p0[1]), fabs(W.p0[2]))));
  return fabs(dotw(n, D3(W.p0[0], W.p0[1], W.p0[2])) - c) <= tol &&
         fabs(dotw(n, D3(W.p1[0], W.p1[1], W.p1[2])) - c) <= tol;
}

// Can a leg from a point of segment A0-A1 to a point of segment B0-B1 cross
// plane Pl inside its box? Such legs fill the tetrahedron of the four ends,
// whose section by the plane lies within the box of the crossings of its six
// edges; "no" when the four ends lie on one side (by more than m) or that
// box, widened by m, misses the plane's box.
__device__ __forceinline__ bool section_reachable(const RPlane& Pl, float3 A0, float3 A1, float3 B0, float3 B1,
                                                  float m) {
  const float3 n = f3(Pl.nf[0], Pl.nf[1], Pl.nf[2]);
  const float3 X[4] = {A0, A1, B0, B1};
  float d[4];
  bool pos = false, neg = false;
  for (int i = 0; i < 4; ++i) {
    d[i] = fdot3(n, X[i]) - Pl.cf;
    pos = pos || d[i] > -m;
    neg = neg || d[i] < m;
  }
  if (!pos || !neg) return false;
  float lo[3] = {3e38f, 3e38f, 3e38f}, hi[3] = {-3e38f, -3e38f, -3e38f};
  bool any = false;
  for (int i = 0; i < 4; ++i)
    for (int j = i + 1; j < 4; ++j) {
      if ((d[i] > m && d[j] > m) || (d[i] < -m && d[j] < -m)) continue;
      const float den = d[i] - d[j];
      float ta = 0.0f, tb = 1.0f;
      if (fabsf(den) > 1e-30f) {
        const float t1 = (d[i] - m) / den, t2 = (d[i] + m) / den;
        ta = fmaxf(0.0f, fminf(t1, t2));
        tb = fminf(1.0f, fmaxf(t1, t2));
      }
      if (ta > tb) continue;
      for (int q = 0; q < 2; ++q) {
        const float t = q ? tb : ta;
        const float x = X[i].x + t * (X[j].x - X[i].x), y = X[i].y + t * (X[j].y - X[i].y),
                    z = X[i].z + t * (X[j].z - X[i].z);
        lo[0] = fminf(lo[0], x); lo[1] = fminf(lo[1], y); lo[2] = fminf(lo[2], z);
        hi[0] = fmaxf(hi[0], x); hi[1] = fmaxf(hi[1], y); hi[2] = fmaxf(hi[2], z);
      }
      any = true;
    }
  if (!any) return false;
  for (int k = 0; k < 3; ++k)
    if (hi[k] < Pl.box[k] - m || lo[k] > Pl.box[3 + k] + m) return false;
  return true;
}

// Wedge pairs with a reflection between them (Sec. III steps 3-5): per
// (transmitter, first wedge, reflector plane), one warp, its lanes over the
// second wedge. By image theory the path Tx -> Q1 -> P -> Q2 -> Rx is the
// chain over w1 and w2's image in the plane; the pair is kept when that
// image and w1 satisfy the pair tests of k_diff_pairs (each partly in the
// other's exterior, some point of the image beyond the transmitter's shadow
// boundary at w1, the transmitter outside w1, a Keller point on w1
// possible) and some leg between the two edges can cross the plane inside
// its box. Entries (t, w1, w2, -2 - p) join
// the pair list (k_diff_triples skips them); the FP64 vertex, line and
// face-plane rules are the exact stage's.
__global__ void __launch_bounds__(256) k_diff_mid_pairs(PathArgs a) {
  const long nblk = (long)a.dntx * a.nw * a.nrp;
  const int lane = threadIdx.x & 31;
  const long nwarp = (long)gridDim.x * (blockDim.x >> 5);
  for (long b = (long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); b < nblk; b += nwarp) {
    const int p = (int)(b % a.nrp);
    const long r = b / a.nrp;
    const int w1 = (int)(r % a.nw), t = (int)(r / a.nw);
    const WedgeF fa = a.wf[w1];
    const float3 T = chain_source32(a, t);
    if (surely_inside(fa, T) || !end_sees(a, t, w1)) continue;  // warp-uniform
    const RPlane& Pl = a.rplanes[p];
    const float3 n = f3(Pl.nf[0], Pl.nf[1], Pl.nf[2]);
    float3 A0, A1;
    edge_ends(fa, A0, A1);
    for (int w0 = 0; w0 < a.nw; w0 += 32) {
      const int w2 = w0 + lane;
      bool keep = false;
      if (w2 < a.nw && w2 != w1) {
        const WedgeF fb = wedge_mirror32(a.wf[w2], n, Pl.cf);
        float3 B0, B1;
        edge_ends(fb, B0, B1);
        const float m = fmaxf(pre_margin_m(A0), pre_margin_m(A1));
        keep = edge_sees(fa, fb, m) && edge_sees(fb, fa, m) && shadow_meets(fa, T, B0, B1);
        if (keep) {
          const float mg = 0.1f + 1e-4f * (fabsf(A0.x) + fabsf(A0.y) + fabsf(A0.z) + fa.len + fb.len);
          keep = section_reachable(Pl, A0, A1, B0, B1, mg) && keller_on_edge(fa, true, T, fb, fb, keller_margin(fa, T));
        }
        if (keep) {  // the exact stage's FP64 rules on the group plane's image
          const Wedge &A = a.wedges[w1], &B = a.wedges[w2];
          const d3w n64 = D3(Pl.n[0], Pl.n[1], Pl.n[2]);
          const Wedge Bm = wedge_mirror64(B, n64, Pl.c);
          keep = !edge_in_plane(A, n64, Pl.c) && !edge_in_plane(B, n64, Pl.c) && !share_vertex(A, Bm) &&
                 !collinear_edges(A, Bm) && !in_face_plane(A, Bm) && !in_face_plane(Bm, A);
        }
      }
      const unsigned mk = __ballot_sync(0xffffffffu, keep);
      if (!mk) continue;
      unsigned at = 0;
      if (lane == 0) at = atomicAdd(&a.ctr->n_dpair, (unsigned)__popc(mk));
      at = __shfl_sync(0xffffffffu, at, 0) + __popc(mk & ((1u << lane) - 1u));
      if (keep) {
        if (at < a.dseq2_cap) a.dseq2[at] = make_int4(t, w1, w2, -2 - p);
        else atomicOr(&a.ctr->err, ERR_DIFF_OVERFLOW);
      }
    }
  }
}

// Triples (w1, w2, w3) from the pairs: (w2, w3) in the relation, w3 not w1,
// and a Keller point on w2 possible between edges 1 and 3 (keller_on_edge).
__global__ void __launch_bounds__(256) k_diff_triples(PathArgs a) {
  const long nw = a.nw;
  const long np = (long)min(a.ctr->n_dpair, a.dseq2_cap), total = np * nw;
  const int lane = threadIdx.x & 31;
  const long stride = (long)gridDim.x * blockDim.x;
  for (long base = (long)blockIdx.x * blockDim.x + (threadIdx.x & ~31); base < total; base += stride) {
    long idx = base + lane;
    bool keep = false;
    int4 pr = make_int4(0, 0, 0, -1);
    int w3 = 0;
    if (idx < total) {
      long p = idx / nw;
      w3 = (int)(idx - p * nw);
      pr = a.dseq2[p];
      size_t bit = (size_t)pr.z * nw + w3;
      keep = pr.w == -1 && w3 != pr.y && ((a.drel[bit >> 5] >> (bit & 31)) & 1u);
      if (keep) {  // the Keller point on the middle edge between the other two
        const WedgeF f2 = a.wf[pr.z];
        keep = keller_on_edge(f2, false, f2.p0, a.wf[pr.y], a.wf[w3], keller_margin(f2, f2.p0));
      }
    }
    unsigned mk = __ballot_sync(0xffffffffu, keep);
    if (!mk) continue;
    unsigned at = 0;
    if (lane == 0) at = atomicAdd(&a.ctr->n_dtrip, (unsigned)__popc(mk));
    at = __shfl_sync(0xffffffffu, at, 0) + __popc(mk & ((1u << lane) - 1u));
    if (keep) {
      if (at < a.dseq3_cap) a.dseq3[at] = make_int4(pr.x, pr.y, pr.z, w3);
      else atomicOr(&a.ctr->err, ERR_DIFF_OVERFLOW);
    }
  }
}

// FP32 Keller points of a chain (the pre-test's estimate): Newton's method
// as in keller_chain, in FP32, from the edges' midpoints. Returns true when
// the cosine mismatch fell below 2e-6 at every edge, or a full Newton step
// would move no point by more than step_tol (metres).
// The iterates may leave the edges: where the length is nearly flat (legs of
// 200 to 2000 m along a road) only the converged point shows how far off its
// edge it lies. Held within 4 m of the edges and cut by convexity instead, a
// highway's chains of two with every reflection left 145,370 candidates for
// the FP64 stage, not 59,700 (24.0 ms a frame, so 20.0), three wedges on a
// 1 km road 13,831, not 126, and the 8 x 8 city 432, not 307 (1446, so 1246 us).
__device__ __forceinline__ float chain_len32(const WedgeF* W, int m, float3 T, float3 R, const float* t) {
  float3 prev = T;
  float L = 0.0f;
  for (int i = 0; i < m; ++i) {
    float3 q = edge_point(W[i], t[i]);
    float3 d = f3(q.x - prev.x, q.y - prev.y, q.z - prev.z);
    L += sqrtf(fdot3(d, d));
    prev = q;
  }
  float3 d = f3(R.x - prev.x, R.y - prev.y, R.z - prev.z);
  return L + sqrtf(fdot3(d, d));
}
__device__ bool keller32(const WedgeF* W, int m, float3 T, float3 R, float* t, float step_tol) {
  for (int i = 0; i < m; ++i) t[i] = 0.5f * W[i].len;
  float Lc = chain_len32(W, m, T, R, t);
  for (int it = 0; it < 30; ++it) {
    float3 X[5];
    X[0] = T;
    for (int i = 0; i < m; ++i) X[i + 1] = edge_point(W[i], t[i]);
    X[m + 1] = R;
    float g[3] = {0.0f, 0.0f, 0.0f}, H[3][3] = {{0.0f, 0.0f, 0.0f}, {0.0f, 0.0f, 0.0f}, {0.0f, 0.0f, 0.0f}};
    for (int j = 0; j <= m; ++j) {
      float3 d = f3(X[j + 1].x - X[j].x, X[j + 1].y - X[j].y, X[j + 1].z - X[j].z);
      float l = sqrtf(fdot3(d, d));
      if (!(l > 0.0f)) return false;
      float3 u = f3(d.x / l, d.y / l, d.z / l);
      int ia = j - 1, ib = j;
      float ca = ia >= 0 ? fdot3(W[ia].e, u) : 0.0f, cb = ib < m ? fdot3(W[ib].e, u) : 0.0f;
      if (ib < m) {
        g[ib] += cb;
        H[ib][ib] += (1.0f - cb * cb) / l;
      }
      if (ia >= 0) {
        g[ia] -= ca;
        H[ia][ia] += (1.0f - ca * ca) / l;
      }
      if (ia >= 0 && ib < m) {
        float h = -(fdot3(W[ia].e, W[ib].e) - ca * cb) / l;
        H[ia][ib] += h;
        H[ib][ia] += h;
      }
    }
    float gmax = 0.0f;
    for (int i = 0; i < m; ++i) gmax = fmaxf(gmax, fabsf(g[i]));
    if (gmax < 2e-6f) return true;
    float A[3][4], dx[3];
    for (int i = 0; i < m; ++i) {
      for (int j = 0; j < m; ++j) A[i][j] = H[i][j];
      A[i][m] = -g[i];
    }
    for (int c = 0; c < m; ++c) {
      int piv = c;
      for (int r = c + 1; r < m; ++r)
        if (fabsf(A[r][c]) > fabsf(A[piv][c])) piv = r;
      if (!(fabsf(A[piv][c]) > 1e-30f)) return false;
      if (piv != c)
        for (int j = 0; j <= m; ++j) {
          float x = A[c][j];
          A[c][j] = A[piv][j];
          A[piv][j] = x;
        }
      for (int r = c + 1; r < m; ++r) {
        float f = A[r][c] / A[c][c];
        for (int j = c; j <= m; ++j) A[r][j] -= f * A[c][j];
      }
    }
    for (int i = m - 1; i >= 0; --i) {
      float v = A[i][m];
      for (int j = i + 1; j < m; ++j) v -= A[i][j] * dx[j];
      dx[i] = v / A[i][i];
    }
    float dfull = 0.0f;
    for (int i = 0; i < m; ++i) dfull = fmaxf(dfull, fabsf(dx[i]));
    float step = 1.0f, tn[3] = {t[0], t[1], t[2]};
    bool moved = false;
    for (int q = 0; q < 30; ++q) {
      for (int i = 0; i < m; ++i) tn[i] = t[i] + step * dx[i];
      float Ln = chain_len32(W, m, T, R, tn);
      if (Ln <= Lc * (1.0f + 1e-6f)) {
        Lc = fminf(Lc, Ln);
        moved = true;
        break;
      }
      step *= 0.5f;
    }
    if (!moved) return gmax < 1e-4f;
    for (int i = 0; i < m; ++i) t[i] = tn[i];
    // the full Newton step (the quadratic model's distance to the
    // stationary point) below step_tol: close enough for the margins
    if (dfull < step_tol) return true;
  }
  return false;
}

// Position margin of the FP32 Keller estimate: 5 cm plus 1e-5 of the
// coordinates' size (FP32 rounding of the geometry and of the solve).
__device__ __forceinline__ float chain_margin(float3 T, float3 R) {
  return 0.05f + 1e-5f * (fabsf(T.x) + fabsf(T.y) + fabsf(T.z) + fabsf(R.x) + fabsf(R.y) + fabsf(R.z));
}

// Is the leg o -> o + dv certainly blocked, whatever its true position within
// `delta` of this one? Only a triangle (other than ex0 .. ex3) that the leg
// crosses strictly inside counts: the crossing must lie within the leg's
// occlusion range (eps_occ, 1 - eps_occ) and at least mu from every edge of
// the triangle in its plane, mu = delta (1 + 1/|cos|) + FP32 slack, |cos|
// the leg's angle to the triangle's normal: a leg displaced by delta moves
// its crossing by at most that much. So the exact leg (FP32 any-hit of the
// FP64 points) is blocked too, and the chain is rejected either way. An
// overflow of the stack or of the visit limit answers "not certain".
__device__ __noinline__ bool leg_surely_blocked(const Bvh& bvh, float3 o, float3 dv, float delta, float eps_occ, int ex0,
                                   int ex1, int ex2, int ex3, TStack& st) {
  const float dl = sqrtf(fdot3(dv, dv));
  if (!(dl > 0.0f)) return false;
  const float slack = 2e-3f + 1e-6f * (fabsf(o.x) + fabsf(o.y) + fabsf(o.z) + dl);
  RayPre rp = ray_pre(o, dv);
  st.reset();
  if (bvh.root1 != kEmpty && !st.push(bvh.root1)) return false;
  int cur = bvh.root0;
  for (int visits = 0;; ++visits) {
    if (visits > bvh.max_visits) return false;
    if (cur == kEmpty) {
      if (st.empty()) break;
      cur = st.pop();
      continue;
    }
    if (cur >= 0) {
      const float4* n = bvh.nodes + 4 * (size_t)DCEM_IDX(cur, bvh.nnodes);
      float4 n0 = __ldg(n), n1 = __ldg(n + 1), n2 = __ldg(n + 2), n3 = __ldg(n + 3);
      float tn0, tn1;
      bool h0 = slab(rp, n0.x, n0.y, n0.z, n0.w, n2.x, n2.y, 1.0f, tn0);
      bool h1 = slab(rp, n1.x, n1.y, n1.z, n1.w, n2.z, n2.w, 1.0f, tn1);
      int c0 = __float_as_int(n3.x), c1 = __float_as_int(n3.y);
      if (h0 && h1) {
        if (!st.push(c1)) return false;
        cur = c0;
      } else {
        cur = h0 ? c0 : h1 ? c1 : kEmpty;
      }
      continue;
    }
    float3 v0, v1, v2;
    int id;
    load_tri(bvh.tris, DCEM_IDX(~cur, bvh.ntris), v0, v1, v2, id);
    cur = kEmpty;
    if (id == ex0 || id == ex1 || id == ex2 || id == ex3) continue;
    float3 e01 = f3(v1.x - v0.x, v1.y - v0.y, v1.z - v0.z), e12 = f3(v2.x - v1.x, v2.y - v1.y, v2.z - v1.z);
    float3 e20 = f3(v0.x - v2.x, v0.y - v2.y, v0.z - v2.z);
    float3 nv = cross3(e01, f3(-e20.x, -e20.y, -e20.z));
    float nn = sqrtf(fdot3(nv, nv)), dn = fdot3(dv, nv);
    if (!(fabsf(dn) > 1e-4f * dl * nn)) continue;  // nearly parallel: not certain
    float u = fdot3(f3(v0.x - o.x, v0.y - o.y, v0.z - o.z), nv) / dn;
    float mu = delta * (1.0f + dl * nn / fabsf(dn)) + slack;
    float nu = mu / dl;
    if (!(u > eps_occ + nu && u < 1.0f - eps_occ - nu)) continue;
    float3 H = f3(o.x + dv.x * u, o.y + dv.y * u, o.z + dv.z * u);
    float d0 = fdot3(cross3(e01, f3(H.x - v0.x, H.y - v0.y, H.z - v0.z)), nv) / (sqrtf(fdot3(e01, e01)) * nn);
    float d1 = fdot3(cross3(e12, f3(H.x - v1.x, H.y - v1.y, H.z - v1.z)), nv) / (sqrtf(fdot3(e12, e12)) * nn);
    float d2 = fdot3(cross3(e20, f3(H.x - v2.x, H.y - v2.y, H.z - v2.z)), nv) / (sqrtf(fdot3(e20, e20)) * nn);
    if (fminf(d0, fminf(d1, d2)) > mu) return true;
  }
  return false;
}

// The FP32 estimate of a chain against the FP64 rules, with margins: false
// only when the exact test rejects the chain too -- a Keller point off its
// edge by more than the position margin, or at some wedge a point inside the
// wedge or the shadow rule missed by more than the angle's rounding bound
// plus the angle the position margin subtends at that point's distance from
// the edge.
// *solved: the estimate converged (t then holds it) -- only then can it
// reject anything.
__device__ __noinline__ bool chain_possible(const WedgeF* W, int m, float3 T, float3 R, float* t, bool* solved) {
  float mt = chain_margin(T, R);
  *solved = keller32(W, m, T, R, t, 0.1f * mt);
  if (!*solved) return true;
  float3 X[5];
  X[0] = T;
  for (int i = 0; i < m; ++i) {
    if (t[i] < -mt || t[i] > W[i].len + mt) return false;
    X[i + 1] = edge_point(W[i], t[i]);
  }
  X[m + 1] = R;
  for (int i = 0; i < m; ++i) {
    float a2[2], tl[2];
    bool sure[2];
    for (int q = 0; q < 2; ++q) {
      float r, dist;
      float2 p = wedge_plane(W[i], X[i + 2 * q], r, dist);
      float3 d = f3(p.x * W[i].t0.x + p.y * W[i].y0.x, p.x * W[i].t0.y + p.y * W[i].y0.y,
                    p.x * W[i].t0.z + p.y * W[i].y0.z);
      a2[q] = wedge_angle32(d, W[i].t0, W[i].y0, r, dist, sure[q], tl[q]);
      // points that move with the estimate (the Keller points) carry its margin
      bool moves = q == 0 ? i > 0 : i < m - 1;
      if (moves) {
        if (!(r > 4.0f * mt)) sure[q] = false;
        else tl[q] += 2.0f * mt / r;
      }
    }
    if ((sure[0] && a2[0] > W[i].npi + tl[0]) || (sure[1] && a2[1] > W[i].npi + tl[1])) return false;
    if (sure[0] && sure[1] && fabsf(a2[1] - a2[0]) < 3.14159265f - (tl[0] + tl[1])) return false;
  }
  return true;
}

// Every (sequence, observer): the observer outside the last wedge and some
// point of the previous edge beyond its shadow boundary at the last wedge,
// then the FP32 Keller estimate against the rules, the legs that are real
// (not those to or from an image) against robust occlusion, and, with a
// reflection, its point on the unfolded leg inside the plane's box (5 cm +
// 1e-4 of the distances; as diffract_refl_candidate). Observers: the
// receivers, and with reflector planes their images (rho = nrx + r * nrpr
// + p) for sequences from a real transmitter; a chain has one reflection.
// Stage 1 of k_diff_multi_pre for sequence sq and observer rho: the
// observer outside the last wedge, some point of the previous edge beyond
// its shadow boundary there, and a Keller point on the last edge possible
// between the previous edge and the observer; an image observer's leg from
// the last edge must be able to cross its plane inside the box.
__device__ __forceinline__ bool multi_stage1(const PathArgs& a, int4 sq, bool three, int rho) {
  const bool mid = !three && sq.w <= -2, obs_img = rho >= a.nrx;
  if (!obs_img && !end_sees(a, a.dntx + rho, three ? sq.w : sq.z)) return false;
  if (obs_img && a.vis && !sees_plane(a, a.dntx + (rho - a.nrx) / a.nrpr, (rho - a.nrx) % a.nrpr)) return false;
  WedgeF fl = a.wf[three ? sq.w : sq.z];
  const WedgeF fp = a.wf[three ? sq.z : sq.y];
  float3 R = chain_observer32(a, rho), P, Q;
  if (mid) {  // a reflection between the wedges: w2 and the receiver mirrored
    const RPlane& Pl = a.rplanes[-2 - sq.w];
    const float3 n = f3(Pl.nf[0], Pl.nf[1], Pl.nf[2]);
    fl = wedge_mirror32(fl, n, Pl.cf);
    R = mirror32(R, n, Pl.cf);
  }
  edge_ends(fp, P, Q);
  bool keep = !surely_inside(fl, R) && shadow_meets(fl, R, P, Q) && keller_on_edge(fl, true, R, fp, fp, keller_margin(fl, R));
  if (keep && !mid && obs_img) {  // the leg from the last edge to the image crosses its plane inside the box
    float3 A1, B1;
    edge_ends(fl, A1, B1);
    float mg = 0.1f + 1e-4f * (fabsf(R.x) + fabsf(R.y) + fabsf(R.z) + fl.len);
    keep = plane_reachable(a.rplanes[(rho - a.nrx) % a.nrpr], R, A1, B1, mg);
  }
  return keep;
}

// Stage 1 of a triple depends on its last two wedges and the receiver only,
// and the triples share their last pairs (8 x 8 city: 112k triples, a few
// thousand pairs): one bit per (related pair whose first wedge is the second
// of some pair, receiver), in rows of dobs1_row words. One warp per related
// pair, its lanes over the receivers.
__global__ void __launch_bounds__(256) k_diff_stage1(PathArgs a) {
  const long nw = a.nw, nch = (nw + 31) / 32, nitem = nw * nch;
  const int lane = threadIdx.x & 31;
  const long nwarp = (long)gridDim.x * (blockDim.x >> 5);
  for (long it = (long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); it < nitem; it += nwarp) {
    const int wp = (int)(it / nch), w0 = (int)(it - (long)wp * nch) * 32;
    if (!((a.dsecond[wp >> 5] >> (wp & 31)) & 1u)) continue;
    const long bit = (long)wp * nw + w0 + lane;
    const bool rel = w0 + lane < nw && ((a.drel[bit >> 5] >> (bit & 31)) & 1u);
    for (unsigned rm = __ballot_sync(0xffffffffu, rel); rm; rm &= rm - 1u) {
      const int wl = w0 + __ffs(rm) - 1;
      unsigned* row = a.dobs1 + ((size_t)wp * nw + wl) * a.dobs1_row;
      for (int c = 0; c < a.dobs1_row; ++c) {
        const int r = 32 * c + lane;
        const unsigned m =
            __ballot_sync(0xffffffffu, r < a.nrx && multi_stage1(a, make_int4(0, 0, wp, wl), true, r));
        if (lane == 0) row[c] = m;
      }
    }
  }
}

// Stage 2 for a pair with a reflection between its wedges: the chain over w1
// and w2's image toward the receiver's image (FP32 Keller estimate against
// the rules), the real first and last legs against robust occlusion (the
// last one mirrored back), and the crossing of the unfolded middle leg with
// the plane inside its box.
__device__ __forceinline__ bool mid_stage2(const PathArgs& a, int4 sq, int rho, TStack& st) {
  const RPlane& Pl = a.rplanes[-2 - sq.w];
  const float3 n = f3(Pl.nf[0], Pl.nf[1], Pl.nf[2]);
  WedgeF Wc[2];
  Wc[0] = a.wf[sq.y];
  Wc[1] = wedge_mirror32(a.wf[sq.z], n, Pl.cf);
  const float3 T = chain_source32(a, sq.x), R = chain_observer32(a, rho), Rm = mirror32(R, n, Pl.cf);
  float t[2];
  bool solved;
  bool keep = chain_possible(Wc, 2, T, Rm, t, &solved);
  if (!keep || !solved) return keep;
  const float delta = chain_margin(T, Rm);
  const float3 Q1 = edge_point(Wc[0], t[0]), Q2m = edge_point(Wc[1], t[1]), Q2 = mirror32(Q2m, n, Pl.cf);
  const Wedge &A = a.wedges[sq.y], &B = a.wedges[sq.z];
  float3 dv = f3(Q1.x - T.x, Q1.y - T.y, Q1.z - T.z);
  if (leg_surely_blocked(a.bvh, T, dv, delta, a.eps_occ, -1, -1, A.ta, A.tb, st)) return false;
  dv = f3(R.x - Q2.x, R.y - Q2.y, R.z - Q2.z);
  if (leg_surely_blocked(a.bvh, Q2, dv, delta, a.eps_occ, B.ta, B.tb, -1, -1, st)) return false;
  dv = f3(Q2m.x - Q1.x, Q2m.y - Q1.y, Q2m.z - Q1.z);
  const float den = fdot3(n, dv), len = sqrtf(fdot3(dv, dv));
  if (fabsf(den) > 1e-6f * len) {
    const float tt = (Pl.cf - fdot3(n, Q1)) / den;
    const float mt = (0.05f + delta + 1e-4f * (len + sqrtf(fdot3(Q1, Q1)))) / len;
    if (tt < -mt || tt > 1.0f + mt) return false;
    const float3 Xp = f3(Q1.x + tt * dv.x, Q1.y + tt * dv.y, Q1.z + tt * dv.z);
    const float mb = 0.05f + delta + 1e-4f * (len + sqrtf(fdot3(Xp, Xp)));
    if (Xp.x < Pl.box[0] - mb || Xp.y < Pl.box[1] - mb || Xp.z < Pl.box[2] - mb || Xp.x > Pl.box[3] + mb ||
        Xp.y > Pl.box[4] + mb || Xp.z > Pl.box[5] + mb)
      return false;
    // the two real legs through the reflection point (a crossing near a
    // leg's end, as the reflector's own at P, does not count)
    float3 d1 = f3(Xp.x - Q1.x, Xp.y - Q1.y, Xp.z - Q1.z), d2 = f3(Q2.x - Xp.x, Q2.y - Xp.y, Q2.z - Xp.z);
    if (leg_surely_blocked(a.bvh, Q1, d1, delta, a.eps_occ, A.ta, A.tb, -1, -1, st) ||
        leg_surely_blocked(a.bvh, Xp, d2, delta, a.eps_occ, -1, -1, B.ta, B.tb, st))
      return false;
  }
  return true;
}

// Stage 2 for an index past stage 1: the FP32 Keller estimate against the
// rules, the real legs against robust occlusion, and with a reflection its
// point on the unfolded leg inside the plane's box.
__device__ __forceinline__ bool multi_stage2(const PathArgs& a, long idx, long n2, long nobs, TStack& st) {
  const long e = idx / nobs;
  const int rho = (int)(idx - e * nobs);
  const bool three = e >= n2;
  const long ei = three ? e - n2 : e;
  const int4 sq = three ? a.dseq3[ei] : a.dseq2[ei];
  if (!three && sq.w <= -2) return mid_stage2(a, sq, rho, st);
  const bool src_img = sq.x >= a.dntx, obs_img = rho >= a.nrx;
  const int wl = three ? sq.w : sq.z, wp = three ? sq.z : sq.y;
  WedgeF Wc[3];
  Wc[0] = a.wf[sq.y];
  Wc[1] = a.wf[three ? wp : wl];  // order 2: (w1, last); order 3: (w1, previous, last)
  Wc[2] = a.wf[wl];
  const int m = three ? 3 : 2;
  const float3 T = chain_source32(a, sq.x), R = chain_observer32(a, rho);
  float t[3];
  bool solved;
  bool keep = chain_possible(Wc, m, T, R, t, &solved);
  if (keep && solved) {
    const int w[3] = {sq.y, sq.z, sq.w};
    const float delta = chain_margin(T, R);
    float3 X[5];
    X[0] = T;
    for (int i = 0; i < m; ++i) X[i + 1] = edge_point(Wc[i], t[i]);
    X[m + 1] = R;
    // a leg certainly blocked rejects the chain (legs to or from an
    // image are not real: the reflection breaks them)
    for (int q = 0; keep && q <= m; ++q) {
      if ((q == 0 && src_img) || (q == m && obs_img)) continue;
      const Wedge* A = q >= 1 ? &a.wedges[w[q - 1]] : nullptr;
      const Wedge* B = q < m ? &a.wedges[w[q]] : nullptr;
      float3 dv = f3(X[q + 1].x - X[q].x, X[q + 1].y - X[q].y, X[q + 1].z - X[q].z);
      if (leg_surely_blocked(a.bvh, X[q], dv, delta, a.eps_occ, A ? A->ta : -1, A ? A->tb : -1,
                             B ? B->ta : -1, B ? B->tb : -1, st))
        keep = false;
    }
    if (keep && (src_img || obs_img)) {  // the reflection point within the plane's box
      const RPlane& Pl = a.rplanes[src_img ? (sq.x - a.dntx) % a.nrpr : (rho - a.nrx) % a.nrpr];
      const float3 n = f3(Pl.nf[0], Pl.nf[1], Pl.nf[2]);
      const float3 a0 = src_img ? X[0] : X[m], a1 = src_img ? X[1] : X[m + 1];
      const float3 dv = f3(a1.x - a0.x, a1.y - a0.y, a1.z - a0.z);
      const float den = fdot3(n, dv), len = sqrtf(fdot3(dv, dv));
      if (fabsf(den) > 1e-6f * len) {
        float tt = (Pl.cf - fdot3(n, a0)) / den;
        float mt = (0.05f + delta + 1e-4f * (len + sqrtf(fdot3(a0, a0)))) / len;
        if (tt < -mt || tt > 1.0f + mt) keep = false;
        float3 Xp = f3(a0.x + tt * dv.x, a0.y + tt * dv.y, a0.z + tt * dv.z);
        float mb = 0.05f + delta + 1e-4f * (len + sqrtf(fdot3(Xp, Xp)));
        if (Xp.x < Pl.box[0] - mb || Xp.y < Pl.box[1] - mb || Xp.z < Pl.box[2] - mb ||
            Xp.x > Pl.box[3] + mb || Xp.y > Pl.box[4] + mb || Xp.z > Pl.box[5] + mb)
          keep = false;
        if (keep) {  // the two real legs through the reflection point (its own crossing is at their end)
          const float4 ev = src_img ? a.txs[(sq.x - a.dntx) / a.nrpr] : a.rx[(rho - a.nrx) / a.nrpr];
          const float3 E = f3(ev.x, ev.y, ev.z);        // the real transmitter or receiver
          const float3 Qn = src_img ? X[1] : X[m];     // the diffraction point next to the reflection
          const Wedge& Wn = a.wedges[src_img ? w[0] : w[m - 1]];
          const float3 d1 = f3(Xp.x - E.x, Xp.y - E.y, Xp.z - E.z), d2 = f3(Qn.x - Xp.x, Qn.y - Xp.y, Qn.z - Xp.z);
          if (leg_surely_blocked(a.bvh, E, d1, delta, a.eps_occ, -1, -1, -1, -1, st) ||
              leg_surely_blocked(a.bvh, Xp, d2, delta, a.eps_occ, -1, -1, Wn.ta, Wn.tb, st))
            keep = false;
        }
      }
    }
  }
  return keep;
}

// One warp per sequence, its lanes over the observers: every (sequence,
// observer) through stage 1; the indices (sequence * nobs + observer) that
// pass wait in a per-warp queue and go through stage 2 (the Newton estimate,
// the legs) 32 at a time, so that the costly stage runs on full warps.
// Observers: the receivers, and with reflector planes their images (rho =
// nrx + r * nrpr + p) for sequences from a real transmitter (a chain has one
// reflection: a sequence from an image sees the receivers only).
__global__ void __launch_bounds__(256) k_diff_multi_pre(PathArgs a) {
  extern __shared__ int sstk[];
  __shared__ long wq[8][64];
  TStack st;
  bind_stack(st, sstk, kStackTrace);
  const long n2 = a.diff_order >= 2 ? (long)min(a.ctr->n_dpair, a.dseq2_cap) : 0;
  const long n3 = a.diff_order >= 3 ? (long)min(a.ctr->n_dtrip, a.dseq3_cap) : 0;
  const long nobs = (long)a.nrx * (1 + a.nrpr);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  // work items: (sequence, run of kObsRun observers), so that the sequences
  // from a real transmitter, which see every observer, split over warps
  constexpr long kObsRun = 512;
  const long nrun = (nobs + kObsRun - 1) / kObsRun, nitem = (n2 + n3) * nrun;
  const long nwarps = (long)gridDim.x * (blockDim.x >> 5);
  long item = (long)blockIdx.x * (blockDim.x >> 5) + wid - nwarps;
  long e = 0, r0 = 0, r1 = 0;  // the item's sequence and observer range (warp-uniform)
  int4 sq = make_int4(0, 0, 0, 0);
  int qn = 0;                  // queued indices of this warp (warp-uniform)
  for (;;) {
    while (r0 >= r1) {  // the next item with observers
      item += nwarps;
      if (item >= nitem) break;
      e = item / nrun;
      sq = e >= n2 ? a.dseq3[e - n2] : a.dseq2[e];
      const long nob = sq.x >= a.dntx || (e < n2 && sq.w <= -2) ? a.nrx : nobs;
      r0 = (item - e * nrun) * kObsRun;
      r1 = min(r0 + kObsRun, nob);
    }
    const bool more = item < nitem;
    if (more) {
      const long rho = r0 + lane;
      bool pass = rho < r1;
      if (pass) {
        if (a.dobs1 && e >= n2 && rho < a.nrx)
          pass = (a.dobs1[((size_t)sq.z * a.nw + sq.w) * a.dobs1_row + (rho >> 5)] >> (rho & 31)) & 1u;
        else
          pass = multi_stage1(a, sq, e >= n2, (int)rho);
      }
      const unsigned mk = __ballot_sync(0xffffffffu, pass);
      if (pass) wq[wid][qn + __popc(mk & ((1u << lane) - 1u))] = e * nobs + rho;
      qn += __popc(mk);
      __syncwarp();
      r0 += 32;
    }
    while (qn >= 32 || (!more && qn > 0)) {
      const int nn = min(qn, 32);
      const long idx = lane < nn ? wq[wid][qn - nn + lane] : -1;
      __syncwarp();
      qn -= nn;
      const bool keep = idx >= 0 && multi_stage2(a, idx, n2, nobs, st);
      const unsigned mk = __ballot_sync(0xffffffffu, keep);
      if (!mk) continue;
      unsigned at = 0;
      if (lane == 0) at = atomicAdd(&a.ctr->n_dsurv, (unsigned)__popc(mk));
      at = __shfl_sync(0xffffffffu, at, 0) + __popc(mk & ((1u << lane) - 1u));
      if (keep) {
        const bool three = idx >= n2 * nobs;
        const unsigned long long code =
            (unsigned long long)(three ? idx - n2 * nobs : idx) | (three ? kMulti3 : kMulti2);
        if (at < a.dsurv_cap) a.dsurv[at] = code;
        else atomicOr(&a.ctr->err, ERR_DIFF_OVERFLOW);
      }
    }
    if (!more) break;
  }
}

// Unfolded length of the chain with edge parameters t.
__device__ __forceinline__ double chain_len(const Wedge* const* E, int m, d3w T, d3w R, const double* t) {
  d3w prev = T;
  double L = 0.0;
  for (int i = 0; i < m; ++i) {
    d3w q = D3(E[i]->p0[0], E[i]->p0[1], E[i]->p0[2]) + D3(E[i]->e[0], E[i]->e[1], E[i]->e[2]) * t[i];
    d3w d = q - prev;
    L += sqrt(dotw(d, d));
    prev = q;
  }
  d3w d = R - prev;
  return L + sqrt(dotw(d, d));
}

// Where Newton's method starts (the length is convex, so the start decides
// the number of steps, not the result): one wedge's closed form, a chain's
// FP32 Keller points where that estimate converges, else the midpoints. An
// FP64 step costs some two thousand cycles of dependent operations; from the
// midpoints a chain takes 5 to 50, from these starts two or three.
__device__ __forceinline__ void keller_start(const Wedge* const* E, int m, d3w T, d3w R, double* t) {
  if (m == 1) {
    const d3w e = D3(E[0]->e[0], E[0]->e[1], E[0]->e[2]), p0 = D3(E[0]->p0[0], E[0]->p0[1], E[0]->p0[2]);
    const d3w dt = T - p0, dr = R - p0;
    const double zt = dotw(dt, e), zr = dotw(dr, e);
    const d3w pt = dt - e * zt, pr = dr - e * zr;
    const double rt = sqrt(dotw(pt, pt)), rr = sqrt(dotw(pr, pr));
    t[0] = rt + rr > 0.0 ? zt + (zr - zt) * rt / (rt + rr) : 0.5 * E[0]->len;
    return;
  }
  WedgeF W[3];
  float tf[3];
  for (int i = 0; i < m; ++i) W[i] = wedge_f(*E[i]);
  const bool ok =
      keller32(W, m, f3((float)T.x, (float)T.y, (float)T.z), f3((float)R.x, (float)R.y, (float)R.z), tf, 1e-3f);
  for (int i = 0; i < m; ++i) t[i] = ok ? (double)tf[i] : 0.5 * E[i]->len;
}

// Keller points: the stationary point (the minimum: the length is convex in
// t) of the unfolded length over the edge parameters, by Newton's method
// from keller_start (at most 50 steps), a step that does not
// shorten the chain halved (at most 40 times) until the cosine mismatch is
// below 1e-8 or the Newton decrement below 1e-15 of the length, full steps
// after that; converged when every edge's mismatch is below 1e-12. A leg shorter than kLegMin stops it: the
// minimum is then at a kink of the length (consecutive edge lines meet),
// where Keller's law has no solution.
constexpr double kLegMin = 1e-6;
__device__ bool keller_chain(const Wedge* const* E, int m, d3w T, d3w R, double* t) {
  keller_start(E, m, T, R, t);
  double Lc = chain_len(E, m, T, R, t);
  for (int it = 0; it < 50; ++it) {
    d3w X[5];
    X[0] = T;
    for (int i = 0; i < m; ++i)
      X[i + 1] = D3(E[i]->p0[0], E[i]->p0[1], E[i]->p0[2]) + D3(E[i]->e[0], E[i]->e[1], E[i]->e[2]) * t[i];
    X[m + 1] = R;
    double g[3] = {0.0, 0.0, 0.0}, H[3][3] = {{0.0, 0.0, 0.0}, {0.0, 0.0, 0.0}, {0.0, 0.0, 0.0}};
    for (int j = 0; j <= m; ++j) {
      d3w d = X[j + 1] - X[j];
      double l = sqrt(dotw(d, d));
      if (!(l > kLegMin)) return false;
      d3w u = d * (1.0 / l);
      int ia = j - 1, ib = j;
      d3w ea = ia >= 0 ? D3(E[ia]->e[0], E[ia]->e[1], E[ia]->e[2]) : D3(0, 0, 0);
      d3w eb = ib < m ? D3(E[ib]->e[0], E[ib]->e[1], E[ib]->e[2]) : D3(0, 0, 0);
      double ca = dotw(ea, u), cb = dotw(eb, u);
      if (ib < m) {
        g[ib] += cb;
        H[ib][ib] += (1.0 - cb * cb) / l;
      }
      if (ia >= 0) {
        g[ia] -= ca;
        H[ia][ia] += (1.0 - ca * ca) / l;
      }
      if (ia >= 0 && ib < m) {
        double h = -(dotw(ea, eb) - ca * cb) / l;
        H[ia][ib] += h;
        H[ib][ia] += h;
      }
    }
    double gmax = 0.0, cut = 0.0;
    for (int i = 0; i < m; ++i) {
      gmax = fmax(gmax, fabs(g[i]));
      cut += fmin(-g[i] * t[i], g[i] * (E[i]->len - t[i]));
    }
    if (gmax < 1e-12) return true;
    // convex: at any y the length is at least L(t) + g.(y - t), so when that
    // exceeds L(t) for every y on the edges (by more than rounding), the
    // minimum lies off an edge and the chain is rejected (kinks off the edges
    // otherwise take the 50 steps of 40 halvings: 4.1M cycles for one chain)
    if (cut > 1e-9 * Lc) return false;
    // H dx = -g by elimination with partial pivoting
    double A[3][4], dx[3];
    for (int i = 0; i < m; ++i) {
      for (int j = 0; j < m; ++j) A[i][j] = H[i][j];
      A[i][m] = -g[i];
    }
    for (int c = 0; c < m; ++c) {
      int piv = c;
      for (int r = c + 1; r < m; ++r)
        if (fabs(A[r][c]) > fabs(A[piv][c])) piv = r;
      if (!(fabs(A[piv][c]) > 1e-300)) return false;
      if (piv != c)
        for (int j = 0; j <= m; ++j) {
          double x = A[c][j];
          A[c][j] = A[piv][j];
          A[piv][j] = x;
        }
      for (int r = c + 1; r < m; ++r) {
        double f = A[r][c] / A[c][c];
        for (int j = c; j <= m; ++j) A[r][j] -= f * A[c][j];
      }
    }
    for (int i = m - 1; i >= 0; --i) {
      double v = A[i][m];
      for (int j = i + 1; j < m; ++j) v -= A[i][j] * dx[j];
      dx[i] = v / A[i][i];
    }
    // near the minimum the full step: the length it saves (the Newton
    // decrement, -g.dx / 2) is below the length's rounding there, so a
    // comparison of lengths cannot judge it -- a mismatch below 1e-8, or a
    // decrement below 1e-15 of the length (long chains reach that floor at
    // larger mismatches)
    double gdx = 0.0;
    for (int i = 0; i < m; ++i) gdx += g[i] * dx[i];
    const bool floor = gmax < 1e-8 || fabs(gdx) <= 2e-15 * Lc;
    double step = 1.0, tn[3] = {0.0, 0.0, 0.0};
    for (int q = 0; q < 40; ++q) {
      for (int i = 0; i < m; ++i) tn[i] = t[i] + step * dx[i];
      double Ln = chain_len(E, m, T, R, tn);
      if (Ln <= Lc || floor) {
        Lc = Ln;
        break;
      }
      step *= 0.5;
    }
    double dmax = 0.0;
    for (int i = 0; i < m; ++i) {
      dmax = fmax(dmax, fabs(tn[i] - t[i]));
      t[i] = tn[i];
    }
    if (dmax == 0.0) return gmax < 1e-9;
  }
  return false;
}

// The Keller points of a chain from src to obs and the rules on the
// unfolded chain: every point inside its edge, every leg longer than 1e-9 m,
// at every wedge both neighbours in the exterior and the next point beyond
// the incident shadow boundary of the previous one. X: the chain's points.
__device__ bool chain_geometry(const Wedge* const* E, int m, d3w src, d3w obs, d3w* X, double* ell,
                               double* phip, double* phi) {
  if (wedge_angle(*E[0], src) > E[0]->n * M_PI || wedge_angle(*E[m - 1], obs) > E[m - 1]->n * M_PI) return false;
  double t[3];
  if (!keller_chain(E, m, src, obs, t)) return false;
  X[0] = src;
  for (int i = 0; i < m; ++i) {
    double uq = t[i] / E[i]->len;
    if (!(uq > 0.0 && uq < 1.0)) return false;
    X[i + 1] = D3(E[i]->p0[0], E[i]->p0[1], E[i]->p0[2]) + D3(E[i]->e[0], E[i]->e[1], E[i]->e[2]) * t[i];
  }
  X[m + 1] = obs;
  for (int q = 0; q <= m; ++q) {
    d3w d = X[q + 1] - X[q];
    ell[q] = sqrt(dotw(d, d));
    if (!(ell[q] > 1e-9)) return false;
  }
  for (int i = 0; i < m; ++i) {
    phip[i] = wedge_angle(*E[i], X[i]);
    phi[i] = wedge_angle(*E[i], X[i + 2]);
    const double nn = E[i]->n;
    if (phip[i] > nn * M_PI || phi[i] > nn * M_PI) return false;
    if (!(fabs(phi[i] - phip[i]) > M_PI)) return false;
  }
  return true;
}

// The reflection point of the unfolded leg a0 -> a1 on plane (n, c): false
// when the leg does not cross the plane between its ends.
__device__ __forceinline__ bool leg_plane(d3w a0, d3w a1, d3w n, double c, d3w& P) {
  double den = dotw(n, a1 - a0);
  if (den == 0.0) return false;
  double t = (c - dotw(n, a0)) / den;
  if (!(t > 0.0 && t < 1.0)) return false;
  P = a0 + (a1 - a0) * t;
  return true;
}

// The specular reflection of field E at a triangle with unit normal nj and
// material mj, incoming direction din, outgoing dout: Fresnel TE / TM in the
// bounce basis of k_val_field (s = din x n, p_in = s x din, p_out = s x dout).
__device__ zv3 reflect_field_d(const PathArgs& a, d3w nj, float4 mj, d3w din, d3w dout, zv3 E) {
  double ct = fabs(dotw(din, nj));
  d3w sv = crossw(din, nj);
  double sn = sqrt(dotw(sv, sv));
  if (sn < 1e-12) {
    d3w ax = fabs(nj.x) < 0.9 ? D3(1, 0, 0) : D3(0, 1, 0);
    sv = unitw(crossw(nj, ax));
  } else {
    sv = sv * (1.0 / sn);
  }
  d3w pin = crossw(sv, din), pout = crossw(sv, dout);
  zd gte, gtm;
  fresnel_d(mj, a.freq, ct, gte, gtm);
  zd ts = gte * zvdot(E, sv), tp = gtm * zvdot(E, pin);
  return zv3{ts * sv.x + tp * pout.x, ts * sv.y + tp * pout.y, ts * sv.z + tp * pout.z};
}

// One (sequence, observer) survivor of order m: with an image source or
// observer, the chain is solved on the plane group's image, the member
// triangle j holding the reflection point is found, and everything is
// redone with j's own plane (the oracle takes each static triangle as the
// mirror). Then the Keller points and rules (chain_geometry), the real legs
// (FP32 any-hit; triangle j excluded at the reflection point, the wedges'
// faces at theirs), and the UTD chain: at each wedge the coefficient acts on
// the arriving field in the wedge's edge-fixed bases; the wave behind it has
// a caustic on the edge (radius s along phi^) and one rho_e behind it
// (radius rho_e + s along beta^), rho_e the arriving wavefront's radius of
// curvature along the edge's projection (Euler's formula; the source's
// distance for its spherical wave); spreading sqrt(rho_e / (s (rho_e + s)))
// and distance parameter L = s (rho_e + s) rho_1 rho_2 sin^2 beta_0 /
// (rho_e (rho_1 + s) (rho_2 + s)) (Kouyoumjian & Pathak 1974, straight
// edge), over the unfolded distances (a plane mirror keeps the wavefront's
// radii); the reflection applies Fresnel in the real directions.
// One survivor of a pair with a reflection between its wedges (Sec. III
// steps 3-5): the FP64 chain over w1 and w2's image in the plane toward the
// receiver's image (chain_geometry), the vertex, line and face-plane rules
// on the image, the reflection point where the unfolded middle leg crosses
// the plane, the member triangle holding it and everything again on that
// triangle's own plane; the four real legs (FP32 any-hit; the wedges' faces
// excluded at Q1 and Q2, the triangle at P); then the field: UTD at w1,
// Fresnel at P in the real directions with the wavefront's principal
// directions mirrored, UTD at w2 in the real directions (its angles are
// those about the image). Record: depth 3, {w1 | diffract, triangle,
// w2 | diffract}.
__device__ __noinline__ void diffract_mid(const PathArgs& a, int4 sq, int r, double k, double lam, unsigned& ovf,
                                          TStack& st) {
  const int w1 = sq.y, w2 = sq.z, tx = sq.x;
  const int link = tx * a.nrx + r;
  const Wedge& A = a.wedges[w1];
  const Wedge& B = a.wedges[w2];
  const float4 rxv = a.rx[r], txv = a.txs[tx];
  const d3w T = D3(txv.x, txv.y, txv.z), R = D3(rxv.x, rxv.y, rxv.z);
  const RPlane& G = a.rplanes[-2 - sq.w];
  d3w n = D3(G.n[0], G.n[1], G.n[2]);
  double c = G.c;
  auto mir = [&](d3w x) { return x - n * (2.0 * (dotw(n, x) - c)); };
  int j = -1;
  float4 mj = make_float4(0.f, 0.f, 0.f, 0.f);
  d3w X[4], Pp = D3(0, 0, 0);
  double ell[3], phip[2], phi[2];
  for (int pass = 0; pass < 2; ++pass) {
    const Wedge Bm = wedge_mirror64(B, n, c);  // w2's image in the plane
    if (edge_in_plane(A, n, c) || edge_in_plane(B, n, c)) return;
    if (share_vertex(A, Bm) || collinear_edges(A, Bm) || in_face_plane(A, Bm) || in_face_plane(Bm, A)) return;
    const Wedge* E[2] = {&A, &Bm};
    if (!chain_geometry(E, 2, T, mir(R), X, ell, phip, phi)) return;
    if (!leg_plane(X[1], X[2], n, c, Pp)) return;
    d3w v0, v1, v2;
    if (pass == 0) {  // the member triangle holding P: its own plane next
      const int exw[4] = {A.ta, A.tb, B.ta, B.tb};
      j = member_at(a, G, Pp, exw, 4, v0, v1, v2, mj);
      if (j < 0) return;
      n = unitw(crossw(v1 - v0, v2 - v0));
      c = dotw(n, v0);
    } else {
      tri64(a, j, v0, v1, v2, mj);
      if (!inside_tri64(v0, v1, v2, Pp)) return;
    }
  }
  const d3w Q1 = X[1], Q2 = mir(X[2]);
  // the real legs: two excluded triangles at each point
  const d3w Y[5] = {T, Q1, Pp, Q2, R};
  const int ex[5][2] = {{-1, -1}, {A.ta, A.tb}, {j, j}, {B.ta, B.tb}, {-1, -1}};
  if (legs_occluded(a, Y, ex, 5, ovf, st)) return;
  unsigned fl = 0;
  const d3w u = D3(a.pol.x, a.pol.y, a.pol.z);
  d3w ip = (Q1 - T) * (1.0 / ell[0]);
  double sn, cs;
  sincos(-k * ell[0], &sn, &cs);
  const zd Ei = Z(cs / ell[0], sn / ell[0]);
  const d3w e0 = polw(u, ip, fl);
  zv3 Ev = {Ei * e0.x, Ei * e0.y, Ei * e0.z};
  double rho1 = ell[0], rho2 = ell[0];
  d3w dir1 = D3(0, 0, 0), dir2 = D3(0, 0, 0);
  const d3w din = unitw(Pp - Q1), dout = unitw(Q2 - Pp);
  for (int i = 0; i < 2; ++i) {
    const Wedge& W = i == 0 ? A : B;
    const d3w dd = i == 0 ? din : unitw(R - Q2);
    const double s = ell[i + 1], nn = W.n;
    if (i == 1) {  // the reflection at P; the wavefront's principal directions mirrored
      Ev = reflect_field_d(a, n, mj, din, dout, Ev);
      dir1 = dir1 - n * (2.0 * dotw(dir1, n));
      dir2 = dir2 - n * (2.0 * dotw(dir2, n));
      ip = dout;
    }
    const d3w e = D3(W.e[0], W.e[1], W.e[2]);
    const double beta0 = acos(fmax(-1.0, fmin(1.0, dotw(ip, e))));
    const double sb = sin(beta0);
    const d3w php = unitw(crossw(e, ip)) * -1.0, ph = unitw(crossw(e, dd));
    const d3w bp = crossw(ip, php), bd = crossw(dd, ph);
    double rhoe;
    if (i == 0) rhoe = ell[0];
    else {
      const double c1 = dotw(bp, dir1), c2 = dotw(bp, dir2);
      rhoe = 1.0 / (c1 * c1 / rho1 + c2 * c2 / rho2);
    }
    const double L = s * (rhoe + s) * rho1 * rho2 * sb * sb / (rhoe * (rho1 + s) * (rho2 + s));
    const float4 ma =
        a.mats[__float_as_int(a.tris[3 * (size_t)DCEM_IDX(a.slot_of_id[DCEM_IDX(W.ta, a.bvh.ntris)], a.bvh.ntris) + 1].w)];
    const float4 mb =
        a.mats[__float_as_int(a.tris[3 * (size_t)DCEM_IDX(a.slot_of_id[DCEM_IDX(W.tb, a.bvh.ntris)], a.bvh.ntris) + 1].w)];
    zd r0s, r0h, rns, rnh;
    fresnel_faces(ma, fabs(sin(phip[i])), mb, fabs(sin(nn * M_PI - phi[i])), a.freq, r0s, r0h, rns, rnh);
    const UtdParts up = utd_parts(nn, phi[i], phip[i], beta0, L, k, fl);
    const zd Ds = utd_coeff(up, r0s, rns), Dh = utd_coeff(up, r0h, rnh);
    sincos(-k * s, &sn, &cs);
    const zd Am = Z(cs, sn) * sqrt(rhoe / (s * (rhoe + s)));
    const zd cb = Ds * zvdot(Ev, bp) * Am * -1.0, cp = Dh * zvdot(Ev, php) * Am * -1.0;
    Ev = zv3{cb * bd.x + cp * ph.x, cb * bd.y + cp * ph.y, cb * bd.z + cp * ph.z};
    rho1 = s;
    dir1 = ph;
    rho2 = rhoe + s;
    dir2 = bd;
    ip = dd;
  }
  const d3w prx = polw(u, ip * -1.0, fl);
  const zd amp = zvdot(Ev, prx) * (lam / (4.0 * M_PI));
  if (diff_lane() != 0) return;  // one lane of the group writes the record
  unsigned uu = atomicAdd(&a.ctr->n_unique, 1u);
  if (uu >= a.ucap) {
    atomicOr(&a.ctr->err, ERR_UNIQUE_OVERFLOW);
    return;
  }
  const int ids[3] = {w1 | kDiffBit, j, w2 | kDiffBit};
  PathRec rec;
  rec.key = seq_key(r, 3, [&](int q) { return ids[q]; });
  rec.rx = link;
  rec.depth = 3;
  rec.ray = -1;
  rec.flags = fl;
  rec.valid = 1;
  rec.pad = 0;
  rec.len = ell[0] + ell[1] + ell[2];
  rec.amp_re = amp.re;
  rec.amp_im = amp.im;
  for (int q = 0; q < kMaxRefl; ++q) {
    rec.tri[q] = q < 3 ? ids[q] : -1;
    rec.pts[q][0] = rec.pts[q][1] = rec.pts[q][2] = 0.0f;
  }
  for (int q = 0; q < 3; ++q) {
    rec.pts[q][0] = (float)Y[q + 1].x;
    rec.pts[q][1] = (float)Y[q + 1].y;
    rec.pts[q][2] = (float)Y[q + 1].z;
  }
  a.prec[uu] = rec;
  unsigned pos = atomicAdd(&a.bucket_cnt[link], 1u);
  if (pos < (unsigned)a.bucket_cap) a.bucket[(size_t)link * a.bucket_cap + pos] = (int)uu;
  else atomicOr(&a.ctr->err, ERR_BUCKET_OVERFLOW);
  atomicAdd(&a.ctr->n_valid, 1u);
}

__device__ __noinline__ void diffract_multi(const PathArgs& a, unsigned long long code, double k, double lam,
                                            unsigned& ovf, TStack& st) {
  const bool three = (code >> kKindShift) == 3ull;
  const int m = three ? 3 : 2;
  const unsigned long long c = code & ((1ull << kKindShift) - 1ull);
  const unsigned long long nobs = (unsigned long long)a.nrx * (1 + a.nrpr);
  const long ei = (long)(c / nobs);
  const int rho = (int)(c - (unsigned long long)ei * nobs);
  const int4 sq = three ? a.dseq3[ei] : a.dseq2[ei];
  if (!three && sq.w <= -2) {  // a reflection between the two wedges
    if (rho < a.nrx) diffract_mid(a, sq, rho, k, lam, ovf, st);
    return;
  }
  const int w[3] = {sq.y, sq.z, sq.w};
  const bool first = sq.x >= a.dntx, last = rho >= a.nrx;  // a reflection before / after the chain
  if (first && last) return;
  const int tx = first ? (sq.x - a.dntx) / a.nrpr : sq.x, r = last ? (rho - a.nrx) / a.nrpr : rho;
  const int pl = first ? (sq.x - a.dntx) % a.nrpr : last ? (rho - a.nrx) % a.nrpr : -1;
  const int link = tx * a.nrx + r;
  const Wedge* E[3] = {&a.wedges[w[0]], &a.wedges[w[1]], three ? &a.wedges[w[2]] : &a.wedges[w[1]]};
  float4 rxv = a.rx[r], txv = a.txs[tx];
  const d3w T = D3(txv.x, txv.y, txv.z), R = D3(rxv.x, rxv.y, rxv.z);
  d3w X[5], Pp = D3(0, 0, 0), nj = D3(0, 0, 0);
  double ell[4], phip[3], phi[3];
  int j = -1;
  float4 mj = make_float4(0.f, 0.f, 0.f, 0.f);
  if (pl < 0) {
    if (!chain_geometry(E, m, T, R, X, ell, phip, phi)) return;
  } else {
    const RPlane Pg = a.rplanes[pl];
    d3w n = D3(Pg.n[0], Pg.n[1], Pg.n[2]);
    double cg = Pg.c;
    for (int pass = 0; pass < 2; ++pass) {
      d3w src = first ? T - n * (2.0 * (dotw(n, T) - cg)) : T;
      d3w obs = last ? R - n * (2.0 * (dotw(n, R) - cg)) : R;
      if (!chain_geometry(E, m, src, obs, X, ell, phip, phi)) return;
      if (!leg_plane(first ? X[0] : X[m], first ? X[1] : X[m + 1], n, cg, Pp)) return;
      if (pass == 0) {  // the member triangle holding the point: its own plane next
        d3w v0, v1, v2;
        int exw[6];
        for (int i = 0; i < m; ++i) {
          exw[2 * i] = E[i]->ta;
          exw[2 * i + 1] = E[i]->tb;
        }
        j = member_at(a, Pg, Pp, exw, 2 * m, v0, v1, v2, mj);
        if (j < 0) return;
        nj = unitw(crossw(v1 - v0, v2 - v0));
        n = nj;
        cg = dotw(nj, v0);
      } else {
        d3w v0, v1, v2;
        tri64(a, j, v0, v1, v2, mj);
        if (!inside_tri64(v0, v1, v2, Pp)) return;
      }
    }
  }
  // the real legs: Y the path's points, two excluded triangles at each
  d3w Y[6];
  int ex[6][2], ny = 0;
  Y[ny] = T; ex[ny][0] = ex[ny][1] = -1; ++ny;
  if (first) { Y[ny] = Pp; ex[ny][0] = ex[ny][1] = j; ++ny; }
  for (int i = 0; i < m; ++i) { Y[ny] = X[i + 1]; ex[ny][0] = E[i]->ta; ex[ny][1] = E[i]->tb; ++ny; }
  if (last) { Y[ny] = Pp; ex[ny][0] = ex[ny][1] = j; ++ny; }
  Y[ny] = R; ex[ny][0] = ex[ny][1] = -1; ++ny;
  if (legs_occluded(a, Y, ex, ny, ovf, st)) return;
  unsigned fl = 0;
  const d3w u = D3(a.pol.x, a.pol.y, a.pol.z);
  d3w ip = (X[1] - X[0]) * (1.0 / ell[0]);  // the real direction into Q_1
  double sn, cs;
  sincos(-k * ell[0], &sn, &cs);
  zd Ei = Z(cs / ell[0], sn / ell[0]);
  zv3 Ev;
  if (first) {
    d3w din = unitw(Pp - T);
    d3w e0 = polw(u, din, fl);
    zv3 E0 = {Z(e0.x), Z(e0.y), Z(e0.z)};
    zv3 Er = reflect_field_d(a, nj, mj, din, ip, E0);
    Ev = zv3{Er.x * Ei, Er.y * Ei, Er.z * Ei};
  } else {
    d3w e0 = polw(u, ip, fl);
    Ev = zv3{Ei * e0.x, Ei * e0.y, Ei * e0.z};
  }
  double rho1 = ell[0], rho2 = ell[0];
  d3w dir1 = D3(0, 0, 0), dir2 = D3(0, 0, 0), dd = ip;
  for (int i = 0; i < m; ++i) {
    const Wedge& W = *E[i];
    const double s = ell[i + 1], nn = W.n;
    const d3w e = D3(W.e[0], W.e[1], W.e[2]);
    dd = (X[i + 2] - X[i + 1]) * (1.0 / s);
    double beta0 = acos(fmax(-1.0, fmin(1.0, dotw(ip, e))));
    double sb = sin(beta0);
    d3w php = unitw(crossw(e, ip)) * -1.0, ph = unitw(crossw(e, dd));
    d3w bp = crossw(ip, php), bd = crossw(dd, ph);
    double rhoe;
    if (i == 0) rhoe = ell[0];
    else {
      double c1 = dotw(bp, dir1), c2 = dotw(bp, dir2);
      rhoe = 1.0 / (c1 * c1 / rho1 + c2 * c2 / rho2);
    }
    double L = s * (rhoe + s) * rho1 * rho2 * sb * sb / (rhoe * (rho1 + s) * (rho2 + s));
    const float4 ma =
        a.mats[__float_as_int(a.tris[3 * (size_t)DCEM_IDX(a.slot_of_id[DCEM_IDX(W.ta, a.bvh.ntris)], a.bvh.ntris) + 1].w)];
    const float4 mb =
        a.mats[__float_as_int(a.tris[3 * (size_t)DCEM_IDX(a.slot_of_id[DCEM_IDX(W.tb, a.bvh.ntris)], a.bvh.ntris) + 1].w)];
    zd r0s, r0h, rns, rnh;
    fresnel_faces(ma, fabs(sin(phip[i])), mb, fabs(sin(nn * M_PI - phi[i])), a.freq, r0s, r0h, rns, rnh);
    const UtdParts up = utd_parts(nn, phi[i], phip[i], beta0, L, k, fl);
    zd Ds = utd_coeff(up, r0s, rns), Dh = utd_coeff(up, r0h, rnh);
    sincos(-k * s, &sn, &cs);
    zd A = Z(cs, sn) * sqrt(rhoe / (s * (rhoe + s)));
    zd cb = Ds * zvdot(Ev, bp) * A * -1.0, cp = Dh * zvdot(Ev, php) * A * -1.0;
    Ev = zv3{cb * bd.x + cp * ph.x, cb * bd.y + cp * ph.y, cb * bd.z + cp * ph.z};
    rho1 = s;
    dir1 = ph;
    rho2 = rhoe + s;
    dir2 = bd;
    ip = dd;
  }
  d3w dlast = dd;
  if (last) {  // reflected last, toward the real receiver
    d3w dout = unitw(R - Pp);
    Ev = reflect_field_d(a, nj, mj, dd, dout, Ev);
    dlast = dout;
  }
  d3w prx = polw(u, dlast * -1.0, fl);
  zd amp = zvdot(Ev, prx) * (lam / (4.0 * M_PI));
  double Ltot = 0.0;
  for (int q = 0; q <= m; ++q) Ltot += ell[q];
  if (diff_lane() != 0) return;  // one lane of the group writes the record
  unsigned uu = atomicAdd(&a.ctr->n_unique, 1u);
  if (uu >= a.ucap) {
    atomicOr(&a.ctr->err, ERR_UNIQUE_OVERFLOW);
    return;
  }
  const int depth = m + (pl >= 0 ? 1 : 0);
  int ids[4];
  for (int q = 0; q < depth; ++q) {
    if (first) ids[q] = q == 0 ? j : (w[q - 1] | kDiffBit);
    else if (last) ids[q] = q == m ? j : (w[q] | kDiffBit);
    else ids[q] = w[q] | kDiffBit;
  }
  PathRec rec;
  rec.key = seq_key(r, depth, [&](int q) { return ids[q]; });
  rec.rx = link;
  rec.depth = depth;
  rec.ray = -1;
  rec.flags = fl;
  rec.valid = 1;
  rec.pad = 0;
  rec.len = Ltot;
  rec.amp_re = amp.re;
  rec.amp_im = amp.im;
  for (int q = 0; q < kMaxRefl; ++q) {
    rec.tri[q] = q < depth ? ids[q] : -1;
    rec.pts[q][0] = rec.pts[q][1] = rec.pts[q][2] = 0.0f;
  }
  for (int q = 1; q + 1 < ny; ++q) {
    rec.pts[q - 1][0] = (float)Y[q].x;
    rec.pts[q - 1][1] = (float)Y[q].y;
    rec.pts[q - 1][2] = (float)Y[q].z;
  }
  a.prec[uu] = rec;
  unsigned pos = atomicAdd(&a.bucket_cnt[link], 1u);
  if (pos < (unsigned)a.bucket_cap) a.bucket[(size_t)link * a.bucket_cap + pos] = (int)uu;
  else atomicOr(&a.ctr->err, ERR_BUCKET_OVERFLOW);
  atomicAdd(&a.ctr->n_valid, 1u);
}

// ---------------------------------------------------------------------------
// two reflections around a first-order diffraction (Sec. III steps 3-5; the
// paper's evaluation allows two reflections and one diffraction per path)
// ---------------------------------------------------------------------------
// Candidates (kind, link, p1, p2, wedge), the reflector planes p1, p2 in path
// order: kind 0 both before the wedge (Tx -> P1 -> P2 -> Q -> Rx), 1 one on
// each side (Tx -> P1 -> Q -> P2 -> Rx), 2 both after it (Tx -> Q -> P1 -> P2
// -> Rx). By image theory the diffraction runs from the transmitter's image
// in the planes before the wedge (taken in path order) toward the receiver's
// image in the planes after it (the last one first); the reflection points
// follow by unfolding back from Q. The candidates are formed per side of the
// wedge (k_refl_single to k_refl_double) or link by link (k_refl_direct).
// Survivors carry 10 in bits 63-62 and 1 in bit 61 over (block * nw + wedge).
constexpr unsigned long long kRefl2Tag = kReflTag | (1ull << 61);
constexpr unsigned long long kRefl2Mask = (1ull << 61) - 1ull;

// Where the legs from S to the points of `box` (lo, hi) cross plane P inside
// P's box: false when none can, else [lo, hi] becomes a box that holds every
// such crossing. Legs to the corners across the plane from S bound the
// crossings of the box's part there; where the plane cuts the box (a corner
// on S's side, or within m of the plane), the cut is itself a set of
// crossings, bounded by the box. No conclusion for S within m of the plane.
__device__ __forceinline__ bool box_window(const RPlane& P, float3 S, float m, float* lo, float* hi) {
  const float3 n = f3(P.nf[0], P.nf[1], P.nf[2]);
  const float ds = fdot3(n, S) - P.cf;
  if (fabsf(ds) <= m) {
    for (int k = 0; k < 3; ++k) {
      lo[k] = P.box[k];
      hi[k] = P.box[3 + k];
    }
    return true;
  }
  float wl[3] = {3e38f, 3e38f, 3e38f}, wh[3] = {-3e38f, -3e38f, -3e38f};
  bool any = false, cut = false;
#pragma unroll 2  // (the kernels that inline this are bound by instruction fetch)
  for (int q = 0; q < 8; ++q) {
    const float3 X = f3((q & 1) ? hi[0] + m : lo[0] - m, (q & 2) ? hi[1] + m : lo[1] - m, (q & 4) ? hi[2] + m : lo[2] - m);
    const float dx = fdot3(n, X) - P.cf, sd = ds > 0.0f ? dx : -dx;  // sd > 0: on S's side
    if (sd >= -m) cut = true;
    if (sd > m) continue;
    any = true;
    const float t = fminf(fmaxf(ds / (ds - dx), 0.0f), 1.0f);
    const float x = S.x + t * (X.x - S.x), y = S.y + t * (X.y - S.y), z = S.z + t * (X.z - S.z);
    wl[0] = fminf(wl[0], x); wl[1] = fminf(wl[1], y); wl[2] = fminf(wl[2], z);
    wh[0] = fmaxf(wh[0], x); wh[1] = fmaxf(wh[1], y); wh[2] = fmaxf(wh[2], z);
  }
  if (!any) return false;
  bool meet = true;
  for (int k = 0; k < 3; ++k) {
    if (cut) {
      wl[k] = fminf(wl[k], lo[k] - m);
      wh[k] = fmaxf(wh[k], hi[k] + m);
    }
    lo[k] = fmaxf(wl[k], P.box[k]) - m;
    hi[k] = fminf(wh[k], P.box[3 + k]) + m;
    meet = meet && lo[k] <= hi[k];
  }
  return meet;
}

// The crossing X of the unfolded leg a0 -> a1 with plane P, within margins
// (delta + 2e-4 of the distances): 0 when it certainly lies off the leg or
// off P's box, 1 with X set, 2 when the leg runs nearly parallel to the
// plane (no conclusion).
__device__ __forceinline__ int refl_cross32(const RPlane& P, float3 a0, float3 a1, float delta, float3& X) {
  const float3 n = f3(P.nf[0], P.nf[1], P.nf[2]);
  const float3 dv = f3(a1.x - a0.x, a1.y - a0.y, a1.z - a0.z);
  const float den = fdot3(n, dv), len = sqrtf(fdot3(dv, dv));
  if (!(fabsf(den) > 1e-6f * len)) return 2;
  const float t = (P.cf - fdot3(n, a0)) / den;
  const float mt = (delta + 2e-4f * (len + sqrtf(fdot3(a0, a0)))) / len;
  if (t < -mt || t > 1.0f + mt) return 0;
  X = f3(a0.x + t * dv.x, a0.y + t * dv.y, a0.z + t * dv.z);
  const float mb = delta + 2e-4f * (len + sqrtf(fdot3(X, X)));
  if (X.x < P.box[0] - mb || X.y < P.box[1] - mb || X.z < P.box[2] - mb || X.x > P.box[3] + mb ||
      X.y > P.box[4] + mb || X.z > P.box[5] + mb)
    return 0;
  return 1;
}

// FP32 pre-test of one candidate: false only when the FP64 test rejects it
// too. S, O: the source and observer of the diffraction (images); S1: the
// transmitter's image in P1 (kind 0), O1: the receiver's image in P2 (kind 2).
// The Keller point's place on the edge and the crossings with the planes
// there come first, the angle rules (diffract_candidate) last.
__device__ __forceinline__ bool refl2_candidate(const WedgeF& W, const RPlane& P1, const RPlane& P2, int kind,
                                                float3 S, float3 S1, float3 O, float3 O1) {
  const float3 e = W.e, p0 = W.p0;
  const float3 dt = f3(S.x - p0.x, S.y - p0.y, S.z - p0.z), dr = f3(O.x - p0.x, O.y - p0.y, O.z - p0.z);
  const float zt = fdot3(dt, e), zr = fdot3(dr, e);
  const float3 pt = f3(dt.x - e.x * zt, dt.y - e.y * zt, dt.z - e.z * zt);
  const float3 pr = f3(dr.x - e.x * zr, dr.y - e.y * zr, dr.z - e.z * zr);
  const float rt = sqrtf(fdot3(pt, pt)), rr = sqrtf(fdot3(pr, pr));
  if (!(rt > 1e-3f && rr > 1e-3f)) return true;  // as diffract_candidate: no conclusion
  const float zq = zt + (zr - zt) * rt / (rt + rr);
  const float mz = 0.05f + 1e-5f * (sqrtf(fdot3(dt, dt)) + sqrtf(fdot3(dr, dr)));
  if (zq < -mz || zq > W.len + mz) return false;  // the Keller point off the edge (as diffract_candidate)
  const float3 Q = f3(p0.x + e.x * zq, p0.y + e.y * zq, p0.z + e.z * zq);
  const float d = 0.1f;
  float3 X;
  if (kind == 0) {
    const int r = refl_cross32(P2, S, Q, d, X);
    if (r == 0) return false;
    if (r == 1 && refl_cross32(P1, S1, X, d, X) == 0) return false;
  } else if (kind == 1) {
    if (refl_cross32(P1, S, Q, d, X) == 0) return false;
    if (refl_cross32(P2, Q, O, d, X) == 0) return false;
  } else {
    const int r = refl_cross32(P1, Q, O, d, X);
    if (r == 0) return false;
    if (r == 1 && refl_cross32(P2, X, O1, d, X) == 0) return false;
  }
  return diffract_candidate(W, make_float4(S.x, S.y, S.z, 0.0f), make_float4(O.x, O.y, O.z, 0.0f));
}

static_assert(kWedgeCluster == 32 && kWedgeGroup == 8, "a mask word holds four groups, a warp four octets");

// The images of block (kind, link, p1, p2): S, O the diffraction's source
// and observer, S1 the transmitter's image in P1 (kind 0), O1 the
// receiver's image in P2 (kind 2).
__device__ __forceinline__ void refl2_images(const PathArgs& a, int kind, int link, const RPlane& P1,
                                             const RPlane& P2, float3& S, float3& S1, float3& O, float3& O1) {
  const float4 tv = a.txs[link / a.nrx], rv = a.rx[link % a.nrx];
  const float3 T = f3(tv.x, tv.y, tv.z), R = f3(rv.x, rv.y, rv.z);
  const float3 n1 = f3(P1.nf[0], P1.nf[1], P1.nf[2]);
  const float3 n2 = f3(P2.nf[0], P2.nf[1], P2.nf[2]);
  S = S1 = T;
  O = O1 = R;
  if (kind == 0) {
    S1 = mirror32(T, n1, P1.cf);
    S = mirror32(S1, n2, P2.cf);
  } else if (kind == 1) {
    S = S1 = mirror32(T, n1, P1.cf);
    O = O1 = mirror32(R, n2, P2.cf);
  } else {
    O1 = mirror32(R, n2, P2.cf);
    O = mirror32(O1, n1, P1.cf);
  }
}

// Survivor codes of one and two reflections around a first-order diffraction.
__device__ __forceinline__ unsigned long long refl1_code(const PathArgs& a, int link, int w, int p, bool first) {
  return kReflTag | ((((unsigned long long)link * a.nw + w) * a.nrp + p) * 2 + (first ? 1 : 0));
}
__device__ __forceinline__ unsigned long long refl2_code(const PathArgs& a, int nlinks, int kind, int link, int p1,
                                                         int p2, int w) {
  const unsigned long long b = (((unsigned long long)kind * nlinks + link) * a.nrp + p1) * a.nrp + p2;
  return kRefl2Tag | (b * a.nw + w);
}
struct ReflCand {
  int kind, link, w, p1, p2;  // kind 0-2 as above; 3: one reflection (p1) before the wedge, 4: after it
};
__device__ __forceinline__ ReflCand refl_decode(const PathArgs& a, int nlinks, unsigned long long code) {
  ReflCand c;
  if ((code >> 61) & 1ull) {
    unsigned long long v = code & kRefl2Mask;
    c.w = (int)(v % (unsigned)a.nw);
    v /= (unsigned)a.nw;
    c.p2 = (int)(v % (unsigned)a.nrp);
    v /= (unsigned)a.nrp;
    c.p1 = (int)(v % (unsigned)a.nrp);
    v /= (unsigned)a.nrp;
    c.link = (int)(v % (unsigned)nlinks);
    c.kind = (int)(v / (unsigned)nlinks);
  } else {
    unsigned long long v = code & ~kReflTag;
    c.kind = (v & 1ull) ? 3 : 4;
    v >>= 1;
    c.p1 = c.p2 = (int)(v % (unsigned)a.nrp);
    v /= (unsigned)a.nrp;
    c.w = (int)(v % (unsigned)a.nw);
    c.link = (int)(v / (unsigned)a.nw);
  }
  return c;
}

// ---- candidates by end point ----
// The candidates (link, wedge, planes) are a product of two sides that are
// nearly independent: the transmitter's image after 0, 1 or 2 reflections
// against a wedge, and the receiver's. Forming each side once and joining
// the two at the wedge costs a few percent of testing every (kind, link,
// plane pair) block on its own (8 x 8 city blocks, 64 receivers, 321 planes:
// 19.8M blocks, 24.5 ms; this form 1.9 ms in all):
//   k_diff_visible the planes and wedges each end point may see at all
//   k_refl_single  every (end point, plane): the wedges that the image sees
//                  through the plane's box. Such a side with no reflection
//                  on the other end gives the one-reflection candidates;
//                  with two reflections on, the sets are also kept as mask
//                  words and the receivers' sides counted per wedge
//   k_refl_lists   the receivers' one-reflection sides listed by wedge
//   k_refl_join    every transmitter side with one reflection against its
//                  wedge's list: one reflection on each side of the wedge
//   k_refl_double  every (end point, plane, plane): the wedges that the
//                  double image sees, against the other ends: both
//                  reflections on one side
// The joins apply the closed-form Keller point and the angle rules
// (side_pair, the rules of diffract_candidate on precomputed sides); what
// passes goes through the full FP32 test (refl_candidates_take).

// A point about a wedge: along the edge, off the edge line, from the edge's
// start, and its angle (sure: tol >= 0).
struct WedgeSide {
  float z, r, l, phi, tol;
};
__device__ __forceinline__ void side_zr(const WedgeF& W, float3 X, WedgeSide& s, float3& p) {
  const float3 d = f3(X.x - W.p0.x, X.y - W.p0.y, X.z - W.p0.z);
  s.z = fdot3(d, W.e);
  p = f3(d.x - W.e.x * s.z, d.y - W.e.y * s.z, d.z - W.e.z * s.z);
  s.r = sqrtf(fdot3(p, p));
  s.l = sqrtf(fdot3(d, d));
}
__device__ __forceinline__ void side_angle(const WedgeF& W, float3 p, WedgeSide& s) {
  bool sure;
  s.phi = wedge_angle32(p, W.t0, W.y0, s.r, s.l, sure, s.tol);
  if (!sure) s.tol = -1.0f;
}
__device__ __forceinline__ WedgeSide wedge_side(const WedgeF& W, float3 X) {
  WedgeSide s;
  float3 p;
  side_zr(W, X, s, p);
  side_angle(W, p, s);
  return s;
}
// The Keller point of two sides within the edge (margins of diffract_candidate)?
__device__ __forceinline__ bool side_keller(float len, const WedgeSide& s, const WedgeSide& o) {
  if (!(s.r > 1e-3f && o.r > 1e-3f)) return true;
  const float zq = s.z + (o.z - s.z) * s.r / (s.r + o.r);
  const float mz = 0.05f + 1e-5f * (s.l + o.l);
  return !(zq < -mz || zq > len + mz);
}
// ... and the angle rules (the angles of both sides known)?
__device__ __forceinline__ bool side_rules(float npi, const WedgeSide& s, const WedgeSide& o) {
  if (!(s.r > 1e-3f && o.r > 1e-3f)) return true;
  const bool ss = s.tol >= 0.0f, so = o.tol >= 0.0f;
  if ((ss && s.phi > npi + s.tol) || (so && o.phi > npi + o.tol)) return false;
  return !(ss && so && fabsf(o.phi - s.phi) < 3.14159265f - (s.tol + o.tol));
}

// Does an image X (of an end point, in plane Pl last) see wedge W: the
// wedge not facing away, and some leg to its edge crossing Pl in its box?
// For a double image, the legs must also have crossed the first plane Pf on
// their way from the single image Xf to the crossings with Pl.
__device__ __forceinline__ bool image_sees(const RPlane& Pl, const WedgeF& W, float3 X, const RPlane* Pf, float3 Xf) {
  float3 A, B;
  edge_ends(W, A, B);
  const float mg = 0.1f + 1e-4f * (fabsf(X.x) + fabsf(X.y) + fabsf(X.z) + W.len);
  float lo[3], hi[3];
  return leg_window(Pl, X, A, B, mg, lo, hi) && (!Pf || box_window(*Pf, Xf, mg, lo, hi)) && !surely_inside(W, X);
}
// ... and a group of wedges, by its box.
__device__ __forceinline__ bool image_sees_group(const PathArgs& a, const RPlane& Pl, int g, float3 X, float m,
                                                 const RPlane* Pf, float3 Xf) {
  const float* gb = a.wgbox + 6 * (size_t)g;
  float lo[3] = {gb[0], gb[1], gb[2]}, hi[3] = {gb[3], gb[4], gb[5]};
  return box_window(Pl, X, m, lo, hi) && (!Pf || box_window(*Pf, Xf, m, lo, hi));
}
// The next four of the lanes in mask `gm`, whose groups are g, to the warp's
// four octets: this lane's place in the wedge order, -1 for none.
__device__ __forceinline__ int octet_wedge(const PathArgs& a, int g, unsigned& gm) {
  const int lane = threadIdx.x & 31;
  int src = -1;
  for (int k = 0; k < 4 && gm; ++k, gm &= gm - 1u)
    if (lane >> 3 == k) src = __ffs(gm) - 1;
  const int i = __shfl_sync(0xffffffffu, g, max(src, 0)) * kWedgeGroup + (lane & 7);
  return src >= 0 && i < a.nw ? i : -1;
}
__device__ __forceinline__ float3 plane_image(const RPlane& P, float3 X) {
  return mirror32(X, f3(P.nf[0], P.nf[1], P.nf[2]), P.cf);
}
__device__ __forceinline__ float image_margin(float3 X, float3 Y) {
  return 0.1f + 1e-4f * (fabsf(X.x) + fabsf(X.y) + fabsf(X.z) + fabsf(Y.x) + fabsf(Y.y) + fabsf(Y.z));
}

// Two FIFO queues per warp in shared memory, so that each stage runs on full
// warps: sides (end point, planes, wedge) waiting to be joined with the
// other ends, and candidates waiting for the full test. At most 31 entries
// wait when up to 32 join, so rings of 64 hold them.
constexpr int kReflWarps = 8, kReflRing = 64;
struct ReflQueues {
  int4 side[kReflWarps][kReflRing];  // item, first plane from it, second or -1, wedge (place in wperm)
  unsigned long long cand[kReflWarps][kReflRing];
};
struct ReflRing {  // warp-uniform
  int sh = 0, st = 0, ch = 0, ct = 0;
};

// The oldest `nn` candidates of the warp through the full FP32 test; those
// that pass join the survivor list.
__device__ __noinline__ void refl_candidates_take(const PathArgs& a, int nlinks, const unsigned long long* q, int head,
                                                  int nn) {
  const int lane = threadIdx.x & 31;
  bool keep = false;
  unsigned long long code = 0;
  if (lane < nn) {
    code = q[(head + lane) & (kReflRing - 1)];
    const ReflCand c = refl_decode(a, nlinks, code);
    const WedgeF W = a.wf[c.w];
    if (c.kind >= 3) {
      keep = diffract_refl_candidate(W, a.rplanes[c.p1], a.txs[c.link / a.nrx], a.rx[c.link % a.nrx], c.kind == 3);
    } else {
      float3 S, S1, O, O1;
      refl2_images(a, c.kind, c.link, a.rplanes[c.p1], a.rplanes[c.p2], S, S1, O, O1);
      keep = refl2_candidate(W, a.rplanes[c.p1], a.rplanes[c.p2], c.kind, S, S1, O, O1);
    }
  }
  const unsigned mk = __ballot_sync(0xffffffffu, keep);
  if (!mk) return;
  unsigned at = 0;
  if (lane == 0) at = atomicAdd(&a.ctr->n_dsurv, (unsigned)__popc(mk));
  at = __shfl_sync(0xffffffffu, at, 0) + __popc(mk & ((1u << lane) - 1u));
  if (keep) {
    if (at < a.dsurv_cap) a.dsurv[at] = code;
    else atomicOr(&a.ctr->err, ERR_DIFF_OVERFLOW);
  }
}

// Lanes with `add` push their candidate; 32 waiting go through the test.
__device__ __forceinline__ void refl_push(const PathArgs& a, int nlinks, unsigned long long* q, ReflRing& r, bool add,
                                          unsigned long long code) {
  const unsigned m = __ballot_sync(0xffffffffu, add);
  if (!m) return;
  const int lane = threadIdx.x & 31;
  if (add) q[(r.ct + __popc(m & ((1u << lane) - 1u))) & (kReflRing - 1)] = code;
  r.ct += __popc(m);
  __syncwarp();
  if (r.ct - r.ch >= 32) {
    refl_candidates_take(a, nlinks, q, r.ch, 32);
    r.ch += 32;
    __syncwarp();
  }
}

// Work items by end point: the transmitters, each split into a.rsub runs of
// receivers (few transmitters against many receivers would otherwise leave
// their pairs to a few warps), then the receivers.
__device__ __forceinline__ int item_end(const PathArgs& a, int ntx, int v) {
  return v < ntx * a.rsub ? v / a.rsub : v - ntx * a.rsub + ntx;
}

// The oldest `nn` sides of the warp against the other ends without a
// reflection: a transmitter's side against the item's run of receivers, a
// receiver's against every transmitter. (Entries name the item, not the end point.)
__device__ __noinline__ void refl_sides_take(const PathArgs& a, int ntx, int nlinks, const int4* sq,
                                             unsigned long long* cq, ReflRing& r, int nn) {
  const int lane = threadIdx.x & 31;
  int4 s = make_int4(0, 0, -1, 0);
  WedgeSide me{};
  WedgeF W{};
  int y0 = 0, y1 = 0, at = 0;
  if (lane < nn) {
    s = sq[(r.sh + lane) & (kReflRing - 1)];
    at = s.w;
    s.w = a.wperm[at];
    const int v = s.x;
    s.x = item_end(a, ntx, v);
    W = a.wf[s.w];
    float3 X = plane_image(a.rplanes[s.y], end_point(a, ntx, s.x));
    if (s.z >= 0) X = plane_image(a.rplanes[s.z], X);
    me = wedge_side(W, X);
    if (s.x < ntx) {
      const int run = (a.nrx + a.rsub - 1) / a.rsub;
      y0 = (v % a.rsub) * run;
      y1 = min(a.nrx, y0 + run);
    } else {
      y1 = ntx;
    }
  }
  const int most = __reduce_max_sync(0xffffffffu, max(y1 - y0, 0));
  for (int k = 0; k < most; ++k) {
    const int y = y0 + k, yx = s.x < ntx ? ntx + y : y;
    bool ok = y < y1 && sees_wedge(a, yx, at);
    if (ok) {
      const float3 Y = end_point(a, ntx, yx);
      WedgeSide o;
      float3 p;
      side_zr(W, Y, o, p);
      ok = side_keller(W.len, me, o);
      if (ok) {
        side_angle(W, p, o);
        ok = side_rules(W.npi, me, o);
      }
    }
    unsigned long long code = 0;
    if (ok) {
      const bool tx = s.x < ntx;
      const int link = tx ? s.x * a.nrx + y : y * a.nrx + (s.x - ntx);
      code = s.z < 0 ? refl1_code(a, link, s.w, s.y, tx)
                     : refl2_code(a, nlinks, tx ? 0 : 2, link, tx ? s.y : s.z, tx ? s.z : s.y, s.w);
    }
    refl_push(a, nlinks, cq, r, ok, code);
  }
}

// The wedges of cluster c that lanes with `bit` hold join the side queue.
__device__ __forceinline__ void side_push(const PathArgs& a, int ntx, int nlinks, int4* sq, unsigned long long* cq,
                                          ReflRing& r, bool bit, int4 s) {
  const unsigned m = __ballot_sync(0xffffffffu, bit);
  if (!m) return;
  const int lane = threadIdx.x & 31;
  if (bit) sq[(r.st + __popc(m & ((1u << lane) - 1u))) & (kReflRing - 1)] = s;
  r.st += __popc(m);
  __syncwarp();
  if (r.st - r.sh >= 32) {
    refl_sides_take(a, ntx, nlinks, sq, cq, r, 32);
    r.sh += 32;
    __syncwarp();
  }
}
__device__ __forceinline__ void refl_flush(const PathArgs& a, int ntx, int nlinks, int4* sq, unsigned long long* cq,
                                           ReflRing& r) {
  if (r.st > r.sh) refl_sides_take(a, ntx, nlinks, sq, cq, r, r.st - r.sh);
  __syncwarp();
  if (r.ct > r.ch) refl_candidates_take(a, nlinks, cq, r.ch, r.ct - r.ch);
}

// One warp per (end point, plane) and part of the wedge groups (`parts` of
// them while there are few end points and planes: in an open scene every
// group is in the image's window): lanes test the groups' boxes first, then
// the wedges, four groups at once.
__global__ void __launch_bounds__(256) k_refl_single(PathArgs a, int ntx, int nlinks, int parts) {
  __shared__ ReflQueues Q;
  const long nitem = ((long)ntx * a.rsub + a.nrx) * a.nrp * parts;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const long nwarp = (long)gridDim.x * kReflWarps;
  const int ng = (a.nw + kWedgeGroup - 1) / kWedgeGroup;
  ReflRing r;
  for (long u = (long)blockIdx.x * kReflWarps + wid; u < nitem; u += nwarp) {
    const long it = u / parts;
    const int p = (int)(it % a.nrp), v = (int)(it / a.nrp), x = item_end(a, ntx, v);
    if (!sees_plane(a, x, p)) continue;
    const RPlane& Pl = a.rplanes[p];
    const float3 E = end_point(a, ntx, x), X = plane_image(Pl, E);
    const float m = image_margin(E, X);
    for (int g0 = 32 * (int)(u % parts); g0 < ng; g0 += 32 * parts) {
      const bool near = g0 + lane < ng && image_sees_group(a, Pl, g0 + lane, X, m, nullptr, X);
      for (unsigned gm = __ballot_sync(0xffffffffu, near); gm;) {
        const int i = octet_wedge(a, g0 + lane, gm);
        int w = 0;
        bool bit = false;
        if (i >= 0) {
          w = a.wperm[i];
          bit = image_sees(Pl, a.wf[w], X, nullptr, X);
        }
        if (bit && a.drefl2) {
          atomicOr(&a.rmask[((long)x * a.nrp + p) * a.nwc + i / kWedgeCluster], 1u << (i % kWedgeCluster));
          if (x >= ntx) atomicAdd(&a.wobs_cnt[w], 1u);
        }
        side_push(a, ntx, nlinks, Q.side[wid], Q.cand[wid], r, bit, make_int4(v, p, -1, i));
      }
    }
  }
  refl_flush(a, ntx, nlinks, Q.side[wid], Q.cand[wid], r);
}

// Room in the observer list for every wedge's receiver sides.
__global__ void k_refl_room(PathArgs a) {
  for (int w = blockIdx.x * blockDim.x + threadIdx.x; w < a.nw; w += gridDim.x * blockDim.x) {
    const unsigned n = a.wobs_cnt[w];
    const unsigned at = n ? atomicAdd(&a.ctr->n_dobs, n) : 0u;
    a.wobs_off[w] = a.wobs_pos[w] = at;
    if (n && (unsigned long long)at + n > a.dobs_cap) atomicOr(&a.ctr->err, ERR_DIFF_OVERFLOW);
  }
}

// The receivers' one-reflection sides into their wedges' lists, from the
// mask words: one warp per (receiver, plane) and part of the words.
__global__ void __launch_bounds__(256) k_refl_lists(PathArgs a, int ntx, int parts) {
  const long nitem = (long)a.nrx * a.nrp * parts;
  const int lane = threadIdx.x & 31;
  const long nwarp = (long)gridDim.x * (blockDim.x >> 5);
  for (long u = (long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); u < nitem; u += nwarp) {
    const long it = u / parts;
    const int p = (int)(it % a.nrp), rx = (int)(it / a.nrp), part = (int)(u % parts);
    const float3 X = plane_image(a.rplanes[p], end_point(a, ntx, ntx + rx));
    const unsigned* row = a.rmask + ((long)(ntx + rx) * a.nrp + p) * a.nwc;
    for (int c0 = 0; c0 < a.nwc; c0 += 32) {
      const unsigned word = c0 + lane < a.nwc && (c0 + lane) % parts == part ? row[c0 + lane] : 0u;
      for (unsigned cm = __ballot_sync(0xffffffffu, word != 0); cm; cm &= cm - 1u) {
        const int src = __ffs(cm) - 1;
        const unsigned wd = __shfl_sync(0xffffffffu, word, src);
        if (!((wd >> lane) & 1u)) continue;
        const int w = a.wperm[(c0 + src) * kWedgeCluster + lane];
        const WedgeSide s = wedge_side(a.wf[w], X);
        const unsigned at = atomicAdd(&a.wobs_pos[w], 1u);
        if (at < a.dobs_cap) a.dobs[at] = DiffObs{rx, p, s.z, s.r, s.l, s.phi, s.tol, 0.0f};
      }
      __syncwarp();
    }
  }
}

// One reflection on each side of the wedge: one warp per (transmitter,
// plane, cluster) mask word and eighth of the lists, its lanes over that
// part of the list of each wedge in the word.
constexpr int kJoinParts = 8;
__global__ void __launch_bounds__(256) k_refl_join(PathArgs a, int ntx, int nlinks) {
  __shared__ unsigned long long cq[kReflWarps][kReflRing];
  const long nitem = (long)ntx * a.nrp * a.nwc * kJoinParts;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const long nwarp = (long)gridDim.x * kReflWarps;
  ReflRing r;
  for (long part = (long)blockIdx.x * kReflWarps + wid; part < nitem; part += nwarp) {
    const long it = part / kJoinParts;
    unsigned word = a.rmask[it];
    if (!word) continue;
    const int c = (int)(it % a.nwc);
    const long tp = it / a.nwc;
    const int p1 = (int)(tp % a.nrp), t = (int)(tp / a.nrp);
    const float3 S = plane_image(a.rplanes[p1], end_point(a, ntx, t));
    for (; word; word &= word - 1u) {
      const int w = a.wperm[c * kWedgeCluster + __ffs(word) - 1];
      const WedgeF W = a.wf[w];
      const WedgeSide me = wedge_side(W, S);
      const unsigned n = a.wobs_cnt[w], off = a.wobs_off[w];
      if ((unsigned long long)off + n > a.dobs_cap) continue;  // the list overflowed: the frame is traced again
      for (unsigned i0 = 32 * (unsigned)(part % kJoinParts); i0 < n; i0 += 32 * kJoinParts) {
        bool ok = i0 + lane < n;
        unsigned long long code = 0;
        if (ok) {
          const DiffObs o = a.dobs[off + i0 + lane];
          const WedgeSide os{o.z, o.r, o.l, o.phi, o.tol};
          ok = side_keller(W.len, me, os) && side_rules(W.npi, me, os);
          if (ok) code = refl2_code(a, nlinks, 1, t * a.nrx + o.rx, p1, o.p, w);
        }
        refl_push(a, nlinks, cq[wid], r, ok, code);
      }
    }
  }
  if (r.ct > r.ch) refl_candidates_take(a, nlinks, cq[wid], r.ch, r.ct - r.ch);
}

// Both reflections on one side of the wedge: lanes take (end point, first
// plane from it, second plane) and keep those whose second plane's box the
// image can reach through the first's; for each of them the warp tests the
// groups' boxes against the double image, then the groups' wedges. `per`
// items a warp: 32, or fewer so that all warps have one (a highway's 8 planes
// and 201 end points make 14,400 items, nearly all of them within reach).
__global__ void __launch_bounds__(256, 3) k_refl_double(PathArgs a, int ntx, int nlinks, int per) {
  __shared__ ReflQueues Q;
  const long nitem = ((long)ntx * a.rsub + a.nrx) * a.nrp * a.nrp;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const long stride = (long)gridDim.x * kReflWarps * per;
  const int ng = (a.nw + kWedgeGroup - 1) / kWedgeGroup;
  ReflRing r;
  for (long base = ((long)blockIdx.x * kReflWarps + wid) * per; base < nitem; base += stride) {
    const long it = lane < per ? base + lane : nitem;
    int v = 0, pa = 0, pb = 0;
    float m = 0.0f;
    bool pass = false;
    if (it < nitem) {
      pb = (int)(it % a.nrp);
      const long q = it / a.nrp;
      pa = (int)(q % a.nrp);
      v = (int)(q / a.nrp);
      const int x = item_end(a, ntx, v);
      if (pa != pb && sees_plane(a, x, pa)) {  // two reflections in a row are on different planes
        const float3 E = end_point(a, ntx, x), X1 = plane_image(a.rplanes[pa], E);
        const RPlane& Pb = a.rplanes[pb];
        m = image_margin(E, plane_image(Pb, X1));
        float lo[3] = {Pb.box[0], Pb.box[1], Pb.box[2]}, hi[3] = {Pb.box[3], Pb.box[4], Pb.box[5]};
        pass = box_window(a.rplanes[pa], X1, m, lo, hi);
      }
    }
    for (unsigned pm = __ballot_sync(0xffffffffu, pass); pm; pm &= pm - 1u) {
      const int who = __ffs(pm) - 1;
      const int uv = __shfl_sync(0xffffffffu, v, who), ux = item_end(a, ntx, uv), ua = __shfl_sync(0xffffffffu, pa, who),
                ub = __shfl_sync(0xffffffffu, pb, who);
      const float um = __shfl_sync(0xffffffffu, m, who);
      const RPlane &Pa = a.rplanes[ua], &Pb = a.rplanes[ub];
      const float3 U1 = plane_image(Pa, end_point(a, ntx, ux)), U = plane_image(Pb, U1);
      // the wedges the other ends see
      const unsigned* opp = a.vis_any + (ux < ntx ? a.nwc : 0);
      const int* grp = a.vis_grp + (ux < ntx ? ng + 1 : 0);
      const int n = grp[0];
      for (int k0 = 0; k0 < n; k0 += 32) {
        const int g = k0 + lane < n ? grp[1 + k0 + lane] : -1;
        const bool near = g >= 0 && image_sees_group(a, Pb, g, U, um, &Pa, U1);
        for (unsigned gm = __ballot_sync(0xffffffffu, near); gm;) {
          const int i = octet_wedge(a, g, gm);
          bool bit = false;
          if (i >= 0 && ((opp[i / kWedgeCluster] >> (i % kWedgeCluster)) & 1u))
            bit = image_sees(Pb, a.wf[a.wperm[i]], U, &Pa, U1);
          side_push(a, ntx, nlinks, Q.side[wid], Q.cand[wid], r, bit, make_int4(uv, ua, ub, i));
        }
      }
    }
  }
  refl_flush(a, ntx, nlinks, Q.side[wid], Q.cand[wid], r);
}

// The same candidates link by link, for open scenes with few transmitters:
// nearly every wedge is within reach of every double image there, so forming
// the sides first saves nothing, and the Keller point's place on the edge (a
// tenth of a side's work) drops most pairs. One warp per (side, link, plane,
// plane). A highway (8 planes, 2400 wedges, 200 links): 1.55 ms a frame by
// k_refl_double, 0.57 ms by this.
__global__ void __launch_bounds__(256, 3) k_refl_direct(PathArgs a, int ntx, int nlinks) {
  __shared__ unsigned long long cq[kReflWarps][kReflRing];
  const long nitem = 2L * nlinks * a.nrp * a.nrp;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const long nwarp = (long)gridDim.x * kReflWarps;
  const int ng = (a.nw + kWedgeGroup - 1) / kWedgeGroup;
  ReflRing r;
  for (long it = (long)blockIdx.x * kReflWarps + wid; it < nitem; it += nwarp) {
    const int pb = (int)(it % a.nrp);
    long q = it / a.nrp;
    const int pa = (int)(q % a.nrp);
    q /= a.nrp;
    const int link = (int)(q % nlinks), t = link / a.nrx, rx = ntx + link % a.nrx;
    const bool tx = q < nlinks;
    const int x = tx ? t : rx, y = tx ? rx : t;
    if (pa == pb || !sees_plane(a, x, pa)) continue;
    const RPlane &Pa = a.rplanes[pa], &Pb = a.rplanes[pb];
    const float3 E = end_point(a, ntx, x), Y = end_point(a, ntx, y), X1 = plane_image(Pa, E), X = plane_image(Pb, X1);
    const float m = image_margin(E, X);
    float lo[3] = {Pb.box[0], Pb.box[1], Pb.box[2]}, hi[3] = {Pb.box[3], Pb.box[4], Pb.box[5]};
    if (!box_window(Pa, X1, m, lo, hi)) continue;
    for (int g0 = 0; g0 < ng; g0 += 32) {
      const int g = g0 + lane;
      const bool near = g < ng && image_sees_group(a, Pb, g, X, m, &Pa, X1);
      for (unsigned gm = __ballot_sync(0xffffffffu, near); gm;) {
        const int i = octet_wedge(a, g, gm);
        bool ok = i >= 0 && sees_wedge(a, y, i);
        unsigned long long code = 0;
        if (ok) {
          const int w = a.wperm[i];
          const WedgeF& W = a.wf[w];
          WedgeSide me, o;
          float3 p;
          side_zr(W, X, me, p);
          side_zr(W, Y, o, p);
          ok = side_keller(W.len, me, o);
          if (ok) code = refl2_code(a, nlinks, tx ? 0 : 2, link, tx ? pa : pb, tx ? pb : pa, w);
        }
        refl_push(a, nlinks, cq[wid], r, ok, code);
      }
    }
  }
  if (r.ct > r.ch) refl_candidates_take(a, nlinks, cq[wid], r.ch, r.ct - r.ch);
}

// ---- occlusion before the exact stage ----
// Nearly every candidate of the tests above has its Keller point and
// reflection points in place and a building in between (8 x 8 city blocks:
// 183k candidates, 313 paths), and the exact stage's FP64 work per
// candidate is two orders of magnitude dearer than an FP32 traversal. So the
// candidates whose legs are certainly blocked (leg_surely_blocked around the
// FP32 estimate of the points) are dropped here. The estimate is trusted to
// the margins of the candidate tests where it is well conditioned: both ends
// half a metre off the edge line, legs more than 3 degrees off the planes
// they cross; elsewhere the candidate is kept. Chains were tested by
// k_diff_multi_pre; with transmission on, a first-order leg may cross walls.

// The crossing of the unfolded leg a0 -> a1 with plane P; false when the leg
// is within 3 degrees of the plane. delta: the larger of its value and the
// crossing's margin.
__device__ __forceinline__ bool plane_cross32(const RPlane& P, float3 a0, float3 a1, float3& X, float& delta) {
  const float3 n = f3(P.nf[0], P.nf[1], P.nf[2]);
  const float3 dv = f3(a1.x - a0.x, a1.y - a0.y, a1.z - a0.z);
  const float den = fdot3(n, dv), len = sqrtf(fdot3(dv, dv));
  if (!(fabsf(den) > 0.05f * len)) return false;
  const float t = (P.cf - fdot3(n, a0)) / den;
  X = f3(a0.x + t * dv.x, a0.y + t * dv.y, a0.z + t * dv.z);
  delta = fmaxf(delta, 0.1f + 2e-4f * (len + sqrtf(fdot3(X, X))));
  return true;
}

__device__ __forceinline__ bool diff_blocked(const PathArgs& a, int nlinks, unsigned long long code, TStack& st) {
  ReflCand c;
  const unsigned kind = (unsigned)(code >> kKindShift);
  if (kind == 2u) {
    c = refl_decode(a, nlinks, code);
  } else if (kind == 0u && a.max_trans == 0) {
    c.kind = 5;
    c.link = (int)(code / (unsigned)a.nw);
    c.w = (int)(code % (unsigned)a.nw);
    c.p1 = c.p2 = 0;
  } else {
    return false;
  }
  const WedgeF W = a.wf[c.w];
  const float4 tv = a.txs[c.link / a.nrx], rv = a.rx[c.link % a.nrx];
  const float3 T = f3(tv.x, tv.y, tv.z), R = f3(rv.x, rv.y, rv.z);
  float3 S = T, S1 = T, O = R, O1 = R;
  if (c.kind <= 2) refl2_images(a, c.kind, c.link, a.rplanes[c.p1], a.rplanes[c.p2], S, S1, O, O1);
  else if (c.kind == 3) S = plane_image(a.rplanes[c.p1], T);
  else if (c.kind == 4) O = plane_image(a.rplanes[c.p1], R);
  WedgeSide s, o;
  float3 p;
  side_zr(W, S, s, p);
  side_zr(W, O, o, p);
  if (!(s.r > 0.5f && o.r > 0.5f)) return false;
  const float zq = s.z + (o.z - s.z) * s.r / (s.r + o.r);
  const float3 Qp = edge_point(W, zq);
  float delta = 0.05f + 1e-5f * (s.l + o.l);
  // the path's points between T and R, and the wedge's place among them
  float3 P[5];
  int np = 0, at = 0;
  P[np++] = T;
  float3 X, Y;
  if (c.kind == 0) {
    if (!plane_cross32(a.rplanes[c.p2], S, Qp, Y, delta) || !plane_cross32(a.rplanes[c.p1], S1, Y, X, delta))
      return false;
    P[np++] = X;
    P[np++] = Y;
  } else if (c.kind == 1 || c.kind == 3) {
    if (!plane_cross32(a.rplanes[c.p1], S, Qp, X, delta)) return false;
    P[np++] = X;
  }
  at = np;
  P[np++] = Qp;
  if (c.kind == 2) {
    if (!plane_cross32(a.rplanes[c.p1], Qp, O, X, delta) || !plane_cross32(a.rplanes[c.p2], X, O1, Y, delta))
      return false;
    P[np++] = X;
    P[np++] = Y;
  } else if (c.kind == 1 || c.kind == 4) {
    if (!plane_cross32(a.rplanes[c.kind == 1 ? c.p2 : c.p1], Qp, O, X, delta)) return false;
    P[np++] = X;
  }
  P[np++] = R;
  const int ta = a.wtopo[c.w].ta, tb = a.wtopo[c.w].tb;
  for (int q = 0; q + 1 < np; ++q) {
    const bool ends = q == at || q + 1 == at;  // the wedge's faces do not block the legs at Q
    const float3 dv = f3(P[q + 1].x - P[q].x, P[q + 1].y - P[q].y, P[q + 1].z - P[q].z);
    if (leg_surely_blocked(a.bvh, P[q], dv, delta, a.eps_occ, ends ? ta : -1, ends ? tb : -1, -1, -1, st)) return true;
  }
  return false;
}

__global__ void __launch_bounds__(64) k_diff_unblocked(PathArgs a, int nlinks, unsigned few) {
  extern __shared__ int sstk[];
  TStack st;
  bind_stack(st, sstk, kStackTrace);
  const unsigned n = min(a.ctr->n_dsurv, a.dsurv_cap);
  const int lane = threadIdx.x & 31;
  // few candidates: a few lanes of every warp, so that all SMs share the
  // traversals' latency; many: full warps of consecutive candidates (which
  // come from one warp above, so their legs run close together)
  // Up to `few` candidates all go on (diff_few). They keep their order, in
  // which survivors of one kind stand together: the exact stage's warps then
  // run one kind's code.
  if (n <= few) {
    for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) a.dexact[i] = a.dsurv[i];
    if (blockIdx.x == 0 && threadIdx.x == 0) a.ctr->n_dexact = n;
    return;
  }
  const unsigned nwarp = gridDim.x * (blockDim.x >> 5), per = min(32u, max(1u, (n + nwarp - 1) / nwarp));
  for (unsigned i0 = (blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) * per; i0 < n; i0 += nwarp * per) {
    const unsigned i = i0 + lane;
    const bool mine = lane < (int)per && i < n;
    const unsigned long long code = mine ? a.dsurv[i] : 0ull;
    const bool keep = mine && !diff_blocked(a, nlinks, code, st);
    const unsigned mk = __ballot_sync(0xffffffffu, keep);
    if (!mk) continue;
    unsigned at = 0;
    if (lane == 0) at = atomicAdd(&a.ctr->n_dexact, (unsigned)__popc(mk));
    at = __shfl_sync(0xffffffffu, at, 0) + __popc(mk & ((1u << lane) - 1u));
    if (keep) a.dexact[at] = code;
  }
}

__device__ __forceinline__ d3w mirror_d(d3w x, d3w n, double c) { return x - n * (2.0 * (dotw(n, x) - c)); }

// One survivor with two reflections: the images, the Keller point and the
// wedge rules (chain_geometry with one wedge) and the reflection points on
// the group planes; the member triangles holding those points; everything
// again on the members' own planes (the oracle's mirrors are the static
// triangles); the four real legs (FP32 any-hit; the triangle excluded at a
// reflection point, the wedge's faces at Q); then the field: the
// transmitter's wave along its first real leg, Fresnel at each reflection
// before the wedge in the real directions, the UTD coefficient over the
// unfolded distances, Fresnel at each reflection after it. Record: depth 3.
__device__ __noinline__ void diffract_refl2(const PathArgs& a, unsigned long long code, double k, double lam,
                                            unsigned& ovf, TStack& st) {
  const int w = (int)(code % (unsigned long long)a.nw);
  unsigned long long b = code / (unsigned long long)a.nw;
  const int p2 = (int)(b % (unsigned long long)a.nrp);
  b /= (unsigned long long)a.nrp;
  const int p1 = (int)(b % (unsigned long long)a.nrp);
  b /= (unsigned long long)a.nrp;
  const unsigned long long nlinks = (unsigned long long)a.dntx * a.nrx;
  const int link = (int)(b % nlinks), kind = (int)(b / nlinks);
  const int nb = kind == 0 ? 2 : kind == 1 ? 1 : 0, na = 2 - nb;
  const Wedge& W = a.wedges[w];
  const Wedge* E[1] = {&W};
  const float4 rxv = a.rx[link % a.nrx], txv = a.txs[link / a.nrx];
  const d3w T = D3(txv.x, txv.y, txv.z), R = D3(rxv.x, rxv.y, rxv.z);
  // the planes of the two reflections in path order: the groups', then the members'
  const int pg[2] = {p1, p2};
  d3w pn[2];
  double pc[2];
  int pj[2] = {-1, -1};
  float4 pm[2] = {make_float4(0.f, 0.f, 0.f, 0.f), make_float4(0.f, 0.f, 0.f, 0.f)};
  for (int i = 0; i < 2; ++i) {
    const RPlane& G = a.rplanes[pg[i]];
    pn[i] = D3(G.n[0], G.n[1], G.n[2]);
    pc[i] = G.c;
  }
  d3w X[3], Y[2];
  double ell[2], phip[1], phi[1];
  for (int pass = 0; pass < 2; ++pass) {
    d3w Sim[3], Oim[3];
    Sim[0] = T;
    for (int i = 0; i < nb; ++i) Sim[i + 1] = mirror_d(Sim[i], pn[i], pc[i]);
    Oim[na] = R;
    for (int i = na - 1; i >= 0; --i) Oim[i] = mirror_d(Oim[i + 1], pn[nb + i], pc[nb + i]);
    if (!chain_geometry(E, 1, Sim[nb], Oim[0], X, ell, phip, phi)) return;
    d3w bp = X[1];
    for (int i = nb - 1; i >= 0; --i) {
      if (!leg_plane(Sim[i + 1], bp, pn[i], pc[i], Y[i])) return;
      bp = Y[i];
    }
    d3w ap = X[1];
    for (int i = 0; i < na; ++i) {
      if (!leg_plane(ap, Oim[i], pn[nb + i], pc[nb + i], Y[nb + i])) return;
      ap = Y[nb + i];
    }
    for (int i = 0; i < 2; ++i) {
      d3w v0, v1, v2;
      float4 mj;
      if (pass == 0) {  // the member triangle holding the point: its own plane next
        const RPlane& G = a.rplanes[pg[i]];
        const int exw[2] = {W.ta, W.tb};
        pj[i] = member_at(a, G, Y[i], exw, 2, v0, v1, v2, mj);
        if (pj[i] < 0) return;
        pm[i] = mj;
        pn[i] = unitw(crossw(v1 - v0, v2 - v0));
        pc[i] = dotw(pn[i], v0);
      } else {
        tri64(a, pj[i], v0, v1, v2, mj);
        if (!inside_tri64(v0, v1, v2, Y[i])) return;
      }
    }
  }
  // the real legs: P the path's points, two excluded triangles at each
  d3w P[5];
  int ex[5][2], ny = 0;
  P[ny] = T; ex[ny][0] = ex[ny][1] = -1; ++ny;
  for (int i = 0; i < nb; ++i) { P[ny] = Y[i]; ex[ny][0] = ex[ny][1] = pj[i]; ++ny; }
  P[ny] = X[1]; ex[ny][0] = W.ta; ex[ny][1] = W.tb; ++ny;
  for (int i = 0; i < na; ++i) { P[ny] = Y[nb + i]; ex[ny][0] = ex[ny][1] = pj[nb + i]; ++ny; }
  P[ny] = R; ex[ny][0] = ex[ny][1] = -1; ++ny;
  if (legs_occluded(a, P, ex, ny, ovf, st)) return;
  unsigned fl = 0;
  const d3w u = D3(a.pol.x, a.pol.y, a.pol.z);
  const d3w ip = (X[1] - X[0]) * (1.0 / ell[0]);  // the real direction into Q
  double sn, cs;
  sincos(-k * ell[0], &sn, &cs);
  const zd Ei = Z(cs / ell[0], sn / ell[0]);
  d3w din = nb ? unitw(P[1] - T) : ip;
  const d3w e0 = polw(u, din, fl);
  zv3 Er = {Z(e0.x), Z(e0.y), Z(e0.z)};
  for (int i = 0; i < nb; ++i) {
    const d3w dout = i == nb - 1 ? ip : unitw(P[i + 2] - P[i + 1]);
    Er = reflect_field_d(a, pn[i], pm[i], din, dout, Er);
    din = dout;
  }
  zv3 Ev = {Er.x * Ei, Er.y * Ei, Er.z * Ei};
  {  // the wedge: UTD over the unfolded distances, a spherical wave arriving
    const double s = ell[1], nn = W.n, rhoe = ell[0], rho1 = ell[0], rho2 = ell[0];
    const d3w e = D3(W.e[0], W.e[1], W.e[2]);
    const d3w dd = (X[2] - X[1]) * (1.0 / s);
    const double beta0 = acos(fmax(-1.0, fmin(1.0, dotw(ip, e))));
    const double sb = sin(beta0);
    const d3w php = unitw(crossw(e, ip)) * -1.0, ph = unitw(crossw(e, dd));
    const d3w bpv = crossw(ip, php), bd = crossw(dd, ph);
    const double L = s * (rhoe + s) * rho1 * rho2 * sb * sb / (rhoe * (rho1 + s) * (rho2 + s));
    const float4 ma =
        a.mats[__float_as_int(a.tris[3 * (size_t)DCEM_IDX(a.slot_of_id[DCEM_IDX(W.ta, a.bvh.ntris)], a.bvh.ntris) + 1].w)];
    const float4 mb =
        a.mats[__float_as_int(a.tris[3 * (size_t)DCEM_IDX(a.slot_of_id[DCEM_IDX(W.tb, a.bvh.ntris)], a.bvh.ntris) + 1].w)];
    zd r0s, r0h, rns, rnh;
    fresnel_faces(ma, fabs(sin(phip[0])), mb, fabs(sin(nn * M_PI - phi[0])), a.freq, r0s, r0h, rns, rnh);
    const UtdParts up = utd_parts(nn, phi[0], phip[0], beta0, L, k, fl);
    const zd Ds = utd_coeff(up, r0s, rns), Dh = utd_coeff(up, r0h, rnh);
    sincos(-k * s, &sn, &cs);
    const zd A = Z(cs, sn) * sqrt(rhoe / (s * (rhoe + s)));
    const zd cb = Ds * zvdot(Ev, bpv) * A * -1.0, cp = Dh * zvdot(Ev, php) * A * -1.0;
    Ev = zv3{cb * bd.x + cp * ph.x, cb * bd.y + cp * ph.y, cb * bd.z + cp * ph.z};
    din = dd;
  }
  for (int i = 0; i < na; ++i) {  // reflected after the wedge, toward the real receiver
    const int at = ny - 1 - na + i;
    const d3w dout = unitw(P[at + 1] - P[at]);
    Ev = reflect_field_d(a, pn[nb + i], pm[nb + i], din, dout, Ev);
    din = dout;
  }
  const d3w prx = polw(u, din * -1.0, fl);
  const zd amp = zvdot(Ev, prx) * (lam / (4.0 * M_PI));
  if (diff_lane() != 0) return;  // one lane of the group writes the record
  unsigned uu = atomicAdd(&a.ctr->n_unique, 1u);
  if (uu >= a.ucap) {
    atomicOr(&a.ctr->err, ERR_UNIQUE_OVERFLOW);
    return;
  }
  int ids[3];
  for (int i = 0; i < nb; ++i) ids[i] = pj[i];
  ids[nb] = w | kDiffBit;
  for (int i = 0; i < na; ++i) ids[nb + 1 + i] = pj[nb + i];
  PathRec rec;
  rec.key = seq_key(link % a.nrx, 3, [&](int q) { return ids[q]; });
  rec.rx = link;
  rec.depth = 3;
  rec.ray = -1;
  rec.flags = fl;
  rec.valid = 1;
  rec.pad = 0;
  rec.len = ell[0] + ell[1];
  rec.amp_re = amp.re;
  rec.amp_im = amp.im;
  for (int q = 0; q < kMaxRefl; ++q) {
    rec.tri[q] = q < 3 ? ids[q] : -1;
    rec.pts[q][0] = rec.pts[q][1] = rec.pts[q][2] = 0.0f;
  }
  for (int q = 1; q + 1 < ny; ++q) {
    rec.pts[q - 1][0] = (float)P[q].x;
    rec.pts[q - 1][1] = (float)P[q].y;
    rec.pts[q - 1][2] = (float)P[q].z;
  }
  a.prec[uu] = rec;
  unsigned pos = atomicAdd(&a.bucket_cnt[link], 1u);
  if (pos < (unsigned)a.bucket_cap) a.bucket[(size_t)link * a.bucket_cap + pos] = (int)uu;
  else atomicOr(&a.ctr->err, ERR_BUCKET_OVERFLOW);
  atomicAdd(&a.ctr->n_valid, 1u);
}

// Pass 1 over every (link, wedge) pair: the FP32 pre-test rejects most of
// them; the survivors' indices go to a list (one atomic per warp).
__global__ void __launch_bounds__(256) k_diffract_pre(PathArgs a, int nlinks) {
  const long total = (long)nlinks * a.nw;
  const int lane = threadIdx.x & 31;
  const long stride = (long)gridDim.x * blockDim.x;
  for (long base = (long)blockIdx.x * blockDim.x + (threadIdx.x & ~31); base < total; base += stride) {
    long idx = base + lane;
    bool keep = false;
    if (idx < total) {
      int link = (int)(idx / a.nw), w = (int)(idx - (long)link * a.nw);
      keep = diffract_candidate(a.wf[w], a.txs[link / a.nrx], a.rx[link % a.nrx]);
    }
    unsigned m = __ballot_sync(0xffffffffu, keep);
    if (!m) continue;
    unsigned at = 0;
    if (lane == 0) at = atomicAdd(&a.ctr->n_dsurv, (unsigned)__popc(m));
    at = __shfl_sync(0xffffffffu, at, 0) + __popc(m & ((1u << lane) - 1u));
    if (keep) {
      if (at < a.dsurv_cap) a.dsurv[at] = (unsigned long long)idx;
      else atomicOr(&a.ctr->err, ERR_DIFF_OVERFLOW);
    }
  }
}

// Pass 2 over the survivors: the exact FP64 test, the occlusion legs and the
// UTD field. The SM's FP64 pipe is narrow and a warp instruction costs it the
// same whatever the number of active lanes, but with the few survivors left
// after the occlusion test the pipe is mostly idle (12% busy on the city) and
// the time is the longest lane's chain of dependent operations plus the
// other lanes' divergent branches: so a survivor takes a group of four lanes
// (see utd_parts), survivor i goes to block i mod grid, slot i / grid, and the
// slots fill the warps one group at a time. More survivors than an SM holds
// groups of (64) keep the instruction pipes busy; there a survivor takes one
// lane, and the slots fill one warp after the other (spread over the warps,
// every warp instruction of the FP64 pipe had a few lanes: 767 us for a
// highway with two reflections, 276 survivors an SM, so 548). With 60 an SM
// (the highway with one) a frame takes 859 us on four lanes, 950 on one; with
// 105 (60 vehicles, four transmitters, two reflections) 1524 and 1344.
constexpr int kDiffThreads = 256;
__global__ void __launch_bounds__(kDiffThreads) k_diffract(PathArgs a) {
  extern __shared__ int sstk[];
  TStack st;
  bind_stack(st, sstk, kStackTrace);
  const unsigned n = min(a.ctr->n_dexact, a.dsurv_cap);
  const double k = 2.0 * M_PI * a.freq / 299792458.0, lam = 299792458.0 / a.freq;
  unsigned ovf = 0;
  constexpr unsigned kWarps = kDiffThreads / 32;
  const unsigned lanes = n > kDiffThreads / kDiffLanes * gridDim.x ? 1 : kDiffLanes;
  if (threadIdx.x == 0) diff_lanes = (int)lanes;
  __syncthreads();
  const unsigned slot = lanes == 1 ? threadIdx.x : (threadIdx.x & 31) / lanes * kWarps + (threadIdx.x >> 5);
  for (unsigned i = blockIdx.x + gridDim.x * slot; i < n; i += gridDim.x * (kDiffThreads / lanes)) {
    const unsigned long long c = a.dexact[i];
    const unsigned kind = (unsigned)(c >> kKindShift);
    if (kind == 2u && ((c >> 61) & 1ull)) diffract_refl2(a, c & kRefl2Mask, k, lam, ovf, st);
    else if (kind == 2u) diffract_refl_pair(a, c & ~kReflTag, k, lam, ovf, st);
    else if (kind != 0u) diffract_multi(a, c, k, lam, ovf, st);
    else diffract_pair(a, (long)c, k, lam, ovf, st);
  }
  if (ovf) {
    atomicAdd(&a.ctr->stack_overflow, 1u);
    atomicOr(&a.ctr->err, ERR_STACK);
  }
}

// ---------------------------------------------------------------------------
// per link: sort paths by key, sum in that order, write them out
// ---------------------------------------------------------------------------
constexpr int kReduceThreads = 256;

// Output offsets of many links (above kScanLinks): the valid paths of each
// group of kReduceGroup links, then (more than kReduceGroup groups) an
// exclusive scan of the groups. (One CTA scanning every link took 110 us for
// 65,536 links, each thread walking its own run of counts.)
constexpr int kReduceGroup = 256;
__global__ void __launch_bounds__(kReduceGroup) k_link_sums(const unsigned* __restrict__ cnt, int n, unsigned cap,
                                                            unsigned* __restrict__ sums) {
  const int i = blockIdx.x * kReduceGroup + threadIdx.x;
  unsigned v = i < n ? min(cnt[i], cap) : 0u;
  v = __reduce_add_sync(0xffffffffu, v);
  __shared__ unsigned part[kReduceGroup / 32];
  if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int k = 1; k < kReduceGroup / 32; ++k) v += part[k];
    sums[blockIdx.x] = v;
  }
}
__global__ void __launch_bounds__(1024) k_link_scan(unsigned* __restrict__ sums, int n) {
  __shared__ unsigned part[32];
  __shared__ unsigned carry;
  const int tid = threadIdx.x, lane = tid & 31;
  if (tid == 0) carry = 0u;
  for (int i0 = 0; i0 < n; i0 += 1024) {
    const unsigned v = i0 + tid < n ? sums[i0 + tid] : 0u;
    unsigned x = v;
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    if (lane == 31) part[tid >> 5] = x;
    __syncthreads();
    if (tid < 32) {
      unsigned p = part[tid];
      for (int o = 1; o < 32; o <<= 1) {
        const unsigned y = __shfl_up_sync(0xffffffffu, p, o);
        if (lane >= o) p += y;
      }
      part[tid] = p;
    }
    __syncthreads();
    const unsigned before = carry + (tid >= 32 ? part[(tid >> 5) - 1] : 0u) + x - v;
    if (i0 + tid < n) sums[i0 + tid] = before;
    __syncthreads();
    if (tid == 0) carry += part[31];
    __syncthreads();
  }
}

// The record of a distinct key as it goes to the caller.
__device__ __forceinline__ void write_path(const PathArgs& a, const PathRec& p, unsigned o) {
  if (o >= a.pout_cap) return;
  dcem_path q;
  q.rx = p.rx % a.nrx;
  q.tx = p.rx / a.nrx;
  q.reserved = 0;
  q.depth = p.depth;
  for (int j = 0; j < kMaxRefl; ++j) {
    q.tri[j] = p.tri[j];
    q.pts[j][0] = p.pts[j][0];
    q.pts[j][1] = p.pts[j][1];
    q.pts[j][2] = p.pts[j][2];
  }
  q.flags = p.flags;
  q.ray = p.ray >= 0 ? a.ray_perm[p.ray] : -1;
  q.key = p.key;
  q.len_m = p.len;
  q.delay_s = p.len / 299792458.0;
  q.amp_re = p.amp_re;
  q.amp_im = p.amp_im;
  (o < a.hrec_cap ? a.hrec : a.pout)[o] = q;
}
// A link's sums as field and powers: thread k of the first half of 2 n
// threads takes link r0 + k's field and coherent power, of the second half
// its incoherent power (a logarithm is some 60 dependent FP64 operations, so
// the block's links take theirs side by side).
__device__ __forceinline__ void write_links(const PathArgs& a, int r0, int n, const double (*sum)[3]) {
  const int tid = threadIdx.x;
  if (tid >= 2 * n) return;
  const int k = tid < n ? tid : tid - n, r = r0 + k;
  const double fr = sum[k][0], fi = sum[k][1], w = tid < n ? fr * fr + fi * fi : sum[k][2];
  if (tid < n && a.out_field) {
    a.out_field[2 * (size_t)r] = fr;
    a.out_field[2 * (size_t)r + 1] = fi;
  }
  double* out = tid < n ? a.out_pc : a.out_pi;
  if (out) out[r] = 10.0 * log10(a.tx_power * w) + 30.0;
}

// One warp per link with up to 32 paths (nearly all: the keys are sorted and
// the sums formed in registers), then the block together for each link with
// more. The sums' order is one for both: position i of the sorted paths goes
// to partial sum i mod 256, in order, then a fixed binary tree over the 256
// partial sums -- whose upper levels add zeros when there are few paths, so
// the warp takes the last five only. One CTA per link took 548 us for 65,536
// links with 21,700 paths. A block takes `per` links: eight, or one while
// there are few links, which may then hold dozens of paths each (the office:
// 48 links with 14 paths on average, 12 us one a block, 41 us eight).
constexpr int kReduceWarps = kReduceThreads / 32;
__global__ void __launch_bounds__(kReduceThreads) k_reduce(PathArgs a, int nlinks, int per) {
  extern __shared__ unsigned long long skey[];   // bucket_cap keys, then bucket_cap ints
  int* sidx = reinterpret_cast<int*>(skey + a.bucket_cap);
  __shared__ double red[3][kReduceThreads], sums[kReduceWarps][3];
  __shared__ unsigned scnt[kReduceWarps], part[kReduceWarps];
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int r0 = blockIdx.x * per, rw = wid < per ? r0 + wid : nlinks;
  const unsigned cap = (unsigned)a.bucket_cap;
  // paths of the links before this block's: the groups' offsets or sums, and
  // the links of the own group (of all links when there are no groups)
  const int g = r0 / kReduceGroup, ng = (nlinks + kReduceGroup - 1) / kReduceGroup;
  unsigned before = 0;
  if (a.link_off) {
    if (ng > kReduceGroup) before = tid == 0 ? a.link_off[g] : 0u;
    else before = tid < g ? a.link_off[tid] : 0u;
  }
  for (int q = (a.link_off ? g * kReduceGroup : 0) + tid; q < r0; q += kReduceThreads) before += min(a.bucket_cnt[q], cap);
  before = __reduce_add_sync(0xffffffffu, before);
  const int cnt = rw < nlinks ? (int)min(a.bucket_cnt[rw], cap) : 0;
  if (lane == 0) {
    part[wid] = before;
    scnt[wid] = (unsigned)cnt;
  }
  // the warp's keys, sorted across its lanes (an odd-even merge network over
  // the next power of two)
  unsigned long long key = ~0ull;
  int idx = -1;
  if (cnt <= 32 && lane < cnt) {
    idx = DCEM_IDX(a.bucket[(size_t)rw * a.bucket_cap + lane], a.ucap);
    key = a.prec[idx].key;
  }
  if (cnt <= 32) {
    for (int k = 2; k < 2 * cnt; k <<= 1)
      for (int j = k >> 1; j > 0; j >>= 1) {
        const unsigned long long ok = __shfl_xor_sync(0xffffffffu, key, j);
        const int oi = __shfl_xor_sync(0xffffffffu, idx, j);
        const bool low = (lane & j) == 0, up = (lane & k) == 0;
        if (low == up ? ok < key : ok > key) {
          key = ok;
          idx = oi;
        }
      }
  }
  __syncthreads();
  unsigned off = 0;
  for (int k = 0; k < kReduceWarps; ++k) off += part[k];
  const unsigned base = off;
  for (int k = 0; k < wid; ++k) off += scnt[k];
  if (cnt <= 32 && rw < nlinks) {
    double sre = 0.0, sim = 0.0, sinc = 0.0;
    if (lane < cnt) {
      const PathRec& p = a.prec[idx];
      sre += p.amp_re;
      sim += p.amp_im;
      sinc += p.amp_re * p.amp_re + p.amp_im * p.amp_im;
      write_path(a, p, off + (unsigned)lane);
    }
    for (int s = 16; s > 0; s >>= 1) {
      sre += __shfl_down_sync(0xffffffffu, sre, s);
      sim += __shfl_down_sync(0xffffffffu, sim, s);
      sinc += __shfl_down_sync(0xffffffffu, sinc, s);
    }
    if (lane == 0) {
      sums[wid][0] = sre;
      sums[wid][1] = sim;
      sums[wid][2] = sinc;
    }
  }
  off = base;
  for (int k = 0; k < per; ++k) {  // links with more paths, the block together
    const int n = (int)scnt[k];
    if (n > 32) {
      const int r = r0 + k;
      int np2 = 1;
      while (np2 < n) np2 <<= 1;
      __syncthreads();
      for (int i = tid; i < np2; i += kReduceThreads) {
        if (i < n) {
          int u = DCEM_IDX(a.bucket[(size_t)r * a.bucket_cap + i], a.ucap);
          skey[i] = a.prec[u].key;
          sidx[i] = u;
        } else {
          skey[i] = ~0ull;
          sidx[i] = -1;
        }
      }
      __syncthreads();
      for (int kk = 2; kk <= np2; kk <<= 1) {
        for (int j = kk >> 1; j > 0; j >>= 1) {
          for (int i = tid; i < np2; i += kReduceThreads) {
            int ixj = i ^ j;
            if (ixj > i) {
              unsigned long long x = skey[i], y = skey[ixj];
              bool up = (i & kk) == 0;
              if ((x > y) == up) {
                skey[i] = y; skey[ixj] = x;
                int t = sidx[i]; sidx[i] = sidx[ixj]; sidx[ixj] = t;
              }
            }
          }
          __syncthreads();
        }
      }
      double sre = 0.0, sim = 0.0, sinc = 0.0;
      for (int i = tid; i < n; i += kReduceThreads) {
        const PathRec& p = a.prec[sidx[i]];
        sre += p.amp_re;
        sim += p.amp_im;
        sinc += p.amp_re * p.amp_re + p.amp_im * p.amp_im;
        write_path(a, p, off + (unsigned)i);
      }
      red[0][tid] = sre;
      red[1][tid] = sim;
      red[2][tid] = sinc;
      __syncthreads();
      for (int s = kReduceThreads / 2; s > 0; s >>= 1) {
        if (tid < s)
          for (int q = 0; q < 3; ++q) red[q][tid] += red[q][tid + s];
        __syncthreads();
      }
      if (tid < 3) sums[k][tid] = red[tid][0];
    }
    off += scnt[k];
  }
  __syncthreads();
  write_links(a, r0, min(per, nlinks - r0), sums);
}

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------
cudaError_t launch_dedupe(const PathArgs& a, int grid, cudaStream_t st) {
  k_dedupe_insert<<<grid, 256, 0, st>>>(a);
  k_dedupe_unique<<<grid, 256, 0, st>>>(a);
  return cudaGetLastError();
}

// Candidates that go to the exact stage without the occlusion test. The stage
// takes a few an SM side by side, its time is one candidate's either way, and
// the longest of the legs here takes 50 us; a wall in every other leg makes the
// test pay from 16 candidates an SM on (us a frame with lines at 0, 16 and 64:
// 4 x 4 city blocks, 12 candidates an SM 661, 691, 683, 20 an SM 784, 785, 810;
// 5 x 5, two wedges, 25 an SM 1371, 1376, 1486; 3 x 3, 2 an SM 325, 305, 303).
// Open scenes' legs are hardly ever blocked: none is tested. Without reflector
// planes there is no telling: 64 (a highway, chains of two, 26 an SM: 2722 with
// the line at 16, 2632 at 64; 2 km with 16 transmitters, 24 an SM: 481 and 424).
static unsigned diff_few(const PathArgs& a, int sms) {
  if (a.open) return 0xffffffffu;
  return (unsigned)sms * (a.nrp > 0 ? 16u : 64u);
}

cudaError_t launch_hidden_planes(const PathArgs& a, unsigned* cnt, cudaStream_t st) {
  cudaError_t e = cudaMemsetAsync(cnt, 0, 2 * sizeof(unsigned), st);
  if (e != cudaSuccess || a.nrp <= 0) return e;
  const int n = std::min(a.nrp, kHiddenSample);
  k_hidden_planes<<<dim3(n, n), 1, kStackTrace * sizeof(int), st>>>(a, cnt);
  return cudaGetLastError();
}

cudaError_t launch_diffract(const PathArgs& args, int nlinks, int sms, cudaStream_t st) {
  PathArgs a = args;
  if (!a.wedges || a.nw <= 0) return cudaSuccess;
  k_wedge_geom<<<(a.nw + 31) / 32, 32, 0, st>>>(a.tris, a.slot_of_id, a.wtopo, a.nw, a.wedges, a.wf);
  if (a.rplanes && a.nrp > 0)
    k_wedge_boxes<<<(a.nw + 255) / 256, 256, 0, st>>>(a.wf, a.wperm, a.nw, a.wgbox);
  if (nlinks > 0) {
    if (a.vis) {  // what the end points see: with reflector planes or chains
      const bool test = a.nrp == 0 || (!a.open && (a.drefl2 || a.diff_order >= 2));
      const long nvis = (long)(nlinks / a.nrx + a.nrx) * ((a.nrp + 31) / 32 + a.nwc);
      k_diff_visible<<<(int)std::min<long>((nvis + 1) / 2, 16L * sms), 64, 64 * kStackTrace * sizeof(int), st>>>(
          a, nlinks / a.nrx, test);
    }
    long total = (long)nlinks * a.nw;
    long g = std::min<long>((total + 255) / 256, 8L * sms);
    k_diffract_pre<<<(int)std::max<long>(g, 1), 256, 0, st>>>(a, nlinks);
    if (a.rplanes && a.nrp > 0) {
      const int ntx = nlinks / a.nrx;
      a.rsub = std::max(1, std::min((a.nrx + 7) / 8, a.nrx / ntx));
      auto warps = [&](long n) { return (int)std::max<long>(std::min<long>((n + 7) / 8, 8L * sms), 1); };
      if (a.drefl2) {
        cudaMemsetAsync(a.wobs_cnt, 0, sizeof(unsigned) * (size_t)a.nw, st);
        cudaMemsetAsync(a.rmask, 0, sizeof(unsigned) * (size_t)(ntx + a.nrx) * a.nrp * a.nwc, st);
      }
      k_diff_visible_any<<<2, 256, 0, st>>>(a, ntx);
      // parts of an item while there are fewer items than warps
      const long room = 64L * sms;
      auto parts = [&](long n) { return (int)std::max<long>(1, std::min<long>(8, room / std::max<long>(n, 1))); };
      const long single = ((long)ntx * a.rsub + a.nrx) * a.nrp, lists = (long)a.nrx * a.nrp;
      k_refl_single<<<warps(single * parts(single)), 256, 0, st>>>(a, ntx, nlinks, parts(single));
      if (a.drefl2) {
        k_refl_room<<<(a.nw + 255) / 256, 256, 0, st>>>(a);
        k_refl_lists<<<warps(lists * parts(lists)), 256, 0, st>>>(a, ntx, parts(lists));
        k_refl_join<<<warps((long)ntx * a.nrp * a.nwc * kJoinParts), 256, 0, st>>>(a, ntx, nlinks);
        auto items = [&] { return ((long)ntx * a.rsub + a.nrx) * a.nrp * a.nrp; };
        if (a.open && nlinks <= 2 * (ntx + a.nrx)) {
          k_refl_direct<<<warps(2L * nlinks * a.nrp * a.nrp), 256, 0, st>>>(a, ntx, nlinks);
        } else {
          if (items() > 32 * room) a.rsub = std::max(1, a.rsub / 4);
          const int per = (int)std::max<long>(1, std::min<long>(32, items() / room));
          k_refl_double<<<warps((items() + per - 1) / per), 256, 0, st>>>(a, ntx, nlinks, per);
        }
      }
    }
    PathArgs b = a;  // chains: transmitters, and the reflector planes applied to them
    if (a.open) b.vis = nullptr;  // nothing to look up: the rows hold what the pre-tests know
    b.dntx = nlinks / a.nrx;
    b.nrpr = a.rplanes && a.diff_order >= 2 ? a.nrp : 0;
    if (a.diff_order >= 2 && a.nw > 1) {
      int nsrc = b.dntx * (1 + b.nrpr);
      long tp = (long)nsrc * a.nw * a.nw;
      cudaMemsetAsync(a.drel, 0, sizeof(unsigned) * (((size_t)a.nw * a.nw + 31) / 32), st);
      if (a.dobs1) cudaMemsetAsync(a.dsecond, 0, sizeof(unsigned) * (size_t)((a.nw + 31) / 32), st);
      const size_t ssm = 256 * kStackTrace * sizeof(int);
      const long rw = (long)a.nw * ((a.nw + 31) / 32);
      k_diff_rel<<<(int)std::max<long>(std::min<long>((rw + 7) / 8, 8L * sms), 1), 256, ssm, st>>>(b);
      k_diff_pairs<<<(int)std::max<long>(std::min<long>((tp + 255) / 256, 8L * sms), 1), 256, 0, st>>>(b, nsrc);
      if (a.dmid && a.rplanes && a.nrp > 0) {
        long nblk = (long)b.dntx * a.nw * a.nrp;
        k_diff_mid_pairs<<<(int)std::max<long>(std::min<long>((nblk + 7) / 8, 8L * sms), 1), 256, 0, st>>>(b);
      }
      if (a.diff_order >= 3) {
        k_diff_triples<<<8 * sms, 256, 0, st>>>(b);
        if (a.dobs1) k_diff_stage1<<<8 * sms, 256, 0, st>>>(b);
      }
      k_diff_multi_pre<<<8 * sms, 256, 256 * kStackTrace * sizeof(int), st>>>(b);
    }
    k_diff_unblocked<<<8 * sms, 64, 64 * kStackTrace * sizeof(int), st>>>(b, nlinks, diff_few(a, sms));
    k_diffract<<<sms, kDiffThreads, kDiffThreads * kStackTrace * sizeof(int), st>>>(b);
  }
  return cudaGetLastError();
}

cudaError_t launch_sticky_probe(const PathArgs& a, int grid, cudaStream_t st) {
  k_sticky_probe<<<grid, 256, 0, st>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_validate(const PathArgs& a, int nlinks, int grid, cudaStream_t st) {
  const size_t osm = 64 * kStackTrace * sizeof(int);
  if (nlinks <= kFewLinks) {
    if (a.prec_df) k_validate<df><<<grid, kFieldThreads, osm, st>>>(a);
    else k_validate<double><<<grid, kFieldThreads, osm, st>>>(a);
    return cudaGetLastError();
  }
  const size_t gsm = 64 * kStackSmall * sizeof(int);
  if (a.prec_df) k_val_geom<df><<<4 * grid, 64, gsm, st>>>(a);
  else k_val_geom<double><<<4 * grid, 64, gsm, st>>>(a);
  // (key, sub-segment) items: one or two lanes of every warp while they are
  // few, so that a warp waits for few different traversals
  k_val_occ<<<4 * grid, 64, osm, st>>>(a);
  k_val_field<<<4 * grid, kFieldThreads, 0, st>>>(a);
  return cudaGetLastError();
}

// The next frame's table: link key -> record index of each distinct key.
__global__ void k_vcache_build(PathArgs a) {
  unsigned nu = min(a.ctr->n_unique, a.ucap);
  const unsigned mask = a.vc_cap - 1u;
  for (unsigned u = blockIdx.x * blockDim.x + threadIdx.x; u < nu; u += gridDim.x * blockDim.x) {
    unsigned long long key = a.ckey[u];
    if (!key) continue;
    unsigned slot = (unsigned)(key & mask);
    for (unsigned p = 0; p < a.vc_cap; ++p) {
      unsigned long long prev = atomicCAS(&a.vc_next_key[slot], 0ull, key);
      if (prev == 0ull || prev == key) {
        a.vc_next_u[slot] = u;
        break;
      }
      slot = (slot + 1u) & mask;
    }
  }
}

cudaError_t launch_vcache_build(const PathArgs& a, int grid, cudaStream_t st) {
  k_vcache_build<<<grid, 256, 0, st>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_reduce(const PathArgs& a, int nlinks, cudaStream_t st) {
  if (nlinks <= 0) return cudaSuccess;
  if (a.link_off) {
    const int ng = (nlinks + kReduceGroup - 1) / kReduceGroup;
    k_link_sums<<<ng, kReduceGroup, 0, st>>>(a.bucket_cnt, nlinks, (unsigned)a.bucket_cap, a.link_off);
    if (ng > kReduceGroup) k_link_scan<<<1, 1024, 0, st>>>(a.link_off, ng);
  }
  size_t smem = (size_t)a.bucket_cap * (sizeof(unsigned long long) + sizeof(int));
  static bool attr = false;
  if (!attr) {
    cudaFuncSetAttribute(k_reduce, cudaFuncAttributeMaxDynamicSharedMemorySize, 160 * 1024);
    attr = true;
  }
  const int per = nlinks <= 1024 ? 1 : kReduceWarps;
  k_reduce<<<(nlinks + per - 1) / per, kReduceThreads, smem, st>>>(a, nlinks, per);
  return cudaGetLastError();
}

DCEM_CHECKS_TAKER(checks_take_paths)

}  // namespace dcem
