// grad.cu -- derivatives of the per-receiver field over a fixed path
// topology, with respect to each material's (eps_r, sigma) and each rigid
// object's (x, y) translation.
//
// The amplitude of a path is Sec. III steps 3, 4 and 6 again: image sources
// of the transmitter in the planes of the path's triangles, back-trace from
// the receiver to the reflection points, Fresnel reflection (TE/TM) with
// vector polarisation, and the amplitude of Eq. 1 with the Friis spreading of
// Eq. 3. Here it is evaluated in FP64 forward-mode dual numbers (value and
// derivative along one parameter): translating an object moves the vertices
// of its triangles, a material parameter enters through the complex
// permittivity. One work item is one (path, parameter) pair, where the
// parameter is that of one bounce's material or object; the first bounce that
// uses a material (object) seeds every bounce that shares it, later ones
// contribute no item. The per-receiver sums run in path order, one warp per
// receiver, so results are the same in every run.
#include "grad.cuh"

#include <algorithm>

namespace dcem {
namespace {

constexpr double kC0 = 299792458.0;
constexpr double kEps0 = 8.8541878128e-12;
constexpr double kPi = 3.141592653589793;

struct Dd {
  double v, d;
};
__device__ __forceinline__ Dd cst(double v) { return Dd{v, 0.0}; }
__device__ __forceinline__ Dd operator+(Dd a, Dd b) { return Dd{a.v + b.v, a.d + b.d}; }
__device__ __forceinline__ Dd operator-(Dd a, Dd b) { return Dd{a.v - b.v, a.d - b.d}; }
__device__ __forceinline__ Dd operator-(Dd a) { return Dd{-a.v, -a.d}; }
__device__ __forceinline__ Dd operator*(Dd a, Dd b) { return Dd{a.v * b.v, a.d * b.v + a.v * b.d}; }
__device__ __forceinline__ Dd operator*(double s, Dd a) { return Dd{s * a.v, s * a.d}; }
__device__ __forceinline__ Dd operator/(Dd a, Dd b) {
  double q = a.v / b.v;
  return Dd{q, (a.d - q * b.d) / b.v};
}
__device__ __forceinline__ Dd dsqrt(Dd a) {
  double r = sqrt(a.v);
  return Dd{r, r > 0.0 ? a.d / (2.0 * r) : 0.0};
}
__device__ __forceinline__ Dd dabs(Dd a) { return a.v < 0.0 ? -a : a; }

struct V3 {
  Dd x, y, z;
};
__device__ __forceinline__ V3 vc(double x, double y, double z) { return V3{cst(x), cst(y), cst(z)}; }
__device__ __forceinline__ V3 operator+(const V3& a, const V3& b) { return V3{a.x + b.x, a.y + b.y, a.z + b.z}; }
__device__ __forceinline__ V3 operator-(const V3& a, const V3& b) { return V3{a.x - b.x, a.y - b.y, a.z - b.z}; }
__device__ __forceinline__ V3 operator-(const V3& a) { return V3{-a.x, -a.y, -a.z}; }
__device__ __forceinline__ V3 scl(Dd s, const V3& a) { return V3{s * a.x, s * a.y, s * a.z}; }
__device__ __forceinline__ Dd vdot(const V3& a, const V3& b) { return a.x * b.x + a.y * b.y + a.z * b.z; }
__device__ __forceinline__ V3 vcross(const V3& a, const V3& b) {
  return V3{a.y * b.z - a.z * b.y, a.z * b.x - a.x * b.z, a.x * b.y - a.y * b.x};
}
__device__ __forceinline__ Dd vnorm(const V3& a) { return dsqrt(vdot(a, a)); }
__device__ __forceinline__ V3 vunit(const V3& a) {
  Dd n = vnorm(a);
  return V3{a.x / n, a.y / n, a.z / n};
}

struct Cd {
  Dd re, im;
};
__device__ __forceinline__ Cd cre(Dd r) { return Cd{r, cst(0.0)}; }
__device__ __forceinline__ Cd operator+(const Cd& a, const Cd& b) { return Cd{a.re + b.re, a.im + b.im}; }
__device__ __forceinline__ Cd operator-(const Cd& a, const Cd& b) { return Cd{a.re - b.re, a.im - b.im}; }
__device__ __forceinline__ Cd operator*(const Cd& a, const Cd& b) {
  return Cd{a.re * b.re - a.im * b.im, a.re * b.im + a.im * b.re};
}
__device__ __forceinline__ Cd operator*(Dd s, const Cd& a) { return Cd{s * a.re, s * a.im}; }
__device__ __forceinline__ Cd operator/(const Cd& a, const Cd& b) {
  Dd den = b.re * b.re + b.im * b.im;
  return Cd{(a.re * b.re + a.im * b.im) / den, (a.im * b.re - a.re * b.im) / den};
}
// principal square root; derivative dz / (2 w)
__device__ __forceinline__ Cd csqrt_d(const Cd& z) {
  double x = z.re.v, y = z.im.v;
  double r = hypot(x, y), wr, wi;
  if (x >= 0.0) {
    double t = sqrt(0.5 * (r + x));
    wr = t;
    wi = t > 0.0 ? y / (2.0 * t) : 0.0;
  } else {
    double t = sqrt(0.5 * (r - x));
    wr = fabs(y) / (2.0 * t);
    wi = copysign(t, y);
  }
  double m = 2.0 * (wr * wr + wi * wi);
  double dr = m > 0.0 ? (z.re.d * wr + z.im.d * wi) / m : 0.0;
  double di = m > 0.0 ? (z.im.d * wr - z.re.d * wi) / m : 0.0;
  return Cd{Dd{wr, dr}, Dd{wi, di}};
}

struct C3 {
  Cd x, y, z;
};
__device__ __forceinline__ Cd cdotv(const C3& e, const V3& v) {
  return v.x * e.x + v.y * e.y + v.z * e.z;
}

// unit vector of u - (u.d) d; u parallel to d falls back to a fixed axis
__device__ __forceinline__ V3 pol_dir(const V3& u, const V3& d) {
  V3 p = u - scl(vdot(u, d), d);
  if (vnorm(p).v < 1e-9) {
    V3 a = fabs(d.x.v) < 0.9 ? vc(1, 0, 0) : vc(0, 1, 0);
    p = a - scl(vdot(a, d), d);
  }
  return vunit(p);
}

// Gamma_TE, Gamma_TM of a half-space with eps_c = eps_r - j sigma / (w eps0)
__device__ __forceinline__ void fresnel_d(Dd eps_r, Dd sigma, bool pec, double freq, Dd ct, Cd& te, Cd& tm) {
  if (pec) {
    te = cre(cst(-1.0));
    tm = cre(cst(1.0));
    return;
  }
  Cd ec{eps_r, (-1.0 / (2.0 * kPi * freq * kEps0)) * sigma};
  Dd sin2 = cst(1.0) - ct * ct;
  Cd root = csqrt_d(ec - cre(sin2));
  Cd c = cre(ct);
  te = (c - root) / (c + root);
  Cd ecc = ec * c;
  tm = (ecc - root) / (ecc + root);
}

__device__ __forceinline__ V3 vertex(const float4& f, int seed_axis) {
  V3 v = vc(f.x, f.y, f.z);
  if (seed_axis == 0) v.x.d = 1.0;
  if (seed_axis == 1) v.y.d = 1.0;
  return v;
}

// Amplitude of path P and its derivative along one parameter: kind 0/1 =
// eps_r / sigma of material `sid`, 2/3 = x / y translation of object `sid`,
// -1 = value only. False if the triangle sequence has no reflection geometry.
__device__ bool path_amp(const GradArgs& g, const dcem_path& P, int kind, int sid, Cd& amp) {
  const int k = P.depth;
  V3 tx = vc(g.tx[0], g.tx[1], g.tx[2]);
  float4 rv = g.rx[P.rx];
  V3 rx = vc(rv.x, rv.y, rv.z);
  V3 img[kMaxRefl + 1], X[kMaxRefl + 2], V0[kMaxRefl], Nn[kMaxRefl];
  Dd er[kMaxRefl], sg[kMaxRefl];
  bool pec[kMaxRefl];
  img[0] = tx;
  for (int j = 0; j < k; ++j) {
    int id = P.tri[j];
    const float4* t = g.tris + 3 * (size_t)g.slot_of_id[id];
    int ax = (kind >= 2 && g.tri_obj[id] == sid) ? kind - 2 : -1;
    V3 v0 = vertex(t[0], ax), v1 = vertex(t[1], ax), v2 = vertex(t[2], ax);
    V3 n = vcross(v1 - v0, v2 - v0);
    Dd nn = vdot(n, n);
    if (!(nn.v > 0.0)) return false;
    Dd h = vdot(img[j] - v0, n) / nn;
    img[j + 1] = img[j] - scl(2.0 * h, n);
    V0[j] = v0;
    Nn[j] = n;
    int m = g.tri_mat[id];
    float4 mt = g.mats[m];
    er[j] = cst(mt.x);
    sg[j] = cst(mt.y);
    pec[j] = mt.z != 0.0f;
    if (kind == 0 && m == sid) er[j].d = 1.0;
    if (kind == 1 && m == sid) sg[j].d = 1.0;
  }
  X[0] = tx;
  X[k + 1] = rx;
  for (int j = k; j >= 1; --j) {
    V3 dir = img[j] - X[j + 1];
    Dd den = vdot(dir, Nn[j - 1]);
    if (den.v == 0.0) return false;
    Dd s = vdot(V0[j - 1] - X[j + 1], Nn[j - 1]) / den;
    X[j] = X[j + 1] + scl(s, dir);
  }
  Dd L = cst(0.0);
  for (int j = 0; j <= k; ++j) L = L + vnorm(X[j + 1] - X[j]);
  if (!(L.v > 0.0)) return false;
  // field with vector polarisation
  V3 u = vc(g.pol[0], g.pol[1], g.pol[2]);
  V3 e0 = pol_dir(u, vunit(X[1] - X[0]));
  C3 E{cre(e0.x), cre(e0.y), cre(e0.z)};
  for (int j = 1; j <= k; ++j) {
    V3 din = vunit(X[j] - X[j - 1]), dout = vunit(X[j + 1] - X[j]);
    V3 nh = vunit(Nn[j - 1]);
    Dd ct = dabs(vdot(din, nh));
    V3 sv = vcross(din, nh);
    Dd sn = vnorm(sv);
    if (sn.v < 1e-12) {  // normal incidence: a fixed unit vector perpendicular to n
      V3 a = fabs(nh.x.v) < 0.9 ? vc(1, 0, 0) : vc(0, 1, 0);
      sv = vunit(vcross(nh, a));
    } else {
      sv = V3{sv.x / sn, sv.y / sn, sv.z / sn};
    }
    V3 pin = vcross(sv, din), pout = vcross(sv, dout);
    Cd gte, gtm;
    fresnel_d(er[j - 1], sg[j - 1], pec[j - 1], g.freq, ct, gte, gtm);
    Cd es = gte * cdotv(E, sv), ep = gtm * cdotv(E, pin);
    E = C3{sv.x * es + pout.x * ep, sv.y * es + pout.y * ep, sv.z * es + pout.z * ep};
  }
  V3 prx = pol_dir(u, -vunit(X[k + 1] - X[k]));
  double lam = kC0 / g.freq, kw = 2.0 * kPi * g.freq / kC0;
  double sp, cp;
  sincos(kw * L.v, &sp, &cp);
  Cd ph{Dd{cp, -kw * L.d * sp}, Dd{-sp, -kw * L.d * cp}};  // e^{-j k L}
  Cd a = cdotv(E, prx) * ph;
  amp = cst(lam / (4.0 * kPi)) * (a / cre(L));
  return true;
}

__global__ void k_grad_items(GradArgs g) {
  long total = (long)g.n_paths * g.W;
  for (long it = blockIdx.x * (long)blockDim.x + threadIdx.x; it < total; it += (long)gridDim.x * blockDim.x) {
    int p = (int)(it / g.W), slot = (int)(it - (long)p * g.W);
    const dcem_path& P = g.paths[p];
    g.param[it] = -1;
    bool good = P.depth >= 0 && P.depth <= g.max_refl && P.rx >= 0 && P.rx < g.nrx;
    for (int j = 0; good && j < P.depth; ++j) good = P.tri[j] >= 0 && P.tri[j] < g.ntri;
    if (!good) {
      if (slot == 0) atomicOr(g.err, 2u);
      continue;
    }
    Cd amp;
    if (slot == 0) {
      if (p > 0 && g.paths[p - 1].rx > P.rx) atomicOr(g.err, 1u);
      if (!path_amp(g, P, -1, -1, amp)) {
        atomicOr(g.err, 4u);
        continue;
      }
      g.items[it] = make_double2(amp.re.v, amp.im.v);
      g.param[it] = -2;
      continue;
    }
    int j = (slot - 1) >> 2, w = (slot - 1) & 3;
    if (j >= P.depth) continue;
    int id = P.tri[j], sid, theta;
    if (w < 2) {
      sid = g.tri_mat[id];
      if (g.mats[sid].z != 0.0f) continue;  // perfect conductor: no material dependence
      bool first = true;
      for (int q = 0; q < j; ++q) first = first && g.tri_mat[P.tri[q]] != sid;
      if (!first) continue;
      theta = 2 * sid + w;
    } else {
      sid = g.tri_obj[id];
      if (sid < 0) continue;
      bool first = true;
      for (int q = 0; q < j; ++q) first = first && g.tri_obj[P.tri[q]] != sid;
      if (!first) continue;
      theta = 2 * g.nmat + 2 * sid + (w - 2);
    }
    if (!path_amp(g, P, w, sid, amp)) continue;  // reported by the value item
    g.items[it] = make_double2(amp.re.d, amp.im.d);
    g.param[it] = theta;
  }
}

// One block per receiver: its paths are contiguous (grouped by rx). The items
// of a path belong to distinct parameters, so the block's threads add a
// path's items side by side, path after path (every sum in path order), to
// accumulators in shared memory while the parameters fit there. (One lane
// adding all items in global memory took 108 us for 256 receivers.)
constexpr int kGradThreads = 128;
__global__ void __launch_bounds__(kGradThreads) k_grad_reduce(GradArgs g, int nparam) {
  extern __shared__ double sacc[];
  __shared__ int range[2];
  __shared__ double se[2];
  const int r = blockIdx.x, tid = threadIdx.x;
  if (tid < 2) {  // the first path with rx >= r, and with rx > r
    int a = 0, b = g.n_paths;
    while (a < b) {
      const int m = (a + b) >> 1;
      if (g.paths[m].rx < r + tid) a = m + 1; else b = m;
    }
    range[tid] = a;
  }
  double* out = g.dfield ? g.dfield + 2 * (size_t)r * nparam : nullptr;
  double* df = nparam <= kGradShared ? sacc : out;
  if (g.need_d)
    for (int t = tid; t < 2 * nparam; t += kGradThreads) df[t] = 0.0;
  __syncthreads();
  const int lo = range[0], hi = range[1];
  double er = 0.0, ei = 0.0;
  for (int p = lo; p < hi; ++p) {
    for (int q = tid; q < (g.need_d ? g.W : 1); q += kGradThreads) {
      const long it = (long)p * g.W + q;
      const int pm = g.param[it];
      if (pm == -2) {
        const double2 v = g.items[it];
        er += v.x;
        ei += v.y;
      } else if (pm >= 0) {
        const double2 v = g.items[it];
        df[2 * pm] += v.x;
        df[2 * pm + 1] += v.y;
      }
    }
    __syncthreads();
  }
  if (tid == 0) {
    if (g.field) {
      g.field[2 * (size_t)r] = er;
      g.field[2 * (size_t)r + 1] = ei;
    }
    const double p = er * er + ei * ei;
    if (g.pcoh) g.pcoh[r] = p > 0.0 ? 10.0 * log10(g.tx_power * p) + 30.0 : -INFINITY;
    se[0] = er;
    se[1] = ei;
  }
  if (!g.need_d) return;
  __syncthreads();
  er = se[0];
  ei = se[1];
  if (out && df != out)
    for (int t = tid; t < 2 * nparam; t += kGradThreads) out[t] = df[t];
  if (g.dpcoh) {
    // P = P_t |E|^2: dP = 2 P_t Re(conj(E) dE), d(dBm) = 10 / ln 10 * dP / P
    const double p = er * er + ei * ei;
    for (int t = tid; t < nparam; t += kGradThreads) {
      const double dr = df[2 * t], di = df[2 * t + 1];
      const double dp = 2.0 * (er * dr + ei * di);
      g.dpcoh[(size_t)r * nparam + t] = p > 0.0 && (dr != 0.0 || di != 0.0) ? 4.342944819032518 * dp / p : 0.0;
    }
  }
}

// ---------------------------------------------------------------------------
// reverse mode: eight lanes per path
// ---------------------------------------------------------------------------
// The forward sweep evaluates the path's geometry in FP64 (image sources,
// back-trace: one lane, the only long chain) and keeps its vertices
// X_0 .. X_{k+1}. A bounce's field quantities (directions, polarisation
// basis, Fresnel coefficients) depend on the vertices only, so each lane
// forms those of its own bounce; carrying the field forward and its adjoint
// back through them is short; then each lane differentiates its own bounce,
// and the parameters' tangents are shared out likewise. Everything of a path
// waits in shared memory. FP64 runs at a small fraction of the FP32 rate and
// a path is a chain of dependent operations: one thread per path that
// recomputed every earlier bounce for each one took 385 us a call (300 paths,
// up to 4 bounces). The backward sweep carries d a / d v for every
// intermediate v (complex: the field is holomorphic in its complex
// intermediates) from a back to the vertices and to each bounce's complex
// permittivity. A material's eps_r and sigma take d a / d eps_c directly; an
// object's translation moves the planes of its triangles, whose effect on the
// vertices is a tangent of the (cheap, real) image geometry, contracted with
// d a / d X.
struct R3 {
  double x, y, z;
};
__device__ __forceinline__ R3 r3(double x, double y, double z) { return R3{x, y, z}; }
__device__ __forceinline__ R3 operator+(R3 a, R3 b) { return r3(a.x + b.x, a.y + b.y, a.z + b.z); }
__device__ __forceinline__ R3 operator-(R3 a, R3 b) { return r3(a.x - b.x, a.y - b.y, a.z - b.z); }
__device__ __forceinline__ R3 operator*(R3 a, double s) { return r3(a.x * s, a.y * s, a.z * s); }
// (not fused: path lengths stay equal to those of a plain FP64 evaluation, and
// the phase is 600 radians a metre; fused, the gradient case's powers and
// derivatives were 3.7 and 2.3 times as far from one, in the same time)
__device__ __forceinline__ double rdot(R3 a, R3 b) { return a.x * b.x + a.y * b.y + a.z * b.z; }
__device__ __forceinline__ R3 rcross(R3 a, R3 b) {
  return r3(a.y * b.z - a.z * b.y, a.z * b.x - a.x * b.z, a.x * b.y - a.y * b.x);
}
__device__ __forceinline__ double rnorm(R3 a) { return sqrt(rdot(a, a)); }
__device__ __forceinline__ R3 runit(R3 a) { return a * (1.0 / rnorm(a)); }

struct Zc {
  double re, im;
};
__device__ __forceinline__ Zc zc(double r, double i = 0.0) { return Zc{r, i}; }
__device__ __forceinline__ Zc operator+(Zc a, Zc b) { return zc(a.re + b.re, a.im + b.im); }
__device__ __forceinline__ Zc operator-(Zc a, Zc b) { return zc(a.re - b.re, a.im - b.im); }
__device__ __forceinline__ Zc operator*(Zc a, Zc b) {
  return zc(fma(a.re, b.re, -(a.im * b.im)), fma(a.re, b.im, a.im * b.re));
}
__device__ __forceinline__ Zc operator*(Zc a, double s) { return zc(a.re * s, a.im * s); }
__device__ __forceinline__ Zc operator/(Zc a, Zc b) {
  double d = b.re * b.re + b.im * b.im;
  return zc((a.re * b.re + a.im * b.im) / d, (a.im * b.re - a.re * b.im) / d);
}
__device__ __forceinline__ Zc zsqrt_p(Zc z) {  // principal branch
  double r = hypot(z.re, z.im);
  if (z.re >= 0.0) {
    double t = sqrt(0.5 * (r + z.re));
    return zc(t, t > 0.0 ? z.im / (2.0 * t) : 0.0);
  }
  double t = sqrt(0.5 * (r - z.re));
  return zc(fabs(z.im) / (2.0 * t), copysign(t, z.im));
}

struct Z3 {
  Zc x, y, z;
};
__device__ __forceinline__ Z3 z3of(R3 v, Zc s) { return Z3{s * v.x, s * v.y, s * v.z}; }  // s v
__device__ __forceinline__ Z3 operator+(const Z3& a, const Z3& b) { return Z3{a.x + b.x, a.y + b.y, a.z + b.z}; }
__device__ __forceinline__ Z3 operator-(const Z3& a, const Z3& b) { return Z3{a.x - b.x, a.y - b.y, a.z - b.z}; }
__device__ __forceinline__ Z3 operator*(const Z3& a, Zc s) { return Z3{a.x * s, a.y * s, a.z * s}; }
__device__ __forceinline__ Z3 operator*(const Z3& a, double s) { return Z3{a.x * s, a.y * s, a.z * s}; }
__device__ __forceinline__ Zc zdot(const Z3& a, R3 v) {
  return zc(fma(a.z.re, v.z, fma(a.y.re, v.y, a.x.re * v.x)), fma(a.z.im, v.z, fma(a.y.im, v.y, a.x.im * v.x)));
}
__device__ __forceinline__ Z3 zcross(R3 a, const Z3& b) {  // real x complex
  return Z3{b.z * a.y - b.y * a.z, b.x * a.z - b.z * a.x, b.y * a.x - b.x * a.y};
}
__device__ __forceinline__ Z3 zcross(const Z3& a, R3 b) {  // complex x real
  return Z3{a.y * b.z - a.z * b.y, a.z * b.x - a.x * b.z, a.x * b.y - a.y * b.x};
}

// Polarisation of an isotropic antenna along unit d: normalize(u - (u.d) d),
// a fixed axis in place of u when u is along d.
struct Pol {
  R3 n, ueff;
  double qn;
};
__device__ __forceinline__ Pol pol_fwd(R3 u, R3 d) {
  Pol p;
  p.ueff = u;
  R3 q = u - d * rdot(u, d);
  p.qn = rnorm(q);
  if (p.qn < 1e-9) {
    p.ueff = fabs(d.x) < 0.9 ? r3(1, 0, 0) : r3(0, 1, 0);
    q = p.ueff - d * rdot(p.ueff, d);
    p.qn = rnorm(q);
  }
  p.n = q * (1.0 / p.qn);
  return p;
}
// d a / d d from d a / d n
__device__ __forceinline__ Z3 pol_bwd(const Pol& p, R3 d, const Z3& nbar) {
  Z3 g = (nbar - z3of(p.n, zdot(nbar, p.n))) * (1.0 / p.qn);
  Zc gd = zdot(g, d);
  return z3of(p.ueff, gd * -1.0) - g * rdot(p.ueff, d);
}

// One bounce's field quantities, from its incoming and outgoing directions.
struct Bounce {
  R3 nh, sv, pin, pout;
  double c, sgn, vn;  // |d_in . n|, its sign, |d_in x n| (fixed s below 1e-12)
  bool fixed_s, pec;
  Zc te, tm, ec, root;
};
__device__ __forceinline__ Bounce bounce_of(R3 din, R3 dout, R3 nrm, double er, double sg, bool pec, double wfac) {
  Bounce b;
  b.nh = runit(nrm);
  double dn = rdot(din, b.nh);
  b.c = fabs(dn);
  b.sgn = dn < 0.0 ? -1.0 : 1.0;
  R3 v = rcross(din, b.nh);
  b.vn = rnorm(v);
  b.fixed_s = b.vn < 1e-12;
  if (b.fixed_s) {  // normal incidence: a fixed unit vector perpendicular to n
    R3 a = fabs(b.nh.x) < 0.9 ? r3(1, 0, 0) : r3(0, 1, 0);
    b.sv = runit(rcross(b.nh, a));
  } else {
    b.sv = v * (1.0 / b.vn);
  }
  b.pin = rcross(b.sv, din);
  b.pout = rcross(b.sv, dout);
  b.pec = pec;
  if (pec) {
    b.te = zc(-1.0);
    b.tm = zc(1.0);
  } else {
    b.ec = zc(er, sg * wfac);
    b.root = zsqrt_p(b.ec - zc(1.0 - b.c * b.c));
    Zc cc = zc(b.c);
    b.te = (cc - b.root) / (cc + b.root);
    Zc ecc = b.ec * b.c;
    b.tm = (ecc - b.root) / (ecc + b.root);
  }
  return b;
}
__device__ __forceinline__ Z3 bounce_apply(const Bounce& b, const Z3& E) {
  return z3of(b.sv, b.te * zdot(E, b.sv)) + z3of(b.pout, b.tm * zdot(E, b.pin));
}

constexpr int kAdjLanes = 8, kAdjGroups = 32 / kAdjLanes;
// A path's state in shared memory (index j: bounce j + 1, i: leg or vertex).
struct AdjPath {
  R3 V0[kMaxRefl], Nn[kMaxRefl], img[kMaxRefl + 1], X[kMaxRefl + 2], dv[kMaxRefl + 1];
  double ell[kMaxRefl + 1], er[kMaxRefl], sg[kMaxRefl], nn[kMaxRefl], den[kMaxRefl], sp[kMaxRefl];
  int mat[kMaxRefl], obj[kMaxRefl], pec[kMaxRefl];
  Bounce b[kMaxRefl];
  Z3 Em[kMaxRefl], Eb[kMaxRefl];       // the field before a bounce, the adjoint of the field after it
  Z3 din[kMaxRefl], dout[kMaxRefl];    // adjoints of a bounce's incoming and outgoing directions
  Z3 t[kMaxRefl + 1];                  // adjoint of a leg's vector
  Zc ebar[kMaxRefl];                   // adjoint of a bounce's permittivity
  Pol pol0, polr;
  Z3 E0b, Er;                          // adjoint of the field at the Tx, the field at the Rx
  Z3 p0, pr;                           // the polarisations' part of the end legs' adjoints
  Zc ph, Pbar, Lbar;
  double L;
  int bad;
};

// One path per group of kAdjLanes lanes, `ppw` groups of each warp at work.
__global__ void __launch_bounds__(32) k_grad_adjoint(GradArgs g, int ppw) {
  __shared__ AdjPath sh[kAdjGroups];
  const int gl = threadIdx.x % kAdjLanes, grp = threadIdx.x / kAdjLanes;
  AdjPath& s = sh[grp];
  const int p = blockIdx.x * ppw + grp;
  bool act = grp < ppw && p < g.n_paths;
  const dcem_path& P = g.paths[act ? p : 0];
  const long base = (long)p * g.W;
  const int k = act ? P.depth : 0;
  if (act) {
    for (int q = gl; q < g.W; q += kAdjLanes) g.param[base + q] = -1;
    bool good = k >= 0 && k <= g.max_refl && P.rx >= 0 && P.rx < g.nrx;
    for (int j = 0; good && j < k; ++j) good = P.tri[j] >= 0 && P.tri[j] < g.ntri;
    if (!good) {
      if (gl == 0) atomicOr(g.err, 2u);
      act = false;
    } else if (gl == 0) {
      if (p > 0 && g.paths[p - 1].rx > P.rx) atomicOr(g.err, 1u);
      s.bad = 0;
    }
  }
  __syncwarp();
  // ---- forward sweep: the triangles at theta
  const double wfac = -1.0 / (2.0 * kPi * g.freq * kEps0);
  const R3 tx = r3(g.tx[0], g.tx[1], g.tx[2]), u = r3(g.pol[0], g.pol[1], g.pol[2]);
  if (act)
    for (int j = gl; j < k; j += kAdjLanes) {
      const int id = P.tri[j];
      const float4* t = g.tris + 3 * (size_t)g.slot_of_id[id];
      const int ob = g.tri_obj[id], m = g.tri_mat[id];
      R3 off = r3(0.0, 0.0, 0.0);
      if (g.theta && ob >= 0) {
        const double* th = g.theta + 2 * g.nmat + 2 * ob;
        const float* xf = g.xf + 12 * (size_t)ob;
        off = r3(th[0] - (double)xf[3], th[1] - (double)xf[7], 0.0);
      }
      R3 v0 = r3(t[0].x, t[0].y, t[0].z) + off, v1 = r3(t[1].x, t[1].y, t[1].z) + off,
         v2 = r3(t[2].x, t[2].y, t[2].z) + off;
      R3 n = rcross(v1 - v0, v2 - v0);
      s.nn[j] = rdot(n, n);
      s.V0[j] = v0;
      s.Nn[j] = n;
      const float4 mt = g.mats[m];
      s.mat[j] = m;
      s.obj[j] = ob;
      s.pec[j] = mt.z != 0.0f;
      s.er[j] = g.theta ? g.theta[2 * m] : (double)mt.x;
      s.sg[j] = g.theta ? g.theta[2 * m + 1] : (double)mt.y;
      if (!(s.nn[j] > 0.0)) s.bad = 1;
    }
  __syncwarp();
  if (act && gl == 0 && !s.bad) {  // image sources, back-trace
    R3 I = tx;
    s.img[0] = I;
    for (int j = 0; j < k; ++j) {
      I = I - s.Nn[j] * (2.0 * rdot(I - s.V0[j], s.Nn[j]) / s.nn[j]);
      s.img[j + 1] = I;
    }
    const float4 rv = g.rx[P.rx];
    R3 Y = r3(rv.x, rv.y, rv.z);
    s.X[0] = tx;
    s.X[k + 1] = Y;
    for (int j = k; j >= 1; --j) {
      const R3 dir = s.img[j] - Y;
      const double den = rdot(dir, s.Nn[j - 1]);
      if (den == 0.0) {
        s.bad = 1;
        break;
      }
      const double q = rdot(s.V0[j - 1] - Y, s.Nn[j - 1]) / den;
      s.den[j - 1] = den;
      s.sp[j - 1] = q;
      Y = Y + dir * q;
      s.X[j] = Y;
    }
  }
  __syncwarp();
  if (act && !s.bad)
    for (int i = gl; i <= k; i += kAdjLanes) {
      const R3 e = s.X[i + 1] - s.X[i];
      const double l = rnorm(e);
      s.ell[i] = l;
      s.dv[i] = e * (1.0 / l);
      if (!(l > 0.0)) s.bad = 1;
    }
  __syncwarp();
  if (act && s.bad) {
    if (gl == 0) atomicOr(g.err, 4u);
    act = false;
  }
  // ---- the bounces, the end polarisations, the phase
  if (act) {
    for (int j = gl; j < k; j += kAdjLanes)
      s.b[j] = bounce_of(s.dv[j], s.dv[j + 1], s.Nn[j], s.er[j], s.sg[j], s.pec[j] != 0, wfac);
    if (gl == kAdjLanes - 1) s.pol0 = pol_fwd(u, s.dv[0]);
    if (gl == kAdjLanes - 2) s.polr = pol_fwd(u, s.dv[k] * -1.0);
    if (gl == kAdjLanes - 3) {
      double L = 0.0, sp, cp;
      for (int i = 0; i <= k; ++i) L += s.ell[i];
      sincos(2.0 * kPi * g.freq / kC0 * L, &sp, &cp);
      s.ph = zc(cp, -sp);  // e^{-j k L}
      s.L = L;
    }
  }
  __syncwarp();
  // ---- the field forward, its adjoint back (from a-bar = 1)
  if (act && gl == 0) {
    const R3 e = s.pol0.n;
    Z3 E = Z3{zc(e.x), zc(e.y), zc(e.z)};
    for (int j = 0; j < k; ++j) {
      s.Em[j] = E;
      E = bounce_apply(s.b[j], E);
    }
    const double lam = kC0 / g.freq, K = lam / (4.0 * kPi);
    const Zc a = zdot(E, s.polr.n) * s.ph * (K / s.L);
    g.items[base] = make_double2(a.re, a.im);
    g.param[base] = -2;
    if (g.need_d) {
      s.Er = E;
      s.Pbar = s.ph * (K / s.L);
      s.Lbar = a * zc(-1.0 / s.L, -(2.0 * kPi * g.freq / kC0));
      Z3 Eb = z3of(s.polr.n, s.Pbar);
      for (int j = k - 1; j >= 0; --j) {
        const Bounce& b = s.b[j];
        s.Eb[j] = Eb;
        Eb = z3of(b.sv, zdot(Eb, b.sv) * b.te) + z3of(b.pin, zdot(Eb, b.pout) * b.tm);
      }
      s.E0b = Eb;
    }
  }
  if (!g.need_d) return;
  __syncwarp();
  // ---- each bounce differentiated at its own directions
  if (act) {
    for (int j = gl; j < k; j += kAdjLanes) {
      const Bounce b = s.b[j];
      const Z3 Em = s.Em[j], Eb = s.Eb[j];
      const R3 di = s.dv[j], dq = s.dv[j + 1];
      const Zc es = zdot(Em, b.sv), ep = zdot(Em, b.pin);
      const Zc A = b.te * es, B = b.tm * ep;
      const Zc Ab = zdot(Eb, b.sv), Bb = zdot(Eb, b.pout);
      Z3 svb = Eb * A + Em * (Ab * b.te);
      const Z3 poutb = Eb * B;
      const Z3 pinb = Em * (Bb * b.tm);
      Z3 din = zcross(pinb, b.sv);
      Zc eb = zc(0.0);
      if (!b.pec) {
        const Zc teb = Ab * es, tmb = Bb * ep;
        const Zc r = b.root, cc = zc(b.c), c2 = zc(b.c * b.c);
        const Zc Dte = cc + r, Dtm = b.ec * b.c + r;
        const Zc w = r - c2 / r;                      // r - c^2 / r
        const Zc dte_dc = w * 2.0 / (Dte * Dte);
        const Zc dte_de = (cc / r) * -1.0 / (Dte * Dte);
        const Zc dtm_dc = b.ec * w * 2.0 / (Dtm * Dtm);
        const Zc dtm_de = cc * (r * 2.0 - b.ec / r) / (Dtm * Dtm);
        const Zc cb = teb * dte_dc + tmb * dtm_dc;
        eb = teb * dte_de + tmb * dtm_de;
        din = din + z3of(b.nh, cb * b.sgn);
      }
      svb = svb + zcross(di, pinb) + zcross(dq, poutb);
      if (!b.fixed_s) {
        const Z3 vb = (svb - z3of(b.sv, zdot(svb, b.sv))) * (1.0 / b.vn);
        din = din + zcross(b.nh, vb);
      }
      s.ebar[j] = eb;
      s.din[j] = din;
      s.dout[j] = zcross(poutb, b.sv);
    }
    if (gl == kAdjLanes - 1) s.p0 = pol_bwd(s.pol0, s.dv[0], s.E0b);
    // the Rx polarisation is taken along -d_k
    if (gl == kAdjLanes - 2) s.pr = pol_bwd(s.polr, s.dv[k] * -1.0, s.Er * s.Pbar);
  }
  __syncwarp();
  // directions and lengths -> the legs' vectors
  if (act)
    for (int i = gl; i <= k; i += kAdjLanes) {
      Z3 db = i < k ? s.din[i] : s.pr * -1.0;
      if (i > 0) db = db + s.dout[i - 1];
      if (i == 0) db = db + s.p0;
      s.t[i] = (db - z3of(s.dv[i], zdot(db, s.dv[i]))) * (1.0 / s.ell[i]) + z3of(s.dv[i], s.Lbar);
    }
  __syncwarp();
  if (!act) return;
  // ---- outputs: each parameter at its first bounce
  for (int j = gl; j < k; j += kAdjLanes) {
    bool first = !s.pec[j];
    for (int q = 0; q < j; ++q) first = first && s.mat[q] != s.mat[j];
    if (!first) continue;
    Zc de = zc(0.0);
    for (int q = j; q < k; ++q)
      if (s.mat[q] == s.mat[j]) de = de + s.ebar[q];
    g.items[base + 1 + 4 * j] = make_double2(de.re, de.im);                 // d / d eps_r
    g.param[base + 1 + 4 * j] = 2 * s.mat[j];
    g.items[base + 2 + 4 * j] = make_double2(-de.im * wfac, de.re * wfac);  // d / d sigma
    g.param[base + 2 + 4 * j] = 2 * s.mat[j] + 1;
  }
  for (int ja = gl; ja < 2 * k; ja += kAdjLanes) {
    const int j = ja >> 1, ax = ja & 1;
    bool first = s.obj[j] >= 0;
    for (int q = 0; q < j; ++q) first = first && s.obj[q] != s.obj[j];
    if (!first) continue;
    // tangent of the image geometry when every plane of object obj[j] moves
    // along axis ax: of the images, then of the vertices from the last back
    // (the images' tangents are kept, the vertices' contracted at once)
    R3 ti[kMaxRefl + 1];
    ti[0] = r3(0, 0, 0);
    const R3 e = r3(ax == 0 ? 1.0 : 0.0, ax == 1 ? 1.0 : 0.0, 0.0);
    for (int q = 0; q < k; ++q) {
      const R3 d0 = s.obj[q] == s.obj[j] ? e : r3(0, 0, 0);
      ti[q + 1] = ti[q] - s.Nn[q] * (2.0 * rdot(ti[q] - d0, s.Nn[q]) / s.nn[q]);
    }
    Zc da = zc(0.0);
    R3 tX = r3(0, 0, 0);
    for (int q = k; q >= 1; --q) {
      const R3 d0 = s.obj[q - 1] == s.obj[j] ? e : r3(0, 0, 0);
      const R3 dir = s.img[q] - s.X[q + 1], tdir = ti[q] - tX;
      const double sq = s.sp[q - 1];
      const double ts = (rdot(d0 - tX, s.Nn[q - 1]) - sq * rdot(tdir, s.Nn[q - 1])) / s.den[q - 1];
      tX = tX + dir * ts + tdir * sq;
      da = da + zdot(s.t[q - 1] - s.t[q], tX);  // vertex q ends leg q - 1 and starts leg q
    }
    g.items[base + 3 + ax + 4 * j] = make_double2(da.re, da.im);
    g.param[base + 3 + ax + 4 * j] = 2 * g.nmat + 2 * s.obj[j] + ax;
  }
}

// Vector-Jacobian product of the received powers: one thread per parameter,
// receivers summed in order, sixteen receivers' values loaded at a time (the
// sum itself is short; one load per addition took 69 us for 256 receivers).
__global__ void k_theta_bar(GradArgs g, int nparam) {
  constexpr int kBatch = 16;
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= nparam) return;
  double acc = 0.0;
  for (int r0 = 0; r0 < g.nrx; r0 += kBatch) {
    double v[kBatch], w[kBatch];
#pragma unroll
    for (int i = 0; i < kBatch; ++i) {
      const int r = min(r0 + i, g.nrx - 1);
      v[i] = g.dpcoh[(size_t)r * nparam + t];
      w[i] = g.pcoh_bar[r];
    }
#pragma unroll
    for (int i = 0; i < kBatch; ++i)
      if (r0 + i < g.nrx) acc += w[i] * v[i];
  }
  g.theta_bar[t] = acc;
}

__global__ void k_pack_rx(const float* __restrict__ rx3, int n, float4* out) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
    out[i] = make_float4(rx3[3 * i], rx3[3 * i + 1], rx3[3 * i + 2], 0.0f);
}

}  // namespace

cudaError_t launch_pack_rx(const float* rx3, int n, float4* out, cudaStream_t st) {
  if (n > 0) k_pack_rx<<<(n + 255) / 256, 256, 0, st>>>(rx3, n, out);
  return cudaGetLastError();
}

static void launch_grad_reduce(const GradArgs& a, int nparam, cudaStream_t st) {
  if (a.nrx <= 0) return;
  const size_t smem = a.need_d && nparam <= kGradShared ? 2 * sizeof(double) * (size_t)nparam : 0;
  k_grad_reduce<<<a.nrx, kGradThreads, smem, st>>>(a, nparam);
}

cudaError_t launch_adjoint(const GradArgs& a, int sms, cudaStream_t st) {
  if (a.n_paths > 0) {
    // one path per warp while there are few, so that a path's FP64 chain has
    // a scheduler to itself; four when they are many
    const int ppw = std::max(1, std::min(kAdjGroups, a.n_paths / (8 * sms)));
    k_grad_adjoint<<<(a.n_paths + ppw - 1) / ppw, 32, 0, st>>>(a, ppw);
  }
  int nparam = grad_nparam(a.nmat, a.nobj);
  launch_grad_reduce(a, nparam, st);
  if (a.theta_bar && nparam > 0) k_theta_bar<<<(nparam + 31) / 32, 32, 0, st>>>(a, nparam);
  return cudaGetLastError();
}

cudaError_t launch_gradients(const GradArgs& a, cudaStream_t st) {
  long total = (long)a.n_paths * a.W;
  if (total > 0) {
    long b = (total + 127) / 128;
    k_grad_items<<<(int)(b < 65535 ? b : 65535), 128, 0, st>>>(a);
  }
  launch_grad_reduce(a, grad_nparam(a.nmat, a.nobj), st);
  return cudaGetLastError();
}

DCEM_CHECKS_TAKER(checks_take_grad)

}  // namespace dcem
