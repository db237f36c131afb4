// Ostrich per-timestep solve and IFT adjoint for many independent worlds, sm_103a.
//
// One CTA runs one world; its whole working set (bodies, constraint rows, contact
// slots, Schur blocks) lives in shared memory.  The work follows the paper:
//   Sec. III-A  backward-Euler kinematics Eq. (1), implicit dynamics Eq. (2);
//   Sec. III-B  joint rows Eq. (3), FB normal contact Eq. (4), friction Eq. (7)
//               with the two cone safeguards, velocity servo Eq. (8);
//   Sec. III-C  kinematic substitution, Schur step Eq. (12), back-substitution
//               Eq. (13), best-iterate backtracking (optional line search);
//   Sec. III-D  adjoint Eqs. (16)-(19) with the forward Schur factor read back from
//               the tape, vector-Jacobian products Eq. (17) with the position
//               pull-back evaluated by forward-mode duals, one row at a time.
// The Schur matrix A = h J M^-1 J^T + C + delta I is never formed densely: rows are
// ordered contact rows first, grouped by body (each group touches one body only,
// so groups do not couple), then the joint/servo rows (the separator).  That block-
// arrowhead structure is factored as Cholesky of each group block, elimination of
// the group-separator coupling, then Cholesky of the reduced separator block.
//
// Included once per precision (ostrich_kernels_f32.cu, ostrich_kernels_f64.cu, which
// define OST_REAL) so that the two compile in parallel.
#include <cuda_runtime.h>
#include <stdint.h>
#include <atomic>
#include "ostrich_scene.h"
#include "ostrich_math.cuh"
#include "ostrich_contacts.cuh"

namespace ost {

// ---------------------------------------------------------------------------
// shared-memory layout of one world
// ---------------------------------------------------------------------------
template <class Real> struct WS {
  int tid;        // this thread's number in the CTA's work (the kernels may turn the warps' order)
  int sum_nth;    // threads whose partial sums the merit and the damping are added up from
  // bodies
  Real *qm, *um, *ubar, *uk, *ut, *ub, *du, *f, *rdyn, *mr, *Iw, *Iwi, *R, *qp;
  Real *sbc;      // per servo: the bias b_c of Eq. (8) (-target, or (x(q-) - target)/h)
  // rows
  // J: 12 per row, both bodies' parts; a contact row touches one body, and the second half
  // of its row holds Y = M^-1 J^T.  ys: Y of the separator rows, 12 per row.
  Real *J, *ys, *C, *rhat, *r2, *lk, *lt, *lb, *dl, *rhs;
  uint32_t *row;  // what each row is: row_word()
  // slots
  Real *sn, *sd, *st1, *st2, *swhat, *srad, *sedge;
  int *srow;      // first row of an active slot, -1 of an inactive one
  int *sid, *sftype;
  // per-body row lists
  uint16_t *bsep;   // offsets in J of the body's parts of the separator rows touching it
  // groups
  int *g0, *gn;
  // Schur storage (block-arrowhead, inverse form): G group blocks, E coupling rows, H their
  // F = E L^-T, S reduced separator; prow the factors' exchange rows, 64 values per warp
  Real *G, *E, *H, *S, *prow, *tmp, *tmp2;
  // scratch
  Real *red;
  int *ints;      // [0] rows, [1] contact rows, [7] contact-generation status bits (4: candidates beyond
                  // the slots), [8], [9] decisions of the exact adjoint, [14] turn of the warps, [15] work item
  Real *scal;     // [2] delta, the damping at the iterate evaluated last
  Real *pcr;      // PCR mode: r, z, p, A p, A z, P A p and the Jacobi diagonal, m_max each
};

// Takes n elements of T from the workspace at base: off is the byte offset of the first
// free byte.  Pointers stay base + offset (no integer round trip), so that the compiler
// sees that they point into shared memory and uses its loads, stores and 32-bit addresses.
struct Carver {
  char* base;
  size_t off;
};
template <class T> __host__ __device__ __forceinline__ T* carve(Carver& p, int n, size_t align = 8) {
  const size_t a = alignof(T) < align ? align : alignof(T);
  const size_t q = (p.off + a - 1) & ~(a - 1);
  p.off = q + sizeof(T) * (size_t)(n > 0 ? n : 1);
  return reinterpret_cast<T*>(p.base + q);
}

// Word of a row: its index in the state's lambda block, its bodies (15: none), type, index among
// its slot's or joint's rows, contact group, and slot or joint.
__device__ __forceinline__ uint32_t row_word(int lam, int b0, int b1, int type, int sub, int grp, int ref) {
  return (uint32_t)(lam | b0 << 8 | (b1 & 15) << 12 | type << 16 | sub << 18 | grp << 21 | ref << 24);
}
static_assert(5 * NJ_CAP + NJ_CAP + 3 * SLOT_CAP <= 256 && NB_CAP <= 8 && SLOT_CAP <= 256, "a row's word holds these");
__device__ __forceinline__ int row_lam(uint32_t x) { return x & 255; }
__device__ __forceinline__ int row_b0(uint32_t x) { return (x >> 8) & 15; }
__device__ __forceinline__ int row_b1(uint32_t x) { const int b = (x >> 12) & 15; return b == 15 ? -1 : b; }
__device__ __forceinline__ int row_type(uint32_t x) { return (x >> 16) & 3; }
__device__ __forceinline__ int row_sub(uint32_t x) { return (x >> 18) & 7; }
__device__ __forceinline__ int row_grp(uint32_t x) { return (x >> 21) & 7; }
__device__ __forceinline__ int row_ref(uint32_t x) { return x >> 24; }

template <class Real> __host__ __device__ __forceinline__ WS<Real> ws_carve(char* base, const SceneLayout& s, size_t* bytes = nullptr) {
  WS<Real> w;
  Carver p = {base, 0};
  int nb = s.nb, m = s.m_max, ns = s.n_slots > 0 ? s.n_slots : 1, ng = s.n_groups > 0 ? s.n_groups : 1;
  int ss = s.ss > 0 ? s.ss : 1, pg = s.pg > 0 ? s.pg : 1;
  w.qm = carve<Real>(p, 7 * nb); w.um = carve<Real>(p, 6 * nb); w.ubar = carve<Real>(p, s.n_servo + 1);
  w.uk = carve<Real>(p, 6 * nb); w.ut = carve<Real>(p, 6 * nb); w.ub = carve<Real>(p, 6 * nb);
  w.du = carve<Real>(p, 6 * nb); w.f = carve<Real>(p, 6 * nb); w.rdyn = carve<Real>(p, 6 * nb);
  w.mr = carve<Real>(p, 6 * nb);
  w.Iw = carve<Real>(p, 9 * nb); w.Iwi = carve<Real>(p, 9 * nb); w.R = carve<Real>(p, 9 * nb);
  w.qp = carve<Real>(p, 7 * nb);
  w.sbc = carve<Real>(p, s.n_servo + 1);
  w.J = carve<Real>(p, 12 * m, 16);
  w.C = carve<Real>(p, m); w.rhat = carve<Real>(p, m); w.lk = carve<Real>(p, m); w.lb = carve<Real>(p, m);
  // r2 is done with once the merit is summed: its place then holds the exchange rows of the
  // register factors (64 values per warp, at most four warps), or four columns of a
  // separator beyond 32 rows
  w.r2 = carve<Real>(p, m > 4 * 64 ? m : 4 * 64, 16);
  w.prow = w.r2;
  static_assert(SEP_CAP <= 64, "four columns of a separator fit the exchange buffer");
  w.row = carve<uint32_t>(p, m);
  w.sn = carve<Real>(p, 3 * ns); w.st1 = carve<Real>(p, 3 * ns); w.st2 = carve<Real>(p, 3 * ns);
  w.srad = carve<Real>(p, 3 * ns); w.sd = carve<Real>(p, ns); w.swhat = carve<Real>(p, ns);
  w.sedge = carve<Real>(p, 2 * ns);
  w.srow = carve<int>(p, ns); w.sid = carve<int>(p, ns); w.sftype = carve<int>(p, ns);
  w.bsep = carve<uint16_t>(p, nb * ss);
  w.g0 = carve<int>(p, ng); w.gn = carve<int>(p, ng);
  const int cm = s.cmax > 0 ? s.cmax : 1, ldg = s.ldg > 0 ? s.ldg : 1, esz = ng * cm * ldg;
  // The coupling rows E live from the assembly to F = E L^-T, when the trial multipliers, the
  // step and the solve's scratch are free: one place for both
  const size_t e0 = (p.off + 15) & ~(size_t)15;
  w.lt = carve<Real>(p, m, 16);
  w.dl = carve<Real>(p, m); w.rhs = carve<Real>(p, m); w.tmp = carve<Real>(p, m); w.tmp2 = carve<Real>(p, m);
  w.E = w.lt;
  if (p.off < e0 + sizeof(Real) * (size_t)esz) p.off = e0 + sizeof(Real) * (size_t)esz;
  // G, H and S in one run (the adjoint keeps up to 14 m pull-back items there).  The separator
  // rows' Y lives from the evaluation to the assembly, F from the elimination on: one place.
  const int hsz = esz > 12 * ss ? esz : 12 * ss;
  int gsz = ng * tri_size(pg);
  if (gsz + hsz + tri_size(ss) < 14 * m) gsz = 14 * m - hsz - tri_size(ss);
  w.G = carve<Real>(p, gsz); w.H = carve<Real>(p, hsz, 16); w.ys = w.H;
  w.S = carve<Real>(p, tri_size(ss));
  w.red = carve<Real>(p, 64); w.ints = carve<int>(p, 16); w.scal = carve<Real>(p, 8);
  w.pcr = s.lin == LIN_PCR ? carve<Real>(p, 7 * m) : nullptr;
  if (bytes) *bytes = p.off;
  return w;
}

// Dynamic shared memory of one world: what the carve takes from a 16-byte aligned base (the
// dynamic shared-memory base is), rounded up to 16 bytes.
template <class Real> __host__ __device__ __forceinline__ size_t ws_layout_bytes(const SceneLayout& s) {
  size_t used = 0;
  ws_carve<Real>(nullptr, s, &used);
  return (used + 15) & ~(size_t)15;
}
template <class Real> size_t ws_bytes(const DevScene& s) { return ws_layout_bytes<Real>(s); }
// All shared memory of a CTA of the step kernels: the working set beside their static scene.
template <class Real> size_t step_smem_total(const DevScene& s) {
  return ws_bytes<Real>(s) + ((sizeof(KScene<Real>) + 15) & ~(size_t)15);
}

// Deterministic block sum (fixed tree), the same in every thread, through w.red[8..].  One
// barrier: between the reads of one call and the writes of the next lies another barrier of
// the caller's, and block_sum2 has places of its own, so that the two may alternate.
template <class Real> __device__ Real block_sum(WS<Real>& w, Real v) {
  const int tid = w.tid, lane = tid & 31, wid = tid >> 5, nw = (blockDim.x + 31) >> 5;
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if (lane == 0) w.red[8 + wid] = v;
  __syncthreads();
  Real acc = Real(0);
  for (int i = 0; i < nw; ++i) acc += w.red[8 + i];
  return acc;
}

// Two deterministic block sums at once (fixed tree, as block_sum): results in a, b.  The same
// rule on barriers.  (512 robots by conjugate residuals, whose iterations hold one of each: 1291 ->
// 1267 us with one barrier instead of three and two; 8192 robots directly 2371 -> 2351.)
template <class Real> __device__ void block_sum2(WS<Real>& w, Real& a, Real& b) {
  const int tid = w.tid, lane = tid & 31, wid = tid >> 5, nw = (blockDim.x + 31) >> 5;
  for (int o = 16; o > 0; o >>= 1) {
    a += __shfl_xor_sync(0xffffffffu, a, o);
    b += __shfl_xor_sync(0xffffffffu, b, o);
  }
  if (lane == 0) { w.red[wid] = a; w.red[16 + wid] = b; }
  __syncthreads();
  Real sa = Real(0), sb = Real(0);
  for (int i = 0; i < nw; ++i) { sa += w.red[i]; sb += w.red[16 + i]; }
  a = sa;
  b = sb;
}

// block maximum (every thread gets it), through w.red[33..]
template <class Real> __device__ Real block_max(WS<Real>& w, Real v) {
  const int tid = w.tid, lane = tid & 31, wid = tid >> 5, nw = (blockDim.x + 31) >> 5;
  for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
  __syncthreads();
  if (lane == 0) w.red[33 + wid] = v;
  __syncthreads();
  Real mx = w.red[33];
  for (int i = 1; i < nw; ++i) mx = fmax(mx, w.red[33 + i]);
  __syncthreads();
  return mx;
}

// two block maxima at once (every thread gets both), through w.red[40..] and w.red[56..]
template <class Real> __device__ void block_max2(WS<Real>& w, Real& a, Real& b) {
  const int tid = w.tid, lane = tid & 31, wid = tid >> 5, nw = (blockDim.x + 31) >> 5;
  for (int o = 16; o > 0; o >>= 1) {
    a = fmax(a, __shfl_xor_sync(0xffffffffu, a, o));
    b = fmax(b, __shfl_xor_sync(0xffffffffu, b, o));
  }
  __syncthreads();
  if (lane == 0) { w.red[40 + wid] = a; w.red[56 + wid] = b; }
  __syncthreads();
  Real ma = w.red[40], mb = w.red[56];
  for (int i = 1; i < nw; ++i) { ma = fmax(ma, w.red[40 + i]); mb = fmax(mb, w.red[56 + i]); }
  __syncthreads();
  a = ma;
  b = mb;
}

// ---------------------------------------------------------------------------
// geometry helpers in any scalar type S
// ---------------------------------------------------------------------------
template <class S> __device__ __forceinline__ void tangent_basis(vec3<S> n, vec3<S>& t1, vec3<S>& t2) {
  vec3<S> e = below_09(fabs(sval(n.x))) ? v3(S(1), S(0), S(0)) : v3(S(0), S(1), S(0));
  vec3<S> t = e - scale(n, dot3(n, e));
  S l = ssqrt(dot3(t, t));
  t1 = scale(t, S(1) / l);
  t2 = cross3(n, t1);
}

// contact point on body b at pose (p, q) for slot kind: box corner (material point) or
// rim (deepest point of the rim circle along -n)
template <class S, class Real> __device__ __forceinline__ vec3<S> slot_point(const KScene<Real>& sc, int b, int local, vec3<S> p,
                                                                 const S* q, vec3<S> n) {
  if (sc.shape[b] == SHAPE_BOX) {
    int k = local;
    vec3<S> rb = v3(S((k & 1) ? sc.half[b][0] : -sc.half[b][0]), S((k & 2) ? sc.half[b][1] : -sc.half[b][1]),
                    S((k & 4) ? sc.half[b][2] : -sc.half[b][2]));
    return p + qrot(q, rb);
  }
  int rim = local / sc.nf;
  vec3<S> a = qrot(q, v3(S(0), S(1), S(0)));
  vec3<S> cen = p + qrot(q, v3(S(0), S(rim ? sc.hw[b] : -sc.hw[b]), S(0)));
  S nd = dot3(n, a);
  vec3<S> perp = n - scale(a, nd);
  S pl = ssqrt(dot3(perp, perp));
  if (upto_1em12(sval(pl))) return cen;
  return cen - scale(perp, S(sc.radius[b]) / pl);
}

// frame (n, d) of a slot: fixed plane, or box edge with normal toward the rim centre at q-
template <class S, class Real> __device__ __forceinline__ void slot_frame2(const KScene<Real>& sc, int b, int local, int ftype,
                                                                           const S* qm7, const Real* nstore, Real dstore,
                                                                           const Real* edge, vec3<S>& n, S& d) {
  if (ftype == 1) {
    int rim = local / sc.nf;
    vec3<S> p = v3(qm7[0], qm7[1], qm7[2]);
    vec3<S> cen = p + qrot(qm7 + 3, v3(S(0), S(rim ? sc.hw[b] : -sc.hw[b]), S(0)));
    S dx = cen.x - S(edge[0]), dz = cen.z - S(edge[1]);
    S len = ssqrt(dx * dx + dz * dz);
    n = v3(dx / len, S(0), dz / len);
    d = n.x * S(edge[0]) + n.z * S(edge[1]);
  } else {
    n = v3(S(nstore[0]), S(nstore[1]), S(nstore[2]));
    d = S(dstore);
  }
}

// ---------------------------------------------------------------------------
// joint geometry in any scalar type S, from body positions and rotation matrices
// ---------------------------------------------------------------------------
// Body-frame to world rotations for the joint helpers: a rotation matrix (the step's
// R(q) in shared memory) or a quaternion normalised once (the adjoint's dual numbers, where
// nine matrix entries per body would cost registers).
template <class S> struct MatRot {
  const S* R;
  __device__ __forceinline__ vec3<S> operator()(vec3<S> v) const { return mat3<S>(R, v); }
};
template <class S> struct QuatRot {
  S w;
  vec3<S> qv;
  __device__ __forceinline__ explicit QuatRot(const S* q) {
    const S inv = S(1) / ssqrt(q[0] * q[0] + q[1] * q[1] + q[2] * q[2] + q[3] * q[3]);
    w = q[0] * inv;
    qv = v3(q[1] * inv, q[2] * inv, q[3] * inv);
  }
  // v + w t + qv x t, t = 2 qv x v (the rotation of qrot, with the normalisation done once)
  __device__ __forceinline__ vec3<S> operator()(vec3<S> v) const {
    vec3<S> t = cross3(qv, v);
    t = v3(t.x + t.x, t.y + t.y, t.z + t.z);
    const vec3<S> c = cross3(qv, t);
    return v3(v.x + w * t.x + c.x, v.y + w * t.y + c.y, v.z + w * t.z + c.z);
  }
};

template <class S, class Real> __device__ __forceinline__ vec3<S> cvec(const Real* a) { return v3(S(a[0]), S(a[1]), S(a[2])); }

// The five rows of joint j (Eq. (3)): Jacobian parts before the rotation-rate map E and the
// constraint values, handed row by row (k = 0..4) to f(k, lin_p, ang_p, lin_c, ang_c, c) so
// that a caller contracts or stores each row without holding all five (each intermediate
// lives only as long as its rows need it).  rotp / rotc: the parent's / child's rotation.
// Revolute: anchor rows (p_p + r_p) - (p_c + r_c) by component, then the alignment rows
// perp_k,p . axis_c.  Prismatic: b_k . d (b_k = R_p perp_k, d = (p_c + r_c) - (p_p + r_p)),
// the alignment rows, and the twist lock perp2_p . perp1_c.
template <class S, class RP, class RC, class F, class Real>
__device__ __forceinline__ void joint_rows_each(const KScene<Real>& sc, int j, vec3<S> pp, const RP& rotp, vec3<S> pc,
                                                const RC& rotc, F&& f) {
  const vec3<S> z = v3(S(0.0), S(0.0), S(0.0));
  if (sc.jtype[j] == JOINT_REVOLUTE) {
    {
      const vec3<S> rp = rotp(cvec<S>(sc.ap[j])), rc = rotc(cvec<S>(sc.ac[j]));
      const vec3<S> d = (pc + rc) - (pp + rp);
      const vec3<S> ex = v3(S(1.0), S(0.0), S(0.0)), ey = v3(S(0.0), S(1.0), S(0.0)), ez = v3(S(0.0), S(0.0), S(1.0));
      f(0, ex, cross3(rp, ex), scale(ex, S(-1.0)), scale(cross3(rc, ex), S(-1.0)), S(0.0) - d.x);
      f(1, ey, cross3(rp, ey), scale(ey, S(-1.0)), scale(cross3(rc, ey), S(-1.0)), S(0.0) - d.y);
      f(2, ez, cross3(rp, ez), scale(ez, S(-1.0)), scale(cross3(rc, ez), S(-1.0)), S(0.0) - d.z);
    }
    const vec3<S> aw = rotc(cvec<S>(sc.axc[j]));
    {
      const vec3<S> b1 = rotp(cvec<S>(sc.p1[j]));
      const vec3<S> a1 = cross3(b1, aw);
      f(3, z, a1, z, scale(a1, S(-1.0)), dot3(b1, aw));
    }
    const vec3<S> b2 = rotp(cvec<S>(sc.p2[j]));
    const vec3<S> a2 = cross3(b2, aw);
    f(4, z, a2, z, scale(a2, S(-1.0)), dot3(b2, aw));
  } else {
    const vec3<S> b1 = rotp(cvec<S>(sc.p1[j])), b2 = rotp(cvec<S>(sc.p2[j]));
    {
      const vec3<S> rp = rotp(cvec<S>(sc.ap[j])), rc = rotc(cvec<S>(sc.ac[j]));
      const vec3<S> d = (pc + rc) - (pp + rp);
      const vec3<S> dr = d + rp;
      f(0, scale(b1, S(-1.0)), cross3(b1, dr), b1, cross3(rc, b1), dot3(b1, d));
      f(1, scale(b2, S(-1.0)), cross3(b2, dr), b2, cross3(rc, b2), dot3(b2, d));
    }
    {
      const vec3<S> aw = rotc(cvec<S>(sc.axc[j]));
      const vec3<S> a1 = cross3(b1, aw), a2 = cross3(b2, aw);
      f(2, z, a1, z, scale(a1, S(-1.0)), dot3(b1, aw));
      f(3, z, a2, z, scale(a2, S(-1.0)), dot3(b2, aw));
    }
    const vec3<S> e1 = rotc(cvec<S>(sc.p1[j]));
    const vec3<S> a3 = cross3(b2, e1);
    f(4, z, a3, z, scale(a3, S(-1.0)), dot3(b2, e1));
  }
}

// Servo row of joint j (Eq. (8)): Jacobian parts before E of the joint rate, the relative
// angular velocity about the parent axis (revolute) or the slide rate d/dt (a . d)
// (prismatic).
template <class S> struct SRow { vec3<S> lin_p, ang_p, lin_c, ang_c; };

template <class S, class RP, class RC, class Real>
__device__ __forceinline__ void servo_row_geom(const KScene<Real>& sc, int j, vec3<S> pp, const RP& rotp, vec3<S> pc,
                                               const RC& rotc, SRow<S>& o) {
  const vec3<S> a = rotp(cvec<S>(sc.axp[j]));
  if (sc.jtype[j] == JOINT_REVOLUTE) {
    o.lin_p = v3(S(0.0), S(0.0), S(0.0)); o.lin_c = o.lin_p;
    o.ang_p = scale(a, S(-1.0)); o.ang_c = a;
  } else {
    const vec3<S> rp = rotp(cvec<S>(sc.ap[j])), rc = rotc(cvec<S>(sc.ac[j]));
    const vec3<S> d = (pc + rc) - (pp + rp);
    o.lin_p = scale(a, S(-1.0)); o.ang_p = cross3(a, d + rp);
    o.lin_c = a; o.ang_c = cross3(rc, a);
  }
}

// The joint coordinate a position servo tracks: the revolute angle about the parent axis a
// from perp1_p to the child's perp1 (atan2), or the prismatic slide a . d.
__device__ __forceinline__ float satan2(float y, float x) { return atan2f(y, x); }
__device__ __forceinline__ double satan2(double y, double x) { return atan2(y, x); }
template <class T> __device__ __forceinline__ dual<T> satan2(dual<T> y, dual<T> x) {
  const T r2 = x.v * x.v + y.v * y.v;
  return dual<T>(satan2(y.v, x.v), (x.v * y.d - y.v * x.d) / r2);
}

template <class S, class RP, class RC, class Real>
__device__ __forceinline__ S joint_coord(const KScene<Real>& sc, int j, vec3<S> pp, const RP& rotp, vec3<S> pc,
                                         const RC& rotc) {
  const vec3<S> a = rotp(cvec<S>(sc.axp[j]));
  if (sc.jtype[j] == JOINT_REVOLUTE) {
    const vec3<S> f = rotp(cvec<S>(sc.p1[j]));
    const vec3<S> e = rotc(cvec<S>(sc.p1[j]));
    return satan2(dot3(e, cross3(a, f)), dot3(e, f));
  }
  const vec3<S> rp = rotp(cvec<S>(sc.ap[j])), rc = rotc(cvec<S>(sc.ac[j]));
  return dot3(a, (pc + rc) - (pp + rp));
}

// ---------------------------------------------------------------------------
// per-world setup: load inputs, contacts, rows, masses, warm start
// ---------------------------------------------------------------------------
// element i of an input vector lives at p[i * stride] (stride = ld for the structure-of-
// arrays state, 1 for a tape record)
template <class Real> struct Src { const Real* p; size_t stride; };

// Asynchronous global -> shared copy of one element (cp.async, cached in L1), committed
// as a group and awaited before use, so that the copies proceed while the CTA computes.
template <class Real> __device__ __forceinline__ void cp_async_elem(Real* smem_dst, const Real* gsrc) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(smem_dst);
  if (sizeof(Real) == 8) asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(s), "l"(gsrc) : "memory");
  else asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(s), "l"(gsrc) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_group 0;\n" ::: "memory"); }

// Integers in a tape of Real elements, bit for bit: the bits of a float, or the value of a
// double (exact for every int).
__device__ __forceinline__ float tape_from_int(int v, float) { return __int_as_float(v); }
__device__ __forceinline__ double tape_from_int(int v, double) { return (double)v; }
__device__ __forceinline__ int tape_to_int(float v) { return __float_as_int(v); }
__device__ __forceinline__ int tape_to_int(double v) { return (int)v; }

// ct_out: when not null, the contact slot table of this step is recorded there (a tape
// record's slot table); ct_in: when not null, the table is read from there instead of
// running the activation (the adjoint, at the taped step: the same set by construction).
template <class Real>
__device__ void world_setup(const KScene<Real>& sc, WS<Real>& w, Src<Real> qmv, Src<Real> umv, Src<Real> ubarv,
                            const StepH<Real>& h, Real* ct_out = nullptr, const Real* ct_in = nullptr) {
  const int tid = w.tid, nth = blockDim.x;
  const int nb = sc.nb;
  for (int i = tid; i < 7 * nb; i += nth) w.qm[i] = qmv.p[i * qmv.stride];
  for (int i = tid; i < 6 * nb; i += nth) w.um[i] = umv.p[i * umv.stride];
  for (int i = tid; i < sc.n_servo; i += nth) w.ubar[i] = ubarv.p[i * ubarv.stride];
  if (tid == 0) w.ints[7] = 0;
  __syncthreads();
  // contact activation (FP32 predicate) and slot frames in working precision; an item is one
  // slot, or on a heightmap one wheel rim, whose candidate faces fill its nf slots in order.
  // (Rare or long pieces stay loops and single call sites: their code is read once per step
  // and only pushes the Newton loop's out of the instruction cache.)
  const bool hm = sc.env == ENV_HEIGHTMAP && !ct_in;
  const int n_rims = hm ? 2 * nb : 0;
#pragma unroll 1
  for (int e = tid; e < n_rims + sc.n_slots; e += nth) {
    SlotAct acts[8];
    int sl, b, local, cnt = 1;
    if (e < n_rims) {
      b = e >> 1;
      if (sc.shape[b] != SHAPE_WHEEL) continue;
      local = (e & 1) * sc.nf; cnt = sc.nf;
      sl = sc.slot_base[b] + local;
    } else {
      sl = e - n_rims;
      b = sc.slot_body[sl];
      if (hm && sc.shape[b] == SHAPE_WHEEL) continue;
      local = sl - sc.slot_base[b];
    }
    if (ct_in) {
      const Real* c = ct_in + CT_PER_SLOT * sl;
      SlotAct& a = acts[0];
      a.active = tape_to_int(c[0]); a.id = tape_to_int(c[1]); a.ftype = tape_to_int(c[2]);
      a.n[0] = (float)c[3]; a.n[1] = (float)c[4]; a.n[2] = (float)c[5]; a.d = (float)c[6];
      a.ex = (float)c[7]; a.ez = (float)c[8];
    } else {
      float q7[7], u6[6];
      for (int k = 0; k < 7; ++k) q7[k] = (float)w.qm[7 * b + k];
      for (int k = 0; k < 6; ++k) u6[k] = (float)w.um[6 * b + k];
      if (e < n_rims) {
        if (activate_rim_hm(sc, b, e & 1, q7, u6, acts)) atomicOr(&w.ints[7], 4);
      } else {
        acts[0] = activate_slot(sc, b, local, q7, u6);
      }
    }
#pragma unroll 1
    for (int f = 0; f < cnt; ++f, ++sl, ++local) {
      const SlotAct a = acts[f];
      w.srow[sl] = a.active ? 0 : -1; w.sid[sl] = a.id; w.sftype[sl] = a.ftype;
      w.sedge[2 * sl] = (Real)a.ex; w.sedge[2 * sl + 1] = (Real)a.ez;
      vec3<Real> n; Real d;
      Real ns[3] = {(Real)a.n[0], (Real)a.n[1], (Real)a.n[2]};
      slot_frame2<Real, Real>(sc, b, local, a.ftype, w.qm + 7 * b, ns, (Real)a.d, w.sedge + 2 * sl, n, d);
      vec3<Real> t1, t2;
      tangent_basis(n, t1, t2);
      w.sn[3 * sl] = n.x; w.sn[3 * sl + 1] = n.y; w.sn[3 * sl + 2] = n.z; w.sd[sl] = d;
      w.st1[3 * sl] = t1.x; w.st1[3 * sl + 1] = t1.y; w.st1[3 * sl + 2] = t1.z;
      w.st2[3 * sl] = t2.x; w.st2[3 * sl + 1] = t2.y; w.st2[3 * sl + 2] = t2.z;
      if (ct_out) {
        Real* c = ct_out + CT_PER_SLOT * sl;
        c[0] = tape_from_int(a.active, Real(0)); c[1] = tape_from_int(a.id, Real(0)); c[2] = tape_from_int(a.ftype, Real(0));
        c[3] = Real(a.n[0]); c[4] = Real(a.n[1]); c[5] = Real(a.n[2]); c[6] = Real(a.d);
        c[7] = Real(a.ex); c[8] = Real(a.ez);
      }
    }
  }
  // bodies: world inertia at q-, external force, warm-start velocity
  for (int b = nth - 1 - tid; b < nb; b += nth) {   // beside the slots' warp
    Real R[9];
    qmat(w.qm + 7 * b + 3, R);
    for (int k = 0; k < 9; ++k) w.R[9 * b + k] = R[k];
    for (int i = 0; i < 3; ++i)
      for (int j = 0; j < 3; ++j) {
        Real a = 0, ai = 0;
        for (int k = 0; k < 3; ++k) {
          a += R[3 * i + k] * sc.inertia[b][k] * R[3 * j + k];
          ai += R[3 * i + k] * sc.iinv[b][k] * R[3 * j + k];
        }
        w.Iw[9 * b + 3 * i + j] = a; w.Iwi[9 * b + 3 * i + j] = ai;
      }
    Real m = sc.mass[b];
    vec3<Real> om = v3(w.um[6 * b + 3], w.um[6 * b + 4], w.um[6 * b + 5]);
    vec3<Real> Io = mat3<Real>(w.Iw + 9 * b, om);
    vec3<Real> gy = cross3(om, Io);
    w.f[6 * b] = 0; w.f[6 * b + 1] = 0; w.f[6 * b + 2] = m * sc.g;
    w.f[6 * b + 3] = -gy.x; w.f[6 * b + 4] = -gy.y; w.f[6 * b + 5] = -gy.z;
    vec3<Real> dw = mat3<Real>(w.Iwi + 9 * b, v3(w.f[6 * b + 3], w.f[6 * b + 4], w.f[6 * b + 5]));
    w.uk[6 * b] = w.um[6 * b];
    w.uk[6 * b + 1] = w.um[6 * b + 1];
    w.uk[6 * b + 2] = rn_fma(h.h, sc.g, w.um[6 * b + 2]);
    w.uk[6 * b + 3] = w.um[6 * b + 3] + h.h * dw.x;
    w.uk[6 * b + 4] = w.um[6 * b + 4] + h.h * dw.y;
    w.uk[6 * b + 5] = w.um[6 * b + 5] + h.h * dw.z;
  }
  __syncthreads();
  // servo biases b_c of Eq. (8): -target (velocity target) or (x(q-) - target)/h (position
  // target, x the joint coordinate at the step's start; w.R holds R(q-) here)
  for (int k = tid; k < sc.n_servo; k += nth) {
    const int j = sc.servo_j[k], bp = sc.jp[j], bc = sc.jc[j];
    if (sc.smode[j] == SERVO_POSITION) {
      const Real x = joint_coord<Real>(sc, j, v3(w.qm[7 * bp], w.qm[7 * bp + 1], w.qm[7 * bp + 2]),
                                       MatRot<Real>{w.R + 9 * bp},
                                       v3(w.qm[7 * bc], w.qm[7 * bc + 1], w.qm[7 * bc + 2]), MatRot<Real>{w.R + 9 * bc});
      w.sbc[k] = (x - w.ubar[k]) / h.h;
    } else {
      w.sbc[k] = -w.ubar[k];
    }
  }
  // row compaction, fixed order: the contact rows of the active slots in slot order (so
  // grouped by body), then the separator rows.  A slot's first row is 3 x the number of
  // active slots before it: warp ballots over the slot table (at most 64 slots) give the
  // prefix counts, and each lane writes its own slot's rows.
  if (tid < 32) {
    const int lane = tid, ns = sc.n_slots;
    const unsigned m0 = __ballot_sync(0xffffffffu, lane < ns && w.srow[lane] >= 0);
    const unsigned m1 = __ballot_sync(0xffffffffu, 32 + lane < ns && w.srow[32 + lane] >= 0);
    const int c0 = __popc(m0);
    for (int c = 0; c < 2; ++c) {
      const int sl = 32 * c + lane;
      if (sl >= ns) continue;
      const unsigned mk = c == 0 ? m0 : m1;
      if (!((mk >> lane) & 1u)) { w.srow[sl] = -1; continue; }
      const int r0 = 3 * ((c == 0 ? 0 : c0) + __popc(mk & ((1u << lane) - 1u)));
      const int bb = sc.slot_body[sl];
      w.srow[sl] = r0;
      const int lam = 5 * sc.nj + sc.n_servo + 3 * sl;
      const int gb = sc.body_group[bb];
      for (int k = 0; k < 3; ++k) {
        const int r = r0 + k;
        w.row[r] = row_word(lam + k, bb, -1, k == 0 ? ROW_NORMAL : ROW_FRIC, k, gb, sl);
      }
    }
    // groups: first row and row count of each body's slots
    for (int g = lane; g < sc.n_groups; g += 32) {
      const int bb = sc.group_body[g], lo = sc.slot_base[bb], hi = lo + sc.slot_count[bb];
      auto before = [&](int x) {   // active slots with index < x
        const unsigned lo0 = x >= 32 ? m0 : (m0 & ((1u << x) - 1u));
        const unsigned lo1 = x <= 32 ? 0u : (x >= 64 ? m1 : (m1 & ((1u << (x - 32)) - 1u)));
        return __popc(lo0) + __popc(lo1);
      };
      w.g0[g] = 3 * before(lo);
      w.gn[g] = 3 * (before(hi) - before(lo));
    }
    if (lane == 0) {
      const int mc = 3 * (c0 + __popc(m1));
      w.ints[1] = mc;
      w.ints[0] = mc + sc.ss;
    }
  }
  __syncthreads();
  {
    const int mc = w.ints[1];
    // separator rows: five per joint, then one per servo
    const int ssd = sc.ss > 0 ? sc.ss : 1;
    for (int a = nth - 1 - tid; a < sc.ss; a += nth) {
      const int r = mc + a;
      // in its bodies' lists (in row order)
      for (int side = 0; side < 2; ++side)
        w.bsep[sc.sep_b[a][side] * ssd + sc.sep_pos[a][side]] = (uint16_t)(12 * r + 6 * side);
      if (a < 5 * sc.nj) {
        const int j = a / 5, k = a - 5 * j;
        w.row[r] = row_word(5 * j + k, sc.jp[j], sc.jc[j], ROW_JOINT, k, 0, j);
      } else {
        const int j = sc.servo_j[a - 5 * sc.nj];
        w.row[r] = row_word(5 * sc.nj + sc.servo_of[j], sc.jp[j], sc.jc[j], ROW_SERVO, 0, 0, j);
      }
    }
  }
  // normal-row scaling what = J_n M^-1 J_n^T at q- (geometric Jacobian, E = I)
  for (int sl = tid; sl < sc.n_slots; sl += nth) {
    if (w.srow[sl] < 0) { w.swhat[sl] = 0; continue; }
    int b = sc.slot_body[sl];
    int local = sl - sc.slot_base[b];
    vec3<Real> n = v3(w.sn[3 * sl], w.sn[3 * sl + 1], w.sn[3 * sl + 2]);
    vec3<Real> p = v3(w.qm[7 * b], w.qm[7 * b + 1], w.qm[7 * b + 2]);
    vec3<Real> x = slot_point<Real>(sc, b, local, p, w.qm + 7 * b + 3, n);
    vec3<Real> a = cross3(x - p, n);
    vec3<Real> ia = mat3<Real>(w.Iwi + 9 * b, a);
    w.swhat[sl] = sc.minv[b] + dot3(a, ia);
  }
  __syncthreads();
}

// first safeguard of Sec. III-B: |lambda_f| <= mu lambda_n (l: a slot's three multipliers)
template <class Real> __device__ __forceinline__ void clamp_slot(const KScene<Real>& sc, Real* l) {
  Real rad = sc.mu * (l[0] > Real(0) ? l[0] : Real(0));
  Real nn = ssqrt(l[1] * l[1] + l[2] * l[2]);
  if (nn > rad) {
    Real f = nn > Real(0) ? rad / nn : Real(0);
    l[1] *= f; l[2] *= f;
  }
}
template <class Real> __device__ __forceinline__ void clamp_cone(const KScene<Real>& sc, WS<Real>& w, Real* lam) {
  for (int sl = w.tid; sl < sc.n_slots; sl += blockDim.x)
    if (w.srow[sl] >= 0) clamp_slot(sc, lam + w.srow[sl]);
}

template <class Real> __device__ __forceinline__ Real rowdot(const Real* Ja, int sa, const Real* Yb, int sb) {
  return Ja[sa] * Yb[sb] + Ja[sa + 1] * Yb[sb + 1] + Ja[sa + 2] * Yb[sb + 2] + Ja[sa + 3] * Yb[sb + 3] +
         Ja[sa + 4] * Yb[sb + 4] + Ja[sa + 5] * Yb[sb + 5];
}

// Six consecutive values of a row (rows are 16-byte aligned and 48 or 96 bytes long), two at
// a time.
__device__ __forceinline__ void load6(const float* p, float* v) {
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    const float2 x = reinterpret_cast<const float2*>(p)[q];
    v[2 * q] = x.x; v[2 * q + 1] = x.y;
  }
}
__device__ __forceinline__ void load6(const double* p, double* v) {
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    const double2 x = reinterpret_cast<const double2*>(p)[q];
    v[2 * q] = x.x; v[2 * q + 1] = x.y;
  }
}
__device__ __forceinline__ void store6(float* p, const float* v) {
#pragma unroll
  for (int q = 0; q < 3; ++q) reinterpret_cast<float2*>(p)[q] = make_float2(v[2 * q], v[2 * q + 1]);
}
__device__ __forceinline__ void store6(double* p, const double* v) {
#pragma unroll
  for (int q = 0; q < 3; ++q) reinterpret_cast<double2*>(p)[q] = make_double2(v[2 * q], v[2 * q + 1]);
}

// J part . Y part, both six values in shared memory
template <class Real> __device__ __forceinline__ Real rowdot6(const Real* J, const Real* Y) {
  Real a[6], b[6];
  load6(J, a);
  load6(Y, b);
  return rowdot(a, 0, b, 0);
}

// y = M^-1 J^T of one body's part of a row: (J_lin / m, Iw^-1 J_ang); the values Eq. (2)'s
// M~^-1 gives the row.
template <class Real>
__device__ __forceinline__ void minv_row6(const KScene<Real>& sc, const WS<Real>& w, int b, const Real* Js, Real* ys) {
  const Real mi = sc.minv[b];
  ys[0] = Js[0] * mi; ys[1] = Js[1] * mi; ys[2] = Js[2] * mi;
  const vec3<Real> ia = mat3<Real>(w.Iwi + 9 * b, v3(Js[3], Js[4], Js[5]));
  ys[3] = ia.x; ys[4] = ia.y; ys[5] = ia.z;
}

// The rows touching body b, in row order: its contact group's, then the separator rows of its
// joints.  f(offset of the body's part of the row in J, row).
template <class Real, class F>
__device__ __forceinline__ void body_rows(const KScene<Real>& sc, const WS<Real>& w, int b, F&& f) {
  const int g = sc.body_group[b], r0 = g >= 0 ? w.g0[g] : 0, n = g >= 0 ? w.gn[g] : 0, tot = n + sc.body_sepn[b];
  const uint16_t* bs = w.bsep + b * (sc.ss > 0 ? sc.ss : 1) - n;
#pragma unroll 4
  for (int t = 0; t < tot; ++t) {
    const unsigned off = t < n ? 12 * (r0 + t) : bs[t];
    f((int)off, (int)(off / 12u));
  }
}

// Separator row a at the iterate (u, lam): one of a joint's five position rows (Eq. (3), as
// joint_rows_each forms them) or a servo row (Eq. (8), as servo_row_geom).  A thread per row:
// all five by one thread are five copies of the row's code and five times its latency.
template <class Real>
__device__ __forceinline__ void sep_row(const KScene<Real>& sc, WS<Real>& w, const Real* u, const Real* lam,
                                        const StepH<Real>& h, int a, int mc) {
  const int i = mc + a, j = row_ref(w.row[i]), bp = sc.sep_b[a][0], bc = sc.sep_b[a][1];
  const int k = a < 5 * sc.nj ? a - 5 * j : 5;           // row of the joint; 5: its servo
  const bool rev = sc.jtype[j] == JOINT_REVOLUTE;
  const vec3<Real> pp = v3(w.qp[7 * bp], w.qp[7 * bp + 1], w.qp[7 * bp + 2]);
  const vec3<Real> pc = v3(w.qp[7 * bc], w.qp[7 * bc + 1], w.qp[7 * bc + 2]);
  const MatRot<Real> rotp{w.R + 9 * bp}, rotc{w.R + 9 * bc};
  const vec3<Real> z = v3(Real(0), Real(0), Real(0));
  vec3<Real> lp = z, ap, lc = z, ac;       // the child's angular part is -ac where neg
  Real c = Real(0);
  const bool neg = k < 5 && (rev || k >= 2);
  if (k < 5 && k >= (rev ? 3 : 2)) {
    // alignment (and a prismatic joint's twist lock): b . v
    const bool first = k == (rev ? 3 : 2);
    const vec3<Real> b = rotp(cvec<Real>(first ? sc.p1[j] : sc.p2[j]));
    const vec3<Real> v = rotc(cvec<Real>(!rev && k == 4 ? sc.p1[j] : sc.axc[j]));
    ap = cross3(b, v);
    ac = ap;
    c = dot3(b, v);
  } else if (k == 5 && rev) {
    // joint rate: the relative angular velocity about the parent axis
    ac = rotp(cvec<Real>(sc.axp[j]));
    ap = scale(ac, Real(-1));
  } else {
    const vec3<Real> rp = rotp(cvec<Real>(sc.ap[j])), rc = rotc(cvec<Real>(sc.ac[j]));
    const vec3<Real> d = (pc + rc) - (pp + rp);
    if (rev) {
      // anchor rows by component
      lp = v3(k == 0 ? Real(1) : Real(0), k == 1 ? Real(1) : Real(0), k == 2 ? Real(1) : Real(0));
      ap = cross3(rp, lp);
      lc = scale(lp, Real(-1));
      ac = cross3(rc, lp);
      c = Real(0) - (k == 0 ? d.x : k == 1 ? d.y : d.z);
    } else {
      // the anchor off the axis along a perpendicular, or the slide rate along the axis
      const vec3<Real> b = rotp(cvec<Real>(k == 0 ? sc.p1[j] : k == 1 ? sc.p2[j] : sc.axp[j]));
      lp = scale(b, Real(-1));
      ap = cross3(b, d + rp);
      lc = b;
      ac = cross3(rc, b);
      c = dot3(b, d);
    }
  }
  const vec3<Real> wp = v3(u[6 * bp + 3], u[6 * bp + 4], u[6 * bp + 5]);
  const vec3<Real> wc = v3(u[6 * bc + 3], u[6 * bc + 4], u[6 * bc + 5]);
  const vec3<Real> ap_ = map_Et(ap, wp, h);
  // E of -ac as (w x ac, -ac): the rounding of the row's other users (joint_rows_each)
  const MapE<Real> Ec(wc, h);
  const vec3<Real> x = cross3(neg ? wc : ac, neg ? ac : wc);
  const vec3<Real> as = neg ? scale(ac, Real(-1)) : ac;
  const vec3<Real> ac_ = v3((as.x + x.x * Ec.hh) * Ec.inv, (as.y + x.y * Ec.hh) * Ec.inv, (as.z + x.z * Ec.hh) * Ec.inv);
  const Real Jr[12] = {lp.x, lp.y, lp.z, ap_.x, ap_.y, ap_.z, lc.x, lc.y, lc.z, ac_.x, ac_.y, ac_.z};
  store6(w.J + 12 * i, Jr);
  store6(w.J + 12 * i + 6, Jr + 6);
  Real r, C = Real(0);
  if (k < 5) {
    r = c / h.h;
  } else {
    // J_c u + alpha lambda_c + b_c
    Real v = Real(0);
#pragma unroll
    for (int q = 0; q < 6; ++q) v = rn_add(v, rn_fma(Jr[q], u[6 * bp + q], rn_mul(Jr[6 + q], u[6 * bc + q])));
    C = sc.alpha[j];
    r = v + C * lam[i] + w.sbc[a - 5 * sc.nj];
  }
  w.r2[i] = r; w.rhat[i] = r; w.C[i] = C;
}

// The rows of contact slot sl: the normal's, the two of friction, or all three.
template <bool NORM, bool FRIC, class Real>
__device__ __forceinline__ void slot_rows(const KScene<Real>& sc, WS<Real>& w, const Real* u, const Real* lam,
                                          const StepH<Real>& h, int sl) {
  const Real hR = h.h;
  int i = w.srow[sl];
  int b = sc.slot_body[sl];
  int local = sl - sc.slot_base[b];
  vec3<Real> p = v3(w.qp[7 * b], w.qp[7 * b + 1], w.qp[7 * b + 2]);
  vec3<Real> n = v3(w.sn[3 * sl], w.sn[3 * sl + 1], w.sn[3 * sl + 2]);
  vec3<Real> t1 = v3(w.st1[3 * sl], w.st1[3 * sl + 1], w.st1[3 * sl + 2]);
  vec3<Real> t2 = v3(w.st2[3 * sl], w.st2[3 * sl + 1], w.st2[3 * sl + 2]);
  vec3<Real> x = slot_point<Real>(sc, b, local, p, w.qp + 7 * b + 3, n);
  vec3<Real> lev = x - p;
  vec3<Real> wk = v3(u[6 * b + 3], u[6 * b + 4], u[6 * b + 5]);
  vec3<Real> dirs[3] = {n, t1, t2};
  Real vel[3];
  const MapE<Real> Ek(wk, h);
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    if (k == 0 ? !NORM : !FRIC) continue;
    vec3<Real> ang = Ek(cross3(lev, dirs[k]));
    Real* Jr = w.J + 12 * (i + k);
    Jr[0] = dirs[k].x; Jr[1] = dirs[k].y; Jr[2] = dirs[k].z; Jr[3] = ang.x; Jr[4] = ang.y; Jr[5] = ang.z;
    vel[k] = dirs[k].x * u[6 * b] + dirs[k].y * u[6 * b + 1] + dirs[k].z * u[6 * b + 2] + ang.x * u[6 * b + 3] +
             ang.y * u[6 * b + 4] + ang.z * u[6 * b + 5];
  }
  const Real kap = sc.kappa, eps = sc.eps;
  const Real hw = hR * w.swhat[sl];
  const Real ln = lam[i];
  if (NORM) {
    // normal row, Eq. (4): phi_eps(c_n/h + kappa lambda_n, h what lambda_n)
    Real cn = dot3(n, x) - w.sd[sl];
    Real a = cn / hR + kap * ln, bb = hw * ln;
    // At an active contact b = h what lambda_n is large (~10 m/s) and a ~ 0, so the
    // textbook forms a + b - s, 1 - a/s and 1 - b/s cancel; in FP32 that leaves ~1e-6
    // m/s of noise in the row, which the small eigenvalue (~kappa) of the impulse split
    // between redundant contacts amplifies to ~1e-3 N and the Newton iteration stalls.
    // The same quantities in forms free of cancellation (exact rearrangements):
    // a + b - s = (2ab - eps^2)/(a + b + s) for a + b > 0;  1 - a/s = (b^2 + eps^2)/(s (s + a))
    // for a > 0;  1 - b/s likewise.
    Real s = ssqrt(a * a + bb * bb + eps * eps);
    const Real apb = a + bb;
    Real phi = apb > Real(0) ? (Real(2) * a * bb - eps * eps) / (apb + s) : apb - s;
    Real fa, fb;
    if constexpr (sizeof(Real) == 8) {
      // (in FP64 one form alone is the cheaper where all lanes agree: 22 robots 1 %)
      fa = a > Real(0) ? (bb * bb + eps * eps) / (s * (s + a)) : Real(1) - a / s;
      fb = bb > Real(0) ? (a * a + eps * eps) / (s * (s + bb)) : Real(1) - bb / s;
    } else {
      // one quotient for either form: a warp with lanes of both kinds would go through two
      // (step and adjoint: 8192 robots 2351 -> 2336 us, 1001 robots on the plane 261 -> 259)
      fa = (a > Real(0) ? bb * bb + eps * eps : a) / (a > Real(0) ? s * (s + a) : s);
      fb = (bb > Real(0) ? a * a + eps * eps : bb) / (bb > Real(0) ? s * (s + bb) : s);
      if (!(a > Real(0))) fa = Real(1) - fa;
      if (!(bb > Real(0))) fb = Real(1) - fb;
    }
    Real scl = fa > Real(1e-12) ? fa : Real(1e-12);
    w.r2[i] = phi; w.rhat[i] = phi / scl; w.C[i] = kap + hw * fb / scl;
  }
  if (!FRIC) return;
  // friction rows, Eq. (7): J_f u + (W + kappa) lambda_f with W from the FB reading
  const Real l1 = lam[i + 1], l2 = lam[i + 2];
  Real vt = ssqrt(vel[1] * vel[1] + vel[2] * vel[2] + eps * eps);
  Real lfn = ssqrt(l1 * l1 + l2 * l2 + eps * eps);
  Real lnp = ln > Real(0) ? ln : Real(0);
  Real g = hw * (sc.mu * lnp - lfn);
  Real sg = ssqrt(vt * vt + g * g + eps * eps);
  // W's numerator max(0, vt - phi_eps(vt, g)) is sg - g >= 0; for g > 0 (sticking) it is
  // the small difference of two large numbers, taken as (vt^2 + eps^2)/(sg + g)
  Real num = g > Real(0) ? (vt * vt + eps * eps) / (sg + g) : sg - g;
  Real den = sc.mu * lnp; if (den < Real(1e-12)) den = Real(1e-12);
  Real W = num / den;
  Real rf1 = vel[1] + (W + kap) * l1, rf2 = vel[2] + (W + kap) * l2;
  Real wgt = hw / (hw + W);
  w.r2[i + 1] = rf1 * wgt; w.r2[i + 2] = rf2 * wgt;
  w.rhat[i + 1] = rf1; w.rhat[i + 2] = rf2;
  w.C[i + 1] = W + kap; w.C[i + 2] = W + kap;
  // radial part of the friction block: rho e e^T, e = lambda_f/|lambda_f|
  Real rho = Real(0);
  if (num > Real(0)) {
    Real fbg = num / sg;                  // 1 - g/sg
    rho = fbg * hw * lfn / den;
  }
  Real e1 = l1 / lfn, e2 = l2 / lfn;
  w.srad[3 * sl] = rho * e1 * e1; w.srad[3 * sl + 1] = rho * e1 * e2; w.srad[3 * sl + 2] = rho * e2 * e2;
}

// ---------------------------------------------------------------------------
// one residual / Jacobian evaluation at iterate (u, lam); returns the merit
// ---------------------------------------------------------------------------
// dyn = false (the adjoint): the rows, their compliance and delta only; the dynamics
// residual and the merit are not formed (the returned merit is 0).
template <bool FEW, class Real>
__device__ Real evaluate(const KScene<Real>& sc, WS<Real>& w, const Real* u, const Real* lam, const StepH<Real>& h, bool dyn = true) {
  const int tid = w.tid, nth = blockDim.x;
  const int nb = sc.nb, m = w.ints[0], mc = w.ints[1];
  const Real hR = h.h;
  // poses at q+ = q- + h G(q-) u, a thread per body and axis (column of the rotation)
  for (int e = tid; e < 3 * nb; e += nth) {
    const int b = e / 3, ax = e - 3 * b;
    Real qp[7];
    kin_body<Real, Real>(w.qm + 7 * b, u + 6 * b, h, qp);
    const vec3<Real> c = qrot(qp + 3, v3(ax == 0 ? Real(1) : Real(0), ax == 1 ? Real(1) : Real(0),
                                         ax == 2 ? Real(1) : Real(0)));
    Real* R = w.R + 9 * b + ax;
    R[0] = c.x; R[3] = c.y; R[6] = c.z;
    if (ax == 0)
      for (int k = 0; k < 7; ++k) w.qp[7 * b + k] = qp[k];
  }
  __syncthreads();
  // contact slots from the first thread on, separator rows from the last: they run beside
  // one another in different warps.  Where warps would idle (few worlds), a slot's friction and
  // its normal (its position's arithmetic twice) run in different warps, the lighter normals
  // beside the separator rows: their roots and quotients are this phase's serial chain, and
  // in FP64 the time of the warp's arithmetic unit (step and adjoint: 1 robot 213 -> 209 us,
  // 22 in FP64 1605 -> 1534, 37 boxes in FP64 881 -> 817).  With the chip full it would be more
  // work for the same units (8192 robots 2.35 -> 2.38 ms).
  const int half = nth >> 1;
  if (FEW && half >= 32 && sc.n_slots <= half) {
    const int sl = tid < half ? tid : tid - half;
    if (sl < sc.n_slots && w.srow[sl] >= 0) {
      if (tid < half) slot_rows<false, true>(sc, w, u, lam, h, sl);
      else slot_rows<true, false>(sc, w, u, lam, h, sl);
    }
  } else {
    for (int sl = tid; sl < sc.n_slots; sl += nth)
      if (w.srow[sl] >= 0) slot_rows<true, true>(sc, w, u, lam, h, sl);
  }
  for (int a = nth - 1 - tid; a < sc.ss; a += nth) sep_row(sc, w, u, lam, h, a, mc);
  __syncthreads();
  // Y = M^-1 J^T of every row and the diagonal J Y of J M^-1 J^T, for the assembly at this
  // iterate and its damping delta = delta_rel * mean diag(h J Y); from the last thread, beside
  // the bodies' residuals below
  for (int i = nth - 1 - tid; i < m; i += nth) {
    Real* Ji = w.J + 12 * i;
    const uint32_t rw = w.row[i];
    Real Yi[6], Jv[6];
    load6(Ji, Jv);
    minv_row6(sc, w, row_b0(rw), Jv, Yi);
    Real d = rowdot(Jv, 0, Yi, 0);
    if (i < mc) {
      store6(Ji + 6, Yi);
    } else {
      // (the direct adjoint, dyn = false, needs no Y, and its F is on its way to that place)
      Real* Ys = w.ys + 12 * (i - mc);
      const bool keep = dyn || sc.lin == LIN_PCR;
      if (keep) store6(Ys, Yi);
      load6(Ji + 6, Jv);
      minv_row6(sc, w, row_b1(rw), Jv, Yi);
      if (keep) store6(Ys + 6, Yi);
      d = d + rowdot(Jv, 0, Yi, 0);
    }
    w.tmp[i] = d;
  }
  if (dyn) {
    // Eq. (10): r_dyn = M (u - u-) - h f - h J^T lambda, per body; merit part |M^-1 r_dyn|^2.
    // The inertia and constraint terms nearly cancel at convergence, so the sum is
    // accumulated with exact products and exact partial sums (acc2).
    if constexpr (FEW && sizeof(Real) == 8) {
      // FP64: what counts is the number of instructions of a warp, each some 60 cycles of its
      // arithmetic unit whatever the lanes in use.  Four threads a sum, four terms a turn: each
      // forms its own term's product and the errors of its product and of its partial sum; the
      // sum itself and that of the errors all four form alike, term by term in acc2's order (19
      // instructions for four terms instead of 40, and the same bits).  Terms past the end are
      // zero and change nothing.  From the last thread on, beside the rows above.  The phase
      // takes 12.3 instead of 17.9 k cycles for a box, 23.7 instead of 27.9 k for a robot; with
      // more worlds, whose warps fill the units, it is the slower one (583 robots + 1 %).
      const int seg = 3 - (tid & 3), lane3 = (threadIdx.x & 31) | 3;
      for (int base = 0; base < 24 * nb; base += nth) {
        const int e = (base + nth - 1 - tid) >> 2, b = e / 6, k = e - 6 * b;
        const bool on = e < 6 * nb;
        const int g = on ? sc.body_group[b] : -1, r0 = g >= 0 ? w.g0[g] : 0, n = g >= 0 ? w.gn[g] : 0;
        const int tot = on ? n + sc.body_sepn[b] : 0, nm = k < 3 ? 2 : 6, T = on ? tot + nm + 1 : 0;
        const uint16_t* bs = w.bsep + (on ? b : 0) * (sc.ss > 0 ? sc.ss : 1) - n;
        Real s = Real(0), cc = Real(0);
        for (int t0 = 0; __any_sync(0xffffffffu, t0 < T); t0 += 4) {
          const int t = t0 + seg, r = t - tot;
          Real x = Real(0), y = Real(0);
          if (t < tot) {
            const unsigned off = t < n ? 12 * (r0 + t) : bs[t];
            x = w.J[off + k];
            y = -hR * lam[off / 12u];
          } else if (on && r < nm) {
            x = k < 3 ? sc.mass[b] : w.Iw[9 * b + 3 * (k - 3) + (r >> 1)];
            const int q = 6 * b + (k < 3 ? k : 3 + (r >> 1));
            if (r & 1) { x = -x; y = w.um[q]; } else { y = u[q]; }
          } else if (on && r == nm) {
            x = -hR;
            y = w.f[6 * b + k];
          }
          const Real p = rn_mul(x, y), ep = rn_fma(x, y, -p);
          Real sb = Real(0), sa = Real(0);
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const Real t1 = rn_add(s, __shfl_sync(0xffffffffu, p, lane3 - q));
            if (seg == q) { sb = s; sa = t1; }
            s = t1;
          }
          const Real bp = rn_sub(sa, sb), es = rn_add(rn_sub(sb, rn_sub(sa, bp)), rn_sub(p, bp));
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            cc = rn_add(cc, __shfl_sync(0xffffffffu, es, lane3 - q));
            cc = rn_add(cc, __shfl_sync(0xffffffffu, ep, lane3 - q));
          }
        }
        if (on && seg == 0) w.rdyn[6 * b + k] = rn_add(s, cc);
      }
    } else {
      for (int task = tid; task < 6 * nb; task += nth) {
        const int b = task / 6, k = task - 6 * (task / 6);
        acc2<Real> rd;
        body_rows(sc, w, b, [&](int off, int i) { rd.add_prod(w.J[off + k], -hR * lam[i]); });
        if (k < 3) {
          const Real m_ = sc.mass[b];
          rd.add_prod(m_, u[6 * b + k]);
          rd.add_prod(-m_, w.um[6 * b + k]);
        } else {
          for (int c = 0; c < 3; ++c) {
            rd.add_prod(w.Iw[9 * b + 3 * (k - 3) + c], u[6 * b + 3 + c]);
            rd.add_prod(-w.Iw[9 * b + 3 * (k - 3) + c], w.um[6 * b + 3 + c]);
          }
        }
        rd.add_prod(-hR, w.f[6 * b + k]);
        w.rdyn[6 * b + k] = rd.value();
      }
    }
  }
  __syncthreads();
  Real part = Real(0);
  for (int b = tid; b < nb && dyn; b += nth) {
    const Real* rv = w.rdyn + 6 * b;
    Real mi = sc.minv[b];
    vec3<Real> iw = mat3<Real>(w.Iwi + 9 * b, v3(rv[3], rv[4], rv[5]));
    Real mr[6] = {rv[0] * mi, rv[1] * mi, rv[2] * mi, iw.x, iw.y, iw.z};
    for (int k = 0; k < 6; ++k) { w.mr[6 * b + k] = mr[k]; part += mr[k] * mr[k]; }
  }
  Real dpart = 0;
  if (tid < w.sum_nth)
    for (int i = tid; i < m; i += w.sum_nth) {
      if (dyn) part += w.r2[i] * w.r2[i];
      dpart += hR * w.tmp[i];
    }
  block_sum2(w, part, dpart);
  if (tid == 0) w.scal[2] = m > 0 ? sc.delta_rel * dpart / Real(m) : Real(0);
  __syncthreads();                         // scal[2] is read by the assembly that follows
  return part;
}

// ---------------------------------------------------------------------------
// Schur assembly, factorisation and solves
// ---------------------------------------------------------------------------


// Row a of the packed lower triangle that entry e lies in: (2 a + 1)^2 <= 8 e + 1 < (2 a + 3)^2.
// Half a unit added under the root keeps it off these squares by more than 1e-5 of its value
// for every triangle here, far beyond the approximate root's error.
__device__ __forceinline__ int tri_row(int e) {
  float r;
  asm("sqrt.approx.f32 %0, %1;" : "=f"(r) : "f"((float)(8 * e + 1) + 0.5f));
  return (int)(0.5f * (r - 1.0f));
}

// The group blocks A_g, their coupling rows E_g and the separator block, all from J and
// Y = M^-1 J^T as the evaluation left them, in 3 x 3 (contact against contact, contact against
// three coupled rows) and 2 x 3 tiles (separator), a tile per thread and turn: a tile reads
// 6 rows for 9 products.  One thread per row, forming its own Y and taking its columns after
// one another, took 9.9 k cycles per Newton iteration of a robot, two threads per row 5.8 k.
template <class Real> __device__ __forceinline__ void assemble(const KScene<Real>& sc, WS<Real>& w, const StepH<Real>& h) {
  const int tid = w.tid, nth = blockDim.x;
  const int mc = w.ints[1], gstr = tri_size(sc.pg), ss = sc.ss, ldg = sc.ldg;
  const Real hR = h.h;
  // delta = delta_rel * mean diag(h J M^-1 J^T), formed by the evaluation at this iterate
  const Real delta = w.scal[2];
  // tiles of group g: its contact pairs, then its contacts by triples of coupled rows
  int g = 0, base = 0;
#pragma unroll 1
  for (int t = tid; ; t += nth) {
    int np = 0, nt = 0, nk = 0;
    for (; g < sc.n_groups; ++g) {
      const int nc = w.gn[g] / 3;
      np = tri_size(nc);
      nk = (sc.cpl_n[g] + 2) / 3;
      nt = np + nc * nk;
      if (t - base < nt) break;
      base += nt;
    }
    if (g >= sc.n_groups) break;
    // three rows a of contact ca against three rows b: those of contact cb <= ca, or three of
    // the group's coupled separator rows
    const int e = t - base, r0 = w.g0[g];
    const bool pair = e < np;
    int ca, cb, ob[3];
    if (pair) {
      ca = tri_row(e);
      cb = e - tri(ca, 0);
#pragma unroll
      for (int b = 0; b < 3; ++b) ob[b] = 12 * (r0 + 3 * cb + b);
    } else {
      ca = 0;
      for (cb = e - np; cb >= nk; cb -= nk) ++ca;
      const int bg = sc.group_body[g], last = sc.cpl_n[g] - 1;
#pragma unroll
      for (int b = 0; b < 3; ++b) {
        const int a = sc.cpl_row[g][3 * cb + b < last ? 3 * cb + b : last];
        ob[b] = 12 * (mc + a) + (sc.sep_b[a][0] == bg ? 0 : 6);
      }
    }
    const int ra = r0 + 3 * ca;
    Real v[3][3], y[3][6], x[6];
#pragma unroll
    for (int a = 0; a < 3; ++a) load6(w.J + 12 * (ra + a) + 6, y[a]);
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      load6(w.J + ob[b], x);
#pragma unroll
      for (int a = 0; a < 3; ++a) v[a][b] = rn_mul(hR, rowdot(x, 0, y[a], 0));
    }
    if (pair) {
      Real* Ga = w.G + g * gstr;
      if (ca == cb) {
        // a contact against itself: the diagonal and the radial friction terms
        const Real* rd = w.srad + 3 * row_ref(w.row[ra]);
#pragma unroll
        for (int a = 0; a < 3; ++a) v[a][a] = rn_add(v[a][a], rn_add(w.C[ra + a], delta));
        v[1][1] = rn_add(v[1][1], rd[0]); v[2][1] = rn_add(v[2][1], rd[1]); v[2][2] = rn_add(v[2][2], rd[2]);
      }
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        Real* Gr = Ga + tri(3 * ca + a, 3 * cb);
#pragma unroll
        for (int b = 0; b < 3; ++b)
          if (a >= b || ca != cb) Gr[b] = v[a][b];
      }
    } else {
      Real* Eb = w.E + (g * sc.cmax + 3 * cb) * ldg + 3 * ca;
#pragma unroll
      for (int b = 0; b < 3; ++b)
        if (3 * cb + b < sc.cpl_n[g])
#pragma unroll
          for (int a = 0; a < 3; ++a) Eb[b * ldg + a] = v[a][b];
    }
  }
  // Separator, in blocks of 6 x 6 rows (a joint's five and its servo row, or so), six tiles each.
  // Entry (a, b) is the sum of J_b . Y_a over the bodies the two rows share, parent parts of
  // row a first; a part no entry of the tile shares is skipped.
  const int nblk = tri_size((ss + 5) / 6);
#pragma unroll 1
  for (int t = nth - 1 - tid; t < 6 * nblk; t += nth) {
    const int blk = t / 6, in = t - 6 * blk, I = tri_row(blk);
    const int a0 = 6 * I + 2 * (in >> 1), b0 = 6 * (blk - tri(I, 0)) + 3 * (in & 1);
    if (b0 > a0 + 1 || a0 >= ss || b0 >= ss) continue;
    const int ar[2] = {a0, a0 + 1 < ss ? a0 + 1 : a0};
    const int br[3] = {b0, b0 + 1 < ss ? b0 + 1 : b0, b0 + 2 < ss ? b0 + 2 : b0};
    Real v[2][3] = {{Real(0), Real(0), Real(0)}, {Real(0), Real(0), Real(0)}};
#pragma unroll 1
    for (int part = 0; part < 4; ++part) {
      const int pa = part >> 1, pb = part & 1;
      bool on[2][3], any = false;
#pragma unroll
      for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b) {
          on[a][b] = sc.sep_b[ar[a]][pa] == sc.sep_b[br[b]][pb];
          any = any || on[a][b];
        }
      if (!any) continue;
      Real y[2][6], x[6];
#pragma unroll
      for (int a = 0; a < 2; ++a) load6(w.ys + 12 * ar[a] + 6 * pa, y[a]);
#pragma unroll
      for (int b = 0; b < 3; ++b) {
        load6(w.J + 12 * (mc + br[b]) + 6 * pb, x);
#pragma unroll
        for (int a = 0; a < 2; ++a) {
          const Real d = rowdot(x, 0, y[a], 0);
          if (on[a][b]) v[a][b] = rn_add(v[a][b], d);
        }
      }
    }
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
      for (int b = 0; b < 3; ++b) {
        const int ra = a0 + a, cb = b0 + b;
        if (ra >= ss || cb > ra) continue;
        Real x = rn_mul(v[a][b], hR);
        if (ra == cb) x = rn_add(x, rn_add(w.C[mc + ra], delta));
        w.S[tri(ra, cb)] = x;
      }
  }
  __syncthreads();
}

// L^-1 of an n x n symmetric positive definite block, in place, by one warp.  A (packed
// lower triangle, tri()) holds the block on entry and L^-1 on return, L L^T = A; colbuf
// holds n values.  Right-looking, one pivot k at a time:
//   pass 1: column k of L below the pivot goes to colbuf; row k of L^-1 is finished,
//           X[k][c] = Xt[k][c] / L[k][k] (its partial sums Xt already sit in row k);
//   pass 2: rank-one updates of the trailing block, A[i][j] -= L[i][k] L[j][k]
//           (k < j <= i), and of the rows of L^-1 below, Xt[i][c] -= L[i][k] X[k][c]
//           (c <= k).  Position (i, k) changes from L[i][k], now in colbuf and never
//           read again, to Xt[i][k].
// Each element of L and of L^-1 receives the same operations in the same order as the
// sequential column-by-column factor and forward substitution (k, resp. l,
// ascending), so the result does not depend on how the rows are shared out.
template <class Real> __device__ void chol_inv_inplace(Real* A, int n, Real* colbuf) {
  const int t = threadIdx.x & 31;
  for (int k = 0; k < n; ++k) {
    const Real akk = A[tri(k, k)];
    const Real inv = pivot_rsqrt(akk > Real(0) ? akk : Real(1e-30));
    const Real xkk = inv;                   // X[k][k], known to every thread
    for (int e = t; e < n; e += 32) {        // the pivot entry itself is left for pass 2
      if (e > k) colbuf[e] = A[tri(e, k)] * inv;
      else if (e < k) A[tri(k, e)] *= inv;
    }
    __syncwarp();
    if (t == 0) A[tri(k, k)] = xkk;
    // lanes own columns (j = t, t + 32, ...)
    for (int j = t; j < n; j += 32) {
      // per column: the multiplier of l_ik (X[k][j], X[k][k] or l_jk) and whether the
      // entry keeps its value (no branch inside the row loop)
      const Real coef = j < k ? A[tri(k, j)] : (j == k ? xkk : colbuf[j]);
      const bool keep = j != k;
      int i = k + 1 > j ? k + 1 : j;
      for (; i + 3 < n; i += 4) {             // four independent rows per pass
        const int i1 = i + 1, i2 = i + 2, i3 = i + 3;
        const Real l0 = colbuf[i], l1 = colbuf[i1], l2 = colbuf[i2], l3 = colbuf[i3];
        Real* a0 = A + tri(i, j);
        Real* a1 = A + tri(i1, j);
        Real* a2 = A + tri(i2, j);
        Real* a3 = A + tri(i3, j);
        const Real o0 = keep ? *a0 : Real(0), o1 = keep ? *a1 : Real(0);
        const Real o2 = keep ? *a2 : Real(0), o3 = keep ? *a3 : Real(0);
        *a0 = o0 - l0 * coef; *a1 = o1 - l1 * coef; *a2 = o2 - l2 * coef; *a3 = o3 - l3 * coef;
      }
      for (; i < n; ++i) {
        const Real lik = colbuf[i];
        Real* aij = A + tri(i, j);
        const Real old = keep ? *aij : Real(0);
        *aij = old - lik * coef;
      }
    }
    __syncwarp();
  }
}

__device__ __forceinline__ void load4(const float* b, float* v) {
  const float4 x = *reinterpret_cast<const float4*>(b);
  v[0] = x.x; v[1] = x.y; v[2] = x.z; v[3] = x.w;
}
__device__ __forceinline__ void load4(const double* b, double* v) {
  const double2 x = reinterpret_cast<const double2*>(b)[0], y = reinterpret_cast<const double2*>(b)[1];
  v[0] = x.x; v[1] = x.y; v[2] = y.x; v[3] = y.y;
}

// Column `lane` of the symmetric n x n block whose packed lower triangle is A (zeros past its
// end); the addresses are clamped rather than the loads predicated, so that all are in flight
// together.
template <int NR, class Real> __device__ __forceinline__ void load_column(const Real* A, int n, int lane, Real (&a)[NR]) {
  const int last = n > 0 ? tri_size(n) - 1 : 0;
#pragma unroll
  for (int r = 0; r < NR; ++r) {
    const int i = r >= lane ? tri(r, 0) + lane : tri(lane, 0) + r;
    const Real v = A[i < last ? i : last];
    a[r] = r < n && lane < n ? v : Real(0);
  }
}

// L^-1 of an n x n symmetric positive definite block in place, as chol_inv_inplace, by TW
// lanes of a warp (32, or 16 with two blocks per warp) with the block in registers:
// 0 < n <= TW; nmax is the largest n in the warp (its lanes leave the loop together).
// Lane j holds column j of the symmetric block, later of L^-1: rows k .. n-1 at the k-th
// pivot, the pivot row always in a[0] (the rows move up by one as they are updated, so
// that one loop body serves every pivot).  Column k of L is row k of the symmetric block
// times 1/L[k][k], so every lane supplies its own entry of it, exchanged through `buf` (2 TW
// values, 16-byte aligned, the team's own; two halves in turn: one warp barrier per
// pivot).  Row k of L^-1 is then final and goes to A.  Every entry receives the operations
// of chol_inv_inplace in the same order.
//
// FP64: its multiply-adds bound it (two a clock per SM), so rows past the end are left out.  Of
// two blocks in a warp the shorter one goes on with the longer one's pivots: on its own, which
// are zero, its lanes would go the other way at the test for a positive pivot, and the warp
// through the root twice (37 boxes, step and adjoint: 754 -> 707 us).
// The reciprocal root is some 1000 cycles of the warp's arithmetic unit, half of a pivot.
// PAIR: a second warp (chol_roots), on another unit, takes the root of the next diagonal --
// which lane k + 1 forms from its own entries alone (a - c c) -- while this one updates the
// rows.  They meet at the named barriers bar and bar + 1 of their 64 threads, both nmax - 1
// times, and exchange through xch (4 values).  The 24 x 24 separator of a robot: 53.2 -> 42.9 k
// cycles.
__device__ __forceinline__ void pair_sync(int id) {
  __syncwarp();
  asm volatile("bar.sync %0, 64;" ::"r"(id) : "memory");
}

template <int TW, bool PAIR = false>
__device__ __forceinline__ void chol_inv_regs(double* A, int n, int nmax, double* buf, double* xch = nullptr,
                                              int bar = 0) {
  const int lane = threadIdx.x & (TW - 1), half = (threadIdx.x & 31) / TW;
  double a[TW];
  load_column(A, n, lane, a);
  double* row = A + lane;
  double inv;
#pragma unroll 1
  for (int k = 0; k < nmax; ++k) {
    if (!PAIR || k == 0) {
      const double akk = __shfl_sync(0xffffffffu, a[0], TW == 32 ? k : (n > k ? half : half ^ 1) * TW + k);
      inv = pivot_rsqrt(akk > 0.0 ? akk : 1e-30);
    } else {
      pair_sync(bar + 1);
      inv = xch[2 + half];
    }
    const bool piv = lane == k;
    const double c = piv ? inv : a[0] * inv;
    double* bk = buf + (k & 1 ? TW : 0);
    if (lane > k) bk[lane - k - 1] = c;
    if (PAIR && lane == k + 1) xch[half] = rn_fma(-c, c, a[1]);
    if (PAIR && k + 1 < nmax) pair_sync(bar);
    if (lane <= k && k < n) *row = c;
    row += k + 1;
    __syncwarp();
#pragma unroll
    for (int q = 0; q < TW; q += 4)
      if (q < nmax - 1 - k) {
        double l[4];
        load4(bk + q, l);
#pragma unroll
        for (int r = 0; r < 4; ++r)
          if (q + r + 1 < TW) a[q + r] = rn_fma(-l[r], c, piv ? 0.0 : a[q + r + 1]);
      }
  }
}

// The second warp of a pair: the reciprocal roots of the pivots after the first.
template <int TW> __device__ __forceinline__ void chol_roots(int n, int nmax, double* xch, int bar) {
  const int half = (threadIdx.x & 31) / TW;
#pragma unroll 1
  for (int k = 1; k < nmax; ++k) {
    pair_sync(bar);
    const double d = xch[TW == 32 || n > k ? half : half ^ 1], inv = pivot_rsqrt(d > 0.0 ? d : 1e-30);
    if ((threadIdx.x & (TW - 1)) == 0) xch[2 + half] = inv;
    pair_sync(bar + 1);
  }
}

// FP32: what bounds a pivot is the chain from row to row -- multiply, exchange, update of the
// next row -- and beside it the reciprocal root of the next diagonal, which lane k + 1 forms
// from its own entries alone (a - c c).  The other rows' updates are put off by one pivot, into
// the shadow of the next exchange, and the rows taken shrink from 32 or 16 by eights as the
// block does.  A 24 x 24 block takes 2.8 k cycles of one warp (5.9 k with the updates in their
// own pivot, tested eight rows at a time; two pivots per exchange with paired
// multiply-adds 4.5 k), a 12 x 12 block 1.3 k (2.8 k).
//
// One pivot k.  On entry a[0] is row k, updated by all pivots before; the other rows still
// lack the update of pivot k - 1, whose column is lp (lp[r]: row k + r) and whose multiplier
// in this lane is cp (the lane's rows restart from 0 where its own column was that pivot).
// Returns with the rows moved up by one, l the column of pivot k (l[r]: row k + 1 + r), c its
// multiplier and inv 1 / L[k+1][k+1].  NS: rows taken.
template <int NS, int TW>
__device__ __forceinline__ void chol_pivot(float (&a)[TW], const float (&lp)[TW], float (&l)[TW], float cp, float& c,
                                           float& inv, int k, int n, float* bk, float* row) {
  const int lane = threadIdx.x & (TW - 1);
  const bool piv = lane == k, kp = lane == k - 1;
  c = piv ? inv : a[0] * inv;
  if (lane > k) bk[lane - k - 1] = c;
  if (lane <= k && k < n) row[lane] = c;
  __syncwarp();
#pragma unroll
  for (int q = 0; q < NS; q += 4) load4(bk + q, l + q);
  a[0] = rn_fma(-lp[1], cp, kp ? 0.0f : a[1]);
  const float d = rn_fma(-c, c, a[0]);
  const float next = pivot_rsqrt(d > 0.0f ? d : 1e-30f);
#pragma unroll
  for (int r = 2; r < NS; ++r) a[r - 1] = rn_fma(-lp[r], cp, kp ? 0.0f : a[r]);
  inv = __shfl_sync(0xffffffffu, next, k + 1, TW);
  a[0] = rn_fma(-l[0], c, piv ? 0.0f : a[0]);
}

// The pivots at which NS rows, but not NS - 8, are needed; two per turn, so that the columns of
// the last two pivots change places without moves.
template <int NS, int TW>
__device__ __forceinline__ void chol_stage(float (&a)[TW], float (&l0)[TW], float (&l1)[TW], float& c0, float& c1,
                                           float& inv, int& k, int n, int nmax, float* buf, float*& row) {
#pragma unroll 1
  for (; k < nmax && (NS == 8 || nmax - k > NS - 8); k += 2) {
    chol_pivot<NS, TW>(a, l1, l0, c1, c0, inv, k, n, buf, row);
    row += k + 1;
    chol_pivot<NS, TW>(a, l0, l1, c0, c1, inv, k + 1, n, buf + TW, row);
    row += k + 2;
  }
}

template <int TW> __device__ __forceinline__ void chol_inv_regs(float* A, int n, int nmax, float* buf) {
  const int lane = threadIdx.x & (TW - 1);
  float a[TW], l0[TW], l1[TW];
  load_column(A, n, lane, a);
#pragma unroll
  for (int r = 0; r < TW; ++r) l1[r] = 0.0f;
  const float a00 = __shfl_sync(0xffffffffu, a[0], 0, TW);
  float inv = pivot_rsqrt(a00 > 0.0f ? a00 : 1e-30f), c0 = 0.0f, c1 = 0.0f;
  float* row = A;
  int k = 0;
  if (TW == 32) {
    chol_stage<TW, TW>(a, l0, l1, c0, c1, inv, k, n, nmax, buf, row);
    chol_stage<TW - 8, TW>(a, l0, l1, c0, c1, inv, k, n, nmax, buf, row);
  }
  chol_stage<16, TW>(a, l0, l1, c0, c1, inv, k, n, nmax, buf, row);
  chol_stage<8, TW>(a, l0, l1, c0, c1, inv, k, n, nmax, buf, row);
}

// The inverse factors of the contact groups' blocks.  Blocks of up to 16 rows (five of a
// wheel's slots active; a robot on flat ground has 6 rows per wheel) go two to a warp, larger
// ones one to a warp, and blocks beyond 32 rows through shared memory.  With few worlds in FP64
// the second half of the warps takes the roots of the first half's pivots, where that leaves
// every warp at most one block (or two of 16 rows).
template <bool FEW, class Real> __device__ __forceinline__ void factor_groups(const KScene<Real>& sc, WS<Real>& w) {
  const int tid = w.tid, wid = tid >> 5, nw = blockDim.x >> 5;
  const int ng = sc.n_groups, gstr = tri_size(sc.pg);
  int big = 0;
  for (int g = 0; g < ng; ++g) big = w.gn[g] > big ? w.gn[g] : big;
  if constexpr (FEW && sizeof(Real) == 8) {
    const int hw = nw >> 1, per = big <= 16 ? 2 : 1;
    if (big <= 32 && ng <= per * hw) {
      const int job = wid < hw ? wid : wid - hw, bar = 1 + 2 * job, half = per == 2 ? (tid >> 4) & 1 : 0;
      const int g0 = per * job, g = g0 + half, na = g0 < ng ? w.gn[g0] : 0;
      const int nb = per == 2 && g0 + 1 < ng ? w.gn[g0 + 1] : 0, nmax = na > nb ? na : nb;
      Real* xch = w.prow + 64 * (hw + job);
      Real* A = w.G + (g < ng ? g : 0) * gstr;
      const int n = g < ng ? w.gn[g] : 0;
      if (wid >= 2 * hw || nmax == 0) return;
      if (per == 2) {
        if (wid < hw) chol_inv_regs<16, true>(A, n, nmax, w.prow + 64 * wid + 32 * half, xch, bar);
        else chol_roots<16>(n, nmax, xch, bar);
      } else {
        if (wid < hw) chol_inv_regs<32, true>(A, n, nmax, w.prow + 64 * wid, xch, bar);
        else chol_roots<32>(n, nmax, xch, bar);
      }
      return;
    }
  }
  if (big <= 16) {
    const int half = (tid >> 4) & 1;
    Real* buf = w.prow + 64 * wid + 32 * half;
    for (int g0 = 2 * wid; g0 < ng; g0 += 2 * nw) {
      const int g = g0 + half, n = g < ng ? w.gn[g] : 0;
      const int na = w.gn[g0], nb = g0 + 1 < ng ? w.gn[g0 + 1] : 0, nmax = na > nb ? na : nb;
      if (nmax > 0) chol_inv_regs<16>(w.G + (g < ng ? g : g0) * gstr, n, nmax, buf);
    }
  } else {
    for (int g = wid; g < ng; g += nw) {
      const int n = w.gn[g];
      if (n <= 32) chol_inv_regs<32>(w.G + g * gstr, n, n, w.prow + 64 * wid);
      else chol_inv_inplace(w.G + g * gstr, n, w.prow + 64 * wid);
    }
  }
}

// One round of P pivots (k .. k+P-1) of the in-place L^-1 by the whole CTA, P <= 4.  Every
// thread forms the P x P pivot block itself: the inverse pivots ip[p] = 1/L[k+p][k+p], the
// block's L below the diagonal and its inverse X.  Pass 1 gives columns k .. k+P-1 of L
// below the block (colbuf, n values per column) and finishes rows k .. k+P-1 of L^-1 left
// of it; pass 2 applies the P rank-one updates, in pivot order, to the trailing block and
// to the rows of L^-1 below.  Every element receives the operations of the one-pivot-per-
// round factor in the same order (k ascending); a round costs two barriers.
template <int P, class Real> __device__ void chol_round(Real* A, int n, int k, Real* colbuf) {
  const int t = threadIdx.x, T = blockDim.x;
  Real a[P][P], l[P][P], x[P][P], xt[P][P], ip[P];
#pragma unroll
  for (int p = 0; p < P; ++p)
#pragma unroll
    for (int q = 0; q < P; ++q) { a[p][q] = q <= p ? A[tri(k + p, k + q)] : Real(0); xt[p][q] = Real(0); }
#pragma unroll
  for (int p = 0; p < P; ++p) {
    ip[p] = pivot_rsqrt(a[p][p] > Real(0) ? a[p][p] : Real(1e-30));
#pragma unroll
    for (int r = p + 1; r < P; ++r) l[r][p] = a[r][p] * ip[p];
#pragma unroll
    for (int r = p + 1; r < P; ++r)
#pragma unroll
      for (int c = p + 1; c <= r; ++c) a[r][c] = a[r][c] - l[r][p] * l[c][p];
  }
#pragma unroll
  for (int p = 0; p < P; ++p) {
#pragma unroll
    for (int q = 0; q < p; ++q) x[p][q] = xt[p][q] * ip[p];
    x[p][p] = ip[p];
#pragma unroll
    for (int r = p + 1; r < P; ++r) {
#pragma unroll
      for (int q = 0; q < p; ++q) xt[r][q] = xt[r][q] - l[r][p] * x[p][q];
      xt[r][p] = Real(0) - l[r][p] * x[p][p];
    }
  }
  // pass 1 writes neither the pivot block nor any entry another thread reads in this pass
  for (int e = t; e < n; e += T) {
    if (e >= k + P) {
      Real v[P];
#pragma unroll
      for (int p = 0; p < P; ++p) v[p] = A[tri(e, k + p)];
#pragma unroll
      for (int p = 0; p < P; ++p) {
        const Real c = v[p] * ip[p];
        colbuf[p * n + e] = c;
#pragma unroll
        for (int r = p + 1; r < P; ++r) v[r] = v[r] - c * l[r][p];
      }
    } else if (e < k) {
      Real y[P];
#pragma unroll
      for (int p = 0; p < P; ++p) y[p] = A[tri(k + p, e)];
#pragma unroll
      for (int p = 0; p < P; ++p) {
        const Real xe = y[p] * ip[p];
        A[tri(k + p, e)] = xe;
#pragma unroll
        for (int r = p + 1; r < P; ++r) y[r] = y[r] - l[r][p] * xe;
      }
    }
  }
  __syncthreads();
  if (t == 0) {
#pragma unroll
    for (int p = 0; p < P; ++p)
#pragma unroll
      for (int q = 0; q <= p; ++q) A[tri(k + p, k + q)] = x[p][q];
  }
  const int nw = T >> 5, lane = t & 31;
  for (int j = lane; j < n; j += 32) {
    // the P multipliers of column j, the first pivot that updates it (columns of the pivot
    // block took the earlier pivots' updates into colbuf) and whether the entry keeps its value
    Real m[P];
    int qs = 0;
    bool keep = true;
    if (j < k) {
#pragma unroll
      for (int p = 0; p < P; ++p) m[p] = A[tri(k + p, j)];
    } else if (j < k + P) {
      qs = j - k;
      keep = false;
#pragma unroll
      for (int p = 0; p < P; ++p) {
        Real xv = Real(0);
#pragma unroll
        for (int q = 0; q < P; ++q) if (q == j - k && q <= p) xv = x[p][q];
        m[p] = xv;
      }
    } else {
#pragma unroll
      for (int p = 0; p < P; ++p) m[p] = colbuf[p * n + j];
    }
    int i = (k + P > j ? k + P : j) + (t >> 5);
    for (; i + 3 * nw < n; i += 4 * nw) {                  // four independent rows per pass
      int ii[4] = {i, i + nw, i + 2 * nw, i + 3 * nw};
      Real v[4];
#pragma unroll
      for (int r = 0; r < 4; ++r) v[r] = keep ? A[tri(ii[r], j)] : Real(0);
#pragma unroll
      for (int p = 0; p < P; ++p)
        if (p >= qs)
#pragma unroll
          for (int r = 0; r < 4; ++r) v[r] = v[r] - colbuf[p * n + ii[r]] * m[p];
#pragma unroll
      for (int r = 0; r < 4; ++r) A[tri(ii[r], j)] = v[r];
    }
    for (; i < n; i += nw) {
      Real v = keep ? A[tri(i, j)] : Real(0);
#pragma unroll
      for (int p = 0; p < P; ++p)
        if (p >= qs) v = v - colbuf[p * n + i] * m[p];
      A[tri(i, j)] = v;
    }
  }
  __syncthreads();
}

// In-place L^-1 of an n x n SPD block by the whole CTA: four pivots per round, the
// remainder two and one at a time.  colbuf holds 4 n values.
template <class Real> __device__ void chol_inv_inplace4(Real* A, int n, Real* colbuf) {
  int k = 0;
  for (; k + 3 < n; k += 4) chol_round<4>(A, n, k, colbuf);
  for (; k + 1 < n; k += 2) chol_round<2>(A, n, k, colbuf);
  if (k < n) chol_round<1>(A, n, k, colbuf);
}

// L_s^-1 of the separator block in place over S: in one warp's registers up to 32 rows (the
// CTA's other warps do not join; with few worlds in FP64 the last of four warps takes the
// pivots' roots), else by the whole CTA through shared memory.  The caller synchronises.
template <bool FEW, class Real> __device__ __forceinline__ void factor_separator(const KScene<Real>& sc, WS<Real>& w) {
  if constexpr (FEW && sizeof(Real) == 8) {
    if (blockDim.x == 128 && sc.ss > 0 && sc.ss <= 32) {
      if (w.tid < 32) chol_inv_regs<32, true>(w.S, sc.ss, sc.ss, w.prow, w.prow + 64 * 3, 1);
      else if (w.tid >= 96) chol_roots<32>(sc.ss, sc.ss, w.prow + 64 * 3, 1);
      return;
    }
  }
  if (sc.ss > 32) chol_inv_inplace4(w.S, sc.ss, w.prow);
  else if (w.tid < 32 && sc.ss > 0) chol_inv_regs<32>(w.S, sc.ss, sc.ss, w.prow);
}

// Two-accumulator dot products (even and odd terms apart, halving the dependent chain):
// a contiguous one, and one down a column of a packed triangle (element (l, c), l = c ..
// n-1, at tri(l, c)).  Eight terms at a time, the loads of all eight in flight together,
// terms past the end zero: the vectors are short (6 to 24), and a plain loop waits for
// shared memory once per pair while its unrolled copies and remainders fill the
// instruction cache.
template <class Real> __device__ __forceinline__ Real dot2c(const Real* a, const Real* b, int n) {
  Real s0 = Real(0), s1 = Real(0);
#pragma unroll 1
  for (int l = 0; l < n; l += 8) {
    Real x[8], y[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      x[q] = l + q < n ? a[l + q] : Real(0);
      y[q] = l + q < n ? b[l + q] : Real(0);
    }
#pragma unroll
    for (int q = 0; q < 8; q += 2) {
      s0 = rn_fma(x[q], y[q], s0);
      s1 = rn_fma(x[q + 1], y[q + 1], s1);
    }
  }
  return rn_add(s0, s1);
}
template <class Real> __device__ __forceinline__ Real dot2col(const Real* T, int c, int n, const Real* b) {
  Real s0 = Real(0), s1 = Real(0);
#pragma unroll 1
  for (int l = c; l < n; l += 8) {
    const Real* Tl = T + tri(l, c);
    Real x[8], y[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      x[q] = l + q < n ? Tl[q * l + ((q * (q + 1)) >> 1)] : Real(0);
      y[q] = l + q < n ? b[l + q] : Real(0);
    }
#pragma unroll
    for (int q = 0; q < 8; q += 2) {
      s0 = rn_fma(x[q], y[q], s0);
      s1 = rn_fma(x[q + 1], y[q + 1], s1);
    }
  }
  return rn_add(s0, s1);
}

// Block-arrowhead factorisation kept in inverse form for row-parallel solves:
//   Li_g = L_g^-1 with L_g L_g^T = A_g (contact groups; stored in G, packed),
//   F_g = E_g L_g^-T (coupled separator rows; stored in H),
//   Lsi = L_s^-1 with L_s L_s^T = S - sum_g F_g F_g^T, the reduced separator (stored in S,
//   packed).
// Here all but the last; factor_separator follows.
template <bool FEW, class Real> __device__ __forceinline__ void factor_eliminate(const KScene<Real>& sc, WS<Real>& w) {
  const int tid = w.tid, nth = blockDim.x;
  const int ldg = sc.ldg, cm = sc.cmax, gstr = tri_size(sc.pg);
  factor_groups<FEW>(sc, w);
  __syncthreads();
  // F_g[k][j] = sum_{l <= j} E_g[k][l] Li_g[j][l], two threads per contact row
  const int mc = w.ints[1];
  for (int r = tid >> 1; r < mc; r += nth >> 1) {
    const int g = row_grp(w.row[r]), j = r - w.g0[g], nc = sc.cpl_n[g];
    const Real* Lj = w.G + g * gstr + tri(j, 0);
    for (int k = tid & 1; k < nc; k += 2)
      w.H[(g * cm + k) * ldg + j] = dot2c(w.E + (g * cm + k) * ldg, Lj, j + 1);
  }
  __syncthreads();
  // S' = S - sum_g F_g F_g^T: two threads per coupled row k1 of a group take its pairs k2 <= k1
  // in turn.  All groups at once, or one after another where a joint's two bodies both
  // carry one and an entry of its rows takes both groups' terms.
  const int ng = sc.n_groups, ng_at_once = sc.sep_shared ? 1 : ng;
  for (int g0 = 0; g0 < ng; g0 += ng_at_once) {
    for (int e = tid >> 1; e < ng_at_once * cm; e += nth >> 1) {
      int g = g0, k1 = e;
      while (k1 >= cm) { k1 -= cm; ++g; }
      const int n = w.gn[g];
      if (n == 0 || k1 >= sc.cpl_n[g]) continue;
      const Real* Fb = w.H + g * cm * ldg;
      Real* Sa = w.S + tri(sc.cpl_row[g][k1], 0);
      for (int k2 = tid & 1; k2 <= k1; k2 += 2) Sa[sc.cpl_row[g][k2]] -= dot2c(Fb + k1 * ldg, Fb + k2 * ldg, n);
    }
    __syncthreads();
  }
  if (ng == 0) __syncthreads();
}

// v <- A^-1 v with the inverse-form block-arrowhead factor, in three parts.
// Groups, forward: y_g = Li_g b_g, then the separator's right-hand side
// b_s' = b_s - sum_g F_g y_g, by the T threads t = 0 .. T-1 that sync() joins (needs no S).
template <class Real, class Sync>
__device__ __forceinline__ void arrow_forward(const KScene<Real>& sc, WS<Real>& w, const Real* v, int t, int T,
                                              Sync&& sync) {
  const int gstr = tri_size(sc.pg), ldg = sc.ldg, cm = sc.cmax, mc = w.ints[1];
  Real* y = w.tmp;
  Real* z = w.tmp2;
  for (int r = t; r < mc; r += T) {
    const int g = row_grp(w.row[r]), r0 = w.g0[g], i = r - r0;
    y[r] = dot2c(w.G + g * gstr + tri(i, 0), v + r0, i + 1);
  }
  sync();
  for (int a = t; a < sc.ss; a += T) {
    Real acc = v[mc + a];
    for (int pa = 0; pa < sc.sep_n[a]; ++pa) {
      const int g = sc.sep_g[a][pa];
      acc -= dot2c(w.H + (g * cm + sc.sep_k[a][pa]) * ldg, y + w.g0[g], w.gn[g]);
    }
    z[a] = acc;
  }
}

// Separator, by one warp: y_s = Lsi b_s', x_s = Lsi^T y_s into v.
template <class Real> __device__ __forceinline__ void arrow_separator(const KScene<Real>& sc, WS<Real>& w, Real* v) {
  const int lane = threadIdx.x & 31, ss = sc.ss, mc = w.ints[1];
  Real* y = w.tmp + mc;
  for (int a = lane; a < ss; a += 32) y[a] = dot2c(w.S + tri(a, 0), w.tmp2, a + 1);
  __syncwarp();
  for (int a = lane; a < ss; a += 32) v[mc + a] = dot2col(w.S, a, ss, y);
}

// Groups, backward, by the whole CTA: x_g = Li_g^T (y_g - F_g^T x_s) into v.
template <class Real> __device__ __forceinline__ void arrow_backward(const KScene<Real>& sc, WS<Real>& w, Real* v) {
  const int tid = w.tid, nth = blockDim.x;
  const int gstr = tri_size(sc.pg), ldg = sc.ldg, cm = sc.cmax, mc = w.ints[1];
  const Real* y = w.tmp;
  Real* z = w.tmp2;
  for (int r = tid; r < mc; r += nth) {
    const int g = row_grp(w.row[r]), i = r - w.g0[g], nc = sc.cpl_n[g];
    const Real* Fb = w.H + g * cm * ldg + i;
    Real s0 = y[r], s1 = Real(0);
#pragma unroll 1
    for (int k = 0; k < nc; k += 8) {
      Real x[8], f[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        x[q] = k + q < nc ? v[mc + sc.cpl_row[g][k + q]] : Real(0);
        f[q] = k + q < nc ? Fb[(k + q) * ldg] : Real(0);
      }
#pragma unroll
      for (int q = 0; q < 8; q += 2) {
        s0 = rn_fma(-f[q], x[q], s0);
        s1 = rn_fma(-f[q + 1], x[q + 1], s1);
      }
    }
    z[r] = rn_add(s0, s1);
  }
  __syncthreads();
  for (int r = tid; r < mc; r += nth) {
    const int g = row_grp(w.row[r]), r0 = w.g0[g], i = r - r0;
    v[r] = dot2col(w.G + g * gstr, i, w.gn[g], z + r0);
  }
  __syncthreads();
}

template <class Real> __device__ __forceinline__ void arrow_solve(const KScene<Real>& sc, WS<Real>& w, Real* v) {
  arrow_forward(sc, w, v, w.tid, blockDim.x, [] { __syncthreads(); });
  __syncthreads();
  if (w.tid < 32) arrow_separator(sc, w, v);
  __syncthreads();
  arrow_backward(sc, w, v);
}

// out_b = sum over rows touching body b of J_row,b^T x_row (6 per body), a thread per
// component; with ACC exact products and exact partial sums.
template <bool ACC, class Real>
__device__ __forceinline__ void jt_apply(const KScene<Real>& sc, WS<Real>& w, const Real* x, Real* out) {
  for (int task = w.tid; task < 6 * sc.nb; task += blockDim.x) {
    const int b = task / 6, k = task - 6 * (task / 6);
    acc2<Real> ca;
    Real acc = Real(0);
    body_rows(sc, w, b, [&](int off, int i) {
      if (ACC) ca.add_prod(w.J[off + k], x[i]);
      else acc += w.J[off + k] * x[i];
    });
    out[task] = ACC ? ca.value() : acc;
  }
}

// M^-1 v per body (6 per body)
template <class Real> __device__ __forceinline__ void minv6(const KScene<Real>& sc, const WS<Real>& w, int b, const Real* v,
                                                            Real* o) {
  Real mi = sc.minv[b];
  o[0] = v[0] * mi; o[1] = v[1] * mi; o[2] = v[2] * mi;
  vec3<Real> a = mat3<Real>(w.Iwi + 9 * b, v3(v[3], v[4], v[5]));
  o[3] = a.x; o[4] = a.y; o[5] = a.z;
}

// Schur solve with iterative refinement: x = A^-1 b with the arrowhead factor, then
// `sweeps` corrections x += A^-1 (b - A x), where A x = h J (M^-1 J^T x) + (C + delta) x
// (+ the radial friction blocks) is formed matrix-free from J.  b is kept in `b`,
// the solution is returned in `x`; t6 (6 per body) and r (rows) are scratch.
template <class Real>
__device__ void schur_solve(const KScene<Real>& sc, WS<Real>& w, const Real* b, Real* x, Real* t6, Real* r, const StepH<Real>& h,
                            int sweeps, Real stop_rel = Real(0)) {
  const int tid = w.tid, nth = blockDim.x, m = w.ints[0];
  const Real hR = h.h;
  // pass -1 solves for x itself (its correction from x = 0 is A^-1 b), so that one inlined
  // copy of the arrowhead solve serves the first solve and the sweeps
  for (int i = tid; i < m; i += nth) { x[i] = Real(0); r[i] = b[i]; }
  __syncthreads();
  const Real delta = w.scal[2];
  for (int sweep = -1; sweep < sweeps; ++sweep) {
    if (sweep >= 0) {
      jt_apply<false>(sc, w, x, t6);
      __syncthreads();
      for (int bb = tid; bb < sc.nb; bb += nth) {
        Real o[6];
        minv6(sc, w, bb, t6 + 6 * bb, o);
        for (int k = 0; k < 6; ++k) t6[6 * bb + k] = o[k];
      }
      __syncthreads();
      for (int i = tid; i < m; i += nth) {
        const Real* Ji = w.J + 12 * i;
        int b0 = row_b0(w.row[i]), b1 = row_b1(w.row[i]);
        acc2<Real> ax;
        for (int k = 0; k < 6; ++k) ax.add_prod(Ji[k], t6[6 * b0 + k]);
        if (b1 >= 0) for (int k = 0; k < 6; ++k) ax.add_prod(Ji[6 + k], t6[6 * b1 + k]);
        acc2<Real> res;                   // r = b - A x, compensated throughout
        res.add(b[i]);
        res.add_prod(-hR, ax.s);
        res.add_prod(-hR, ax.c);
        res.add_prod(-(w.C[i] + delta), x[i]);
        int t = row_type(w.row[i]), sub = row_sub(w.row[i]);
        if (t == ROW_FRIC) {
          const Real* rd = w.srad + 3 * row_ref(w.row[i]);
          if (sub == 1) { res.add_prod(-rd[0], x[i]); res.add_prod(-rd[1], x[i + 1]); }
          else { res.add_prod(-rd[1], x[i - 1]); res.add_prod(-rd[2], x[i]); }
        }
        r[i] = res.value();
      }
      __syncthreads();
    }
    arrow_solve(sc, w, r);
    Real cmax = Real(0), xmax = Real(0);
    for (int i = tid; i < m; i += nth) {
      x[i] += r[i];
      cmax = fmax(cmax, fabs(r[i]));
      xmax = fmax(xmax, fabs(x[i]));
    }
    __syncthreads();
    // optional early stop once the correction no longer changes x at working precision
    if (sweep >= 0 && stop_rel > Real(0)) {
      block_max2(w, cmax, xmax);
      if (cmax <= stop_rel * xmax) break;
    }
  }
}

// ---------------------------------------------------------------------------
// matrix-free Schur operator and preconditioned conjugate residual (Sec. III-C)
// ---------------------------------------------------------------------------
// out = A v, A = h J M^-1 J^T + C + delta I (+ the radial friction blocks), from the rows:
// t6 = J^T v per body component (a thread per component, over the rows touching the
// body), then per row h J_i M^-1 t6 plus the diagonal and radial terms.  ACC: exact
// products and compensated sums throughout (the adjoint's solve).  Returns this thread's
// part of v . out; the caller reduces it (the rows are written by their owning threads).
template <class Real, bool ACC>
__device__ Real schur_apply(const KScene<Real>& sc, WS<Real>& w, const Real* v, Real* out, Real* t6, const StepH<Real>& h) {
  const int tid = w.tid, nth = blockDim.x, m = w.ints[0];
  jt_apply<ACC>(sc, w, v, t6);
  __syncthreads();
  const Real hR = h.h, delta = w.scal[2];
  Real part = Real(0);
  for (int i = tid; i < m; i += nth) {
    const Real* Ji = w.J + 12 * i;
    acc2<Real> ca;
    Real ax = Real(0);
    for (int side = 0; side < 2; ++side) {
      const int b = (side ? row_b1(w.row[i]) : row_b0(w.row[i]));
      if (b < 0) continue;
      Real o[6];
      minv6(sc, w, b, t6 + 6 * b, o);
      for (int q = 0; q < 6; ++q) {
        if (ACC) ca.add_prod(Ji[6 * side + q], o[q]);
        else ax += Ji[6 * side + q] * o[q];
      }
    }
    Real y;
    const int t = row_type(w.row[i]), sub = row_sub(w.row[i]);
    if (ACC) {
      acc2<Real> ya;
      ya.add_prod(hR, ca.s);
      ya.add_prod(hR, ca.c);
      ya.add_prod(w.C[i] + delta, v[i]);
      if (t == ROW_FRIC) {
        const Real* rd = w.srad + 3 * row_ref(w.row[i]);
        if (sub == 1) { ya.add_prod(rd[0], v[i]); ya.add_prod(rd[1], v[i + 1]); }
        else { ya.add_prod(rd[1], v[i - 1]); ya.add_prod(rd[2], v[i]); }
      }
      y = ya.value();
    } else {
      y = hR * ax + (w.C[i] + delta) * v[i];
      if (t == ROW_FRIC) {
        const Real* rd = w.srad + 3 * row_ref(w.row[i]);
        y += sub == 1 ? rd[0] * v[i] + rd[1] * v[i + 1] : rd[1] * v[i - 1] + rd[2] * v[i];
      }
    }
    out[i] = y;
    part += v[i] * y;
  }
  return part;
}

// Jacobi preconditioner: the inverse diagonal of A, stored per row by the row's thread
template <class Real> __device__ void pcr_jacobi(const KScene<Real>& sc, WS<Real>& w, const StepH<Real>& h) {
  const int tid = w.tid, nth = blockDim.x, m = w.ints[0], mc = w.ints[1];
  const Real hR = h.h, delta = w.scal[2];
  Real* pd = w.pcr + 6 * sc.m_max;
  for (int i = tid; i < m; i += nth) {
    const Real* Ji = w.J + 12 * i;
    const Real* Ys = w.ys + 12 * (i - mc);
    const Real jy = i < mc ? rowdot6(Ji, Ji + 6) : rowdot6(Ji, Ys) + rowdot6(Ji + 6, Ys + 6);
    Real d = hR * jy + w.C[i] + delta;
    if (row_type(w.row[i]) == ROW_FRIC) d += w.srad[3 * row_ref(w.row[i]) + (row_sub(w.row[i]) == 1 ? 0 : 2)];
    pd[i] = Real(1) / d;
  }
}

// Block-Jacobi preconditioner: each contact group's block and the (unreduced) separator
// block of A, as assembled, factored in place to their inverse Cholesky factors (G, S)
template <class Real> __device__ __forceinline__ void factor_blocks(const KScene<Real>& sc, WS<Real>& w) {
  factor_groups<false>(sc, w);
  __syncthreads();
  factor_separator<false>(sc, w);
  __syncthreads();
}

// out = P v.  Jacobi: per row, by the row's thread (no synchronisation).  Block Jacobi:
// L^-T L^-1 v per block (reads other rows of v: synchronises on entry and between the two
// triangular products); out is written by the rows' threads.
template <class Real> __device__ void pcr_precond(const KScene<Real>& sc, WS<Real>& w, const Real* v, Real* out) {
  const int tid = w.tid, nth = blockDim.x, m = w.ints[0], mc = w.ints[1];
  if (sc.pc == PC_JACOBI) {
    const Real* pd = w.pcr + 6 * sc.m_max;
    for (int i = tid; i < m; i += nth) out[i] = pd[i] * v[i];
    return;
  }
  const int gstr = tri_size(sc.pg), ss = sc.ss;
  Real* y = w.tmp;
  __syncthreads();
  for (int r = tid; r < m; r += nth) {
    Real acc = Real(0);
    if (r < mc) {
      const int g = row_grp(w.row[r]), r0 = w.g0[g], i = r - r0;
      const Real* Li = w.G + g * gstr + tri(i, 0);
      for (int l = 0; l <= i; ++l) acc += Li[l] * v[r0 + l];
    } else {
      const int a = r - mc;
      const Real* La = w.S + tri(a, 0);
      for (int b = 0; b <= a; ++b) acc += La[b] * v[mc + b];
    }
    y[r] = acc;
  }
  __syncthreads();
  for (int r = tid; r < m; r += nth) {
    Real acc = Real(0);
    if (r < mc) {
      const int g = row_grp(w.row[r]), r0 = w.g0[g], i = r - r0, n = w.gn[g];
      const Real* Lb = w.G + g * gstr;
      for (int l = i; l < n; ++l) acc += Lb[tri(l, i)] * y[r0 + l];
    } else {
      const int a = r - mc;
      for (int b = a; b < ss; ++b) acc += w.S[tri(b, a)] * y[mc + b];
    }
    out[r] = acc;
  }
}

// Preconditioned conjugate residual on A x = b from x = 0 (A SPD, P SPD):
//   r = b, z = P r, p = z;  per iteration
//   alpha = (z, A z) / (A p, P A p);  x += alpha p;  r -= alpha A p;  z -= alpha P A p
//   beta = (z', A z') / (z, A z);  p = z' + beta p;  A p = A z' + beta A p
// one operator product and one preconditioner application per iteration; x_k minimises
// |L^T (b - A x)| (P = L L^T) over K_k(P A, P b).  At most `iters` iterations; with rtol > 0
// it stops after the first iteration with |r| <= rtol |b| and sets *conv.  Breakdown (a
// denominator that is not positive: the exact solution reached) stops it too.  Every
// decision is taken on block-reduced values, so all threads leave together.  t6: 6 nb
// scratch.  Returns the iterations taken.
template <class Real, bool ACC>
__device__ int pcr_solve(const KScene<Real>& sc, WS<Real>& w, const Real* b, Real* x, int iters, Real rtol, Real* t6,
                         const StepH<Real>& h, int* conv) {
  const int tid = w.tid, nth = blockDim.x, m = w.ints[0], M = sc.m_max;
  Real *r = w.pcr, *z = r + M, *p = z + M, *Ap = p + M, *Az = Ap + M, *q = Az + M;
  Real bb = Real(0);
  for (int i = tid; i < m; i += nth) { x[i] = Real(0); r[i] = b[i]; bb += b[i] * b[i]; }
  pcr_precond(sc, w, r, z);
  __syncthreads();
  Real rho = schur_apply<Real, ACC>(sc, w, z, Az, t6, h);
  for (int i = tid; i < m; i += nth) { p[i] = z[i]; Ap[i] = Az[i]; }
  block_sum2(w, rho, bb);
  *conv = 0;
  if (!(bb > Real(0))) { *conv = 1; return 0; }
  const Real target = rtol * rtol * bb;
  int k = 0;
  for (; k < iters; ++k) {
    pcr_precond(sc, w, Ap, q);
    Real den = Real(0);
    for (int i = tid; i < m; i += nth) den += Ap[i] * q[i];
    den = block_sum(w, den);
    if (!(den > Real(0)) || !(rho > Real(0))) break;
    const Real alpha = rho / den;
    Real rr = Real(0);
    for (int i = tid; i < m; i += nth) {
      x[i] += alpha * p[i];
      r[i] -= alpha * Ap[i];
      z[i] -= alpha * q[i];
      rr += r[i] * r[i];
    }
    __syncthreads();
    Real rho1 = schur_apply<Real, ACC>(sc, w, z, Az, t6, h);
    block_sum2(w, rho1, rr);
    const Real beta = rho1 / rho;
    rho = rho1;
    for (int i = tid; i < m; i += nth) { p[i] = z[i] + beta * p[i]; Ap[i] = Az[i] + beta * Ap[i]; }
    if (rtol > Real(0) && rr <= target) { *conv = 1; ++k; break; }
  }
  __syncthreads();
  return k;
}

// The adjoint's PCR solve, restarted on the true residual: x = 0, r = b; then up to 8
// times: PCR on A dx = r (asking for |r'| <= max(rtol |b| / |r|, floor) |r|, floor 1e-4 in
// FP32: what one FP32 run's recurrence reliably attains), x += dx, and the true residual
// r = b - A x formed with the compensated product.  It stops when |r| <= rtol |b|, when a
// correction no longer changes x at working precision (max |dx| <= 2^-23 max |x| in FP32,
// 2^-52 in FP64), or after `iters` PCR iterations in all.  The Schur matrix's condition
// number (~1e5-1e6 with contact compliance) turns a residual of rtol into a solution error
// of up to cond x rtol, hence the FP32 default rtol of 1e-10, far below what one FP32 run
// reaches.  dx, rt: m-row scratch.  Returns the PCR iterations; *conv = 1 when either
// stopping test was met.
template <class Real>
__device__ int pcr_solve_refined(const KScene<Real>& sc, WS<Real>& w, const Real* b, Real* x, int iters, Real rtol,
                                 Real* t6, Real* dx, Real* rt, const StepH<Real>& h, int* conv) {
  const int tid = w.tid, nth = blockDim.x, m = w.ints[0];
  const Real floor = sizeof(Real) == 4 ? Real(1e-4) : Real(0);
  const Real ulp = sizeof(Real) == 4 ? Real(1.1920929e-7) : Real(2.220446049250313e-16);
  Real bb = Real(0);
  for (int i = tid; i < m; i += nth) { x[i] = Real(0); rt[i] = b[i]; bb += b[i] * b[i]; }
  bb = block_sum(w, bb);
  Real rr = bb;
  Real* Ax = w.pcr + 4 * sc.m_max;     // free between PCR runs
  int its = 0;
  *conv = 0;
  for (int restart = 0; restart < 8; ++restart) {
    if (!(rr > rtol * rtol * bb)) { *conv = 1; break; }
    if (its >= iters) break;
    int c2 = 0;
    Real inner = rtol * ssqrt(bb / rr);
    if (inner < floor) inner = floor;
    its += pcr_solve<Real, true>(sc, w, rt, dx, iters - its, inner, t6, h, &c2);
    Real dmax = Real(0), xmax = Real(0);
    for (int i = tid; i < m; i += nth) {
      x[i] += dx[i];
      dmax = fmax(dmax, fabs(dx[i]));
      xmax = fmax(xmax, fabs(x[i]));
    }
    __syncthreads();
    schur_apply<Real, true>(sc, w, x, Ax, t6, h);
    Real r2 = Real(0);
    for (int i = tid; i < m; i += nth) {
      acc2<Real> r;
      r.add(b[i]);
      r.add(-Ax[i]);
      rt[i] = r.value();
      r2 += rt[i] * rt[i];
    }
    rr = block_sum(w, r2);
    dmax = block_max(w, dmax);
    xmax = block_max(w, xmax);
    if (restart > 0 && dmax <= ulp * xmax) { *conv = 1; break; }
  }
  if (!(rr > rtol * rtol * bb)) *conv = 1;
  return its;
}

// ---------------------------------------------------------------------------
// forward step kernel
// ---------------------------------------------------------------------------
// The scene lives in a CTA's shared memory, in working precision: kernels index its per-body and
// per-row tables with thread-dependent indices, which the constant (parameter) cache would
// serialise across a warp.  Every CTA forms it as it starts (once per world, or once per
// persistent CTA), each value by one thread, the servo compliance by a division in FP64.
template <class Real> __device__ __forceinline__ void scene_to_shared(const DevScene& src, double h, KScene<Real>& dst) {
  const SceneLayout& sl = src;
  SceneLayout& dl = dst;
  const int* s = reinterpret_cast<const int*>(&sl);
  int* d = reinterpret_cast<int*>(&dl);
  const int tid = threadIdx.x, nth = blockDim.x;
  for (int i = tid; i < (int)(sizeof(SceneLayout) / sizeof(int)); i += nth) d[i] = s[i];
  for (int b = tid; b < src.nb; b += nth) {
    dst.mass[b] = Real(src.mass[b]);
    dst.minv[b] = Real(1) / dst.mass[b];
    dst.radius[b] = Real(src.radius[b]);
    dst.hw[b] = Real(src.hw[b]);
    for (int k = 0; k < 3; ++k) {
      dst.inertia[b][k] = Real(src.inertia[b][k]);
      dst.iinv[b][k] = Real(1) / dst.inertia[b][k];
      dst.half[b][k] = Real(src.half[b][k]);
    }
  }
  for (int j = nth - 1 - tid; j < src.nj; j += nth) {   // from the last thread, beside the bodies
    for (int k = 0; k < 3; ++k) {
      dst.ap[j][k] = Real(src.ap[j][k]); dst.ac[j][k] = Real(src.ac[j][k]);
      dst.axp[j][k] = Real(src.axp[j][k]); dst.axc[j][k] = Real(src.axc[j][k]);
      dst.p1[j][k] = Real(src.p1[j][k]); dst.p2[j][k] = Real(src.p2[j][k]);
    }
    // servo compliance alpha of Eq. (8): 1/kp (velocity target), 1/(kd + h kp) (position)
    dst.alpha[j] = Real(src.smode[j] == SERVO_POSITION ? 1.0 / (src.kd[j] + h * src.kp[j]) : 1.0 / src.kp[j]);
  }
  if (tid == 0) {
    dst.mu = Real(src.mu); dst.g = Real(src.g);
    for (int i = 0; i < 5; ++i) dst.box[i] = Real(src.box[i]);
    dst.hsp = Real(src.hsp); dst.hox = Real(src.hox); dst.hoy = Real(src.hoy);
    dst.tol = Real(src.tol); dst.delta_rel = Real(src.delta_rel); dst.kappa = Real(src.kappa);
    dst.eps = Real(src.eps); dst.margin = Real(src.margin); dst.pcr_rtol_adj = Real(src.pcr_rtol_adj);
    dst.hs.h = Real(h); dst.hs.hh = Real(0.5 * h);
    dst.heights = src.heights;
  }
  __syncthreads();
}

// The thread's number in its CTA's work.  The CTA's first warp does most of the work that one
// warp does alone (the separator's factor and solve, the bodies' sums).  A warp's scheduler
// follows from its slot on the SM, and CTAs of two warps would all put their first warps on
// the same two of the four: every second CTA takes its warps in the other order (8192
// robots: 3.06 -> 2.66 ms, step + adjoint, for the step's).  The numbering changes no result.
// Four warps have a scheduler each; turning them too made the terrain slower (1.20 -> 1.53 ms).
template <class Real> __device__ __forceinline__ void turn_warps(WS<Real>& w) {
  if (threadIdx.x == 0) {
    unsigned slot;
    asm volatile("mov.u32 %0, %%warpid;" : "=r"(slot));
    w.ints[14] = (int)(slot >> 2);
  }
  __syncthreads();
  w.tid = blockDim.x == 64 ? (int)((threadIdx.x + 32u * (unsigned)w.ints[14]) & 63u) : (int)threadIdx.x;
}

// One world's step; `item` is the launch's work index (the CTA index of a one-CTA-per-
// world launch, or the index a persistent CTA took from the queue).
template <class Real, bool FEW>
__device__ __forceinline__ void step_world(const KScene<Real>& sc, WS<Real>& w, const StepArgs& a, int item) {
  const int tid = w.tid, nth = blockDim.x;
  const int world = a.list ? a.list[item] : a.world0 + item;
  if (world < 0 || world >= a.n_worlds) return;
  const TapeLayout tl = tape_layout(sc);
  Real* tpw = nullptr;    // this world's tape record (nullptr: the step records nothing)
  if (a.tape) {
    const int slot = a.list ? (a.list_slot ? a.list_slot[item] : -1) : 0;
    if (slot >= 0 && (!a.list || slot < a.tape_slots))
      tpw = reinterpret_cast<Real*>(a.tape) + ((size_t)slot * a.n_worlds + world) * tl.total;
  }
  const int ld = a.ld, nb = sc.nb;
  const Real* sin = reinterpret_cast<const Real*>(a.state_in);
  const Real* ctl = reinterpret_cast<const Real*>(a.controls);
  const StepH<Real> h = sc.hs;
  // this world's inputs (structure of arrays, world index fastest)
  Src<Real> sq = {sin + world, (size_t)ld}, su = {sin + (size_t)7 * nb * ld + world, (size_t)ld};
  Src<Real> sb = {ctl ? ctl + world : sin, ctl ? (size_t)ld : (size_t)0};
  world_setup<Real>(sc, w, sq, su, sb, h, tpw ? tpw + tl.off_ct : nullptr);
  const int m = w.ints[0], mc = w.ints[1];
  // warm start: lambda from the previous step on the active rows, into the trial buffers;
  // the loop's evaluation takes it as its first trial
  for (int i = tid; i < 6 * nb; i += nth) w.ut[i] = w.uk[i];
  for (int i = tid; i < m; i += nth) w.lt[i] = sin[(size_t)(13 * nb + row_lam(w.row[i])) * ld + world];
  __syncthreads();
  clamp_cone(sc, w, w.lt);
  __syncthreads();
  double* trace = a.trace ? a.trace + (size_t)world * (sc.budget + 2) : nullptr;
  Real merit = Real(0);
  Real best = Real(INFINITY);
  int best_k = -1, k = 0, conv = 0;
  const Real tol2 = sc.tol * sc.tol;
  const int n_alpha = sc.ls ? 4 : 1;
  // phase 0: the warm start; 1: a Newton trial; 2: the returned iterate when it is not the
  // last one evaluated (the best iterate from k_min on, or the NaN iterate)
  int phase = 0;
  bool nan0 = false;
  uint32_t status = 0;
  Real mret = merit;
  Real alpha = Real(1);
  int ai = 0;
  for (;;) {
    // the loop's one evaluation: of the trial iterate, the warm start or the returned
    // iterate; step control: the full step (Sec. III-C) or backtracking on the merit
    const Real mt = evaluate<FEW>(sc, w, w.ut, w.lt, h);
    if (phase == 1 && !(mt < merit) && ai + 1 < n_alpha) {
      ++ai;
      alpha *= Real(0.5);
      for (int i = tid; i < 6 * nb; i += nth) w.ut[i] = w.uk[i] + alpha * w.du[i];
      for (int i = tid; i < m; i += nth) w.lt[i] = w.lk[i] + alpha * w.dl[i];
      __syncthreads();
      clamp_cone(sc, w, w.lt);
      __syncthreads();
      continue;
    }
    for (int i = tid; i < 6 * nb; i += nth) w.uk[i] = w.ut[i];
    for (int i = tid; i < m; i += nth) w.lk[i] = w.lt[i];
    if (phase == 2) {
      mret = mt;
    } else {
      merit = mt;
      if (trace && tid == 0) trace[phase == 0 ? 0 : k + 1] = (double)merit;
      // A NaN merit at the warm start (a non-finite input, or an input that has blown up)
      // makes every Newton step NaN: the iterate is set to NaN at once instead of after
      // the whole budget of NaN iterations, and the step returns it with status bits 1 and 2.
      if (phase == 0) nan0 = !(merit == merit);
      else ++k;
    }
    __syncthreads();
    bool fin = phase == 2 || nan0 || k >= sc.budget;
    if (phase != 2) {
      phase = 1;
      if (!fin) {
        if (k >= sc.kmin && merit < best) {
          best = merit; best_k = k;
          for (int i = tid; i < 6 * nb; i += nth) w.ub[i] = w.uk[i];
          for (int i = tid; i < m; i += nth) w.lb[i] = w.lk[i];
        }
        if (merit < tol2) { conv = 1; fin = true; }
      }
      if (fin) {
        // the returned iterate: the last one (evaluated: the workspace holds its rows), or
        // the best from k_min on, or the NaN iterate, which go through the evaluation first
        mret = merit;
        if (!conv) {
          status |= 1u;
          if (nan0 || (!(k >= sc.kmin && merit < best) && best_k >= 0)) {
            const Real qnan = Real(NAN);
            for (int i = tid; i < 6 * nb; i += nth) w.ut[i] = nan0 ? qnan : w.ub[i];
            for (int i = tid; i < m; i += nth) w.lt[i] = nan0 ? qnan : w.lb[i];
            __syncthreads();
            phase = 2;
            continue;
          }
        }
      }
    }
    // a recording direct-mode step factors the returned iterate for the tape at the loop's
    // own assembly and factorisation below; otherwise the loop ends here
    if (fin && !(tpw && sc.lin == LIN_DIRECT)) break;
    // Schur step, Eq. (12): (h J M^-1 J^T + C + delta) dl = J M^-1 r_dyn - rhat, by the
    // block-arrowhead factor or by PCR (the preconditioner formed at this iterate)
    const bool direct = sc.lin == LIN_DIRECT;
    if (direct || sc.pc == PC_BLOCK) {
      assemble(sc, w, h);
      if (direct) {
        factor_eliminate<FEW>(sc, w);
        if (fin) {
          factor_separator<FEW>(sc, w);
          break;
        }
      } else {
        factor_blocks(sc, w);
      }
    } else {
      pcr_jacobi(sc, w, h);
    }
    // right-hand side J M^-1 r_dyn - rhat.  Direct: by the second warp, with the groups'
    // forward pass, beside the first warp's factorisation of the separator (neither needs the
    // other), straight into dl, solved in place.
    const bool beside = direct && nth > 32 && sc.ss <= 32;
    Real* rhs = direct ? w.dl : w.rhs;
    const int t0 = beside ? tid - 32 : tid, T = beside ? 32 : nth;
    if constexpr (FEW && sizeof(Real) == 8) {
      if (beside && (tid < 32 || tid >= 96)) factor_separator<FEW>(sc, w);
    } else {
      if (beside && tid < 32) factor_separator<FEW>(sc, w);
    }
    if (t0 >= 0 && t0 < T) {
      for (int i = t0; i < m; i += T) {
        const Real* Ji = w.J + 12 * i;
        const int b0 = row_b0(w.row[i]), b1 = row_b1(w.row[i]);
        acc2<Real> jm;
        for (int q = 0; q < 6; ++q) jm.add_prod(Ji[q], w.mr[6 * b0 + q]);
        if (b1 >= 0) for (int q = 0; q < 6; ++q) jm.add_prod(Ji[6 + q], w.mr[6 * b1 + q]);
        jm.add(-w.rhat[i]);
        rhs[i] = jm.value();
      }
      if (beside) {
        __syncwarp();
        arrow_forward(sc, w, w.dl, t0, T, [] { __syncwarp(); });
      }
    }
    __syncthreads();
    if (direct) {
      if (!beside) {
        arrow_forward(sc, w, w.dl, tid, nth, [] { __syncthreads(); });
        factor_separator<FEW>(sc, w);
        __syncthreads();
      }
      if (tid < 32) arrow_separator(sc, w, w.dl);
      __syncthreads();
      arrow_backward(sc, w, w.dl);
    } else {
      int pconv;
      pcr_solve<Real, false>(sc, w, w.rhs, w.dl, sc.pcr_iters, Real(0), w.du, h, &pconv);
    }
    // Eq. (13): du = M^-1 (h J^T dl - r_dyn), and the full-step trial (mr is free once the
    // right-hand side is formed)
    for (int task = tid; task < 6 * nb; task += nth) {
      const int b = task / 6, k = task - 6 * (task / 6);
      Real jt = Real(0);
      body_rows(sc, w, b, [&](int off, int i) { jt += w.J[off + k] * w.dl[i]; });
      w.mr[task] = h.h * jt - w.rdyn[task];
    }
    __syncthreads();
    ai = 0;
    alpha = Real(1);
    for (int task = tid; task < 6 * nb; task += nth) {
      const int b = task / 6, k = task - 6 * (task / 6);
      const Real* t = w.mr + 6 * b;
      const Real* Iv = w.Iwi + 9 * b + 3 * (k - 3);
      const Real d = k < 3 ? t[k] * sc.minv[b] : Iv[0] * t[3] + Iv[1] * t[4] + Iv[2] * t[5];
      w.du[task] = d;
      w.ut[task] = w.uk[task] + alpha * d;
    }
    for (int i = nth - 1 - tid; i < sc.ss; i += nth) w.lt[mc + i] = w.lk[mc + i] + alpha * w.dl[mc + i];
    for (int sl = nth - 1 - tid; sl < sc.n_slots; sl += nth) {
      if (w.srow[sl] < 0) continue;
      const int i = w.srow[sl];
      for (int q = 0; q < 3; ++q) w.lt[i + q] = w.lk[i + q] + alpha * w.dl[i + q];
      clamp_slot(sc, w.lt + i);
    }
    __syncthreads();
  }
  if (!(mret == mret) || !(fabs((double)mret) < 1e300)) status |= 2u;
  status |= (uint32_t)w.ints[7];
  if (tpw) {
    // the returned iterate with (direct mode) its Schur factor, formed by the loop's last
    // pass; PCR records no matrix (the adjoint forms its operator and preconditioner at
    // the taped iterate)
    Real* tp = tpw;
    for (int i = tid; i < 7 * nb; i += nth) tp[tl.off_qm + i] = w.qm[i];
    for (int i = tid; i < 6 * nb; i += nth) { tp[tl.off_um + i] = w.um[i]; tp[tl.off_u + i] = w.uk[i]; }
    for (int i = tid; i < sc.n_servo; i += nth) tp[tl.off_ubar + i] = w.ubar[i];
    for (int i = tid; i < sc.m_max; i += nth) tp[tl.off_lam + i] = Real(0);
    __syncthreads();
    for (int i = tid; i < m; i += nth) tp[tl.off_lam + row_lam(w.row[i])] = w.lk[i];
    if (sc.lin == LIN_DIRECT) {
      for (int i = tid; i < sc.n_groups * tri_size(sc.pg); i += nth) tp[tl.off_G + i] = w.G[i];
      for (int i = tid; i < sc.n_groups * sc.cmax * sc.ldg; i += nth) tp[tl.off_H + i] = w.H[i];
      for (int i = tid; i < tri_size(sc.ss); i += nth) tp[tl.off_S + i] = w.S[i];
    }
  }
  // outputs: q+ (normalised quaternions), u+, lambda+, impulses h lambda, contact ids
  Real* so = reinterpret_cast<Real*>(a.state_out);
  Real* imp = reinterpret_cast<Real*>(a.impulses);
  for (int b = tid; b < nb; b += nth) {
    Real qp[7];
    kin_body<Real, Real>(w.qm + 7 * b, w.uk + 6 * b, h, qp);
    Real nq = ssqrt(qp[3] * qp[3] + qp[4] * qp[4] + qp[5] * qp[5] + qp[6] * qp[6]);
    for (int c = 3; c < 7; ++c) qp[c] /= nq;
    for (int c = 0; c < 7; ++c) so[(size_t)(7 * b + c) * ld + world] = qp[c];
    for (int c = 0; c < 6; ++c) so[(size_t)(7 * nb + 6 * b + c) * ld + world] = w.uk[6 * b + c];
  }
  for (int i = tid; i < sc.m_max; i += nth) {
    so[(size_t)(13 * nb + i) * ld + world] = Real(0);
    if (imp) imp[(size_t)i * ld + world] = Real(0);
  }
  __syncthreads();
  for (int i = tid; i < m; i += nth) {
    int li = row_lam(w.row[i]);
    so[(size_t)(13 * nb + li) * ld + world] = w.lk[i];
    if (imp) imp[(size_t)li * ld + world] = h.h * w.lk[i];
  }
  if (a.ids)
    for (int sl = tid; sl < sc.n_slots; sl += nth) a.ids[(size_t)sl * ld + world] = w.srow[sl] >= 0 ? w.sid[sl] : -1;
  if (tid == 0) {
    if (a.status) a.status[world] = status;
    if (a.cost) a.cost[world] = k;
    if (a.iters) a.iters[world] = k | (m << 16);
  }
}

// At most 128 threads per world, registers capped at 128 in FP32: eight robot worlds of 64
// threads per SM then, which their 24.9 KB of workspace allows too.
// FEW: see few_worlds; a kernel of its own, because as a branch of this one its code cost the
// large launches 1 %.
template <class Real, bool FEW>
__global__ void __launch_bounds__(128, sizeof(Real) == 4 ? 4 : 3) step_kernel(const DevScene scp, const StepArgs a) {
  extern __shared__ __align__(16) char smem[];
  __shared__ __align__(16) KScene<Real> ssc;
  scene_to_shared(scp, a.h, ssc);
  WS<Real> w = ws_carve<Real>(smem, ssc);
  turn_warps(w);
  w.sum_nth = a.sum_threads;
  // one CTA per world, or persistent: take work items until the queue is exhausted (no CTA
  // waits on another).  One call site for both: a second inlined copy would double the code.
  for (;;) {
    int it = blockIdx.x;
    if (a.queue) {
      __syncthreads();
      if (threadIdx.x == 0) w.ints[15] = atomicAdd(a.queue, 1);
      __syncthreads();
      it = w.ints[15];
      if (it >= a.n_items) break;
      if (a.order) it = a.order[it];
    }
    step_world<Real, FEW>(ssc, w, a, it);
    if (!a.queue) break;
  }
}

// Heaviest-first order of the worlds by their previous step's Newton iterations (a
// counting sort over 0..63, one CTA): worlds that took the most iterations start first,
// so the last wave is short.  Worlds of equal count may come in any order; a world's
// result does not depend on when it runs.
static __global__ void lpt_order_kernel(const int32_t* cost, int n, int32_t* order) {
  __shared__ int bins[64], start[64];
  for (int i = threadIdx.x; i < 64; i += blockDim.x) bins[i] = 0;
  __syncthreads();
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    int c = cost[i];
    c = c < 0 ? 0 : (c > 63 ? 63 : c);
    atomicAdd(&bins[c], 1);
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    int acc = 0;
    for (int c = 63; c >= 0; --c) { start[c] = acc; acc += bins[c]; }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    int c = cost[i];
    c = c < 0 ? 0 : (c > 63 ? 63 : c);
    order[atomicAdd(&start[c], 1)] = i;
  }
}

// ---------------------------------------------------------------------------
// adjoint kernel
// ---------------------------------------------------------------------------
// Body part of Psi: g_q . q+(q-) + w_u . (M(q-)(u* - u-) - h f(q-, u-)), along (b, dc).
template <class Real>
__device__ Real body_vjp(const KScene<Real>& sc, const WS<Real>& w, int b, int dc, const Real* gq, const Real* wu, const StepH<Real>& h) {
  typedef dual<Real> D;
  D qm[7], qp[7];
  for (int c = 0; c < 7; ++c) qm[c] = D(w.qm[7 * b + c], c == dc ? Real(1) : Real(0));
  kin_body<D, Real>(qm, w.uk + 6 * b, h, qp);
  D acc(Real(0));
  for (int c = 0; c < 7; ++c) acc = acc + D(gq[7 * b + c]) * qp[c];
  // angular part depends on q- through I_w(q-) = R diag(I) R^T
  vec3<D> dw = v3(D(w.uk[6 * b + 3] - w.um[6 * b + 3]), D(w.uk[6 * b + 4] - w.um[6 * b + 4]), D(w.uk[6 * b + 5] - w.um[6 * b + 5]));
  vec3<D> om = v3(D(w.um[6 * b + 3]), D(w.um[6 * b + 4]), D(w.um[6 * b + 5]));
  auto Iw_apply = [&](vec3<D> v) {
    vec3<D> vb = v3(D(Real(0)), D(Real(0)), D(Real(0)));
    // R^T v via rotating by the conjugate quaternion
    D qc[4] = {qm[3], D(Real(0)) - qm[4], D(Real(0)) - qm[5], D(Real(0)) - qm[6]};
    vb = qrot(qc, v);
    vb = v3(vb.x * D(sc.inertia[b][0]), vb.y * D(sc.inertia[b][1]), vb.z * D(sc.inertia[b][2]));
    return qrot(qm + 3, vb);
  };
  vec3<D> Idw = Iw_apply(dw);
  vec3<D> gy = cross3(om, Iw_apply(om));        // f_ang = -gy
  vec3<D> ra = Idw + scale(gy, D(h.h));     // angular r_dyn minus the lambda terms
  acc = acc + D(wu[6 * b + 3]) * ra.x + D(wu[6 * b + 4]) * ra.y + D(wu[6 * b + 5]) * ra.z;
  return acc.d;
}

}  // namespace ost
#include "ostrich_adjoint.cuh"
namespace ost {

// One world's adjoint (Sec. III-D) in mode MODE (ADJ_PAPER or ADJ_EXACT).
// FP32, paper mode: registers capped at 128, so that eight robot worlds of 64 threads run per SM as
// in the step (8192 robots, step + adjoint: 2.57 -> 2.45 ms although the capped code spills
// some).  The exact mode's shared memory allows three anyway.
template <class Real, int MODE>
__global__ void __launch_bounds__(128, sizeof(Real) == 4 && MODE == ADJ_PAPER ? 4 : 3) adjoint_kernel(const DevScene scp, const AdjArgs a) {
  extern __shared__ __align__(16) char smem[];
  __shared__ __align__(16) KScene<Real> ssc;
  __shared__ __align__(16) AdjLists al;
  unsigned char* bgl = al.bgl;
  int *bgn = al.bgn, *item0 = al.item0, *ncon = al.ncon, *jpre = al.jpre, *cpre = al.cpre;
  scene_to_shared(scp, a.h, ssc);
  const KScene<Real>& sc = ssc;
  WS<Real> w = ws_carve<Real>(smem, sc);
  turn_warps(w);
  w.sum_nth = a.sum_threads;
  ExWS<Real> ex = {};
  if (MODE == ADJ_EXACT) ex = ex_carve<Real>(smem + ws_layout_bytes<Real>(sc), sc);
  const int tid = w.tid, nth = blockDim.x;
  const int world = a.list ? a.list[blockIdx.x] : a.world0 + blockIdx.x;
  if (world < 0 || world >= a.n_worlds) return;
  const int slot = a.list ? (a.list_slot ? a.list_slot[blockIdx.x] : -1) : 0;
  if (slot < 0 || (a.list && slot >= a.tape_slots)) return;
  const int ld = a.ld, nb = sc.nb;
  const StepH<Real> h = sc.hs;
  const Real hR = h.h;
  const TapeLayout tl = tape_layout(sc);
  const Real* tp = reinterpret_cast<const Real*>(a.tape) + ((size_t)slot * a.n_worlds + world) * tl.total;
  if (sc.lin == LIN_DIRECT) {
    // the taped factor, copied to shared memory in the background of the setup and the
    // evaluation (neither touches G, H or S); awaited before the solve
    for (int i = tid; i < sc.n_groups * tri_size(sc.pg); i += nth) cp_async_elem(w.G + i, tp + tl.off_G + i);
    for (int i = tid; i < sc.n_groups * sc.cmax * sc.ldg; i += nth) cp_async_elem(w.H + i, tp + tl.off_H + i);
    for (int i = tid; i < tri_size(sc.ss); i += nth) cp_async_elem(w.S + i, tp + tl.off_S + i);
    cp_async_commit();
  }
  Src<Real> sq = {tp + tl.off_qm, 1}, su = {tp + tl.off_um, 1}, sb = {tp + tl.off_ubar, 1};
  world_setup<Real>(sc, w, sq, su, sb, h, (Real*)nullptr, tp + tl.off_ct);   // the step's contact set
  const int m = w.ints[0], mc = w.ints[1];
  for (int i = tid; i < 6 * nb; i += nth) w.uk[i] = tp[tl.off_u + i];
  for (int i = tid; i < m; i += nth) w.lk[i] = tp[tl.off_lam + row_lam(w.row[i])];
  __syncthreads();
  evaluate<false>(sc, w, w.uk, w.lk, h, false);   // J (with E at u*), C, delta, poses at q+
  if (tid < 32) {
    // a lane per body: its groups, and by prefix sums over the bodies the places of its
    // pull-back items and the joint and contact groups before it
    const int lane = tid;
    const bool tr = MODE == ADJ_PAPER && sc.pullback == 1;
    int nc = 0, ng = 0;
    bool dual_pos = false;
    if (lane < nb) {
      ng = body_groups(sc, w, lane, bgl, nc);
      for (int k = 0; k < ng; ++k) dual_pos = dual_pos || position_needs_dual(sc, w, bgl[lane * GROUPS_PER_BODY + k], tr);
      bgn[lane] = ng;
      ncon[lane] = nc;
    }
    dual_pos = __any_sync(0xffffffffu, dual_pos);
    int pi = lane < nb ? 7 * (ng + 1) : 0, pj = ng - nc, pc = nc;
    for (int o = 1; o < NB_CAP; o <<= 1) {             // inclusive sums
      const int ui = __shfl_up_sync(0xffffffffu, pi, o), uj = __shfl_up_sync(0xffffffffu, pj, o);
      const int uc = __shfl_up_sync(0xffffffffu, pc, o);
      if (lane >= o) { pi += ui; pj += uj; pc += uc; }
    }
    if (lane == 0) { item0[0] = 0; jpre[0] = 0; cpre[0] = 0; al.n_first = dual_pos ? 7 : 4; }
    if (lane < nb) { item0[lane + 1] = pi; jpre[lane + 1] = pj; cpre[lane + 1] = pc; }
  }
  if (sc.lin == LIN_DIRECT) {
    cp_async_wait_all();     // this thread's copies of the taped factor; the barrier below
                             // (before the solve) makes every thread's visible
  } else if (MODE == ADJ_EXACT) {
    // PCR mode tapes no factor: the exact mode's GMRES preconditioner is the direct factor,
    // formed here at the taped iterate
    assemble(sc, w, h);
    factor_eliminate<false>(sc, w);
    factor_separator<false>(sc, w);
    __syncthreads();
  } else if (sc.pc == PC_BLOCK) {
    // the PCR operator and preconditioner of the forward pass, at the taped iterate
    assemble(sc, w, h);
    factor_blocks(sc, w);
  } else {
    pcr_jacobi(sc, w, h);
  }
  // incoming cotangent: normalisation Jacobian of the output quaternions, then g
  Real* gq = w.lb;      // the best-iterate buffer is free in the adjoint; m_max >= 7 nb
  Real* gu = w.du;
  const Real* din = reinterpret_cast<const Real*>(a.dL_dnext);
  for (int b = tid; b < nb; b += nth) {
    Real qp[7];
    kin_body<Real, Real>(w.qm + 7 * b, w.uk + 6 * b, h, qp);
    Real nq = ssqrt(qp[3] * qp[3] + qp[4] * qp[4] + qp[5] * qp[5] + qp[6] * qp[6]);
    Real qh[4] = {qp[3] / nq, qp[4] / nq, qp[5] / nq, qp[6] / nq};
    Real gin[4];
    for (int c = 0; c < 4; ++c) gin[c] = din[(size_t)(7 * b + 3 + c) * ld + world];
    Real dp = qh[0] * gin[0] + qh[1] * gin[1] + qh[2] * gin[2] + qh[3] * gin[3];
    for (int c = 0; c < 3; ++c) gq[7 * b + c] = din[(size_t)(7 * b + c) * ld + world];
    for (int c = 0; c < 4; ++c) gq[7 * b + 3 + c] = (gin[c] - qh[c] * dp) / nq;
    for (int c = 0; c < 6; ++c) gu[6 * b + c] = din[(size_t)(7 * nb + 6 * b + c) * ld + world];
    // g = grad_u L + h G(q-)^T grad_q L; G^T for the quaternion block is 1/2 vec(g (x) q-*)
    const Real* q = w.qm + 7 * b + 3;
    const Real* g4 = gq + 7 * b + 3;
    Real vx = -g4[0] * q[1] + g4[1] * q[0] - g4[2] * q[3] + g4[3] * q[2];
    Real vy = -g4[0] * q[2] + g4[1] * q[3] + g4[2] * q[0] - g4[3] * q[1];
    Real vz = -g4[0] * q[3] - g4[1] * q[2] + g4[2] * q[1] + g4[3] * q[0];
    gu[6 * b] += hR * gq[7 * b]; gu[6 * b + 1] += hR * gq[7 * b + 1]; gu[6 * b + 2] += hR * gq[7 * b + 2];
    gu[6 * b + 3] += hR * Real(0.5) * vx; gu[6 * b + 4] += hR * Real(0.5) * vy; gu[6 * b + 5] += hR * Real(0.5) * vz;
    Real mg[6];
    minv6(sc, w, b, gu + 6 * b, mg);
    for (int c = 0; c < 6; ++c) w.mr[6 * b + c] = mg[c];
  }
  __syncthreads();
  Real* wl = w.dl;
  Real* wu = w.ub;
  if (MODE == ADJ_PAPER) {
    // Eq. (18): A w_lambda = -h J M^-1 g, with the forward factor (the refinement's
    // matrix-free product takes delta as the evaluation at the iterate formed it, scal[2]);
    // the right-hand side is formed with exact products: its rounding would otherwise
    // reach the null space of J^T, where A's eigenvalue is only kappa
    for (int i = tid; i < m; i += nth) {
      const Real* Ji = w.J + 12 * i;
      int b0 = row_b0(w.row[i]), b1 = row_b1(w.row[i]);
      acc2<Real> jm;
      for (int k = 0; k < 6; ++k) jm.add_prod(Ji[k], w.mr[6 * b0 + k]);
      if (b1 >= 0) for (int k = 0; k < 6; ++k) jm.add_prod(Ji[6 + k], w.mr[6 * b1 + k]);
      w.rhs[i] = -hR * jm.value();
    }
    __syncthreads();
    if (sc.lin == LIN_DIRECT) {
      // refined until a correction no longer changes w_lambda at working precision (at
      // most refine_adj sweeps)
      schur_solve(sc, w, w.rhs, wl, w.f, w.lt, h, sc.refine_adj, Real(sizeof(Real) == 4 ? 1.2e-7 : 0.0));
    } else {
      // a single PCR solve with the forward pass's operator and preconditioner (Sec. III-D)
      int pconv = 0;
      const int its = pcr_solve_refined<Real>(sc, w, w.rhs, wl, sc.pcr_iters_adj, sc.pcr_rtol_adj, w.f, w.lt,
                                              w.tmp2, h, &pconv);
      if (tid == 0 && a.krylov) a.krylov[world] = its | (pconv ? 0 : (1 << 16));
    }
    // Eq. (19): w_u = -M^-1 (g + J^T w_lambda)
    jt_apply<true>(sc, w, wl, w.f);     // f is free now
    __syncthreads();
    for (int b = tid; b < nb; b += nth) {
      Real t[6], o[6];
      for (int c = 0; c < 6; ++c) t[c] = gu[6 * b + c] + w.f[6 * b + c];
      minv6(sc, w, b, t, o);
      for (int c = 0; c < 6; ++c) wu[6 * b + c] = -o[c];
    }
    __syncthreads();
  } else {
    // exact IFT: local Jacobians of every group at the returned iterate, then GMRES on
    // J_F^T [w_u; w_lambda] = [-g; 0] preconditioned by the paper's matrix
    exact_slot_terms(sc, w, ex, h);
    __syncthreads();
    for (int task = tid; task < 6 * nb; task += nth) exact_task(sc, w, ex, bgl, bgn, task / 6, task % 6, h);
    for (int i = tid; i < 6 * nb; i += nth) ex.r[i] = -gu[i];
    for (int i = tid; i < m; i += nth) ex.r[6 * nb + i] = Real(0);
    __syncthreads();
    Real msum = Real(0);
    for (int b = 0; b < nb; ++b) msum += sc.mass[b];
    const Real sigma = msum / (Real(nb) * hR);
    int conv = 0;
    const int its = exact_gmres(sc, w, ex, h, sigma, Real(sizeof(Real) == 4 ? 1e-6 : 1e-13), &conv);
    for (int i = tid; i < 6 * nb; i += nth) wu[i] = ex.x[i];
    for (int i = tid; i < m; i += nth) wl[i] = ex.x[6 * nb + i];
    if (tid == 0 && a.krylov) a.krylov[world] = its | (conv ? 0 : (1 << 16));
    __syncthreads();
  }
  // Eq. (17) with xi = theta, the physical parameters: explicit partials of the rows
  // that hold them, contracted with the adjoint.  Servo gain k_p: the servo row of
  // Eq. (8) holds lambda_c / k_p, so d/dk_p = -lambda_c / k_p^2.  Body mass m_b: the
  // linear rows of Eq. (10), m_b (v - v-) - h m_b g, so d/dm_b = (v - v-) - h g e_z.
  // Principal moment I_k: the angular rows, I_w (w - w-) + h w- x (I_w w-) with
  // I_w = R diag(I) R^T at q-, so d/dI_k = r_k (r_k . (w - w-)) + h (r_k . w-) (w- x r_k),
  // r_k the k-th column of R(q-).  Friction coefficient mu (exact mode; the paper's
  // frozen W holds it): the friction rows of Eq. (7) through W.
  if (a.dL_dkp) {
    Real* dkp = reinterpret_cast<Real*>(a.dL_dkp);
    for (int i = mc + 5 * sc.nj + tid; i < m; i += nth) {
      // d alpha / d k_p: -1/k_p^2 (velocity target), -h/(k_d + h k_p)^2 (position target)
      const int j = row_ref(w.row[i]);
      const Real al = sc.alpha[j];
      const Real dal = sc.smode[j] == SERVO_POSITION ? -hR * al * al : -al * al;
      dkp[(size_t)(i - mc - 5 * sc.nj) * ld + world] = wl[i] * w.lk[i] * dal;
    }
  }
  if (a.dL_dmass) {
    Real* dm = reinterpret_cast<Real*>(a.dL_dmass);
    for (int b = tid; b < nb; b += nth) {
      Real acc = 0;
      for (int k = 0; k < 3; ++k) acc += wu[6 * b + k] * (w.uk[6 * b + k] - w.um[6 * b + k]);
      acc += wu[6 * b + 2] * (-hR * sc.g);
      dm[(size_t)b * ld + world] = acc;
    }
  }
  if (a.dL_dinertia) {
    Real* di = reinterpret_cast<Real*>(a.dL_dinertia);
    for (int b = tid; b < nb; b += nth) {
      Real R[9];
      qmat(w.qm + 7 * b + 3, R);                 // R(q-); w.R holds R(q+) after the evaluation
      const vec3<Real> wm = v3(w.um[6 * b + 3], w.um[6 * b + 4], w.um[6 * b + 5]);
      const vec3<Real> dw = v3(w.uk[6 * b + 3] - wm.x, w.uk[6 * b + 4] - wm.y, w.uk[6 * b + 5] - wm.z);
      const vec3<Real> ww = v3(wu[6 * b + 3], wu[6 * b + 4], wu[6 * b + 5]);
      for (int k = 0; k < 3; ++k) {
        const vec3<Real> rk = v3(R[k], R[3 + k], R[6 + k]);
        const vec3<Real> c = cross3(wm, rk);
        const Real s1 = dot3(rk, dw), s2 = hR * dot3(rk, wm);
        di[(size_t)(3 * b + k) * ld + world] =
            ww.x * (rk.x * s1 + c.x * s2) + ww.y * (rk.y * s1 + c.y * s2) + ww.z * (rk.z * s1 + c.z * s2);
      }
    }
  }
  if (a.dL_dmu) {
    Real part = Real(0);
    if (MODE == ADJ_EXACT) {
      typedef dual<Real> D;
      for (int sl = tid; sl < sc.n_slots; sl += nth) {
        if (w.srow[sl] < 0) continue;
        const int i = w.srow[sl], b = sc.slot_body[sl];
        CGroup<Real> g;
        contact_group<Real, Real>(sc, w, sl, b, w.qm + 7 * b, w.uk + 6 * b, h, g);
        D rf[2];
        friction_rows<D, Real>(sc, D(g.vel[1]), D(g.vel[2]), D(w.lk[i]), w.lk[i + 1], w.lk[i + 2],
                               hR * w.swhat[sl], D(sc.mu, Real(1)), rf);
        part += wl[i + 1] * rf[0].d + wl[i + 2] * rf[1].d;
      }
    }
    const Real tot = block_sum(w, part);
    if (tid == 0) reinterpret_cast<Real*>(a.dL_dmu)[world] = tot;
  }
  // dL/du- = -M w_u - h (df/du-)^T w_u ;  dL/dubar = -w_lambda of the servo rows
  Real* dout = reinterpret_cast<Real*>(a.dL_dstate);
  for (int b = tid; b < nb; b += nth) {
    Real mb = sc.mass[b];
    for (int c = 0; c < 3; ++c) dout[(size_t)(7 * nb + 6 * b + c) * ld + world] = -mb * wu[6 * b + c];
    vec3<Real> wa = v3(wu[6 * b + 3], wu[6 * b + 4], wu[6 * b + 5]);
    vec3<Real> om = v3(w.um[6 * b + 3], w.um[6 * b + 4], w.um[6 * b + 5]);
    vec3<Real> Iwa = mat3<Real>(w.Iw + 9 * b, wa);
    vec3<Real> t1 = mat3<Real>(w.Iw + 9 * b, cross3(om, wa));
    vec3<Real> t2 = cross3(mat3<Real>(w.Iw + 9 * b, om), wa);
    vec3<Real> d = v3(-Iwa.x - hR * (t1.x - t2.x), -Iwa.y - hR * (t1.y - t2.y), -Iwa.z - hR * (t1.z - t2.z));
    dout[(size_t)(7 * nb + 6 * b + 3) * ld + world] = d.x;
    dout[(size_t)(7 * nb + 6 * b + 4) * ld + world] = d.y;
    dout[(size_t)(7 * nb + 6 * b + 5) * ld + world] = d.z;
  }
  for (int i = tid; i < sc.m_max; i += nth) dout[(size_t)(13 * nb + i) * ld + world] = Real(0);
  Real* dctl = reinterpret_cast<Real*>(a.dL_dcontrols);
  if (dctl)   // d b_c / d target: -1 (velocity target), -1/h (position target)
    for (int i = mc + 5 * sc.nj + tid; i < m; i += nth)
      dctl[(size_t)(i - mc - 5 * sc.nj) * ld + world] = sc.smode[row_ref(w.row[i])] == SERVO_POSITION ? -wl[i] / hR : -wl[i];
  // dL/dq-: one work item per (body b, coordinate c of its q-, group touching b or the
  // body's own terms), each a dual-number evaluation along that coordinate; the items of a
  // coordinate are summed in a fixed order
  const bool trunc = MODE == ADJ_PAPER && sc.pullback == 1;
  Real* item = w.G;     // the factor (G, H, S, one carved run; E lies over dl = wl and is not part
                        // of it) is no longer needed; sum_b 7 (groups_b + 1) <= 14 m_max items
  // taken in cost order (every joint item, then every contact item, then the body terms)
  // so that the threads' loads even out; each item is stored at its place in the per-body
  // layout, which fixes the order of the sums below.  First the four quaternion coordinates,
  // and the three positions after them where a group has no closed form for those.  A
  // non-finite item means a non-finite value among what the duals multiply: a zero derivative
  // times it is NaN along the positions too, which their closed form would lose, so that
  // world takes a second pass, over all positions.
  int c0 = 0, nco = al.n_first;
  bool all_dual = false;
  for (;;) {
    const int nbc = c0 ? 3 : 4, nj_items = nco * jpre[nb], nc_items = nco * cpre[nb];
    const int n_items = nj_items + nc_items + nbc * nb;
    bool lost = false;
    for (int e = tid; e < n_items; e += nth) {
      int b = 0, c, k;
      if (e < nj_items) {
        while (e >= nco * jpre[b + 1]) ++b;
        const int nj = bgn[b] - ncon[b], r = e - nco * jpre[b];
        c = r / nj;
        k = 1 + ncon[b] + (r - c * nj);
      } else if (e < nj_items + nc_items) {
        const int e2 = e - nj_items;
        while (e2 >= nco * cpre[b + 1]) ++b;
        const int nc = ncon[b], r = e2 - nco * cpre[b];
        c = r / nc;
        k = 1 + (r - c * nc);
      } else {
        const int e3 = e - nj_items - nc_items;
        b = e3 / nbc;
        c = e3 - nbc * b;
        k = 0;
      }
      c += c0;
      c = c < 4 ? 3 + c : c - 4;
      const int grp = k ? bgl[b * GROUPS_PER_BODY + k - 1] : 0;
      if (c < 3 && !all_dual && !position_needs_dual(sc, w, grp, trunc)) continue;
      const Real v =
          k == 0 ? body_vjp(sc, w, b, c, gq, wu, h) : group_vjp_q<Real, MODE>(sc, w, ex, grp, b, c, wl, wu, trunc, h);
      item[item0[b] + c * (bgn[b] + 1) + k] = v;
      lost = lost || !isfinite(v);
    }
    if (!__syncthreads_or(lost) || all_dual) break;
    all_dual = true;
    c0 = 4; nco = 3;
  }
  const Real inv_h = Real(1) / hR;
  for (int e = tid; e < nb * 7; e += nth) {
    const int b = e / 7, c = e % 7;
    acc2<Real> acc;        // the terms cancel strongly: compensated sum
    const int base = item0[b] + c * (bgn[b] + 1);
    for (int k = 0; k <= bgn[b]; ++k) {
      const int grp = k ? bgl[b * GROUPS_PER_BODY + k - 1] : 0;
      if (c >= 3 || all_dual || (k && position_needs_dual(sc, w, grp, trunc))) acc.add(item[base + k]);
      else acc.add(k ? group_pull_position<Real, MODE>(sc, w, ex, grp, b, c, wl, inv_h) : gq[7 * b + c]);
    }
    dout[(size_t)(7 * b + c) * ld + world] = acc.value();
  }
}

// ---------------------------------------------------------------------------
// launchers (called by the C ABI)
// ---------------------------------------------------------------------------
// The dynamic shared-memory limit of a kernel is raised once per device and size; a
// launch inside a stream capture then issues nothing but the launch itself.
template <class K> cudaError_t ensure_smem(K kernel, size_t smem, int* done_dev, size_t* done_size) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 64 && done_size[dev] >= smem && done_dev[dev]) return cudaSuccess;
  e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  // all of the unified L1 as shared memory: the working sets live there, global traffic is small
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, (int)cudaSharedmemCarveoutMaxShared);
  if (e == cudaSuccess && dev < 64) { done_dev[dev] = 1; if (smem > done_size[dev]) done_size[dev] = smem; }
  return e;
}

// Whether a launch of n worlds is few for the chip: at most four per SM in FP32, two in FP64.
// Most of its schedulers would idle, and what counts is one world's latency.  The line, by
// the robot's step without and with all that follows from it (us): FP32, 1 world 149 / 136, two
// per SM 253 / 235, four 273 / 260, five 306 / 387; FP64, one per SM 1413 / 1092, two 1552 / 1215,
// three 1506 / 1450, but four 1901 / 2249 and their adjoint 207 / 275 (its arithmetic units
// are full).  Boxes: FP32 four per SM 139 / 128, FP64 two 682 / 556.  The line takes no account of
// how many worlds a scene's workspace lets run at once: where they run in turns there is
// the more to gain (eight chained boxes, FP32, 58 KB, three per SM at once: four per SM 2194 /
// 1895; FP64, 114 KB, one at once: two per SM 13170 / 9425).  A context of 128 threads with
// 64 slots gains nothing in FP32 (terrain, four per SM 267 / 275).
template <class Real> bool few_worlds(int n) {
  static std::atomic<int> sms[64];
  int dev = 0, k = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) { cudaGetLastError(); return false; }
  if (!(k = sms[dev].load(std::memory_order_relaxed))) {
    if (cudaDeviceGetAttribute(&k, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) { cudaGetLastError(); return false; }
    sms[dev].store(k, std::memory_order_relaxed);
  }
  return n <= (sizeof(Real) == 4 ? 4 : 2) * k;
}

// Threads of a world's CTA in a launch of few worlds for a context set to `threads`: four warps
// share its rows and tiles.  Scenes of at most a warp's rows gain nothing from more than two.
// The sums over all rows keep the order of `threads` (sum_threads), so results do not depend on
// this.  The conjugate-residual solver and the exact adjoint sum over the whole CTA in more
// places: they keep their threads.
inline int few_threads(const DevScene& sc, int threads) {
  if (sc.lin != LIN_DIRECT) return threads;
  const int t = sc.m_max <= 32 ? 64 : 128;
  return threads > t ? threads : t;
}

// Threads per world of a step of n worlds for a context set to `threads`.
template <class Real> int step_threads(const DevScene& sc, int threads, int n) {
  return few_worlds<Real>(n) ? few_threads(sc, threads) : threads;
}

template <class Real>
cudaError_t launch_step(const DevScene& sc, const StepArgs& a, int threads, cudaStream_t st) {
  static int done_dev[2][64] = {{0}};
  static size_t done_size[2][64] = {{0}};
  int n = a.list ? a.n_list : a.n_worlds - a.world0;
  const bool few = few_worlds<Real>(n);
  auto kernel = few ? step_kernel<Real, true> : step_kernel<Real, false>;
  size_t smem = ws_bytes<Real>(sc);
  // both kernels at once: a launch of another number of worlds may be under capture
  cudaError_t e = ensure_smem(step_kernel<Real, false>, smem, done_dev[0], done_size[0]);
  if (e == cudaSuccess) e = ensure_smem(step_kernel<Real, true>, smem, done_dev[1], done_size[1]);
  if (e != cudaSuccess) return e;
  if (n <= 0) return cudaSuccess;
  StepArgs b = a;
  b.sum_threads = threads;
  if (few) threads = few_threads(sc, threads);
  if (a.queue) {
    // persistent: as many CTAs as fit on the device at once, fed from the queue
    int dev = 0, n_sms = 0, per_sm = 0;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&n_sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, smem)) != cudaSuccess)
      return e;
    if (per_sm < 1) per_sm = 1;
    int grid = n_sms * per_sm < n ? n_sms * per_sm : n;
    if ((e = cudaMemsetAsync(a.queue, 0, sizeof(int), st)) != cudaSuccess) return e;
    if (a.order && a.cost) {
      lpt_order_kernel<<<1, 1024, 0, st>>>(a.cost + a.world0, n, const_cast<int32_t*>(a.order));
      if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    b.n_items = n;
    kernel<<<grid, threads, smem, st>>>(sc, b);
    return cudaGetLastError();
  }
  kernel<<<n, threads, smem, st>>>(sc, b);
  return cudaGetLastError();
}

template <class Real>
cudaError_t launch_adjoint(const DevScene& sc, const AdjArgs& a, int threads, cudaStream_t st) {
  static int done_dev[2][64] = {{0}};
  static size_t done_size[2][64] = {{0}};
  const int mode = a.mode == ADJ_EXACT ? ADJ_EXACT : ADJ_PAPER;
  auto kernel = mode == ADJ_EXACT ? adjoint_kernel<Real, ADJ_EXACT> : adjoint_kernel<Real, ADJ_PAPER>;
  const size_t smem = adj_smem_bytes<Real>(sc, mode);
  cudaError_t e = ensure_smem(kernel, smem, done_dev[mode], done_size[mode]);
  if (e != cudaSuccess) return e;
  int n = a.list ? a.n_list : a.n_worlds - a.world0;
  if (n <= 0) return cudaSuccess;
  AdjArgs b = a;
  b.sum_threads = threads;
  if (mode == ADJ_PAPER && few_worlds<Real>(n)) threads = few_threads(sc, threads);
  kernel<<<n, threads, smem, st>>>(sc, b);
  return cudaGetLastError();
}

template cudaError_t launch_step<OST_REAL>(const DevScene&, const StepArgs&, int, cudaStream_t);
template cudaError_t launch_adjoint<OST_REAL>(const DevScene&, const AdjArgs&, int, cudaStream_t);
template int step_threads<OST_REAL>(const DevScene&, int, int);
template size_t ws_bytes<OST_REAL>(const DevScene&);
template size_t step_smem_total<OST_REAL>(const DevScene&);
template size_t adj_smem_total<OST_REAL>(const DevScene&, int);

}  // namespace ost
