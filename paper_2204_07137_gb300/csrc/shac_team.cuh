// Lane form of a forward substep: a team whose lanes cover every link and DOF
// keeps the environment's state and every per-link quantity in registers.
//
// Lane d owns DOF d and, when d is the first DOF of its link, that link; links
// without a DOF (fixed joints) take the lanes after the DOFs.  So one lane holds
// a hinge's coordinate, velocity, pose, inertia and matrix row, and only three
// exchanges of a substep go through shared memory: the subtree sums, the
// right-hand vectors of the mass matrix, and the factor's transpose.
//
//   poses, velocities, accelerations: sums and products along each link's path
//     to the root by shuffles: a specialised build (and the reverse pass) by pointer
//     doubling, in round r a lane combining its value with that of its 2^r-th ancestor
//     (ceil(log2(levels)) rounds); the generic build a level of the tree a round;
//   composite inertias and total forces: subtree sums, one component per lane;
//   specialised: M = L^T L, eliminated leaves first (the last DOF first), so L has no
//     entry outside the pairs (DOF, ancestor DOF): a specialised build, which knows
//     the ancestors, skips the others and factors the DOFs of one tree level together;
//   generic: M = L L^T, root first.
//
// The generic build's forward substep does the general kernels' operations in their
// order (but for the muscles' sums), so a model has the same states, bit for bit, in
// both forms.  A window's gradients jump where a contact, friction or limit switch is
// decided by rounding; with other roundings one of some 80,000 environments came out
// with a gradient some percent off the general kernels' (2 % of the batches of 1531
// ant-like environments over two steps), with the same roundings none.  It costs the
// generic windows about a tenth (1531 environments, h = 8: 1.67 -> 1.78 ms; the general
// kernels 3.97; 512 of the deeper humanoid-like model 7.3 -> 8.8; 19.8).
//
// What bounds it is latency: at 2048 environments an SM holds seven warps, so a
// substep costs its dependent instructions, not its arithmetic.  The per-link
// passes over shared-memory scratch that this form replaces cost a store, a
// barrier and a load between any two of them.  Measured on the ant-like model:
// specialised, 2048 environments, h = 8, forward + adjoint 2.09 -> 1.01 ms (a substep's
// cycles at T = 16, before the roundings above: forward 10.8 k -> 4.4 k, reverse
// 11.5 k -> 5.0 k); the generic kernels on 1531 environments, h = 2: 0.99 -> 0.47 ms.
#pragma once
#include "shac_device.cuh"

namespace shac {

// This lane's share of the model (DevModel::ln_i, ln_f: one column per lane).
enum { LI_LINK = 0, LI_JT, LI_ANC, LI_Q, LI_ACT, LI_C0, LI_C1, LI_DESC, LI_ROW, LI_DLINK, LI_DEPTH, LI_ON_ROOT, LI_N };
enum { LF_AXIS = 0, LF_JROT = 3, LF_JPOS = 12, LF_COM = 15, LF_ICOM = 18, LF_MASS = 24, LF_ARM, LF_DAMP, LF_GEAR,
       LF_QLO, LF_QHI, LF_CPOS, LF_CRAD = LF_CPOS + 3, LF_BASE, LF_N = LF_BASE + 3 };
constexpr int LANE_COLS = 32;
// A row of the mass matrix on its lane: up the tree in the generic build, down it
// in a specialised one (see Dense).
#ifdef SHAC_SPEC_ANC
constexpr int MASS_COLS = LI_DESC;
#else
constexpr int MASS_COLS = LI_ROW;
#endif
constexpr int MSLOTS = 32;   // columns of the muscles' via-point items
constexpr int LINK_CONTACTS = 16;   // contacts of a link whose switches one record word holds

struct LaneConst {
  int link, jt, qi, act, c0, c1, dlink, depth, ms0, ms1;
  unsigned anc, cols;   // cols: entries of the lane's mass-matrix row
  bool own;             // lane < nv
  bool on_root;         // the link is of the free root's tree
  V3 axis, jpos, com, cpos, base;   // cpos, crad: the link's first contact; base: -g on a root link
  M33 jrot;
  float icom[6];
  float mass, arm, damp, gear, qlo, qhi, crad;
  float klim;
};

__device__ __forceinline__ LaneConst lane_const(const DevModel& M, int lane) {
  const int* I = M.ln_i + lane;
  const float* F = M.ln_f + lane;
  auto gi = [&](int k) { return __ldg(I + LANE_COLS * k); };
  auto gf = [&](int k) { return __ldg(F + LANE_COLS * k); };
  LaneConst c;
  c.link = gi(LI_LINK); c.jt = gi(LI_JT); c.anc = (unsigned)gi(LI_ANC); c.qi = gi(LI_Q); c.act = gi(LI_ACT);
  c.c0 = gi(LI_C0); c.c1 = gi(LI_C1); c.cols = (unsigned)gi(MASS_COLS); c.dlink = gi(LI_DLINK);
  c.depth = gi(LI_DEPTH);
  c.ms0 = c.ms1 = 0;
  if (M.nseg > 0 && c.link >= 0) { c.ms0 = __ldg(M.ms_ptr + c.link); c.ms1 = __ldg(M.ms_ptr + c.link + 1); }
  c.own = lane < M.nv;
  c.on_root = gi(LI_ON_ROOT) != 0;
  c.axis = v3(gf(LF_AXIS), gf(LF_AXIS + 1), gf(LF_AXIS + 2));
  c.jpos = v3(gf(LF_JPOS), gf(LF_JPOS + 1), gf(LF_JPOS + 2));
  c.com = v3(gf(LF_COM), gf(LF_COM + 1), gf(LF_COM + 2));
#pragma unroll
  for (int k = 0; k < 9; ++k) c.jrot.m[k] = gf(LF_JROT + k);
#pragma unroll
  for (int k = 0; k < 6; ++k) c.icom[k] = gf(LF_ICOM + k);
  c.mass = gf(LF_MASS); c.arm = gf(LF_ARM); c.damp = gf(LF_DAMP); c.gear = gf(LF_GEAR);
  c.qlo = gf(LF_QLO); c.qhi = gf(LF_QHI);
  c.cpos = v3(gf(LF_CPOS), gf(LF_CPOS + 1), gf(LF_CPOS + 2)); c.crad = gf(LF_CRAD);
  c.base = v3(gf(LF_BASE), gf(LF_BASE + 1), gf(LF_BASE + 2));
  c.klim = M.klim;
  return c;
}

// State in registers: the lane's joint coordinate (one-DOF joints) and its
// DOF's velocity with their compensations; the free root's pose and velocity on
// every lane (its rotation is a factor of every lane's work).
struct LaneState {
  float q, qc, qd, qdc;
  float rq[7], rqc[3];
  float rqd[6], rqdc[3];   // rqdc: compensations of the body velocity
};

__device__ __forceinline__ float team_shfl(float x, int src, int nl) { return __shfl_sync(0xffffffffu, x, src, nl); }
__device__ __forceinline__ V3 team_shfl(V3 x, int src, int nl) {
  return v3(team_shfl(x.x, src, nl), team_shfl(x.y, src, nl), team_shfl(x.z, src, nl));
}

// Sums of a and b along the path to the root (own value included) in the forward
// substep.  A specialised build doubles.  The generic build takes the levels of the
// tree in turn, the links of level r adding their parents': the general kernels' order
// of additions, so that states come out the same to the last bit in both.
__device__ __forceinline__ void path_sums(const DevModel& M, const LaneConst& c, int nl, V3& a, V3& b) {
#ifdef SHAC_SPEC_ANC
#pragma unroll
  for (int r = 0; r < M.nround; ++r) {
    const unsigned s = (c.anc >> (6 * r)) & 63u;
    const V3 pa = team_shfl(a, (int)(s & 31u), nl), pb = team_shfl(b, (int)(s & 31u), nl);
    if (s < 32u) { a = a + pa; b = b + pb; }
  }
#else
  const int src = (int)(c.anc & 31u);
  for (int r = 1; r <= M.deepest; ++r) {
    const V3 pa = team_shfl(a, src, nl), pb = team_shfl(b, src, nl);
    if (c.depth == r) { a = a + pa; b = b + pb; }
  }
#endif
}

// 1 / sqrt(x): rsqrtf (documented maximum error 2 ulp) and one Newton step of
// y -> y (3 - x y^2) / 2, to a relative error below 1.5 * 2^-24; 0 gives infinity and
// infinity 0, where the step has no value.  Serves muscle lengths and, in the reverse
// pass, sliding speeds and the quaternion's norm.  200 environments of the 152-muscle
// model, specialised, h = 3, take 0.71 ms forward and 1.47 ms back with it, 0.73 and
// 1.56 ms with 1.f / sqrtf(x) for the lengths; the ant-like model's window on the ground
// 0.73 ms back with it and 0.75 with 1.f / sqrtf(x) for the speeds (1531, h = 8).
__device__ __forceinline__ float rsqrt_refined(float x) {
  const float y = rsqrtf(x), e = fmaf(-x * y, y, 1.f);
  return fabsf(e) < 1.f ? fmaf(0.5f * y, e, y) : y;
}

// 16-byte shared-memory accesses (o a multiple of 4).
__device__ __forceinline__ void sts4(const SMem& w, int o, float a, float b, float c, float d) {
  *reinterpret_cast<float4*>(&w[o]) = make_float4(a, b, c, d);
}
__device__ __forceinline__ float4 lds4(const SMem& w, int o) { return *reinterpret_cast<const float4*>(&w[o]); }

// Exchange buffers (offsets from o_X, multiples of 4 floats): per link the 16
// components of [Ic, F] in 20 floats (the 16-byte accesses of eight lanes then
// meet eight distinct bank groups), per DOF the vector Ic S in 8, then the
// factor's rows.
constexpr int XB = 20, XF = 8;
__host__ __device__ constexpr int dense_stride(int nm) { return (nm + 3) / 4 * 4 + ((nm + 3) / 4 % 2 ? 0 : 4); }
__host__ __device__ constexpr int lane_xchg_floats(int L, int nm) {
  return XB * L + (XF * nm + dense_stride(nm) * nm > XF * L ? XF * nm + dense_stride(nm) * nm : XF * L);
}

// ---- substep record of the lane form -------------------------------------
// What the reverse pass reads, one block per substep (offsets in floats, every
// array of 16-byte elements indexed by link or DOF, so that lanes read and
// write consecutive 16 bytes):
//   8 float4 [link]: R, P, spatial inertia, velocity, external wrench (32 of 34); in the
//                    place of the inertia's mass, a model constant, the contacts' switches
//   1 float4 [DOF]:  qd, qdd, 1 / L_kk, q (one-DOF joints)
//   rows of the unit factor, float4 [entry / 4][DOF]
//   free root: q 7, qd 6, qdd 6, pad
//   1 float2 [link]: the external wrench's last two
//   via points of the muscle segments, x y z planes in item order (below)
struct LaneRecord {
  int dof, fac, root, fx, items;   // offsets; items: floats before the via points
  int rs;                          // DOFs per factor row block (odd beyond 8: column reads then spread over the banks)
};
__host__ __device__ constexpr int record_row_stride(int nv) { return nv > 8 ? (nv | 1) : nv; }
__host__ __device__ inline LaneRecord lane_record(int L, int nv, int nm, int root_free) {
  LaneRecord r;
  r.rs = record_row_stride(nv);
  r.dof = 32 * L;
  r.fac = r.dof + 4 * nv;
  r.root = r.fac + 4 * ((nm + 3) / 4) * r.rs;
  r.fx = r.root + (root_free ? 20 : 0);
  r.items = (r.fx + 2 * L + 3) / 4 * 4;
  return r;
}

__device__ __forceinline__ void stg4(float* p, float a, float b, float c, float d) {
  *reinterpret_cast<float4*>(p) = make_float4(a, b, c, d);
}

// Request a record's copy to shared memory (n floats, 16 bytes per copy, all in
// flight together); record_wait waits for this lane's copies (the caller's team
// barrier makes them visible to the team).
__device__ __forceinline__ void record_request(const SMem& w, int o, const float* src, int n, int lane, int nl) {
  for (int j = lane; j < n / 4; j += nl) {
    const unsigned dst = (unsigned)__cvta_generic_to_shared(&w[o + 4 * j]);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(dst), "l"(src + 4 * j) : "memory");
  }
  asm volatile("cp.async.commit_group;\n" ::: "memory");
}
__device__ __forceinline__ void record_wait() { asm volatile("cp.async.wait_group 0;\n" ::: "memory"); }

// Subtree sums of NC values a link; on return this lane's DOF's link's sums
// (lanes from nv on: their link's or the first link's, not used).  Each link's
// values go to its block of the exchange buffer, one component per lane adds
// child to parent, last link first.  A specialised build does so at constant
// addresses (150 cycles for the ant-like model's nine links and 16 components).
// With the tree known at run time only, a chain's running sum (parent = i - 1)
// stays in a register, the next link's value and parent are read ahead, and only
// a branch goes back to memory.
template <int NC>
__device__ __forceinline__ void lane_sums(const DevModel& M, const SMem& w, float (&x)[NC], const LaneConst& c,
                                          bool link, int lane, int nl) {
  constexpr int N4 = (NC + 3) / 4;
  if (link) {
#pragma unroll
    for (int j = 0; j < N4; ++j)
      sts4(w, M.o_X + XB * c.link + 4 * j, x[4 * j], 4 * j + 1 < NC ? x[4 * j + 1 < NC ? 4 * j + 1 : 0] : 0.f,
           4 * j + 2 < NC ? x[4 * j + 2 < NC ? 4 * j + 2 : 0] : 0.f, 4 * j + 3 < NC ? x[4 * j + 3 < NC ? 4 * j + 3 : 0] : 0.f);
  }
  team_sync(nl);
  for (int k = lane; k < NC; k += nl) {
#ifdef SHAC_SPEC_PARENTS
#pragma unroll
    for (int i = M.L - 1; i > 0; --i) {
      const int p = link_parent(M, i);
      if (p >= 0) w[M.o_X + XB * p + k] += w[M.o_X + XB * i + k];
    }
#else
    const int o = M.o_X + k;
    int a = o + XB * (M.L - 1), p = M.par8[M.L - 1];
    float v = w[a], carry = 0.f;
    for (int i = M.L - 1; i > 0; --i) {
      const float vn = w[a - XB];
      const int pn = M.par8[i - 1];
      const float s = v + carry;
      w[a] = s;
      // a branch's parent takes the sum in memory; otherwise the same access adds
      // nothing to this link's own (spent) block, which costs less than a jump
      const bool chain = p == i - 1, up = !chain && p >= 0;
      const int b = up ? o + XB * p : a;
      w[b] += up ? s : 0.f;
      carry = chain ? s : 0.f;
      v = vn;
      p = pn;
      a -= XB;
    }
    w[a] = v + carry;
#endif
  }
  team_sync(nl);
#pragma unroll
  for (int j = 0; j < N4; ++j) {
    const float4 v = lds4(w, M.o_X + XB * c.dlink + 4 * j);
    x[4 * j] = v.x;
    if (4 * j + 1 < NC) x[4 * j + 1 < NC ? 4 * j + 1 : 0] = v.y;
    if (4 * j + 2 < NC) x[4 * j + 2 < NC ? 4 * j + 2 : 0] = v.z;
    if (4 * j + 3 < NC) x[4 * j + 3 < NC ? 4 * j + 3 : 0] = v.w;
  }
  team_sync(nl);   // the blocks are free again
}

// Assembly of the lane's row of M + diag(arm) and the factor's rows in the record,
// common to both eliminations below.
template <int NM>
struct DenseRows {
  static constexpr int ST = dense_stride(NM);
  // row[b] = (xw, xv) . (vector of DOF b at of) for the columns in c.cols, zero
  // elsewhere; lanes from nv on: identity rows.
  // The columns go in groups whose vectors are all read before the first product
  // (one at a time, every column waited for its own reads: 54 cycles each).
  static constexpr int GROUP = 7;
  template <int B0, int... B>
  static __device__ __forceinline__ void assemble_group(const SMem& w, int of, V3 sw, V3 sv, const LaneConst& c,
                                                        int lane, float (&row)[NM], float& diag, iseq<B...>) {
    float4 f0[sizeof...(B)];
    float2 f1[sizeof...(B)];
    ([&] {
      f0[B] = lds4(w, of + XF * (B0 + B));
      f1[B] = *reinterpret_cast<const float2*>(&w[of + XF * (B0 + B) + 4]);
    }(), ...);
    ([&] {
      const float p = dot(sw, v3(f0[B].x, f0[B].y, f0[B].z)) + dot(sv, v3(f0[B].w, f1[B].x, f1[B].y));
      float v = ((c.cols >> (B0 + B)) & 1u) ? p : 0.f;
      if (B0 + B == lane) { v += c.arm; diag = v; }
      row[B0 + B] = v;
    }(), ...);
  }
  template <int B0 = 0>
  static __device__ __forceinline__ void assemble(const SMem& w, int of, V3 sw, V3 sv, const LaneConst& c, int lane,
                                                  float (&row)[NM], float& diag) {
    if constexpr (B0 < NM) {
      assemble_group<B0>(w, of, sw, sv, c, lane, row, diag, make_iseq<(NM - B0 < GROUP ? NM - B0 : GROUP)>{});
      assemble<B0 + GROUP>(w, of, sw, sv, c, lane, row, diag);
    }
  }
  // One lane's row of the factor (in the form ls) to the record: 16 bytes of every
  // row side by side.
  static __device__ __forceinline__ void store_row(float* fac, int rs, const float (&ls)[NM], int lane) {
#pragma unroll
    for (int k = 0; k < (NM + 3) / 4; ++k)
      stg4(fac + 4 * (k * rs + lane), ls[4 * k], 4 * k + 1 < NM ? ls[4 * k + 1 < NM ? 4 * k + 1 : 0] : 0.f,
           4 * k + 2 < NM ? ls[4 * k + 2 < NM ? 4 * k + 2 : 0] : 0.f,
           4 * k + 3 < NM ? ls[4 * k + 3 < NM ? 4 * k + 3 : 0] : 0.f);
  }
  // The record's factor: entries k > lane of this lane's column and, below, all of
  // its row (both zero elsewhere).
  static __device__ __forceinline__ void load_record(const SMem& w, int of, int rs, int n, int lane, float (&lc)[NM],
                                                     float (&ls)[NM]) {
    const int oc = of + 4 * (lane >> 2) * rs + (lane & 3);
#pragma unroll
    for (int k = 0; k < NM; ++k) {
      const bool use = lane < k && k < n;
      const float v = w[use ? oc + 4 * k : of];
      lc[k] = use ? v : 0.f;
    }
#pragma unroll
    for (int k = 0; k < (NM + 3) / 4; ++k) {
      const float4 v = lds4(w, of + 4 * (k * rs + (lane < n ? lane : 0)));
      const float t[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (4 * k + j < NM) ls[4 * k + j < NM ? 4 * k + j : 0] = lane < n ? t[j] : 0.f;
    }
  }
};

#ifdef SHAC_SPEC_ANC
// A specialised build eliminates leaves first, M = L^T L.  It has the ancestor masks
// as literals, so it knows which entries of the factor exist and which DOFs may be
// eliminated together.
constexpr unsigned kAncMask[] = {SHAC_SPEC_ANC};
constexpr int kAncCount = sizeof(kAncMask) / sizeof(kAncMask[0]);
__host__ __device__ constexpr bool has_entry(int k, int j) { return k < kAncCount && j < k && ((kAncMask[k] >> j) & 1u); }
__host__ __device__ constexpr int dof_level(int k) {   // number of ancestors
  if (k >= kAncCount) return -1;
  int n = -1;
  for (int b = 0; b < 32; ++b) n += (kAncMask[k] >> b) & 1u;
  return n;
}

// Lane a holds row[b] = M_ab for its descendants b >= a (and itself), its
// diagonal in diag and the right-hand side in b.  Eliminating DOF k: L_kk =
// sqrt(pivot), L_ka = M_ak / L_kk on lane a, M_aj -= L_ka L_kj, and the forward
// substitution y_k = b_k / L_kk, b_a -= L_ka y_k in the same pass.  L_ka goes to
// row k of the factor in shared memory, where lane k reads it for the backward
// substitution and the record keeps it for the adjoint: the unit factor, row k
// holding L_kj / L_kk for j < k, next to 1 / L_kk.
template <int NM>
struct Dense : DenseRows<NM> {
  using Rows = DenseRows<NM>;
  static constexpr int ST = Rows::ST;
  template <int K, int J>
  static __device__ __forceinline__ void update(float (&row)[NM], float lk, int nl) {
    if constexpr (has_entry(K, J)) row[J] = fmaf(-lk, team_shfl(lk, J, nl), row[J]);
  }
  template <int K, int... J>
  static __device__ __forceinline__ void updates(float (&row)[NM], float lk, int nl, iseq<J...>) {
    (update<K, J>(row, lk, nl), ...);
  }
  template <int LV, int K>
  static __device__ __forceinline__ void pivot(float diag, float (&inv)[NM], float b, float (&y)[NM], int nl) {
    if constexpr (dof_level(K) == LV) {
      inv[K] = rsqrtf(team_shfl(diag, K, nl));
      y[K] = team_shfl(b, K, nl) * inv[K];
    }
  }
  template <int LV, int K>
  static __device__ __forceinline__ void column(const SMem& w, int ol, float (&row)[NM], float& diag, float& idiag,
                                                const float (&inv)[NM], float& b, const float (&y)[NM], int lane,
                                                int nl) {
    if constexpr (dof_level(K) == LV) {
      const float lk = row[K] * inv[K];
      if (lane < K) {
        w[ol + ST * K + lane] = lk;
        diag = fmaf(-lk, lk, diag);
        b = fmaf(-lk, y[K], b);
      }
      if (lane == K) { idiag = inv[K]; b = y[K]; }
      updates<K>(row, lk, nl, make_iseq<K>{});
    }
  }
  template <int LV, int... K>
  static __device__ __forceinline__ void level(const SMem& w, int ol, float (&row)[NM], float& diag, float& idiag,
                                               float (&inv)[NM], float& b, float (&y)[NM], int lane, int nl,
                                               iseq<K...>) {
    (pivot<LV, K>(diag, inv, b, y, nl), ...);
    (column<LV, K>(w, ol, row, diag, idiag, inv, b, y, lane, nl), ...);
  }
  template <int... LV>
  static __device__ __forceinline__ void factor(const SMem& w, int ol, float (&row)[NM], float& diag, float& idiag,
                                                float& b, int lane, int nl, iseq<LV...>) {
    float inv[NM], y[NM];
    (level<NM - 1 - LV>(w, ol, row, diag, idiag, inv, b, y, lane, nl, make_iseq<NM>{}), ...);
  }
  // L x = y with row `lane` of L scaled by 1 / L_kk: z_a -= (L_ak / L_aa) x_k,
  // a level's x_k read together.
  template <int LV, int K>
  static __device__ __forceinline__ void back_read(float z, float (&x)[NM], int nl) {
    if constexpr (dof_level(K) == LV) x[K] = team_shfl(z, K, nl);
  }
  template <int LV, int K>
  static __device__ __forceinline__ void back_apply(float& z, const float (&x)[NM], const float (&ls)[NM]) {
    if constexpr (dof_level(K) == LV) z = fmaf(-ls[K], x[K], z);
  }
  template <int LV, int... K>
  static __device__ __forceinline__ void back_level(float& z, float (&x)[NM], const float (&ls)[NM], int nl,
                                                    iseq<K...>) {
    (back_read<LV, K>(z, x, nl), ...);
    (back_apply<LV, K>(z, x, ls), ...);
  }
  template <int... LV>
  static __device__ __forceinline__ void back(float& z, const float (&ls)[NM], int nl, iseq<LV...>) {
    float x[NM];
    (back_level<LV>(z, x, ls, nl, make_iseq<NM>{}), ...);
  }
  // row `lane` of the factor in shared memory, scaled, zero from the diagonal on
  static __device__ __forceinline__ void load_row(const SMem& w, int ol, float idiag, int lane, float (&ls)[NM]) {
    const int o = ol + ST * (lane < NM ? lane : 0);
    float t[(NM + 3) / 4 * 4];
#pragma unroll
    for (int k = 0; k < (NM + 3) / 4; ++k) {
      const float4 v = lds4(w, o + 4 * k);
      t[4 * k] = v.x; t[4 * k + 1] = v.y; t[4 * k + 2] = v.z; t[4 * k + 3] = v.w;
    }
#pragma unroll
    for (int k = 0; k < NM; ++k) ls[k] = lane > k ? t[k] * idiag : 0.f;
  }

  // Assemble, factor and solve (M + diag(arm)) x = b; returns x of this lane's
  // DOF and 1 / L_kk in idiag.  sw, sv: the lane's motion subspace; fn, ff: Ic S of
  // its DOF, which every lane's row needs (the vectors at of).
  static __device__ __forceinline__ void put_vector(const SMem& w, int of, int lane, V3 sw, V3 sv, V3 fn, V3 ff) {
    sts4(w, of + XF * lane, fn.x, fn.y, fn.z, ff.x);
    *reinterpret_cast<float2*>(&w[of + XF * lane + 4]) = make_float2(ff.y, ff.z);
  }
  static __device__ __forceinline__ float solve(const SMem& w, float* fac, int rs, int of, int ol, V3 sw, V3 sv, V3 fn,
                                                V3 ff, float b, const LaneConst& c, int lane, int nl, float& idiag) {
    float row[NM], diag = 1.f;
    Rows::assemble(w, of, sw, sv, c, lane, row, diag);
    factor(w, ol, row, diag, idiag, b, lane, nl, make_iseq<NM>{});
    team_sync(nl);
    float ls[NM];
    load_row(w, ol, idiag, lane, ls);
    if (fac && c.own) Rows::store_row(fac, rs, ls, lane);
    float z = b * idiag;
    back(z, ls, nl, make_iseq<NM>{});
    return z;
  }
  // x = (L^T L)^{-1} b from the record: b_a -= (L_ka / L_kk) b_k leaves first,
  // scaled by 1 / L_kk^2, then back as above.
  template <int LV, int K>
  static __device__ __forceinline__ void fwd_read(float b, float (&y)[NM], int nl) {
    if constexpr (dof_level(K) == LV) y[K] = team_shfl(b, K, nl);
  }
  template <int LV, int K>
  static __device__ __forceinline__ void fwd_apply(float& b, const float (&y)[NM], const float (&lc)[NM]) {
    if constexpr (dof_level(K) == LV) b = fmaf(-lc[K], y[K], b);
  }
  template <int LV, int... K>
  static __device__ __forceinline__ void fwd_level(float& b, float (&y)[NM], const float (&lc)[NM], int nl,
                                                   iseq<K...>) {
    (fwd_read<LV, K>(b, y, nl), ...);
    (fwd_apply<LV, K>(b, y, lc), ...);
  }
  template <int... LV>
  static __device__ __forceinline__ float solve_record(const SMem& w, int of, int rs, int n, float idiag, float b,
                                                       int lane, int nl, iseq<LV...>) {
    float y[NM], lc[NM], ls[NM];
    Rows::load_record(w, of, rs, n, lane, lc, ls);
    (fwd_level<NM - 1 - LV>(b, y, lc, nl, make_iseq<NM>{}), ...);
    float z = b * (idiag * idiag);
    back(z, ls, nl, make_iseq<NM>{});
    return z;
  }
};
#else
// The generic build eliminates root first, M = L L^T, one DOF at a time, with the
// general kernels' operations in their order (dense_substep): a model's states then
// do not depend on which of the two forms its batch takes, to the last bit, and no
// contact, friction or limit switch of a window falls differently in them.  With the
// tree known at run time only, leaves first would take as many steps.
//
// Lane a holds row[b] = M_ab for its ancestors b <= a, its diagonal in diag and the
// right-hand side in b.  Eliminating DOF k: L_ik = M_ik / L_kk on the lanes i > k,
// M_ij -= L_ik L_jk, and the forward substitution y_k = b_k / L_kk, b_i -= L_ik y_k in
// the same pass.  Column k goes to shared memory, where lane k reads it for the
// backward substitution; the record keeps the rows, next to 1 / L_kk.
template <int NM>
struct Dense : DenseRows<NM> {
  using Rows = DenseRows<NM>;
  static constexpr int ST = Rows::ST;
  template <int K, int... J>
  static __device__ __forceinline__ void trailing(float (&row)[NM], float lk, int nl, iseq<J...>) {
    ((row[K + 1 + J] = fmaf(-lk, team_shfl(lk, K + 1 + J, nl), row[K + 1 + J])), ...);
  }
  template <int K>
  static __device__ __forceinline__ void column(const SMem& w, int ol, float (&row)[NM], float& diag, float& idiag,
                                                float& b, int lane, int nl) {
    const float inv = rsqrtf(team_shfl(diag, K, nl));
    const float yk = team_shfl(b, K, nl) * inv;
    const float lk = row[K] * inv;
    row[K] = lk;
    if (lane == K) { idiag = inv; b = yk; }
    if (lane > K) {
      diag = fmaf(-lk, lk, diag);
      b = fmaf(-lk, yk, b);
    }
    trailing<K>(row, lk, nl, make_iseq<NM - K - 1>{});
  }
  template <int... K>
  static __device__ __forceinline__ void factor(const SMem& w, int ol, float (&row)[NM], float& diag, float& idiag,
                                                float& b, int lane, int nl, iseq<K...>) {
    (column<K>(w, ol, row, diag, idiag, b, lane, nl), ...);
  }
  // L^T x = y: x_k = y_k / L_kk, y_a -= L_ka x_k, the last DOF first; lc: this lane's
  // column of L.
  template <int K>
  static __device__ __forceinline__ void back_step(float& b, const float (&lc)[NM], float idiag, int lane, int nl) {
    const float xk = team_shfl(b * idiag, K, nl);
    b = lane == K ? xk : fmaf(-lc[K], xk, b);
  }
  template <int... K>
  static __device__ __forceinline__ void back(float& b, const float (&lc)[NM], float idiag, int lane, int nl, iseq<K...>) {
    (back_step<NM - 1 - K>(b, lc, idiag, lane, nl), ...);
  }
  // Assemble, factor and solve (M + diag(arm)) x = b; returns x of this lane's
  // DOF and 1 / L_kk in idiag.  sw, sv: the lane's motion subspace, which every lane's
  // row needs (the vectors at of); fn, ff: Ic S of its DOF.
  static __device__ __forceinline__ void put_vector(const SMem& w, int of, int lane, V3 sw, V3 sv, V3 fn, V3 ff) {
    sts4(w, of + XF * lane, sw.x, sw.y, sw.z, sv.x);
    *reinterpret_cast<float2*>(&w[of + XF * lane + 4]) = make_float2(sv.y, sv.z);
  }
  static __device__ __forceinline__ float solve(const SMem& w, float* fac, int rs, int of, int ol, V3 sw, V3 sv, V3 fn,
                                                V3 ff, float b, const LaneConst& c, int lane, int nl, float& idiag) {
    float row[NM], diag = 1.f;
    Rows::assemble(w, of, fn, ff, c, lane, row, diag);
    factor(w, ol, row, diag, idiag, b, lane, nl, make_iseq<NM>{});
#pragma unroll
    for (int k = 0; k < NM; ++k) row[k] = k < lane ? row[k] : 0.f;
    if (lane < NM) {
#pragma unroll
      for (int k = 0; k < (NM + 3) / 4; ++k)
        sts4(w, ol + ST * lane + 4 * k, row[4 * k], 4 * k + 1 < NM ? row[4 * k + 1 < NM ? 4 * k + 1 : 0] : 0.f,
             4 * k + 2 < NM ? row[4 * k + 2 < NM ? 4 * k + 2 : 0] : 0.f,
             4 * k + 3 < NM ? row[4 * k + 3 < NM ? 4 * k + 3 : 0] : 0.f);
    }
    if (fac && c.own) Rows::store_row(fac, rs, row, lane);
    team_sync(nl);
    float lc[NM];
#pragma unroll
    for (int k = 0; k < NM; ++k) {   // zero in the row's own upper part
      const float v = w[ol + ST * k + (lane < NM ? lane : 0)];
      lc[k] = lane < k ? v : 0.f;
    }
    back(b, lc, idiag, lane, nl, make_iseq<NM>{});
    return b;
  }
  // x = (L L^T)^{-1} b from the record
  template <int K>
  static __device__ __forceinline__ void fwd_step(float& b, const float (&ls)[NM], float idiag, int lane, int nl) {
    const float yk = team_shfl(b * idiag, K, nl);
    b = lane == K ? yk : fmaf(-ls[K], yk, b);
  }
  template <int... K>
  static __device__ __forceinline__ float solve_record(const SMem& w, int of, int rs, int n, float idiag, float b,
                                                       int lane, int nl, iseq<K...>) {
    float lc[NM], ls[NM];
    Rows::load_record(w, of, rs, n, lane, lc, ls);
    (fwd_step<K>(b, ls, idiag, lane, nl), ...);
    back(b, lc, idiag, lane, nl, iseq<K...>{});
    return b;
  }
};
#endif

// Position update of the free root (replicated on every lane) from its new
// velocity: p += h R v, quat <- normalise(quat + h/2 quat (x) (w, 0)); see
// lk_integrate.
__device__ __forceinline__ void root_integrate(const DevModel& M, const M33& R, LaneState& s) {
  const V3 v = v3(s.rqd[3], s.rqd[4], s.rqd[5]), vc = v3(s.rqdc[0], s.rqdc[1], s.rqdc[2]);
  const V3 dp = M.h * mul(R, v) + M.h * mul(R, vc);
  s.rq[0] = two_sum(s.rq[0], dp.x + s.rqc[0], s.rqc[0]);
  s.rq[1] = two_sum(s.rq[1], dp.y + s.rqc[1], s.rqc[1]);
  s.rq[2] = two_sum(s.rq[2], dp.z + s.rqc[2], s.rqc[2]);
  const V3 u = v3(s.rq[3], s.rq[4], s.rq[5]), om = v3(s.rqd[0], s.rqd[1], s.rqd[2]);
  const float qw = s.rq[6], hh = 0.5f * M.h;
  const V3 n = u + hh * (qw * om + cross(u, om));
  const float nw = qw - hh * dot(u, om);
  const float inv = rsqrtf(dot(n, n) + nw * nw);
  s.rq[3] = n.x * inv; s.rq[4] = n.y * inv; s.rq[5] = n.z * inv; s.rq[6] = nw * inv;
}

// Contacts and local force of this lane's link (lk_local), from registers: the
// spatial inertia si, the external wrench (wn, wf) and F.
struct LaneLink {
  M33 R;
  V3 P, Vw, Vv, aw, av;
  float si[10];         // m, h, Io
  V3 wn, wf, fn, ff;
  // two bits a contact, the link's first lowest: touching, and sliding slowly (the
  // viscous branch).  The reverse pass takes the branches the forward took from here: a
  // test repeated from the record, within rounding of its switch, could fall the other
  // way and give the gradient of another force than the one that acted.
  unsigned contacts;
};
// COMPOSITE: the composite inertia's product with a motion subspace, whose y component
// rounds as the general kernels' (si_mul of shac_device.cuh).
template <bool COMPOSITE = false>
__device__ __forceinline__ void si_mul(const float (&si)[10], V3 xw, V3 xv, V3& yn, V3& yf) {
  const V3 h = v3(si[1], si[2], si[3]);
  yn = v3(sum3(si[4], xw.x, si[7], xw.y, si[8], xw.z),
          COMPOSITE ? sum3(si[5], xw.y, si[7], xw.x, si[9], xw.z) : sum3(si[7], xw.x, si[5], xw.y, si[9], xw.z),
          sum3(si[8], xw.x, si[9], xw.y, si[6], xw.z)) + cross(h, xv);
  yf = si[0] * xv - cross(h, xw);
}
__device__ __forceinline__ void lane_local(const DevModel& M, const LaneConst& c, float zroot,
                                           LaneLink& k) {
  const V3 cm = k.P + mul(k.R, c.com);
  M33 Ic;
  Ic.m[0] = c.icom[0]; Ic.m[4] = c.icom[1]; Ic.m[8] = c.icom[2];
  Ic.m[1] = Ic.m[3] = c.icom[3]; Ic.m[2] = Ic.m[6] = c.icom[4]; Ic.m[5] = Ic.m[7] = c.icom[5];
  const M33 Iw = mulBT(mul(k.R, Ic), k.R);
  spatial_inertia(Iw, c.mass, cm, k.si);
  k.wn = k.wf = v3(0.f, 0.f, 0.f);
  k.contacts = 0u;
  V3 xl = c.cpos;
  float rad = c.crad;
  for (int e = c.c0; e < c.c1;) {   // contact spheres (the model of lk_local)
    V3 x = k.P + mul(k.R, xl);
    x.z -= rad;
    const float d = x.z + zroot;
    V3 f = v3(0.f, 0.f, 0.f);
    if (d < 0.f) {
      const V3 vp = k.Vv + cross(k.Vw, x);
      const float fn = (-M.ke + M.kd * vp.z) * d;
      const float vt = sqrtf(sum2(vp.x, vp.x, vp.y, vp.y));
      const float fmax = M.mu * fabsf(fn);
      const bool slow = M.kt * vt <= fmax;
      const float sc = slow ? M.kt : fmax / vt;
      k.contacts |= (slow ? 3u : 1u) << (2 * (e - c.c0));
      f.x = -sc * vp.x; f.y = -sc * vp.y;
      f.z = fn;
    }
    k.wn = k.wn + cross(x, f);
    k.wf = k.wf + f;
    if (++e < c.c1) {
      const int ci = __ldg(M.lc_idx + e);
      xl = cld3(M.item_pos + 3 * ci);
      rad = __ldg(M.crad + ci);
    }
  }
  V3 bn, bf;
  si_mul(k.si, k.aw, k.av, k.fn, k.ff);
  si_mul(k.si, k.Vw, k.Vv, bn, bf);
  k.fn = k.fn + cross(k.Vw, bn) + cross(k.Vv, bf) - k.wn;
  k.ff = k.ff + cross(k.Vw, bf) - k.wf;
}

// Segments a lane takes together: all their reads come before the first store
// (which could alias them for all the compiler knows), so their latencies overlap.
constexpr int SEG_GROUP = 2;

// Muscles of the lane form.  The via-point items are laid out in MSLOTS columns
// of mrows (row j of column s at j * MSLOTS + (s + j) % MSLOTS: both a row and
// the consecutive items of a link, which neighbouring lanes write, lie on
// different banks; without the shift a segment step took 770 cycles, with it
// 580), every column one link's items
// and every link at least its share of columns, so that the per-link sums take
// mrows conflict-free steps whatever the distribution of the items over the
// links (a lane per link takes as many steps as the busiest link has items: 99
// of the 152-muscle model's 608, where 22 rows serve).  The unused places hold
// zeros.  512 environments of that model, h = 2: 7.27 -> 1.41 ms, the scratch of
// an environment down from 60 to 36 KB, so that all of them are resident.  Planes of MSLOTS * mrows floats: points x y z at o_MX, forces (reverse:
// the points' cotangents) x y z at o_MF.
__device__ __forceinline__ void muscle_clear(const DevModel& M, const SMem& w, int lane, int nl) {
  zero_range(w, M.o_MX, 3 * MSLOTS * M.mrows, lane, nl);
  zero_range(w, M.o_MF, 3 * MSLOTS * M.mrows, lane, nl);
}
__device__ __forceinline__ void muscle_put_pose(const DevModel& M, const SMem& w, int link, const M33& R, V3 P) {
  if (link < 0) return;
  const int o = M.o_MP + 12 * link;
  sts4(w, o, R.m[0], R.m[1], R.m[2], R.m[3]);
  sts4(w, o + 4, R.m[4], R.m[5], R.m[6], R.m[7]);
  sts4(w, o + 8, R.m[8], P.x, P.y, P.z);
}
// One segment's constants: its ends in their links' frames, fmax, links, muscle
// and places.
struct Segment {
  V3 p0, p1;
  float fmax;
  int l0, l1, mus, i0, i1;
};
__device__ __forceinline__ Segment muscle_segment(const DevModel& M, int sg) {
  const float4 a = __ldg(reinterpret_cast<const float4*>(M.sg_f) + sg);
  const float4 b = __ldg(reinterpret_cast<const float4*>(M.sg_f) + M.nseg + sg);
  const unsigned pl = (unsigned)__ldg(M.sg_place + sg), id = __float_as_uint(b.w);
  Segment s;
  s.p0 = v3(a.x, a.y, a.z); s.fmax = a.w; s.p1 = v3(b.x, b.y, b.z);
  s.l0 = (int)(id & 255u); s.l1 = (int)((id >> 8) & 255u); s.mus = (int)(id >> 16);
  s.i0 = (int)(pl & 0xffffu); s.i1 = (int)(pl >> 16);
  return s;
}
__device__ __forceinline__ V3 plane_ld(const SMem& w, int o, int n, int i) { return v3(w[o + i], w[o + n + i], w[o + 2 * n + i]); }
__device__ __forceinline__ void plane_st(const SMem& w, int o, int n, int i, V3 v) {
  w[o + i] = v.x; w[o + n + i] = v.y; w[o + 2 * n + i] = v.z;
}
__device__ __forceinline__ void muscle_forward(const DevModel& M, const SMem& w, int lane, int nl) {
  const int n = MSLOTS * M.mrows;
  auto point = [&](int link, V3 p) {
    const int o = M.o_MP + 12 * link;
    const float4 a = lds4(w, o), b = lds4(w, o + 4), c = lds4(w, o + 8);
    M33 R;
    R.m[0] = a.x; R.m[1] = a.y; R.m[2] = a.z; R.m[3] = a.w; R.m[4] = b.x; R.m[5] = b.y; R.m[6] = b.z; R.m[7] = b.w;
    R.m[8] = c.x;
    return v3(c.y, c.z, c.w) + mul(R, p);
  };
  for (int s0 = lane; s0 < M.nseg; s0 += SEG_GROUP * nl) {   // seg_forward
    V3 x0[SEG_GROUP], x1[SEG_GROUP], f[SEG_GROUP];
    int i0[SEG_GROUP], i1[SEG_GROUP];
#pragma unroll
    for (int g = 0; g < SEG_GROUP; ++g) {
      const Segment s = muscle_segment(M, min(s0 + g * nl, M.nseg - 1));
      x0[g] = point(s.l0, s.p0); x1[g] = point(s.l1, s.p1);
      i0[g] = s.i0; i1[g] = s.i1;
      const float a = fminf(fmaxf(w[M.o_ACT + M.ntact + s.mus], 0.f), 1.f);
      const V3 dv = x1[g] - x0[g];
      f[g] = (a * s.fmax) * (rsqrt_refined(dot(dv, dv)) * dv);
    }
#pragma unroll
    for (int g = 0; g < SEG_GROUP; ++g) {
      if (s0 + g * nl < M.nseg) {
        plane_st(w, M.o_MX, n, i0[g], x0[g]);
        plane_st(w, M.o_MX, n, i1[g], x1[g]);
        plane_st(w, M.o_MF, n, i0[g], f[g]);
        plane_st(w, M.o_MF, n, i1[g], -f[g]);
      }
    }
  }
  team_sync(nl);
  for (int c = lane; c < MSLOTS; c += nl) {
    V3 wn = v3(0.f, 0.f, 0.f), wf = wn;
#pragma unroll 4
    for (int j = 0; j < M.mrows; ++j) {
      const V3 x = plane_ld(w, M.o_MX, n, MSLOTS * j + ((c + j) & (MSLOTS - 1))), f = plane_ld(w, M.o_MF, n, MSLOTS * j + ((c + j) & (MSLOTS - 1)));
      wn = wn + cross(x, f);
      wf = wf + f;
    }
    st3(w, M.o_MW + 12 * c, wn);
    st3(w, M.o_MW + 12 * c + 3, wf);
  }
  team_sync(nl);
}
// Reverse of every segment (seg_adjoint) from the recorded points: the
// activations' cotangents into o_ACTB, per column the sums of the points'
// cotangents x_bar and of x_bar x^T.
__device__ __forceinline__ void muscle_reverse(const DevModel& M, const SMem& w, int lane, int nl) {
  const int n = MSLOTS * M.mrows;
  for (int s0 = lane; s0 < M.nseg; s0 += SEG_GROUP * nl) {
    V3 b0[SEG_GROUP], b1[SEG_GROUP];
    float ab[SEG_GROUP];
    int i0[SEG_GROUP], i1[SEG_GROUP];
#pragma unroll
    for (int k = 0; k < SEG_GROUP; ++k) {
      const Segment s = muscle_segment(M, min(s0 + k * nl, M.nseg - 1));
      const V3 x0 = plane_ld(w, M.o_MX, n, s.i0), x1 = plane_ld(w, M.o_MX, n, s.i1);
      const V3 n0 = ld3(w, M.o_MB + 6 * s.l0), e0 = ld3(w, M.o_MB + 6 * s.l0 + 3);
      const V3 n1 = ld3(w, M.o_MB + 6 * s.l1), e1 = ld3(w, M.o_MB + 6 * s.l1 + 3);
      i0[k] = s.i0; i1[k] = s.i1;
      const float araw = w[M.o_ACT + M.ntact + s.mus];
      const float F = fminf(fmaxf(araw, 0.f), 1.f) * s.fmax;
      const V3 dv = x1 - x0;
      const float il = rsqrt_refined(dot(dv, dv));
      const V3 u = il * dv, f = F * u;
      const V3 g = (cross(x0, n0) - e0) - (cross(x1, n1) - e1);   // f0_bar - f1_bar
      const V3 ub = F * g;
      const V3 dvb = il * (ub - dot(u, ub) * u);
      b0[k] = cross(n0, f) - dvb;
      b1[k] = dvb - cross(n1, f);
      ab[k] = (araw > 0.f && araw < 1.f) ? dot(u, g) * s.fmax : 0.f;
    }
#pragma unroll
    for (int k = 0; k < SEG_GROUP; ++k) {
      if (s0 + k * nl < M.nseg) {
        plane_st(w, M.o_MF, n, i0[k], b0[k]);
        plane_st(w, M.o_MF, n, i1[k], b1[k]);
        w[M.o_SEGA + s0 + k * nl] = ab[k];
      }
    }
  }
  team_sync(nl);
  for (int mu = lane; mu < M.nm; mu += nl) {
    float sa = 0.f;
    for (int sg = __ldg(M.mus_seg_ptr + mu); sg < __ldg(M.mus_seg_ptr + mu + 1); ++sg) sa += w[M.o_SEGA + sg];
    w[M.o_ACTB + M.ntact + mu] += sa;
  }
  for (int c = lane; c < MSLOTS; c += nl) {
    V3 Pb = v3(0.f, 0.f, 0.f);
    M33 Q;
#pragma unroll
    for (int j = 0; j < 9; ++j) Q.m[j] = 0.f;
#pragma unroll 4
    for (int j = 0; j < M.mrows; ++j) {
      const V3 x = plane_ld(w, M.o_MX, n, MSLOTS * j + ((c + j) & (MSLOTS - 1))), xb = plane_ld(w, M.o_MF, n, MSLOTS * j + ((c + j) & (MSLOTS - 1)));
      Pb = Pb + xb;
      add_outer(Q, xb, x);
    }
    st3(w, M.o_MW + 12 * c, Pb);
    stm(w, M.o_MW + 12 * c + 3, Q);
  }
  team_sync(nl);
}

// One forward substep.  tau0: gear * action of this lane's DOF.  rec: where the
// substep's record (LaneRecord) goes, straight from registers (null: nowhere; a
// run-time test, so that one body serves both and the recomputing adjoint
// repeats the forward's rounding).
__device__ __forceinline__ void lane_substep(const DevModel& M, const SMem& w, const LaneConst& c, LaneState& s,
                                             float tau0, float* rec, int lane, int nl, int nm) {
  const LaneRecord ro = lane_record(M.L, M.nv, nm, M.root_free);
  // local pose and joint velocity in the link frame
  const bool root = M.root_free && lane == 0;
  LaneLink k;
  M33 R0;                                   // the free root's rotation, on every lane
  k.R = mul(c.jrot, axis_angle(c.axis, c.jt == J_REV ? s.q : 0.f));
  k.P = c.jpos;
  if (c.jt == J_PRIS) k.P = k.P + s.q * mul(k.R, c.axis);
  if (M.root_free) {
    R0 = quat_to_R(s.rq[3], s.rq[4], s.rq[5], s.rq[6]);
    if (root) {
      k.R = R0;
      k.P = v3(0.f, 0.f, 0.f);
    }
  }
  // world pose: T_i = T_anc T_i, the ancestor twice as far in every round, or the
  // parent, a level in every round (path_sums)
#ifdef SHAC_SPEC_ANC
#pragma unroll
  for (int r = 0; r < M.nround; ++r) {
    const unsigned a = (c.anc >> (6 * r)) & 63u;
    const int src = (int)(a & 31u);
    const bool take = a < 32u;
#else
  const int src = (int)(c.anc & 31u);
  for (int r = 1; r <= M.deepest; ++r) {
    const bool take = c.depth == r;
#endif
    M33 Rp;
#pragma unroll
    for (int j = 0; j < 9; ++j) Rp.m[j] = team_shfl(k.R.m[j], src, nl);
    const V3 Pp = team_shfl(k.P, src, nl);
    if (take) {
      k.P = Pp + mul(Rp, k.P);
      k.R = mul(Rp, k.R);
    }
  }
  // motion subspace, joint velocity, velocities and accelerations (qdd = 0)
  const V3 ax = mul(k.R, c.axis);
  V3 sw = c.jt == J_REV ? ax : v3(0.f, 0.f, 0.f);
  V3 sv = c.jt == J_REV ? cross(k.P, ax) : (c.jt == J_PRIS ? ax : v3(0.f, 0.f, 0.f));
  V3 uw = s.qd * sw, uv = s.qd * sv;
  if (M.root_free) {
    if (root) {
      uw = uv = v3(0.f, 0.f, 0.f);          // a DOF at a time, as lk_subspace_vel
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        uw = uw + s.rqd[j] * col(R0, j);
        uv = uv + s.rqd[3 + j] * col(R0, j);
      }
    }
    if (lane < 6) {                         // the root's columns (its origin is the reference point)
      const int d = lane % 3;
      const V3 e = d == 0 ? col(R0, 0) : (d == 1 ? col(R0, 1) : col(R0, 2));
      sw = lane < 3 ? e : v3(0.f, 0.f, 0.f);
      sv = lane < 3 ? v3(0.f, 0.f, 0.f) : e;
    }
  }
  k.Vw = uw; k.Vv = uv;
  path_sums(M, c, nl, k.Vw, k.Vv);
  k.aw = cross(k.Vw, uw);
  k.av = cross(k.Vw, uv) + cross(k.Vv, uw);
  k.av = k.av + c.base;
  path_sums(M, c, nl, k.aw, k.av);
  lane_local(M, c, c.on_root ? s.rq[2] : 0.f, k);
  const bool link = c.link >= 0;
  if (M.nseg > 0) {   // muscles: a segment spans two links, so the poses go through memory
    muscle_put_pose(M, w, c.link, k.R, k.P);
    team_sync(nl);
    muscle_forward(M, w, lane, nl);
    if (rec) {
      for (int j = lane; j < 3 * MSLOTS / 4 * M.mrows; j += nl) {
        const float4 v = lds4(w, M.o_MX + 4 * j);
        stg4(rec + ro.items + 4 * j, v.x, v.y, v.z, v.w);
      }
    }
    if (link) {
      V3 wn = v3(0.f, 0.f, 0.f), wf = wn;
      for (int s_ = c.ms0; s_ < c.ms1; ++s_) {
        wn = wn + ld3(w, M.o_MW + 12 * s_);
        wf = wf + ld3(w, M.o_MW + 12 * s_ + 3);
      }
      k.wn = k.wn + wn; k.wf = k.wf + wf;
      k.fn = k.fn - wn; k.ff = k.ff - wf;
    }
  }
  if (rec && link) {
    float* r = rec + 4 * c.link;
    const int fs = 4 * M.L;
    stg4(r, k.R.m[0], k.R.m[1], k.R.m[2], k.R.m[3]);
    stg4(r + fs, k.R.m[4], k.R.m[5], k.R.m[6], k.R.m[7]);
    stg4(r + 2 * fs, k.R.m[8], k.P.x, k.P.y, k.P.z);
    stg4(r + 3 * fs, __uint_as_float(k.contacts), k.si[1], k.si[2], k.si[3]);
    stg4(r + 4 * fs, k.si[4], k.si[5], k.si[6], k.si[7]);
    stg4(r + 5 * fs, k.si[8], k.si[9], k.Vw.x, k.Vw.y);
    stg4(r + 6 * fs, k.Vw.z, k.Vv.x, k.Vv.y, k.Vv.z);
    stg4(r + 7 * fs, k.wn.x, k.wn.y, k.wn.z, k.wf.x);
    *reinterpret_cast<float2*>(rec + ro.fx + 2 * c.link) = make_float2(k.wf.y, k.wf.z);
  }
  // composite inertias and total forces of this lane's DOF's link
  const int of = M.o_X + XB * M.L;
  float x[16];
#pragma unroll
  for (int j = 0; j < 10; ++j) x[j] = k.si[j];
  x[10] = k.fn.x; x[11] = k.fn.y; x[12] = k.fn.z;
  x[13] = k.ff.x; x[14] = k.ff.y; x[15] = k.ff.z;
  lane_sums(M, w, x, c, link, lane, nl);
  // right-hand side and the vectors Ic S
  float b = 0.f;
  V3 fn, ff;
  {
    const float ic[10] = {x[0], x[1], x[2], x[3], x[4], x[5], x[6], x[7], x[8], x[9]};
    si_mul<true>(ic, sw, sv, fn, ff);
    if (lane < nm) Dense<2>::put_vector(w, of, lane, sw, sv, fn, ff);
    if (c.own) {
      float t = tau0;
      if (c.jt == J_REV || c.jt == J_PRIS) {
        if (s.q < c.qlo) t += c.klim * (c.qlo - s.q);
        else if (s.q > c.qhi) t += c.klim * (c.qhi - s.q);
      }
      b = t - c.damp * s.qd - (dot(sw, v3(x[10], x[11], x[12])) + dot(sv, v3(x[13], x[14], x[15])));
    }
  }
  team_sync(nl);
  float idiag = 1.f, qdd = 0.f;
  const int ol = of + XF * nm;
  switch (nm) {
#define SHAC_CASE(N) case N: qdd = Dense<N>::solve(w, rec ? rec + ro.fac : nullptr, ro.rs, of, ol, sw, sv, fn, ff, b, c, lane, nl, idiag); break;
    SHAC_DENSE_CASES(SHAC_CASE)
#undef SHAC_CASE
    default: break;
  }
  if (!c.own) qdd = 0.f;
  if (rec) {
    if (c.own) stg4(rec + ro.dof + 4 * lane, s.qd, qdd, idiag, s.q);
    if (M.root_free) {
      float a[6];
#pragma unroll
      for (int j = 0; j < 6; ++j) a[j] = team_shfl(qdd, j, nl);
      if (lane == 0) {
        float* r = rec + ro.root;
        stg4(r, s.rq[0], s.rq[1], s.rq[2], s.rq[3]);
        stg4(r + 4, s.rq[4], s.rq[5], s.rq[6], s.rqd[0]);
        stg4(r + 8, s.rqd[1], s.rqd[2], s.rqd[3], s.rqd[4]);
        stg4(r + 12, s.rqd[5], a[0], a[1], a[2]);
        stg4(r + 16, a[3], a[4], a[5], 0.f);
      }
    }
  }
  // semi-implicit Euler: the DOF's velocity, then the position of its joint
  s.qd = two_sum(s.qd, M.h * qdd + s.qdc, s.qdc);
  if (c.jt == J_REV || c.jt == J_PRIS) {
    const float y = M.h * s.qd + (M.h * s.qdc + s.qc);
    s.q = two_sum(s.q, y, s.qc);
  }
  if (M.root_free) {
#pragma unroll
    for (int j = 0; j < 6; ++j) s.rqd[j] = team_shfl(s.qd, j, nl);
#pragma unroll
    for (int j = 0; j < 3; ++j) s.rqdc[j] = team_shfl(s.qdc, 3 + j, nl);
    root_integrate(M, R0, s);
  }
}

// Load and clear the state at a step start / write it to scratch (o_Q, o_QD).
__device__ __forceinline__ void lane_from_scratch(const DevModel& M, const SMem& w, const LaneConst& c, int lane,
                                                  LaneState& s) {
  const bool dof1 = c.jt == J_REV || c.jt == J_PRIS;
  s.q = dof1 ? w[M.o_Q + c.qi] : 0.f;
  s.qd = c.own ? w[M.o_QD + lane] : 0.f;
  s.qc = s.qdc = 0.f;
#pragma unroll
  for (int j = 0; j < 7; ++j) s.rq[j] = M.root_free ? w[M.o_Q + j] : 0.f;
#pragma unroll
  for (int j = 0; j < 6; ++j) s.rqd[j] = M.root_free ? w[M.o_QD + j] : 0.f;
#pragma unroll
  for (int j = 0; j < 3; ++j) s.rqc[j] = s.rqdc[j] = 0.f;
}
__device__ __forceinline__ void lane_to_scratch(const DevModel& M, const SMem& w, const LaneConst& c, int lane,
                                                const LaneState& s) {
  if (c.own) w[M.o_QD + lane] = s.qd;
  if (c.jt == J_REV || c.jt == J_PRIS) w[M.o_Q + c.qi] = s.q;
  if (M.root_free && lane == 0) {
#pragma unroll
    for (int j = 0; j < 7; ++j) w[M.o_Q + j] = s.rq[j];
  }
}

// Cotangents in registers: this lane's one-DOF coordinate, its DOF's velocity
// and action, and the free root's pose (on every lane).
struct LaneBars {
  float qb, qdb, actb;
  float rqb[7];
};

// Sums of four vectors along the path to the root (own value included), by doubling.
__device__ __forceinline__ void path_sums2(const DevModel& M, unsigned anc, int nl, V3& a, V3& b, V3& c, V3& d) {
#pragma unroll
  for (int r = 0; r < M.nround; ++r) {
    const unsigned s = (anc >> (6 * r)) & 63u;
    const int src = (int)(s & 31u);
    const V3 pa = team_shfl(a, src, nl), pb = team_shfl(b, src, nl);
    const V3 pc = team_shfl(c, src, nl), pd = team_shfl(d, src, nl);
    if (s < 32u) { a = a + pa; b = b + pb; c = c + pc; d = d + pd; }
  }
}

// One reverse substep in lane form: the record's copy in shared memory (o_R)
// holds the substep, g the cotangents of its end state; on return g holds those
// of its start state.  The next record is requested as soon as this one is in
// registers, so its copy runs under the rest of the pass.
__device__ __forceinline__ void lane_reverse(const DevModel& M, const SMem& w, const LaneConst& c, LaneBars& g,
                                             const float* rec, const float* next, int lane, int nl, int nm) {
  const LaneRecord ro = lane_record(M.L, M.nv, nm, M.root_free);
  const bool link = c.link >= 0, one = c.jt == J_REV || c.jt == J_PRIS;
  const bool root = M.root_free && lane == 0;
  const float h = M.h;
  record_wait();
  team_sync(nl);
  if (M.nseg > 0) record_request(w, M.o_MX, rec + ro.items, 3 * MSLOTS * M.mrows, lane, nl);
  // this lane's part of the record
  LaneLink k;
  float q = 0.f, qd = 0.f, qdd = 0.f, idiag = 1.f;
  {
    const int o = M.o_R + 4 * (link ? c.link : 0), fs = 4 * M.L;
    const float4 a0 = lds4(w, o), a1 = lds4(w, o + fs), a2 = lds4(w, o + 2 * fs), a3 = lds4(w, o + 3 * fs);
    const float4 a4 = lds4(w, o + 4 * fs), a5 = lds4(w, o + 5 * fs), a6 = lds4(w, o + 6 * fs), a7 = lds4(w, o + 7 * fs);
    const float2 a8 = *reinterpret_cast<const float2*>(&w[M.o_R + ro.fx + 2 * (link ? c.link : 0)]);
    k.R.m[0] = a0.x; k.R.m[1] = a0.y; k.R.m[2] = a0.z; k.R.m[3] = a0.w;
    k.R.m[4] = a1.x; k.R.m[5] = a1.y; k.R.m[6] = a1.z; k.R.m[7] = a1.w;
    k.R.m[8] = a2.x; k.P = v3(a2.y, a2.z, a2.w);
    k.contacts = __float_as_uint(a3.x); k.si[0] = c.mass; k.si[1] = a3.y; k.si[2] = a3.z; k.si[3] = a3.w;
    k.si[4] = a4.x; k.si[5] = a4.y; k.si[6] = a4.z; k.si[7] = a4.w;
    k.si[8] = a5.x; k.si[9] = a5.y; k.Vw = v3(a5.z, a5.w, a6.x); k.Vv = v3(a6.y, a6.z, a6.w);
    k.wn = v3(a7.x, a7.y, a7.z); k.wf = v3(a7.w, a8.x, a8.y);
    if (c.own) {
      const float4 d = lds4(w, M.o_R + ro.dof + 4 * lane);
      qd = d.x; qdd = d.y; idiag = d.z; q = d.w;
    }
  }
  // integrator: q' = q + h qd', qd' = qd + h qdd; the free root's pose on every lane
  if (one) g.qdb += h * g.qb;
  float rqd[6], rqdd[6], zroot = 0.f;
  M33 R0;
  float rx = 0.f, ry = 0.f, rz = 0.f, rw = 1.f;
  if (M.root_free) {
    const int o = M.o_R + ro.root;
    const float4 b0 = lds4(w, o), b1 = lds4(w, o + 4), b2 = lds4(w, o + 8), b3 = lds4(w, o + 12), b4 = lds4(w, o + 16);
    zroot = c.on_root ? b0.z : 0.f; rx = b0.w; ry = b1.x; rz = b1.y; rw = b1.z;
    rqd[0] = b1.w; rqd[1] = b2.x; rqd[2] = b2.y; rqd[3] = b2.z; rqd[4] = b2.w; rqd[5] = b3.x;
    rqdd[0] = b3.y; rqdd[1] = b3.z; rqdd[2] = b3.w; rqdd[3] = b4.x; rqdd[4] = b4.y; rqdd[5] = b4.z;
    R0 = quat_to_R(rx, ry, rz, rw);
    const V3 vb1 = v3(rqd[3], rqd[4], rqd[5]) + h * v3(rqdd[3], rqdd[4], rqdd[5]);
    const V3 om1 = v3(rqd[0], rqd[1], rqd[2]) + h * v3(rqdd[0], rqdd[1], rqdd[2]);
    const V3 pb = v3(g.rqb[0], g.rqb[1], g.rqb[2]);
    const V3 va = h * mulT(R0, pb);
    M33 B;
#pragma unroll
    for (int j = 0; j < 9; ++j) B.m[j] = 0.f;
    add_outer(B, h * pb, vb1);
    float xb = 0.f, yb = 0.f, zb = 0.f, wb = 0.f;
    quat_to_R_adj(rx, ry, rz, rw, B, xb, yb, zb, wb);
    const V3 u = v3(rx, ry, rz);
    const float hh = 0.5f * h;
    const V3 nu = u + hh * (rw * om1 + cross(u, om1));
    const float nw = rw - hh * dot(u, om1);
    const float inv = rsqrt_refined(dot(nu, nu) + nw * nw);
    const V3 qu1 = inv * nu;
    const float qw1 = inv * nw;
    const V3 qub = v3(g.rqb[3], g.rqb[4], g.rqb[5]);
    const float qwb = g.rqb[6];
    const float pr = dot(qu1, qub) + qw1 * qwb;
    const V3 nub = inv * (qub - pr * qu1);
    const float nwb = inv * (qwb - pr * qw1);
    const V3 ub = nub + hh * cross(om1, nub) - (hh * nwb) * om1;
    const float wbq = nwb + hh * dot(om1, nub);
    const V3 omb = hh * (rw * nub + cross(nub, u)) - (hh * nwb) * u;
    g.rqb[3] = ub.x + xb; g.rqb[4] = ub.y + yb; g.rqb[5] = ub.z + zb; g.rqb[6] = wbq + wb;
    const float add[6] = {omb.x, omb.y, omb.z, va.x, va.y, va.z};
#pragma unroll
    for (int j = 0; j < 6; ++j)
      if (lane == j) g.qdb += add[j];
  }
  // lambda = M^{-1} (h qd_bar)
  float lam = c.own ? h * g.qdb : 0.f;
  switch (nm) {
#define SHAC_CASE(N) case N: lam = Dense<N>::solve_record(w, M.o_R + ro.fac, ro.rs, M.nv, idiag, lam, lane, nl, make_iseq<N>{}); break;
    SHAC_DENSE_CASES(SHAC_CASE)
#undef SHAC_CASE
    default: break;
  }
  if (!c.own) lam = 0.f;
  team_sync(nl);   // every lane has read the record
  if (next) record_request(w, M.o_R, next, ro.items, lane, nl);
  // joint terms: velocity u, S qdd and -lambda S, then (A, F_bar) as path sums
  V3 sw = v3(0.f, 0.f, 0.f), sv = sw;
  const V3 ax = mul(k.R, c.axis);
  if (c.jt == J_REV) { sw = ax; sv = cross(k.P, ax); }
  if (c.jt == J_PRIS) sv = ax;
  V3 uw = qd * sw, uv = qd * sv;
  V3 nb = -lam * sw, fb = -lam * sv;
  k.aw = qdd * sw; k.av = qdd * sv;
  float rl[6];
  if (M.root_free) {
#pragma unroll
    for (int j = 0; j < 6; ++j) rl[j] = team_shfl(lam, j, nl);
    if (root) {
      uw = mul(R0, v3(rqd[0], rqd[1], rqd[2])); uv = mul(R0, v3(rqd[3], rqd[4], rqd[5]));
      k.aw = mul(R0, v3(rqdd[0], rqdd[1], rqdd[2])); k.av = mul(R0, v3(rqdd[3], rqdd[4], rqdd[5]));
      nb = -mul(R0, v3(rl[0], rl[1], rl[2])); fb = -mul(R0, v3(rl[3], rl[4], rl[5]));
    }
  }
  k.aw = k.aw + cross(k.Vw, uw);
  k.av = k.av + cross(k.Vw, uv) + cross(k.Vv, uw);
  k.av = k.av + c.base;
  path_sums2(M, c.anc, nl, k.aw, k.av, nb, fb);
  // the joint forces of this lane's DOF (dof_adj_force)
  if (c.own) {
    g.actb += lam * c.gear;
    if (one && (q < c.qlo || q > c.qhi)) g.qb -= lam * c.klim;
    g.qdb -= lam * c.damp;
  }
  // local force and its reverse (lk_adj_local)
  V3 bn, bf, abn, abf;
  si_mul(k.si, k.aw, k.av, k.fn, k.ff);
  si_mul(k.si, k.Vw, k.Vv, bn, bf);
  k.fn = k.fn + cross(k.Vw, bn) + cross(k.Vv, bf) - k.wn;
  k.ff = k.ff + cross(k.Vw, bf) - k.wf;
  si_mul(k.si, nb, fb, abn, abf);
  // total forces and A_bar
  float xs[12] = {k.fn.x, k.fn.y, k.fn.z, k.ff.x, k.ff.y, k.ff.z, abn.x, abn.y, abn.z, abf.x, abf.y, abf.z};
  lane_sums(M, w, xs, c, link, lane, nl);
  const V3 Fn = v3(xs[0], xs[1], xs[2]), Ff = v3(xs[3], xs[4], xs[5]);
  const V3 an = v3(xs[6], xs[7], xs[8]), af = v3(xs[9], xs[10], xs[11]);
  V3 hb = v3(0.f, 0.f, 0.f);
  M33 G;
#pragma unroll
  for (int j = 0; j < 9; ++j) G.m[j] = 0.f;
  si_adj(hb, G, k.aw, k.av, nb, fb);
  V3 vwb = cross(bn, nb) + cross(bf, fb);
  V3 vvb = cross(bf, nb);
  {
    const V3 bnb = cross(nb, k.Vw), bfb = cross(nb, k.Vv) + cross(fb, k.Vw);
    V3 t1, t2;
    si_mul(k.si, bnb, bfb, t1, t2);
    vwb = vwb + t1;
    vvb = vvb + t2;
    si_adj(hb, G, k.Vw, k.Vv, bnb, bfb);
  }
  V3 Pb;
  M33 Rb;
  {   // spatial inertia about the reference point -> pose cotangents (zero for a massless link)
    const float m = c.mass;
    const V3 cm = k.P + mul(k.R, c.com);
    const float trG = G.m[0] + G.m[4] + G.m[8];
    M33 Gs, Ic;
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
      for (int b = 0; b < 3; ++b) Gs.m[3 * a + b] = G.m[3 * a + b] + G.m[3 * b + a];
    Ic.m[0] = c.icom[0]; Ic.m[4] = c.icom[1]; Ic.m[8] = c.icom[2];
    Ic.m[1] = Ic.m[3] = c.icom[3]; Ic.m[2] = Ic.m[6] = c.icom[4]; Ic.m[5] = Ic.m[7] = c.icom[5];
    Pb = m * hb + m * (2.f * trG * cm - mul(Gs, cm));
    Rb = mul(mul(Gs, k.R), Ic);
    add_outer(Rb, Pb, c.com);
  }
  float depth = 0.f;   // cotangent of the root height through the contact depths
  V3 xl = c.cpos;
  float rad = c.crad;
  for (int e = c.c0; e < c.c1;) {
    const unsigned on = k.contacts >> (2 * (e - c.c0));
    if (on & 1u) {
      V3 x = k.P + mul(k.R, xl);
      x.z -= rad;
      const float dep = x.z + zroot;
      const V3 vp = k.Vv + cross(k.Vw, x);
      const float fn = (-M.ke + M.kd * vp.z) * dep;
      const bool slow = (on & 2u) != 0u;
      const float iv = slow ? 0.f : rsqrt_refined(sum2(vp.x, vp.x, vp.y, vp.y));   // 1 / |v_t|
      const float fmax = M.mu * fabsf(fn);
      const V3 neb = -nb;
      const V3 fbar = cross(neb, x) - fb;
      float fnb = fbar.z;
      V3 f, vpb = v3(0.f, 0.f, 0.f);
      f.z = fn;
      const float sc = slow ? M.kt : fmax * iv;
      f.x = -sc * vp.x; f.y = -sc * vp.y;
      vpb.x = -sc * fbar.x;
      vpb.y = -sc * fbar.y;
      if (!slow) {
        const float sb = -(fbar.x * vp.x + fbar.y * vp.y) * iv;
        fnb += sb * (fn >= 0.f ? M.mu : -M.mu);
        const float vtb = -sb * sc * iv;
        vpb.x += vtb * vp.x;
        vpb.y += vtb * vp.y;
      }
      V3 xb = cross(f, neb);
      const float db = fnb * (-M.ke + M.kd * vp.z);   // fn = (-ke + kd ddot) d, d = x.z + root height
      xb.z += db;
      depth += db;
      vpb.z += fnb * M.kd * dep;
      vwb = vwb + cross(x, vpb);
      vvb = vvb + vpb;
      xb = xb + cross(vpb, k.Vw);
      Pb = Pb + xb;
      add_outer(Rb, xb, xl);
    }
    if (++e < c.c1) {
      const int ci = __ldg(M.lc_idx + e);
      xl = cld3(M.item_pos + 3 * ci);
      rad = __ldg(M.crad + ci);
    }
  }
  V3 Pm = v3(0.f, 0.f, 0.f);   // muscles: their points' cotangents and moments sum x_bar x^T
  M33 Qm;
#pragma unroll
  for (int j = 0; j < 9; ++j) Qm.m[j] = 0.f;
  if (M.nseg > 0) {
    if (link) {
      st3(w, M.o_MB + 6 * c.link, nb);
      st3(w, M.o_MB + 6 * c.link + 3, fb);
    }
    if (next) asm volatile("cp.async.wait_group 1;\n" ::: "memory");   // the via points, requested first
    else record_wait();
    team_sync(nl);
    muscle_reverse(M, w, lane, nl);
    if (link) {
      for (int s_ = c.ms0; s_ < c.ms1; ++s_) {
        const int o = M.o_MW + 12 * s_;
        Pm = Pm + ld3(w, o);
#pragma unroll
        for (int j = 0; j < 9; ++j) Qm.m[j] += w[o + 3 + j];
      }
    }
  }
  // V_bar's own term with A_bar, and its sums
  vwb = vwb + cross(uw, an) + cross(uv, af);
  vvb = vvb + cross(uw, af);
  {
    float xv[6] = {vwb.x, vwb.y, vwb.z, vvb.x, vvb.y, vvb.z};
    lane_sums(M, w, xv, c, link, lane, nl);
    vwb = v3(xv[0], xv[1], xv[2]); vvb = v3(xv[3], xv[4], xv[5]);
  }
  // one-DOF joint terms and the moment Q of this link's own pose cotangents
  if (one) {
    const V3 tw = cross(an, k.Vw) + cross(af, k.Vv) + vwb, tv = cross(af, k.Vw) + vvb;
    g.qdb += dot(sw, tw) + dot(sv, tv);
    const V3 sbw = -lam * Fn + qdd * an + qd * tw, sbv = -lam * Ff + qdd * af + qd * tv;
    V3 ab;
    if (c.jt == J_REV) {
      ab = sbw + cross(sbv, k.P);
      Pb = Pb + cross(ax, sbv);
    } else {
      ab = sbv;
    }
    add_outer(Rb, ab, c.axis);
  }
  M33 Q = mulBT(Rb, k.R);
  add_outer(Q, Pb, k.P);
  if (M.nseg > 0) {
    Pb = Pb + Pm;
#pragma unroll
    for (int j = 0; j < 9; ++j) Q.m[j] += Qm.m[j];
  }
  float xq[13] = {Q.m[0], Q.m[1], Q.m[2], Q.m[3], Q.m[4], Q.m[5], Q.m[6], Q.m[7], Q.m[8], Pb.x, Pb.y, Pb.z, depth};
  lane_sums(M, w, xq, c, link, lane, nl);
  // q_bar: a revolute joint's is a . (axial(Q) - P x P_bar), a prismatic one's a . P_bar
  if (one) {
    const V3 axial = v3(xq[7] - xq[5], xq[2] - xq[6], xq[3] - xq[1]), pb = v3(xq[9], xq[10], xq[11]);
    g.qb += c.jt == J_REV ? dot(ax, axial - cross(k.P, pb)) : dot(ax, pb);
  }
  if (M.root_free) {   // the root's six DOFs and its quaternion: lanes 0 to 5 hold the root's sums, the others' values
                       // are not used
    const V3 w3 = v3(rqd[0], rqd[1], rqd[2]), v3_ = v3(rqd[3], rqd[4], rqd[5]);
    const V3 Vw0 = mul(R0, w3), Vv0 = mul(R0, v3_);
    const V3 tw = cross(an, Vw0) + cross(af, Vv0) + vwb, tv = cross(af, Vw0) + vvb;
    const V3 bw = mulT(R0, tw), bv = mulT(R0, tv);
    const float add[6] = {bw.x, bw.y, bw.z, bv.x, bv.y, bv.z};
#pragma unroll
    for (int j = 0; j < 6; ++j)
      if (lane == j) g.qdb += add[j];
    M33 T;
#pragma unroll
    for (int j = 0; j < 9; ++j) T.m[j] = xq[j];
    T = mul(T, R0);   // the root origin is the reference point (P = 0)
    add_outer(T, Fn, v3(-rl[0], -rl[1], -rl[2]));
    add_outer(T, an, v3(rqdd[0], rqdd[1], rqdd[2]));
    add_outer(T, tw, w3);
    add_outer(T, Ff, v3(-rl[3], -rl[4], -rl[5]));
    add_outer(T, af, v3(rqdd[3], rqdd[4], rqdd[5]));
    add_outer(T, tv, v3_);
    quat_to_R_adj(rx, ry, rz, rw, T, g.rqb[3], g.rqb[4], g.rqb[5], g.rqb[6]);
    g.rqb[2] += xq[12];
  }
}

// Cotangents from and to scratch (o_QB, o_QDB; the step's reward adjoint runs there).
__device__ __forceinline__ void bars_from_scratch(const DevModel& M, const SMem& w, const LaneConst& c, int lane,
                                                  LaneBars& g) {
  g.qb = c.jt == J_REV || c.jt == J_PRIS ? w[M.o_QB + c.qi] : 0.f;
  g.qdb = c.own ? w[M.o_QDB + lane] : 0.f;
  g.actb = c.own && c.act >= 0 ? w[M.o_ACTB + c.act] : 0.f;
#pragma unroll
  for (int j = 0; j < 7; ++j) g.rqb[j] = M.root_free ? w[M.o_QB + j] : 0.f;
}
__device__ __forceinline__ void bars_to_scratch(const DevModel& M, const SMem& w, const LaneConst& c, int lane,
                                                const LaneBars& g) {
  if (c.jt == J_REV || c.jt == J_PRIS) w[M.o_QB + c.qi] = g.qb;
  if (c.own) w[M.o_QDB + lane] = g.qdb;
  if (c.own && c.act >= 0) w[M.o_ACTB + c.act] = g.actb;
  if (M.root_free && lane == 0) {
#pragma unroll
    for (int j = 0; j < 7; ++j) w[M.o_QB + j] = g.rqb[j];
  }
}

}  // namespace shac
