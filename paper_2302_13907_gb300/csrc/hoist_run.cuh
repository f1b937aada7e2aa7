// Half step marched along theta: one thread owns four z cells of a row and walks
// a run of theta planes, with the loads of the next plane in flight (as stored, in
// registers) while it computes the present one.
//
// What bounds the tile-by-tile kernels on the lean cells is latency: a thread
// loads, waits and computes once, 24 warps an SM do not cover it, and in 16-bit
// storage the instructions (590 a warp and plane for the velocities) take longer
// than the bytes.  The march keeps 13 loads a thread in flight throughout, reads
// the theta neighbours once (they are the present values of the plane before or
// after), and with 32-bit offsets and the material table in shared memory takes
// 420.  196 x 64 x 1056 cells, BF16: 217 us a step tile by tile, 193 here;
// FP16-SR 342 and 285 (288 with its layer in whole tiles, z_sum); FP32 on 136 x
// 32 x 3104 cells 294 and 269.  Its interior
// launches reach 66 and 57 % of the DRAM throughput (53 and 46 % tile by tile); what
// is left is issue slots (57 to 61 % busy) and the start of every run.
//
// The radial layer (RAD) takes the same march in FP32 with its memory variables
// loaded ahead too, two blocks an SM: 212 x 64 x 8224 cells, the launches beside
// the one-pass step take 410 us of a step, tile by tile 455.  On 136 x 32 x 3104
// cells it is the slower one (260 us a step against 247): too few runs to fill two
// blocks an SM.  The tuner measures both.
#pragma once

#include "hoist_body.cuh"

namespace cwell {
namespace {

// Loads of the next plane: volatile, so that the compiler leaves them ahead of
// the present plane's arithmetic instead of sinking them to their use.
__device__ __forceinline__ float4 ld_ahead4(const float *p) {
  float4 v;
  asm volatile("ld.global.nc.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p));
  return v;
}
__device__ __forceinline__ uint2 ld_ahead8(const void *p) {
  uint2 v;
  asm volatile("ld.global.nc.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "l"(p));
  return v;
}
__device__ __forceinline__ unsigned ld_ahead2(const void *p) {
  unsigned short v;
  asm volatile("ld.global.nc.u16 %0, [%1];" : "=h"(v) : "l"(p));
  return v;
}

// four values of a row, and one, as stored
template <typename T>
struct Raw4 {
  uint2 v;
  __device__ __forceinline__ void ld(const T *p) { v = ld_ahead8(p); }
  __device__ __forceinline__ void zero() { v = make_uint2(0u, 0u); }
  __device__ __forceinline__ void get(float (&d)[4]) const {
    const float2 a = u32_to_f2(v.x, (const T *)nullptr), b = u32_to_f2(v.y, (const T *)nullptr);
    d[0] = a.x, d[1] = a.y, d[2] = b.x, d[3] = b.y;
  }
};
template <>
struct Raw4<float> {
  float4 v;
  __device__ __forceinline__ void ld(const float *p) { v = ld_ahead4(p); }
  __device__ __forceinline__ void zero() { v = make_float4(0.f, 0.f, 0.f, 0.f); }
  __device__ __forceinline__ void get(float (&d)[4]) const { d[0] = v.x, d[1] = v.y, d[2] = v.z, d[3] = v.w; }
};
template <typename T>
struct Raw1 {
  unsigned v;
  __device__ __forceinline__ void ld(const T *p) { v = ld_ahead2(p); }
  __device__ __forceinline__ void zero() { v = 0u; }
  __device__ __forceinline__ float get() const { return u32_to_f2(v, (const T *)nullptr).x; }
};
template <>
struct Raw1<float> {
  float v;
  __device__ __forceinline__ void ld(const float *p) { asm volatile("ld.global.nc.f32 %0, [%1];" : "=f"(v) : "l"(p)); }
  __device__ __forceinline__ void zero() { v = 0.f; }
  __device__ __forceinline__ float get() const { return v; }
};
// four material IDs and the one after them
struct RawId {
  uint2 v;
  unsigned e;
  __device__ __forceinline__ void ld(const uint16_t *p) { v = ld_ahead8(p), e = ld_ahead2(p + 4); }
  __device__ __forceinline__ void zero() { v = make_uint2(0u, 0u), e = 0; }
  __device__ __forceinline__ unsigned id(int q) const {
    return q == 4 ? e : q == 0 ? v.x & 0xffffu : q == 1 ? v.x >> 16 : q == 2 ? v.y & 0xffffu : v.y >> 16;
  }
};

// Material table of a block in shared memory (in L1 its words lose their lines to
// the fields' streams: 203 us a BF16 step against 193): {rho} (velocities) or {1/mu} and
// {lambda, lambda + 2 mu} (stresses)
constexpr int RUN_MATS = 2048;  // larger tables keep the kernels that look up in L1
inline int run_table_bytes(int n_mat, bool vel) { return n_mat * (vel ? 4 : 12); }
template <bool VEL>
__device__ __forceinline__ void run_table(const KParams &p, float2 *tab) {
  float *t1 = VEL ? (float *)tab : (float *)(tab + p.n_mat);
  for (int m = threadIdx.y * 32 + threadIdx.x; m < p.n_mat; m += 128) {
    t1[m] = __ldg((VEL ? p.m_rho : p.m_imu) + m);
    if (!VEL) tab[m] = __ldg(p.m_lam + m);
  }
  __syncthreads();
}

// element at a 32-bit byte offset from a field's base (launch: the arrays are
// below 4 GB), so that the base stays in uniform registers and an access costs
// no 64-bit address arithmetic of its own
template <typename T>
__device__ __forceinline__ T *at(T *base, unsigned o) {
  return (T *)((std::conditional_t<std::is_const<T>::value, const char, char> *)base + o);
}

// memory variables of the radial layer of one plane and component group
struct RadPlane {
  float4 v[6];
};
struct NoRad {};
// memory variables are rewritten by the thread that reads them: not the read-only path
__device__ __forceinline__ float4 ld_own4(const float *p) {
  float4 v;
  asm volatile("ld.global.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p));
  return v;
}
// a half step's access to them: load_rad (next plane's, ahead), take_rad,
// rad (recursion of one value), put_rad
#define RUN_RADIAL(R0, Q0)                                                                             \
  auto load_rad = [&](unsigned o) {                                                                    \
    if constexpr (RAD) {                                                                               \
      if (rp) {                                                                                        \
        _Pragma("unroll") for (int u = 0; u < 6; u++)                                                  \
            nr_.v[u] = ld_own4(at((const float *)p.psr[u < 3 ? R0 + u : Q0 + u - 3], o));              \
      }                                                                                                \
    }                                                                                                  \
  };                                                                                                   \
  auto take_rad = [&](float(&psi)[RAD ? 6 : 1][4]) {                                                   \
    if constexpr (RAD) {                                                                               \
      _Pragma("unroll") for (int u = 0; u < 6; u++) {                                                  \
        psi[u][0] = nr_.v[u].x, psi[u][1] = nr_.v[u].y, psi[u][2] = nr_.v[u].z, psi[u][3] = nr_.v[u].w; \
      }                                                                                                \
    }                                                                                                  \
  };                                                                                                   \
  auto rad = [&](float(&psi)[RAD ? 6 : 1][4], int u, int e, float a, float b, float D) {               \
    if constexpr (RAD) return stretch_reg(psi[u][e], a, b, D);                                         \
    else return D;                                                                                     \
  };                                                                                                   \
  auto put_rad = [&](float(&psi)[RAD ? 6 : 1][4], unsigned o) {                                        \
    if constexpr (RAD) {                                                                               \
      if (rp) {                                                                                        \
        _Pragma("unroll") for (int u = 0; u < 6; u++) stv(at(p.psr[u < 3 ? R0 + u : Q0 + u - 3], o), psi[u]); \
      }                                                                                                \
    }                                                                                                  \
  };

// what a plane of the velocity march loads: plane j, and of plane j + 1 the
// sigma_phi and IDs v_phi needs
template <typename T>
struct VelPlane {
  Raw4<T> srr, srp, srz, spz, szz, msrr, mspp, psrp, psrz, vr, vp, vz, sppn;
  RawId idm, idn;
  Raw1<T> szz4, srzm, spzm;
};

// RAD: rows i >= nr carry the radial memory variables (read, updated and written
// with the plane; recursion as in stretch()); fo: the set written (p.f: in place)
template <typename T, bool RAD>
__device__ __forceinline__ void vel_run(const KParams &p, void *const *fo, const float *rho_of, int j, const int J,
                                        const int i, const int k0) {
  constexpr unsigned B = sizeof(T), IB = B / 2;  // bytes of a value; o / IB: the offset in the IDs
  const unsigned pl = (unsigned)(p.plane * B), row = (unsigned)p.NZp * B, end = p.nth * pl;
  const T *srr = (const T *)p.f[F_SRR], *spp = (const T *)p.f[F_SPP], *szz = (const T *)p.f[F_SZZ];
  const T *srp = (const T *)p.f[F_SRP], *spz = (const T *)p.f[F_SPZ], *srz = (const T *)p.f[F_SRZ];
  const T *vr = (const T *)p.f[F_VR], *vp = (const T *)p.f[F_VP], *vz = (const T *)p.f[F_VZ];
  const bool im = i >= 1, ip = i + 1 < p.NR, km = k0 > 0;
  const float inv_ri = __ldg(p.inv_ri + i), inv_rh = __ldg(p.inv_rh + i);
  const float dtv = p.dtv, idr = p.inv_dr, idz = p.inv_dz, idth = p.inv_dth;
  const bool rp = RAD && i >= p.nr;
  float4 abr = z4(), abq = z4();
  if (rp) abr = __ldg(p.ab_r + i), abq = __ldg(p.ab_q + i);
  // byte offset of the plane in a memory variable, and from plane to plane
  const unsigned rpl = RAD ? (unsigned)(p.pml_r * p.NZp) * 4u : 0u;
  unsigned cr = rp ? j * rpl + ((unsigned)(i - p.nr) * p.NZp + k0) * 4u : 0u;
  std::conditional_t<RAD, RadPlane, NoRad> nr_;
  RUN_RADIAL(R_VR, Q_VR)
  int n = 0;
  if constexpr (std::is_same<T, half_sr>::value) n = *p.step + p.step_off;

  auto load = [&](VelPlane<T> &b, unsigned c, unsigned cn) {
    b.srr.ld(at(srr, c)), b.srp.ld(at(srp, c)), b.srz.ld(at(srz, c)), b.spz.ld(at(spz, c)), b.szz.ld(at(szz, c));
    b.vr.ld(at(vr, c)), b.vp.ld(at(vp, c)), b.vz.ld(at(vz, c));
    b.sppn.ld(at(spp, cn)), b.idn.ld(at(p.id, cn / IB));
    b.szz4.ld(at(szz, c) + 4);
    if (km) b.srzm.ld(at(srz, c) - 1), b.spzm.ld(at(spz, c) - 1);
    else b.srzm.zero(), b.spzm.zero();
    if (im) b.msrr.ld(at(srr, c - row)), b.mspp.ld(at(spp, c - row)), b.idm.ld(at(p.id, (c - row) / IB));
    else b.msrr.zero(), b.mspp.zero(), b.idm.zero();
    if (ip) b.psrp.ld(at(srp, c + row)), b.psrz.ld(at(srz, c + row));
    else b.psrp.zero(), b.psrz.zero();
  };

  unsigned c = j * pl + i * row + k0 * B, cn = end - c > pl ? c + pl : c + pl - end;
  VelPlane<T> nx;
  load_rad(cr);
  // of plane j - 1: sigma_rphi, sigma_phiz; of plane j: sigma_phi, rho
  float srp0[4], spz0[4], spp_[4], rho[5];
  {
    const unsigned cm = c >= pl ? c - pl : c - pl + end;
    Raw4<T> a, b, d;
    RawId u;
    a.ld(at(srp, cm)), b.ld(at(spz, cm)), d.ld(at(spp, c)), u.ld(at(p.id, c / IB));
    load(nx, c, cn);
    a.get(srp0), b.get(spz0), d.get(spp_);
#pragma unroll
    for (int e = 0; e < 5; e++) rho[e] = rho_of[u.id(e)];
  }
#pragma unroll 1
  for (int l = 0; l < J; l++) {
    float a_srr[4], a_srp[4], a_srz[4], a_spz[4], a_szz[4], m_srr[4], m_spp[4], p_srp[4], p_srz[4], n_spp[4];
    float o_r[4], o_p[4], o_z[4], rho_m[4], rho_n[5];
    nx.srr.get(a_srr), nx.srp.get(a_srp), nx.srz.get(a_srz), nx.spz.get(a_spz), nx.szz.get(a_szz);
    nx.msrr.get(m_srr), nx.mspp.get(m_spp), nx.psrp.get(p_srp), nx.psrz.get(p_srz), nx.sppn.get(n_spp);
    nx.vr.get(o_r), nx.vp.get(o_p), nx.vz.get(o_z);
    const float szz4 = nx.szz4.get(), srzm = nx.srzm.get(), spzm = nx.spzm.get();
#pragma unroll
    for (int e = 0; e < 4; e++) rho_m[e] = rho_of[nx.idm.id(e)];
#pragma unroll
    for (int e = 0; e < 5; e++) rho_n[e] = rho_of[nx.idn.id(e)];
    const unsigned cw = c, crw = cr;
    c = cn;
    cn = end - c > pl ? c + pl : c + pl - end;
    float psi[RAD ? 6 : 1][4];
    take_rad(psi);
    if (l + 1 < J) {
      load(nx, c, cn);
      cr = c < cw ? cr - (p.nth - 1) * rpl : cr + rpl;
      load_rad(cr);
    }
#pragma unroll
    for (int e = 0; e < 4; e++) {
      if (im) {
        const float q = 0.5f * (a_srr[e] + m_srr[e]) - 0.5f * (spp_[e] + m_spp[e]) + (a_srp[e] - srp0[e]) * idth;
        const float dr = a_srr[e] - m_srr[e], dz = a_srz[e] - (e ? a_srz[e - 1] : srzm);
        const float t = rp ? rad(psi, 0, e, abr.x, abr.y, dr * idr) + rad(psi, 3, e, abq.x, abq.y, q * inv_ri)
                           : mul_add2(dr, idr, q, inv_ri);
        o_r[e] += vel_coef(dtv, rho_m[e] + rho[e]) * __fmaf_rn(dz, idz, t);
      }
      {
        const float q = (p_srp[e] + a_srp[e]) + (n_spp[e] - spp_[e]) * idth;
        const float dr = p_srp[e] - a_srp[e], dz = a_spz[e] - (e ? a_spz[e - 1] : spzm);
        const float t = rp ? rad(psi, 1, e, abr.z, abr.w, dr * idr) + rad(psi, 4, e, abq.z, abq.w, q * inv_rh)
                           : mul_add2(dr, idr, q, inv_rh);
        o_p[e] += vel_coef(dtv, rho[e] + rho_n[e]) * __fmaf_rn(dz, idz, t);
      }
      {
        const float q = mul_add2(0.5f, p_srz[e] + a_srz[e], a_spz[e] - spz0[e], idth);
        const float dr = p_srz[e] - a_srz[e], dz = (e < 3 ? a_szz[e + 1] : szz4) - a_szz[e];
        const float t = rp ? rad(psi, 2, e, abr.z, abr.w, dr * idr) + rad(psi, 5, e, abq.z, abq.w, q * inv_rh)
                           : mul_add2(dr, idr, q, inv_rh);
        o_z[e] += vel_coef(dtv, rho[e] + rho[e + 1]) * __fmaf_rn(dz, idz, t);
      }
    }
    SrKey sk{0ull, 0ull, 0};
    if constexpr (std::is_same<T, half_sr>::value) {
      sk = sr_key(p, n, j, i, k0);
      j = j == p.nth - 1 ? 0 : j + 1;
    }
    if (im) st_field<T, 4, false>(at((T *)fo[F_VR], cw), o_r, sk, F_VR);
    st_field<T, 4, false>(at((T *)fo[F_VP], cw), o_p, sk, F_VP);
    st_field<T, 4, false>(at((T *)fo[F_VZ], cw), o_z, sk, F_VZ);
    put_rad(psi, crw);
#pragma unroll
    for (int e = 0; e < 4; e++) srp0[e] = a_srp[e], spz0[e] = a_spz[e], spp_[e] = n_spp[e];
#pragma unroll
    for (int e = 0; e < 5; e++) rho[e] = rho_n[e];
  }
}

// what a plane of the stress march loads: plane j, and of plane j + 1 the v_r,
// v_z and IDs the shear strains need
template <typename T>
struct StrPlane {
  Raw4<T> vp, pvr, mvp, mvz, rr, pp, zz, rp, pz, rz, vrn, vzn;
  RawId idn, idmn;
  Raw1<T> vr4, vp4, vzm;
};

template <typename T, bool RAD>
__device__ __forceinline__ void str_run(const KParams &p, void *const *fo, const float2 *lam_of, const float *imu_of, int j,
                                        const int J, const int i, const int k0) {
  constexpr unsigned B = sizeof(T), IB = B / 2;  // bytes of a value; o / IB: the offset in the IDs
  const unsigned pl = (unsigned)(p.plane * B), row = (unsigned)p.NZp * B, end = p.nth * pl;
  const T *vr = (const T *)fo[F_VR], *vp = (const T *)fo[F_VP], *vz = (const T *)fo[F_VZ];
  const T *srr = (const T *)p.f[F_SRR], *spp = (const T *)p.f[F_SPP], *szz = (const T *)p.f[F_SZZ];
  const T *srp = (const T *)p.f[F_SRP], *spz = (const T *)p.f[F_SPZ], *srz = (const T *)p.f[F_SRZ];
  const bool im = i >= 1, ip = i + 1 < p.NR, km = k0 > 0;
  const float inv_ri = __ldg(p.inv_ri + i), inv_rh = __ldg(p.inv_rh + i);
  const float dts = p.dts, idr = p.inv_dr, idz = p.inv_dz, idth = p.inv_dth;
  const bool rp = RAD && i >= p.nr;
  float4 abr = z4(), abq = z4();
  if (rp) abr = __ldg(p.ab_r + i), abq = __ldg(p.ab_q + i);
  const unsigned rpl = RAD ? (unsigned)(p.pml_r * p.NZp) * 4u : 0u;
  unsigned cr = rp ? j * rpl + ((unsigned)(i - p.nr) * p.NZp + k0) * 4u : 0u;
  std::conditional_t<RAD, RadPlane, NoRad> nr_;
  RUN_RADIAL(R_ERR, Q_EPP)
  const bool src_cell = i == p.src_i && p.src_k >= k0 && p.src_k < k0 + 4;
  int n = 0;
  if constexpr (std::is_same<T, half_sr>::value) n = *p.step + p.step_off;

  auto load = [&](StrPlane<T> &b, unsigned c, unsigned cn) {
    b.vp.ld(at(vp, c)), b.vrn.ld(at(vr, cn)), b.vzn.ld(at(vz, cn)), b.idn.ld(at(p.id, cn / IB));
    b.rr.ld(at(srr, c)), b.pp.ld(at(spp, c)), b.zz.ld(at(szz, c)), b.rp.ld(at(srp, c)), b.pz.ld(at(spz, c)), b.rz.ld(at(srz, c));
    b.vr4.ld(at(vr, c) + 4), b.vp4.ld(at(vp, c) + 4);
    if (km) b.vzm.ld(at(vz, c) - 1);
    else b.vzm.zero();
    if (im) b.mvp.ld(at(vp, c - row)), b.mvz.ld(at(vz, c - row)), b.idmn.ld(at(p.id, (cn - row) / IB));
    else b.mvp.zero(), b.mvz.zero(), b.idmn.zero();
    if (ip) b.pvr.ld(at(vr, c + row));
    else b.pvr.zero();
  };

  unsigned c = j * pl + i * row + k0 * B, cn = end - c > pl ? c + pl : c + pl - end;
  StrPlane<T> nx;
  load_rad(cr);
  // of plane j - 1: v_phi; of plane j: v_r, v_z, IDs, 1/mu of rows i and i - 1
  float vp0[4], vr0[4], vz0[4], imu[5], imm[5];
  RawId u;
  {
    const unsigned cm = c >= pl ? c - pl : c - pl + end;
    Raw4<T> a, b, d;
    RawId m;
    a.ld(at(vp, cm)), b.ld(at(vr, c)), d.ld(at(vz, c)), u.ld(at(p.id, c / IB));
    if (im) m.ld(at(p.id, (c - row) / IB));
    else m.zero();
    load(nx, c, cn);
    a.get(vp0), b.get(vr0), d.get(vz0);
#pragma unroll
    for (int e = 0; e < 5; e++) {
      imu[e] = imu_of[u.id(e)];
      imm[e] = imu_of[m.id(e)];
    }
  }
#pragma unroll 1
  for (int l = 0; l < J; l++) {
    float a_vp[4], n_vr[4], n_vz[4], p_vr[4], m_vp[4], m_vz[4], orr[4], opp[4], ozz[4], orp[4], opz[4], orz[4];
    float imn[5], immn[5];
    float2 lam[4];
    nx.vp.get(a_vp), nx.vrn.get(n_vr), nx.vzn.get(n_vz), nx.pvr.get(p_vr), nx.mvp.get(m_vp), nx.mvz.get(m_vz);
    nx.rr.get(orr), nx.pp.get(opp), nx.zz.get(ozz), nx.rp.get(orp), nx.pz.get(opz), nx.rz.get(orz);
    const float vr4 = nx.vr4.get(), vp4 = nx.vp4.get(), vzm = nx.vzm.get();
#pragma unroll
    for (int e = 0; e < 5; e++) {
      imn[e] = imu_of[nx.idn.id(e)];
      immn[e] = imu_of[nx.idmn.id(e)];
      if (e < 4) lam[e] = lam_of[u.id(e)];
    }
    u = nx.idn;
    const unsigned cw = c, crw = cr;
    c = cn;
    cn = end - c > pl ? c + pl : c + pl - end;
    float psi[RAD ? 6 : 1][4];
    take_rad(psi);
    if (l + 1 < J) {
      load(nx, c, cn);
      cr = c < cw ? cr - (p.nth - 1) * rpl : cr + rpl;
      load_rad(cr);
    }
    float src[4] = {0.f, 0.f, 0.f, 0.f};
    if (src_cell && (p.src_j < 0 || p.src_j == j)) {
      const int m = *p.step + p.step_off;
      const float w = m < p.n_wav ? __ldg(p.wav + m) : 0.f;
#pragma unroll
      for (int e = 0; e < 4; e++)
        if (k0 + e == p.src_k) src[e] = w;
    }
#pragma unroll
    for (int e = 0; e < 4; e++) {
      float err = __fmul_rn(p_vr[e] - vr0[e], idr);
      float epp = __fmul_rn(mul_add2(0.5f, vr0[e] + p_vr[e], a_vp[e] - vp0[e], idth), inv_rh);
      const float ezz = __fmul_rn(vz0[e] - (e ? vz0[e - 1] : vzm), idz);
      if (rp) err = rad(psi, 0, e, abr.z, abr.w, err), epp = rad(psi, 3, e, abq.z, abq.w, epp);
      const float l = lam[e].x, l2m = lam[e].y;
      orr[e] = __fadd_rn(orr[e], __fmaf_rn(dts, mul_add2(l2m, err, l, __fadd_rn(epp, ezz)), src[e]));
      opp[e] = __fadd_rn(opp[e], __fmaf_rn(dts, mul_add2(l, __fadd_rn(err, ezz), l2m, epp), src[e]));
      ozz[e] = __fadd_rn(ozz[e], __fmaf_rn(dts, mul_add2(l2m, ezz, l, __fadd_rn(err, epp)), src[e]));
      if (im) {
        {
          const float q = mul_add2(n_vr[e] - vr0[e], idth, -0.5f, a_vp[e] + m_vp[e]), dr = a_vp[e] - m_vp[e];
          const float t = rp ? rad(psi, 1, e, abr.x, abr.y, dr * idr) + rad(psi, 4, e, abq.x, abq.y, q * inv_ri)
                             : mul_add2(dr, idr, q, inv_ri);
          const float mu = mu_harm(imm[e] + imu[e] + immn[e] + imn[e]);
          orp[e] += dts * mu * t;
        }
        const float dz = (e < 3 ? vr0[e + 1] : vr4) - vr0[e], dr = vz0[e] - m_vz[e];
        const float t = rp ? dz * idz + rad(psi, 2, e, abr.x, abr.y, dr * idr) : mul_add2(dz, idz, dr, idr);
        const float mu = mu_harm(imm[e] + imu[e] + imm[e + 1] + imu[e + 1]);
        orz[e] += dts * mu * t;
      }
      float q = __fmul_rn(__fmul_rn(n_vz[e] - vz0[e], idth), inv_rh);
      if (rp) q = rad(psi, 5, e, abq.z, abq.w, q);
      const float t = __fmaf_rn((e < 3 ? a_vp[e + 1] : vp4) - a_vp[e], idz, q);
      const float mu = mu_harm(imu[e] + imn[e] + imu[e + 1] + imn[e + 1]);
      opz[e] += dts * mu * t;
    }
    SrKey sk{0ull, 0ull, 0};
    if constexpr (std::is_same<T, half_sr>::value) sk = sr_key(p, n, j, i, k0);
    j = j == p.nth - 1 ? 0 : j + 1;
    st_field<T, 4, false>(at((T *)fo[F_SRR], cw), orr, sk, F_SRR);
    st_field<T, 4, false>(at((T *)fo[F_SPP], cw), opp, sk, F_SPP);
    st_field<T, 4, false>(at((T *)fo[F_SZZ], cw), ozz, sk, F_SZZ);
    st_field<T, 4, false>(at((T *)fo[F_SPZ], cw), opz, sk, F_SPZ);
    if (im) {
      st_field<T, 4, false>(at((T *)fo[F_SRP], cw), orp, sk, F_SRP);
      st_field<T, 4, false>(at((T *)fo[F_SRZ], cw), orz, sk, F_SRZ);
    }
    put_rad(psi, crw);
#pragma unroll
    for (int e = 0; e < 4; e++) vp0[e] = a_vp[e], vr0[e] = n_vr[e], vz0[e] = n_vz[e];
#pragma unroll
    for (int e = 0; e < 5; e++) imu[e] = imn[e], imm[e] = immn[e];
  }
}

}  // namespace
}  // namespace cwell
