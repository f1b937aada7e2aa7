// One-pass step (tile codes 40xx, FP32): both halves of the leapfrog step for
// the lean cells (no PML memory variable) in one kernel, double-buffered, so
// that every field crosses memory once per step: 74 bytes per cell-update
// (nine fields read, nine written, the ID) against 112 for a velocity and a
// stress launch.
//
// A block owns R = 9 rows x 120 z cells and marches theta.  One warp per row
// (plus one row below and one above, whose velocities it recomputes), four z
// cells per lane; lanes 0 and 31 are the z halo.  Each theta plane of the six
// stresses and the IDs (R + 2 rows of 512 / 256 bytes) comes into a ring of
// four shared-memory slots by TMA (one cp.async.bulk.tensor box per array,
// mbarrier completion), issued by a producer warp while two planes are in use
// (one untiled bulk copy per row, 77 a plane, kept the ring waiting: 2.7 us a
// plane with or without the stores); the old velocities, which only their own
// cell reads, are loaded into registers one plane ahead.  The material table sits in
// shared memory ({rho, 1/mu, lambda, lambda + 2 mu}, one 16-byte word per ID).
// At march index j the warps
//   A. compute v_r and v_z of plane j and v_phi of plane j - 1 from the stress
//      planes j - 1 and j, write the owned ones and put all three in shared
//      memory (three rotating buffers, so that one barrier per plane suffices);
//   B. compute all six stresses of plane j - 1 from the velocities of planes
//      j - 2 (v_phi, a register), j - 1 and j, and write them.
// r neighbours come from shared memory, z neighbours by shuffle, theta
// neighbours from the ring slot or registers of the plane before; material
// values of a plane are looked up once and kept for the next one.
//
// A run of J planes reads J + 2 and recomputes one plane of v_r, v_z and
// v_phi each.  Whole rounds of one item per SM take theta in d runs (code 4000
// + 100 m + d), the tiles left over in more and shorter ones; one block per SM
// walks the (tile, run) items, its ring running on from item to item (m even),
// or every item has its own block (m odd: no fixed share of the items per SM,
// but a pipeline fill per item).  The tuner times both with theta in one run (d = 1);
// other d are for opts.tile.
//
// Measured: 196 x 64 x 8224 cells 1.27 ms a launch (74 bytes a cell: 5.5 TB/s)
// where the split halves take 0.83 + 1.03 ms on the same cells; the step with its
// edge launches 1.68 ms (1.73 before the radial layer was marched) against 2.15.  136 x 32 x 3104: 0.26 ms against 0.29.
//
// What bounds it: DRAM.  Halo rows and columns (11 x 128 read for 9 x 120
// owned) are shared with blocks that run at the same time and come from L2.
// The cells with memory variables (radial PML, z ends) and the one-cell rim the
// march may not recompute them from keep the split bodies, out of place:
// their velocities beside this kernel, their stresses after it.
//
// Every mbarrier wait is bounded; a wait that gives up sets bit 1 of the
// status word, the row warps leave together, and the producer first waits
// (bounded) for the copies it has issued.
#include "hoist_body.cuh"
#include "tma_util.cuh"

namespace cwell {
namespace {

constexpr int PZ = 120;   // owned z cells per tile
constexpr int PW = 128;   // staged z cells per row
constexpr int PSLOT = 4;  // ring slots
enum { S_SRR = 0, S_SPP, S_SZZ, S_SRP, S_SPZ, S_SRZ };

template <int R>
struct PassSmem {
  static constexpr int ROWS = R + 2, WARPS = ROWS + 1;       // row warps and the producer
  static constexpr int FIELD = ROWS * PW;                    // floats
  static constexpr int SLOT_BYTES = 6 * FIELD * 4 + FIELD * 2;
  static constexpr int EXCH = 3 * FIELD;                     // v_r, v_z, v_phi of one march index
  static constexpr int EXCH_OFF = PSLOT * SLOT_BYTES;
  static constexpr int BAR_OFF = EXCH_OFF + 3 * EXCH * 4;
  static constexpr int TAB_OFF = BAR_OFF + 64;
  static constexpr int BYTES = TAB_OFF + 128;  // + the material table; 128: slack for aligning the base
};

__device__ __forceinline__ void mbar_arrive(uint64_t *bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
// barrier of the row warps that also tells all of them whether any failed
template <int THREADS>
__device__ __forceinline__ bool row_barrier_or(bool fail) {
  uint32_t r;
  asm volatile(
      "{\n .reg .pred p, q;\n setp.ne.u32 p, %1, 0;\n barrier.cta.red.or.pred q, 1, %2, p;\n selp.u32 %0, 1, 0, q;\n}\n"
      : "=r"(r)
      : "r"((uint32_t)fail), "n"(THREADS)
      : "memory");
  return r != 0;
}

__device__ __forceinline__ void lds4(float (&d)[4], const float *p) {
  const float4 v = *reinterpret_cast<const float4 *>(p);
  d[0] = v.x, d[1] = v.y, d[2] = v.z, d[3] = v.w;
}
__device__ __forceinline__ void sts4(float *p, const float (&v)[4]) {
  *reinterpret_cast<float4 *>(p) = make_float4(v[0], v[1], v[2], v[3]);
}
__device__ __forceinline__ void cpy4(float (&d)[4], const float (&s)[4]) {
#pragma unroll
  for (int e = 0; e < 4; e++) d[e] = s[e];
}

// item t of the launch: z tile fastest, then r tile, then theta run; the first
// tiles1 tiles in runs of run1 planes, the rest, which would leave SMs idle in a
// last round, in shorter runs of run2
struct PassItem {
  int i0, ks, j0, J;  // first owned row, first staged z cell, first owned plane, planes
};
__device__ __forceinline__ PassItem pass_item(const PassParams &q, int R, int t) {
  const bool first = t < q.items1;
  const int n = first ? q.tiles1 : q.tiles - q.tiles1, run = first ? q.run1 : q.run2;
  if (!first) t -= q.items1;
  const int tile = t % n + (first ? 0 : q.tiles1);
  PassItem it;
  it.ks = q.ks0 + (tile % q.nzt) * PZ;
  it.i0 = (tile / q.nzt) * R;
  it.j0 = t / n * run;
  it.J = min(run, q.k.nth - it.j0);
  return it;
}

// an old velocity: used once, kept out of the way in L1
__device__ __forceinline__ void ld_once(float (&d)[4], const float *p) {
  asm volatile("ld.global.nc.L1::no_allocate.v4.f32 {%0, %1, %2, %3}, [%4];"
      : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
      : "l"(p));
}

template <int R>
__global__ void __launch_bounds__(PassSmem<R>::WARPS * 32, 1) 
    pass_step(const __grid_constant__ FusedMaps maps, const __grid_constant__ PassParams q) {
  using SM = PassSmem<R>;
  constexpr unsigned FULL = 0xffffffffu;
  extern __shared__ unsigned char smem_raw[];
  unsigned char *smem = smem_raw + ((128 - (smem_u32(smem_raw) & 127)) & 127);
  float *exch = reinterpret_cast<float *>(smem + SM::EXCH_OFF);
  uint64_t *full = reinterpret_cast<uint64_t *>(smem + SM::BAR_OFF), *empty = full + PSLOT;
  float4 *tab = reinterpret_cast<float4 *>(smem + SM::TAB_OFF);
  const KParams &p = q.k;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nth = p.nth, NR = p.NR, NZp = p.NZp;
  if (threadIdx.x == 0) {
    for (int s = 0; s < PSLOT; s++) mbar_init(&full[s], 1), mbar_init(&empty[s], SM::ROWS);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  for (int m = threadIdx.x; m < q.n_mat; m += SM::WARPS * 32) {
    const float2 l = __ldg(p.m_lam + m);
    tab[m] = make_float4(__ldg(p.m_rho + m), __ldg(p.m_imu + m), l.x, l.y);
  }
  __syncthreads();

  if (warp == SM::ROWS) {  // ---- producer: the planes of every item in the order they are used
    int slot = 0;
    unsigned eph = 0;  // bit s: parity of the next completion of empty[s]
    long long n = 0;   // planes issued
    bool ok = true;
    for (int t = blockIdx.x; t < q.items && ok; t += gridDim.x) {
      const PassItem it = pass_item(q, R, t);
      for (int l = 0; l < it.J + 2; l++, n++) {
        if (n >= PSLOT) {
          ok = __all_sync(FULL, mbar_wait(&empty[slot], (eph >> slot) & 1u));
          eph ^= 1u << slot;
          if (!ok) break;
        }
        int j = it.j0 - 1 + l;
        j = j < 0 ? j + nth : j >= nth ? j - nth : j;
        unsigned char *d = smem + slot * SM::SLOT_BYTES;
        if (lane == 0) {  // cells outside the array arrive as zeros
          mbar_expect_tx(&full[slot], SM::SLOT_BYTES);
          for (int f = 0; f < 6; f++)
            tma_load_4d(d + f * SM::FIELD * 4, &maps.f[F_SRR + f], it.ks, it.i0 - 1, j, 0, &full[slot]);
          tma_load_4d(d + 6 * SM::FIELD * 4, &maps.id, it.ks, it.i0 - 1, j, 0, &full[slot]);
        }
        __syncwarp();
        slot = slot == PSLOT - 1 ? 0 : slot + 1;
      }
    }
    if (!ok) {
      if (lane == 0) atomicOr(q.status, 2);
      // the copies issued last may still be writing their slots: wait (bounded) for them
      for (long long c = n > PSLOT ? n - PSLOT : 0; c < n; c++) (void)mbar_wait(&full[c % PSLOT], (unsigned)(c / PSLOT) & 1u);
    }
    return;
  }

  // ---- row warps
  const float dtv2 = 2.f * p.dtv, dts = p.dts, dts4 = 4.f * p.dts, idr = p.inv_dr, idz = p.inv_dz, idth = p.inv_dth;
  int s0 = 0;              // ring slot of plane j - 1
  unsigned fph = 0;        // bit s: parity of the next completion of full[s]
  int xb = 0;              // exchange buffer of the march index
  // fail: a wait of this warp gave up; every warp goes on to the next barrier,
  // which tells all of them, and they leave together (stop)
  bool fail = false, stop = false;
  const int at = warp * PW + lane * 4;  // this thread's cells in a staged field
  auto wait_full = [&](int s) {
    const bool ok = mbar_wait(&full[s], (fph >> s) & 1u);
    fph ^= 1u << s;
    return __any_sync(FULL, !ok) != 0;
  };
  auto release = [&](int s) {  // this row is done with the plane in slot s
    __syncwarp();
    if (lane == 0) mbar_arrive(&empty[s]);
  };
  for (int t = blockIdx.x; t < q.items && !stop; t += gridDim.x) {
    const PassItem it = pass_item(q, R, t);
    const int i = it.i0 - 1 + warp, k0 = it.ks + lane * 4;
    const bool row_ok = i >= 0 && i < NR && i <= q.r1;  // rows whose values any owned cell reads
    const bool own = warp >= 1 && warp <= R && i < q.r1 && lane >= 1 && lane <= 30 && k0 >= q.z0 && k0 < q.z1;
    const bool ids_ok = row_ok && k0 < NZp;
    const int ic = min(max(i, 0), NR - 1);
    const float inv_ri = __ldg(p.inv_ri + ic), inv_rh = __ldg(p.inv_rh + ic);
    const bool im = i >= 1, do_r = row_ok && warp >= 1, do_pz = row_ok && warp <= R;
    // element of this thread's cells in the plane v_r and v_z are computed for
    long long o = (long long)it.j0 * p.plane + (long long)ic * NZp + k0;
    const bool src_cell = own && i == p.src_i && p.src_k >= k0 && p.src_k < k0 + 4;
    const bool force_cell = row_ok && i == q.force_i && q.force_k >= k0 && q.force_k < k0 + 4;

    // values of the plane before, carried from one march index to the next
    float rho0[4], imu0[4], smc0[4], vr0[4], vz0[4], vpm[4];
    float2 lam0[4];
    zero(vr0), zero(vz0), zero(vpm);
    // old velocities of the next march index: v_r, v_z of plane j, v_phi of plane j - 1
    float nr_[4], nz_[4], np_[4];
    zero(nr_), zero(nz_), zero(np_);
    const long long wrap = (long long)nth * p.plane;
    auto fetch = [&](int j, long long oj) {
      if (ids_ok) {
        const long long a = j >= nth ? oj - wrap : oj, b = j == 0 ? oj - p.plane + wrap : oj - p.plane;
        ld_once(nr_, (const float *)p.f[F_VR] + a);
        ld_once(nz_, (const float *)p.f[F_VZ] + a);
        ld_once(np_, (const float *)p.f[F_VP] + b);
      }
    };
    // material values of the staged plane in slot s: rho, 1/mu, the sum of 1/mu
    // over rows i - 1 and i, lambda's
    auto material = [&](int s, float (&rho)[4], float (&rho_m)[4], float (&imu)[4], float (&smc)[4], float2 (&lam)[4]) {
      const uint16_t *ids = (const uint16_t *)(smem + s * SM::SLOT_BYTES + 6 * SM::FIELD * 4) + at;
      uint2 a = make_uint2(0u, 0u), b = make_uint2(0u, 0u);
      if (ids_ok) {
        a = *reinterpret_cast<const uint2 *>(ids);
        if (warp >= 1 && im) b = *reinterpret_cast<const uint2 *>(ids - PW);
      }
      const unsigned c[4] = {a.x & 0xffffu, a.x >> 16, a.y & 0xffffu, a.y >> 16};
      const unsigned m[4] = {b.x & 0xffffu, b.x >> 16, b.y & 0xffffu, b.y >> 16};
#pragma unroll
      for (int e = 0; e < 4; e++) {
        const float4 v = tab[c[e]];
        const float2 w = *reinterpret_cast<const float2 *>(tab + m[e]);
        rho[e] = v.x, imu[e] = v.y, lam[e] = make_float2(v.z, v.w);
        rho_m[e] = w.x, smc[e] = w.y + v.y;
      }
    };

    fetch(it.j0, o);
    zero(rho0), zero(imu0), zero(smc0);
#pragma unroll
    for (int e = 0; e < 4; e++) lam0[e] = make_float2(0.f, 0.f);
    if (!fail) fail = wait_full(s0);  // plane j0 - 1: only its material values are needed before the first march index
    if (!fail) {
      float unused[4];
      material(s0, rho0, unused, imu0, smc0, lam0);
    }
    for (int l = 1; l <= it.J + 1; l++, o += p.plane) {
      const int j = it.j0 - 1 + l;  // march index (j may equal nth: plane 0 again)
      const int s1 = s0 == PSLOT - 1 ? 0 : s0 + 1;
      if (!fail) fail = wait_full(s1);
      const float *S0 = (const float *)(smem + s0 * SM::SLOT_BYTES) + at;  // plane j - 1
      const float *S1 = (const float *)(smem + s1 * SM::SLOT_BYTES) + at;  // plane j
      float vr1[4], vz1[4], vp0[4], rho1[4] = {}, imu1[4] = {}, smc1[4] = {};
      float2 lam1[4] = {};
      float *X = exch + xb * SM::EXCH + at;
      const float *Xp = exch + (xb == 0 ? 2 : xb - 1) * SM::EXCH + at;
      zero(vr1), zero(vz1), zero(vp0);
      if (!fail) {
        // ---- A: v_r and v_z of plane j, v_phi of plane j - 1
        float rho_m[4], or_[4], oz_[4], op_[4];
        material(s1, rho1, rho_m, imu1, smc1, lam1);
        cpy4(or_, nr_), cpy4(oz_, nz_), cpy4(op_, np_);
        if (l <= it.J) fetch(j + 1, o + p.plane);
        float a_srp[4], a_srz[4], a_spz[4], a_spp[4], c_spp[4], c_srp[4], c_spz[4];
        lds4(a_srp, S1 + S_SRP * SM::FIELD);
        lds4(a_srz, S1 + S_SRZ * SM::FIELD);
        lds4(a_spz, S1 + S_SPZ * SM::FIELD);
        lds4(a_spp, S1 + S_SPP * SM::FIELD);
        lds4(c_spp, S0 + S_SPP * SM::FIELD);
        lds4(c_srp, S0 + S_SRP * SM::FIELD);
        lds4(c_spz, S0 + S_SPZ * SM::FIELD);
        const float srz_km = __shfl_up_sync(FULL, a_srz[3], 1), spz_km = __shfl_up_sync(FULL, c_spz[3], 1);
        const float rho_k4 = __shfl_down_sync(FULL, rho1[0], 1);
        if (do_r) {
          float a_srr[4], m_srr[4], m_spp[4];
          lds4(a_srr, S1 + S_SRR * SM::FIELD);
          lds4(m_srr, S1 + S_SRR * SM::FIELD - PW);
          lds4(m_spp, S1 + S_SPP * SM::FIELD - PW);
#pragma unroll
          for (int e = 0; e < 4; e++) {
            const float Dr = (a_srr[e] - m_srr[e]) * idr;
            const float Q = (0.5f * (a_srr[e] + m_srr[e]) - 0.5f * (a_spp[e] + m_spp[e]) + (a_srp[e] - c_srp[e]) * idth) * inv_ri;
            const float Dz = (a_srz[e] - (e ? a_srz[e - 1] : srz_km)) * idz;
            const float v = or_[e] + dtv2 * rcp_fast(rho_m[e] + rho1[e]) * (Dr + Q + Dz);
            vr1[e] = im ? v : or_[e];
          }
        }
        if (do_pz) {
          float a_szz[4], p_srz[4], p_srp[4];
          lds4(a_szz, S1 + S_SZZ * SM::FIELD);
          zero(p_srz), zero(p_srp);
          if (i + 1 < NR) {
            lds4(p_srz, S1 + S_SRZ * SM::FIELD + PW);
            lds4(p_srp, S0 + S_SRP * SM::FIELD + PW);
          }
          const float szz_k4 = __shfl_down_sync(FULL, a_szz[0], 1);
#pragma unroll
          for (int e = 0; e < 4; e++) {
            {
              const float s1v = p_srz[e], s0v = a_srz[e];
              const float Dr = (s1v - s0v) * idr;
              const float Q = (0.5f * (s1v + s0v) + (a_spz[e] - c_spz[e]) * idth) * inv_rh;
              const float Dz = ((e < 3 ? a_szz[e + 1] : szz_k4) - a_szz[e]) * idz;
              vz1[e] = oz_[e] + dtv2 * rcp_fast(rho1[e] + (e < 3 ? rho1[e + 1] : rho_k4)) * (Dr + Q + Dz);
            }
            {
              const float s1v = p_srp[e], s0v = c_srp[e];
              const float Dr = (s1v - s0v) * idr;
              const float Q = ((s1v + s0v) + (a_spp[e] - c_spp[e]) * idth) * inv_rh;
              const float Dz = (c_spz[e] - (e ? c_spz[e - 1] : spz_km)) * idz;
              vp0[e] = op_[e] + dtv2 * rcp_fast(rho0[e] + rho1[e]) * (Dr + Q + Dz);
            }
          }
        }
        if (force_cell) {  // point force (v_r or v_z), on the recomputed halo as well
          const int st = *p.step + p.step_off, jj = j >= nth ? j - nth : j;
          const float w = st < p.n_wav ? __ldg(q.force_w + jj) * __ldg(q.force_wav + st) : 0.f;
#pragma unroll
          for (int e = 0; e < 4; e++)
            if (k0 + e == q.force_k) {
              if (q.force_vz) vz1[e] += w;
              else vr1[e] += w;
            }
        }
        sts4(X, vr1);
        sts4(X + SM::FIELD, vz1);
        sts4(X + 2 * SM::FIELD, vp0);
        if (own) {
          if (l <= it.J) {
            Vec<float, 4>::st((float *)q.out.f[F_VR] + o, vr1);
            Vec<float, 4>::st((float *)q.out.f[F_VZ] + o, vz1);
          }
          if (l >= 2) Vec<float, 4>::st((float *)q.out.f[F_VP] + (o - p.plane), vp0);
        }
      }
      stop = row_barrier_or<SM::ROWS * 32>(fail);
      if (stop) break;
      // ---- B: the stresses of plane j - 1
      if (l >= 2 && warp >= 1 && warp <= R && i < q.r1) {
        float p_vr[4], m_vz[4], m_vp[4];
        lds4(p_vr, Xp + PW);
        lds4(m_vz, Xp + SM::FIELD - PW);
        lds4(m_vp, X + 2 * SM::FIELD - PW);
        const float vr_k4 = __shfl_down_sync(FULL, vr0[0], 1), vp_k4 = __shfl_down_sync(FULL, vp0[0], 1);
        const float vz_km = __shfl_up_sync(FULL, vz0[3], 1);
        const float sjc_0 = imu0[0] + imu1[0];  // 1/mu over planes j - 1 and j
        const float sjc_k4 = __shfl_down_sync(FULL, sjc_0, 1), smc_k4 = __shfl_down_sync(FULL, smc0[0], 1);
        if (own) {
          float orr[4], opp[4], ozz[4], orp[4], opz[4], orz[4];
          lds4(orr, S0 + S_SRR * SM::FIELD);
          lds4(opp, S0 + S_SPP * SM::FIELD);
          lds4(ozz, S0 + S_SZZ * SM::FIELD);
          lds4(orp, S0 + S_SRP * SM::FIELD);
          lds4(opz, S0 + S_SPZ * SM::FIELD);
          lds4(orz, S0 + S_SRZ * SM::FIELD);
          float sjc[5] = {sjc_0, imu0[1] + imu1[1], imu0[2] + imu1[2], imu0[3] + imu1[3], sjc_k4};
#pragma unroll
          for (int e = 0; e < 4; e++) {
            const float smc_e1 = e < 3 ? smc0[e + 1] : smc_k4;
            const float err = (p_vr[e] - vr0[e]) * idr;
            const float epp = ((vp0[e] - vpm[e]) * idth + 0.5f * (vr0[e] + p_vr[e])) * inv_rh;
            const float ezz = (vz0[e] - (e ? vz0[e - 1] : vz_km)) * idz;
            orr[e] += dts * (lam0[e].y * err + lam0[e].x * (epp + ezz));
            opp[e] += dts * (lam0[e].y * epp + lam0[e].x * (err + ezz));
            ozz[e] += dts * (lam0[e].y * ezz + lam0[e].x * (err + epp));
            if (im) {
              const float gr = (vp0[e] - m_vp[e]) * idr;
              const float Q = ((vr1[e] - vr0[e]) * idth - 0.5f * (vp0[e] + m_vp[e])) * inv_ri;
              orp[e] += dts4 * rcp_fast(smc0[e] + smc1[e]) * (gr + Q);
              const float gz = ((e < 3 ? vr0[e + 1] : vr_k4) - vr0[e]) * idz;
              const float gw = (vz0[e] - m_vz[e]) * idr;
              orz[e] += dts4 * rcp_fast(smc0[e] + smc_e1) * (gz + gw);
            }
            const float Q = (vz1[e] - vz0[e]) * idth * inv_rh;
            const float gz = ((e < 3 ? vp0[e + 1] : vp_k4) - vp0[e]) * idz;
            opz[e] += dts4 * rcp_fast(sjc[e] + sjc[e + 1]) * (Q + gz);
          }
          if (src_cell && (p.src_j < 0 || p.src_j == j - 1)) {
            const int st = *p.step + p.step_off;
            const float w = st < p.n_wav ? __ldg(p.wav + st) : 0.f;
#pragma unroll
            for (int e = 0; e < 4; e++)
              if (k0 + e == p.src_k) orr[e] += w, opp[e] += w, ozz[e] += w;
          }
          const long long os = o - p.plane;
          Vec<float, 4>::st((float *)q.out.f[F_SRR] + os, orr);
          Vec<float, 4>::st((float *)q.out.f[F_SPP] + os, opp);
          Vec<float, 4>::st((float *)q.out.f[F_SZZ] + os, ozz);
          Vec<float, 4>::st((float *)q.out.f[F_SRP] + os, orp);
          Vec<float, 4>::st((float *)q.out.f[F_SPZ] + os, opz);
          Vec<float, 4>::st((float *)q.out.f[F_SRZ] + os, orz);
        }
      }
      release(s0);
      s0 = s1;
      xb = xb == 2 ? 0 : xb + 1;
      cpy4(rho0, rho1), cpy4(imu0, imu1), cpy4(smc0, smc1), cpy4(vr0, vr1), cpy4(vz0, vz1), cpy4(vpm, vp0);
#pragma unroll
      for (int e = 0; e < 4; e++) lam0[e] = lam1[e];
    }
    if (!stop) {  // the last plane of the run
      release(s0);
      s0 = s0 == PSLOT - 1 ? 0 : s0 + 1;
    }
  }
  if (stop && lane == 0) atomicOr(q.status, 2);
}

constexpr int PASS_R = 9;

}  // namespace

bool pass_region(const KParams &p, int *r1, int *z0, int *z1) {
  const int za = (p.pml_z + 3) / 4 * 4, zb = std::max(za, (p.NZ - p.pml_z - 1) / 4 * 4);
  // the recomputed rim (row r1's v_r, the cells z0 - 1 and z1) must be lean too
  *r1 = p.nr < p.NR ? p.nr - 1 : p.NR;
  *z0 = za >= p.pml_z + 1 ? za : za + 4;
  *z1 = zb;
  return *r1 >= 4 && *z1 - *z0 >= 32 && p.i_lo == 0 && p.i_hi == p.NR && p.k_lo == 0 && p.k_hi >= p.NZ;
}

size_t pass_smem_bytes(int n_mat) { return PassSmem<PASS_R>::BYTES + (size_t)n_mat * 16; }

int pass_box_rows() { return PASS_R + 2; }

cudaError_t launch_pass(int code, const FusedMaps &maps, const PassParams &pp, cudaStream_t s) {
  const int runs = pass_runs(code);
  PassParams q = pp;
  if (!pass_region(q.k, &q.r1, &q.z0, &q.z1) || runs < 1) return cudaErrorInvalidValue;
  q.ks0 = (q.z0 - 4) / 8 * 8;  // 16-byte aligned ID rows; lane 0 is halo
  // tile zt owns [ks0 + 4 + 120 zt, ks0 + 124 + 120 zt)
  q.nzt = (q.z1 - (q.ks0 + 4) + PZ - 1) / PZ;
  const long long tiles = (long long)((q.r1 + PASS_R - 1) / PASS_R) * q.nzt;
  if (tiles * q.k.nth > 0x7fffffffLL) return cudaErrorInvalidValue;
  q.tiles = (int)tiles;
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  sms = std::max(sms, 1);
  // whole rounds of one item per SM in runs theta / d, the tiles left over in as
  // many runs (of two planes or more) as the SMs take in one round
  auto run_of = [&](int d) { return (q.k.nth + d - 1) / d; };
  auto count = [&](int run) { return (q.k.nth + run - 1) / run; };
  q.run1 = run_of(runs);
  q.tiles1 = (int)(tiles * count(q.run1) / sms * sms / count(q.run1));
  const int rest = q.tiles - q.tiles1;
  q.run2 = std::min(q.run1, std::max(2, run_of(rest > 0 ? std::max(1, sms / rest) : 1)));
  q.items1 = q.tiles1 * count(q.run1);
  q.items = q.items1 + rest * count(q.run2);
  const int bytes = (int)pass_smem_bytes(q.n_mat);
  cudaError_t e = cudaFuncSetAttribute(pass_step<PASS_R>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
  if (e != cudaSuccess) return e;
  const int grid = pass_per_tile(code) ? q.items : std::min(q.items, sms);
  pass_step<PASS_R><<<grid, PassSmem<PASS_R>::WARPS * 32, bytes, s>>>(maps, q);
  return cudaGetLastError();
}

}  // namespace cwell
