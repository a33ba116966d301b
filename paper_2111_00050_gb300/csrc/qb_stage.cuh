// The shared-memory resident path of spaces whose sectors are all small: one CTA takes a
// sector and runs every RK4 stage of the call on it, with only CTA barriers between stages
// (the sectors are independent, so no CTA ever waits on another).  The arithmetic and the
// order of every ket's sums are the direct stage kernel's (qb_block.cuh): the states agree
// bit for bit.
//
// A stage launch of such a space costs 5 to 12 us, most of it latency; in one CTA a stage is
// a chain of shared-memory reads.  The targets do not change from stage to stage: they are
// ranked once per call and kept as 16-bit indices beside the four vectors (psi, its weighted
// copy and two stage vectors), record by record, so that the lanes read them in order.
#pragma once
#include "qb_block.cuh"

namespace qb {

struct ResArgs {
  double2* psi;        // global psi [total]
  float4* psif;        // global double-float copy of psi in the weighted basis [total] (read, written back)
  const float4* diag;  // per-ket diagonal
  float2 scale;        // two-body scale, double-float
  double dt;
  int64_t steps;
  int order;           // Taylor order of a step (stages per step)
  int cap;             // kets per sector the shared buffers hold (a multiple of 4)
  float4 *w1, *w2;     // stage vectors [total] and counter of the cooperative launch
  uint32_t* barrier;
  uint32_t polls;      // of a CTA at a barrier before it gives up
  bool later;          // not the call's first launch
  int* status;
};

// Whether the resident kernel keeps each ket's own records alone (SPARSE): where a ket takes part
// in few of them (Tables::bk_share).  One stage, every record / own records (us): M = 16, 969 kets
// (share 0.02) 63 / 2.9; M = 9, 220 kets (0.05; the register kernel) 7.7 / 1.8; M = 8, 495 (0.09) 12.5
// / 3.2; M = 6, 210 (0.13) 7.0 / 3.1, 1,287 (0.36) 9.4 / 9.0; M = 4, 495 (0.42) 3.5 / 3.8.
inline bool resident_sparse(const Tables& t) { return t.bk_share < 0.3f && t.bk_kc != 2 && t.bk_kc != 3; }

// bytes of one ket's target indices: w 16-bit entries a record, and the fifth partner's; of its
// own records alone, their numbers and how many there are
inline size_t resident_index_bytes(const Tables& t) {
  const size_t rec = t.bk_kc == 2 ? 4 : t.bk_kc == 5 ? 10 : 8;
  return resident_sparse(t) ? t.bk_most * (rec + 2) + 2 : t.bk_nrec * rec;
}

// Shared memory of the resident kernel holding `cap` kets per sector.
inline size_t resident_smem(const Tables& t, int cap) {
  return blk_smem_bytes(t, t.is_complex != 0) + (size_t)cap * (64 + resident_index_bytes(t)) +
         (resident_sparse(t) ? kFirstBytes : 0);
}

// SPARSE: a ket's targets are kept for the records that it takes part in, with their numbers, and
// the lanes walk each its own; else for every record, which the lanes walk in step.
template <int MT, int KC, bool CPLX, bool SPARSE>
__global__ void __launch_bounds__(1024, 1) resident_kernel(const Tables t, const ResArgs r) {
  constexpr int NT = Rec<KC>::n, RW = Rec<KC>::w, NW = occ_words<MT>();
  const int T = t.bk_T, nrec = t.bk_nrec, cap = r.cap;
  float2* sG = reinterpret_cast<float2*>(blk_smem);
  float2* sGi = sG + T;
  uint2* sinfo = reinterpret_cast<uint2*>(sG + (CPLX ? 2 : 1) * T);
  double2* spsi = reinterpret_cast<double2*>(sinfo + ((nrec + 1) & ~1));
  float4* spsif = reinterpret_cast<float4*>(spsi + cap);
  float4* sw1 = spsif + cap;
  float4* sw2 = sw1 + cap;
  const int rows = SPARSE ? t.bk_most : nrec;
  uint16_t* sidx = reinterpret_cast<uint16_t*>(sw2 + cap);      // [rows][cap][RW]
  uint16_t* sidx5 = sidx + (size_t)rows * cap * RW;             // [rows][cap]
  uint16_t* srec = sidx5 + (NT > 4 ? (size_t)rows * cap : 0);   // [rows][cap] numbers of the records
  uint16_t* scnt = srec + (size_t)rows * cap;                   // [cap]
  uint16_t* first = scnt + cap;                                 // [256]
  const int tid = threadIdx.x, nthr = blockDim.x;
  for (int i = tid; i < T; i += nthr) {
    sG[i] = __ldg(t.bk_G + i);
    if (CPLX) sGi[i] = __ldg(t.bk_Gi + i);
  }
  for (int i = tid; i < nrec; i += nthr) sinfo[i] = __ldg(t.bk_info + i);
  __syncthreads();
  if (SPARSE) first_records(sinfo, nrec, first);
  const int64_t off = __ldg(t.sec_off + blockIdx.x);
  const int D = (int)(__ldg(t.sec_off + blockIdx.x + 1) - off);
  if (D > cap) {  // not reached: the host sizes the buffers for the largest sector
    if (tid == 0) atomicOr(r.status, 4);
    return;
  }

  // the sector's state, and its kets' targets by block base and place (qb_block.cuh)
  bool bad = false;
  for (int i = tid; i < D; i += nthr) {
    const int64_t g = off + i;
    spsi[i] = r.psi[g];
    spsif[i] = r.psif[g];  // the weighted double-float copy
    const uint64_t word = __ldg(t.occ + g);
    uint32_t ob[NW];
    unpack_occ<MT, NW>(t, word, ob);
    uint32_t blk = __ldg(t.rblk + g / 32), f = __ldg(t.fill + g / 32 * 32);
    for (int64_t k = g / 32 * 32 + 1; k <= g; ++k) {  // blocks begun since the round's first ket
      const uint32_t fk = __ldg(t.fill + k);
      blk += fk != f + 1u;
      f = fk;
    }
    const uint32_t* base = t.bk_base + (size_t)blk * T;
    RecordWalk walk(t, SPARSE ? word : 0ull);
    int row = 0;
    for (;; ++row) {
      if (SPARSE ? !walk.next(sinfo, first) : row == nrec) break;
      if (SPARSE && row == rows) {  // not reached: bk_most bounds them
        bad = true;
        break;
      }
      const int rec = SPARSE ? walk.rec : row;
      if (SPARSE) srec[(size_t)row * cap + i] = (uint16_t)rec;
      const uint2 info = sinfo[rec];
      const float Af = (occ_float23<NW>(ob, info.x, (info.x & 0x8000u) != 0u) - 8388608.0f) *
                       (occ_float23<NW>(ob, info.x >> 16, (info.x & 0x80000000u) != 0u) - __uint_as_float(info.y));
      const int n = (int)((info.x >> 4) & 7);
      for (int c = 0; c < (NT > 4 ? 5 : RW); ++c) {
        const int sl = c < 4 ? RW * rec + c : 4 * nrec + rec;
        uint32_t k = 0;
        if (Af != 0.f && c < n) {
          const uint32_t place = c < 4 ? __ldg(reinterpret_cast<const uint16_t*>(t.bk_map) +
                                               ((size_t)rec * t.bk_S + f) * RW + c)
                                       : __ldg(t.bk_map5 + (size_t)rec * t.bk_S + f);
          k = __ldg(base + sl) + place - (uint32_t)off;
          if (k >= (uint32_t)D) {
            bad = true;
            k = 0;
          }
        }
        if (c < 4)
          sidx[((size_t)row * cap + i) * RW + c] = (uint16_t)k;
        else
          sidx5[(size_t)row * cap + i] = (uint16_t)k;
      }
    }
    if (SPARSE) scnt[i] = (uint16_t)row;
  }
  if (bad) atomicOr(r.status, 1);
  __syncthreads();

  DfArgs a{};
  a.diag = r.diag;
  a.scale[0] = r.scale;
  a.psi = spsi;
  a.psif = spsif;
  dfl bil_l{0.f, 0.f};
  dfc bil_w[1] = {dfc{0ull, 0ull}};
  double dot64 = 0.0;
  for (int64_t it = 0; it < r.steps; ++it) {
    for (int d = r.order; d >= 1; --d) {
      const int j = r.order - d;
      const float4* vin = (j == 0) ? spsif : ((j - 1) % 2 == 0 ? sw1 : sw2);
      a.vin = vin;
      a.out = (d == 1) ? spsif : (j % 2 == 0 ? sw1 : sw2);
      a.zre = r.dt / d;
      const float zh = (float)a.zre;
      a.zf = make_float2(zh, (float)(a.zre - (double)zh));
      for (int i = tid; i < ((D + 31) & ~31); i += nthr) {
        const bool valid = i < D;
        const int ii = valid ? i : D - 1;
        uint32_t ob[NW];
        unpack_occ<MT, NW>(t, valid ? __ldg(t.occ + off + ii) : 0ull, ob);
        dfc acc[1] = {dfc{0ull, 0ull}};
        float4 x[NT];
#pragma unroll
        for (int c = 0; c < NT; ++c) x[c] = make_float4(0.f, 0.f, 0.f, 0.f);
        const uint16_t* ip = sidx + (size_t)ii * RW;
        const uint16_t* ip5 = sidx5 + ii;
        const int cnt = !SPARSE ? nrec : valid ? (int)scnt[ii] : 0;
        for (int row = 0; SPARSE ? __any_sync(0xffffffffu, row < cnt) : row < nrec; ++row) {
          const int rec = !SPARSE ? row : row < cnt ? (int)srec[(size_t)row * cap + ii] : 0;
          const uint2 info = sinfo[rec];
          const float Af = (occ_float23<NW>(ob, info.x, (info.x & 0x8000u) != 0u) - 8388608.0f) *
                           (occ_float23<NW>(ob, info.x >> 16, (info.x & 0x80000000u) != 0u) - __uint_as_float(info.y));
          const bool act = SPARSE ? row < cnt : Af != 0.f;
          if (SPARSE ? act : (bool)__any_sync(0xffffffffu, act)) {
            const int n = KC == 0 ? (int)((info.x >> 4) & 7) : NT;
            uint2 k2 = make_uint2(0u, 0u);
            if constexpr (RW == 2)
              k2.x = *reinterpret_cast<const uint32_t*>(ip + (size_t)row * cap * RW);
            else
              k2 = *reinterpret_cast<const uint2*>(ip + (size_t)row * cap * RW);
            if (act) {  // a lane that lacks the pair keeps its last values
              x[0] = vin[k2.x & 0xffffu];
              if (KC > 0 || n > 1) x[1] = vin[k2.x >> 16];
              if constexpr (NT > 2)
                if (KC > 0 || n > 2) x[2] = vin[k2.y & 0xffffu];
              if constexpr (NT > 3)
                if (KC > 0 || n > 3) x[3] = vin[k2.y >> 16];
              if constexpr (NT > 4) x[4] = vin[ip5[(size_t)row * cap]];
            }
            add_record<KC, CPLX, false>(acc[0], x, sG, sGi, rec, nrec, n, 0, Af);
            if (KC > 0 || (info.x & 0x80u)) acc[0] = dfc_renorm(acc[0]);
          }
        }
        if (valid) stage_epilogue<MT, 1, KIND_STAGE, false, NW, true>(t, a, d == 1 ? 1 : 0, off + i, i, acc, ob, bil_l, bil_w, dot64);
      }
      __syncthreads();
    }
  }
  for (int i = tid; i < D; i += nthr) {
    r.psi[off + i] = spsi[i];
    r.psif[off + i] = spsif[i];
  }
}

// Barrier of a cooperative grid: the CTAs arrive at a counter and wait until `target` have.
// The wait is bounded (kWaitPolls, a minute or so, longer than another stream's kernel should
// hold the SMs that the grid's last CTAs wait for): on its end kLate is set in the launch's
// status and the CTA leaves, as every other one does at the next barrier.
constexpr int kLate = 8;
__device__ __forceinline__ bool grid_barrier(uint32_t* counter, uint32_t target, uint32_t polls, int* status) {
  __syncthreads();
  int late = 0;
  if (threadIdx.x == 0) {
    __threadfence();
    atomicAdd(counter, 1u);
    uint32_t seen = 0;
    for (uint32_t n = 0; n < polls && seen < target; ++n)
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(counter) : "memory");
    late = seen < target;
    if (late) atomicOr(status, kLate);
    __threadfence();
  }
  return __syncthreads_or(late) == 0;
}

// Sectors of at most reg_kets(M) kets with a fixed partner count: one ket a thread, its
// targets, pair factors, psi and weights in registers for the whole call, so that a stage
// reads shared memory for the gathered values (and the couplings, by broadcast) only.  The
// records are unrolled: with one or two warps a sector the general kernel's chain of
// dependent reads per record is all latency.  One RK4 stage of the 42-ket M = 5 sector: 1.1 us
// (general kernel 3.1; 4.6 when every stage ranked its targets).
constexpr int reg_kets(int M) { return M == 5 ? 512 : 256; }  // 126 registers a thread, 202 (M = 7), 255 (M = 9)

//
// GRID: the same over the whole space, one CTA an SM in a cooperative launch, for spaces whose
// sectors are too large for a CTA but whose kets all find a thread.  The stage vectors lie in
// global memory (L2), with a grid barrier in the place of the CTA's.  Launched stage by stage
// such a space pays for the launch, its tables and its chain of dependent reads every time (us a
// stage, stage launches / grid): M = 5, 3,060 kets 5.5 / 3.5, 33,649 kets 6.8 / 4.1, 53,130 kets
// 8.2 / 5.1; M = 7, 19,448 kets 10.1 / 4.5, 27,132 kets 10.2 / 6.1.  M = 9 does not fit its
// registers (12,870 kets 12.2 / 12.1) and stays with the stage launches.
template <int MT, bool GRID>
__global__ void __launch_bounds__(reg_kets(MT), 1) resident_reg_kernel(const Tables t, const ResArgs r) {
  constexpr int KC = (MT - 1) / 2, NT = Rec<KC>::n, RW = Rec<KC>::w, NW = occ_words<MT>();
  constexpr int NR = MT * (MT + 1) / 2;
  static_assert(KC >= 2 && KC <= 4, "two or four 16-bit targets a record");
  const int T = t.bk_T;
  // a launch after one of the same call that gave up does nothing
  if (GRID && r.later && __syncthreads_or(threadIdx.x == 0 && (*reinterpret_cast<volatile int*>(r.status) & kLate) != 0)) return;
  float2* sG = reinterpret_cast<float2*>(blk_smem);
  // two vectors of the stages: [2][cap] in shared memory, or the workspace's
  float4* const buf0 = GRID ? r.w1 : reinterpret_cast<float4*>(blk_smem + blk_smem_bytes(t, false));
  float4* const buf1 = GRID ? r.w2 : buf0 + r.cap;
  const int i = GRID ? (int)(blockIdx.x * blockDim.x + threadIdx.x) : (int)threadIdx.x;
  for (int k = threadIdx.x; k < T; k += blockDim.x) sG[k] = __ldg(t.bk_G + k);
  const int64_t off = GRID ? 0 : __ldg(t.sec_off + blockIdx.x);
  const int D = (int)(GRID ? t.total : __ldg(t.sec_off + blockIdx.x + 1) - off);
  const bool valid = i < D;
  const int64_t g = off + (valid ? i : 0);
  uint32_t ix[NR][RW / 2];
  float A[NR];
  double2 psi = r.psi[g];
  float4 pf = r.psif[g];
  const float4 dg4 = __ldg(r.diag + g);
  const double wk = __ldg(t.wk + g), wi = __ldg(t.wi + g);
  bool bad = !GRID && D > r.cap;
  {
    uint32_t ob[NW];
    unpack_occ<MT, NW>(t, valid ? __ldg(t.occ + g) : 0ull, ob);
    uint32_t blk = __ldg(t.rblk + g / 32), f = __ldg(t.fill + g / 32 * 32);
    for (int64_t k = g / 32 * 32 + 1; k <= g; ++k) {  // blocks begun since the round's first ket
      const uint32_t fk = __ldg(t.fill + k);
      blk += fk != f + 1u;
      f = fk;
    }
    const uint32_t* base = t.bk_base + (size_t)blk * T;
    const unsigned char* mp = t.bk_map + (size_t)f * (2 * RW);
#pragma unroll
    for (int rec = 0; rec < NR; ++rec) {
      const uint2 info = __ldg(t.bk_info + rec);
      A[rec] = (occ_float23<NW>(ob, info.x, (info.x & 0x8000u) != 0u) - 8388608.0f) *
               (occ_float23<NW>(ob, info.x >> 16, (info.x & 0x80000000u) != 0u) - __uint_as_float(info.y));
      const MapRec<KC> m = load_map<KC>(mp + (size_t)rec * t.bk_S * (2 * RW), nullptr);
      const BaseRec<KC> b = load_base<KC>(base, rec, NR);
      uint32_t k[4] = {b.a.x + (m.a.x & 0xffffu), b.a.y + (m.a.x >> 16), b.a.z + (m.a.y & 0xffffu), b.a.w + (m.a.y >> 16)};
#pragma unroll
      for (int c = 0; c < RW; ++c) {
        k[c] -= (uint32_t)off;
        if (A[rec] == 0.f || c >= NT || k[c] >= (uint32_t)D) {
          bad |= A[rec] != 0.f && c < NT;
          k[c] = valid ? (uint32_t)i : 0u;  // a pair the ket lacks: factor 0 on the ket's own value
        }
      }
      ix[rec][0] = k[0] | (k[1] << 16);
      if constexpr (RW == 4) ix[rec][1] = k[2] | (k[3] << 16);
    }
  }
  if (bad) atomicOr(r.status, 1);
  if (!GRID && D > r.cap) return;  // not reached: the host sizes the buffers for the largest sector
  const dfl sc{r.scale.x, r.scale.y};
  const dfl dg = df_add(dfl{dg4.x, dg4.y}, df_mul(sc, dfl{dg4.z, dg4.w}));
  float4 own = pf;
  int cur = 0;
  uint32_t round = 0;
  auto sync = [&]() -> bool {  // false: the grid's barrier gave up
    if (GRID) return grid_barrier(r.barrier, ++round * gridDim.x, r.polls, r.status);
    __syncthreads();
    return true;
  };
  if (valid) buf0[i] = pf;
  if (!sync()) return;
  for (int64_t it = 0; it < r.steps; ++it) {
    for (int d = r.order; d >= 1; --d) {
      const float4* vin = cur ? buf1 : buf0;
      dfc acc{0ull, 0ull};
#pragma unroll
      for (int rec = 0; rec < NR; ++rec) {
        float4 x[NT];
        x[0] = vin[ix[rec][0] & 0xffffu];
        x[1] = vin[ix[rec][0] >> 16];
        if constexpr (NT > 2) x[2] = vin[ix[rec][RW / 2 - 1] & 0xffffu];
        if constexpr (NT > 3) x[3] = vin[ix[rec][RW / 2 - 1] >> 16];
        add_record<KC, false, false>(acc, x, sG, sG, rec, NR, NT, 0, A[rec]);
        acc = dfc_renorm(acc);
      }
      // the stage's output, with the arithmetic of stage_epilogue
      dfl ar, ai;
      f2_unpack(acc.h, ar.h, ai.h);
      f2_unpack(acc.l, ar.l, ai.l);
      const dfl hr = df_add(df_mul(dg, df_re(own)), df_mul(sc, ar));
      const dfl hi = df_add(df_mul(dg, df_im(own)), df_mul(sc, ai));
      const double zre = r.dt / d;
      if (d > 1) {
        const float zh = (float)zre;
        const dfl zf{zh, (float)(zre - (double)zh)};
        own = df_pack(df_add(df_re(pf), df_mul(zf, hi)), df_add(df_im(pf), df_neg(df_mul(zf, hr))));
      } else {
        psi.x = psi.x + wk * (zre * df_to(hi));
        psi.y = psi.y + wk * (-zre * df_to(hr));
        own = pf = df_pack(df_of(psi.x * wi), df_of(psi.y * wi));
      }
      cur ^= 1;
      if (valid) (cur ? buf1 : buf0)[i] = own;
      if (!sync()) return;
    }
  }
  if (valid) {
    r.psi[g] = psi;
    r.psif[g] = pf;
  }
}

template <int MT>
int resident_reg_launch(const Tables& t, const ResArgs& r, int threads, cudaStream_t st) {
  auto k = resident_reg_kernel<MT, false>;
  const size_t smem = blk_smem_bytes(t, false) + (size_t)r.cap * 32;
  int per = 0, sms = 0;
  const int rc = occupancy_cached(k, smem, &per, &sms, threads);
  if (rc) return rc;
  k<<<t.n_sectors, threads, smem, st>>>(t, r);
  QB_CUDA(cudaGetLastError());
  return QB_OK;
}

// The cooperative launch, by the call that holds the device's turn (coop_turn): it needs every
// SM, and the barrier's counter and the status beside it are the space's.
template <int MT>
int grid_reg_launch(const Tables& t, const ResArgs& r0, cudaStream_t st) {
  auto k = resident_reg_kernel<MT, true>;
  const size_t smem = blk_smem_bytes(t, false);
  int per = 0, sms = 0;
  const int rc = occupancy_cached(k, smem, &per, &sms, reg_kets(MT));
  if (rc) return rc;
  ResArgs r = r0;
  Tables tt = t;
  const int threads = ((int)((t.total + sms - 1) / sms) + 31) & ~31;
  const int grid = (int)((t.total + threads - 1) / threads);
  // the barrier's counter: 31 bits of arrivals a launch
  const int64_t most = (int64_t)0x7fffffff / ((int64_t)grid * r.order) - 1;
  void* args[] = {&tt, &r};
  for (int64_t left = r0.steps; left > 0; left -= r.steps) {
    r.steps = std::min(left, most);
    r.later = left < r0.steps;
    QB_CUDA(cudaMemsetAsync(r.barrier, 0, (r.later ? 1 : 2) * sizeof(uint32_t), st));  // the status once
    QB_CUDA(cudaLaunchCooperativeKernel(reinterpret_cast<const void*>(k), dim3(grid), dim3(threads), args, smem, st));
  }
  return QB_OK;
}
// Whether every ket finds a thread and a 16-bit target
inline bool grid_reg_fits(const Tables& t, int sms) {
  return !t.fa_on && (t.M == 5 || t.M == 7) && t.bk_kc > 0 &&
         t.total <= std::min<int64_t>(65536, (int64_t)sms * reg_kets(t.M));
}

template <int MT, int KC, bool CPLX, bool SPARSE>
int resident_launch_k(const Tables& t, const ResArgs& r, int threads, cudaStream_t st) {
  auto k = resident_kernel<MT, KC, CPLX, SPARSE>;
  const size_t smem = resident_smem(t, r.cap);
  int per = 0, sms = 0;
  const int rc = occupancy_cached(k, smem, &per, &sms, threads);  // raises the function's shared-memory limit
  if (rc) return rc;
  k<<<t.n_sectors, threads, smem, st>>>(t, r);
  QB_CUDA(cudaGetLastError());
  return QB_OK;
}

// Kets per sector up to which the resident path is the faster one (in spaces of at most 64
// kets per SM, one CTA or two each).  One stage, resident against stage launches (us): the
// register kernel, M = 5: 42 kets 1.1 / 5.3, 51 sectors of up to 201 kets 1.9 / 5.5; M = 7, 50
// sectors of up to 246: 3.8 / 8.0.  The general kernel, M = 6, 132 kets 8.1 / 11.8, 335 kets
// 11.7 / 11.8; exact momentum M = 7, 151 kets 7.7 / 10.8; but M = 5, 612 kets 7.1 / 5.6.
inline int resident_most(const Tables& t) {
  const bool reg = t.bk_kc >= 2 && t.bk_kc <= 4 && t.M <= 9;
  return reg ? reg_kets(t.M) : 256;
}

int resident_launch_m5(const Tables&, const ResArgs&, int, cudaStream_t);
int resident_launch_m7(const Tables&, const ResArgs&, int, cudaStream_t);
int resident_launch_m9(const Tables&, const ResArgs&, int, cudaStream_t);
int resident_launch_m11(const Tables&, const ResArgs&, int, cudaStream_t);
int resident_launch_any(const Tables&, const ResArgs&, int, cudaStream_t);
int grid_launch_m5(const Tables&, const ResArgs&, cudaStream_t);
int grid_launch_m7(const Tables&, const ResArgs&, cudaStream_t);

// Every sector resident, `threads` threads each.
inline int resident_launch(const Tables& t, const ResArgs& r, int threads, cudaStream_t st) {
  if (t.bk_kc > 0) {
    switch (t.M) {
      case 5: return resident_launch_m5(t, r, threads, st);
      case 7: return resident_launch_m7(t, r, threads, st);
      case 9: return resident_launch_m9(t, r, threads, st);
      case 11: return resident_launch_m11(t, r, threads, st);
      default: break;
    }
  }
  return resident_launch_any(t, r, threads, st);
}

}  // namespace qb
