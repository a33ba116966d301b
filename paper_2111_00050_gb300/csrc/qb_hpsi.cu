// H psi in FP64 for one state (qb_hpsi), ranked by blocks as the stage kernels are
// (qb_block.cuh, qb_factor.cuh), in the unweighted basis:
//
//   direct     per row and pair (r, s), sqrt(n_r (n_s - d)) sum_c G_c sqrt((n_p + 1)(n_q + 1 + d_pq)) psi_target
//   factored   g_k(m) = lam_k sum_{p <= q in k} c_pq sqrt((m_p + 1)(m_q + 1 + d)) psi(m + e_p + e_q), then
//              sum_{r <= s} c_rs sqrt(n_r (n_s - d)) g_{r+s}(n - e_r - e_s)
//
// FP64 runs at 1/64 of the FP32 rate: 4 operations a term and 4 a pair are 3.2 ms of the
// direct M = 11, N = 20 sector (2.7M kets, 396M terms); the factored passes take 3 a pair each,
// 0.9 ms.
#include <cuda_runtime.h>

#include <mutex>

#include "qb_factor.cuh"
#include "qb_internal.h"

namespace qb {

// Share of the records (Tables::bk_share) up to which each lane walks its own ket's.  All records in
// step / own (us): M = 16, 969 kets (0.02) 216 / 57; M = 14, 116,280 (0.1) 711 / 255; M = 11, 167,960
// (0.19) 588 / 306; M = 8, 43,758 (0.29) 118 / 107; M = 6, 5,005 (0.34) 44 / 48; M = 7, 50,388 (0.39)
// 93 / 83, M = 6, 38,760 (0.48) 52 / 56.
constexpr float kHpsiShare = 0.3f;

struct HpsiArgs {
  const double2* psi;
  double2* out;
  double2* g;  // factored: [fa_nG]
  int* status;
};

// n_m as an integer
template <int NW>
__device__ __forceinline__ int occ_int(const uint32_t (&ob)[NW], int m) {
  const bool m8 = m >= 8;
  return (int)(__byte_perm(m8 ? ob[2] : ob[0], m8 ? ob[3] : ob[1], (uint32_t)(m & 7)) & 0xffu);
}

// the row's one-body sum; with DIAG also its two-body diagonal, pairs in order
template <bool DIAG>
__device__ __forceinline__ double row_diag(const Tables& t, const uint32_t (&ob)[4], const double* w, const double* gd) {
  double d = 0.0, dl = 0.0;
  for (int m = 0; m < t.M; ++m) d += w[m] * occ_int<4>(ob, m);
  if (DIAG) {
    int ai = 0;
    for (int r = 0; r < t.M; ++r)
      for (int s = r; s < t.M; ++s, ++ai) {
        const int k = occ_int<4>(ob, r) * (occ_int<4>(ob, s) - (r == s ? 1 : 0));
        if (k > 0) dl += gd[ai] * (double)k;
      }
  }
  return d + dl;
}

// SPARSE: each lane walks the records of its own ket (qb_block.cuh, sparse_stage_kernel), with the
// same sums.
template <int KC, bool CPLX, bool SPARSE>
__global__ void __launch_bounds__(512, 2) hpsi_direct_kernel(const Tables t, const HpsiArgs a) {
  constexpr int NT = Rec<KC>::n, RW = Rec<KC>::w;
  const int T = t.bk_T, nrec = t.bk_nrec, M = t.M;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
  double* ssq = reinterpret_cast<double*>(blk_smem);       // [nmax + 3] sqrt(k)
  double* sw = ssq + t.nmax + 3;                           // [M]
  double* sgd = sw + M;                                    // [n_ann]
  double2* sG = reinterpret_cast<double2*>(blk_smem + (((t.nmax + 3 + M + t.n_ann) * 8 + 15) & ~15));  // [T]
  uint2* sinfo = reinterpret_cast<uint2*>(sG + T);         // [nrec]
  uint32_t* spq = reinterpret_cast<uint32_t*>(sinfo + nrec);  // [T] p | q << 8
  for (int i = threadIdx.x; i < t.nmax + 3; i += blockDim.x) ssq[i] = __ldg(reinterpret_cast<const double*>(t.blob + t.o_sqrt) + i);
  for (int i = threadIdx.x; i < M; i += blockDim.x) sw[i] = __ldg(reinterpret_cast<const double*>(t.blob + t.o_w) + i);
  for (int i = threadIdx.x; i < t.n_ann; i += blockDim.x) sgd[i] = __ldg(reinterpret_cast<const double*>(t.blob + t.o_gd) + i);
  for (int i = threadIdx.x; i < T; i += blockDim.x) {
    const uint32_t j = __ldg(t.bk_combo + i);  // combo of the slot, or none
    sG[i] = j == 0xffffffffu ? make_double2(0.0, 0.0) : __ldg(reinterpret_cast<const double2*>(t.blob + t.o_G) + j);
    spq[i] = j == 0xffffffffu ? 0u : __ldg(reinterpret_cast<const uint32_t*>(t.blob + t.o_pq) + j) & 0xffffu;
  }
  for (int i = threadIdx.x; i < nrec; i += blockDim.x) sinfo[i] = __ldg(t.bk_info + i);
  __syncthreads();
  uint16_t* first = reinterpret_cast<uint16_t*>(spq + T);
  if (SPARSE) first_records(sinfo, nrec, first);
  const int64_t total = t.total, step = (int64_t)gridDim.x * warps;
  int64_t rd = (total - 1) / 32 - ((int64_t)blockIdx.x * warps + warp);
  for (; rd >= 0; rd -= step) {
    const int64_t g = rd * 32 + lane;
    const bool valid = g < total;
    const RoundIn in = load_round(t.occ, t.fill, t.rblk, rd, total, lane);
    const uint32_t* base = t.bk_base + (size_t)block_of_lane(in, lane, valid) * T;
    const unsigned char* mp = t.bk_map + (size_t)in.fill * (2 * RW);
    const uint16_t* mp5 = t.bk_map5 + in.fill;
    uint32_t ob[4];
    unpack_occ<0, 4>(t, valid ? in.word : 0ull, ob);  // an invalid lane: no pair acts
    double acc_re = 0.0, acc_im = 0.0, pr = 0.0, pi = 0.0;
    bool bad = false;
    MapRec<KC> mcur;
    BaseRec<KC> bcur;
    RecordWalk walk(t, SPARSE && valid ? in.word : 0ull);
    auto load = [&](int rec) {
      mcur = load_map<KC>(mp + (size_t)rec * t.bk_S * (2 * RW), mp5 + (size_t)rec * t.bk_S);
      bcur = load_base<KC>(base, rec, nrec);
    };
    bool on = SPARSE ? walk.next(sinfo, first) : nrec > 0;
    if (on) load(SPARSE ? walk.rec : 0);
    // (a lane without a further record of its own waits at the loop's end)
    for (int at = 0; SPARSE ? on : at < nrec; ++at) {
      const int rec = SPARSE ? walk.rec : at;
      const MapRec<KC> mnow = mcur;
      const BaseRec<KC> bnow = bcur;
      if (SPARSE) on = walk.next(sinfo, first);
      if (!SPARSE || on) load(SPARSE ? walk.rec : min(at + 1, nrec - 1));
      const uint2 info = sinfo[rec];
      const int r = (int)((info.x & 7) | ((info.x >> 12) & 8)), s = (int)(((info.x >> 16) & 7) | ((info.x >> 28) & 8));
      const int nr = occ_int<4>(ob, r), ns = occ_int<4>(ob, s) - (r == s ? 1 : 0);
      const bool act = nr >= 1 && ns >= 1;
      if (SPARSE ? act : (bool)__any_sync(0xffffffffu, act)) {
        const int n = KC == 0 ? (int)((info.x >> 4) & 7) : NT;
        uint32_t rk[NT];
        rk[0] = bnow.a.x + (mnow.a.x & 0xffffu);
        rk[1] = bnow.a.y + (mnow.a.x >> 16);
        if constexpr (NT > 2) rk[2] = bnow.a.z + (mnow.a.y & 0xffffu);
        if constexpr (NT > 3) rk[3] = bnow.a.w + (mnow.a.y >> 16);
        if constexpr (NT > 4) rk[4] = bnow.b + mnow.b;
        uint32_t top = rk[0];
#pragma unroll
        for (int c = 1; c < NT; ++c)
          if (KC > 0 || c < n) top = max(top, rk[c]);
        const bool ok = act && top < (uint32_t)total;
        bad |= act && !ok;
        if (ok) {
          double2 x[NT];
#pragma unroll
          for (int c = 0; c < NT; ++c)
            if (KC > 0 || c < n) x[c] = __ldg(a.psi + rk[c]);
#pragma unroll
          for (int c = 0; c < NT; ++c) {
            if (KC == 0 && c >= n) continue;
            const int sl = c < 4 ? RW * rec + c : 4 * nrec + rec;
            const int p = spq[sl] & 0xff, q = spq[sl] >> 8;
            const double Bf = ssq[occ_int<4>(ob, p) + 1] * ssq[occ_int<4>(ob, q) + 1 + (p == q ? 1 : 0)];
            const double2 G = sG[sl];
            const double cr = G.x * Bf;
            if (CPLX) {
              const double ci = G.y * Bf;
              pr += cr * x[c].x - ci * x[c].y;
              pi += cr * x[c].y + ci * x[c].x;
            } else {
              pr += cr * x[c].x;
              pi += cr * x[c].y;
            }
          }
          if (KC > 0 || (info.x & 0x80u)) {  // the pair is complete
            const double A = ssq[nr] * ssq[ns];
            acc_re += A * pr;
            acc_im += A * pi;
            pr = pi = 0.0;
          }
        }
      }
    }
    __syncwarp();
    if (bad) atomicOr(a.status, 1);
    if (valid) {
      const double dg = row_diag<true>(t, ob, sw, sgd);
      const double2 x = a.psi[g];
      a.out[g] = make_double2(dg * x.x + acc_re, dg * x.y + acc_im);
    }
  }
}

// modes of an annihilation slot (p | q << 8), from the pairs of its class
template <int NT>
__global__ void __launch_bounds__(1024, 1) hpsi_ann_kernel(const Tables t, const HpsiArgs a) {
  constexpr int PL = NT > 4 ? 2 : 1, NS = NT > 0 ? NT : 4;
  const int nrec = t.fa_nrec, nc = t.fa_nc, Ta = fa_Ta(t);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
  double* ssq = reinterpret_cast<double*>(blk_smem);  // [nmax + 3]
  double* slam = ssq + t.nmax + 3;                    // [nc]
  uint2* srec = reinterpret_cast<uint2*>(slam + nc);  // [nrec]
  uint32_t* spq = reinterpret_cast<uint32_t*>(srec + nrec);  // [Ta] p | q << 8
  for (int i = threadIdx.x; i < t.nmax + 3; i += blockDim.x) ssq[i] = __ldg(reinterpret_cast<const double*>(t.blob + t.o_sqrt) + i);
  for (int i = threadIdx.x; i < nc; i += blockDim.x) slam[i] = __ldg(t.fa_lam64 + i);
  for (int i = threadIdx.x; i < nrec; i += blockDim.x) srec[i] = __ldg(t.fa_rec + i);
  for (int i = threadIdx.x; i < Ta; i += blockDim.x) spq[i] = __ldg(t.fa_pqa + i);
  __syncthreads();
  const int64_t total = t.total, step = (int64_t)gridDim.x * warps;
  for (int64_t rd = (t.fa_low - 1) / 32 - ((int64_t)blockIdx.x * warps + warp); rd >= 0; rd -= step) {
    const int64_t rn = t.fa_perm ? (int64_t)__ldg(t.fa_perm + rd) : rd;
    const int64_t g = rn * 32 + lane;
    const bool valid = g < t.fa_low;
    const RoundIn in = load_round(t.fa_occ, t.fa_fill, t.fa_rblk, rn, t.fa_low, lane);
    const uint32_t* base = t.fa_basea + (size_t)block_of_lane(in, lane, valid) * fa_rowa(t);
    const uint32_t* gb = base + Ta;
    const uint2* mp = t.fa_mapa + in.fill;
    uint32_t ob[4];
    unpack_occ<0, 4>(t, in.word, ob);
    const uint32_t mask = nrec > 32 ? ~0u : __reduce_or_sync(0xffffffffu, valid ? __ldg(gb + nc) : 0u);
    double re = 0.0, im = 0.0;
    bool bad = false;
    for (int rec = 0; rec < nrec; ++rec) {
      if (nrec <= 32 && !((mask >> rec) & 1u)) continue;
      uint32_t ix[NS];
      const uint4 b0 = __ldg(reinterpret_cast<const uint4*>(base) + rec * PL);
      const uint2 m0 = __ldg(mp + (size_t)(rec * PL) * t.bk_S);
      ix[0] = b0.x + (m0.x & 0xffffu);
      ix[1] = b0.y + (m0.x >> 16);
      ix[2] = b0.z + (m0.y & 0xffffu);
      if constexpr (NS > 3) ix[3] = b0.w + (m0.y >> 16);
      if constexpr (NS > 4) {
        const uint4 b1 = __ldg(reinterpret_cast<const uint4*>(base) + rec * PL + 1);
        const uint2 m1 = __ldg(mp + (size_t)(rec * PL + 1) * t.bk_S);
        ix[4] = b1.x + (m1.x & 0xffffu);
        if constexpr (NS > 5) ix[5] = b1.y + (m1.x >> 16);
      }
      const bool act = valid && b0.x != kNoIndex;
      if (!__any_sync(0xffffffffu, act)) continue;
      const uint32_t info = srec[rec].x;
      const int n = (int)((info >> 8) & 15), k = (int)(info & 0xffu);
      uint32_t top = ix[0];
#pragma unroll
      for (int c = 1; c < NS; ++c)
        if (c < n) top = max(top, ix[c]);
      const bool ok = act && top < (uint32_t)total;
      bad |= act && !ok;
      if (!ok) continue;
      double2 x[NS];
#pragma unroll
      for (int c = 0; c < NS; ++c)
        if (c < n) x[c] = __ldg(a.psi + ix[c]);
#pragma unroll
      for (int c = 0; c < NS; ++c) {
        if (c >= n) continue;
        const uint32_t pq = spq[rec * PL * 4 + c];
        const int p = pq & 0xff, q = pq >> 8;
        double cf = ssq[occ_int<4>(ob, p) + 1] * ssq[occ_int<4>(ob, q) + 1 + (p == q ? 1 : 0)];
        if (p != q) cf += cf;  // both orders
        re += cf * x[c].x;
        im += cf * x[c].y;
      }
      if (info & 0x10000u) {  // the class is complete
        a.g[__ldg(gb + k) + (uint32_t)g] = make_double2(slam[k] * re, slam[k] * im);
        re = im = 0.0;
      }
    }
    if (bad) atomicOr(a.status, 1);
  }
}

__global__ void __launch_bounds__(1024, 1) hpsi_cre_kernel(const Tables t, const HpsiArgs a) {
  const int ng = t.fa_ng, Tc = fa_Tc(t), M = t.M;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
  double* ssq = reinterpret_cast<double*>(blk_smem);  // [nmax + 3]
  double* sw = ssq + t.nmax + 3;                      // [M]
  uint32_t* sinfo = reinterpret_cast<uint32_t*>(sw + M);  // [Tc]
  for (int i = threadIdx.x; i < t.nmax + 3; i += blockDim.x) ssq[i] = __ldg(reinterpret_cast<const double*>(t.blob + t.o_sqrt) + i);
  for (int i = threadIdx.x; i < M; i += blockDim.x) sw[i] = __ldg(reinterpret_cast<const double*>(t.blob + t.o_w) + i);
  for (int i = threadIdx.x; i < Tc; i += blockDim.x) sinfo[i] = __ldg(reinterpret_cast<const uint32_t*>(t.fa_info) + i);
  __syncthreads();
  const uint32_t nG = (uint32_t)t.fa_nG;
  const int npair = M * (M + 1) / 2;
  const int64_t total = t.total, step = (int64_t)gridDim.x * warps;
  for (int64_t rd = (total - 1) / 32 - ((int64_t)blockIdx.x * warps + warp); rd >= 0; rd -= step) {
    const int64_t g = rd * 32 + lane;
    const bool valid = g < total;
    const RoundIn in = load_round(t.occ, t.fill, t.rblk, rd, total, lane);
    const uint4* base = reinterpret_cast<const uint4*>(t.fa_basec) + (size_t)block_of_lane(in, lane, valid) * ng;
    const uint2* mp = t.fa_mapc + in.fill;
    uint32_t ob[4];
    unpack_occ<0, 4>(t, valid ? in.word : 0ull, ob);  // an invalid lane: no pair acts
    double re = 0.0, im = 0.0;
    bool bad = false;
    uint2 mcur = __ldg(mp);
    uint4 bcur = __ldg(base);
    for (int gi = 0; gi < ng; ++gi) {
      const int nx = min(gi + 1, ng - 1);
      const uint2 mnext = __ldg(mp + (size_t)nx * t.bk_S);
      const uint4 bnext = __ldg(base + nx);
      const uint32_t ix[4] = {bcur.x + (mcur.x & 0xffffu), bcur.y + (mcur.x >> 16), bcur.z + (mcur.y & 0xffffu),
                              bcur.w + (mcur.y >> 16)};
      double2 x[4];
      int nr[4], ns[4];
      bool ok[4];
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const uint32_t sel = sinfo[4 * gi + c];
        const int r = (int)((sel & 7) | ((sel >> 12) & 8)), s = (int)(((sel >> 16) & 7) | ((sel >> 28) & 8));
        nr[c] = occ_int<4>(ob, r);
        ns[c] = occ_int<4>(ob, s) - (r == s ? 1 : 0);
        const bool act = 4 * gi + c < npair && nr[c] >= 1 && ns[c] >= 1;
        ok[c] = act && ix[c] < nG;
        bad |= act && !ok[c];
        if (ok[c]) x[c] = __ldg(a.g + ix[c]);
      }
#pragma unroll
      for (int c = 0; c < 4; ++c)
        if (ok[c]) {
          double cf = ssq[nr[c]] * ssq[ns[c]];
          if (4 * gi + c < npair - M) cf += cf;  // r < s: both orders
          re += cf * x[c].x;
          im += cf * x[c].y;
        }
      mcur = mnext;
      bcur = bnext;
    }
    if (bad) atomicOr(a.status, 1);
    if (valid) {
      const double dg = row_diag<false>(t, ob, sw, nullptr);
      const double2 x = a.psi[g];
      a.out[g] = make_double2(dg * x.x + re, dg * x.y + im);
    }
  }
}

template <typename K>
static int hpsi_run(K k, const Tables& t, const HpsiArgs& a, int64_t rows, int max_warps, size_t smem, cudaStream_t st) {
  int warps = 0, grid = 0;
  const int rc = stage_geometry(k, rows, 0, max_warps, smem, &warps, &grid);
  if (rc) return rc;
  k<<<grid, 32 * warps, smem, st>>>(t, a);
  QB_CUDA(cudaGetLastError());
  return QB_OK;
}

template <int KC, bool CPLX>
static int hpsi_direct(const Tables& t, const HpsiArgs& a, cudaStream_t st) {
  const size_t smem = (((size_t)(t.nmax + 3 + t.M + t.n_ann) * 8 + 15) & ~(size_t)15) + (size_t)t.bk_T * 20 + (size_t)t.bk_nrec * 8;
  if (t.bk_share < kHpsiShare) return hpsi_run(hpsi_direct_kernel<KC, CPLX, true>, t, a, t.total, 16, smem + kFirstBytes, st);
  return hpsi_run(hpsi_direct_kernel<KC, CPLX, false>, t, a, t.total, 16, smem, st);
}

int launch_hpsi(Space& s, const void* d_v, void* d_out, void* stream) {
  cudaStream_t st = (cudaStream_t)stream;
  const Tables& t = s.t;
  HpsiArgs a{};
  a.psi = (const double2*)d_v;
  a.out = (double2*)d_out;
  a.status = reinterpret_cast<int*>(s.d_scratch);
  int rc = QB_OK;
  if (!t.fa_on) {
    if (t.is_complex) {
      rc = hpsi_direct<0, true>(t, a, st);
    } else {
      switch (t.bk_kc) {
        case 2: rc = hpsi_direct<2, false>(t, a, st); break;
        case 3: rc = hpsi_direct<3, false>(t, a, st); break;
        case 4: rc = hpsi_direct<4, false>(t, a, st); break;
        case 5: rc = hpsi_direct<5, false>(t, a, st); break;
        default: rc = hpsi_direct<0, false>(t, a, st); break;
      }
    }
    if (rc) return rc;
    return check_status(s, st);
  }
  // The vector of B_k psi is the space's, made by the first call; the call holds it until
  // its work is done.  Without the memory for it the rows are ranked one by one.
  std::lock_guard<std::mutex> lock(s.hpsi_mu);
  if (!s.d_hpsi && cudaMalloc(&s.d_hpsi, sizeof(double2) * (size_t)t.fa_nG) != cudaSuccess) {
    cudaGetLastError();
    s.d_hpsi = nullptr;
    rc = launch_hpsi_rows(s, d_v, d_out, st);
    return rc ? rc : check_status(s, st);
  }
  a.g = reinterpret_cast<double2*>(s.d_hpsi);
  const size_t sa = (size_t)(t.nmax + 3 + t.fa_nc) * 8 + (size_t)t.fa_nrec * 8 + (size_t)fa_Ta(t) * 4;
  switch (t.fa_nt) {
    case 4: rc = hpsi_run(hpsi_ann_kernel<4>, t, a, t.fa_low, 32, sa, st); break;
    case 5: rc = hpsi_run(hpsi_ann_kernel<5>, t, a, t.fa_low, 32, sa, st); break;
    case 6: rc = hpsi_run(hpsi_ann_kernel<6>, t, a, t.fa_low, 32, sa, st); break;
    default: rc = t.fa_nt == 0 ? hpsi_run(hpsi_ann_kernel<0>, t, a, t.fa_low, 32, sa, st)
                               : fail(QB_EINTERNAL, "pairs a class");
  }
  if (!rc) rc = hpsi_run(hpsi_cre_kernel, t, a, t.total, 32, (size_t)(t.nmax + 3 + t.M) * 8 + (size_t)fa_Tc(t) * 4, st);
  // (on an error the stream is drained too: the next call reuses the vector)
  if (rc) {
    cudaStreamSynchronize(st);
    return rc;
  }
  return check_status(s, st);
}

}  // namespace qb
