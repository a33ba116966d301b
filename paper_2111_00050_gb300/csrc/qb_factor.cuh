// The RK4 stage of couplings that factor by momentum class (a contact interaction):
//
//   H_2 = sum_k lam_k B_k^dag B_k,   B_k = sum over ordered (p, q) of class k of a_p a_q
//
// (class k: p + q = k mod M, or p + q = k with exact momentum).  Instead of the pairs
// {r, s} -> {p, q} one by one, (M + 1) / 2 times more terms, a stage makes two passes:
//
//   ann_kernel   g_k(m) = lam_k sum_{p <= q in k} c_pq f(m + e_p + e_q) on the kets m of two
//                particles fewer, c = 2 - [p = q].  In the weighted basis the annihilation
//                pair has no further factor: the products are sums.
//   cre_kernel   (W^-1 H_2 W f)(n) = sum_{r <= s} c_rs n_r (n_s - [r = s]) g_{r+s}(n - e_r - e_s),
//                the factor an exact integer, then the stage's epilogue.
//
// Per ket of M = 7 (N = 36) that is 41 gathers and 41 sums of 8 or 11 operations instead of
// 62 of 14.  Both passes rank by blocks as the direct kernel does (qb_block.cuh): the map of
// a pair holds the place of a filling after the pair is added or taken away.
#pragma once
#include "qb_block.cuh"

namespace qb {

inline size_t ann_smem_bytes(const Tables& t) { return ((size_t)t.fa_nrec * 8 + t.fa_nc * 8 + 15) & ~(size_t)15; }

// Rows of bases per lower block: the annihilation slots, then where each class's entries
// start less the number of the lower ket.  kNoIndex: the raised sector is not held.

// DOT: no vector; sum_k lam_k |B_k psi|^2 over CTAs, partial[block].  A ket's values are scaled by
// the power of two of its weight and the sum over its classes, formed in double-float, by the
// rest squared in FP64: the weight rounded to 48 bits erred alike in the many kets that share it
// (positive states of 245,157 kets, M = 7, against 64 bits 1.1e-15, now 4e-16, the direct form 7e-16).
// EVERY: every record of every lower ket is taken (all momenta held).
// SIDE: member blockIdx.y of a sweep, with a vector of its own (here and below).
template <int NT, bool DOT, bool EVERY, bool SIDE>
__global__ void __launch_bounds__(1024, 1) ann_kernel(const Tables t, const DfArgs a) {
  constexpr int PL = NT > 4 ? 2 : 1;       // groups of four pairs a record
  constexpr int NS = NT > 0 ? NT : 4;      // pairs of a record
  const int nrec = t.fa_nrec, nc = t.fa_nc;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
  uint2* srec = reinterpret_cast<uint2*>(blk_smem);
  float2* slam = reinterpret_cast<float2*>(srec + nrec);
  for (int i = threadIdx.x; i < nrec; i += blockDim.x) srec[i] = __ldg(t.fa_rec + i);
  for (int i = threadIdx.x; i < nc; i += blockDim.x) slam[i] = __ldg(t.fa_lam + i);
  __syncthreads();
  const int64_t total = t.total;
  const float4* vin = a.vin + (SIDE ? (size_t)blockIdx.y * total : 0);
  float4* g_out = a.g + (SIDE ? (size_t)blockIdx.y * t.fa_nG : 0);
  double dot64 = 0.0;

  // Rounds of a layer are taken in an order that walks its sectors side by side (fa_perm):
  // a ket f(n) is read from every lower sector, at about the same place, and is still in
  // L1 / L2 then.  (A launch over part of the lower kets takes them as they come.)
  const uint32_t* perm = a.low0 == 0 && a.low1 == t.fa_low ? t.fa_perm : nullptr;
  const int64_t r0 = a.low0 / 32, step = (int64_t)gridDim.x * warps;
  int64_t rd = (a.low1 - 1) / 32 - ((int64_t)blockIdx.x * warps + warp);
  auto round_of = [&](int64_t r) { return perm ? (int64_t)__ldg(perm + max(r, r0)) : max(r, r0); };
  int64_t rn = round_of(rd), rn2 = round_of(rd - step);
  RoundIn next = load_round(t.fa_occ, t.fa_fill, t.fa_rblk, rn, t.fa_low, lane);
  chain_wait();
  for (; rd >= r0; rd -= step) {
      const int64_t g = rn * 32 + lane;
      const bool valid = g >= a.low0 && g < a.low1;
      const RoundIn in = next;
      rn = rn2;
      next = load_round(t.fa_occ, t.fa_fill, t.fa_rblk, rn, t.fa_low, lane);
      rn2 = round_of(rd - 2 * step);
      const uint32_t* base = t.fa_basea + (size_t)block_of_lane(in, lane, g < t.fa_low) * fa_rowa(t);
      const uint32_t* gb = base + fa_Ta(t);
      const uint2* mp = t.fa_mapa + in.fill;
      float w2 = 1.f;    // the power of two of the weight, for the values
      double wm2 = 0.0;  // and the square of the rest, for the ket's sum
      dfl dsum{0.f, 0.f};
      if (DOT && valid) {  // w(m) sqrt(N (N - 1)) with the centring powers of two, N the raised number
        int rem = 0;
        for (int m = 0; m < t.M; ++m) rem += occ_of(in.word, m, t.occ_bits);
        const double w = t.fa_wk ? __ldg(t.fa_wk + g) : ket_weight_word<0>(t, in.word).x;
        const double c = sqrt((double)(rem + 2) * (rem + 1)) * __ldg(t.wscale + rem + 2).x * __ldg(t.wscale + rem).y;
        const uint32_t hw = (uint32_t)__double2hiint(w * c);
        const double m = __hiloint2double((int)((hw & 0xfffffu) | 0x3ff00000u), __double2loint(w * c));
        w2 = __uint_as_float((((hw >> 20) & 0x7ffu) - 896u) << 23);  // within 2^+-90
        wm2 = m * m;
      }
      bool bad = false;
      dfc acc{0ull, 0ull};
      float4 x[NS];
#pragma unroll
      for (int c = 0; c < NS; ++c) x[c] = make_float4(0.f, 0.f, 0.f, 0.f);
      // the records whose raised sector some lane's block has (one class of M where the
      // space holds one momentum)
      uint32_t mask = ~0u;
      if (!EVERY && nrec <= 32) mask = __reduce_or_sync(0xffffffffu, valid ? __ldg(gb + nc) : 0u);
      uint2 mcur[PL];
      uint4 bcur[PL];
      auto load = [&](int rec) {
#pragma unroll
        for (int p = 0; p < PL; ++p) {
          mcur[p] = __ldg(mp + (size_t)(rec * PL + p) * t.bk_S);
          bcur[p] = __ldg(reinterpret_cast<const uint4*>(base) + rec * PL + p);
        }
      };
      auto following = [&](int rec) {  // the next record to take, or nrec
        if (EVERY || nrec > 32) return rec + 1;
        const uint32_t rest = rec < 31 ? mask & (~0u << (rec + 1)) : 0u;
        return rest ? __ffs(rest) - 1 : nrec;
      };
      int rec = EVERY || (mask & 1u) ? 0 : following(0);
      if (rec < nrec) load(rec);
      for (int rnext; rec < nrec; rec = rnext) {
        rnext = following(rec);
        uint32_t ix[NS];
        ix[0] = bcur[0].x + (mcur[0].x & 0xffffu);
        ix[1] = bcur[0].y + (mcur[0].x >> 16);
        ix[2] = bcur[0].z + (mcur[0].y & 0xffffu);
        if constexpr (NS > 3) ix[3] = bcur[0].w + (mcur[0].y >> 16);
        if constexpr (NS > 4) ix[4] = bcur[PL - 1].x + (mcur[PL - 1].x & 0xffffu);
        if constexpr (NS > 5) ix[5] = bcur[PL - 1].y + (mcur[PL - 1].x >> 16);
        const bool act = valid && bcur[0].x != kNoIndex;
        if (rnext < nrec) load(rnext);
        if (!__any_sync(0xffffffffu, act)) continue;
        const uint32_t info = srec[rec].x;
        const int n = NT > 0 ? NT : (int)((info >> 8) & 15), dbl = NT > 0 ? NT - 1 : (int)((info >> 12) & 7);
        uint32_t top = ix[0];
#pragma unroll
        for (int c = 1; c < NS; ++c)
          if (NT > 0 || c < n) top = max(top, ix[c]);
        const bool ok = act && top < (uint32_t)total;
        bad |= act && !ok;
#pragma unroll
        for (int c = 0; c < NS; ++c)
          if (ok && (NT > 0 || c < n)) x[c] = vin[ix[c]];
        if constexpr (NT > 0) {
          acc = dfc{f2_pack(x[0].x, x[0].y), f2_pack(x[0].z, x[0].w)};
        } else {
          if (dbl == 0) acc = dfc{f2_add(acc.h, acc.h), f2_add(acc.l, acc.l)};
          dfc_add(acc, f2_pack(x[0].x, x[0].y), f2_pack(x[0].z, x[0].w));
        }
#pragma unroll
        for (int c = 1; c < NS; ++c) {
          if (c == dbl) acc = dfc{f2_add(acc.h, acc.h), f2_add(acc.l, acc.l)};
          if (c < n) dfc_add(acc, f2_pack(x[c].x, x[c].y), f2_pack(x[c].z, x[c].w));
        }
        if (NT == 0 && dbl == 4) acc = dfc{f2_add(acc.h, acc.h), f2_add(acc.l, acc.l)};
        if (NT > 0 || (info & 0x10000u) != 0u) {  // the class is complete
          const int k = NT > 0 ? rec : (int)(info & 0xffu);
          const float2 lm = slam[k];
          const dfc sm = dfc_renorm(acc);
          dfl gr, gi;
          f2_unpack(sm.h, gr.h, gi.h);
          f2_unpack(sm.l, gr.l, gi.l);
          if constexpr (DOT) {
            gr = dfl{w2 * gr.h, w2 * gr.l};
            gi = dfl{w2 * gi.h, w2 * gi.l};
            const dfl v = df_mul(dfl{lm.x, lm.y}, df_add(df_mul(gr, gr), df_mul(gi, gi)));
            if (ok) dsum = df_add(dsum, v);
          } else {
            gr = df_renorm(df_mul(dfl{lm.x, lm.y}, gr));
            gi = df_renorm(df_mul(dfl{lm.x, lm.y}, gi));
            if (ok) g_out[__ldg(gb + k) + (uint32_t)g] = df_pack(gr, gi);
          }
          acc = dfc{0ull, 0ull};
        }
      }
      if (bad) atomicOr(a.status, 1);
      if (DOT) dot64 += df_to(dsum) * wm2;
  }
  if constexpr (DOT) {
    __shared__ double red[32];
    for (int o = 16; o > 0; o >>= 1) dot64 += __shfl_down_sync(0xffffffffu, dot64, o);
    if (lane == 0) red[warp] = dot64;
    __syncthreads();
    if (threadIdx.x == 0) {
      double sum = 0.0;
      for (int w = 0; w < warps; ++w) sum += red[w];
      a.partial[blockIdx.x] = sum;
    }
  }
}

// the creation pairs in order: r < s, then r = s
template <int MT>
struct PairList {
  int r[MT * (MT + 1) / 2], s[MT * (MT + 1) / 2];
  constexpr PairList() : r(), s() {
    int i = 0;
    for (int p = 0; p < MT; ++p)
      for (int q = p + 1; q < MT; ++q, ++i) {
        r[i] = p;
        s[i] = q;
      }
    for (int p = 0; p < MT; ++p, ++i) r[i] = s[i] = p;
  }
};

inline size_t cre_smem_bytes(const Tables& t, int MT) { return MT > 0 ? 0 : (size_t)fa_Tc(t) * 12; }

template <int MT, int KIND, bool SIDE>
__global__ void __launch_bounds__((blk_max_threads<1, KIND>()), 1)
    cre_kernel(const Tables t, const DfArgs a, const int mode) {
  constexpr int NW = occ_words<MT>();
  constexpr bool BIL = (KIND == KIND_BIL);
  constexpr int kMB = (MT > 0) ? MT : 16;
  const int M = (MT > 0) ? MT : t.M;
  const int ng = t.fa_ng;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
  uint4* sinfo = reinterpret_cast<uint4*>(blk_smem);
  float4* scoef = reinterpret_cast<float4*>(sinfo + ng);
  if constexpr (MT == 0) {  // else the pairs are constants
    for (int i = threadIdx.x; i < ng; i += blockDim.x) sinfo[i] = __ldg(t.fa_info + i);
    for (int i = threadIdx.x; i < 2 * ng; i += blockDim.x) scoef[i] = __ldg(t.fa_coef + i);
    __syncthreads();
  }
  const uint32_t nG = (uint32_t)t.fa_nG;
  const float4* g_in = a.g + (SIDE ? (size_t)blockIdx.y * nG : 0);
  dfl bil_l{0.f, 0.f};
  dfc bil_w[BIL ? (kMB + 1) / 2 : 1];
#pragma unroll
  for (int q = 0; q < (BIL ? (kMB + 1) / 2 : 1); ++q) bil_w[q] = dfc{0ull, 0ull};
  double dot64 = 0.0;

  const int64_t r0 = a.row0 / 32, step = (int64_t)gridDim.x * warps;
  int64_t rd = (a.row1 - 1) / 32 - ((int64_t)blockIdx.x * warps + warp);
  RoundIn next = load_round(t.occ, t.fill, t.rblk, max(rd, r0), t.total, lane);
  chain_wait();
  for (; rd >= r0; rd -= step) {
      const int64_t g = rd * 32 + lane;
      const bool valid = g >= a.row0 && g < a.row1;
      const RoundIn in = next;
      next = load_round(t.occ, t.fill, t.rblk, max(rd - step, r0), t.total, lane);
      const uint4* base = reinterpret_cast<const uint4*>(t.fa_basec) + (size_t)block_of_lane(in, lane, g < t.total) * ng;
      uint32_t ob[NW];
      unpack_occ<MT, NW>(t, valid ? in.word : 0ull, ob);  // an invalid lane: no pair acts
      const uint2* mp = t.fa_mapc + in.fill;
      dfc acc[1] = {dfc{0ull, 0ull}};
      bool bad = false;
      if constexpr (MT > 0) {
        // unrolled: the pairs are constants, a factor is one product of two registers; the
        // pairs r < s first, their sum doubled, then the pairs r = s
        constexpr PairList<MT> pr{};
        constexpr int NP = MT * (MT + 1) / 2, NO = MT * (MT - 1) / 2, NG = (NP + 3) / 4;
        float nf[MT];
#pragma unroll
        for (int m = 0; m < MT; ++m) nf[m] = occ_float<NW>(ob, m);
        float4 x[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) x[c] = make_float4(0.f, 0.f, 0.f, 0.f);
        uint2 mcur = __ldg(mp);
        uint4 bcur = __ldg(base);
#pragma unroll
        for (int gi = 0; gi < NG; ++gi) {
          const uint32_t ix[4] = {bcur.x + (mcur.x & 0xffffu), bcur.y + (mcur.x >> 16), bcur.z + (mcur.y & 0xffffu),
                                  bcur.w + (mcur.y >> 16)};
          if (gi + 1 < NG) {
            mcur = __ldg(mp + (size_t)(gi + 1) * t.bk_S);
            bcur = __ldg(base + gi + 1);
          }
          float A[4];
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            const int i = 4 * gi + c;
            if (i >= NP) break;
            A[c] = i < NO ? nf[pr.r[i]] * nf[pr.s[i]] : nf[pr.r[i]] * (nf[pr.r[i]] - 1.f);  // exact
            const bool act = A[c] != 0.f, ok = act && ix[c] < nG;
            bad |= act && !ok;
            if (ok) x[c] = g_in[ix[c]];
          }
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            const int i = 4 * gi + c;
            if (i >= NP) break;
            if (i == NO) acc[0] = dfc{f2_add(acc[0].h, acc[0].h), f2_add(acc[0].l, acc[0].l)};
            if (__any_sync(0xffffffffu, A[c] != 0.f))
              dfc_fma_int(acc[0], f2_pack(A[c], A[c]), f2_pack(-A[c], -A[c]), f2_pack(x[c].x, x[c].y),
                          f2_pack(x[c].z, x[c].w));
          }
          acc[0] = dfc_renorm(acc[0]);  // keep |lo| below an ulp of hi
        }
      } else {
        float4 x[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) x[c] = make_float4(0.f, 0.f, 0.f, 0.f);
        uint2 mcur = __ldg(mp);
        uint4 bcur = __ldg(base);
        for (int gi = 0; gi < ng; ++gi) {
          if (gi + 1 < ng) {
            mp += t.bk_S;
            ++base;
          }
          const uint2 mnext = __ldg(mp);
          const uint4 bnext = __ldg(base);
          const uint4 sl = sinfo[gi];
          const float4 ca = scoef[2 * gi], cb = scoef[2 * gi + 1];
          const uint32_t sel[4] = {sl.x, sl.y, sl.z, sl.w};
          const float del[4] = {ca.x, ca.z, cb.x, cb.z}, mul[4] = {ca.y, ca.w, cb.y, cb.w};
          const uint32_t ix[4] = {bcur.x + (mcur.x & 0xffffu), bcur.y + (mcur.x >> 16), bcur.z + (mcur.y & 0xffffu),
                                  bcur.w + (mcur.y >> 16)};
          float A[4];
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            A[c] = (occ_float23<NW>(ob, sel[c], (sel[c] & 0x8000u) != 0u) - 8388608.0f) * mul[c] *
                   (occ_float23<NW>(ob, sel[c] >> 16, (sel[c] & 0x80000000u) != 0u) - del[c]);  // exact
            const bool act = A[c] != 0.f, ok = act && ix[c] < nG;
            bad |= act && !ok;
            if (ok) x[c] = g_in[ix[c]];
          }
#pragma unroll
          for (int c = 0; c < 4; ++c)
            if (__any_sync(0xffffffffu, A[c] != 0.f))
              dfc_fma_int(acc[0], f2_pack(A[c], A[c]), f2_pack(-A[c], -A[c]), f2_pack(x[c].x, x[c].y),
                          f2_pack(x[c].z, x[c].w));
          acc[0] = dfc_renorm(acc[0]);  // keep |lo| below an ulp of hi
          mcur = mnext;
          bcur = bnext;
        }
      }
      if (bad) atomicOr(a.status, 1);
      if (valid)
        stage_epilogue<MT, 1, KIND, true, NW>(t, a, mode, g, SIDE ? g + (int64_t)blockIdx.y * t.total : g, acc, ob, bil_l,
                                              bil_w, dot64, SIDE ? (int)blockIdx.y : 0);
  }
  if constexpr (BIL) bil_reduce<kMB>(a, M, bil_l, bil_w);
}

template <int NT, bool DOT, bool SIDE>
int ann_launch(const Tables& t, const DfArgs& a, int members, int shape, cudaStream_t st, int* grid_out) {
  auto k = t.fa_every ? ann_kernel<NT, DOT, true, SIDE> : ann_kernel<NT, DOT, false, SIDE>;
  const size_t smem = ann_smem_bytes(t);
  int grid = 0, warps = 0;
  const int rc = stage_geometry(k, a.low1 - a.low0, shape, 32, smem, &warps, &grid);
  if (rc) return rc;
  QB_CUDA(chain_launch(k, dim3((unsigned)grid, (unsigned)members), 32 * warps, smem, st, t, a));
  if (grid_out) *grid_out = grid;
  return QB_OK;
}

template <int MT, int KIND, bool SIDE>
int cre_launch(const Tables& t, const DfArgs& a, int mode, int members, int shape, cudaStream_t st, int* grid_out) {
  auto k = cre_kernel<MT, KIND, SIDE>;
  const size_t smem = cre_smem_bytes(t, MT);
  int grid = 0, warps = 0;
  const int rc = stage_geometry(k, a.row1 - a.row0, shape, blk_max_threads<1, KIND>() / 32, smem, &warps, &grid);
  if (rc) return rc;
  QB_CUDA(chain_launch(k, dim3((unsigned)grid, (unsigned)members), 32 * warps, smem, st, t, a, mode));
  if (grid_out) *grid_out = grid;
  return QB_OK;
}

// One stage of a factored space: NT pairs a class (0: any), MT modes (0: any).  The members
// of a sweep take a pass in one launch with a vector g each (side_by_side), or their two passes
// one after the other through one.
template <int MT, int NT>
int fac_launch(const Tables& t, const DfArgs& a0, int mode, int B, bool bil, int shape, cudaStream_t st, int* grid) {
  if (mode < 0 || mode > 4) return fail(QB_EINTERNAL, "bad stage mode");
  if (mode == 4) {
    if (B != 1) return fail(QB_EUNSUPPORTED, "the <x|H|x> reduction runs one state at a time");
    return ann_launch<NT, true, false>(t, a0, 1, shape, st, grid);
  }
  if (bil && B != 1) return fail(QB_EUNSUPPORTED, "bilinear stages run one state at a time");
  if (B != 1 && t.exact) return fail(QB_EUNSUPPORTED, "exact momentum: batched sweeps are not built");
  if (B != 1 && B != 2 && B != 4 && B != 8) return fail(QB_EINVAL, "batch must be 1, 2, 4 or 8");
  const int members = B > 1 && a0.g_members >= B ? B : 1;
  for (int b = 0; b < B; b += members) {
    DfArgs a = a0;
    a.vin += (size_t)b * t.total;
    if (a.psif) a.psif += (size_t)b * t.total;
    if (a.psi) a.psi += (size_t)b * t.total;
    a.out += (size_t)b * t.total;
    if (b > 0) a.scale[0] = a0.scale[b];
    int rc = QB_OK;
    if (a.low1 > a.low0)
      rc = members > 1 ? ann_launch<NT, false, true>(t, a, members, shape, st, nullptr)
                       : ann_launch<NT, false, false>(t, a, 1, shape, st, nullptr);
    if (rc) return rc;
    rc = bil           ? cre_launch<MT, KIND_BIL, false>(t, a, mode, 1, shape, st, grid)
         : members > 1 ? cre_launch<MT, KIND_STAGE, true>(t, a, mode, members, shape, st, grid)
                       : cre_launch<MT, KIND_STAGE, false>(t, a, mode, 1, shape, st, grid);
    if (rc) return rc;
  }
  return QB_OK;
}

}  // namespace qb
