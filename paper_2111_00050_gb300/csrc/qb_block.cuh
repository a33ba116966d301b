// The hot kernel: one Horner RK4 stage of every sector (and every member of a
// batched coupling sweep) in one launch, with the matrix-free sector H psi in
// double-float arithmetic, in the weighted basis f = psi / w(n).
//
//   stage d (d = 4, 3, 2):  out = f + (-i dt/d) W^-1 H W v    (double-float out)
//   stage 1:                psi = psi + (-i dt) H v, f = psi / w
//                                                     (FP64 psi, plus its weighted copy)
//
// H is Eq. (Ham) restricted to sectors of fixed N and momentum (Sec. III B).  Per row
// (ket n) the off-diagonal terms are the disjoint pairs {r, s} -> {p, q} of equal
// momentum; in the weighted basis, w(n) = sqrt(N! / prod n_m!) up to a power of two
// per N, the element of target n' = n - e_r - e_s + e_p + e_q is
// G_{pq,rs} n_r (n_s - [r = s]): the ratio w(n') / w(n) cancels the creation square
// roots and squares the annihilation ones.  G is the multiplicity-summed symmetrised
// coupling; the diagonal is precomputed per ket.
//
// Ranking by blocks.  The kets of a sector that share the occupations of the first P
// modes are consecutive; such a block is the list of fillings of the last M - P modes
// with a given particle number and momentum (its class), the same list wherever that
// class occurs.  A term sends every ket of a block into one target block, so that the
// target's index in the state vector splits into
//   base[block][term]   where the target block starts: one row of 32-bit indices per
//                       block, written when the space is built, and
//   map[term][filling]  where the changed filling stands in its class: 16-bit places,
//                       written once, read in order by consecutive lanes.
// A warp takes 32 consecutive kets, one per lane, and walks the annihilation pairs in
// step: the pair, its couplings and (nearly always) the bases are the same for all
// lanes, the map is read coalesced and the gathered targets are near-consecutive.
#pragma once
#include "qb_device.cuh"

namespace qb {

// What a stage launch computes besides (or instead of) its output vector:
//   KIND_STAGE  the RK4 / adjoint stage alone (modes 0 to 3);
//   KIND_BIL    with the adjoint's bilinears fused (modes 2, 3);
//   KIND_DOT    <x|H|x> only (mode 4): Re(conj(psi_n) (H psi)_n) summed in FP64,
//               with each off-diagonal term and its Hermitian reverse taken once
//               (the partners of a pair that come after it, counted twice).
enum { KIND_STAGE = 0, KIND_BIL = 1, KIND_DOT = 2 };

extern __shared__ __align__(16) unsigned char blk_smem[];

// words of occupation bytes, four modes a word (two at least: occ_float23)
template <int MT>
__host__ __device__ constexpr int occ_words() {
  return MT > 0 ? (MT > 4 ? (MT + 3) / 4 : 2) : 4;
}

// 2^23 + n_m as a float, exactly: the byte becomes the last one of 2^23.  The mode is in
// the low bits of m (three for two or three words, then m8 = mode >= 8; the bits above pick
// bytes that are dropped).
template <int NW>
__device__ __forceinline__ float occ_float23(const uint32_t (&ob)[NW], uint32_t m, bool m8) {
  uint32_t w;
  if constexpr (NW == 2) w = __byte_perm(ob[0], ob[1], m);
  if constexpr (NW == 3) w = __byte_perm(m8 ? ob[2] : ob[0], ob[1], m);
  if constexpr (NW == 4) w = __byte_perm(m8 ? ob[2] : ob[0], m8 ? ob[3] : ob[1], m);
  return __uint_as_float(__byte_perm(w, 0x4B000000u, 0x7650u));
}
// A stage's launch may start while the one before it drains: it stages its tables, then waits
// for that launch's end and lets the next one start.  (Only then: the launch after next must
// not start beside the one before, whose vectors its L1 could keep.)  What earlier stages write
// is read by plain loads, which also cost the gathers less than loads for constant data: a step
// of the 62.9M-ket contact space 19.6 -> 18.8 ms.  The overlap: 100 steps of 245,157 kets at
// M = 7 14.4 -> 14.1 ms, 10 of 230,230 at M = 6 2.09 -> 1.96, nothing where a stage takes 1 ms.
__device__ __forceinline__ void chain_wait() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;");
}
template <typename... P, typename... A>
inline cudaError_t chain_launch(void (*k)(P...), dim3 grid, int block, size_t smem, cudaStream_t st, A... args) {
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t c{};
  c.gridDim = grid;
  c.blockDim = dim3((unsigned)block);
  c.dynamicSmemBytes = smem;
  c.stream = st;
  c.attrs = &at;
  c.numAttrs = 1;
  return cudaLaunchKernelEx(&c, k, P(args)...);
}

// Values that a stage reads once (the kets' words and fillings, the diagonal, the vectors of the
// epilogue) are not kept in L1, whose lines the gathers, the maps and the bases reuse.  One step
// of the M = 9, N = 27 long-range space (23.5M kets) 20.8 -> 20.3 ms, 20 steps with gradient of
// the M = 5, 2.3M-ket space 48.0 -> 47.1; maps read that way cost as much again (55.7).
__device__ __forceinline__ float4 ld_once(const float4* p) {
  float4 v;
  asm volatile("ld.global.L1::no_allocate.v4.f32 {%0, %1, %2, %3}, [%4];"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
               : "l"(p)
               : "memory");
  return v;
}
__device__ __forceinline__ uint64_t ld_once(const uint64_t* p) {
  uint64_t v;
  asm volatile("ld.global.nc.L1::no_allocate.u64 %0, [%1];" : "=l"(v) : "l"(p));
  return v;
}
__device__ __forceinline__ uint32_t ld_once(const uint32_t* p) {
  uint32_t v;
  asm volatile("ld.global.nc.L1::no_allocate.u32 %0, [%1];" : "=r"(v) : "l"(p));
  return v;
}

template <int NW>
__device__ __forceinline__ float occ_float(const uint32_t (&ob)[NW], int m) {
  return occ_float23<NW>(ob, (uint32_t)(m & 7), m >= 8) - 8388608.0f;
}

// Occupation bytes of a packed occupation word
template <int MT, int NW>
__device__ __forceinline__ void unpack_occ(const Tables& t, uint64_t word, uint32_t (&ob)[NW]) {
  constexpr int kMB = (MT > 0) ? MT : 16;
#pragma unroll
  for (int k = 0; k < NW; ++k) ob[k] = 0u;
#pragma unroll
  for (int m = 0; m < kMB; ++m) {
    if (MT == 0 && m >= t.M) break;
    ob[m >> 2] |= (uint32_t)occ_of(word, m, t.occ_bits) << (8 * (m & 3));
  }
}

// Terms per record: KC partners of a pair (odd M, momentum mod M: every pair has
// (M - 1) / 2), or groups of up to four partners (KC = 0).  Slots of a record: the
// first four terms side by side (two for KC = 2), a fifth in an array of its own.
template <int KC>
struct Rec {
  static constexpr int n = KC == 0 ? 4 : KC;
  static constexpr int w = KC == 2 ? 2 : 4;
  static_assert(KC >= 0 && KC <= 5 && KC != 1, "partners per pair");
};

template <int KC>
struct MapRec {  // one filling's map entries of one record
  uint2 a;
  uint32_t b;
};

template <int KC>
__device__ __forceinline__ MapRec<KC> load_map(const unsigned char* mp, const uint16_t* mp5) {
  MapRec<KC> r;
  r.b = 0u;
  if constexpr (KC == 2) {
    r.a = make_uint2(__ldg(reinterpret_cast<const uint32_t*>(mp)), 0u);
  } else {
    r.a = __ldg(reinterpret_cast<const uint2*>(mp));
    if constexpr (KC == 5) r.b = __ldg(mp5);
  }
  return r;
}

template <int KC>
struct BaseRec {  // a block's bases of one record
  uint4 a;
  uint32_t b;
};
template <int KC>
__device__ __forceinline__ BaseRec<KC> load_base(const uint32_t* base, int rec, int nrec) {
  BaseRec<KC> r;
  r.b = 0u;
  if constexpr (KC == 2) {
    const uint2 v = __ldg(reinterpret_cast<const uint2*>(base) + rec);
    r.a = make_uint4(v.x, v.y, 0u, 0u);
  } else {
    r.a = __ldg(reinterpret_cast<const uint4*>(base) + rec);
    if constexpr (KC == 5) r.b = __ldg(base + 4 * nrec + rec);
  }
  return r;
}

// acc += the terms of one record: coefficient G n_r (n_s - [r = s]) = G Af, gathered values x
template <int KC, bool CPLX, bool DOT>
__device__ __forceinline__ void add_record(dfc& acc, const float4 (&x)[Rec<KC>::n], const float2* sG, const float2* sGi,
                                           int rec, int nrec, int n, int c_first, float Af) {
  constexpr int NT = Rec<KC>::n, RW = Rec<KC>::w;
#pragma unroll
  for (int c = 0; c < NT; ++c) {
    if ((KC == 0 && c >= n) || (DOT && c < c_first)) continue;  // the same for all lanes
    const int sl = c < 4 ? RW * rec + c : 4 * nrec + rec;
    const float2 g2 = sG[sl];
    const dfl cr = df_mul_f(dfl{g2.x, g2.y}, Af);
    const f2 xh = f2_pack(x[c].x, x[c].y), xl = f2_pack(x[c].z, x[c].w);
    dfc_fma(acc, f2_pack(cr.h, cr.h), f2_pack(-cr.h, -cr.h), f2_pack(cr.l, cr.l), xh, xl);
    if (CPLX) {
      // + (-c_i x_im, c_i x_re): lanes of x swapped, coefficient (-c_i, c_i)
      const float2 gi = sGi[sl];
      const dfl ci = df_mul_f(dfl{gi.x, gi.y}, Af);
      dfc_fma(acc, f2_pack(-ci.h, ci.h), f2_pack(ci.h, -ci.h), f2_pack(-ci.l, ci.l), f2_pack(x[c].y, x[c].x),
              f2_pack(x[c].w, x[c].z));
    }
  }
}

// Everything of a ket's row that the epilogue needs, and the epilogue: forms the
// stage's output (or the bilinears, or the <x|H|x> summand) from the off-diagonal sum.
// WHOLE: acc is the whole two-body part (factored couplings), else its off-diagonal part.
// RESIDENT: the state's vectors lie in shared memory.  gr: the ket; ri: its entry of the vectors;
// member: of the sweep, the first of B.
template <int MT, int B, int KIND, bool WHOLE, int NW, bool RESIDENT = false>
__device__ __forceinline__ void stage_epilogue(const Tables& t, const DfArgs& a, int mode, int64_t gr, int64_t ri,
                                               const dfc (&acc)[B], const uint32_t (&ob)[NW], dfl& bil_l, dfc* bil_w,
                                               double& dot64, int member = 0) {
  constexpr bool BIL = (KIND == KIND_BIL), DOT = (KIND == KIND_DOT);
  constexpr int kMB = (MT > 0) ? MT : 16;
  const int M = (MT > 0) ? MT : t.M;
  const int64_t total = t.total;
  const float4 dg4 = ld_once(a.diag + gr);
  const dfl zf{a.zf.x, a.zf.y};
  // the ket weight where true values are formed
  double2 wk = make_double2(1.0, 1.0);
  if (BIL || DOT || mode == 1 || mode == 3) wk = make_double2(__ldg(t.wk + gr), __ldg(t.wi + gr));
#pragma unroll
  for (int b = 0; b < B; ++b) {
    dfl acc_r, acc_i;
    f2_unpack(acc[b].h, acc_r.h, acc_i.h);
    f2_unpack(acc[b].l, acc_r.l, acc_i.l);
    if (DOT) {  // each term stands for itself and its reverse (H Hermitian): twice the real part
      acc_r = dfl{2.f * acc_r.h, 2.f * acc_r.l};
      acc_i = dfl{2.f * acc_i.h, 2.f * acc_i.l};
    }
    const dfl sc{a.scale[b + member].x, a.scale[b + member].y};
    const dfl dg = WHOLE ? dfl{dg4.x, dg4.y} : df_add(dfl{dg4.x, dg4.y}, df_mul(sc, dfl{dg4.z, dg4.w}));
    const float4 xo = a.vin[(size_t)b * total + ri];
    const dfl hr = df_add(df_mul(dg, df_re(xo)), df_mul(sc, acc_r));
    const dfl hi = df_add(df_mul(dg, df_im(xo)), df_mul(sc, acc_i));
    if (DOT) {
      // <x|H|x>: Re(conj(psi_n) (H psi)_n) = w^2 Re(conj(f_n) (W^-1 H W f)_n), w^2 in
      // FP64 (w^2 alone may leave the fp32 range); no output
      const dfl val = df_add(df_mul(df_re(xo), hr), df_mul(df_im(xo), hi));
      dot64 += df_to(val) * wk.x * wk.x;
      continue;
    }
    if (BIL && b == 0) {
      // H_L x (two-body part at scale 1) and the pair vector of this row, as true
      // values: each factor times w (w^2 alone may leave the fp32 range)
      const float4 pp = ld_once(a.pair + ri);
      const dfl wd = df_of(wk.x);
      const dfl dl{dg4.z, dg4.w};
      const dfl lr = df_mul(wd, WHOLE ? acc_r : df_add(df_mul(dl, df_re(xo)), acc_r));
      const dfl li = df_mul(wd, WHOLE ? acc_i : df_add(df_mul(dl, df_im(xo)), acc_i));
      const dfl pr = df_mul(wd, df_re(pp)), pi = df_mul(wd, df_im(pp));
      const dfl xr = df_mul(wd, df_re(xo)), xi = df_mul(wd, df_im(xo));
      // Im(conj(p) h) = p.re h.im - p.im h.re
      bil_l = df_add(bil_l, df_add(df_mul(pr, li), df_neg(df_mul(pi, lr))));
      // Im(conj(x) p) = x.re p.im - x.im p.re, weighted by each occupation
      const dfl tx = df_add(df_mul(xr, pi), df_neg(df_mul(xi, pr)));
      // two modes a packed sum, the occupations exact
      const f2 th = f2_pack(tx.h, tx.h), tl = f2_pack(tx.l, tx.l);
#pragma unroll
      for (int q = 0; q < kMB; q += 2) {
        if (q >= M) break;
        const float n0 = occ_float<NW>(ob, q), n1 = q + 1 < kMB ? occ_float<NW>(ob, q + 1) : 0.f;
        dfc_fma_int(bil_w[q / 2], f2_pack(n0, n1), f2_pack(-n0, -n1), th, tl);
        bil_w[q / 2] = dfc_renorm(bil_w[q / 2]);
      }
    }
    if (mode == 0 || mode == 2) {
      dfl orr = df_mul(zf, hi), oi = df_neg(df_mul(zf, hr));  // z H x with z = -i zre
      if (mode == 0) {
        const float4* pf = a.psif + (size_t)b * total + ri;
        const float4 p0 = RESIDENT ? *pf : ld_once(pf);
        orr = df_add(df_re(p0), orr);
        oi = df_add(df_im(p0), oi);
      }
      a.out[(size_t)b * total + ri] = df_pack(orr, oi);
    } else {  // modes 1 and 3: back to the FP64 vector, one weight per ket
      double sr = a.zre * df_to(hi), si = -a.zre * df_to(hr);
      if (mode == 3) {
        for (int k = 0; k < a.nbasef; ++k) {
          const float4 e = ld_once(a.basef[k] + (size_t)b * total + ri);
          sr += df_to(df_re(e));
          si += df_to(df_im(e));
        }
      }
      const double2 p0 = a.psi[(size_t)b * total + ri];
      const double nr = p0.x + wk.x * sr, ni = p0.y + wk.x * si;
      a.psi[(size_t)b * total + ri] = make_double2(nr, ni);
      a.out[(size_t)b * total + ri] = df_pack(df_of(nr * wk.y), df_of(ni * wk.y));
    }
  }
}

// The kets of one warp round: 32 consecutive ones, lane by lane.  Fillings of different
// classes are numbered with a gap, so that a ket belongs to the block of the ket before it
// exactly when its filling follows that one's; the block of a round's first ket is stored.
struct RoundIn {
  uint64_t word;   // packed occupations
  uint32_t fill;   // number of the filling
  uint32_t first;  // block of lane 0
};
__device__ __forceinline__ RoundIn load_round(const uint64_t* occ, const uint32_t* fill, const uint32_t* rblk, int64_t r,
                                              int64_t n, int lane) {
  RoundIn in;
  const int64_t g = min(r * 32 + lane, n - 1);
  in.word = ld_once(occ + g);
  in.fill = ld_once(fill + g);
  in.first = __ldg(rblk + r);
  return in;
}
__device__ __forceinline__ uint32_t block_of_lane(const RoundIn& in, int lane, bool inside) {
  const uint32_t prev = __shfl_up_sync(0xffffffffu, in.fill, 1);
  const uint32_t heads = __ballot_sync(0xffffffffu, inside && lane > 0 && in.fill != prev + 1u);
  return in.first + __popc(heads & (0xffffffffu >> (31 - lane)));
}

// Threads a CTA's registers are planned for (65,536 registers per SM): the one-state stages
// at 64 a thread, the bilinear ones at 80 (one stage of 2.3M kets at M = 5: 265 us at 128,
// 200 at 80, 192 at 64 where that does not spill), the sweep members at 128.
template <int B, int KIND>
__host__ __device__ constexpr int blk_max_threads() {
  return KIND == KIND_BIL ? 768 : (B == 1 ? 1024 : 512);
}

// per-CTA sums of the bilinears in a fixed order: lanes by shuffles, warps in turn
template <int kMB>
__device__ __forceinline__ void bil_reduce(const DfArgs& a, int M, const dfl& bil_l, const dfc* bil_w) {
  __shared__ double red[32][17];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
  const int nq = M + 1;
  for (int q = 0; q < nq; ++q) {
    double val = (q == 0) ? df_to(bil_l) : 0.0;
#pragma unroll
    for (int u = 0; u < kMB; ++u)
      if (q == u + 1) {
        float h0, h1, l0, l1;
        f2_unpack(bil_w[u / 2].h, h0, h1);
        f2_unpack(bil_w[u / 2].l, l0, l1);
        val = u % 2 ? (double)h1 + (double)l1 : (double)h0 + (double)l0;
      }
    for (int o = 16; o > 0; o >>= 1) val += __shfl_down_sync(0xffffffffu, val, o);
    if (lane == 0) red[warp][q] = val;
  }
  __syncthreads();
  if (threadIdx.x < nq) {
    double sum = 0.0;
    for (int w = 0; w < warps; ++w) sum += red[w][threadIdx.x];
    a.partial[(size_t)blockIdx.x * nq + threadIdx.x] = sum;
  }
}

// Mode counts up to which the walk over the pairs is unrolled (28 records of 3 terms at
// M = 7).  One step of the M = 7, n_tot = 4 long-range space 155 -> 151 us; at M = 9 (45
// records of 4 terms) the code leaves the instruction cache: 21.2 -> 30.5 ms at N = 27.
constexpr int kUnrollM = 7;
// the pairs r <= s in order
template <int MT>
struct OrderedPairs {
  int r[MT * (MT + 1) / 2], s[MT * (MT + 1) / 2];
  constexpr OrderedPairs() : r(), s() {
    int i = 0;
    for (int p = 0; p < MT; ++p)
      for (int q = p; q < MT; ++q, ++i) {
        r[i] = p;
        s[i] = q;
      }
  }
};

// Shared memory: couplings (real, imaginary) of the slots and the record words
__host__ __device__ inline size_t blk_smem_bytes(const Tables& t, bool cplx) {
  return (size_t)t.bk_T * 8 * (cplx ? 2 : 1) + (((size_t)t.bk_nrec * 8 + 15) & ~(size_t)15);
}

// U: records whose gathers are in flight together.  One where every SM has its 32 warps;
// four in CTAs of up to 256 threads (255 registers) for the spaces that leave a warp or two
// per scheduler, where every gather's latency shows.
template <int MT, bool FIX, int B, bool CPLX, int KIND, int U>
__global__ void __launch_bounds__((U > 1 ? 256 : blk_max_threads<B, KIND>()), 1)
    blk_stage_kernel(const Tables t, const DfArgs a, const int mode) {
  constexpr int KC = FIX ? (MT - 1) / 2 : 0;
  constexpr int NT = Rec<KC>::n, RW = Rec<KC>::w, NW = occ_words<MT>();
  constexpr bool BIL = (KIND == KIND_BIL), DOT = (KIND == KIND_DOT);
  constexpr int kMB = (MT > 0) ? MT : 16;
  const int M = (MT > 0) ? MT : t.M;
  const int T = t.bk_T, nrec = t.bk_nrec;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = blockDim.x >> 5;

  float2* sG = reinterpret_cast<float2*>(blk_smem);
  float2* sGi = sG + T;
  uint2* sinfo = reinterpret_cast<uint2*>(sG + (CPLX ? 2 : 1) * T);
  for (int i = threadIdx.x; i < T; i += blockDim.x) {
    sG[i] = __ldg(t.bk_G + i);
    if (CPLX) sGi[i] = __ldg(t.bk_Gi + i);
  }
  for (int i = threadIdx.x; i < nrec; i += blockDim.x) sinfo[i] = __ldg(t.bk_info + i);
  __syncthreads();  // the only CTA-wide barrier: warps run independently afterwards

  const int64_t total = t.total;
  dfl bil_l{0.f, 0.f};
  dfc bil_w[BIL ? (kMB + 1) / 2 : 1];
#pragma unroll
  for (int q = 0; q < (BIL ? (kMB + 1) / 2 : 1); ++q) bil_w[q] = dfc{0ull, 0ull};
  double dot64 = 0.0;

  // the last rounds (the most particles, the most pairs per ket) first
  const int64_t r0 = a.row0 / 32, step = (int64_t)gridDim.x * warps;
  int64_t rd = (a.row1 - 1) / 32 - ((int64_t)blockIdx.x * warps + warp);
  RoundIn next = load_round(t.occ, t.fill, t.rblk, max(rd, r0), total, lane);
  chain_wait();
  for (; rd >= r0; rd -= step) {
      const int64_t g = rd * 32 + lane;
      const bool valid = g >= a.row0 && g < a.row1;
      const RoundIn in = next;
      next = load_round(t.occ, t.fill, t.rblk, max(rd - step, r0), total, lane);
      const uint32_t* base = t.bk_base + (size_t)block_of_lane(in, lane, g < total) * T;
      uint32_t ob[NW];
      unpack_occ<MT, NW>(t, valid ? in.word : 0ull, ob);  // an invalid lane: no pair acts
      const unsigned char* mp = t.bk_map + (size_t)in.fill * (2 * RW);
      const uint16_t* mp5 = t.bk_map5 + in.fill;

      dfc acc[B];  // (re, im) of the off-diagonal sum, double-float, packed
#pragma unroll
      for (int b = 0; b < B; ++b) acc[b] = dfc{0ull, 0ull};
      bool bad = false;  // a target fell outside the state

      // ---- the annihilation pairs (r <= s) in step, U records' gathers and the next U records'
      // maps and bases in flight.  A lane that lacks a pair has the coefficient 0 and keeps its
      // last gathered values.
      float4 x[U][NT];
#pragma unroll
      for (int u = 0; u < U; ++u)
#pragma unroll
        for (int c = 0; c < NT; ++c) x[u][c] = make_float4(0.f, 0.f, 0.f, 0.f);
      MapRec<KC> mcur[U], mnext[U];
      BaseRec<KC> bcur[U], bnext[U];
      auto load = [&](int rec0, MapRec<KC> (&mr)[U], BaseRec<KC> (&br)[U]) {
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int rec = min(rec0 + u, nrec - 1);
          mr[u] = load_map<KC>(mp + (size_t)rec * t.bk_S * (2 * RW), mp5 + (size_t)rec * t.bk_S);
          br[u] = load_base<KC>(base, rec, nrec);
        }
      };
      if constexpr (FIX && U == 1 && B == 1 && !CPLX && MT <= kUnrollM) {
        // unrolled: the pairs are constants, a pair's factor is one product of two registers; the
        // maps and bases two records ahead (one ahead: one stage of 245,157 kets at M = 7 37.7 us,
        // now 36.2; reading the next targets into L1 or L2 by prefetch as well: 41.1)
        constexpr OrderedPairs<MT> pr{};
        constexpr int NR = MT * (MT + 1) / 2;
        float nf[MT];
#pragma unroll
        for (int m = 0; m < MT; ++m) nf[m] = occ_float<NW>(ob, m);
        load(0, mcur, bcur);
        uint32_t rkn[NT];
        auto targets = [&](uint32_t (&k)[NT]) {
          k[0] = bcur[0].a.x + (mcur[0].a.x & 0xffffu);
          k[1] = bcur[0].a.y + (mcur[0].a.x >> 16);
          if constexpr (NT > 2) k[2] = bcur[0].a.z + (mcur[0].a.y & 0xffffu);
          if constexpr (NT > 3) k[3] = bcur[0].a.w + (mcur[0].a.y >> 16);
          if constexpr (NT > 4) k[4] = bcur[0].b + mcur[0].b;
        };
        targets(rkn);
        load(1, mcur, bcur);
#pragma unroll
        for (int rec = 0; rec < NR; ++rec) {
          uint32_t rk[NT];
#pragma unroll
          for (int c = 0; c < NT; ++c) rk[c] = rkn[c];
          if (rec + 1 < NR) {
            targets(rkn);
            if (rec + 2 < NR) load(rec + 2, mcur, bcur);
          }
          const float Af = pr.r[rec] != pr.s[rec] ? nf[pr.r[rec]] * nf[pr.s[rec]] : nf[pr.r[rec]] * (nf[pr.r[rec]] - 1.f);
          uint32_t top = rk[0];
#pragma unroll
          for (int c = 1; c < NT; ++c) top = max(top, rk[c]);
          const bool act = Af != 0.f, ok = act && top < (uint32_t)total;
          bad |= act && !ok;
          const int c_first = DOT ? (int)((sinfo[rec].x >> 8) & 7) : 0;
#pragma unroll
          for (int c = 0; c < NT; ++c)
            if (ok && (!DOT || c >= c_first)) x[0][c] = a.vin[rk[c]];
          if (__any_sync(0xffffffffu, act)) {
            add_record<KC, CPLX, DOT>(acc[0], x[0], sG, sGi, rec, NR, NT, c_first, Af);
            acc[0] = dfc_renorm(acc[0]);
          }
        }
      } else if (nrec > 0) {
      load(0, mcur, bcur);
      for (int rec0 = 0; rec0 < nrec; rec0 += U) {
        load(rec0 + U, mnext, bnext);
        float Af[U];
        uint32_t rk[U][NT], infox[U];
        bool ok[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const bool in_list = U == 1 || rec0 + u < nrec;
          const uint2 info = sinfo[in_list ? rec0 + u : rec0];
          infox[u] = info.x;
          Af[u] = (occ_float23<NW>(ob, info.x, (info.x & 0x8000u) != 0u) - 8388608.0f) *
                  (occ_float23<NW>(ob, info.x >> 16, (info.x & 0x80000000u) != 0u) - __uint_as_float(info.y));
          if (!in_list) Af[u] = 0.f;
          const int n = KC == 0 ? (int)((info.x >> 4) & 7) : NT;
          rk[u][0] = bcur[u].a.x + (mcur[u].a.x & 0xffffu);
          rk[u][1] = bcur[u].a.y + (mcur[u].a.x >> 16);
          if constexpr (NT > 2) rk[u][2] = bcur[u].a.z + (mcur[u].a.y & 0xffffu);
          if constexpr (NT > 3) rk[u][3] = bcur[u].a.w + (mcur[u].a.y >> 16);
          if constexpr (NT > 4) rk[u][4] = bcur[u].b + mcur[u].b;
          uint32_t top = rk[u][0];
#pragma unroll
          for (int c = 1; c < NT; ++c)
            if (KC > 0 || c < n) top = max(top, rk[u][c]);
          const bool act = Af[u] != 0.f;
          ok[u] = act && top < (uint32_t)total;
          bad |= act && !ok[u];
          const int c_first = DOT ? (int)((info.x >> 8) & 7) : 0;
#pragma unroll
          for (int c = 0; c < NT; ++c)
            if (ok[u] && (KC > 0 || c < n) && (!DOT || c >= c_first)) x[u][c] = a.vin[rk[u][c]];
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
          if (!__any_sync(0xffffffffu, Af[u] != 0.f)) continue;
          const int rec = rec0 + u;
          const int n = KC == 0 ? (int)((infox[u] >> 4) & 7) : NT;
          const int c_first = DOT ? (int)((infox[u] >> 8) & 7) : 0;
#pragma unroll
          for (int b = 0; b < B; ++b) {
            if (b > 0) {
#pragma unroll
              for (int c = 0; c < NT; ++c)
                if (ok[u] && (KC > 0 || c < n)) x[u][c] = a.vin[(size_t)b * total + rk[u][c]];
            }
            add_record<KC, CPLX, DOT>(acc[b], x[u], sG, sGi, rec, nrec, n, c_first, Af[u]);
          }
          // keep |lo| below an ulp of hi between pairs
          if (KC > 0 || (infox[u] & 0x80u)) {
#pragma unroll
            for (int b = 0; b < B; ++b) acc[b] = dfc_renorm(acc[b]);
          }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
          mcur[u] = mnext[u];
          bcur[u] = bnext[u];
        }
      }
      }
      if (bad) atomicOr(a.status, 1);
      if (valid) stage_epilogue<MT, B, KIND, false, NW>(t, a, mode, g, g, acc, ob, bil_l, bil_w, dot64);
  }

  if constexpr (DOT) {
    // the CTA's sum in a fixed order: lanes by shuffles, warps in turn; partial[block]
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
  if constexpr (BIL) bil_reduce<kMB>(a, M, bil_l, bil_w);
}

// The records that a ket takes part in, one after the other: the pairs (r, s) of its occupied
// modes in order, each with its records.
struct RecordWalk {
  uint32_t occ, two, rm, sm;  // modes with a particle, with two; modes r and s still to come
  int r, rec;
  __device__ __forceinline__ RecordWalk(const Tables& t, uint64_t word) : occ(0u), two(0u), sm(0u), r(0), rec(-1) {
    for (int m = 0; m < t.M; ++m) {
      const int n = occ_of(word, m, t.occ_bits);
      occ |= (n > 0 ? 1u : 0u) << m;
      two |= (n > 1 ? 1u : 0u) << m;
    }
    rm = occ;
  }
  // the next record in rec; false when there is none (first: first record of each pair)
  __device__ __forceinline__ bool next(const uint2* sinfo, const uint16_t* first) {
    if (rec >= 0 && (sinfo[rec].x & 0x80u) == 0u) {
      ++rec;
      return true;
    }
    while ((rm | sm) != 0u) {
      if (sm == 0u) {
        r = __ffs(rm) - 1;
        rm &= rm - 1;
        sm = occ & (~0u << r);
        if (((two >> r) & 1u) == 0u) sm &= ~(1u << r);
        continue;
      }
      const int s = __ffs(sm) - 1;
      sm &= sm - 1;
      const uint32_t f = first[r * 16 + s];
      if (f != 0xffffu) {
        rec = (int)f;
        return true;
      }
    }
    return false;
  }
};
// first[r * 16 + s]: the first record of the pair, or 0xffff (a CTA's threads together, between
// two barriers)
constexpr size_t kFirstBytes = 512;
__device__ __forceinline__ void first_records(const uint2* sinfo, int nrec, uint16_t* first) {
  for (int i = threadIdx.x; i < 256; i += blockDim.x) first[i] = 0xffffu;
  __syncthreads();
  for (int i = threadIdx.x; i < nrec; i += blockDim.x) {
    const uint32_t x = sinfo[i].x;
    if (i == 0 || (sinfo[i - 1].x & 0x80u) != 0u)
      first[((x & 7) | ((x >> 12) & 8)) * 16 + (((x >> 16) & 7) | ((x >> 28) & 8))] = (uint16_t)i;
  }
  __syncthreads();
}

// The same stage with each lane on the records of its own ket instead of all lanes on every
// record in step: scattered reads of maps, bases and couplings, but no work for pairs that a ket
// lacks, which with many modes and few particles are nearly all.  A pair that a ket lacks adds
// zero in the kernel above, so that the states agree bit for bit.  The lanes stay together in the
// products where a sweep's members share a record whose partners vary (IN_STEP): with four
// members, M = 10, 184,756 kets, a stage 292 us apart, 280 in step; with two 172 and 189.
template <int KC, int B, bool CPLX, int KIND>
__global__ void __launch_bounds__((blk_max_threads<B, KIND>()), 1)
    sparse_stage_kernel(const Tables t, const DfArgs a, const int mode) {
  constexpr int NT = Rec<KC>::n, RW = Rec<KC>::w, NW = occ_words<0>();
  constexpr bool BIL = (KIND == KIND_BIL), IN_STEP = KC == 0 && B >= 4;
  const int T = t.bk_T, nrec = t.bk_nrec;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
  float2* sG = reinterpret_cast<float2*>(blk_smem);
  float2* sGi = sG + T;
  uint2* sinfo = reinterpret_cast<uint2*>(sG + (CPLX ? 2 : 1) * T);
  uint16_t* first = reinterpret_cast<uint16_t*>(blk_smem + blk_smem_bytes(t, CPLX));
  for (int i = threadIdx.x; i < T; i += blockDim.x) {
    sG[i] = __ldg(t.bk_G + i);
    if (CPLX) sGi[i] = __ldg(t.bk_Gi + i);
  }
  for (int i = threadIdx.x; i < nrec; i += blockDim.x) sinfo[i] = __ldg(t.bk_info + i);
  __syncthreads();
  first_records(sinfo, nrec, first);

  const int64_t total = t.total;
  dfl bil_l{0.f, 0.f};
  dfc bil_w[BIL ? 8 : 1];
#pragma unroll
  for (int q = 0; q < (BIL ? 8 : 1); ++q) bil_w[q] = dfc{0ull, 0ull};
  double dot64 = 0.0;
  const int64_t r0 = a.row0 / 32, step = (int64_t)gridDim.x * warps;
  int64_t rd = (a.row1 - 1) / 32 - ((int64_t)blockIdx.x * warps + warp);
  RoundIn in_next = load_round(t.occ, t.fill, t.rblk, max(rd, r0), total, lane);
  chain_wait();
  for (; rd >= r0; rd -= step) {
    const int64_t g = rd * 32 + lane;
    const bool valid = g >= a.row0 && g < a.row1;
    const RoundIn in = in_next;
    in_next = load_round(t.occ, t.fill, t.rblk, max(rd - step, r0), total, lane);
    const uint32_t* base = t.bk_base + (size_t)block_of_lane(in, lane, g < total) * T;
    uint32_t ob[NW];
    unpack_occ<0, NW>(t, valid ? in.word : 0ull, ob);
    const unsigned char* mp = t.bk_map + (size_t)in.fill * (2 * RW);
    const uint16_t* mp5 = t.bk_map5 + in.fill;
    dfc acc[B];
#pragma unroll
    for (int b = 0; b < B; ++b) acc[b] = dfc{0ull, 0ull};
    bool bad = false;
    RecordWalk walk(t, valid ? in.word : 0ull);
    MapRec<KC> m{};
    BaseRec<KC> bs{};
    bool act = walk.next(sinfo, first);
    auto load = [&]() {
      if (act) {
        m = load_map<KC>(mp + (size_t)walk.rec * t.bk_S * (2 * RW), mp5 + (size_t)walk.rec * t.bk_S);
        bs = load_base<KC>(base, walk.rec, nrec);
      }
    };
    load();
    while (__any_sync(0xffffffffu, act)) {
      const bool on = act;
      const int rec = walk.rec;
      uint32_t rk[NT];
      rk[0] = bs.a.x + (m.a.x & 0xffffu);
      rk[1] = bs.a.y + (m.a.x >> 16);
      if constexpr (NT > 2) rk[2] = bs.a.z + (m.a.y & 0xffffu);
      if constexpr (NT > 3) rk[3] = bs.a.w + (m.a.y >> 16);
      if constexpr (NT > 4) rk[4] = bs.b + m.b;
      if (on) act = walk.next(sinfo, first);
      load();
      if (!IN_STEP && !on) continue;
      const int ri = on ? rec : 0;
      const uint2 info = sinfo[ri];
      const float Af = (occ_float23<NW>(ob, info.x, (info.x & 0x8000u) != 0u) - 8388608.0f) *
                       (occ_float23<NW>(ob, info.x >> 16, (info.x & 0x80000000u) != 0u) - __uint_as_float(info.y));
      const int n = !on ? 0 : KC == 0 ? (int)((info.x >> 4) & 7) : NT;
      uint32_t top = rk[0];
#pragma unroll
      for (int c = 1; c < NT; ++c)
        if (KC > 0 || c < n) top = max(top, rk[c]);
      const bool ok = on && top < (uint32_t)total;
      bad |= on && !ok;
      if (!IN_STEP && !ok) continue;
      const int terms = IN_STEP ? __reduce_max_sync(0xffffffffu, n) : n;  // beyond n: zeros
      const bool done = on && (KC > 0 || (info.x & 0x80u) != 0u);
#pragma unroll
      for (int b = 0; b < B; ++b) {
        float4 x[NT];
#pragma unroll
        for (int c = 0; c < NT; ++c)
          x[c] = (!IN_STEP || ok) && (KC > 0 || c < n) ? a.vin[(size_t)b * total + rk[c]] : make_float4(0.f, 0.f, 0.f, 0.f);
        add_record<KC, CPLX, false>(acc[b], x, sG, sGi, ri, nrec, terms, 0, IN_STEP && !on ? 0.f : Af);
        if (IN_STEP) {
          const dfc sum = dfc_renorm(acc[b]);
          if (done) acc[b] = sum;
        } else if (done) {
          acc[b] = dfc_renorm(acc[b]);
        }
      }
    }
    if (bad) atomicOr(a.status, 1);
    if (valid) stage_epilogue<0, B, KIND, false, NW>(t, a, mode, g, g, acc, ob, bil_l, bil_w, dot64);
  }
  if constexpr (BIL) bil_reduce<16>(a, t.M, bil_l, bil_w);
}

// Tile shapes: warps per CTA (a warp takes 32 kets at a time)
constexpr int kTileShapes = 5;
__host__ __device__ constexpr int tile_warps(int ts) { return ts == 1 ? 16 : ts == 2 ? 24 : ts == 3 ? 12 : ts == 4 ? 8 : 32; }

// Rounds of 32 kets per SM up to which the four-record kernel runs: the CTA of 8 warps that
// its registers allow is then one wave.  One stage, one record against four (us): M = 5,
// 3,003 kets 7.6 / 6.0, 33,649 kets 8.1 / 7.2; M = 7, 19,448 kets 12.5 / 10.6; M = 11, 16,796
// kets 28.4 / 19.2.  The generic kernel (partner counts that vary) gains nothing by it (M = 6,
// 27,132 kets: 11.7 / 13.0).
constexpr int kFewWarps = 8;

// Warps per CTA and grid of a launch over `rows` kets.  While a small space leaves SMs
// without work the CTA shrinks, so that its rounds spread over every SM.
template <typename K>
inline int stage_geometry(K k, int64_t rows, int shape, int max_warps, size_t smem, int* warps_out, int* grid) {
  int per = 0, sms = 0, dev = 0;
  QB_CUDA(cudaGetDevice(&dev));
  QB_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  int warps = std::min(tile_warps(shape), max_warps);
  const int64_t rounds = rows / 32 + 2;  // unaligned ends: at most one more
  while (warps > 2 && rounds <= (int64_t)sms * (warps / 2)) warps >>= 1;
  const int rc = occupancy_cached(k, smem, &per, &sms, 32 * warps);
  if (rc) return rc;
  *warps_out = warps;
  *grid = (int)std::min<int64_t>((int64_t)sms * std::min(per, 16), (rounds + warps - 1) / warps);
  return QB_OK;
}

// One stage over the rows [a.row0, a.row1).
template <int MT, bool FIX, int B, bool CPLX, int KIND, int U>
int blk_launch_u(const Tables& t, const DfArgs& a, int mode, int shape, cudaStream_t st, int* grid_out) {
  auto k = blk_stage_kernel<MT, FIX, B, CPLX, KIND, U>;
  const size_t smem = blk_smem_bytes(t, CPLX);
  int warps = 0, grid = 0;
  const int rc = stage_geometry(k, a.row1 - a.row0, shape, (U > 1 ? 256 : blk_max_threads<B, KIND>()) / 32, smem, &warps,
                                &grid);
  if (rc) return rc;
  QB_CUDA(chain_launch(k, grid, 32 * warps, smem, st, t, a, mode));
  if (grid_out) *grid_out = grid;
  return QB_OK;
}

template <int KC, int B, bool CPLX, int KIND>
int sparse_launch(const Tables& t, const DfArgs& a, int mode, int shape, cudaStream_t st, int* grid_out) {
  auto k = sparse_stage_kernel<KC, B, CPLX, KIND>;
  const size_t smem = blk_smem_bytes(t, CPLX) + kFirstBytes;
  int warps = 0, grid = 0;
  const int rc = stage_geometry(k, a.row1 - a.row0, shape, blk_max_threads<B, KIND>() / 32, smem, &warps, &grid);
  if (rc) return rc;
  QB_CUDA(chain_launch(k, grid, 32 * warps, smem, st, t, a, mode));
  if (grid_out) *grid_out = grid;
  return QB_OK;
}
// Share of a space's records that a ket takes part in on average (Tables::bk_share), up to which
// each lane walks its own ket's.  One stage, all records in step / own records (us): one state, M =
// 12, 18,564 kets (share 0.10) 53 / 21; M = 10, 19,448 kets (0.15) 32 / 29; M = 8, 6,435 (0.2) 15 /
// 19; M = 9, 5,005 (0.14) 11 / 13; M = 11, 167,960 (0.19) 125 / 71, 16,796 of one momentum (0.24)
// 18 / 45.  Two members, M = 9, 92,378 (0.26) 66 / 53, M = 7, 19,448 (0.33) 18 / 24; four, M = 10, 184,756
// (0.24) 355 / 280, M = 7, 245,157 (0.47) 127 / 128; eight, M = 5, 1.2M kets (0.79) 521 / 459.  Partners
// that vary, eight members: M = 6, 5,005 kets (0.34) 56 / 66.  With bilinears (a gradient of
// three steps), M = 12, 18,564 kets 3.1 / 2.0 ms, M = 11, 31,824 (0.14) 1.8 / 2.2.
template <int KC, int B, int KIND>
constexpr float sparse_share() {
  if (KIND == KIND_BIL) return KC == 0 ? 0.16f : KC >= 4 ? 0.1f : 0.f;
  if (B == 1) return KC == 0 ? 0.16f : KC == 4 ? 0.12f : KC == 5 ? 0.2f : 0.f;
  if (B == 2) return KC == 0 ? 0.25f : KC >= 4 ? 0.37f : 0.18f;
  if (KC == 0) return 0.3f;
  return B == 4 ? 0.45f : 2.f;  // eight: always
}

template <int MT, bool FIX, int B, bool CPLX, int KIND>
int blk_launch(const Tables& t, const DfArgs& a, int mode, int shape, cudaStream_t st, int* grid_out) {
  constexpr int KC = FIX ? (MT - 1) / 2 : 0;
  constexpr float line = KIND == KIND_DOT ? 0.f : sparse_share<KC, B, KIND>();
  if constexpr (line > 1.f) {
    return sparse_launch<KC, B, CPLX, KIND>(t, a, mode, shape, st, grid_out);
  } else {
    if constexpr (line > 0.f)
      if (t.bk_share < line) return sparse_launch<KC, B, CPLX, KIND>(t, a, mode, shape, st, grid_out);
    if constexpr (FIX && B == 1 && KIND == KIND_STAGE) {
      int dev = 0, sms = 0;
      QB_CUDA(cudaGetDevice(&dev));
      QB_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
      if ((a.row1 - a.row0) / 32 <= (int64_t)sms * kFewWarps)
        return blk_launch_u<MT, FIX, B, CPLX, KIND, 4>(t, a, mode, shape, st, grid_out);
    }
    return blk_launch_u<MT, FIX, B, CPLX, KIND, 1>(t, a, mode, shape, st, grid_out);
  }
}

// the kinds and batch sizes of one kernel family (real or complex couplings)
template <int MT, bool FIX>
int blk_launch_kind(const Tables& t, const DfArgs& a, int mode, int B, bool bil, int shape, cudaStream_t st, int* grid) {
  if (mode < 0 || mode > 4) return fail(QB_EINTERNAL, "bad stage mode");
  if (mode == 4) {
    if (B != 1) return fail(QB_EUNSUPPORTED, "the <x|H|x> reduction runs one state at a time");
    return blk_launch<MT, FIX, 1, false, KIND_DOT>(t, a, mode, shape, st, grid);
  }
  if (bil) {
    if (B != 1) return fail(QB_EUNSUPPORTED, "bilinear stages run one state at a time");
    return blk_launch<MT, FIX, 1, false, KIND_BIL>(t, a, mode, shape, st, grid);
  }
  if (B != 1 && t.exact) return fail(QB_EUNSUPPORTED, "exact momentum: batched sweeps are not built");
  switch (B) {
    case 1: return blk_launch<MT, FIX, 1, false, KIND_STAGE>(t, a, mode, shape, st, grid);
    case 2: return blk_launch<MT, FIX, 2, false, KIND_STAGE>(t, a, mode, shape, st, grid);
    case 4: return blk_launch<MT, FIX, 4, false, KIND_STAGE>(t, a, mode, shape, st, grid);
    case 8:
      if constexpr (!FIX)
        if (t.bk_share < sparse_share<0, 8, KIND_STAGE>()) {  // as two groups of four (eight at once
          DfArgs h = a;                                       // M = 10, 184,756 kets: 626 us, so 559)
          const int rc = blk_launch<MT, FIX, 4, false, KIND_STAGE>(t, h, mode, shape, st, grid);
          if (rc) return rc;
          const size_t n = 4 * (size_t)t.total;
          h.vin += n;
          h.out += n;
          if (h.psi) h.psi += n;
          if (h.psif) h.psif += n;
          for (int b = 0; b < 4; ++b) h.scale[b] = a.scale[b + 4];
          return blk_launch<MT, FIX, 4, false, KIND_STAGE>(t, h, mode, shape, st, grid);
        }
      return blk_launch<MT, FIX, 8, false, KIND_STAGE>(t, a, mode, shape, st, grid);
    default: return fail(QB_EINVAL, "batch must be 1, 2, 4 or 8");
  }
}

// one translation unit each (qb_stage_m*.cu): the mode counts with a fixed partner count
// (odd M, momentum mod M, real couplings), and everything else; and the factored stages
int stage_launch_m5(const Tables&, const DfArgs&, int, int, bool, int, cudaStream_t, int*);
int stage_launch_m7(const Tables&, const DfArgs&, int, int, bool, int, cudaStream_t, int*);
int stage_launch_m9(const Tables&, const DfArgs&, int, int, bool, int, cudaStream_t, int*);
int stage_launch_m11(const Tables&, const DfArgs&, int, int, bool, int, cudaStream_t, int*);
int stage_launch_any(const Tables&, const DfArgs&, int, int, bool, bool, int, cudaStream_t, int*);
int fac_launch_m7(const Tables&, const DfArgs&, int, int, bool, int, cudaStream_t, int*);
int fac_launch_m9(const Tables&, const DfArgs&, int, int, bool, int, cudaStream_t, int*);
int fac_launch_m11(const Tables&, const DfArgs&, int, int, bool, int, cudaStream_t, int*);
int fac_launch_any(const Tables&, const DfArgs&, int, int, bool, int, cudaStream_t, int*);

// One stage over rows [a.row0, a.row1) in the weighted basis (factored spaces: the lower
// kets [a.low0, a.low1) and a.g as well).  bil: the bilinear instantiations (adjoint modes
// 2, 3); mode 4 is the <x|H|x> reduction (partial[block]; a factored space: its two-body
// part); shape: tile shape (0: the default).
inline int stage_launch(const Tables& t, const DfArgs& a, int mode, int B, bool cplx, cudaStream_t st,
                        int* grid_out = nullptr, bool bil = false, int shape = 0) {
  if (t.fa_on) {
    switch (t.M) {
      case 7: return fac_launch_m7(t, a, mode, B, bil, shape, st, grid_out);
      case 9: return fac_launch_m9(t, a, mode, B, bil, shape, st, grid_out);
      case 11: return fac_launch_m11(t, a, mode, B, bil, shape, st, grid_out);
      default: break;
    }
    return fac_launch_any(t, a, mode, B, bil, shape, st, grid_out);
  }
  if (t.bk_kc > 0 && !cplx) {
    switch (t.M) {
      case 5: return stage_launch_m5(t, a, mode, B, bil, shape, st, grid_out);
      case 7: return stage_launch_m7(t, a, mode, B, bil, shape, st, grid_out);
      case 9: return stage_launch_m9(t, a, mode, B, bil, shape, st, grid_out);
      case 11: return stage_launch_m11(t, a, mode, B, bil, shape, st, grid_out);
      default: break;
    }
  }
  return stage_launch_any(t, a, mode, B, cplx, bil, shape, st, grid_out);
}

}  // namespace qb
