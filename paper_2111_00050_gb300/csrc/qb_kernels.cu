// sm_103a kernels of the qb library: matrix-free sector H psi fused into the
// Horner-form RK4 stages, combinatorial unrank / rank, initial states,
// observable moments with deterministic two-pass reductions.
//
// Paper: Eberhardt, Zamora, Kopp & Abel, arXiv:2111.00050.  The Hamiltonian is
// Eq. (Ham); sectors are the special Hilbert spaces of Sec. III B; the state of
// every sector evolves independently (Sec. III B), so one launch covers all
// sectors of a space (and all members of a batched coupling sweep).
#include <cuda_runtime.h>

#include <algorithm>
#include <chrono>
#include <cmath>
#include <mutex>
#include <string>
#include <vector>

#include "qb_internal.h"

#include "qb_device.cuh"
#include "qb_block.cuh"
#include "qb_factor.cuh"
#include "qb_stage.cuh"

namespace qb {

// ------------------------------------------------------------ H psi kernels

enum { MODE_HPSI = 0, MODE_DOT = 1 };

struct StageArgs {
  const double2* vin;  // gathered vector(s) [B][total]
  double2* out;        // output(s) [B][total]
  double scale[8];     // two-body scale per member
  double* partial;     // MODE_DOT: [gridDim.x][2]
  int* status;         // device status word (bounds violations)
};

template <int MODE, int B, bool CPLX>
__global__ void __launch_bounds__(kBlock) hpsi_kernel(const Tables t, const StageArgs a) {
  extern __shared__ __align__(16) unsigned char smem[];
  load_blob(t, smem);
  const View v = make_view(t, smem);
  const RowScratch rs = row_scratch(smem + blob_smem(t));
  const int tid = threadIdx.x;
  const int M = t.M;
  const int64_t total = t.total;
  double dot_re = 0.0, dot_im = 0.0;

  for (int64_t base = (int64_t)blockIdx.x * kBlock; base < total; base += (int64_t)gridDim.x * kBlock) {
    const int64_t g = base + tid;
    if (g >= total) break;
    const int sid = find_sector(t, g);
    const int64_t off = __ldg(t.sec_off + sid);
    const int64_t D = __ldg(t.sec_off + sid + 1) - off;
    const int N = __ldg(t.sec_N + sid), K = __ldg(t.sec_K + sid);
    const int64_t me = setup_row(t, v, rs, N, K, D, g - off);
    if (me != g - off) atomicOr(a.status, 2);

    const uint8_t* occ = rs.occ + tid;
    const int32_t* idx = rs.idx + tid;
    const int32_t* pe = rs.pe + tid;
    uint32_t occmask = 0, twomask = 0;
    double dw = 0.0;
    for (int m = 0; m < M; ++m) {
      int nm = occ[m * kBlock];
      occmask |= (nm >= 1 ? 1u : 0u) << m;
      twomask |= (nm >= 2 ? 1u : 0u) << m;
      dw += v.w[m] * nm;
    }
    const int64_t rank_base = D - 1 - pe[(M - 1) * kBlock];
    double dl = 0.0;
    double acc_re[B], acc_im[B];
#pragma unroll
    for (int b = 0; b < B; ++b) acc_re[b] = acc_im[b] = 0.0;

    // flattened iteration over annihilation pairs r <= s with n_r (n_s - [r==s]) > 0
    uint32_t rm = occmask, sm = 0;
    int r = 0;
    while (true) {
      if (sm == 0) {
        if (rm == 0) break;
        r = __ffs(rm) - 1;
        rm &= rm - 1;
        sm = occmask & (~0u << r);
        if (!((twomask >> r) & 1u)) sm &= ~(1u << r);
        if (sm == 0) continue;
      }
      const int s = __ffs(sm) - 1;
      sm &= sm - 1;
      const int ai = v.pairidx[r * 16 + s];
      const int nr = occ[r * kBlock], ns = occ[s * kBlock];
      const double A = v.sq[nr] * v.sq[ns - (r == s ? 1 : 0)];
      dl += v.gd[ai] * (double)(nr * (ns - (r == s ? 1 : 0)));
      double pr[B], pi[B];
#pragma unroll
      for (int b = 0; b < B; ++b) pr[b] = pi[b] = 0.0;
      const int j1 = v.ann[ai + 1];
      for (int j = v.ann[ai]; j < j1; ++j) {
        const uint32_t w4 = v.pq[j];
        const int p = w4 & 0xff, q = (w4 >> 8) & 0xff, lo = (w4 >> 16) & 0xff, hi = w4 >> 24;
        const int np_ = occ[p * kBlock], nq = occ[q * kBlock];
        const double Bf = v.sq[np_ + 1] * v.sq[nq + 1 + (p == q ? 1 : 0)];
        int64_t rk = rank_base + pe[hi * kBlock] - pe[lo * kBlock];
        for (int m = lo + 1; m <= hi; ++m) rk -= v.E[idx[m * kBlock] + delta_shift(t, v, j, m)];
        if (rk < 0 || rk >= D) {
          atomicOr(a.status, 1);
          rk = 0;
        }
        const double cr = v.G[2 * j] * Bf;
#pragma unroll
        for (int b = 0; b < B; ++b) {
          const double2 x = __ldg(a.vin + (size_t)b * total + off + rk);
          if (CPLX) {
            const double ci = v.G[2 * j + 1] * Bf;
            pr[b] += cr * x.x - ci * x.y;
            pi[b] += cr * x.y + ci * x.x;
          } else {
            pr[b] += cr * x.x;
            pi[b] += cr * x.y;
          }
        }
      }
#pragma unroll
      for (int b = 0; b < B; ++b) {
        acc_re[b] += A * pr[b];
        acc_im[b] += A * pi[b];
      }
    }

#pragma unroll
    for (int b = 0; b < B; ++b) {
      const double sc = a.scale[b];
      const double2 x = a.vin[(size_t)b * total + g];
      const double dg = dw + sc * dl;
      const double hr = dg * x.x + sc * acc_re[b];
      const double hi = dg * x.y + sc * acc_im[b];
      if (MODE == MODE_HPSI) {
        a.out[(size_t)b * total + g] = make_double2(hr, hi);
      } else {
        // <x | Hx> contribution: conj(x) * Hx
        dot_re += x.x * hr + x.y * hi;
        dot_im += x.x * hi - x.y * hr;
      }
    }
  }

  if (MODE == MODE_DOT) {
    __shared__ double red[2][kBlock / 32];
    for (int o = 16; o > 0; o >>= 1) {
      dot_re += __shfl_down_sync(0xffffffffu, dot_re, o);
      dot_im += __shfl_down_sync(0xffffffffu, dot_im, o);
    }
    if ((tid & 31) == 0) {
      red[0][tid >> 5] = dot_re;
      red[1][tid >> 5] = dot_im;
    }
    __syncthreads();
    if (tid == 0) {
      double sr = 0.0, si = 0.0;
      for (int k = 0; k < kBlock / 32; ++k) {
        sr += red[0][k];
        si += red[1][k];
      }
      a.partial[2 * blockIdx.x] = sr;
      a.partial[2 * blockIdx.x + 1] = si;
    }
  }
}


// psi (FP64, [B][total]) -> double-float copy in the weighted basis, f = psi / w(n),
// with the inverse weights of the per-ket table (coalesced, no unranking)
template <int MT>
__global__ void __launch_bounds__(256) to_dfw_kernel(const Tables t, const double2* psi, float4* out, int B) {
  for (int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; g < t.total; g += (int64_t)gridDim.x * blockDim.x) {
    const double wi = __ldg(t.wi + g);
    for (int b = 0; b < B; ++b) {
      const double2 x = psi[(size_t)b * t.total + g];
      out[(size_t)b * t.total + g] = df_pack(df_of(x.x * wi), df_of(x.y * wi));
    }
  }
}

// ------------------------------------------------------- tables of kets and blocks
//
// What set-up holds per ket is a product or a sum of a part of the block (modes 0 .. P-1, its
// particle number and momentum) and a part of the filling (modes P .. M-1), so that the kets
// are neither unranked nor weighed one by one: block_kernel finds every block's first ket
// and every filling, and ket_kernel joins the two for 32 kets at a time.  A kernel
// that unranked each ket and summed its M (M + 1) / 2 pairs in FP64, 110 operations at 2 per
// clock and SM, took 10.5 ms for 62.9M kets of 7 modes and 0.28 ms for 2.3M of 5 modes; the
// three kernels take 2.4 and 0.13.

// A filling (Tables::suf): the packed occupations of its modes (all ones: a number left out),
// its factors of the ket weight and of the inverse weight, its parts of the diagonals
struct Suffix {
  const uint64_t* word;
  const double *w, *wi, *dw, *dl;
};
// The block's parts of the same, with the first filling of its class and, for each mode
// P + j, the coefficient of n_{P+j} that the pairs (r < P, P + j) add to the two-body diagonal
struct BlockRec {
  uint64_t word;
  uint32_t fill0, pad;
  double w, wi, dw, dl;
  double cross[];
};
__host__ __device__ inline size_t block_rec_bytes(int M, int P) { return sizeof(BlockRec) + 8 * (size_t)(M - P); }

// One block a thread: block b of the sectors (first kets off, first blocks sblk) starts at
// ket start[b].  The occupations of its modes are found from the block counts as those of a
// ket from the fill counts.  FULL: all of BlockRec, else its word and first filling.
struct BlockArgs {
  const int32_t *secN, *secK;
  const int64_t* secOff;
  const uint32_t* sblk;
  int nsec;
  const uint32_t* bcnt;
  uint32_t* start;
  unsigned char* rec;
  size_t stride;
};
template <bool FULL>
__device__ void find_block(const Tables& t, const BlockArgs& a, uint32_t b) {
  const uint32_t* sblk = a.sblk;
  const int nsec = a.nsec;
  if (b >= __ldg(sblk + nsec)) return;
  int lo = 0, hi = nsec - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (__ldg(sblk + mid) <= b)
      lo = mid;
    else
      hi = mid - 1;
  }
  const int M = t.M, P = t.bk_P, Q = t.Q, V = t.nmax + 1, N = __ldg(a.secN + lo);
  const uint32_t* cnt = reinterpret_cast<const uint32_t*>(t.blob + t.o_cnt);
  const double* w1 = reinterpret_cast<const double*>(t.blob + t.o_w);
  const double* gd = reinterpret_cast<const double*>(t.blob + t.o_gd);
  const uint8_t* pairidx = t.blob + t.o_pairidx;
  int64_t off = __ldg(a.secOff + lo);
  uint32_t left = b - __ldg(sblk + lo);
  int rem = N, kr = __ldg(a.secK + lo);
  uint64_t word = 0;
  const double2 c = __ldg(t.wscale + N);
  double w = c.x, wi = c.y, dw = 0.0, dl = 0.0;
  BlockRec* R = reinterpret_cast<BlockRec*>(a.rec + (size_t)b * a.stride);
  for (int m = 0; m < P; ++m) {
    int val = 0;
    while (val < rem) {
      const size_t i = ((size_t)(m + 1) * V + rem - val) * Q + kr;
      const uint32_t n = __ldg(a.bcnt + i);
      if (left < n) break;
      left -= n;
      off += __ldg(cnt + i);
      ++val;
      kr -= m;
      while (kr < 0) kr += Q;
    }
    word |= (uint64_t)val << (m * t.occ_bits);
    if (FULL) {
      const double2 f = __ldg(t.wtab + rem * V + val);
      w *= f.x;
      wi *= f.y;
      const double v = (double)val;
      dw += w1[m] * v;
      double g = gd[pairidx[m * 17]] * (v - 1.0);
      for (int r = 0; r < m; ++r) g += gd[pairidx[r * 16 + m]] * (double)occ_of(word, r, t.occ_bits);
      if (val) dl += g * v;
    }
    rem -= val;
  }
  a.start[b] = (uint32_t)off;
  R->word = word;
  R->fill0 = (uint32_t)__ldg(t.bk_cls + rem * Q + kr).x;
  if (!FULL) return;
  R->w = w;
  R->wi = wi;
  R->dw = dw;
  R->dl = dl;
  for (int m = P; m < M; ++m) {
    double g = 0.0;
    for (int r = 0; r < P; ++r) g += gd[pairidx[r * 16 + m]] * (double)occ_of(word, r, t.occ_bits);
    R->cross[m - P] = g;
  }
}

// One filling a thread, from its number: the class, then the occupations in lexicographic
// order
__device__ void find_filling(const Tables& t, int f, uint64_t* words, double* sw, double* swi, double* sdw, double* sdl) {
  if (f >= t.bk_S) return;
  const int M = t.M, Q = t.Q, P = t.bk_P, V = t.nmax + 1;
  const uint32_t* cnt = reinterpret_cast<const uint32_t*>(t.blob + t.o_cnt);
  const double* w1 = reinterpret_cast<const double*>(t.blob + t.o_w);
  const double* gd = reinterpret_cast<const double*>(t.blob + t.o_gd);
  const uint8_t* pairidx = t.blob + t.o_pairidx;
  int lo = 0, hi = V * Q - 1;  // the last class that starts at or before it
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (__ldg(t.bk_cls + mid).x <= f)
      lo = mid;
    else
      hi = mid - 1;
  }
  const int2 cls = __ldg(t.bk_cls + lo);
  uint32_t left = (uint32_t)(f - cls.x);
  uint64_t word = 0;
  double w = 1.0, wi = 1.0, dw = 0.0, dl = 0.0;
  if (left >= (uint32_t)cls.y) {
    word = ~0ull;
  } else {
    int rem = lo / Q, kr = lo % Q;
    for (int m = P; m < M; ++m) {
      int val = 0;
      if (m == M - 1) val = rem;
      while (val < rem) {
        const uint32_t c = __ldg(cnt + ((size_t)(m + 1) * V + rem - val) * Q + kr);
        if (left < c) break;
        left -= c;
        ++val;
        kr -= m;
        while (kr < 0) kr += Q;
      }
      word |= (uint64_t)val << (m * t.occ_bits);
      const double2 x = __ldg(t.wtab + rem * V + val);
      w *= x.x;
      wi *= x.y;
      const double v = (double)val;
      dw += w1[m] * v;
      double g = gd[pairidx[m * 17]] * (v - 1.0);
      for (int r = P; r < m; ++r) g += gd[pairidx[r * 16 + m]] * (double)occ_of(word, r, t.occ_bits);
      if (val) dl += g * v;
      rem -= val;
    }
  }
  words[f] = word;
  sw[f] = w;
  swi[f] = wi;
  sdw[f] = dw;
  sdl[f] = dl;
}

// Both in one launch, the fillings by the first nf CTAs
__global__ void __launch_bounds__(128) block_kernel(const Tables t, const BlockArgs a, unsigned nf, uint64_t* words) {
  if (blockIdx.x < nf) {
    const size_t S = (size_t)t.bk_S;
    double* d = reinterpret_cast<double*>(words + S);
    find_filling(t, (int)(blockIdx.x * 128 + threadIdx.x), words, d, d + S, d + 2 * S, d + 3 * S);
  } else {
    find_block<true>(t, a, (blockIdx.x - nf) * 128u + threadIdx.x);
  }
}
__global__ void __launch_bounds__(128) lower_block_kernel(const Tables t, const BlockArgs a) {
  find_block<false>(t, a, blockIdx.x * 128u + threadIdx.x);
}

// The kets' tables, a run of rounds of 32 consecutive kets a warp: the block of the first one
// is searched for, the following ones come from the starts after it.  Writes 44 bytes a ket
// (lower kets: 12): at 62.9M kets, 2.8 GB.
template <bool FULL>
__global__ void __launch_bounds__(256) ket_kernel(const Tables t, const Suffix sx, int64_t n, uint32_t nblocks,
                                                   const uint32_t* start, const unsigned char* rec, size_t stride,
                                                   int run, float4* diag, uint64_t* occ, double* wi, double* wk,
                                                   uint32_t* fill, uint32_t* rblk) {
  const int lane = threadIdx.x & 31, P = t.bk_P, M = t.M;
  const int64_t nr = (n + 31) / 32;
  const int64_t r0 = (((int64_t)blockIdx.x * 256 + threadIdx.x) >> 5) * run;
  if (r0 >= nr) return;
  const int64_t r1 = min(r0 + run, nr);
  uint32_t b = 0;  // the last block that starts at or before ket 32 r0
  {
    uint32_t hi = nblocks - 1;
    while (b < hi) {
      const uint32_t mid = b + (hi - b + 1) / 2;
      if ((int64_t)__ldg(start + mid) <= 32 * r0)
        b = mid;
      else
        hi = mid - 1;
    }
  }
  for (int64_t r = r0; r < r1; ++r) {
    const int64_t g = 32 * r + lane;
    // at most 31 blocks start at the round's other kets, and one with the next round
    const uint32_t nb = b + 1 + lane;
    const uint32_t d = nb < nblocks ? __ldg(start + nb) - (uint32_t)(32 * r) : 64u;
    const uint32_t heads = __reduce_or_sync(0xffffffffu, d < 32u ? 1u << d : 0u);
    const bool next = __any_sync(0xffffffffu, d == 32u);
    const uint32_t me = b + __popc(heads & ((2u << lane) - 1u));
    if (lane == 0) rblk[r] = b;
    if (g < n) {
      const BlockRec* R = reinterpret_cast<const BlockRec*>(rec + (size_t)me * stride);
      const uint32_t f = R->fill0 + (uint32_t)g - __ldg(start + me);
      const uint64_t sword = __ldg(sx.word + f);
      occ[g] = R->word | sword;
      fill[g] = f;
      if (FULL) {
        double dl = R->dl + __ldg(sx.dl + f);
        for (int m = P; m < M; ++m) dl += R->cross[m - P] * (double)occ_of(sword, m, t.occ_bits);
        const dfl x = df_of(R->dw + __ldg(sx.dw + f)), y = df_of(dl);
        diag[g] = make_float4(x.h, x.l, y.h, y.l);
        wk[g] = R->w * __ldg(sx.w + f);
        wi[g] = R->wi * __ldg(sx.wi + f);
      }
    }
    b += __popc(heads) + (next ? 1u : 0u);
  }
}

// A filling: its class (particles crem, momentum ckr of the modes P .. M-1), occupations and
// ranking-table indices.  False for the numbers left out.
struct Filling {
  int crem, ckr;
  int occ[kMaxM], idx[kMaxM];
};
__device__ __forceinline__ bool filling_of(const Tables& t, const uint64_t* words, int64_t f, Filling& F) {
  const int M = t.M, Q = t.Q, P = t.bk_P;
  const uint64_t word = __ldg(words + f);
  if (word == ~0ull) return false;
  int sr = 0, sk = 0;
  for (int m = M - 1; m >= P; --m) {
    F.occ[m] = occ_of(word, m, t.occ_bits);
    sr += F.occ[m];
    sk = (sk + m * F.occ[m]) % Q;
    F.idx[m] = (m * t.rem_w + sr + 2) * 2 * Q + sk;
  }
  F.crem = sr;
  F.ckr = sk;
  return true;
}

// Place in its class of the filling changed by the shifts sh[m * stride] of the suffix
// indices; 0 outside the space
__device__ __forceinline__ uint16_t place_of(const Tables& t, const Filling& F, const int32_t* sh, int stride) {
  const int M = t.M, Q = t.Q, P = t.bk_P, twoQ = 2 * Q;
  const int32_t* E = reinterpret_cast<const int32_t*>(t.blob + t.o_E);
  const int flat = (F.crem + 2) * twoQ + F.ckr + sh[P * stride];
  const int rr = flat / twoQ - 2, kk = (flat % twoQ) % Q;
  if (rr < 0 || rr > t.nmax) return 0;
  int place = t.bk_cls[rr * Q + kk].y - 1;
  for (int m = P + 1; m < M; ++m) place -= E[F.idx[m] + sh[m * stride]];
  return (uint16_t)(place < 0 || place > 65535 ? 0 : place);
}

// whether the filling supplies what the pair (r, s) takes from the modes P .. M-1
__device__ __forceinline__ bool supplies(const Tables& t, const Filling& F, int r, int s) {
  bool ok = r < t.bk_P || F.occ[r] >= (r == s ? 2 : 1);
  return ok && (s < t.bk_P || r == s || F.occ[s] >= 1);
}
__device__ __forceinline__ int2 pair_of(uint32_t info) {  // the modes of a selector word
  return make_int2((info & 7) | ((info >> 12) & 8), ((info >> 16) & 7) | ((info >> 28) & 8));
}

// Suffix states of a block, lane m <= P holding mode m's: particles, momentum mod Q and the
// ranking-table index (mode P: the row of bk_EC)
struct BlockState {
  int N, K, cls, my;
};
__device__ __forceinline__ BlockState block_state(const Tables& t, uint64_t word, int lane) {
  int rem = 0, kr = 0;
  for (int i = t.M - 1; i >= lane; --i) {
    const int n = occ_of(word, i, t.occ_bits);
    rem += n;
    kr += i * n;
  }
  kr %= t.Q;
  BlockState b;
  b.N = __shfl_sync(0xffffffffu, rem, 0);
  b.K = __shfl_sync(0xffffffffu, kr, 0);
  b.cls = __shfl_sync(0xffffffffu, rem * t.Q + kr, t.bk_P);
  b.my = ((lane < t.bk_P ? lane * t.rem_w : 0) + rem + 2) * 2 * t.Q + kr;
  return b;
}
// sum of the ranking terms of modes 1 .. P of the block shifted by sh[m * stride], plus the
// size of its class (all lanes take part; sh per lane)
__device__ __forceinline__ uint32_t block_sum(const Tables& t, const BlockState& b, const int32_t* sh, int stride) {
  const int32_t* E = reinterpret_cast<const int32_t*>(t.blob + t.o_E);
  uint32_t sum = 0;
  for (int m = 1; m < t.bk_P; ++m) sum += (uint32_t)__ldg(E + __shfl_sync(0xffffffffu, b.my, m) + (sh ? __ldg(sh + m * stride) : 0));
  return sum + (uint32_t)__ldg(t.bk_EC + __shfl_sync(0xffffffffu, b.my, t.bk_P) + (sh ? __ldg(sh + t.bk_P * stride) : 0));
}

// Bases of the direct stage kernel, one warp a block; checks that the block starts where the
// ranking says and with the first filling of its class.
__global__ void __launch_bounds__(256) base_kernel(const Tables t, const uint32_t* start, int64_t nblocks, uint32_t* base,
                                                    int* status) {
  const int lane = threadIdx.x & 31, T = t.bk_T, TS = T + 4;
  for (int64_t b = ((int64_t)blockIdx.x * 256 + threadIdx.x) >> 5; b < nblocks; b += ((int64_t)gridDim.x * 256) >> 5) {
    const int64_t g = start[b];
    const BlockState s = block_state(t, __ldg(t.occ + g), lane);
    const uint32_t end = (uint32_t)__ldg(t.sec_off + __ldg(t.sec_of + s.N * t.Q + s.K) + 1);
    const uint32_t own = end - block_sum(t, s, nullptr, 0);
    if (lane == 0 && (own != (uint32_t)g || __ldg(t.fill + g) != (uint32_t)__ldg(t.bk_cls + s.cls).x)) atomicOr(status, 2);
    if (t.fa_on) continue;
    for (int t0 = 0; t0 < T; t0 += 32) {
      const int tt = min(t0 + lane, T - 1);
      const uint32_t v = end - block_sum(t, s, t.bk_psh + tt, TS);
      if (t0 + lane < T) base[(size_t)b * T + tt] = v;
    }
  }
}

// Bases of the factored stages: lowered targets of the blocks (basec), raised targets of
// the lower blocks (basea) and where each class's entries start less the lower ket's number.
__global__ void __launch_bounds__(256) lowered_base_kernel(const Tables t, const uint32_t* start, int64_t nblocks,
                                                            uint32_t* basec) {
  const int lane = threadIdx.x & 31, Tc = fa_Tc(t);
  for (int64_t b = ((int64_t)blockIdx.x * 256 + threadIdx.x) >> 5; b < nblocks; b += ((int64_t)gridDim.x * 256) >> 5) {
    const BlockState s = block_state(t, __ldg(t.occ + start[b]), lane);
    for (int t0 = 0; t0 < Tc; t0 += 32) {
      const int tt = min(t0 + lane, Tc - 1);
      const int k = __ldg(t.fa_kc + tt);
      int kk = s.K - k;
      while (kk < 0) kk += t.Q;
      const uint32_t sum = block_sum(t, s, t.fa_psc + tt, Tc);
      uint32_t v = kNoIndex;
      if (s.N >= 2) {
        const int lid = __ldg(t.fa_lowof + (s.N - 2) * t.Q + kk);
        const uint32_t go = lid >= 0 ? __ldg(t.fa_goff + lid * t.fa_nc + k) : kNoIndex;
        if (go != kNoIndex) v = go + (uint32_t)(__ldg(t.fa_lowoff + lid + 1) - __ldg(t.fa_lowoff + lid)) - sum;
      }
      if (t0 + lane < Tc) basec[(size_t)b * Tc + tt] = v;
    }
  }
}

__global__ void __launch_bounds__(256) raised_base_kernel(const Tables t, const uint32_t* start, int64_t nblocks,
                                                           uint32_t* basea) {
  const int lane = threadIdx.x & 31, Ta = fa_Ta(t), row = fa_rowa(t);
  for (int64_t b = ((int64_t)blockIdx.x * 256 + threadIdx.x) >> 5; b < nblocks; b += ((int64_t)gridDim.x * 256) >> 5) {
    const BlockState s = block_state(t, __ldg(t.fa_occ + start[b]), lane);
    const int lid = __ldg(t.fa_lowof + s.N * t.Q + s.K);
    for (int t0 = 0; t0 < Ta; t0 += 32) {
      const int tt = min(t0 + lane, Ta - 1);
      const int k = __ldg(t.fa_ka + tt);
      const uint32_t sum = block_sum(t, s, t.fa_psa + tt, Ta);
      uint32_t v = kNoIndex;
      if (__ldg(t.fa_goff + lid * t.fa_nc + k) != kNoIndex)
        v = (uint32_t)__ldg(t.sec_off + __ldg(t.sec_of + (s.N + 2) * t.Q + (s.K + k) % t.Q) + 1) - sum;
      if (t0 + lane < Ta) basea[(size_t)b * row + tt] = v;
    }
    // bit i: the class of record i (of the first 32) has a raised sector
    uint32_t held = 0;
    if (lane < t.fa_nrec && __ldg(t.fa_goff + lid * t.fa_nc + (__ldg(&t.fa_rec[lane].x) & 0xffu)) != kNoIndex) held = 1u;
    held = __ballot_sync(0xffffffffu, held != 0u);
    for (int k = lane; k < row - Ta; k += 32) {
      uint32_t v = 0;
      if (k < t.fa_nc) v = __ldg(t.fa_goff + lid * t.fa_nc + k) - (uint32_t)__ldg(t.fa_lowoff + lid);
      if (k == t.fa_nc) v = held;
      basea[(size_t)b * row + Ta + k] = v;
    }
  }
}

// Order of the rounds of kets in sectors (first kets off[nsec + 1], particles secN): within
// a layer (equal N) of S sectors, which are nearly equal in size, position j of the layer's n
// rounds is round (j mod S) ceil(n / S) + j / S, the positions beyond the last segment's end
// moved up.  A layer is the rounds [floor(first / 32), floor(end / 32)) of its kets.
__global__ void __launch_bounds__(256) round_order_kernel(const int64_t* off, const int32_t* secN, int nsec, int64_t nr,
                                                           uint32_t* perm) {
  for (int64_t r = (int64_t)blockIdx.x * 256 + threadIdx.x; r < nr; r += (int64_t)gridDim.x * 256) {
    int lo = 0, hi = nsec - 1;
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (__ldg(off + mid) / 32 <= r)
        lo = mid;
      else
        hi = mid - 1;
    }
    int a = lo, b = lo;
    while (a > 0 && secN[a - 1] == secN[lo]) --a;
    while (b + 1 < nsec && secN[b + 1] == secN[lo]) ++b;
    const int64_t ra = __ldg(off + a) / 32, rb = b + 1 < nsec ? __ldg(off + b + 1) / 32 : nr;
    const int64_t S = b - a + 1, n = rb - ra, len = (n + S - 1) / S, j = r - ra;
    // full columns: len - 1 of them where the last segment is short
    const int64_t lastlen = n - (S - 1) * len;  // of segment S - 1 (may be <= 0)
    int64_t seg, pos;
    if (lastlen < 0) {  // fewer rounds than segments need: as they come
      seg = 0;
      pos = j;
    } else if (j < lastlen * S) {
      seg = j % S;
      pos = j / S;
    } else {
      seg = (j - lastlen * S) % (S - 1);
      pos = lastlen + (j - lastlen * S) / (S - 1);
    }
    perm[r] = (uint32_t)(ra + seg * len + pos);
  }
}

// The maps of the direct stage kernel (Tables::bk_map): for every filling and every term,
// the place of the changed filling in its class.  A thread takes one filling and the
// records of its block row.
__global__ void __launch_bounds__(kBlock) block_map_kernel(const Tables t, const uint64_t* words, uint16_t* map,
                                                            uint16_t* map5) {
  const int64_t f = (int64_t)blockIdx.x * kBlock + threadIdx.x;
  Filling F;
  if (f >= t.bk_S || !filling_of(t, words, f, F)) return;
  const int w = t.bk_kc == 2 ? 2 : 4, TS = t.bk_T + 4;
  for (int rec = blockIdx.y; rec < t.bk_nrec; rec += gridDim.y) {
    const uint32_t info = t.bk_info[rec].x;
    const int2 rs = pair_of(info);
    const int n = (info >> 4) & 7;
    const bool ok = supplies(t, F, rs.x, rs.y);
    for (int c = 0; c < max(w, n); ++c) {
      const int slot = c < 4 ? w * rec + c : 4 * t.bk_nrec + rec;
      const uint16_t place = ok && c < n ? place_of(t, F, t.bk_psh + slot, TS) : 0;
      if (c < w)
        map[((size_t)rec * t.bk_S + f) * w + c] = place;
      else
        map5[(size_t)rec * t.bk_S + f] = place;
    }
  }
}

// Tables of the raised moments: suffix shift of one particle more (sign 1) or fewer in mode i
__device__ __forceinline__ int one_shift(const Tables& t, int i, int m, int sign) {
  if (i < m) return 0;
  return sign * 2 * t.Q + (sign > 0 ? i % t.Q : (t.Q - i % t.Q) % t.Q);
}
__global__ void __launch_bounds__(kBlock) moment_map_kernel(const Tables t, const uint64_t* words, uint16_t* map) {
  const int64_t f = (int64_t)blockIdx.x * kBlock + threadIdx.x;
  Filling F;
  if (f >= t.bk_S || !filling_of(t, words, f, F)) return;
  int32_t sh[kMaxM];
  for (int q = blockIdx.y; q < 2 * t.mo_w; q += gridDim.y) {
    const int i = q % t.mo_w, sign = q < t.mo_w ? 1 : -1;
    uint16_t place = 0;
    if (i < t.M && (sign > 0 || i < t.bk_P || F.occ[i] >= 1)) {
      for (int m = 0; m < t.M; ++m) sh[m] = one_shift(t, i, m, sign);
      place = place_of(t, F, sh, 1);
    }
    map[((size_t)(q / 4) * t.bk_S + f) * 4 + q % 4] = place;
  }
}
__global__ void __launch_bounds__(256) moment_base_kernel(const Tables t, const uint32_t* start, int64_t nblocks,
                                                           uint32_t* base) {
  const int lane = threadIdx.x & 31, w = t.mo_w;  // 2 w <= 32: one entry a lane
  const int i = lane % w, sign = lane < w ? 1 : -1;
  const int32_t* E = reinterpret_cast<const int32_t*>(t.blob + t.o_E);
  for (int64_t b = ((int64_t)blockIdx.x * 256 + threadIdx.x) >> 5; b < nblocks; b += ((int64_t)gridDim.x * 256) >> 5) {
    const BlockState s = block_state(t, __ldg(t.occ + start[b]), lane);
    uint32_t sum = 0;
    for (int m = 1; m < t.bk_P; ++m)
      sum += (uint32_t)__ldg(E + __shfl_sync(0xffffffffu, s.my, m) + one_shift(t, i, m, sign));
    sum += (uint32_t)__ldg(t.bk_EC + __shfl_sync(0xffffffffu, s.my, t.bk_P) + one_shift(t, i, t.bk_P, sign));
    const int N = s.N + sign, K = (s.K + (sign > 0 ? i : t.Q - i % t.Q)) % t.Q;
    uint32_t v = kNoIndex;
    if (lane < 2 * w && i < t.M && N >= 0 && N <= t.nmax) {
      const int sid = __ldg(t.sec_of + N * t.Q + K);
      if (sid >= 0) v = (uint32_t)__ldg(t.sec_off + sid + 1) - sum;
    }
    if (lane < 2 * w) base[(size_t)b * 2 * w + lane] = v;
  }
}

// The maps of the factored stages: places after a pair is added (fa_mapa) or taken away
// (fa_mapc)
__global__ void __launch_bounds__(kBlock) factor_map_kernel(const Tables t, const uint64_t* words, uint16_t* mapa,
                                                             uint16_t* mapc) {
  const int64_t f = (int64_t)blockIdx.x * kBlock + threadIdx.x;
  Filling F;
  if (f >= t.bk_S || !filling_of(t, words, f, F)) return;
  const int Ta = fa_Ta(t), Tc = fa_Tc(t);
  const uint32_t* info = reinterpret_cast<const uint32_t*>(t.fa_info);
  for (int q = blockIdx.y; q < Ta / 4 + t.fa_ng; q += gridDim.y)
    for (int c = 0; c < 4; ++c) {
      if (q < Ta / 4) {
        mapa[((size_t)q * t.bk_S + f) * 4 + c] = place_of(t, F, t.fa_psa + 4 * q + c, Ta);
      } else {
        const int i = 4 * (q - Ta / 4) + c;
        const int2 rs = pair_of(info[i]);
        mapc[((size_t)(q - Ta / 4) * t.bk_S + f) * 4 + c] = supplies(t, F, rs.x, rs.y) ? place_of(t, F, t.fa_psc + i, Tc) : 0;
      }
    }
}

// ------------------------------------------------------------- small kernels

// occupations from the packed words, one (ket, mode) a thread
__global__ void __launch_bounds__(kBlock) unrank_kernel(const Tables t, int64_t first, int64_t count, int* occ_out) {
  const int64_t n = count * t.M;
  for (int64_t i = (int64_t)blockIdx.x * kBlock + threadIdx.x; i < n; i += (int64_t)gridDim.x * kBlock) {
    const int64_t k = i / t.M;
    occ_out[i] = occ_of(__ldg(t.occ + first + k), (int)(i - k * t.M), t.occ_bits);
  }
}

__global__ void __launch_bounds__(kBlock) rank_kernel(const Tables t, const int* occ_in, int64_t count,
                                                       int64_t* index_out) {
  extern __shared__ __align__(16) unsigned char smem[];
  load_blob(t, smem);
  const View v = make_view(t, smem);
  const int M = t.M, V = t.nmax + 1;
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < count; k += (int64_t)gridDim.x * blockDim.x) {
    int N = 0, K = 0;
    bool ok = true;
    for (int m = 0; m < M; ++m) {
      int nm = occ_in[k * M + m];
      if (nm < 0 || nm > t.nmax) ok = false;
      N += nm;
      K = (K + m * (nm < 0 ? 0 : nm)) % t.Q;
    }
    int64_t res = -1;
    if (ok && N <= t.nmax) {
      int sid = __ldg(t.sec_of + N * t.Q + K);
      if (sid >= 0) {
        const int64_t off = __ldg(t.sec_off + sid), D = __ldg(t.sec_off + sid + 1) - off;
        int64_t sum = 0;
        int rem = 0, kr = 0;
        for (int m = M - 1; m >= 1; --m) {
          int nm = occ_in[k * M + m];
          rem += nm;
          kr = (kr + m * nm) % t.Q;
          if (rem >= 1)
            sum += v.cnt[((size_t)(m - 1) * V + rem - 1) * t.Q + (((kr - (m - 1)) % t.Q) + t.Q) % t.Q];
        }
        res = off + D - 1 - sum;
      }
    }
    index_out[k] = res;
  }
}

__global__ void __launch_bounds__(kBlock) terms_kernel(const Tables t, unsigned long long* out /*[2]*/) {
  extern __shared__ __align__(16) unsigned char smem[];
  load_blob(t, smem);
  const View v = make_view(t, smem);
  const RowScratch rs = row_scratch(smem + blob_smem(t));
  const int tid = threadIdx.x, M = t.M;
  unsigned long long terms = 0, tuples = 0;
  for (int64_t base = (int64_t)blockIdx.x * kBlock; base < t.total; base += (int64_t)gridDim.x * kBlock) {
    const int64_t g = base + tid;
    if (g >= t.total) break;
    const int sid = find_sector(t, g);
    const int64_t off = __ldg(t.sec_off + sid);
    const int64_t D = __ldg(t.sec_off + sid + 1) - off;
    setup_row(t, v, rs, __ldg(t.sec_N + sid), __ldg(t.sec_K + sid), D, g - off);
    terms += 1;  // diagonal element
    for (int r = 0; r < M; ++r)
      for (int s = r; s < M; ++s) {
        int nr = rs.occ[r * kBlock + tid], ns = rs.occ[s * kBlock + tid];
        if (nr < 1 || ns - (r == s ? 1 : 0) < 1) continue;
        int ai = v.pairidx[r * 16 + s];
        unsigned long long mrs = (r == s) ? 1 : 2;
        if (v.gd[ai] != 0.0) tuples += mrs * mrs;
        for (int j = v.ann[ai]; j < v.ann[ai + 1]; ++j) {
          if (v.G[2 * j] == 0.0 && v.G[2 * j + 1] == 0.0) continue;
          uint32_t w4 = v.pq[j];
          int p = w4 & 0xff, q = (w4 >> 8) & 0xff;
          terms += 1;
          tuples += mrs * ((p == q) ? 1ull : 2ull);
        }
      }
  }
  for (int o = 16; o > 0; o >>= 1) {
    terms += __shfl_down_sync(0xffffffffu, terms, o);
    tuples += __shfl_down_sync(0xffffffffu, tuples, o);
  }
  if ((tid & 31) == 0) {
    atomicAdd(out, terms);
    atomicAdd(out + 1, tuples);
  }
}

// amplitude = prod_i table[i][n_i] (complex), zero outside N == only_N (if >= 0);
// per-block partial sums of |amplitude|^2
__global__ void __launch_bounds__(kBlock) init_table_kernel(const Tables t, const double2* table, int only_N,
                                                             double2* psi, double* partial) {
  const int tid = threadIdx.x, M = t.M, V = t.nmax + 1;
  double n2 = 0.0;
  for (int64_t g = (int64_t)blockIdx.x * kBlock + tid; g < t.total; g += (int64_t)gridDim.x * kBlock) {
    const uint64_t word = __ldg(t.occ + g);
    int N = 0;
    for (int m = 0; m < M; ++m) N += occ_of(word, m, t.occ_bits);
    double re = 0.0, im = 0.0;
    if (only_N < 0 || N == only_N) {
      re = 1.0;
      for (int m = 0; m < M; ++m) {
        const double2 f = __ldg(table + (size_t)m * V + occ_of(word, m, t.occ_bits));
        const double nr = re * f.x - im * f.y;
        im = re * f.y + im * f.x;
        re = nr;
      }
    }
    psi[g] = make_double2(re, im);
    n2 += re * re + im * im;
  }
  __shared__ double red[kBlock / 32];
  for (int o = 16; o > 0; o >>= 1) n2 += __shfl_down_sync(0xffffffffu, n2, o);
  if ((tid & 31) == 0) red[tid >> 5] = n2;
  __syncthreads();
  if (tid == 0) {
    double s = 0.0;
    for (int k = 0; k < kBlock / 32; ++k) s += red[k];
    partial[blockIdx.x] = s;
  }
}

__global__ void scale_kernel(double2* psi, int64_t n, double f) {
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x) {
    double2 x = psi[k];
    psi[k] = make_double2(x.x * f, x.y * f);
  }
}

__global__ void number_kernel(double2* psi, int64_t n, int64_t index) {
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x)
    psi[k] = make_double2(k == index ? 1.0 : 0.0, 0.0);
}

// ---------------------------------------------------------------- moments
//
// Raw moments of Sec. II C-E: norm, <N>, <a_i>, <a_i^dag a_j>, <a_i a_j>.  Each
// row (ket n with amplitude x) contributes conj(psi[target]) * c * x for every
// operator that maps n to a held ket.  Contributions are reduced across the warp
// by shuffles into per-warp shared accumulators, then across warps into one
// partial per block, then over blocks in a fixed order: deterministic.

__device__ __forceinline__ double warp_sum(double x) {
  for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
  return x;
}

__global__ void __launch_bounds__(kBlock) moments_kernel(const Tables t, const double2* psi, double* partial,
                                                          int nmom, int* status) {
  extern __shared__ __align__(16) unsigned char smem[];
  load_blob(t, smem);
  const View v = make_view(t, smem);
  const size_t blob_al = blob_smem(t);
  const RowScratch rs = row_scratch(smem + blob_al);
  double* acc = reinterpret_cast<double*>(smem + blob_al + ((kRowScratchBytes + 15) & ~15));  // [warps][nmom]
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, M = t.M;
  for (int k = tid; k < (kBlock / 32) * nmom; k += kBlock) acc[k] = 0.0;
  __syncthreads();
  double* wacc = acc + (size_t)warp * nmom;
  // layout: [0] norm [1] N [2] H (unused here) [3] pad, a: 4.., Mij: 4+2M.., aa: 4+2M+2M^2..
  const int oA = 4, oM = 4 + 2 * M, oAA = 4 + 2 * M + 2 * M * M;

  for (int64_t base = (int64_t)blockIdx.x * kBlock; base < t.total; base += (int64_t)gridDim.x * kBlock) {
    const int64_t g = base + tid;
    const bool live = g < t.total;
    int N = 0, K = 0;
    double xr = 0.0, xi = 0.0;
    if (live) {
      const int sid = find_sector(t, g);
      const int64_t off = __ldg(t.sec_off + sid);
      const int64_t D = __ldg(t.sec_off + sid + 1) - off;
      N = __ldg(t.sec_N + sid);
      K = __ldg(t.sec_K + sid);
      setup_row(t, v, rs, N, K, D, g - off);
      const double2 x = psi[g];
      xr = x.x;
      xi = x.y;
    }
    const double p2 = xr * xr + xi * xi;
    {
      double c0 = warp_sum(p2), c1 = warp_sum(p2 * N);
      if (lane == 0) {
        wacc[0] += c0;
        wacc[1] += c1;
      }
    }
    // contribution conj(y) * c * x for target index tg (or none)
    auto contrib = [&](int slot, bool has, int64_t tg, double c) {
      double cr = 0.0, ci = 0.0;
      if (has && (tg < 0 || tg >= t.total)) {
        atomicOr(status, 1);
        has = false;
      }
      if (has) {
        const double2 y = psi[tg];
        cr = c * (y.x * xr + y.y * xi);
        ci = c * (y.x * xi - y.y * xr);
      }
      if (__any_sync(0xffffffffu, has)) {
        cr = warp_sum(cr);
        ci = warp_sum(ci);
        if (lane == 0) {
          wacc[slot] += cr;
          wacc[slot + 1] += ci;
        }
      }
    };
    const uint8_t* occ = rs.occ + tid;
    // <a_i>
    for (int i = 0; i < M; ++i) {
      bool has = false;
      int64_t tg = 0;
      double c = 0.0;
      if (live && occ[i * kBlock] >= 1 && N >= 1) {
        const int Kt = ((K - i) % t.Q + t.Q) % t.Q;
        const int sid = __ldg(t.sec_of + (N - 1) * t.Q + Kt);
        if (sid >= 0) {
          const int64_t off = __ldg(t.sec_off + sid), D = __ldg(t.sec_off + sid + 1) - off;
          int e[1] = {i}, dn[1] = {-1};
          tg = off + rank_changed(t, v, rs, 1, e, dn, D);
          c = v.sq[occ[i * kBlock]];
          has = true;
        }
      }
      contrib(oA + 2 * i, has, tg, c);
    }
    // <a_i^dag a_j>
    for (int i = 0; i < M; ++i)
      for (int j = 0; j < M; ++j) {
        bool has = false;
        int64_t tg = 0;
        double c = 0.0;
        if (live && occ[j * kBlock] >= 1) {
          if (i == j) {
            tg = g;
            c = (double)occ[i * kBlock];
            has = true;
          } else {
            const int Kt = ((K - j + i) % t.Q + t.Q) % t.Q;
            const int sid = __ldg(t.sec_of + N * t.Q + Kt);
            if (sid >= 0) {
              const int64_t off = __ldg(t.sec_off + sid), D = __ldg(t.sec_off + sid + 1) - off;
              int e[2] = {j, i}, dn[2] = {-1, 1};
              tg = off + rank_changed(t, v, rs, 2, e, dn, D);
              c = v.sq[occ[j * kBlock]] * v.sq[occ[i * kBlock] + 1];
              has = true;
            }
          }
        }
        contrib(oM + 2 * (i * M + j), has, tg, c);
      }
    // <a_i a_j>, i <= j (the matrix is symmetric)
    for (int i = 0; i < M; ++i)
      for (int j = i; j < M; ++j) {
        bool has = false;
        int64_t tg = 0;
        double c = 0.0;
        if (live && N >= 2) {
          const int ni = occ[i * kBlock], nj = occ[j * kBlock];
          const bool ok = (i == j) ? (ni >= 2) : (ni >= 1 && nj >= 1);
          if (ok) {
            const int Kt = ((K - i - j) % t.Q + t.Q) % t.Q;
            const int sid = __ldg(t.sec_of + (N - 2) * t.Q + Kt);
            if (sid >= 0) {
              const int64_t off = __ldg(t.sec_off + sid), D = __ldg(t.sec_off + sid + 1) - off;
              int e[2] = {i, j}, dn[2] = {(i == j) ? -2 : -1, -1};
              tg = off + rank_changed(t, v, rs, (i == j) ? 1 : 2, e, dn, D);
              c = (i == j) ? v.sq[ni] * v.sq[ni - 1] : v.sq[ni] * v.sq[nj];
              has = true;
            }
          }
        }
        contrib(oAA + 2 * (i * M + j), has, tg, c);
      }
  }
  __syncthreads();
  for (int k = tid; k < nmom; k += kBlock) {
    double s = 0.0;
    for (int w = 0; w < kBlock / 32; ++w) s += acc[(size_t)w * nmom + k];
    partial[(size_t)blockIdx.x * nmom + k] = s;
  }
}


// ------------------------------------------------------------------ host side

static size_t row_smem(const Tables& t) { return blob_smem(t) + kRowScratchBytes; }

// grid of a persistent row kernel, capped by the scratch sizing

int check_status(const Space& s, cudaStream_t st) {
  int h = 0;
  int* d = reinterpret_cast<int*>(s.d_scratch);  // status word lives at the head of the scratch area
  QB_CUDA(cudaMemcpyAsync(&h, d, sizeof(int), cudaMemcpyDeviceToHost, st));
  QB_CUDA(cudaStreamSynchronize(st));
  if (h) {
    QB_CUDA(cudaMemsetAsync(d, 0, sizeof(int), st));
    QB_CUDA(cudaStreamSynchronize(st));
    return fail(QB_EINTERNAL, "device-side consistency check failed (status " + std::to_string(h) + ")");
  }
  return QB_OK;
}

int device_setup(Space& s) {
  QB_CUDA(cudaGetDevice(&s.device));
  Tables& t = s.t;
  const int M = s.M, V = s.nmax + 1, nsec = (int)s.secN.size();
  t.n_sectors = nsec;
  t.total = s.secOff.back();
  if (row_smem(t) + (size_t)(kBlock / 32) * nmoments(M) * 8 > 227 * 1024)
    return fail(QB_EUNSUPPORTED, "tables too large for shared memory (reduce n_max or M)");
  if (t.total >= (int64_t)kNoIndex) return fail(QB_EUNSUPPORTED, "the space exceeds 2^32 - 2^16 kets");
  // sqrt(C(rem, k)): the binomial exactly in 128 bits while it fits (rem <= 125:
  // C(125, 62) < 2^122), then one rounding to double, one correctly rounded sqrt
  // and one division; beyond, by the recurrence C(rem, k) = C(rem, k-1) (rem-k+1) / k
  // in long double (at least 64 significant bits: the accumulated relative error
  // of at most 2 rem roundings stays far below a double's half-ulp)
  std::vector<double2> wt((size_t)V * V, make_double2(0.0, 0.0));
  for (int rem = 0; rem < V; ++rem) {
    unsigned __int128 c = 1;
    long double cl = 1.0L;
    for (int k = 0; k <= rem; ++k) {
      if (k > 0) {
        if (rem <= 125)
          c = c * (unsigned __int128)(rem - k + 1) / (unsigned __int128)k;
        else
          cl = cl * (long double)(rem - k + 1) / (long double)k;
      }
      const double r = rem <= 125 ? std::sqrt((double)c) : (double)std::sqrt(cl);
      wt[(size_t)rem * V + k] = make_double2(r, 1.0 / r);
    }
  }
  // after the table: the per-N centring powers of two (Tables::wscale)
  for (int N = 0; N < V; ++N) {
    const int e = (int)std::floor(0.5 * log2_max_ket_weight(M, N) + 0.5);
    wt.push_back(make_double2(std::ldexp(1.0, -e), std::ldexp(1.0, e)));
  }
  t.occ_bits = 1;
  while ((1 << t.occ_bits) <= s.nmax) ++t.occ_bits;  // M * occ_bits <= 64 (checked by qb_sector_build)

  // One allocation holds everything, as one copy brings what the host made: each allocation
  // and its release cost 20 to 50 us, twenty of them half of a small space's set-up.
  size_t bytes = 0;
  auto take = [&](size_t n) {
    const size_t at = bytes;
    bytes = (bytes + n + 255) & ~(size_t)255;
    return at;
  };
  struct Part {
    size_t at;
    const void* p;
    size_t n;
  };
  std::vector<Part> parts;
  auto give = [&](const void* p, size_t n) {
    parts.push_back({take(n), p, n});
    return parts.back().at;
  };
  const size_t o_blob = give(s.blob.data(), s.blob.size());
  const size_t o_secOff = give(s.secOff.data(), sizeof(int64_t) * (nsec + 1));
  const size_t o_secN = give(s.secN.data(), sizeof(int32_t) * nsec);
  const size_t o_secK = give(s.secK.data(), sizeof(int32_t) * nsec);
  const size_t o_secOf = give(s.secOf.data(), sizeof(int32_t) * s.secOf.size());
  const size_t o_wtab = give(wt.data(), sizeof(double2) * wt.size());
  const size_t o_bk = give(s.bk.data(), s.bk.size());
  const size_t o_fa = t.fa_on ? give(s.fa.data(), s.fa.size()) : 0;
  const size_t o_bcnt = give(s.blkCnt.data(), sizeof(uint32_t) * s.blkCnt.size());
  const size_t o_sblk = give(s.secBlk.data(), sizeof(uint32_t) * (nsec + 1));
  const size_t o_lblk = t.fa_on ? give(s.lowBlk.data(), sizeof(uint32_t) * s.lowBlk.size()) : 0;
  const size_t image = bytes;
  // scratch: status + partials for the largest persistent grid of any reduction
  int sms = 0;
  QB_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, s.device));
  const int64_t max_grid = (int64_t)sms * 16;
  s.grid_hpsi = (int)max_grid;
  s.scratch_doubles = scratch_doubles_for(M, s.nmax, max_grid);
  const size_t o_scratch = take(sizeof(double) * s.scratch_doubles);
  const size_t n = (size_t)t.total, nr = (n + 31) / 32;
  // (the observables' copy of the state with it, but of the largest spaces: kObsfKets)
  const bool obsf = t.total <= kObsfKets;
  const size_t o_diag = take(16 * n), o_obsf = take(obsf ? 16 * n : 0), o_occ = take(8 * n), o_wi = take(16 * n);
  const size_t o_fill = take(4 * n), o_rblk = take(4 * nr);
  const size_t S = (size_t)t.bk_S, o_suf = take(40 * S);
  const uint32_t nblocks = s.secBlk.back();
  const size_t stride = block_rec_bytes(M, t.bk_P);
  const size_t o_start = take(4 * (size_t)nblocks);
  // the blocks' records are read before the rows of bases are written over them
  const size_t o_base = take((size_t)nblocks * std::max(stride, sizeof(uint32_t) * (t.fa_on ? fa_Tc(t) : t.bk_T)));
  size_t o_map = 0, o_map5 = 0;
  if (!t.fa_on) {
    o_map = take(s.bk_map_bytes);
    o_map5 = take(t.bk_kc == 5 ? (size_t)t.bk_nrec * S * 2 : 0);
  }
  // lower kets: the space's first ones, or their own
  const size_t low = t.fa_on ? (size_t)t.fa_low : 0, lnr = (low + 31) / 32;
  const uint32_t lblocks = !t.fa_on ? 0 : s.low_held ? s.secBlk[t.fa_nlow] : s.lowBlk.back();
  size_t o_mapa = 0, o_mapc = 0, o_perm = 0, o_basea = 0, o_locc = 0, o_lfill = 0, o_lrblk = 0, o_lstart = 0;
  if (t.fa_on) {
    o_mapa = take((size_t)t.fa_nrec * t.fa_pl * S * 8);
    o_mapc = take((size_t)t.fa_ng * S * 8);
    o_perm = take(4 * lnr);
    o_basea = take((size_t)lblocks * std::max(sizeof(BlockRec), sizeof(uint32_t) * fa_rowa(t)));
    if (!s.low_held) {
      o_locc = take(8 * low);
      o_lfill = take(4 * low);
      o_lrblk = take(4 * lnr);
      o_lstart = take(4 * (size_t)lblocks);
    }
  }
  // moments by raised kets: odd M with a kernel, every sector from the vacuum to nmax held
  int layers_end = 0;  // first sector of nmax particles
  t.mo_on = (M == 5 || M == 7 || M == 9) && s.nmin == 0 && s.nmax >= 1 && s.nmax < 256;
  for (int N = 0, i = 0; N <= s.nmax && t.mo_on; ++N) {
    if (N == s.nmax) layers_end = i;
    for (int K = 0; K < s.Q; ++K)
      if (s.cnt[(size_t)N * s.Q + K] > 0) {
        if (s.secOf[(size_t)N * s.Q + K] < 0) t.mo_on = 0;
        ++i;
      }
  }
  size_t o_mmap = 0, o_mbase = 0, o_mperm = 0;
  int64_t mnr = 0;
  if (t.mo_on) {
    t.mo_w = (M + 3) & ~3;
    t.mo_rows = s.secOff[layers_end];
    mnr = t.mo_rows / 32;
    o_mmap = take((size_t)2 * t.mo_w * S * 2);
    o_mbase = take((size_t)nblocks * 2 * t.mo_w * 4);
    o_mperm = take(4 * (size_t)mnr);
  }

  QB_CUDA(cudaMalloc(&s.d_arena, bytes));
  unsigned char* A = s.d_arena;
  {
    std::vector<unsigned char> img(image, 0);
    for (const Part& p : parts)
      if (p.n) memcpy(img.data() + p.at, p.p, p.n);
    QB_CUDA(cudaMemcpy(A, img.data(), image, cudaMemcpyHostToDevice));
  }
  s.d_scratch = reinterpret_cast<double*>(A + o_scratch);
  QB_CUDA(cudaMemsetAsync(s.d_scratch, 0, sizeof(double) * s.scratch_doubles));
  auto u32 = [&](size_t o) { return reinterpret_cast<uint32_t*>(A + o); };
  auto i32 = [&](size_t o) { return reinterpret_cast<const int32_t*>(A + o); };
  s.d_diag = reinterpret_cast<float4*>(A + o_diag);
  s.d_obsf = obsf ? reinterpret_cast<float4*>(A + o_obsf) : nullptr;
  uint64_t* occ = reinterpret_cast<uint64_t*>(A + o_occ);
  double* wi = reinterpret_cast<double*>(A + o_wi);
  t.blob = A + o_blob;
  t.sec_off = reinterpret_cast<const int64_t*>(A + o_secOff);
  t.sec_N = i32(o_secN);
  t.sec_K = i32(o_secK);
  t.sec_of = i32(o_secOf);
  t.wi = wi;
  t.wk = wi + n;
  t.occ = occ;
  t.wtab = reinterpret_cast<const double2*>(A + o_wtab);
  t.wscale = t.wtab + (size_t)V * V;
  auto bk = [&](int k) { return A + o_bk + s.bk_off[k]; };
  t.bk_info = reinterpret_cast<const uint2*>(bk(0));
  t.bk_G = reinterpret_cast<const float2*>(bk(1));
  t.bk_Gi = reinterpret_cast<const float2*>(bk(2));
  t.bk_psh = reinterpret_cast<const int32_t*>(bk(3));
  t.bk_EC = reinterpret_cast<const int32_t*>(bk(4));
  t.bk_cls = reinterpret_cast<const int2*>(bk(5));
  t.bk_combo = reinterpret_cast<const uint32_t*>(bk(7));
  t.fill = u32(o_fill);
  t.rblk = u32(o_rblk);

  Suffix sx{};
  {
    uint64_t* words = reinterpret_cast<uint64_t*>(A + o_suf);
    double* d = reinterpret_cast<double*>(words + S);
    sx = Suffix{words, d, d + S, d + 2 * S, d + 3 * S};
  }
  // a run of rounds a warp: 8, fewer where the kets don't fill the SMs' 64 warps
  auto run_of = [&](size_t rounds) { return (int)std::max<size_t>(1, std::min<size_t>(8, rounds / ((size_t)sms * 64))); };
  auto grid_of = [&](size_t rounds) { return (unsigned)(((rounds + run_of(rounds) - 1) / run_of(rounds) + 7) / 8); };
  uint32_t* start = u32(o_start);
  const unsigned nf = (unsigned)((S + 127) / 128);
  block_kernel<<<nf + (nblocks + 127) / 128, 128>>>(
      t, BlockArgs{t.sec_N, t.sec_K, t.sec_off, u32(o_sblk), nsec, u32(o_bcnt), start, A + o_base, stride}, nf,
      reinterpret_cast<uint64_t*>(A + o_suf));
  ket_kernel<true><<<grid_of(nr), 256>>>(t, sx, t.total, nblocks, start, A + o_base, stride, run_of(nr), s.d_diag, occ, wi,
                                         wi + n, u32(o_fill), u32(o_rblk));
  QB_CUDA(cudaGetLastError());
  const int base_grid = sms * 8;
  base_kernel<<<base_grid, 256>>>(t, start, nblocks, u32(o_base), reinterpret_cast<int*>(s.d_scratch));
  QB_CUDA(cudaGetLastError());
  const unsigned fill_grid = (unsigned)((S + kBlock - 1) / kBlock);
  if (!t.fa_on) {
    t.bk_base = u32(o_base);
    t.bk_map = A + o_map;
    t.bk_map5 = reinterpret_cast<const uint16_t*>(A + o_map5);
    if (t.bk_nrec > 0) {
      const dim3 grid(fill_grid, (unsigned)std::min(t.bk_nrec, 8));
      block_map_kernel<<<grid, kBlock>>>(t, sx.word, reinterpret_cast<uint16_t*>(A + o_map),
                                         reinterpret_cast<uint16_t*>(A + o_map5));
      QB_CUDA(cudaGetLastError());
    }
  } else {
    auto at = [&](int k) { return A + o_fa + s.fa_off[k]; };
    t.fa_rec = reinterpret_cast<const uint2*>(at(0));
    t.fa_lam = reinterpret_cast<const float2*>(at(1));
    t.fa_ka = reinterpret_cast<const int32_t*>(at(2));
    t.fa_kc = reinterpret_cast<const int32_t*>(at(3));
    t.fa_psa = reinterpret_cast<const int32_t*>(at(4));
    t.fa_psc = reinterpret_cast<const int32_t*>(at(5));
    t.fa_info = reinterpret_cast<const uint4*>(at(6));
    t.fa_coef = reinterpret_cast<const float4*>(at(7));
    t.fa_lowof = reinterpret_cast<const int32_t*>(at(8));
    t.fa_lowoff = reinterpret_cast<const int64_t*>(at(9));
    t.fa_goff = reinterpret_cast<const uint32_t*>(at(10));
    t.fa_lam64 = reinterpret_cast<const double*>(at(15));
    t.fa_pqa = reinterpret_cast<const uint32_t*>(at(16));
    t.fa_mapa = reinterpret_cast<const uint2*>(A + o_mapa);
    t.fa_mapc = reinterpret_cast<const uint2*>(A + o_mapc);
    t.fa_basec = u32(o_base);
    t.fa_basea = u32(o_basea);
    t.fa_perm = u32(o_perm);
    const int32_t *lowN = reinterpret_cast<const int32_t*>(at(11)), *lowK = reinterpret_cast<const int32_t*>(at(12));
    uint32_t* lstart = start;
    if (s.low_held) {
      t.fa_occ = t.occ;
      t.fa_fill = t.fill;
      t.fa_wk = t.wk;
      t.fa_rblk = t.rblk;
    } else {
      lstart = u32(o_lstart);
      t.fa_occ = reinterpret_cast<const uint64_t*>(A + o_locc);
      t.fa_fill = u32(o_lfill);
      t.fa_wk = nullptr;
      t.fa_rblk = u32(o_lrblk);
      lower_block_kernel<<<(lblocks + 127) / 128, 128>>>(
          t, BlockArgs{lowN, lowK, t.fa_lowoff, u32(o_lblk), t.fa_nlow, u32(o_bcnt), lstart, A + o_basea, sizeof(BlockRec)});
      ket_kernel<false><<<grid_of(lnr), 256>>>(t, sx, t.fa_low, lblocks, lstart, A + o_basea, sizeof(BlockRec), run_of(lnr),
                                               nullptr, reinterpret_cast<uint64_t*>(A + o_locc), nullptr, nullptr,
                                               u32(o_lfill), u32(o_lrblk));
      QB_CUDA(cudaGetLastError());
    }
    round_order_kernel<<<base_grid, 256>>>(t.fa_lowoff, lowN, t.fa_nlow, (int64_t)lnr, u32(o_perm));
    lowered_base_kernel<<<base_grid, 256>>>(t, start, nblocks, u32(o_base));
    raised_base_kernel<<<base_grid, 256>>>(t, lstart, lblocks, u32(o_basea));
    const dim3 grid(fill_grid, (unsigned)std::min(fa_Ta(t) / 4 + t.fa_ng, 8));
    factor_map_kernel<<<grid, kBlock>>>(t, sx.word, reinterpret_cast<uint16_t*>(A + o_mapa),
                                        reinterpret_cast<uint16_t*>(A + o_mapc));
    QB_CUDA(cudaGetLastError());
  }
  if (t.mo_on) {
    t.mo_map = reinterpret_cast<const uint2*>(A + o_mmap);
    t.mo_base = u32(o_mbase);
    moment_map_kernel<<<dim3(fill_grid, 8), kBlock>>>(t, sx.word, reinterpret_cast<uint16_t*>(A + o_mmap));
    moment_base_kernel<<<base_grid, 256>>>(t, start, nblocks, u32(o_mbase));
    if (mnr > 0) {
      round_order_kernel<<<base_grid, 256>>>(t.sec_off, t.sec_N, t.n_sectors, mnr, u32(o_mperm));
      t.mo_perm = u32(o_mperm);
    }
    QB_CUDA(cudaGetLastError());
  }
  QB_CUDA(cudaDeviceSynchronize());
  return QB_OK;
}

// Members of a sweep whose vectors of B_k f lie side by side, so that each of the two passes is
// one launch for all of them: all, where that takes 256 MB at most.  A pass over so few kets is
// one or two waves of the SMs, and eight in turn pay for that and for the launch eight times (one
// stage of eight members, us: M = 16, 20,349 kets 312, side by side 86; M = 7, 50,388 104 / 36; M = 11,
// 167,960 361 / 186, M = 7, 245,157 202 / 175; M = 9, 817,190, beyond the line, 691 / 686).
constexpr int64_t kSideEntries = 16ll << 20;
int side_by_side(const Space& s, int batch) {
  return batch * s.t.fa_nG <= kSideEntries ? batch : 1;
}

// workspace: two double-float stage vectors and the double-float copy of psi,
// each [batch][total] x 16 bytes, and for factored couplings the vectors of B_k f
int64_t workspace_bytes(const Space& s, int batch) {
  return 16 * (3 * (int64_t)batch * s.secOff.back() + (s.t.fa_on ? side_by_side(s, batch) * s.t.fa_nG : 0));
}

template <int MODE, int B, bool CPLX>
static int launch_stage(const Space& s, const StageArgs& a, cudaStream_t st, int* grid_out = nullptr) {
  auto k = hpsi_kernel<MODE, B, CPLX>;
  const size_t smem = row_smem(s.t);
  int grid = 0;
  int rc = persistent_grid(k, smem, s.t.total, &grid);
  if (rc) return rc;
  if (grid_out) *grid_out = grid;
  k<<<grid, kBlock, smem, st>>>(s.t, a);
  QB_CUDA(cudaGetLastError());
  return QB_OK;
}

template <int MODE, int B>
static int launch_stage_c(const Space& s, const StageArgs& a, cudaStream_t st, int* grid_out = nullptr) {
  return s.t.is_complex ? launch_stage<MODE, B, true>(s, a, st, grid_out)
                        : launch_stage<MODE, B, false>(s, a, st, grid_out);
}

int launch_hpsi_rows(const Space& s, const void* d_v, void* d_out, cudaStream_t st) {
  StageArgs a{};
  a.vin = (const double2*)d_v;
  a.out = (double2*)d_out;
  a.scale[0] = 1.0;
  a.status = reinterpret_cast<int*>(s.d_scratch);
  return launch_stage_c<MODE_HPSI, 1>(s, a, st);
}

// plain = true: one launch per sector per stage (the comparison baseline of
// qb_evolve_plain); otherwise one launch per stage covers every sector.
// Steps are issued one launch per stage for every sector (plain = false) or one
// launch per sector per stage (plain = true, the comparison baseline of
// qb_evolve_plain).  The batched path captures chunks of kGraphSteps steps into
// a CUDA graph once the first step has run (and the launch geometry is cached),
// and replays the graph; a capture that the runtime refuses falls back to issuing
// the launches directly.
constexpr int64_t kGraphSteps = 32;

// lower kets whose entries a per-sector launch fills (factored couplings): the layer of two
// particles fewer, before the first sector of its particle number
static void lower_range(const Space& s, int sec, int64_t* low0, int64_t* low1) {
  *low0 = *low1 = 0;
  if (!s.t.fa_on || (sec > 0 && s.secN[sec] == s.secN[sec - 1])) return;
  const auto r = std::equal_range(s.lowN.begin(), s.lowN.end(), s.secN[sec] - 2);
  *low0 = s.lowOff[r.first - s.lowN.begin()];
  *low1 = s.lowOff[r.second - s.lowN.begin()];
}

template <int B>
static int rk4_issue(Space& s, DfArgs& a, double dt, int64_t steps, float4* w1, float4* w2, float4* psif,
                     cudaStream_t st, bool plain) {
  const bool cplx = s.t.is_complex != 0;
  const int K = s.order;
  for (int64_t it = 0; it < steps; ++it) {
    // Horner (order K = 4): v = psi + z/4 H psi; v = psi + z/3 H v; v = psi + z/2 H v;
    // psi = psi + z H v; stage j of K reads the previous output and writes w1 / w2
    // alternately, the last one the weighted copy of psi
    for (int d = K; d >= 1; --d) {
      const int j = K - d;
      a.vin = (j == 0) ? psif : ((j - 1) % 2 == 0 ? w1 : w2);
      a.out = (d == 1) ? psif : (j % 2 == 0 ? w1 : w2);
      a.zre = dt / d;
      const float zh = (float)a.zre;
      a.zf = make_float2(zh, (float)(a.zre - (double)zh));
      if (!plain) {
        a.low0 = 0;
        a.low1 = s.t.fa_on ? s.t.fa_low : 0;
        a.row0 = 0;
        a.row1 = s.t.total;
        int rc = stage_launch(s.t, a, d == 1 ? 1 : 0, B, cplx, st, nullptr, false, s.tile_shape);
        if (rc) return rc;
      } else {
        for (size_t sec = 0; sec + 1 < s.secOff.size(); ++sec) {
          a.row0 = s.secOff[sec];
          a.row1 = s.secOff[sec + 1];
          lower_range(s, (int)sec, &a.low0, &a.low1);
          int rc = stage_launch(s.t, a, d == 1 ? 1 : 0, B, cplx, st, nullptr, false, s.tile_shape);
          if (rc) return rc;
        }
      }
    }
  }
  return QB_OK;
}

// Cooperative launches take turns: one call at a time on a device holds the turn, from before it
// clears its barrier's counter until its stream is drained.  (Two at once could each hold the
// SMs that the other's last CTAs need, and calls on one space share its counter.)  The turn is
// a host lock and leaves nothing on the streams: a wait for another stream's event can close a
// circle of waits with the caller's own, and an event that a caller's stream capture has taken
// up refuses every later wait.  A call waits for it about as long as its own launch would run
// (5 us a stage), between a millisecond and a second, and then goes stage by stage.
static std::unique_lock<std::timed_mutex> coop_turn(const Space& s, int64_t steps) {
  constexpr int kDevices = 64;
  static std::timed_mutex turn[kDevices];
  if (s.device < 0 || s.device >= kDevices) return {};
  const int64_t us = std::min<int64_t>(std::max<int64_t>(5 * s.order * std::min<int64_t>(steps, 1000000), 1000), 1000000);
  return std::unique_lock<std::timed_mutex>(turn[s.device], std::chrono::microseconds(us));
}

template <int B>
static int rk4_loop(Space& s, double2* psi, const double* scale, double dt, int64_t steps, float4* w1, float4* w2,
                    float4* psif, cudaStream_t st, bool plain, std::unique_lock<std::timed_mutex>& turn) {
  {
    // the stages run in the weighted basis f = psi / w
    int rc = launch_to_dfw(s, psi, psif, B, st);
    if (rc) return rc;
  }
  DfArgs a{};
  for (int b = 0; b < B; ++b) {
    const float h = (float)scale[b];
    a.scale[b] = make_float2(h, (float)(scale[b] - (double)h));
  }
  a.diag = s.d_diag;
  a.psi = psi;
  a.psif = psif;
  a.g = psif + (size_t)B * s.t.total;
  a.g_members = side_by_side(s, B);
  a.status = reinterpret_cast<int*>(s.d_scratch);
  a.nbasef = 0;
  if (plain) return rk4_issue<B>(s, a, dt, steps, w1, w2, psif, st, true);
  // A space of small sectors runs resident, all steps in one launch.
  if (B == 1 && !s.t.fa_on) {
    int optin = 0, sms = 0;
    QB_CUDA(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, s.device));
    QB_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, s.device));
    const int cap = (int)std::min<int64_t>((s.maxDim + 3) & ~int64_t(3), 65536);
    ResArgs r{};
    r.psi = psi;
    r.psif = psif;
    r.diag = s.d_diag;
    r.scale = a.scale[0];
    r.dt = dt;
    r.steps = steps;
    r.order = s.order;
    r.cap = cap;
    r.w1 = w1;
    r.w2 = w2;
    r.status = a.status;
    if (s.maxDim <= std::min(s.resident_max_kets, resident_most(s.t)) && s.t.total <= 64LL * sms && resident_smem(s.t, cap) + 1024 <= (size_t)optin)
      return resident_launch(s.t, r, (int)std::min<int64_t>(1024, (s.maxDim + 31) & ~int64_t(31)), st);
    // One cooperative launch where the kets find a thread each.
    if (s.resident_max_kets > 0 && grid_reg_fits(s.t, sms)) {
      turn = coop_turn(s, steps);
      r.barrier = reinterpret_cast<uint32_t*>(s.d_scratch + 1);
      r.status = reinterpret_cast<int*>(r.barrier) + 1;
      r.polls = s.wait_polls;
      if (turn.owns_lock()) return s.M == 5 ? grid_launch_m5(s.t, r, st) : grid_launch_m7(s.t, r, st);
    }
  }
  if (steps < 2 * kGraphSteps) return rk4_issue<B>(s, a, dt, steps, w1, w2, psif, st, false);
  // first step directly: fills the launch-geometry cache outside any capture
  int rc = rk4_issue<B>(s, a, dt, 1, w1, w2, psif, st, false);
  if (rc) return rc;
  int64_t left = steps - 1;
  cudaGraph_t graph = nullptr;
  cudaGraphExec_t exec = nullptr;
  bool captured = false;
  // capture on the space's private stream (the caller's may be the legacy default
  // stream, which cannot capture); the graph is launched on the caller's stream
  if (!s.capture_stream) QB_CUDA(cudaStreamCreateWithFlags(&s.capture_stream, cudaStreamNonBlocking));
  if (cudaStreamBeginCapture(s.capture_stream, cudaStreamCaptureModeThreadLocal) == cudaSuccess) {
    rc = rk4_issue<B>(s, a, dt, kGraphSteps, w1, w2, psif, s.capture_stream, false);
    const cudaError_t ec = cudaStreamEndCapture(s.capture_stream, &graph);
    if (rc) {
      if (graph) cudaGraphDestroy(graph);
      return rc;
    }
    if (ec == cudaSuccess && graph && cudaGraphInstantiate(&exec, graph, 0) == cudaSuccess) captured = true;
  }
  cudaGetLastError();  // a refused capture leaves a sticky-free error; clear it
  if (captured) {
    for (; left >= kGraphSteps; left -= kGraphSteps) {
      const cudaError_t e = cudaGraphLaunch(exec, st);
      if (e != cudaSuccess) {
        cudaGraphExecDestroy(exec);
        cudaGraphDestroy(graph);
        return fail(QB_ECUDA, std::string("cudaGraphLaunch: ") + cudaGetErrorString(e));
      }
    }
    cudaGraphExecDestroy(exec);
    cudaGraphDestroy(graph);
  } else if (graph) {
    cudaGraphDestroy(graph);
  }
  return rk4_issue<B>(s, a, dt, left, w1, w2, psif, st, false);
}

int launch_rk4(Space& s, void* d_psi, int batch, const double* scale, double dt, int64_t steps, void* d_work,
               void* stream, bool plain) {
  cudaStream_t st = (cudaStream_t)stream;
  const int64_t n = (int64_t)batch * s.secOff.back();
  double2* psi = (double2*)d_psi;
  float4* w1 = (float4*)d_work;
  float4* w2 = w1 + n;
  float4* psif = w2 + n;
  std::unique_lock<std::timed_mutex> turn;  // of a cooperative launch, held until the stream is drained
  int rc;
  switch (batch) {
    case 1: rc = rk4_loop<1>(s, psi, scale, dt, steps, w1, w2, psif, st, plain, turn); break;
    case 2: rc = rk4_loop<2>(s, psi, scale, dt, steps, w1, w2, psif, st, plain, turn); break;
    case 4: rc = rk4_loop<4>(s, psi, scale, dt, steps, w1, w2, psif, st, plain, turn); break;
    case 8: rc = rk4_loop<8>(s, psi, scale, dt, steps, w1, w2, psif, st, plain, turn); break;
    default: return fail(QB_EINVAL, "batch must be 1, 2, 4 or 8");
  }
  if (rc) {
    if (turn.owns_lock()) cudaStreamSynchronize(st);
    return rc;
  }
  if (turn.owns_lock()) {  // with the launch's own status, which no other call on the space reads or clears
    int h[4];
    QB_CUDA(cudaMemcpyAsync(h, s.d_scratch, sizeof(h), cudaMemcpyDeviceToHost, st));
    QB_CUDA(cudaStreamSynchronize(st));
    rc = h[0] ? check_status(s, st) : QB_OK;
    if (h[3] & kLate) return fail(QB_ETIMEOUT, "a wait between the stages of a cooperative launch ran out");
    if (h[3]) return fail(QB_EINTERNAL, "device-side consistency check failed (status " + std::to_string(h[3]) + ")");
    return rc;
  }
  return check_status(s, st);
}

int launch_to_dfw(const Space& s, const void* psi, void* psif, int B, void* stream) {
  int dev = 0, sms = 0;
  QB_CUDA(cudaGetDevice(&dev));
  QB_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  const int64_t want = (s.t.total + 255) / 256;
  const int grid = (int)std::max<int64_t>(1, std::min<int64_t>(want, (int64_t)sms * 8));
  auto k = to_dfw_kernel<0>;
  switch (s.M) {
    case 5: k = to_dfw_kernel<5>; break;
    case 7: k = to_dfw_kernel<7>; break;
    case 9: k = to_dfw_kernel<9>; break;
    case 11: k = to_dfw_kernel<11>; break;
    default: break;
  }
  k<<<grid, 256, 0, (cudaStream_t)stream>>>(s.t, (const double2*)psi, (float4*)psif, B);
  QB_CUDA(cudaGetLastError());
  return QB_OK;
}

int launch_unrank(const Space& s, int64_t first, int64_t count, int* d_occ, void* stream) {
  cudaStream_t st = (cudaStream_t)stream;
  int grid = 0;
  int rc = persistent_grid(unrank_kernel, 0, count * s.M, &grid);
  if (rc) return rc;
  unrank_kernel<<<grid, kBlock, 0, st>>>(s.t, first, count, d_occ);
  QB_CUDA(cudaGetLastError());
  return check_status(s, st);
}

int launch_rank(const Space& s, const int* d_occ, int64_t count, int64_t* d_index, void* stream) {
  cudaStream_t st = (cudaStream_t)stream;
  const size_t smem = blob_smem(s.t);
  int grid = 0;
  int rc = persistent_grid(rank_kernel, smem, count, &grid);
  if (rc) return rc;
  rank_kernel<<<grid, kBlock, smem, st>>>(s.t, d_occ, count, d_index);
  QB_CUDA(cudaGetLastError());
  QB_CUDA(cudaStreamSynchronize(st));
  return QB_OK;
}

int launch_terms(const Space& s, int64_t* terms, int64_t* tuples, void* stream) {
  cudaStream_t st = (cudaStream_t)stream;
  const size_t smem = row_smem(s.t);
  int grid = 0;
  int rc = persistent_grid(terms_kernel, smem, s.t.total, &grid);
  if (rc) return rc;
  unsigned long long* d = reinterpret_cast<unsigned long long*>(partial_area(s));
  QB_CUDA(cudaMemsetAsync(d, 0, 16, st));
  terms_kernel<<<grid, kBlock, smem, st>>>(s.t, d);
  QB_CUDA(cudaGetLastError());
  unsigned long long h[2];
  QB_CUDA(cudaMemcpyAsync(h, d, 16, cudaMemcpyDeviceToHost, st));
  QB_CUDA(cudaStreamSynchronize(st));
  *terms = (int64_t)h[0];
  if (tuples) *tuples = (int64_t)h[1];
  return QB_OK;
}

int launch_init_table(const Space& s, const double* table_host, int only_N, void* d_psi, double* norm2,
                      void* stream) {
  cudaStream_t st = (cudaStream_t)stream;
  int grid = 0;
  int rc = persistent_grid(init_table_kernel, 0, s.t.total, &grid);
  if (rc) return rc;
  double* part = partial_area(s);
  double* tab = table_area(s);
  const size_t tab_bytes = sizeof(double) * 2 * (size_t)s.M * (s.nmax + 1);
  QB_CUDA(cudaMemcpyAsync(tab, table_host, tab_bytes, cudaMemcpyHostToDevice, st));
  init_table_kernel<<<grid, kBlock, 0, st>>>(s.t, (const double2*)tab, only_N, (double2*)d_psi, part);
  QB_CUDA(cudaGetLastError());
  double* fin = init_final(s);
  sum_rows_kernel<<<1, kSumThreads, 0, st>>>(part, grid, 1, 1.0, false, fin);
  QB_CUDA(cudaGetLastError());
  QB_CUDA(cudaMemcpyAsync(norm2, fin, sizeof(double), cudaMemcpyDeviceToHost, st));
  QB_CUDA(cudaStreamSynchronize(st));
  return QB_OK;
}

int launch_scale(const Space& s, void* d_psi, double factor, void* stream) {
  cudaStream_t st = (cudaStream_t)stream;
  scale_kernel<<<1216, 256, 0, st>>>((double2*)d_psi, s.t.total, factor);
  QB_CUDA(cudaGetLastError());
  return QB_OK;
}

int launch_number(const Space& s, int64_t index, void* d_psi, void* stream) {
  cudaStream_t st = (cudaStream_t)stream;
  number_kernel<<<1216, 256, 0, st>>>((double2*)d_psi, s.t.total, index);
  QB_CUDA(cudaGetLastError());
  return QB_OK;
}

// ----------------------------------------------- allocation-free observables
//
// qb_observables_noalloc serves callers that must not allocate device memory
// while they run: code inside a memory-budgeted service or a custom allocator
// that forbids cudaMalloc / cudaFree after start-up, or a host thread that must
// not touch the allocator (which may synchronise the device).  It computes the
// same observables as qb_observables, but its reduction partials live in one
// fixed, file-scope device array instead of the space's scratch buffer.
//
// The array holds kNoAllocDoubles doubles (1 MiB) on every GPU that loads the
// library, for the life of the process.  Every call shares it and it keeps the
// last call's contents; the status word is cleared at the start of each call.
// Calls that overlap on the GPU (several streams or threads at once) race on it.
// The first call on each device looks up the array's device address
// (cudaGetSymbolAddress) with that device current; make that first call before
// any stream capture.  The address is cached per device for the process: one CUDA
// context per device for the life of the process is assumed (a cudaDeviceReset
// would reload the module and leave the cached address stale).

constexpr int64_t kNoAllocDoubles = 131072;  // 1 MiB
static __device__ __align__(256) double g_noalloc_scratch[kNoAllocDoubles];
static double* g_noalloc_ptr[256];  // device address of the array, per device
static std::mutex g_noalloc_mu;

static int noalloc_scratch(double** out) {
  int dev = 0;
  QB_CUDA(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 256) return fail(QB_EUNSUPPORTED, "device ordinal beyond 255");
  std::lock_guard<std::mutex> lock(g_noalloc_mu);
  if (!g_noalloc_ptr[dev]) {
    void* p = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
    if (e != cudaSuccess || !p)
      return fail(QB_ECUDA, std::string("cudaGetSymbolAddress(g_noalloc_scratch): ") + cudaGetErrorString(e));
    g_noalloc_ptr[dev] = static_cast<double*>(p);
  }
  *out = g_noalloc_ptr[dev];
  return QB_OK;
}

// <psi|H psi> partials of at most `grid` CTAs (the size the fixed array was carved
// for); *launched receives the CTA count, the number of partials to reduce
template <bool CPLX>
static int noalloc_dot(const Space& s, const StageArgs& a, int grid, cudaStream_t st, int* launched) {
  const size_t smem = row_smem(s.t);
  auto k = hpsi_kernel<MODE_DOT, 1, CPLX>;
  int g0 = 0;
  int rc = persistent_grid(k, smem, s.t.total, &g0);
  if (rc) return rc;
  *launched = std::min(grid, g0);
  k<<<*launched, kBlock, smem, st>>>(s.t, a);
  QB_CUDA(cudaGetLastError());
  return QB_OK;
}

}  // namespace qb

using namespace qb;

extern "C" int qb_observables_noalloc(qb_space* space, const void* d_psi, qb_obs* out, void* stream) {
  Space* sp = reinterpret_cast<Space*>(space);
  if (!sp || !out) return fail(QB_EINVAL, "space and out must be non-NULL");
  if (!d_psi || (reinterpret_cast<uintptr_t>(d_psi) & 15)) return fail(QB_EINVAL, "d_psi must be 16-byte aligned");
  int dev = 0;
  QB_CUDA(cudaGetDevice(&dev));
  if (dev != sp->device) return fail(QB_EINVAL, "the space was built on another device");
  double* scr = nullptr;
  int rc = noalloc_scratch(&scr);
  if (rc) return rc;
  cudaStream_t st = (cudaStream_t)stream;
  const int M = sp->M;
  const int nmom = nmoments(M);
  // layout (doubles): [0, 2) status word | partials [G nmom] | final [nmom] |
  // dot partials [2 G] | dot final [2]; G CTAs, capped so that it fits
  const int64_t fixed = 2 + nmom + 2 + 8;
  const int64_t gcap = (kNoAllocDoubles - fixed) / (nmom + 2);
  if (gcap < 32)
    return fail(QB_EUNSUPPORTED, "the moments of this space need more than the fixed 1 MiB scratch of "
                                 "qb_observables_noalloc (M too large)");
  const size_t smem = row_smem(sp->t) + ((kRowScratchBytes + 15) & ~15) - kRowScratchBytes +
                      (size_t)(kBlock / 32) * nmom * sizeof(double) + 16;
  int grid = 0;
  rc = persistent_grid(moments_kernel, smem, sp->t.total, &grid);
  if (rc) return rc;
  grid = (int)std::min<int64_t>(grid, gcap);
  int* status = reinterpret_cast<int*>(scr);
  double* part = scr + 2;
  double* fin = part + (int64_t)grid * nmom;
  double* dpart = fin + nmom;
  double* dfin = dpart + 2 * (int64_t)grid;
  QB_CUDA(cudaMemsetAsync(status, 0, sizeof(int), st));
  moments_kernel<<<grid, kBlock, smem, st>>>(sp->t, (const double2*)d_psi, part, nmom, status);
  QB_CUDA(cudaGetLastError());
  sum_rows_kernel<<<nmom, kSumThreads, 0, st>>>(part, grid, nmom, 1.0, false, fin);
  QB_CUDA(cudaGetLastError());
  StageArgs a{};
  a.vin = (const double2*)d_psi;
  a.scale[0] = 1.0;
  a.status = status;
  a.partial = dpart;
  int gdot = 0;
  rc = sp->t.is_complex ? noalloc_dot<true>(*sp, a, grid, st, &gdot) : noalloc_dot<false>(*sp, a, grid, st, &gdot);
  if (rc) return rc;
  sum_rows_kernel<<<2, kSumThreads, 0, st>>>(dpart, gdot, 2, 1.0, false, dfin);
  QB_CUDA(cudaGetLastError());
  std::vector<double> raw(nmom, 0.0);
  double h2[2];
  int hs = 0;
  QB_CUDA(cudaMemcpyAsync(raw.data(), fin, sizeof(double) * nmom, cudaMemcpyDeviceToHost, st));
  QB_CUDA(cudaMemcpyAsync(h2, dfin, sizeof(h2), cudaMemcpyDeviceToHost, st));
  QB_CUDA(cudaMemcpyAsync(&hs, status, sizeof(int), cudaMemcpyDeviceToHost, st));
  QB_CUDA(cudaStreamSynchronize(st));
  if (hs) return fail(QB_EINTERNAL, "device-side consistency check failed (status " + std::to_string(hs) + ")");
  raw[2] = h2[0];
  if (!(raw[0] > 0.0)) return fail(QB_EINVAL, "the state has zero norm");
  derive(M, raw.data(), out);
  return QB_OK;
}

namespace qb {

}  // namespace qb
