// Two-body bilinears <bra, a_p^dag a_q^dag a_r a_s ket> of weighted double-float vectors, the
// coupling gradient's inner products, by blocks of kets (qb_block.cuh).
//
// In the weighted basis b = bra / w, f = ket / w
//   <bra, a_p^dag a_q^dag a_r a_s ket> = sum_n conj(b_t) k f_n w_n^2,  k = n_r (n_s - [r = s]),
// t the ket n with r, s taken away and p, q added: the target that the direct stage kernel
// ranks for the same term.  f_n w_n^2 is formed by two products (w_n^2 alone may leave the fp32
// range), the weight with a third part (dft_mul).  A task is one to four records (pairs (r, s)
// with their partners), up to eight sums, over a share of the kets; the sums of a lane over up to
// 32 kets are double-float, those of the lanes of three floats (tfc_add, more bits than FP64), those
// of the warps' flushes, the warps and the CTAs FP64, in a fixed order.
//
// Bound by the issue of the 24 packed operations of a complex product and of what they take
// (58% of the issue slots, 16 warps an SM).  The 45 operators of 435,897 kets at M = 5: 77 us
// (lanes added in double-float and weights of 48 bits: 74); the moments kernel, one entry a lane and
// every target ranked anew from the ranking table, took 145 us, a form that gathered record by
// record 94.
#include <cuda_runtime.h>

#include <algorithm>
#include <string>
#include <vector>

#include "qb_device.cuh"
#include "qb_internal.h"
#include "qb_block.cuh"

namespace qb {

constexpr int kTbCols = 8;     // complex sums of a task
constexpr int kTbWarps = 8;    // warps per CTA
constexpr int kTbRounds = 32;  // rounds of a warp between flushes to FP64
template <int KC>
__host__ __device__ constexpr int tb_records() { return kTbCols / Rec<KC>::n; }

// acc += conj(x) v
__device__ __forceinline__ void conj_fma(dfc& acc, float4 x, dfc v) {
  dfc_fma(acc, f2_pack(x.x, x.x), f2_pack(-x.x, -x.x), f2_pack(x.z, x.z), v.h, v.l);
  float rh, ih, rl, il;
  f2_unpack(v.h, rh, ih);
  f2_unpack(v.l, rl, il);
  dfc_fma(acc, f2_pack(x.y, x.y), f2_pack(-x.y, -x.y), f2_pack(x.w, x.w), f2_pack(ih, -rh), f2_pack(il, -rl));
}

// Tasks blockIdx.y < ngr: records; the others: eight pairs' diagonal operators each.
// partial[task][gridDim.x][2 kTbCols].
template <int MT, bool FIX>
__global__ void __launch_bounds__(32 * kTbWarps, 2) tb_kernel(const Tables t, const float4* bra, const float4* ket,
                                                              int ngr, double* partial, int* status) {
  constexpr int KC = FIX ? (MT - 1) / 2 : 0;
  constexpr int NT = Rec<KC>::n, RW = Rec<KC>::w, NW = occ_words<MT>(), R = tb_records<KC>();
  __shared__ double sum[kTbWarps][2 * kTbCols];
  __shared__ int pairs[kTbCols];
  __shared__ uint2 sinfo[R];
  const int M = (MT > 0) ? MT : t.M;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, task = blockIdx.y;
  const bool diag = task >= ngr;
  if (lane < 2 * kTbCols) sum[warp][lane] = 0.0;
  if (threadIdx.x < kTbCols) {  // pair number -> r | s << 8
    int a = (task - ngr) * kTbCols + (int)threadIdx.x, r = 0;
    while (diag && r < M && a >= M - r) a -= M - r++;
    pairs[threadIdx.x] = diag && r < M ? r | ((r + a) << 8) : -1;
  }
  if (threadIdx.x < R && !diag) sinfo[threadIdx.x] = __ldg(t.bk_info + min(task * R + (int)threadIdx.x, t.bk_nrec - 1));
  __syncthreads();
  const int64_t total = t.total, nr = (total + 31) / 32;
  dfc acc[kTbCols];
#pragma unroll
  for (int j = 0; j < kTbCols; ++j) acc[j] = dfc{0ull, 0ull};
  bool bad = false;
  // the lanes' sums: in three exchanges each half of the lanes takes half of the columns, two
  // more add the four lanes of a column (all eight columns by FP64 shuffles took longer than
  // the products where a warp has few rounds)
  auto flush = [&]() {
    f2 rest[kTbCols];  // third parts (tfc_add)
#pragma unroll
    for (int j = 0; j < kTbCols; ++j) rest[j] = 0ull;
#pragma unroll
    for (int w = kTbCols / 2; w >= 1; w >>= 1) {
      const bool up = (lane & (4 * w)) != 0;
#pragma unroll
      for (int j = 0; j < kTbCols / 2; ++j) {
        if (j >= w) break;
        const dfc mine = up ? acc[j + w] : acc[j], other = up ? acc[j] : acc[j + w];
        const f2 rmine = up ? rest[j + w] : rest[j], rother = up ? rest[j] : rest[j + w];
        acc[j] = mine;
        rest[j] = rmine;
        tfc_add(acc[j], rest[j], __shfl_xor_sync(0xffffffffu, other.h, 4 * w), __shfl_xor_sync(0xffffffffu, other.l, 4 * w),
                w < kTbCols / 2 ? __shfl_xor_sync(0xffffffffu, rother, 4 * w) : 0ull);
      }
    }
#pragma unroll
    for (int o = 2; o >= 1; o >>= 1)
      tfc_add(acc[0], rest[0], __shfl_xor_sync(0xffffffffu, acc[0].h, o), __shfl_xor_sync(0xffffffffu, acc[0].l, o),
              __shfl_xor_sync(0xffffffffu, rest[0], o));
    if ((lane & 3) == 0) {  // column lane / 4
      const double2 v = tfc_to(acc[0], rest[0]);
      sum[warp][lane / 2] += v.x;
      sum[warp][lane / 2 + 1] += v.y;
    }
#pragma unroll
    for (int j = 0; j < kTbCols; ++j) acc[j] = dfc{0ull, 0ull};
  };
  int held = 0;
  const int64_t step = (int64_t)gridDim.x * kTbWarps;
  int64_t rd = (int64_t)blockIdx.x * kTbWarps + warp;
  // the next round's ket is read ahead
  RoundIn next = load_round(t.occ, t.fill, t.rblk, min(rd, nr - 1), total, lane);
  float4 knext = __ldg(ket + min(rd * 32 + lane, total - 1));
  double wnext = __ldg(t.wk + min(rd * 32 + lane, total - 1));
  for (; rd < nr; rd += step) {
    const RoundIn in = next;
    const float4 kv = knext;
    const dft wd = dft_of(wnext);
    const int64_t g = rd * 32 + lane;
    const bool valid = g < total;
    {
      const int64_t gn = min(g + 32 * step, total - 1);
      next = load_round(t.occ, t.fill, t.rblk, min(rd + step, nr - 1), total, lane);
      knext = __ldg(ket + gn);
      wnext = __ldg(t.wk + gn);
    }
    const dfl yr = dft_mul(wd, dft_mul(wd, df_re(kv))), yi = dft_mul(wd, dft_mul(wd, df_im(kv)));
    const f2 yh = f2_pack(yr.h, yi.h), yl = f2_pack(yr.l, yi.l);
    uint32_t ob[NW];
    unpack_occ<MT, NW>(t, valid ? in.word : 0ull, ob);  // an invalid lane: no pair acts
    if (!diag) {
      const uint32_t* base = t.bk_base + (size_t)block_of_lane(in, lane, valid) * t.bk_T;
      const unsigned char* mp = t.bk_map + (size_t)in.fill * (2 * RW);
      const uint16_t* mp5 = t.bk_map5 + in.fill;
      // every record's maps and bases, then every gather, then the products
      MapRec<KC> m[R];
      BaseRec<KC> b[R];
#pragma unroll
      for (int u = 0; u < R; ++u) {
        const int rec = min(task * R + u, t.bk_nrec - 1);
        m[u] = load_map<KC>(mp + (size_t)rec * t.bk_S * (2 * RW), mp5 + (size_t)rec * t.bk_S);
        b[u] = load_base<KC>(base, rec, t.bk_nrec);
      }
      float4 x[R][NT];
      float Af[R];
#pragma unroll
      for (int u = 0; u < R; ++u) {
        const uint2 info = sinfo[u];
        Af[u] = (occ_float23<NW>(ob, info.x, (info.x & 0x8000u) != 0u) - 8388608.0f) *
                (occ_float23<NW>(ob, info.x >> 16, (info.x & 0x80000000u) != 0u) - __uint_as_float(info.y));
        if (task * R + u >= t.bk_nrec) Af[u] = 0.f;
        const int n = KC == 0 ? (int)((info.x >> 4) & 7) : NT;
        const uint32_t rk[5] = {b[u].a.x + (m[u].a.x & 0xffffu), b[u].a.y + (m[u].a.x >> 16),
                                b[u].a.z + (m[u].a.y & 0xffffu), b[u].a.w + (m[u].a.y >> 16), b[u].b + m[u].b};
#pragma unroll
        for (int c = 0; c < NT; ++c) {
          const bool act = Af[u] != 0.f && (KC > 0 || c < n), ok = act && rk[c] < (uint32_t)total;
          bad |= act && !ok;
          x[u][c] = make_float4(0.f, 0.f, 0.f, 0.f);
          if (ok) x[u][c] = __ldg(bra + rk[c]);
        }
      }
#pragma unroll
      for (int u = 0; u < R; ++u) {
        if (!__any_sync(0xffffffffu, Af[u] != 0.f)) continue;
        dfc v{0ull, 0ull};
        dfc_fma_int(v, f2_pack(Af[u], Af[u]), f2_pack(-Af[u], -Af[u]), yh, yl);
        v = dfc_renorm(v);
#pragma unroll
        for (int c = 0; c < NT; ++c) conj_fma(acc[u * NT + c], x[u][c], v);
      }
    } else if (valid) {
      dfc z{0ull, 0ull};
      conj_fma(z, __ldg(bra + g), dfc{yh, yl});
      z = dfc_renorm(z);
#pragma unroll
      for (int j = 0; j < kTbCols; ++j) {
        const int rs = pairs[j];
        if (rs < 0) break;
        const int r = rs & 0xff, s = rs >> 8;
        const float k = occ_float<NW>(ob, r) * (occ_float<NW>(ob, s) - (r == s ? 1.f : 0.f));
        dfc_fma_int(acc[j], f2_pack(k, k), f2_pack(-k, -k), z.h, z.l);
      }
    }
#pragma unroll
    for (int j = 0; j < kTbCols; ++j) acc[j] = dfc_renorm(acc[j]);
    if (++held == kTbRounds) {
      flush();
      held = 0;
    }
  }
  __syncwarp();
  flush();
  if (bad) atomicOr(status, 1);
  __syncthreads();
  if (threadIdx.x < 2 * kTbCols) {
    double s = 0.0;
    for (int w = 0; w < kTbWarps; ++w) s += sum[w][threadIdx.x];
    partial[((size_t)task * gridDim.x + blockIdx.x) * (2 * kTbCols) + threadIdx.x] = s;
  }
}

// d_acc[2e, 2e + 1] += weight * the sum over the shares of operator e's column, one CTA each
__global__ void __launch_bounds__(kSumThreads) tb_sum_kernel(const double* partial, const int* cols, int shares,
                                                              double weight, double* acc) {
  __shared__ double red[kSumThreads / 32][2];
  const int e = blockIdx.x, c = cols[e];
  const double* p = partial + (size_t)(c / kTbCols) * shares * (2 * kTbCols) + 2 * (c % kTbCols);
  double re = 0.0, im = 0.0;
  for (int k = threadIdx.x; k < shares; k += kSumThreads) {
    re += p[(size_t)k * (2 * kTbCols)];
    im += p[(size_t)k * (2 * kTbCols) + 1];
  }
  for (int o = 16; o > 0; o >>= 1) {
    re += __shfl_down_sync(0xffffffffu, re, o);
    im += __shfl_down_sync(0xffffffffu, im, o);
  }
  if ((threadIdx.x & 31) == 0) {
    red[threadIdx.x >> 5][0] = re;
    red[threadIdx.x >> 5][1] = im;
  }
  __syncthreads();
  if (threadIdx.x < 2) {
    double s = 0.0;
    for (int w = 0; w < kSumThreads / 32; ++w) s += red[w][threadIdx.x];
    acc[2 * e + threadIdx.x] += weight * s;
  }
}

static int tb_per(const Tables& t) {
  switch (t.bk_kc) {
    case 2: return tb_records<2>();
    case 3: return tb_records<3>();
    case 4: return tb_records<4>();
    case 5: return tb_records<5>();
    default: return tb_records<0>();
  }
}

std::vector<int> tb_columns(const Space& s, const std::vector<int>& ops) {
  const Tables& t = s.t;
  const Combos& c = s.combos;
  const int per = t.bk_kc > 0 ? t.bk_kc : 4, R = tb_per(t), ngr = (t.bk_nrec + R - 1) / R;
  std::vector<int> first(c.annR.size());  // first record of each pair
  for (size_t a = 0, rec = 0; a < first.size(); ++a) {
    first[a] = (int)rec;
    rec += (size_t)((c.annStart[a + 1] - c.annStart[a] + per - 1) / per);
  }
  std::vector<int> cols;
  for (int w : ops) {
    const int a1 = w & 0xff, a2 = (w >> 8) & 0xff, a = c.pairidx[(w >> 16) & 0xff][(w >> 24) & 0xff];
    if (c.pairidx[a1][a2] == a) {
      cols.push_back(ngr * kTbCols + a);
      continue;
    }
    int j = c.annStart[a];
    while (j < c.annStart[a + 1] && (int)(c.pq[j] & 0xffff) != (a1 | (a2 << 8))) ++j;
    const int k = j - c.annStart[a], rec = first[a] + k / per;
    cols.push_back(rec / R * kTbCols + rec % R * per + k % per);
  }
  return cols;
}

template <int MT, bool FIX>
static int tb_launch(const Space& s, const float4* bra, const float4* ket, const int* cols, int n_ops, double weight,
                     double* acc, cudaStream_t st) {
  const Tables& t = s.t;
  const int R = tb_per(t), ngr = (t.bk_nrec + R - 1) / R, tasks = ngr + (t.n_ann + kTbCols - 1) / kTbCols;
  // shares: a round a warp, at most about four waves of the SMs' 16 warps, and what the
  // partial sums' area holds
  const int64_t G = max_grid_of(s), rounds = (t.total + 31) / 32;
  const int64_t most = std::min<int64_t>(G * nmoments(s.M) / (2 * kTbCols * tasks), std::max<int64_t>(1, G / 2 / tasks));
  const int shares = (int)std::max<int64_t>(1, std::min((rounds + kTbWarps - 1) / kTbWarps, most));
  tb_kernel<MT, FIX><<<dim3((unsigned)shares, (unsigned)tasks), 32 * kTbWarps, 0, st>>>(
      t, bra, ket, ngr, partial_area(s), reinterpret_cast<int*>(s.d_scratch));
  QB_CUDA(cudaGetLastError());
  tb_sum_kernel<<<n_ops, kSumThreads, 0, st>>>(partial_area(s), cols, shares, weight, acc);
  QB_CUDA(cudaGetLastError());
  return QB_OK;
}

int launch_tb_blocks(const Space& s, const float4* bra, const float4* ket, const int* cols, int n_ops, double weight,
                     double* acc, cudaStream_t st) {
  if (s.t.bk_kc > 0) {
    switch (s.M) {
      case 5: return tb_launch<5, true>(s, bra, ket, cols, n_ops, weight, acc, st);
      case 7: return tb_launch<7, true>(s, bra, ket, cols, n_ops, weight, acc, st);
      case 9: return tb_launch<9, true>(s, bra, ket, cols, n_ops, weight, acc, st);
      case 11: return tb_launch<11, true>(s, bra, ket, cols, n_ops, weight, acc, st);
      default: break;
    }
  }
  return tb_launch<0, false>(s, bra, ket, cols, n_ops, weight, acc, st);
}

}  // namespace qb
