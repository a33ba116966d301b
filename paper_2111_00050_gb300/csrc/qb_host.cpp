// Host side of the qb library: model validation, sector tables, the C ABI
// entry points, the small Hermitian eigensolve behind the Penrose-Onsager
// test, breaktime detection and the mean-field integrator.
//
// Paper: Eberhardt, Zamora, Kopp & Abel, arXiv:2111.00050.
#include <cuda_runtime.h>

#include <algorithm>
#include <array>
#include <cmath>
#include <complex>
#include <cstring>
#include <string>
#include <vector>

#include "qb_internal.h"

namespace qb {

static thread_local std::string g_err;

void set_error(const std::string& msg) { g_err = msg; }

int fail(int code, const std::string& msg) {
  g_err = msg;
  return code;
}

typedef std::complex<double> cd;

static int label_shift(int M) { return (M % 2) ? (M - 1) / 2 : 0; }
static int modp(long long a, int M) {
  long long r = a % M;
  return (int)(r < 0 ? r + M : r);
}
static size_t align16(size_t x) { return (x + 15) & ~(size_t)15; }

// Validates and symmetrises the coupling tensor (see qb_model in qb.h).
static int prepare_model(const qb_model* model, std::vector<double>& w, std::vector<double>& Lsym) {
  if (!model || !model->w || !model->L) return fail(QB_EINVAL, "model, model->w and model->L must be non-NULL");
  const int M = model->M;
  if (M < 1 || M > QB_MAX_MODES) return fail(QB_EUNSUPPORTED, "M must be in [1, QB_MAX_MODES]");
  const int c = label_shift(M);
  w.assign(model->w, model->w + M);
  for (int p = 0; p < M; ++p)
    if (!std::isfinite(w[p])) return fail(QB_EINVAL, "w has a non-finite entry");
  const size_t M4 = (size_t)M * M * M * M;
  auto Lat = [&](int p, int q, int r, int s) {
    size_t t = (((size_t)p * M + q) * M + r) * M + s;
    return cd(model->L[2 * t], model->L[2 * t + 1]);
  };
  double lmax = 0.0;
  for (int p = 0; p < M; ++p)
    for (int q = 0; q < M; ++q)
      for (int r = 0; r < M; ++r)
        for (int s = 0; s < M; ++s) {
          cd v = Lat(p, q, r, s);
          if (!std::isfinite(v.real()) || !std::isfinite(v.imag())) return fail(QB_EINVAL, "L has a non-finite entry");
          lmax = std::max(lmax, std::abs(v));
          const long long dP = (long long)(p - c) + (q - c) - (r - c) - (s - c);
          bool cons = model->exact_momentum ? dP == 0 : modp(dP, M) == 0;
          if (!cons && v != cd(0, 0))
            return fail(QB_EINVAL, model->exact_momentum ? "L is nonzero on a tuple that does not conserve momentum"
                                                         : "L is nonzero on a tuple that does not conserve momentum mod M");
        }
  Lsym.assign(2 * M4, 0.0);
  for (int p = 0; p < M; ++p)
    for (int q = 0; q < M; ++q)
      for (int r = 0; r < M; ++r)
        for (int s = 0; s < M; ++s) {
          cd v = 0.25 * (Lat(p, q, r, s) + Lat(q, p, r, s) + Lat(p, q, s, r) + Lat(q, p, s, r));
          size_t t = (((size_t)p * M + q) * M + r) * M + s;
          Lsym[2 * t] = v.real();
          Lsym[2 * t + 1] = v.imag();
        }
  auto S = [&](int p, int q, int r, int s) {
    size_t t = (((size_t)p * M + q) * M + r) * M + s;
    return cd(Lsym[2 * t], Lsym[2 * t + 1]);
  };
  for (int p = 0; p < M; ++p)
    for (int q = 0; q < M; ++q)
      for (int r = 0; r < M; ++r)
        for (int s = 0; s < M; ++s)
          if (std::abs(S(p, q, r, s) - std::conj(S(r, s, p, q))) > 1e-12 * std::max(1.0, lmax))
            return fail(QB_EINVAL, "the symmetrised coupling is not Hermitian: L_{pq;rs} != conj(L_{rs;pq})");
  return QB_OK;
}

// The block tables of the stage kernel (Tables::bk_*), all but the maps, which the
// device fills.  The suffix takes as many modes as keep the maps within kMapBytes and a
// class within 16-bit places: longer blocks mean fewer rows of bases, while the maps are
// read beside the gathers and should stay in L2.  One step of the M = 9, N = 27 long-range
// space (23.5M kets) takes 22.8 ms with 6 MB, 21.5 with 24 and 21.8 with 80; of the M = 7,
// n_tot = 16 contact space 24.3, 23.9 and 23.9.
//
// With many modes that leaves blocks of a few kets, each with a row of bases for hundreds of
// terms (M = 16, n_max = 14, long-range: 2.4 KB a ket, 345 GB).  Where the rows would take more
// than kBaseBytes a ket, or than kBaseRoom in all and 16 bytes a ket, the suffix grows on while
// maps and rows together shrink (that space, 145M kets: 9 GB).  It costs no time: one step of
// M = 16, 5.3M kets, 1,486 B a ket 25.2 ms, 274 B 25.3; M = 13, 1.1M kets, 702 B 4.15, 279 B 4.06;
// M = 12, 2.7M kets, 368 B 7.12, 212 B 7.06.
constexpr int64_t kMapBytes = 24ll << 20;
constexpr int64_t kBaseBytes = 256, kBaseRoom = 8ll << 30;

// Blocks of the fillings of modes m .. M-1 (m <= P): [P + 1][nmax + 1][Q]
static std::vector<uint32_t> block_counts(const Space& sp, int P) {
  const int V = sp.nmax + 1, Q = sp.Q;
  auto CI = [&](int m, int n, int k) { return ((size_t)m * V + n) * Q + k; };
  std::vector<uint32_t> c((size_t)(P + 1) * V * Q, 0);
  for (int n = 0; n < V; ++n)
    for (int k = 0; k < Q; ++k) c[CI(P, n, k)] = sp.cnt[CI(P, n, k)] > 0;
  for (int m = P - 1; m >= 0; --m)
    for (int n = 0; n < V; ++n)
      for (int k = 0, j = modp(-m, Q); k < Q; ++k, j = j + 1 == Q ? 0 : j + 1)
        c[CI(m, n, k)] = c[CI(m + 1, n, k)] + (n > 0 ? c[CI(m, n - 1, j)] : 0);
  return c;
}

static void build_block_tables(Space& sp, bool factored) {
  Tables& t = sp.t;
  const std::vector<int>&annR = sp.combos.annR, &annS = sp.combos.annS, &annStart = sp.combos.annStart;
  const std::vector<uint32_t>& pq = sp.combos.pq;
  const std::vector<double>& G = sp.combos.G;
  const std::vector<std::array<int, 16>>& delta = sp.combos.delta;
  const unsigned char(*pairidx)[16] = sp.combos.pairidx;
  const int M = sp.M, nmax = sp.nmax, Q = sp.Q, twoQ = 2 * Q;
  t.bk_kc = (M % 2 == 1 && M >= 5 && M <= 11 && !sp.exact && !t.is_complex) ? (M - 1) / 2 : 0;
  const int w = t.bk_kc == 2 ? 2 : 4, per = t.bk_kc > 0 ? t.bk_kc : 4;
  struct Record {
    int pair, first, n;
    bool last;
  };
  std::vector<Record> recs;
  for (size_t a = 0; a < annR.size(); ++a)
    for (int j = annStart[a]; j < annStart[a + 1]; j += per)
      recs.push_back({(int)a, j, std::min(per, annStart[a + 1] - j), j + per >= annStart[a + 1]});
  const int nrec = (int)recs.size();
  t.bk_nrec = nrec;
  t.bk_T = std::max(4, (nrec * (t.bk_kc == 5 ? 5 : w) + 3) & ~3);
  const int TS = t.bk_T + 4;

  auto CI = [&](int m, int n, int k) { return ((size_t)m * (nmax + 1) + n) * Q + k; };
  // map bytes per filling (factored: the pairs added, four a group, and taken away)
  const int64_t per_fill = factored ? 8 * ((M * (M + 1) / 2 + 3) / 4 + (sp.exact ? 2 * M : M) * ((M + 8) / 8))
                                    : (int64_t)std::max(1, nrec) * (t.bk_kc == 5 ? 10 : 2 * w);
  // fillings of the modes q .. M-1 with their gaps; -1: a class exceeds 16-bit places
  auto fillings = [&](int q) {
    int64_t S = 0;
    for (int n = 0; n <= nmax; ++n)
      for (int k = 0; k < Q; ++k) {
        const int64_t c = (int64_t)sp.cnt[CI(q, n, k)];
        if (c > 65535) return (int64_t)-1;
        S += c + 1;
      }
    return S;
  };
  auto row_bytes = [&](const std::vector<uint32_t>& c) {  // of bases, from the counts of blocks
    int64_t rows = 0, low = 0;
    for (size_t i = 0; i < sp.secN.size(); ++i) rows += c[CI(0, sp.secN[i], sp.secK[i])];
    if (!factored) return 4ll * t.bk_T * rows;
    for (size_t i = 0; i < sp.lowN.size(); ++i) low += c[CI(0, sp.lowN[i], sp.lowK[i])];
    return 4ll * (fa_Tc(t) * rows + fa_rowa(t) * low);
  };
  int P = M - 1;
  int64_t S = fillings(P);
  while (P > 0) {
    const int64_t s = fillings(P - 1);
    if (s < 0 || s * per_fill > kMapBytes) break;
    --P;
    S = s;
  }
  const int64_t total = sp.secOff.back(), room = std::min(kBaseBytes * total, std::max(kBaseRoom, 16 * total));
  sp.blkCnt = block_counts(sp, P);
  for (int64_t rows = row_bytes(sp.blkCnt); P > 0 && rows > room; --P) {
    std::vector<uint32_t> counts = block_counts(sp, P - 1);
    const int64_t s = fillings(P - 1), next = row_bytes(counts);
    if (s < 0 || s > 0x7fffffff || s * per_fill + next >= S * per_fill + rows) break;
    sp.blkCnt.swap(counts);
    S = s;
    rows = next;
  }
  t.bk_S = (int)S;
  t.bk_P = P;
  // A ket takes part in the records of a pair (r, s) if it is a ket of two particles fewer with
  // them added: summed by the pairs' momentum classes.
  {
    std::vector<int> of(annR.size(), 0), in_class(std::min(Q, 2 * M - 1), 0);
    int most = 0;
    for (const Record& R : recs) {
      most = std::max(most, ++of[R.pair]);
      ++in_class[(annR[R.pair] + annS[R.pair]) % Q];
    }
    double taken = 0.0;
    for (size_t i = 0; i < sp.secN.size(); ++i)
      for (int k = 0; k < (int)in_class.size() && sp.secN[i] >= 2; ++k)
        taken += (double)in_class[k] * (double)sp.cnt[CI(0, sp.secN[i] - 2, sp.secK[i] - k + (sp.secK[i] < k ? Q : 0))];
    t.bk_share = nrec > 0 ? (float)(taken / ((double)nrec * (double)sp.secOff.back())) : 1.f;
    // (p modes occupied, of which nmax / 2 twice at most)
    const int64_t p = std::min(M, nmax);
    t.bk_most = (int)std::min<int64_t>(nrec, most * (p * (p - 1) / 2 + std::min(M, nmax / 2)));
  }

  std::vector<uint32_t> info(2 * (size_t)std::max(1, nrec));
  std::vector<float> Gr(2 * (size_t)t.bk_T, 0.f), Gi(2 * (size_t)t.bk_T, 0.f);
  std::vector<int32_t> psh((size_t)M * TS, 0), EC((size_t)t.rem_w * twoQ, 0), cls(2 * (size_t)(nmax + 1) * Q);
  std::vector<uint32_t> combo(t.bk_T, 0xffffffffu);
  for (int i = 0; i < nrec; ++i) {
    const Record& R = recs[i];
    int after = 0;  // first partner with a larger pair index (partners ascend)
    for (int c = 0; c < R.n; ++c) {
      const int j = R.first + c, sl = c < 4 ? w * i + c : 4 * nrec + i;
      if ((int)pairidx[pq[j] & 0xff][(pq[j] >> 8) & 0xff] < R.pair) after = c + 1;
      for (int k = 0; k < 2; ++k) {
        float* g = (k ? Gi : Gr).data() + 2 * (size_t)sl;
        g[0] = (float)G[2 * j + k];
        g[1] = (float)(G[2 * j + k] - (double)g[0]);
      }
      combo[sl] = (uint32_t)j;
      for (int m = 1; m < M; ++m) psh[(size_t)m * TS + sl] = delta[j][m];
    }
    const uint32_t r = (uint32_t)annR[R.pair], q = (uint32_t)annS[R.pair];
    info[2 * i] = (r & 7) | ((uint32_t)R.n << 4) | (R.last ? 0x80u : 0u) | ((uint32_t)after << 8) |
                  (r >= 8 ? 0x8000u : 0u) | ((q & 7) << 16) | (q >= 8 ? 0x80000000u : 0u);
    info[2 * i + 1] = r == q ? 0x4B000001u : 0x4B000000u;  // 2^23 + [r = s]
  }
  for (int rr = 0; rr < t.rem_w; ++rr)
    for (int kk = 0; kk < twoQ; ++kk) {
      const int rem = rr - 2;
      int64_t v = 0;
      if (P >= 1 && rem >= 1 && rem - 1 <= nmax) v = (int64_t)sp.cnt[CI(P - 1, rem - 1, modp(kk - (P - 1), Q))];
      if (rem >= 0 && rem <= nmax) v += (int64_t)sp.cnt[CI(P, rem, kk % Q)];
      EC[(size_t)rr * twoQ + kk] = (int32_t)v;
    }
  int32_t first = 0;
  for (int n = 0; n <= nmax; ++n)
    for (int k = 0; k < Q; ++k) {
      const int32_t c = (int32_t)sp.cnt[CI(P, n, k)];
      cls[2 * ((size_t)n * Q + k)] = first;
      cls[2 * ((size_t)n * Q + k) + 1] = c;
      first += c + 1;
    }
  auto put = [&](int k, const void* p, size_t bytes) {
    sp.bk_off[k] = sp.bk.size();
    sp.bk.insert(sp.bk.end(), (const unsigned char*)p, (const unsigned char*)p + bytes);
    sp.bk.resize((sp.bk.size() + 255) & ~(size_t)255);
  };
  put(0, info.data(), 4 * info.size());
  put(1, Gr.data(), 4 * Gr.size());
  put(2, Gi.data(), 4 * Gi.size());
  put(3, psh.data(), 4 * psh.size());
  put(4, EC.data(), 4 * EC.size());
  put(5, cls.data(), 4 * cls.size());
  put(7, combo.data(), 4 * combo.size());
  sp.bk_map_bytes = ((size_t)std::max(1, nrec) * t.bk_S * 2 * w + 255) & ~(size_t)255;
}

// Blocks (Tables::rblk) of the sectors and of the lower sectors, from whose counts the device
// finds block b of a sector as it finds a ket from the fill counts.
static void count_blocks(Space& sp) {
  const int V = sp.nmax + 1, Q = sp.Q;
  auto CI = [&](int m, int n, int k) { return ((size_t)m * V + n) * Q + k; };
  auto run = [&](const std::vector<int>& N, const std::vector<int>& K, std::vector<uint32_t>& out) {
    out.assign(1, 0);
    for (size_t i = 0; i < N.size(); ++i) out.push_back(out.back() + sp.blkCnt[CI(0, N[i], K[i])]);
  };
  run(sp.secN, sp.secK, sp.secBlk);
  if (sp.t.fa_on) run(sp.lowN, sp.lowK, sp.lowBlk);
}

// Whether the two-body part factors into one operator per momentum class,
// sum_k lam_k B_k^dag B_k (a contact interaction): every symmetrised coupling of a class
// is the same real number.  Then builds the tables of the factored stages (Tables::fa_*)
// and the list of lower sectors; called once the sectors are known.
//
// Where the line lies (one stage, direct against factored kernels, us): two launches cost
// more than one, so small spaces stay direct (M = 7, 19,448 kets: 10.5 / 13.5; 245,157: 38 / 27;
// M = 9, 35,530: 17.4 / 14.2; M = 11, 16,796: 19.0 / 14.9), and with three pairs a class
// (M = 5) the second pass costs what the fewer terms save (2.3M kets: 138 / 149).
constexpr int kFactorMinM = 6;
constexpr int64_t factor_min(int M) { return M >= 9 ? 16384 : 32768; }

static bool build_factored(Space& sp) {
  Tables& t = sp.t;
  const int M = sp.M, nmax = sp.nmax, Q = sp.Q, twoQ = 2 * Q;
  t.fa_on = 0;
  if (M < kFactorMinM || sp.secOff.back() < factor_min(M) || sp.secOff.back() >= (int64_t)kNoIndex) return false;
  const int nc = sp.exact ? 2 * M - 1 : M;
  std::vector<std::vector<std::pair<int, int>>> cls(nc);  // pairs p < q first, then p = q
  for (int d = 0; d < 2; ++d)
    for (int p = 0; p < M; ++p)
      for (int q = d ? p : p + 1; q < (d ? p + 1 : M); ++q) cls[(p + q) % (sp.exact ? 2 * M : M)].push_back({p, q});
  auto LS = [&](std::pair<int, int> a, std::pair<int, int> b) {
    const size_t ix = (((size_t)a.first * M + a.second) * M + b.first) * M + b.second;
    return cd(sp.Lsym[2 * ix], sp.Lsym[2 * ix + 1]);
  };
  std::vector<float> lam(2 * (size_t)nc);
  std::vector<double> lam64(nc);
  for (int k = 0; k < nc; ++k) {
    const cd l0 = LS(cls[k][0], cls[k][0]);
    if (l0.imag() != 0.0) return false;
    for (auto a : cls[k])
      for (auto b : cls[k])
        if (LS(a, b) != l0) return false;
    lam64[k] = l0.real();
    lam[2 * k] = (float)l0.real();
    lam[2 * k + 1] = (float)(l0.real() - (double)lam[2 * k]);
  }
  // lower sectors and the vector of B_k f
  sp.lowN.clear();
  sp.lowK.clear();
  sp.lowOff.assign(1, 0);
  std::vector<int32_t> lowof((size_t)(nmax + 1) * Q, -1);
  std::vector<uint32_t> goff;
  int64_t nG = 0;
  for (int n = std::max(0, sp.nmin - 2); n + 2 <= nmax; ++n)
    for (int k0 = 0; k0 < Q; ++k0) {
      // within a layer in the order of the space's sectors (ascending label sum)
      const int c = label_shift(M);
      const int K = sp.exact ? k0 : modp((long long)k0 + (long long)c * n, Q);
      const int64_t D = (int64_t)sp.cnt[((size_t)0 * (nmax + 1) + n) * Q + K];
      if (D == 0) continue;
      bool any = false;
      std::vector<uint32_t> row(nc, kNoIndex);
      for (int k = 0; k < nc; ++k) {
        if (sp.secOf[(size_t)(n + 2) * Q + (K + k) % Q] < 0) continue;
        if (sp.exact && K + k > (M - 1) * (n + 2)) continue;
        if (nG + D >= (int64_t)kNoIndex) return false;
        row[k] = (uint32_t)nG;
        nG += D;
        any = true;
      }
      if (!any) continue;
      lowof[(size_t)n * Q + K] = (int32_t)sp.lowN.size();
      sp.lowN.push_back(n);
      sp.lowK.push_back(K);
      sp.lowOff.push_back(sp.lowOff.back() + D);
      goff.insert(goff.end(), row.begin(), row.end());
    }
  const int nlow = (int)sp.lowN.size();
  if (nlow == 0) return false;
  const int64_t total = sp.secOff.back();
  if (total > kObsfKets) {  // 120 bytes a ket: tables, state and workspace of a direct step
    size_t avail = 0, all = 0;
    if (cudaMemGetInfo(&avail, &all) != cudaSuccess) return false;
    if (120.0 * (double)total + 16.0 * (double)nG + 12.0 * (double)sp.lowOff.back() > 0.9 * (double)all) return false;
  }
  sp.low_held = nlow <= (int)sp.secN.size();
  for (int i = 0; i < nlow && sp.low_held; ++i)
    sp.low_held = sp.secN[i] == sp.lowN[i] && sp.secK[i] == sp.lowK[i] && sp.secOff[i] == sp.lowOff[i];

  // annihilation records
  const bool fix = M % 2 == 1 && !sp.exact;
  t.fa_nt = fix && M <= 11 ? (M + 1) / 2 : 0;
  t.fa_pl = t.fa_nt > 4 ? 2 : 1;
  const int per = t.fa_nt > 0 ? t.fa_nt : 4;
  std::vector<uint32_t> rec;
  std::vector<std::pair<int, int>> slot;  // pair of each annihilation slot (first < 0: unused)
  std::vector<int32_t> ka;
  for (int k = 0; k < nc; ++k) {
    const int n = (int)cls[k].size();
    int noff = 0;
    while (noff < n && cls[k][noff].first != cls[k][noff].second) ++noff;
    for (int j = 0; j < n; j += per) {
      const int m = std::min(per, n - j);
      const int dbl = noff > j && noff <= j + m ? noff - j : 7;
      rec.push_back((uint32_t)k | ((uint32_t)m << 8) | ((uint32_t)(t.fa_nt ? 7 : dbl) << 12) |
                    (j + per >= n ? 0x10000u : 0u));
      rec.push_back(0u);
      for (int c = 0; c < 4 * t.fa_pl; ++c) {
        slot.push_back(c < m ? cls[k][j + c] : std::pair<int, int>(-1, -1));
        ka.push_back(k);
      }
    }
  }
  t.fa_nrec = (int)rec.size() / 2;
  t.fa_nc = nc;
  // creation groups: the pairs r < s, then r = s
  std::vector<std::pair<int, int>> cre;
  for (int r = 0; r < M; ++r)
    for (int s = r + 1; s < M; ++s) cre.push_back({r, s});
  for (int r = 0; r < M; ++r) cre.push_back({r, r});
  while (cre.size() % 4) cre.push_back({-1, -1});
  t.fa_ng = (int)cre.size() / 4;
  const int Ta = fa_Ta(t), Tc = fa_Tc(t);
  std::vector<int32_t> kc(Tc, 0), psa((size_t)M * Ta, 0), psc((size_t)M * Tc, 0);
  std::vector<uint32_t> info(Tc, 0u), pqa(Ta, 0u);
  for (int i = 0; i < Ta; ++i)
    if (slot[i].first >= 0) pqa[i] = (uint32_t)slot[i].first | ((uint32_t)slot[i].second << 8);
  std::vector<float> coef(2 * (size_t)Tc, 0.f);
  auto shift = [&](std::pair<int, int> pr, int m, int sign) {
    const int dc = (pr.first >= m) + (pr.second >= m);
    const int dk = (pr.first >= m ? pr.first : 0) + (pr.second >= m ? pr.second : 0);
    return sign * dc * twoQ + modp((long long)sign * dk, Q);
  };
  for (int i = 0; i < Ta; ++i)
    for (int m = 0; m < M && slot[i].first >= 0; ++m) psa[(size_t)m * Ta + i] = shift(slot[i], m, 1);
  for (int i = 0; i < Tc; ++i) {
    if (cre[i].first < 0) continue;
    const uint32_t r = (uint32_t)cre[i].first, q = (uint32_t)cre[i].second;
    kc[i] = sp.exact ? (int)(r + q) : (int)((r + q) % M);
    for (int m = 0; m < M; ++m) psc[(size_t)m * Tc + i] = shift(cre[i], m, -1);
    info[i] = (r & 7) | (r >= 8 ? 0x8000u : 0u) | ((q & 7) << 16) | (q >= 8 ? 0x80000000u : 0u);
    coef[2 * i] = r == q ? 8388609.f : 8388608.f;
    coef[2 * i + 1] = r == q ? 1.f : 2.f;
  }
  sp.fa.clear();
  int at = 0;
  auto put = [&](const void* p, size_t bytes) {
    sp.fa_off[at++] = sp.fa.size();
    sp.fa.insert(sp.fa.end(), (const unsigned char*)p, (const unsigned char*)p + bytes);
    sp.fa.resize((sp.fa.size() + 255) & ~(size_t)255);
  };
  put(rec.data(), 4 * rec.size());
  put(lam.data(), 4 * lam.size());
  put(ka.data(), 4 * ka.size());
  put(kc.data(), 4 * kc.size());
  put(psa.data(), 4 * psa.size());
  put(psc.data(), 4 * psc.size());
  put(info.data(), 4 * info.size());
  put(coef.data(), 4 * coef.size());
  put(lowof.data(), 4 * lowof.size());
  put(sp.lowOff.data(), 8 * sp.lowOff.size());
  put(goff.data(), 4 * goff.size());
  put(sp.lowN.data(), 4 * sp.lowN.size());
  put(sp.lowK.data(), 4 * sp.lowK.size());
  at = 15;
  put(lam64.data(), 8 * lam64.size());
  put(pqa.data(), 4 * pqa.size());
  t.fa_nlow = nlow;
  t.fa_every = std::find(goff.begin(), goff.end(), kNoIndex) == goff.end() ? 1 : 0;
  t.fa_low = sp.lowOff.back();
  t.fa_nG = nG;
  t.fa_on = 1;
  return true;
}

// Builds the fill counts, ranking table, coupling combinations and the
// shared-memory image of the space.
static int build_tables(Space& sp) {
  const int M = sp.M, nmax = sp.nmax, Q = sp.Q;
  // cnt[m][n][k]: fillings of modes m..M-1 with n particles, sum_i i n_i = k mod Q.
  // With Q = (M-1) nmax + 1 no momentum sum of the space wraps: the counts, the
  // ranking table and the coupling combinations below are those of exact
  // conservation, and a wrapped (negative) index lands on a zero count.
  auto CI = [&](int m, int n, int k) { return ((size_t)m * (nmax + 1) + n) * Q + k; };
  sp.cnt.assign((size_t)(M + 1) * (nmax + 1) * Q, 0);
  sp.cnt[CI(M, 0, 0)] = 1;
  // either mode m is empty or one particle of it is taken away
  for (int m = M - 1; m >= 0; --m)
    for (int n = 0; n <= nmax; ++n)
      for (int k = 0, j = modp(-m, Q); k < Q; ++k, j = j + 1 == Q ? 0 : j + 1) {
        const uint64_t acc = sp.cnt[CI(m + 1, n, k)] + (n > 0 ? sp.cnt[CI(m, n - 1, j)] : 0);
        sp.cnt[CI(m, n, k)] = std::min<uint64_t>(acc, 1ull << 62);
      }
  for (uint64_t v : sp.cnt)
    if (v >= (1ull << 31)) return fail(QB_EUNSUPPORTED, "a sub-sector count reaches 2^31; reduce n_max");

  Tables& t = sp.t;
  t.M = M;
  t.Q = Q;
  t.exact = sp.exact;
  t.nmax = nmax;
  t.rem_w = nmax + 5;
  t.n_ann = M * (M + 1) / 2;
  const int twoQ = 2 * Q;

  // annihilation pairs (r <= s) and their creation partners (p <= q) in the same
  // momentum class, excluding the pair itself (those are diagonal)
  auto LS = [&](int p, int q, int r, int s) {
    size_t ix = (((size_t)p * M + q) * M + r) * M + s;
    return cd(sp.Lsym[2 * ix], sp.Lsym[2 * ix + 1]);
  };
  sp.combos = Combos();
  std::vector<int>&annR = sp.combos.annR, &annS = sp.combos.annS, &annStart = sp.combos.annStart;
  std::vector<uint32_t>& pq = sp.combos.pq;
  std::vector<double>& G = sp.combos.G;
  std::vector<std::array<int, 16>>& delta = sp.combos.delta;
  std::vector<double> gd;
  unsigned char(*pairidx)[16] = sp.combos.pairidx;
  memset(pairidx, 0xff, 256);
  bool cplx = false;
  for (int r = 0; r < M; ++r)
    for (int s = r; s < M; ++s) {
      int a = (int)annR.size();
      pairidx[r][s] = pairidx[s][r] = (unsigned char)a;
      annR.push_back(r);
      annS.push_back(s);
      annStart.push_back((int)pq.size());
      double mrs = (r == s) ? 1.0 : 2.0;
      gd.push_back(mrs * mrs * LS(r, s, r, s).real());
      int k = (r + s) % Q;
      for (int p = 0; p < M; ++p)
        for (int q = p; q < M; ++q) {
          if ((p + q) % Q != k || (p == r && q == s)) continue;
          double mpq = (p == q) ? 1.0 : 2.0;
          // combos with a zero coupling are kept: for odd M every pair then has
          // (M-1)/2 partners, which the specialised stage kernels unroll
          cd g = std::conj(mpq * mrs * LS(p, q, r, s));
          if (g.imag() != 0.0) cplx = true;
          int lo = std::min(r, p), hi = std::max(s, q);
          pq.push_back((uint32_t)p | ((uint32_t)q << 8) | ((uint32_t)lo << 16) | ((uint32_t)hi << 24));
          G.push_back(g.real());
          G.push_back(g.imag());
          std::array<int, 16> d{};
          int dn[16] = {0};
          dn[r] -= 1;
          dn[s] -= 1;
          dn[p] += 1;
          dn[q] += 1;
          for (int m = lo + 1; m <= hi; ++m) {
            int dc = 0, dk = 0;
            for (int e = m; e < M; ++e) {
              dc += dn[e];
              dk += dn[e] * e;
            }
            d[m] = dc * twoQ + modp(dk, Q);
          }
          delta.push_back(d);
        }
    }
  annStart.push_back((int)pq.size());
  t.n_combo = (int)pq.size();
  t.is_complex = cplx ? 1 : 0;


  // the image that the row kernels stage in shared memory
  size_t off = 0;
  t.o_cnt = (int)off;
  off = align16(off + sizeof(uint32_t) * (size_t)(M + 1) * (nmax + 1) * Q);
  t.o_E = (int)off;
  off = align16(off + sizeof(int32_t) * (size_t)M * t.rem_w * twoQ);
  t.o_ann = (int)off;
  off = align16(off + sizeof(int32_t) * (size_t)(t.n_ann + 1));
  t.o_pairidx = (int)off;
  off = align16(off + 256);
  t.o_delta = (int)off;
  off = align16(off + (size_t)(sp.exact ? 32 : 16) * std::max(1, t.n_combo));
  t.o_sqrt = (int)off;
  off = align16(off + sizeof(double) * (size_t)(nmax + 3));
  t.o_pq = (int)off;
  off = align16(off + sizeof(uint32_t) * (size_t)std::max(1, t.n_combo));
  t.o_G = (int)off;
  off = align16(off + sizeof(double) * 2 * (size_t)std::max(1, t.n_combo));
  t.o_w = (int)off;
  off = align16(off + sizeof(double) * (size_t)M);
  t.o_gd = (int)off;
  off = align16(off + sizeof(double) * (size_t)t.n_ann);
  t.blob_bytes = (int)off;
  // mod M: the moments kernel holds two ranking-table byte offsets per 32-bit word, so the
  // table must span at most 64 KB (every space within the other limits does but M = 9 with
  // 97 <= n_max <= 108, whose sectors exceed 2^31 kets anyway)
  if (!sp.exact && (int64_t)M * t.rem_w * twoQ * 4 > 65536)
    return fail(QB_EUNSUPPORTED, "the ranking table exceeds 64 KB (reduce n_max)");
  // exact momentum: the fill counts and the ranking table grow with (M-1) n_max
  // and stay in global memory for every kernel
  t.sm_from = sp.exact ? t.o_ann : 0;
  sp.blob.assign(off, 0);
  unsigned char* b = sp.blob.data();
  uint32_t* cnt32 = (uint32_t*)(b + t.o_cnt);
  for (size_t i = 0; i < sp.cnt.size(); ++i) cnt32[i] = (uint32_t)sp.cnt[i];
  int32_t* E = (int32_t*)(b + t.o_E);
  for (int m = 1; m < M; ++m)
    for (int rr = 3; rr < t.rem_w && rr - 3 <= nmax; ++rr)
      for (int kk = 0, j = modp(1 - m, Q); kk < twoQ; ++kk, j = j + 1 == Q ? 0 : j + 1)
        E[((size_t)m * t.rem_w + rr) * twoQ + kk] = (int32_t)sp.cnt[CI(m - 1, rr - 3, j)];
  double* sq = (double*)(b + t.o_sqrt);
  for (int k = 0; k < nmax + 3; ++k) sq[k] = std::sqrt((double)k);
  memcpy(b + t.o_pq, pq.data(), sizeof(uint32_t) * pq.size());
  memcpy(b + t.o_G, G.data(), sizeof(double) * G.size());
  if (sp.exact) {  // int16 shifts (|shift| <= 5Q)
    if (5LL * Q > 32767) return fail(QB_EUNSUPPORTED, "exact momentum: (M-1) n_max too large for 16-bit shifts");
    int16_t* dl = (int16_t*)(b + t.o_delta);
    for (int j = 0; j < t.n_combo; ++j)
      for (int m = 0; m < 16; ++m) dl[(size_t)j * 16 + m] = (int16_t)delta[j][m];
  } else {
    uint8_t* dl = (uint8_t*)(b + t.o_delta);
    for (int j = 0; j < t.n_combo; ++j)
      for (int m = 0; m < 16; ++m) dl[(size_t)j * 16 + m] = (uint8_t)(delta[j][m] + kDeltaBias);
  }
  memcpy(b + t.o_ann, annStart.data(), sizeof(int32_t) * annStart.size());
  memcpy(b + t.o_pairidx, pairidx, 256);
  memcpy(b + t.o_w, sp.w.data(), sizeof(double) * M);
  memcpy(b + t.o_gd, gd.data(), sizeof(double) * gd.size());
  return QB_OK;
}

// rank of an occupation vector within the space (host mirror of the device
// ranking, used for number-state initialisation); -1 if absent
static int64_t host_rank(const Space& sp, const int* occ) {
  const int M = sp.M;
  int N = 0;
  long long K = 0;
  for (int i = 0; i < M; ++i) {
    if (occ[i] < 0) return -1;
    N += occ[i];
    K += (long long)i * occ[i];
  }
  if (N > sp.nmax || N < 0) return -1;
  const int Q = sp.Q;
  int Kk = modp(K, Q);
  int sid = sp.secOf[(size_t)N * Q + Kk];
  if (sid < 0) return -1;
  auto CI = [&](int m, int n, int k) { return ((size_t)m * (sp.nmax + 1) + n) * Q + k; };
  int64_t sum = 0;
  int rem = 0;
  long long kr = 0;
  for (int m = M - 1; m >= 1; --m) {
    rem += occ[m];
    kr += (long long)m * occ[m];
    if (rem >= 1) sum += (int64_t)sp.cnt[CI(m - 1, rem - 1, modp(kr - (m - 1), Q))];
  }
  return sp.secOff[sid] + sp.secDim[sid] - 1 - sum;
}

// ---------------------------------------------------------------- eigensolve

// Eigen-decomposition of a Hermitian n x n matrix (n <= QB_MAX_MODES) by cyclic complex
// Jacobi rotations: eig receives the eigenvalues ascending, vec the unit eigenvector of the
// largest one (its phase is arbitrary).  The rotated-out entries are set to zero, so that a
// few sweeps end it; on the real 2n x 2n embedding, four times the entries, most of a
// small space's qb_observables was this (M = 7: 0.4 of 0.56 ms).
static void hermitian_eig(int n, const double* A /*[n*n] complex*/, double* eig, double* vec /*[n] complex*/) {
  cd S[QB_MAX_MODES][QB_MAX_MODES], V[QB_MAX_MODES][QB_MAX_MODES];
  for (int i = 0; i < n; ++i)
    for (int j = 0; j < n; ++j) {  // the Hermitian part
      const double re = 0.5 * (A[2 * (i * n + j)] + A[2 * (j * n + i)]);
      const double im = 0.5 * (A[2 * (i * n + j) + 1] - A[2 * (j * n + i) + 1]);
      S[i][j] = cd(re, im);
      V[i][j] = i == j ? 1.0 : 0.0;
    }
  auto mul = [](cd a, cd b) { return cd(a.real() * b.real() - a.imag() * b.imag(), a.real() * b.imag() + a.imag() * b.real()); };
  for (int sweep = 0; sweep < 100; ++sweep) {
    double off = 0.0, tot = 0.0;
    for (int i = 0; i < n; ++i)
      for (int j = 0; j < n; ++j) {
        const double v = std::norm(S[i][j]);
        tot += v;
        if (i != j) off += v;
      }
    if (off <= 1e-32 * tot || off == 0.0) break;
    for (int p = 0; p < n - 1; ++p)
      for (int q = p + 1; q < n; ++q) {
        const double m = std::abs(S[p][q]);
        if (m == 0.0) continue;
        const cd ph = S[p][q] / m;  // e^{i phi}
        const double app = S[p][p].real(), aqq = S[q][q].real();
        const double theta = (aqq - app) / (2.0 * m);
        const double tt = (theta >= 0 ? 1.0 : -1.0) / (std::fabs(theta) + std::sqrt(theta * theta + 1.0));
        const double c = 1.0 / std::sqrt(tt * tt + 1.0), s = tt * c;
        const cd sp = s * ph, sm = std::conj(sp);
        // columns: u_p = c e_p - s e^{-i phi} e_q, u_q = s e^{i phi} e_p + c e_q
        for (int k = 0; k < n; ++k) {
          const cd x = S[k][p], y = S[k][q];
          S[k][p] = c * x - mul(sm, y);
          S[k][q] = mul(sp, x) + c * y;
          const cd vx = V[k][p], vy = V[k][q];
          V[k][p] = c * vx - mul(sm, vy);
          V[k][q] = mul(sp, vx) + c * vy;
        }
        for (int k = 0; k < n; ++k) {  // rows: the adjoint
          const cd x = S[p][k], y = S[q][k];
          S[p][k] = c * x - mul(sp, y);
          S[q][k] = mul(sm, x) + c * y;
        }
        S[p][q] = S[q][p] = 0.0;
        S[p][p] = S[p][p].real();
        S[q][q] = S[q][q].real();
      }
  }
  int order[QB_MAX_MODES];
  for (int i = 0; i < n; ++i) order[i] = i;
  std::sort(order, order + n, [&](int a, int b) { return S[a][a].real() < S[b][b].real(); });
  for (int k = 0; k < n; ++k) eig[k] = S[order[k]][order[k]].real();
  const int top = order[n - 1];
  double nrm = 0.0;
  for (int i = 0; i < n; ++i) nrm += std::norm(V[i][top]);
  nrm = std::sqrt(nrm);
  for (int i = 0; i < n; ++i) {
    vec[2 * i] = V[i][top].real() / nrm;
    vec[2 * i + 1] = V[i][top].imag() / nrm;
  }
}

// Derived observables of Sec. II C-E from the raw moments.
void derive(int M, const double* raw, qb_obs* o) {
  memset(o, 0, sizeof(*o));
  double nrm = raw[0];
  o->norm = nrm;
  o->N = raw[1] / nrm;
  o->H = raw[2] / nrm;
  const double* A = raw + 4;
  const double* Mm = A + 2 * M;
  const double* AA = Mm + 2 * M * M;
  std::vector<cd> a(M), Mij((size_t)M * M), aa((size_t)M * M);
  for (int i = 0; i < M; ++i) a[i] = cd(A[2 * i], A[2 * i + 1]) / nrm;
  for (int i = 0; i < M * M; ++i) Mij[i] = cd(Mm[2 * i], Mm[2 * i + 1]) / nrm;
  // <a_k a_l> is symmetric; the device fills k <= l only
  for (int k = 0; k < M; ++k)
    for (int l = 0; l < M; ++l) {
      const int u = (k <= l) ? k * M + l : l * M + k;
      aa[(size_t)k * M + l] = cd(AA[2 * u], AA[2 * u + 1]) / nrm;
    }
  for (int i = 0; i < M; ++i) {
    o->a[2 * i] = a[i].real();
    o->a[2 * i + 1] = a[i].imag();
  }
  std::vector<double> mflat(2 * (size_t)M * M);
  for (int i = 0; i < M * M; ++i) {
    o->Mij[2 * i] = mflat[2 * i] = Mij[i].real();
    o->Mij[2 * i + 1] = mflat[2 * i + 1] = Mij[i].imag();
    o->aa[2 * i] = aa[i].real();
    o->aa[2 * i + 1] = aa[i].imag();
  }
  double ntot = 0.0, dsum = 0.0;
  for (int j = 0; j < M; ++j) {
    ntot += Mij[(size_t)j * M + j].real();
    dsum += Mij[(size_t)j * M + j].real() - std::norm(a[j]);
  }
  o->n_tot = ntot;
  o->Q = dsum / ntot;
  hermitian_eig(M, mflat.data(), o->eig, o->xi);
  o->lam_p = o->eig[M - 1];
  o->PO = 1.0 - o->lam_p / ntot;
  o->gap = (M > 1) ? o->eig[M - 1] - o->eig[M - 2] : INFINITY;
  for (int i = 0; i < M; ++i) {
    double d = Mij[(size_t)i * M + i].real() - std::norm(a[i]);
    cd var = aa[(size_t)i * M + i] - a[i] * a[i];
    o->Vminus[i] = 1.0 + 2.0 * d - 2.0 * std::abs(var);
  }
  std::vector<cd> xi(M);
  for (int k = 0; k < M; ++k) xi[k] = cd(o->xi[2 * k], o->xi[2 * k + 1]);
  cd dd = 0, var = 0;
  for (int k = 0; k < M; ++k)
    for (int l = 0; l < M; ++l) {
      dd += std::conj(xi[k]) * xi[l] * (Mij[(size_t)k * M + l] - std::conj(a[k]) * a[l]);
      var += xi[k] * xi[l] * (aa[(size_t)k * M + l] - a[k] * a[l]);
    }
  o->Vminus_p = 1.0 + 2.0 * dd.real() - 2.0 * std::abs(var);
}

double log2_max_ket_weight(int M, int N) {
  // N! / prod n_m! is largest for the most even occupation: N mod M modes hold
  // floor(N / M) + 1 particles, the rest floor(N / M)
  const int q = N / M, r = N % M;
  const double ln = std::lgamma(N + 1.0) - r * std::lgamma(q + 2.0) - (M - r) * std::lgamma(q + 1.0);
  return 0.5 * ln / std::log(2.0);
}

}  // namespace qb

using namespace qb;

extern "C" {

const char* qb_last_error(void) { return g_err.c_str(); }

int qb_sector_build(const qb_model* model, int n_min, int n_max, const int* p_list, int n_p, qb_space** out) {
  if (!out) return fail(QB_EINVAL, "out must be non-NULL");
  *out = nullptr;
  Space* sp = new (std::nothrow) Space();
  if (!sp) return fail(QB_ENOMEM, "host allocation failed");
  int rc = prepare_model(model, sp->w, sp->Lsym);
  if (rc) {
    delete sp;
    return rc;
  }
  const int M = model->M;
  sp->M = M;
  if (n_min < 0 || n_max < n_min) {
    delete sp;
    return fail(QB_EINVAL, "need 0 <= n_min <= n_max");
  }
  int bits = 1;
  while ((1 << bits) <= n_max) ++bits;
  if (M * bits > 64 || n_max > 250) {
    delete sp;
    return fail(QB_EUNSUPPORTED, "occupation vectors do not pack into 64 bits (M * bits(n_max) > 64)");
  }
  // the stages hold psi / w(n) as fp32 pairs; the centred weights of the deepest sector
  // must stay within the range that keeps them exact (log2 w_max(n_max) <= 160)
  if (log2_max_ket_weight(M, n_max) > kMaxLog2KetWeight) {
    delete sp;
    return fail(QB_EUNSUPPORTED, "ket weights sqrt(N!/prod n!) of the deepest sector exceed 2^160 (reduce n_max): "
                                 "the weighted stage vectors would leave the fp32 exponent range");
  }
  sp->nmin = n_min;
  sp->nmax = n_max;
  sp->exact = model->exact_momentum ? 1 : 0;
  // exact: a modulus above every momentum sum (and above 2(M-1), so that pair
  // momenta never wrap either)
  sp->Q = sp->exact ? std::max((M - 1) * n_max + 1, 2 * M - 1) : M;
  rc = build_tables(*sp);
  if (rc) {
    delete sp;
    return rc;
  }
  std::vector<int> Ps;
  if (p_list) {
    if (n_p < 0) {
      delete sp;
      return fail(QB_EINVAL, "n_p must be >= 0");
    }
    for (int i = 0; i < n_p; ++i) Ps.push_back(sp->exact ? p_list[i] : modp(p_list[i], M));
    std::sort(Ps.begin(), Ps.end());
    Ps.erase(std::unique(Ps.begin(), Ps.end()), Ps.end());
  } else if (sp->exact) {
    // every label sum reachable with N <= n_max: sum_i (i - c) n_i in [-c n_max, (M-1-c) n_max]
    const int c0 = label_shift(M);
    for (int P = -c0 * n_max; P <= (M - 1 - c0) * n_max; ++P) Ps.push_back(P);
  } else {
    for (int P = 0; P < M; ++P) Ps.push_back(P);
  }
  const int c = label_shift(M);
  const int Q = sp->Q;
  sp->secOf.assign((size_t)(n_max + 1) * Q, -1);
  sp->secOff.push_back(0);
  for (int N = n_min; N <= n_max; ++N)
    for (int P : Ps) {
      // index momentum K = sum_i i n_i = P + c N; exact: must lie in [0, (M-1) N]
      const long long Kx = (long long)P + (long long)c * N;
      if (sp->exact && (Kx < 0 || Kx > (long long)(M - 1) * N)) continue;
      int K = modp(Kx, Q);
      uint64_t D = sp->cnt[((size_t)0 * (n_max + 1) + N) * Q + K];
      if (D == 0) continue;
      sp->secOf[(size_t)N * Q + K] = (int)sp->secN.size();
      sp->secN.push_back(N);
      sp->secP.push_back(P);
      sp->secK.push_back(K);
      sp->secDim.push_back((int64_t)D);
      sp->secOff.push_back(sp->secOff.back() + (int64_t)D);
      sp->maxDim = std::max(sp->maxDim, (int64_t)D);
    }
  if (sp->secN.empty()) {
    delete sp;
    return fail(QB_EINVAL, "no non-empty sector in the requested range");
  }
  build_block_tables(*sp, build_factored(*sp));
  count_blocks(*sp);
  rc = device_setup(*sp);
  if (rc) {
    qb_space_free(reinterpret_cast<qb_space*>(sp));
    return rc;
  }
  *out = reinterpret_cast<qb_space*>(sp);
  return QB_OK;
}

void qb_space_free(qb_space* space) {
  Space* sp = reinterpret_cast<Space*>(space);
  if (!sp) return;
  cudaFree(sp->d_arena);
  if (sp->own_obsf) cudaFree(sp->d_obsf);
  cudaFree(sp->d_hpsi);
  if (sp->capture_stream) cudaStreamDestroy(sp->capture_stream);
  delete sp;
}

int qb_space_info(const qb_space* space, int64_t* total_states, int* n_sectors, int64_t* max_dim) {
  const Space* sp = reinterpret_cast<const Space*>(space);
  if (!sp) return fail(QB_EINVAL, "space is NULL");
  if (total_states) *total_states = sp->secOff.back();
  if (n_sectors) *n_sectors = (int)sp->secN.size();
  if (max_dim) *max_dim = sp->maxDim;
  return QB_OK;
}

int qb_space_sectors(const qb_space* space, int* N, int* P, int64_t* dim, int64_t* offset) {
  const Space* sp = reinterpret_cast<const Space*>(space);
  if (!sp) return fail(QB_EINVAL, "space is NULL");
  for (size_t i = 0; i < sp->secN.size(); ++i) {
    if (N) N[i] = sp->secN[i];
    if (P) P[i] = sp->secP[i];
    if (dim) dim[i] = sp->secDim[i];
    if (offset) offset[i] = sp->secOff[i];
  }
  return QB_OK;
}

int qb_space_basis(const qb_space* space, int64_t first, int64_t count, int* d_occ, void* stream) {
  const Space* sp = reinterpret_cast<const Space*>(space);
  if (!sp) return fail(QB_EINVAL, "space is NULL");
  if (first < 0 || count < 0 || first + count > sp->secOff.back())
    return fail(QB_EINVAL, "ket range outside the space");
  if (count == 0) return QB_OK;
  if (!d_occ) return fail(QB_EINVAL, "d_occ is NULL");
  return launch_unrank(*sp, first, count, d_occ, stream);
}

int qb_space_rank(const qb_space* space, const int* d_occ, int64_t count, int64_t* d_index, void* stream) {
  const Space* sp = reinterpret_cast<const Space*>(space);
  if (!sp) return fail(QB_EINVAL, "space is NULL");
  if (count < 0) return fail(QB_EINVAL, "count < 0");
  if (count == 0) return QB_OK;
  if (!d_occ || !d_index) return fail(QB_EINVAL, "NULL device pointer");
  return launch_rank(*sp, d_occ, count, d_index, stream);
}

int qb_space_terms(const qb_space* space, int64_t* terms, int64_t* tuples, void* stream) {
  const Space* sp = reinterpret_cast<const Space*>(space);
  if (!sp || !terms) return fail(QB_EINVAL, "space and terms must be non-NULL");
  return launch_terms(*sp, terms, tuples, stream);
}

static int check_state_ptr(const void* p) {
  if (!p) return fail(QB_EINVAL, "state pointer is NULL");
  if (((uintptr_t)p) & 15) return fail(QB_EINVAL, "state pointer must be 16-byte aligned");
  return QB_OK;
}

int qb_init_number(qb_space* space, const int* occ, void* d_psi, void* stream) {
  Space* sp = reinterpret_cast<Space*>(space);
  if (!sp || !occ) return fail(QB_EINVAL, "space and occ must be non-NULL");
  int rc = check_state_ptr(d_psi);
  if (rc) return rc;
  int64_t k = host_rank(*sp, occ);
  if (k < 0) return fail(QB_EINVAL, "the occupation vector is not a ket of the space");
  return launch_number(*sp, k, d_psi, stream);
}

// table[i][v] = prefactor_i * zeta_i^v / sqrt(v!) for v = 0..nmax, as complex
static void amp_table(const Space& sp, const double* z, double scale, double mode_pref_log, std::vector<double>& tab,
                      bool coherent) {
  const int M = sp.M, V = sp.nmax + 1;
  tab.assign(2 * (size_t)M * V, 0.0);
  for (int i = 0; i < M; ++i) {
    cd zi = cd(z[2 * i], z[2 * i + 1]) * scale;
    double r = std::abs(zi), th = std::arg(zi);
    double pref = coherent ? -0.5 * r * r : 0.0;
    for (int v = 0; v < V; ++v) {
      double re = 0.0, im = 0.0;
      if (v == 0) {
        re = std::exp(pref);
      } else if (r > 0.0) {
        double lg = pref + v * std::log(r) - 0.5 * std::lgamma((double)v + 1.0);
        double mag = std::exp(lg);
        re = mag * std::cos(v * th);
        im = mag * std::sin(v * th);
      }
      tab[2 * ((size_t)i * V + v)] = re;
      tab[2 * ((size_t)i * V + v) + 1] = im;
    }
  }
  (void)mode_pref_log;
}

int qb_init_coherent(qb_space* space, const double* z, void* d_psi, double* kept_norm, void* stream) {
  Space* sp = reinterpret_cast<Space*>(space);
  if (!sp || !z) return fail(QB_EINVAL, "space and z must be non-NULL");
  int rc = check_state_ptr(d_psi);
  if (rc) return rc;
  for (int i = 0; i < 2 * sp->M; ++i)
    if (!std::isfinite(z[i])) return fail(QB_EINVAL, "z has a non-finite entry");
  std::vector<double> tab;
  amp_table(*sp, z, 1.0, 0.0, tab, true);
  double n2 = 0.0;
  rc = launch_init_table(*sp, tab.data(), -1, d_psi, &n2, stream);
  if (rc) return rc;
  if (!(n2 > 0.0)) return fail(QB_EINVAL, "the coherent state has no weight on the space");
  if (kept_norm) *kept_norm = n2;
  return launch_scale(*sp, d_psi, 1.0 / std::sqrt(n2), stream);
}

int qb_init_field_number(qb_space* space, const double* z, int n_tot, void* d_psi, void* stream) {
  Space* sp = reinterpret_cast<Space*>(space);
  if (!sp || !z) return fail(QB_EINVAL, "space and z must be non-NULL");
  int rc = check_state_ptr(d_psi);
  if (rc) return rc;
  double zz = 0.0;
  for (int i = 0; i < sp->M; ++i) {
    if (!std::isfinite(z[2 * i]) || !std::isfinite(z[2 * i + 1])) return fail(QB_EINVAL, "z has a non-finite entry");
    zz += z[2 * i] * z[2 * i] + z[2 * i + 1] * z[2 * i + 1];
  }
  if (!(zz > 0.0)) return fail(QB_EINVAL, "z must be nonzero");
  if (n_tot < sp->nmin || n_tot > sp->nmax) return fail(QB_EINVAL, "n_tot is outside the space");
  std::vector<double> tab;
  amp_table(*sp, z, 1.0 / std::sqrt(zz), 0.0, tab, false);
  // sqrt(n_tot!) folded into mode 0's table
  double pref = std::exp(0.5 * std::lgamma((double)n_tot + 1.0));
  for (int v = 0; v <= sp->nmax; ++v) {
    tab[2 * v] *= pref;
    tab[2 * v + 1] *= pref;
  }
  double n2 = 0.0;
  rc = launch_init_table(*sp, tab.data(), n_tot, d_psi, &n2, stream);
  if (rc) return rc;
  if (!(n2 > 0.0)) return fail(QB_EINVAL, "the field number state has no weight on the space");
  // exact normalisation is 1 by the multinomial theorem on the full sector set;
  // renormalise anyway so that a partial P list still yields a unit vector
  return launch_scale(*sp, d_psi, 1.0 / std::sqrt(n2), stream);
}

int64_t qb_workspace_bytes(const qb_space* space, int batch) {
  const Space* sp = reinterpret_cast<const Space*>(space);
  if (!sp || batch < 1) return -1;
  return workspace_bytes(*sp, batch);
}

int qb_hpsi(qb_space* space, const void* d_psi, void* d_out, void* stream) {
  Space* sp = reinterpret_cast<Space*>(space);
  if (!sp) return fail(QB_EINVAL, "space is NULL");
  int rc = check_state_ptr(d_psi);
  if (rc) return rc;
  rc = check_state_ptr(d_out);
  if (rc) return rc;
  if (d_psi == d_out) return fail(QB_EINVAL, "d_psi and d_out must differ");
  return launch_hpsi(*sp, d_psi, d_out, stream);
}

int qb_evolve(qb_space* space, void* d_psi, double dt, int64_t steps, void* d_work, void* stream) {
  double one = 1.0;
  return qb_evolve_batch(space, d_psi, 1, &one, dt, steps, d_work, stream);
}

int qb_evolve_batch(qb_space* space, void* d_psi, int batch, const double* scale, double dt, int64_t steps,
                    void* d_work, void* stream) {
  Space* sp = reinterpret_cast<Space*>(space);
  if (!sp || !scale) return fail(QB_EINVAL, "space and scale must be non-NULL");
  if (batch < 1 || batch > 8) return fail(QB_EINVAL, "batch must be in [1, 8]");
  if (steps < 0) return fail(QB_EINVAL, "steps < 0");
  if (!std::isfinite(dt)) return fail(QB_EINVAL, "dt is not finite");
  int rc = check_state_ptr(d_psi);
  if (rc) return rc;
  if (steps == 0) return QB_OK;
  rc = check_state_ptr(d_work);
  if (rc) return rc;
  for (int b = 0; b < batch; ++b)
    if (!std::isfinite(scale[b])) return fail(QB_EINVAL, "scale has a non-finite entry");
  return launch_rk4(*sp, d_psi, batch, scale, dt, steps, d_work, stream);
}

int qb_space_set_resident_max(qb_space* space, int resident_max_kets) {
  Space* sp = reinterpret_cast<Space*>(space);
  if (!sp) return fail(QB_EINVAL, "space is NULL");
  if (resident_max_kets < 0) return fail(QB_EINVAL, "resident_max_kets must be >= 0");
  sp->resident_max_kets = resident_max_kets;
  return QB_OK;
}

int qb_space_set_tile_shape(qb_space* space, int shape) {
  Space* sp = reinterpret_cast<Space*>(space);
  if (!sp) return fail(QB_EINVAL, "space is NULL");
  if (shape < 0 || shape >= QB_TILE_SHAPES) return fail(QB_EINVAL, "shape must be in [0, QB_TILE_SHAPES)");
  sp->tile_shape = shape;
  return QB_OK;
}

int qb_space_set_order(qb_space* space, int order) {
  Space* sp = reinterpret_cast<Space*>(space);
  if (!sp) return fail(QB_EINVAL, "space is NULL");
  if (order < 2 || order > 4) return fail(QB_EINVAL, "order must be 2, 3 or 4");
  sp->order = order;
  return QB_OK;
}

int qb_evolve_plain(qb_space* space, void* d_psi, double dt, int64_t steps, void* d_work, void* stream) {
  Space* sp = reinterpret_cast<Space*>(space);
  if (!sp) return fail(QB_EINVAL, "space is NULL");
  if (steps < 0) return fail(QB_EINVAL, "steps < 0");
  if (!std::isfinite(dt)) return fail(QB_EINVAL, "dt is not finite");
  int rc = check_state_ptr(d_psi);
  if (rc) return rc;
  if (steps == 0) return QB_OK;
  rc = check_state_ptr(d_work);
  if (rc) return rc;
  double one = 1.0;
  return launch_rk4(*sp, d_psi, 1, &one, dt, steps, d_work, stream, true);
}

int qb_observables(qb_space* space, const void* d_psi, qb_obs* out, void* stream) {
  Space* sp = reinterpret_cast<Space*>(space);
  if (!sp || !out) return fail(QB_EINVAL, "space and out must be non-NULL");
  int rc = check_state_ptr(d_psi);
  if (rc) return rc;
  const int M = sp->M;
  std::vector<double> raw(4 + 2 * M + 4 * (size_t)M * M, 0.0);
  rc = launch_moments(*sp, d_psi, raw.data(), stream);
  if (rc) return rc;
  if (!(raw[0] > 0.0)) return fail(QB_EINVAL, "the state has zero norm");
  derive(M, raw.data(), out);
  return QB_OK;
}

int qb_evolve_observe(qb_space* space, void* d_psi, double dt, int64_t steps, int obs_every, qb_obs* series,
                      void* d_work, void* stream) {
  if (obs_every < 1 || steps < 0 || steps % obs_every != 0)
    return fail(QB_EINVAL, "steps must be a non-negative multiple of obs_every >= 1");
  if (!series) return fail(QB_EINVAL, "series is NULL");
  int64_t nobs = steps / obs_every;
  int rc = qb_observables(space, d_psi, &series[0], stream);
  if (rc) return rc;
  series[0].t = 0.0;
  for (int64_t k = 1; k <= nobs; ++k) {
    rc = qb_evolve(space, d_psi, dt, obs_every, d_work, stream);
    if (rc) return rc;
    rc = qb_observables(space, d_psi, &series[k], stream);
    if (rc) return rc;
    series[k].t = (double)k * obs_every * dt;
  }
  return QB_OK;
}

int qb_breaktime(const double* values, int n, double dt_obs, double thr, double* t_br, int* flag) {
  if (!values || !t_br || !flag || n < 0) return fail(QB_EINVAL, "bad arguments");
  for (int k = 0; k < n; ++k) {
    if (values[k] >= thr) {
      if (k == 0) {
        *t_br = 0.0;
        *flag = QB_AT_START;
      } else {
        double f = (thr - values[k - 1]) / (values[k] - values[k - 1]);
        *t_br = ((double)(k - 1) + f) * dt_obs;
        *flag = QB_CROSSED;
      }
      return QB_OK;
    }
  }
  *t_br = NAN;
  *flag = QB_NOT_CROSSED;
  return QB_OK;
}

int qb_squeezing(const double* vminus, int n, double dt_obs, double thr, double* t_sqz, int* flag, double* v_min,
                 double* t_min) {
  if (!vminus || !t_sqz || !flag || !v_min || !t_min || n < 1 || !(dt_obs > 0.0))
    return fail(QB_EINVAL, "bad arguments");
  *t_sqz = NAN;
  *flag = QB_NOT_CROSSED;
  for (int k = 0; k < n; ++k) {
    if (vminus[k] <= thr) {
      if (k == 0) {
        *t_sqz = 0.0;
        *flag = QB_AT_START;
      } else {
        const double f = (vminus[k - 1] - thr) / (vminus[k - 1] - vminus[k]);
        *t_sqz = ((double)(k - 1) + f) * dt_obs;
        *flag = QB_CROSSED;
      }
      break;
    }
  }
  int kmin = 0;
  for (int k = 1; k < n; ++k)
    if (vminus[k] < vminus[kmin]) kmin = k;
  *v_min = vminus[kmin];
  *t_min = kmin * dt_obs;
  if (kmin > 0 && kmin < n - 1) {
    // vertex of the parabola through (-1, a), (0, b), (1, c) in units of dt_obs
    const double a = vminus[kmin - 1], b = vminus[kmin], c = vminus[kmin + 1];
    const double den = a - 2.0 * b + c;
    if (den > 0.0) {
      const double u = 0.5 * (a - c) / den;  // in [-1/2, 1/2] since b is the smallest
      *t_min = (kmin + u) * dt_obs;
      *v_min = b - 0.25 * (a - c) * u;
    }
  }
  return QB_OK;
}

int qb_interaction_per_occupation(const qb_model* model, const double* z, double* ntot_chi) {
  if (!model || !z || !ntot_chi) return fail(QB_EINVAL, "bad arguments");
  std::vector<double> w, Ls;
  int rc = prepare_model(model, w, Ls);
  if (rc) return rc;
  const int M = model->M;
  std::vector<cd> zz(M);
  double n = 0.0;
  for (int p = 0; p < M; ++p) {
    if (!std::isfinite(z[2 * p]) || !std::isfinite(z[2 * p + 1])) return fail(QB_EINVAL, "z has a non-finite entry");
    zz[p] = cd(z[2 * p], z[2 * p + 1]);
    n += std::norm(zz[p]);
  }
  if (!(n > 0.0)) return fail(QB_EINVAL, "z must be nonzero");
  cd acc = 0.0;
  for (int p = 0; p < M; ++p)
    for (int q = 0; q < M; ++q)
      for (int r = 0; r < M; ++r)
        for (int s = 0; s < M; ++s) {
          const size_t t = (((size_t)p * M + q) * M + r) * M + s;
          acc += cd(Ls[2 * t], Ls[2 * t + 1]) * std::conj(zz[p]) * std::conj(zz[q]) * zz[r] * zz[s];
        }
  *ntot_chi = acc.real() / n;
  return QB_OK;
}

int qb_fit(const double* x, const double* y, int n, int kind, double* c0, double* c1) {
  if (!x || !y || !c0 || !c1 || n < 2 || (kind != 0 && kind != 1)) return fail(QB_EINVAL, "bad arguments");
  double sx = 0.0, sy = 0.0, sxx = 0.0, sxy = 0.0;
  for (int k = 0; k < n; ++k) {
    if (!(x[k] > 0.0) || (kind == 0 && !(y[k] > 0.0))) return fail(QB_EINVAL, "the fit needs positive data");
    const double u = std::log(x[k]), v = kind == 0 ? std::log(y[k]) : y[k];
    sx += u;
    sy += v;
    sxx += u * u;
    sxy += u * v;
  }
  const double det = n * sxx - sx * sx;
  if (!(det > 0.0)) return fail(QB_EINVAL, "the fit needs two distinct x");
  const double slope = (n * sxy - sx * sy) / det, icpt = (sy - slope * sx) / n;
  *c1 = slope;
  *c0 = kind == 0 ? std::exp(icpt) : icpt;
  return QB_OK;
}

int qb_meanfield(const qb_model* model, const double* z0, double dt, int64_t steps, int every, double* traj) {
  if (!model || !model->w || !model->L || !z0 || !traj || every < 1 || steps < 0)
    return fail(QB_EINVAL, "bad arguments");
  const int M = model->M;
  if (M < 1 || M > QB_MAX_MODES) return fail(QB_EUNSUPPORTED, "M must be in [1, QB_MAX_MODES]");
  std::vector<cd> G((size_t)M * M * M * M);
  for (int k = 0; k < M; ++k)
    for (int q = 0; q < M; ++q)
      for (int r = 0; r < M; ++r)
        for (int s = 0; s < M; ++s) {
          size_t t1 = (((size_t)k * M + q) * M + r) * M + s, t2 = (((size_t)q * M + k) * M + r) * M + s;
          G[t1] = cd(model->L[2 * t1], model->L[2 * t1 + 1]) + cd(model->L[2 * t2], model->L[2 * t2 + 1]);
        }
  auto rhs = [&](const std::vector<cd>& a, std::vector<cd>& f) {
    for (int k = 0; k < M; ++k) {
      cd acc = model->w[k] * a[k];
      for (int q = 0; q < M; ++q)
        for (int r = 0; r < M; ++r)
          for (int s = 0; s < M; ++s) acc += G[(((size_t)k * M + q) * M + r) * M + s] * std::conj(a[q]) * a[r] * a[s];
      f[k] = cd(0, -1) * acc;
    }
  };
  std::vector<cd> a(M), k1(M), k2(M), k3(M), k4(M), u(M);
  for (int i = 0; i < M; ++i) a[i] = cd(z0[2 * i], z0[2 * i + 1]);
  int64_t row = 0;
  for (int i = 0; i < M; ++i) {
    traj[2 * i] = a[i].real();
    traj[2 * i + 1] = a[i].imag();
  }
  for (int64_t st = 1; st <= steps; ++st) {
    rhs(a, k1);
    for (int i = 0; i < M; ++i) u[i] = a[i] + 0.5 * dt * k1[i];
    rhs(u, k2);
    for (int i = 0; i < M; ++i) u[i] = a[i] + 0.5 * dt * k2[i];
    rhs(u, k3);
    for (int i = 0; i < M; ++i) u[i] = a[i] + dt * k3[i];
    rhs(u, k4);
    for (int i = 0; i < M; ++i) a[i] += dt / 6.0 * (k1[i] + 2.0 * k2[i] + 2.0 * k3[i] + k4[i]);
    if (st % every == 0) {
      ++row;
      for (int i = 0; i < M; ++i) {
        traj[2 * (row * M + i)] = a[i].real();
        traj[2 * (row * M + i) + 1] = a[i].imag();
      }
    }
  }
  return QB_OK;
}

}  // extern "C"
