// Internal structures shared by the host code (qb_host.cpp) and the CUDA
// kernels (qb_kernels.cu).  Not part of the public ABI (include/qb.h).
#pragma once
#include <array>
#include <cstdint>
#include <mutex>
#include <string>
#include <vector>

#include <cuda_runtime.h>

#include "../../include/qb.h"

namespace qb {

// Shifts of a suffix-state index are stored as unsigned bytes offset by this bias
// (a shift lies in [-4M, 5M) for M <= 16).
constexpr int kDeltaBias = 64;

// Spaces of more kets than these leave memory for the caller's vectors: the observables' copy
// of the state is allocated by the first call that needs it, and contact couplings are
// factored only where the vector of B_k f fits beside what a step needs without it.
constexpr int64_t kObsfKets = 1ll << 28;

// Polls of a grid barrier before its CTA gives up: a minute or so
constexpr uint32_t kWaitPolls = 1u << 27;

// 32-bit indices of kets and of entries of B_k f stay below this
constexpr uint32_t kNoIndex = 0xffff0000u;

// Everything a kernel needs to walk one space, passed by value.
//
// Ranking of a ket n within its sector (N, K), K = sum_i i n_i mod M (mode
// index momentum), in lexicographic order (n_0 most significant):
//   rank(n) = D - 1 - sum_{m=1}^{M-1} E_m(rem_m, krem_m),
//   rem_m = sum_{i>=m} n_i,  krem_m = sum_{i>=m} i n_i mod M,
//   E_m(rem, k) = cnt[m-1][rem-1][(k - (m-1)) mod M]  (0 for rem < 1),
// where cnt[m][n][k] counts the fillings of modes m..M-1 with n particles and
// index momentum k.  E is stored as E[m][rem + 2][kk] for kk in [0, 2M) with
// E[..][kk] = E_m(rem, kk mod M), so that shifting (rem, krem) by a term's
// (dc, dk mod M) is one integer add on the flat index:
//   idx(m, rem, krem) = (m * rem_w + rem + 2) * 2M + krem.
struct Tables {
  int M;
  int Q;         // momentum modulus of the tables: M (mod-M conservation) or (M-1) nmax + 1 (exact)
  int exact;     // 1: momentum conserved exactly (Q exceeds every momentum sum)
  int sm_from;   // first byte of the image the row kernels stage in shared memory (cnt, E stay global below it)
  int nmax;      // largest N of the space
  int rem_w;     // nmax + 5
  int n_ann;     // M(M+1)/2 unordered annihilation pairs (r <= s)
  int n_combo;   // (annihilation pair, creation pair) combinations, zero couplings included
  int is_complex;
  int blob_bytes;  // size of the shared-memory image
  // byte offsets of the sub-tables inside the image
  int o_cnt;     // uint32 [(M+1)][nmax+1][Q]
  int o_E;       // int32  [M][rem_w][2Q]
  int o_sqrt;    // double [nmax+3]            sqrt(k)
  int o_pq;      // uint32 [n_combo]           p | q<<8 | lo<<16 | hi<<24
  int o_G;       // double [n_combo][2]        conj(mult * L^sym_{pq;rs}) (re, im)
  int o_delta;   // uint8  [n_combo][16]       kDeltaBias + flat-index shift of the suffix state at mode m
                 //   (exact: int16 [n_combo][16], the shift itself)
  int o_ann;     // int32  [n_ann + 1]         first combo of annihilation pair a
  int o_pairidx; // uint8  [16][16]            pair index of (r <= s)
  int o_w;       // double [M]                 one-body w_p
  int o_gd;      // double [n_ann]             diagonal two-body coefficient mult_rs^2 L^sym_{rs;rs}
  const unsigned char* blob;  // device pointer to the image
  // sectors
  int n_sectors;
  const int64_t* sec_off;  // [n_sectors + 1]
  const int32_t* sec_N;    // [n_sectors]
  const int32_t* sec_K;    // [n_sectors] index momentum
  const int32_t* sec_of;   // [(nmax + 1) * Q] sector id of (N, K) or -1
  int64_t total;
  // ket weights w(n) = sqrt(N! / prod_m n_m!) = prod_m sqrt(C(rem_m, n_m)), rem_m the
  // particles in modes m..M-1: entry [rem * (nmax + 1) + k] = (sqrt(C(rem, k)), its inverse)
  const double2* wtab;
  // per particle number N: (2^-e_N, 2^e_N), e_N = round(log2(w_max(N)) / 2) with w_max(N)
  // the largest ket weight of N particles in M modes; the stages use w(n) 2^-e_N, which
  // keeps every weight of the sector within [2^-k, 2^k], k = log2(w_max) / 2 + 1/2.  A
  // constant per sector is a similarity inside each diagonal block of H, so the
  // weighted operator is unchanged; a power of two changes no rounding.
  const double2* wscale;
  // packed occupation vector of every ket (written with the diagonal): n_m in bits
  // [m * occ_bits, (m + 1) * occ_bits), occ_bits the bit length of nmax
  int occ_bits;
  const uint64_t* occ;  // [total]
  const double* wi;     // [total] 1 / w(n) of every ket (the centred ket weight; ket_weight)
  const double* wk;     // [total] w(n)
  // Block tables of the stage kernel (qb_block.cuh).  A block is the run of kets of a
  // sector that share the occupations of modes 0 .. P-1; its class (rem, kr) is the
  // particle number and index momentum of the other modes, whose fillings are numbered
  // class by class (rem, then kr; lexicographic within a class), S in all.  The terms are
  // grouped into records: one annihilation pair with its bk_kc partners, or (bk_kc = 0)
  // with up to four of them.
  int bk_kc;                // partners per pair where that is fixed (2 to 5), else 0
  int bk_P;                 // modes of the block prefix
  int bk_S;                 // fillings of the modes bk_P .. M-1 with up to nmax particles, and one number
                            //   left out after each class
  const uint32_t* fill;     // [total] number of the filling of every ket
  int bk_nrec;              // records
  float bk_share;           // share of the records that a ket takes part in, on average
  int bk_most;              // records that a ket takes part in, at most
  int bk_T;                 // term slots (a multiple of 4): record i holds [w i, w i + w), w = 2 for
                            //   bk_kc = 2, else 4; a fifth partner sits at 4 n_rec + i
  const uint32_t* rblk;     // [ceil(total / 32)] block of every 32nd ket
  const uint32_t* bk_base;  // [blocks][T] index in the state of the first ket of each slot's target block
  const uint2* bk_info;     // [n_rec] x: r mod 8 | terms << 4 | last record of its pair << 7 | first partner after
                            //   the pair << 8 | (r >= 8) << 15 | s mod 8 << 16 | (s >= 8) << 31; y: the float
                            //   2^23 + [r = s]
  const float2* bk_G;       // [T] real coupling (hi, lo); bk_Gi: imaginary
  const float2* bk_Gi;
  const uint32_t* bk_combo; // [T] combination of the slot, or 0xffffffff
  const int32_t* bk_psh;    // [M][T + 4] shift of the suffix index at mode m (a term conserves N and K: 0 for m = 0; 0 for unused slots)
  const int32_t* bk_EC;     // [rem_w][2Q] ranking-table rows of mode P plus the size of the class
  const int2* bk_cls;       // [nmax + 1][Q] (first filling, size) of each class
  const unsigned char* bk_map;  // [n_rec][S] place of the changed filling in its class, w 16-bit entries
  const uint16_t* bk_map5;      // [n_rec][S] of the fifth partner
  // Factored couplings (qb_factor.cuh): H_2 = sum_k lam_k B_k^dag B_k, B_k the sum of a_p a_q
  // over the ordered pairs of momentum class k (fa_on = 1).  B_k f lives on the lower kets, the
  // kets of two particles fewer; its entries of every (lower sector, class) whose raised
  // sector is held form one vector of fa_nG.  Annihilation records: a class with its pairs in
  // fa_pl groups of four (odd M, momentum mod M: fa_nt pairs, the pair p = q last), or
  // (fa_nt = 0) up to four pairs of a class.  Creation groups: four pairs (r, s) each.
  int fa_on, fa_nt, fa_pl, fa_nrec, fa_nc, fa_ng;
  int fa_every;                // 1: every class of every lower sector has its raised sector
  int fa_nlow;                 // lower sectors
  int64_t fa_low;              // lower kets
  int64_t fa_nG;
  const uint2* fa_rec;         // [fa_nrec] x: class | pairs << 8 | double the sum before pair (0-4; 7: never) << 12 |
                               //   last record of the class << 16
  const float2* fa_lam;        // [fa_nc] lam_k (hi, lo)
  const double* fa_lam64;      // [fa_nc] lam_k
  const uint32_t* fa_pqa;      // [fa_Ta] p | q << 8 of each annihilation slot
  const int32_t* fa_ka;        // [fa_Ta] class of each annihilation slot
  const int32_t* fa_kc;        // [fa_Tc] class of each creation slot
  const int32_t* fa_psa;       // [M][fa_Ta] shift of the suffix index when the slot's pair is added
  const int32_t* fa_psc;       // [M][fa_Tc] when it is taken away
  const uint4* fa_info;        // [fa_ng] mode selectors of four pairs, as bk_info's x
  const float4* fa_coef;       // [2 fa_ng] (2^23 + [r = s], 2 - [r = s]; 0 for an unused slot) of two pairs each
  const uint2* fa_mapa;        // [fa_nrec][fa_pl][S] places after adding the pairs
  const uint2* fa_mapc;        // [fa_ng][S] places after taking the pairs away
  const int32_t* fa_lowof;     // [nmax + 1][Q] lower sector of (N, K) or -1
  const int64_t* fa_lowoff;    // [fa_nlow + 1]
  const uint32_t* fa_goff;     // [fa_nlow][fa_nc] first entry of (lower sector, class), or kNoIndex
  const uint64_t* fa_occ;      // [fa_low] packed occupations of the lower kets
  const uint32_t* fa_fill;     // [fa_low] and the numbers of their fillings
  const uint32_t* fa_rblk;     // [ceil(fa_low / 32)] block of every 32nd lower ket
  const uint32_t* fa_basea;    // [lower blocks][fa_rowa] raised target blocks, then the classes' entries (qb_factor.cuh)
  const uint32_t* fa_basec;    // [blocks][fa_Tc] index in the vector of B_k f of the lowered target blocks
  const uint32_t* fa_perm;     // [ceil(fa_low / 32)] order of the rounds (qb_factor.cuh), or NULL
  // Moments by raised and lowered kets (qb_observe.cu), for spaces that hold every sector up
  // to nmax (mo_on): rows of 2 mo_w entries per block, the target blocks after a particle is
  // added to (taken from) each mode, and the places, mo_w / 4 groups of four modes.
  int mo_on, mo_w;
  int64_t mo_rows;             // kets of fewer than nmax particles
  const uint32_t* mo_base;     // [blocks][2 mo_w]
  const uint2* mo_map;         // [2][mo_w / 4][S]
  const uint32_t* mo_perm;     // [mo_rows / 32] order of the rounds
  const double* fa_wk;         // [fa_low] their ket weights, or NULL
};
// a row of fa_basea: the slots, the classes' entries, the mask of records with a held class
__host__ __device__ inline int fa_rowa(const Tables& t) { return t.fa_nrec * t.fa_pl * 4 + ((t.fa_nc + 4) & ~3); }
__host__ __device__ inline int fa_Ta(const Tables& t) { return t.fa_nrec * t.fa_pl * 4; }
__host__ __device__ inline int fa_Tc(const Tables& t) { return t.fa_ng * 4; }

// The (annihilation pair, creation pair) combinations of a space, pair by pair
struct Combos {
  std::vector<int> annR, annS, annStart;       // pairs (r <= s) and their first combos
  std::vector<uint32_t> pq;                    // p | q << 8 | lo << 16 | hi << 24
  std::vector<double> G;                       // coupling (re, im)
  std::vector<std::array<int, 16>> delta;      // shift of the suffix index at each mode
  unsigned char pairidx[16][16];
};

struct Space {
  int M = 0;
  int Q = 0;       // momentum modulus (Tables::Q)
  int exact = 0;   // momentum conserved exactly
  int nmax = 0, nmin = 0;
  std::vector<double> w;                  // [M]
  std::vector<double> Lsym;               // [M^4][2]
  std::vector<int> secN, secP, secK;      // per sector
  std::vector<int64_t> secDim, secOff;    // secOff has n_sectors + 1 entries
  std::vector<uint64_t> cnt;              // host copy of the fill counts
  std::vector<int> secOf;                 // [(nmax+1) * Q]
  std::vector<unsigned char> blob;        // host copy of the shared-memory image
  Combos combos;
  std::vector<unsigned char> bk;          // block tables but the maps and bases
  size_t bk_off[8] = {0};                 // byte offsets of info, G, Gi, psh, EC, cls, (6 unused) and combo in bk
  std::vector<unsigned char> fa;          // tables of the factored couplings but the maps and bases
  size_t fa_off[17] = {0};
  std::vector<int> lowN, lowK;            // lower sectors
  std::vector<int64_t> lowOff;
  bool low_held = false;                  // the lower kets are the space's first kets
  size_t bk_map_bytes = 0;
  int64_t maxDim = 0;
  std::vector<uint32_t> blkCnt;           // [P + 1][nmax + 1][Q] blocks of the fillings of modes m .. M-1
  std::vector<uint32_t> secBlk, lowBlk;   // first block of each sector (lower sector), and their number
  // device memory of the space: one allocation that holds every table (device_setup), the
  // pointers below and the tables' into it
  unsigned char* d_arena = nullptr;
  double* d_scratch = nullptr;  // reduction partials
  float4* d_diag = nullptr;     // per ket: one-body and two-body diagonal as double-float pairs
  float4* d_obsf = nullptr;     // double-float copy of the state being observed (qb_observables)
  bool own_obsf = false;        // an allocation of its own, made by the first call (kObsfKets)
  void* d_hpsi = nullptr;      // FP64 vector of B_k psi (qb_hpsi of a factored space), made by the first call
  std::mutex hpsi_mu;          // held by the call that uses it
  int64_t scratch_doubles = 0;
  Tables t{};
  cudaStream_t capture_stream = nullptr;  // private stream on which RK4 chunks are captured into graphs
  int resident_max_kets = 1024;           // spaces whose sectors are all up to this size run shared-memory resident
  int order = 4;                          // Taylor order of a time step (4: RK4)
  uint32_t wait_polls = kWaitPolls;       // of a cooperative launch's CTA at a barrier
  int tile_shape = 0;                     // tile shape of the single-state stage kernel (qb_stage.cuh)
  int device = 0;
  int grid_hpsi = 0;  // persistent grid sizes per kernel family
};

// error handling
void set_error(const std::string& msg);
int fail(int code, const std::string& msg);
// reads the space's device status word (clearing it): QB_EINTERNAL if a device-side
// check failed since the last read
int check_status(const Space& s, cudaStream_t st);

// Raw moments of one state (doubles): [0] norm, [1] <N> norm, [2] <H> norm, [3] unused,
// then <a_i> [M], <a_i^dag a_j> [M*M], <a_i a_j> [M*M] as (re, im) pairs.
__host__ __device__ inline int nmoments(int M) { return 4 + 2 * M + 4 * M * M; }
// Columns of the per-CTA partials of the observables' first pass: norm, <N>, <n_i> [M].
__host__ __device__ inline int nprep(int M) { return M + 2; }

// Scratch layout of a space (doubles), sized at set-up for the largest persistent grid
// G = SMs * 16:  status word (first half of [0, 1)), counter and status of the cooperative
// launch ([1, 2)) | moment sums [nmom] | <H> sum [2] | first-pass sums [nprep]
// (these, the first finals_doubles, come back in one copy) | moment partials [G nmom] |
// bilinear / <H> partials [(M + 1) G] | first-pass partials [nprep G] | amplitude table
// [2 M (nmax + 1)] | initial-state norm [2]
// (even, as G is: the amplitude table is read as pairs)
inline int64_t finals_doubles(int M) { return (2 + nmoments(M) + 2 + nprep(M) + 1) & ~1; }
inline int64_t scratch_doubles_for(int M, int nmax, int64_t G) {
  return finals_doubles(M) + G * nmoments(M) + (int64_t)(M + 1) * G + G * nprep(M) + 2 * (int64_t)M * (nmax + 1) + 2;
}
inline int64_t max_grid_of(const Space& s) { return s.scratch_doubles > 0 ? (int64_t)s.grid_hpsi : 0; }
inline double* final_area(const Space& s) { return s.d_scratch + 2; }
inline double* dot_final(const Space& s) { return final_area(s) + nmoments(s.M); }
inline double* prep_final(const Space& s) { return dot_final(s) + 2; }
inline double* partial_area(const Space& s) { return s.d_scratch + finals_doubles(s.M); }
inline double* dot_area(const Space& s) { return partial_area(s) + max_grid_of(s) * nmoments(s.M); }
inline double* prep_area(const Space& s) { return dot_area(s) + (int64_t)(s.M + 1) * max_grid_of(s); }
inline double* table_area(const Space& s) { return prep_area(s) + max_grid_of(s) * nprep(s.M); }
inline double* init_final(const Space& s) { return table_area(s) + 2 * (size_t)s.M * (s.nmax + 1); }

// launchers (qb_kernels.cu); all return a QB_* status
int launch_hpsi(Space& s, const void* d_v, void* d_out, void* stream);
int launch_hpsi_rows(const Space& s, const void* d_v, void* d_out, cudaStream_t st);  // thread per row, no tables of blocks
int launch_rk4(Space& s, void* d_psi, int batch, const double* scale, double dt, int64_t steps, void* d_work,
               void* stream, bool plain = false);
int launch_unrank(const Space& s, int64_t first, int64_t count, int* d_occ, void* stream);
int launch_rank(const Space& s, const int* d_occ, int64_t count, int64_t* d_index, void* stream);
int launch_terms(const Space& s, int64_t* terms, int64_t* tuples, void* stream);
int launch_init_table(const Space& s, const double* table_host, int only_N, void* d_psi, double* norm2,
                      void* stream);
int launch_scale(const Space& s, void* d_psi, double factor, void* stream);
int launch_number(const Space& s, int64_t index, void* d_psi, void* stream);
// raw moments: out[0]=norm, out[1]=<N>, out[2]=<H>, then a[M], Mij[M*M], aa[M*M] complex
int launch_moments(Space& s, const void* d_psi, double* out_host, void* stream);
// d_acc[2e], d_acc[2e + 1] += weight * <bra, O_e ket> (re, im) for the two-body operators
// O_e = a_a1^dag a_a2^dag a_c1 a_c2 listed in d_tb[e] = a1 | a2 << 8 | c1 << 16 | c2 << 24;
// bra and ket are weighted double-float vectors of the space (as the stage kernels hold them)
int launch_tb_bilinear(Space& s, const float4* bra, const float4* ket, const int* d_tb, int n_tb, double weight,
                       double* d_acc, void* stream);
// The same by blocks of kets, for spaces with the direct stage tables (fa_on = 0): tb_columns
// gives each operator's column of the partial sums, which the launch takes as d_tb
std::vector<int> tb_columns(const Space& s, const std::vector<int>& ops);
int launch_tb_blocks(const Space& s, const float4* bra, const float4* ket, const int* cols, int n_ops, double weight,
                     double* acc, cudaStream_t st);
int64_t workspace_bytes(const Space& s, int batch);
int side_by_side(const Space& s, int batch);  // members of a sweep with a vector of B_k f each
// psi [B][total] -> double-float copy in the weighted basis f = psi / w(n) (the stages' basis)
int launch_to_dfw(const Space& s, const void* psi, void* psif, int B, void* stream);
// observables of Sec. II C-E from the raw moments (host)
void derive(int M, const double* raw, qb_obs* out);
// log2 of the largest ket weight sqrt(N! / prod_m n_m!) over all occupations of N
// particles in M modes (the most even one), and the largest log2 weight a space may
// reach: the stage vectors hold psi / w as fp32 pairs, so the centred weights
// w 2^-e_N must stay within 2^+-80 (qb_sector_build refuses deeper spaces)
double log2_max_ket_weight(int M, int N);
constexpr double kMaxLog2KetWeight = 160.0;
int device_setup(Space& s);

}  // namespace qb
