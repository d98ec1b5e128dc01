// Sigma vector and environment updates on the tensor cores (tcgen05, BF16 operands, FP32
// accumulation).  The sigma is the same two-stage contraction as the FP64 plan:
//   stage 1: X_beta^T[qr, ql'] = sum_{n2'} Rt_beta^{n2 n2'}[qr, qr'] psi[ql', n1', n2', qr']^T
//   stage 2: sigma[ql, qr]   += sum_{beta, n1'} Lt_beta^{n1 n1'}[ql, ql'] X_beta^T[qr, ql']^T
// with every operand stored as 1 to 3 BF16 slices (x = s0 + s1 + s2, each the
// BF16 rounding of the remainder).  With 3 slices the products s_i t_j with
// i + j <= 2 are summed (6 tensor-core products), which carries the operands
// to about 2^-24 relative accuracy; with 1 slice it is a single BF16 pass.
// Coefficients +-1 of the W-contracted operators become the negate bit of the
// instruction descriptor; other coefficients are folded into a scaled copy.
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <exception>
#include <future>
#include <iterator>
#include <limits>
#include <map>
#include <numeric>
#include <unordered_map>

#include "engine.hpp"
#include "kernels_tc.hpp"
#include "kernels_tma.hpp"

namespace gbdmrg {

namespace {

inline int pad8(int x) { return (x + 7) & ~7; }

// FP64 block -> nsl BF16 slices; writes wcols columns per row (the block's columns
// and its zero padding), rows ldd elements apart in the destination
struct ConvJob {
  const double* src;
  __nv_bfloat16* dst;
  long slice_stride;
  int rows, cols, lds, ldd, nsl;
  double scale;
  int wcols;
};

// Elements of a job spread over the grid (32-bit division when the job has fewer than
// 2^31 elements, as every job of these layouts has).  The FP64 value y is split once into
// a + lo (two FP32 values, a = fl32(y), lo = fl32(y - a)), and the BF16 slices are taken
// from a by exact FP32 subtractions, lo entering the last slice: two FP64 operations per
// element instead of several per slice (the FP64 units of this GPU issue at a small
// fraction of the FP32 rate).  The slices carry y to ~2^-25 relative for three slices,
// as a direct FP64 splitting does.
__device__ __forceinline__ void conv_element(const ConvJob& jb, long i, int j) {
  const double y = j < jb.cols ? jb.scale * jb.src[i * jb.lds + j] : 0.0;
  float a = __double2float_rn(y);
  const float lo = jb.nsl > 1 ? __double2float_rn(y - (double)a) : 0.0f;
  __nv_bfloat16* d = jb.dst + i * jb.ldd + j;
  for (int sl = 0; sl < jb.nsl; ++sl) {
    const __nv_bfloat16 h = __float2bfloat16_rn(sl + 1 == jb.nsl ? a + lo : a);
    d[(long)sl * jb.slice_stride] = h;
    a -= __bfloat162float(h);
  }
}

__global__ void conv_kernel(const ConvJob* __restrict__ jobs) {
  const ConvJob jb = jobs[blockIdx.y];
  const long n = (long)jb.rows * jb.wcols;
  if (n < (1L << 31)) {
    const unsigned w = (unsigned)jb.wcols;
    for (unsigned e = blockIdx.x * blockDim.x + threadIdx.x; e < (unsigned)n; e += gridDim.x * blockDim.x) {
      const unsigned i = e / w;
      conv_element(jb, (long)i, (int)(e - i * w));
    }
  } else {
    for (long e = (long)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += (long)gridDim.x * blockDim.x)
      conv_element(jb, e / jb.wcols, (int)(e % jb.wcols));
  }
}

// FP64 block -> nsl BF16 slices in the column-group layout of the TMA-staged matrices (8
// columns of consecutive rows contiguous): element (i, j) of slice s goes to
// dst[s * slice_stride + (j / 8) * group + i * 8 + j % 8], columns [cols, wcols) are zero
// (wcols a multiple of 8).
struct GroupJob {
  const double* src;
  __nv_bfloat16* dst;
  long slice_stride, group;
  int rows, cols, lds, wcols;
  double scale;
};

// Memory-bound (8 bytes read, 2 written per slice and element): a thread takes 8 columns
// of one row, 64 contiguous bytes of the source, and writes 16 bytes per slice; consecutive
// threads take consecutive rows, so a warp writes 512 contiguous bytes.  Each value is split
// as in conv_element.  src is read `shift` elements further than the job says (the jobs of
// psi are made for one vector and serve any).
template <int NSL>
__global__ void conv_groups_kernel(const GroupJob* __restrict__ jobs, long shift) {
  const GroupJob jb = jobs[blockIdx.y];
  const int ng = jb.wcols >> 3;
  const unsigned n = (unsigned)jb.rows * (unsigned)ng;
  for (unsigned e = blockIdx.x * blockDim.x + threadIdx.x; e < n; e += gridDim.x * blockDim.x) {
    const int q = (int)(e / (unsigned)jb.rows), i = (int)(e - (unsigned)q * (unsigned)jb.rows);
    const double* s = jb.src + shift + (long)i * jb.lds + q * 8;
    const int nc = jb.cols - q * 8;
    uint32_t w[NSL][4];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const double y = u < nc ? jb.scale * s[u] : 0.0;
      float a = __double2float_rn(y);
      const float lo = NSL > 1 ? __double2float_rn(y - (double)a) : 0.0f;
#pragma unroll
      for (int sl = 0; sl < NSL; ++sl) {
        const __nv_bfloat16 h = __float2bfloat16_rn(sl + 1 == NSL ? a + lo : a);
        const uint32_t b = (uint32_t)__bfloat16_as_ushort(h);
        w[sl][u / 2] = (u & 1) ? (w[sl][u / 2] | (b << 16)) : b;
        a -= __bfloat162float(h);
      }
    }
    __nv_bfloat16* d = jb.dst + (long)q * jb.group + (long)i * 8;
#pragma unroll
    for (int sl = 0; sl < NSL; ++sl)
      *reinterpret_cast<uint4*>(d + sl * jb.slice_stride) = make_uint4(w[sl][0], w[sl][1], w[sl][2], w[sl][3]);
  }
}

// transposed gather FP32 -> FP64: dst[i * cols + j] = src[j * lds + i]
struct UnconvJob {
  const float* src;
  double* dst;
  int rows, cols, lds;
};

// dst is written `shift` elements further than the job says
__global__ void unconv_kernel(const UnconvJob* __restrict__ jobs, long shift) {
  const UnconvJob jb = jobs[blockIdx.y];
  const long n = (long)jb.rows * jb.cols;
  for (long e = (long)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += (long)gridDim.x * blockDim.x) {
    const int i = (int)(e / jb.cols), j = (int)(e % jb.cols);
    jb.dst[shift + e] = (double)jb.src[(long)j * jb.lds + i];
  }
}

// blocks per job of the per-job copy kernels (blockIdx.y = job): with many jobs one block
// each (its threads stride over the job), so that no launch holds thousands of idle
// blocks sized for its largest job; with few jobs enough blocks for the largest
static long job_blocks(int njobs, long maxel) {
  if (njobs >= 1024) return 1;
  return std::min<long>(std::max<long>(1, (maxel + 255) / 256), 64);
}

void launch_unconv(const UnconvJob* jobs, int njobs, long maxel, cudaStream_t s, long shift = 0) {
  for (int o0 = 0; o0 < njobs; o0 += 65535) {
    int no = std::min(65535, njobs - o0);
    const long g = job_blocks(njobs, maxel);
    unconv_kernel<<<dim3((unsigned)g, no), 256, 0, s>>>(jobs + o0, shift);
    count_launches(1);
  }
  cuda_check(cudaGetLastError(), "unconv launch");
}

// zero n elements at p + s * stride + r * pitch for every slice s < nsl and r < reps
struct ZeroJob {
  __nv_bfloat16* p;
  long n, stride;
  int nsl;
  int reps = 1;
  long pitch = 0;
};

__global__ void zero_kernel(const ZeroJob* __restrict__ jobs) {
  const ZeroJob jb = jobs[blockIdx.y];
  const __nv_bfloat16 z = __float2bfloat16_rn(0.0f);
  for (int sl = 0; sl < jb.nsl; ++sl)
    for (int r = 0; r < jb.reps; ++r)
      for (long e = (long)blockIdx.x * blockDim.x + threadIdx.x; e < jb.n; e += (long)gridDim.x * blockDim.x)
        jb.p[sl * jb.stride + r * jb.pitch + e] = z;
}

void launch_zero(const ZeroJob* jobs, int njobs, long maxel, cudaStream_t s) {
  for (int o0 = 0; o0 < njobs; o0 += 65535) {
    int no = std::min(65535, njobs - o0);
    const long g = job_blocks(njobs, maxel);
    zero_kernel<<<dim3((unsigned)g, no), 256, 0, s>>>(jobs + o0);
    count_launches(1);
  }
  cuda_check(cudaGetLastError(), "zero launch");
}

void launch_conv(const DArr<ConvJob>& jobs, int njobs, long maxel, cudaStream_t s) {
  for (int o0 = 0; o0 < njobs; o0 += 65535) {
    int no = std::min(65535, njobs - o0);
    const long g = job_blocks(njobs, maxel);
    conv_kernel<<<dim3((unsigned)g, no), 256, 0, s>>>(jobs.p + o0);
    count_launches(1);
  }
  cuda_check(cudaGetLastError(), "conv launch");
}

void launch_conv_groups(const DArr<GroupJob>& jobs, int njobs, int nsl, long maxel, cudaStream_t s, long shift = 0) {
  for (int o0 = 0; o0 < njobs; o0 += 65535) {
    const int no = std::min(65535, njobs - o0);
    const dim3 g((unsigned)job_blocks(njobs, maxel / 8), no);
    const GroupJob* j = jobs.p + o0;
    if (nsl == 1)
      conv_groups_kernel<1><<<g, 256, 0, s>>>(j, shift);
    else if (nsl == 2)
      conv_groups_kernel<2><<<g, 256, 0, s>>>(j, shift);
    else
      conv_groups_kernel<3><<<g, 256, 0, s>>>(j, shift);
    count_launches(1);
  }
  cuda_check(cudaGetLastError(), "conv launch");
}

struct TcBuilder {
  std::vector<TcTile> tiles;
  std::vector<TcTask> tasks;
  std::vector<TcTerm> terms;
  void begin(const TcTask& t) {
    tasks.push_back(t);
    tasks.back().t0 = tasks.back().t1 = (int)terms.size();
  }
  void term(const __nv_bfloat16* A, long sA, int lda, const __nv_bfloat16* B, long sB, int ldb, int k, bool neg,
            int nsl) {
    if (k <= 0) return;
    terms.push_back({A, B, sA, sB, lda, ldb, k, neg ? 1 : 0, nsl});
    tasks.back().t1 = (int)terms.size();
  }
  bool end() {
    TcTask& t = tasks.back();
    if (t.t1 == t.t0) { tasks.pop_back(); return false; }
    const int idx = (int)tasks.size() - 1;
    for (int r0 = 0; r0 < t.m; r0 += TC_TILE_M)
      for (int c0 = 0; c0 < t.n; c0 += TC_TILE_N) tiles.push_back({idx, r0, c0});
    return true;
  }
};

}  // namespace

// padded BF16 layout of one operator class: per-block offsets (elements)
static std::vector<long> padded_offsets(const OpLayout& L, long* total) {
  std::vector<long> off(L.blocks.size());
  long t = 0;
  for (size_t b = 0; b < L.blocks.size(); ++b) {
    off[b] = t;
    t += (long)L.blocks[b].rows * pad8(L.blocks[b].cols);
  }
  *total = t;
  return off;
}

// ---------------------------------------------------------------- TMA-staged single-pass plan

// H_eff.psi in one BF16 pass with both stages as TMA-staged grouped GEMMs over a few
// large matrices (one tensor map each):
//   stage 1, per input group g': X_g'^T = A1_g' Psi_g'^T, where A1_g' stacks, for every
//     bond state beta and every (n2, qr) column block of the output group g = g' + dQ_beta,
//     the row block [Rt_beta^{n2 n2'}[qr, qr'] over the column blocks (n2', qr') of g'];
//     row blocks with the same pattern of non-zero site blocks n2' are stacked together,
//     and a tile multiplies only the K blocks of its pattern (no product with an absent
//     site block).  Each output row goes through a row map to its place in X_g'^T, whose
//     rows are, per beta, the column blocks of g in the row order of sigma^T_g.
//   stage 2, per output block: sigma^T_g[rows, (ql, n1)] += sum_{beta, n1'}
//     X_g'^T[beta rows, (ql', n1')] Lt_beta^{n1 n1'}[ql, ql']^T, a long contraction over
//     the operator terms (the paper's sum over left-right terms, Eq. Hpartition), cut
//     into parts that add with FP32 vector reductions.
// Every block is padded to 16 rows and columns with zeros, so a K step of 16 never
// mixes two blocks and padding contributes exact zeros.
struct TmaPlan {
  int precision = 4;  // the context's precision when the plan was built
  int nsl = 1;  // BF16 slices per operand (1: one pass; 2 or 3: slice products i + j < nsl)
  DArr<__nv_bfloat16> psi_b, a1, xt, lmir;
  DArr<float> sig_t;
  long sig_total = 0;
  DArr<GroupJob> psi_jobs, a1_jobs, l_jobs;
  int n_psi_jobs = 0, n_a1_jobs = 0, n_l_jobs = 0;
  long psi_maxel = 0, a1_maxel = 0, l_maxel = 0;
  DArr<UnconvJob> sig_jobs;
  int n_sig_jobs = 0;
  long sig_maxel = 0;
  DArr<CUtensorMap> maps;
  DArr<long> rowmap;
  // device copies of a launch's copy lists
  struct Lists {
    DArr<int> cta_stage, sorder, tpiece0;
    DArr<long> sfirst;
    DArr<TmStage> stages;
    DArr<TmPiece> pieces;
    int grid = 0, slots = 0, slot_bytes = 0;
    long total = 0;
    // the stage counts on the host (reduce mode: sets the tiles' stages and segments,
    // so it comes before the tiles are uploaded); throws on a malformed term
    void plan(int mode, int nsl, std::vector<TmTile>& tiles, const std::vector<TmTerm>& terms, cudaStream_t s) {
      TmListPlan lp;
      if (!tma_plan_lists(mode, nsl, tiles, terms, lp)) throw Error(ST_ECUDA, "internal: malformed TMA term list");
      grid = lp.grid;
      slots = lp.slots;
      slot_bytes = lp.slot_bytes;
      total = lp.total;
      cta_stage.upload(lp.cta_stage, s);
      sorder.upload(lp.sorder, s);
      sfirst.upload(lp.sfirst, s);
      tpiece0.upload(lp.tpiece0, s);
      stages.alloc((size_t)std::max<long>(lp.total, 1), s);
      pieces.alloc((size_t)std::max<long>(lp.total, 1) * tma_pieces(mode, nsl), s);
    }
    // the lists themselves, on the device, from the uploaded tiles and terms
    void fill(int mode, int nsl, const TmTile* d_tiles, int ntiles, const TmTerm* d_terms, cudaStream_t s) {
      cuda_check(launch_fill_lists(mode, nsl, d_tiles, ntiles, d_terms, tpiece0.p, sorder.p, sfirst.p, total, stages.p,
                                   pieces.p, s),
                 "list fill");
    }
    TmListsDev dev() const { return {grid, slots, slot_bytes, cta_stage.p, stages.p, pieces.p}; }
  };
  struct Chunk {
    DArr<TmTile> t1, t2;
    DArr<TmTerm> m1, m2;
    Lists l1, l2;
    int n1 = 0, n2 = 0;
    DArr<ZeroJob> z;
    int nz = 0;
    long zmax = 0;
    // the chunk's stacked right operators, where not all of them are held (n_a1_jobs == 0)
    DArr<GroupJob> a1;
    int n_a1 = 0;
    long a1_maxel = 0;
    // host copies, kept when the plan may be fused into a batched launch
    std::vector<TmTile> ht1, ht2;
    std::vector<TmTerm> hm1, hm2;
    std::vector<ZeroJob> hz;
    std::vector<GroupJob> ha1;
  };
  std::vector<Chunk> chunks;
  bool host_copies = false;
  std::vector<CUtensorMap> hmaps;
  std::vector<long> hrowmap;
  std::vector<GroupJob> h_psi_jobs;
  std::vector<UnconvJob> h_sig_jobs;
  DArr<int> err;
  double stats[9] = {0, 0, 0, 0, 0, 0, 0, 0, 0};
};

void tma_plan_free(TmaPlan* p) { delete p; }

void tma_plan_stats(const SigmaPlan& plan, double* out) {
  // (statistics are reported for precisions 4-6)
  for (int i = 0; i < 9; ++i) out[i] = plan.tm && plan.tm->precision >= 4 ? plan.tm->stats[i] : 0.0;
}

namespace {
inline int pad16(int x) { return (x + 15) & ~15; }
}  // namespace

// conversion jobs must write inside their destination buffer, in whole 16-byte groups
static void check_group_jobs(const std::vector<GroupJob>& jobs, int nsl, const DArr<__nv_bfloat16>& buf) {
  for (const GroupJob& j : jobs)
    if (j.rows < 1 || j.wcols < j.cols || j.wcols % 8 || (long)j.rows * (j.wcols / 8) >= (1L << 31) || j.dst < buf.p ||
        (j.dst - buf.p) % 8 || j.group % 8 || j.slice_stride % 8 ||
        j.dst + (nsl - 1) * j.slice_stride + (j.wcols / 8 - 1) * j.group + (long)j.rows * 8 > buf.p + buf.n)
      throw Error(ST_ECUDA, "internal: conversion job outside its buffer");
}

// longest tiles first (static round-robin over the persistent CTAs); tiles of equal
// length keep their order, so the N tiles of one row tile stay adjacent
static void longest_first(std::vector<TmTile>& t, const std::vector<TmTerm>& m) {
  // (a counting sort: the lengths are small whole numbers)
  std::vector<int> len(t.size());
  int top = 0;
  for (size_t i = 0; i < t.size(); ++i) {
    long ks = 0;
    for (int j = t[i].t0; j < t[i].t1; ++j) ks += (m[j].k + 63) / 64;
    len[i] = (int)std::min<long>(ks, 1 << 20);
    top = std::max(top, len[i]);
  }
  std::vector<size_t> at((size_t)top + 2, 0);  // tiles longer than the index
  for (int l : len) ++at[(size_t)(top - l) + 1];
  for (size_t l = 1; l < at.size(); ++l) at[l] += at[l - 1];
  std::vector<TmTile> out(t.size());
  for (size_t i = 0; i < t.size(); ++i) out[at[(size_t)(top - len[i])]++] = t[i];
  t.swap(out);
}

// The lists are made group by group on the host threads: K=24, M=512, three slices 18 ms, 38 ms in
// one thread.
void build_tma_plan(Context& c, Tilde& lt, Tilde& rt, int k, SigmaPlan& plan, int nsl) {
  const auto& mid = c.mpo.bonds[k + 1];
  Env& Lenv = *lt.env;
  Env& Renv = *rt.env;
  const Bond& Lb = Lenv.bond;
  const Bond& Rb = Renv.bond;
  const PsiLayout& P = plan.psi;
  auto* tp = new TmaPlan();
  plan.tm.reset(tp);
  if (nsl < 1 || nsl > 3) throw Error(ST_EINVAL, "TMA plan: 1 to 3 slices");
  tp->nsl = nsl;
  tp->precision = c.precision;
  // counted beside the work lists
  std::future<double> flops = std::async(std::launch::async | std::launch::deferred,
                                         [&] { return count_sigma_flops(c.mpo, k, Lb, Rb); });
  tp->host_copies = c.keep_host_plans && c.precision <= 3;  // what a batch takes
  const int nL = Lb.nsec(), nR = Rb.nsec();
  const int nmid = (int)mid.size();
  // slice pairs (i, j), i + j < nsl, multiplied per piece
  const int npair = nsl == 1 ? 1 : nsl == 2 ? 3 : 6;
  // ---- groups of the cut: rows (ql, n1) and columns (n2, qr), blocks padded to 16
  std::map<std::pair<int, int>, int> gidx;
  std::vector<std::pair<int, int>> gq;
  std::vector<std::vector<std::array<int, 3>>> grow, gcol;  // (ql, n1, off), (n2, qr, off)
  std::vector<int> gR, gC;
  {
    std::map<std::pair<int, int>, std::pair<std::vector<std::array<int, 3>>, std::vector<std::array<int, 3>>>> tmp;
    for (int ql = 0; ql < nL; ++ql)
      for (int n1 = 0; n1 < 4; ++n1) tmp[{Lb.qa[ql] + LQA[n1], Lb.qb[ql] + LQB[n1]}].first.push_back({ql, n1, 0});
    for (int qr = 0; qr < nR; ++qr)
      for (int n2 = 0; n2 < 4; ++n2) tmp[{Rb.qa[qr] - LQA[n2], Rb.qb[qr] - LQB[n2]}].second.push_back({n2, qr, 0});
    for (auto& kv : tmp) {
      if (kv.second.first.empty() || kv.second.second.empty()) continue;
      gidx[kv.first] = (int)gq.size();
      gq.push_back(kv.first);
      auto rows = kv.second.first, cols = kv.second.second;
      int R = 0, C = 0;
      for (auto& r : rows) { r[2] = R; R += pad16(Lb.dim[r[0]]); }
      for (auto& cc : cols) { cc[2] = C; C += pad16(Rb.dim[cc[1]]); }
      grow.push_back(rows);
      gcol.push_back(cols);
      gR.push_back(R);
      gC.push_back(C);
    }
  }
  const int ng = (int)gq.size();
  // (group, offset, index of the block in its group) of every row block (ql, n1) and
  // column block (n2, qr)
  std::vector<std::array<int, 3>> rpos((size_t)nL * 4, {-1, 0, -1}), cpos((size_t)nR * 4, {-1, 0, -1});
  for (int g = 0; g < ng; ++g) {
    for (size_t i = 0; i < grow[g].size(); ++i) rpos[grow[g][i][0] * 4 + grow[g][i][1]] = {g, grow[g][i][2], (int)i};
    for (size_t i = 0; i < gcol[g].size(); ++i) cpos[gcol[g][i][1] * 4 + gcol[g][i][0]] = {g, gcol[g][i][2], (int)i};
  }
  auto group_of = [&](int a, int b) {
    auto it = gidx.find({a, b});
    return it == gidx.end() ? -1 : it->second;
  };
  // output group of bond state beta for input group g' (-1: none)
  std::vector<int> gout((size_t)nmid * ng, -1);
  // input group g' = g - dQ_beta of bond state beta for output group g (-1: none)
  std::vector<int> gin((size_t)nmid * ng, -1);
  std::map<std::pair<int, int>, int> dq_first;  // quantum-number change -> the first bond state with it
  for (int beta = 0; beta < nmid; ++beta) {
    int* go = gout.data() + (size_t)beta * ng;
    int* gi = gin.data() + (size_t)beta * ng;
    const int first = dq_first.emplace(std::make_pair(mid[beta].dna, mid[beta].dnb), beta).first->second;
    if (first != beta) {
      std::copy_n(gout.data() + (size_t)first * ng, ng, go);
      std::copy_n(gin.data() + (size_t)first * ng, ng, gi);
      continue;
    }
    for (int g = 0; g < ng; ++g) {
      go[g] = group_of(gq[g].first + mid[beta].dna, gq[g].second + mid[beta].dnb);
      gi[g] = group_of(gq[g].first - mid[beta].dna, gq[g].second - mid[beta].dnb);
    }
  }
  // ---- Psi_g (BF16, R_g x C_g) and sigma^T_g (FP32, C_g x R_g)
  std::vector<long> goff(ng), sgoff(ng);
  long ptot = 0, stot = 0;
  for (int g = 0; g < ng; ++g) {
    goff[g] = ptot;
    ptot += (long)gR[g] * gC[g];
    sgoff[g] = stot;
    stot += (long)gC[g] * gR[g];
  }
  tp->psi_b.alloc(std::max<long>(ptot, 8) * nsl, c.stream);
  cuda_check(cudaMemsetAsync(tp->psi_b.p, 0, tp->psi_b.n * sizeof(__nv_bfloat16), c.stream), "memset");
  tp->sig_total = std::max<long>(stot, 4);
  tp->sig_t.alloc(tp->sig_total, c.stream);
  {
    std::vector<GroupJob> pj;
    std::vector<UnconvJob> sj;
    for (size_t b = 0; b < P.blocks.size(); ++b) {
      const Block& B = P.blocks[b];
      const auto rp = rpos[B.rs * 4 + P.b1[b]];
      const auto cp = cpos[B.cs * 4 + P.b2[b]];
      if (rp[0] < 0 || rp[0] != cp[0]) throw Error(ST_ECUDA, "internal: psi block outside its group");
      const int g = rp[0];
      // Psi_g: gR rows x gC columns in column groups of 8
      pj.push_back({plan.in.p + B.off, tp->psi_b.p + (goff[g] + (long)cp[1] * gR[g]) * nsl + (long)rp[1] * 8,
                    (long)gR[g] * 8, (long)gR[g] * 8 * nsl, B.rows, B.cols, B.cols, pad16(B.cols), 1.0});
      tp->psi_maxel = std::max<long>(tp->psi_maxel, (long)B.rows * pad16(B.cols));
      sj.push_back({tp->sig_t.p + sgoff[g] + (long)cp[1] * gR[g] + rp[1], plan.out.p + B.off, B.rows, B.cols, gR[g]});
      tp->sig_maxel = std::max<long>(tp->sig_maxel, (long)B.rows * B.cols);
    }
    check_group_jobs(pj, nsl, tp->psi_b);
    for (const UnconvJob& u : sj)
      if (u.src < tp->sig_t.p || u.src + (long)(u.cols - 1) * u.lds + u.rows > tp->sig_t.p + tp->sig_total)
        throw Error(ST_ECUDA, "internal: gather job outside sigma^T");
    tp->psi_jobs.upload(pj, c.stream);
    tp->n_psi_jobs = (int)pj.size();
    tp->sig_jobs.upload(sj, c.stream);
    tp->n_sig_jobs = (int)sj.size();
    if (tp->host_copies) {
      tp->h_psi_jobs = pj;
      tp->h_sig_jobs = sj;
    }
    cuda_check(cudaStreamSynchronize(c.stream), "sync");
  }
  // ---- stage-1 row blocks: per input group g', every (beta, n2) with at least one
  // non-zero site block n2' of Rt_beta towards the column blocks of g'
  struct RowBlk {
    int beta, n2, qr, rows, mask;
    int bl[4];  // per n2' in the mask: the operator block of Rt_beta^{n2 n2'}
  };
  std::vector<std::vector<RowBlk>> rb(ng);
  host_parallel(ng, (long)nmid * ng, [&](long gp) {
    for (int beta = 0; beta < nmid; ++beta) {
      const int g = gout[(size_t)beta * ng + gp];
      if (g < 0) continue;
      for (const auto& cb : gcol[g]) {
        const int n2 = cb[0], qr = cb[1];
        RowBlk x{beta, n2, qr, Rb.dim[qr], 0, {-1, -1, -1, -1}};
        for (int n2p = 0; n2p < 4; ++n2p) {
          const TRef& r = rt.ref[beta][n2 * 4 + n2p];
          if (!r.p) continue;
          const int qrp = Rb.find(gq[gp].first + LQA[n2p], gq[gp].second + LQB[n2p]);
          if (qrp < 0 || cpos[qrp * 4 + n2p][0] != gp) continue;
          const OpLayout& Lay = Renv.cls[r.cls];
          const int bl = Lay.blk_of_col[qrp];
          if (bl < 0 || Lay.blocks[bl].rs != qr) continue;
          x.mask |= 1 << n2p;
          x.bl[n2p] = bl;
        }
        if (x.mask) rb[gp].push_back(x);
      }
    }
  });
  size_t nrb = 0;
  for (const auto& v : rb) nrb += v.size();
  std::vector<char> xhas((size_t)nmid * ng, 0);  // [beta][g'] has X^T rows
  for (int gp = 0; gp < ng; ++gp)
    for (const RowBlk& x : rb[gp]) xhas[(size_t)x.beta * ng + gp] = 1;
  // chunks of bond states whose X^T fit the budget (one chunk unless the budget is small)
  std::vector<size_t> xsz(nmid, 0);
  for (int beta = 0; beta < nmid; ++beta)
    for (int gp = 0; gp < ng; ++gp)
      if (xhas[(size_t)beta * ng + gp]) xsz[beta] += (size_t)gC[gout[(size_t)beta * ng + gp]] * gR[gp];
  const long budget_mb = c.precision >= 4 ? c.tma_budget_mb : (long)c.chunk_budget_mb;
  const size_t budget = (size_t)std::max<long>(1, budget_mb) * (1u << 20) / (sizeof(__nv_bfloat16) * nsl);
  // The stacked right operators hold a block once for every bond state and site block that reads it
  // (K=40, M=2000: 12 GB a slice, of a 3.5 GB environment) and are made once per plan, which is
  // quicker than to make those of a chunk in every sigma.  Precisions 1-3 bound their intermediates
  // to leave room for other problems: they do the latter where the whole stack and the vectors of a
  // solve would take more than half of the memory that there is (K=24, M=1500, three
  // slices: 12.9 ms per sigma and 13 GB with the whole stack, 24.9 ms and 5 GB chunk by chunk).
  std::vector<size_t> ssz(nmid, 0);
  for (int gp = 0; gp < ng; ++gp)
    for (const RowBlk& x : rb[gp]) ssz[x.beta] += (size_t)x.rows * gC[gp];
  bool held = true;
  size_t stack_max = std::numeric_limits<size_t>::max();
  if (c.precision <= 3) {
    const size_t el = sizeof(__nv_bfloat16) * nsl;
    size_t x = 0, stack = 0;
    for (int beta = 0; beta < nmid; ++beta) {
      x += xsz[beta];
      stack += ssz[beta];
    }
    const size_t vectors = (size_t)P.nnz * sizeof(double) * 56;  // subspace, its sigma vectors, the others
    const size_t need = (stack + std::min(x, budget)) * el + vectors;
    if (need > (256u << 20)) {  // (the question takes longer than a small plan)
      const size_t left = device_memory_left();
      held = need <= left / 2;
      if (!held) stack_max = left / 8 / el;
    }
  }
  std::vector<std::pair<int, int>> chunks;
  for (int b0 = 0; b0 < nmid;) {
    int b1 = b0;
    size_t tot = 0, stack = 0;
    while (b1 < nmid && (b1 == b0 || (tot + xsz[b1] <= budget && (held || stack + ssz[b1] <= stack_max)))) {
      tot += xsz[b1];
      stack += ssz[b1++];
    }
    chunks.push_back({b0, b1});
    b0 = b1;
  }
  const int nch = (int)chunks.size();
  // stacks of their own layout: one, or one per chunk
  const int nstack = held ? 1 : nch;
  auto stack_of = [&](int ci) { return held ? 0 : ci; };
  std::vector<int> chunk_of(nmid, 0);
  for (int ci = 0; ci < nch; ++ci)
    for (int b = chunks[ci].first; b < chunks[ci].second; ++b) chunk_of[b] = ci;
  // X^T layout per chunk: regions per g' (Sum_beta C_g(beta) rows x R_g' columns in column
  // groups of 8; element offsets below count one slice);
  // xrow[beta][g'] = first row of beta's block in its region
  std::vector<std::vector<long>> xreg(nch, std::vector<long>(ng, 0)), xregrows(nch, std::vector<long>(ng, 0));
  std::vector<long> xrow((size_t)nmid * ng, -1);
  size_t maxchunk = 0;
  for (int ci = 0; ci < nch; ++ci) {
    long off = 0;
    for (int gp = 0; gp < ng; ++gp) {
      xreg[ci][gp] = off;
      long rows = 0;
      for (int beta = chunks[ci].first; beta < chunks[ci].second; ++beta)
        if (xhas[(size_t)beta * ng + gp]) {
          xrow[(size_t)beta * ng + gp] = rows;
          rows += gC[gout[(size_t)beta * ng + gp]];
        }
      xregrows[ci][gp] = rows;
      off += rows * gR[gp];
    }
    maxchunk = std::max(maxchunk, (size_t)off);
  }
  tp->xt.alloc(std::max<size_t>(maxchunk, 8) * nsl, c.stream);
  cuda_check(cudaMemsetAsync(tp->xt.p, 0, tp->xt.n * sizeof(__nv_bfloat16), c.stream), "memset");
  // ---- A1 per g': row blocks sorted by (chunk, mask), beta order kept inside a run
  host_parallel(ng, (long)nrb, [&](long gp) {
    std::stable_sort(rb[gp].begin(), rb[gp].end(), [&](const RowBlk& a, const RowBlk& b) {
      if (chunk_of[a.beta] != chunk_of[b.beta]) return chunk_of[a.beta] < chunk_of[b.beta];
      return a.mask < b.mask;
    });
  });
  // (a run starts on a row group of 16, as the boxes of its tiles have to)
  std::vector<std::vector<long>> a1off(nstack, std::vector<long>(ng, 0)), a1rows(nstack, std::vector<long>(ng, 0));
  std::vector<long> stack_el(nstack, 0);
  for (int gp = 0; gp < ng; ++gp) {
    const RowBlk* prev = nullptr;
    for (const RowBlk& x : rb[gp]) {
      long& rows = a1rows[stack_of(chunk_of[x.beta])][gp];
      if (prev && (chunk_of[prev->beta] != chunk_of[x.beta] || prev->mask != x.mask)) rows = (rows + 15) / 16 * 16;
      rows += x.rows;
      prev = &x;
    }
    for (int st = 0; st < nstack; ++st) {
      a1rows[st][gp] = (a1rows[st][gp] + 15) / 16 * 16;
      a1off[st][gp] = stack_el[st];
      stack_el[st] += a1rows[st][gp] * gC[gp];
    }
  }
  const long a1tot = *std::max_element(stack_el.begin(), stack_el.end());
  tp->a1.alloc(std::max<long>(a1tot, 8) * nsl, c.stream);
  cuda_check(cudaMemsetAsync(tp->a1.p, 0, tp->a1.n * sizeof(__nv_bfloat16), c.stream), "memset");
  struct Run {
    int chunk, mask;
    long r0, r1;
  };
  std::vector<std::vector<Run>> runs(ng);
  // per A1 row: its row in the X^T region of its chunk (columns: blocks of g', each its
  // own submatrix of the region)
  std::vector<std::vector<std::vector<long>>> rowdst(nstack, std::vector<std::vector<long>>(ng));
  // conversion jobs stack by stack, in each group by group: job0[stack * ng + group] the first
  std::vector<size_t> job0((size_t)nstack * ng + 1, 0);
  for (int gp = 0; gp < ng; ++gp)
    for (const RowBlk& x : rb[gp])
      job0[(size_t)stack_of(chunk_of[x.beta]) * ng + gp + 1] += (size_t)__builtin_popcount((unsigned)x.mask);
  for (size_t i = 1; i < job0.size(); ++i) job0[i] += job0[i - 1];
  std::vector<GroupJob> aconv(job0.back());
  std::vector<long> amaxel((size_t)nstack * ng, 0);
  host_parallel(ng, (long)aconv.size(), [&](long gp) {
    long row = 0;
    int st = -1;
    GroupJob* job = nullptr;
    for (int s = 0; s < nstack; ++s) rowdst[s][gp].assign((size_t)a1rows[s][gp], -1);
    for (const RowBlk& x : rb[gp]) {
      const int ci = chunk_of[x.beta];
      if (stack_of(ci) != st) {
        st = stack_of(ci);
        row = 0;
        job = aconv.data() + job0[(size_t)st * ng + gp];
      }
      if (runs[gp].empty() || runs[gp].back().chunk != ci || runs[gp].back().mask != x.mask) {
        row = (row + 15) / 16 * 16;
        runs[gp].push_back({ci, x.mask, row, row});
      }
      runs[gp].back().r1 = row + x.rows;
      const long xr0 = xrow[(size_t)x.beta * ng + gp] + (long)cpos[x.qr * 4 + x.n2][1];
      std::vector<long>& dst = rowdst[st][gp];
      for (int i = 0; i < x.rows; ++i) dst[(size_t)(row + i)] = xr0 + i;
      for (int n2p = 0; n2p < 4; ++n2p) {
        if (!((x.mask >> n2p) & 1)) continue;
        const TRef& r = rt.ref[x.beta][x.n2 * 4 + n2p];
        const Block& B = Renv.cls[r.cls].blocks[x.bl[n2p]];
        // the K block (n2', qr') of g': columns coff .. coff + pad16(d(qr')) of A1
        const int coff = cpos[B.cs * 4 + n2p][1];
        const long rows = a1rows[st][gp];
        *job++ = {r.p + B.off, tp->a1.p + (a1off[st][gp] + rows * coff) * nsl + row * 8, rows * 8,
                  rows * 8 * nsl, B.rows, B.cols, B.cols, pad16(B.cols), r.coef};
        long& most = amaxel[(size_t)st * ng + gp];
        most = std::max<long>(most, (long)B.rows * pad16(B.cols));
      }
      row += x.rows;
    }
  });
  check_group_jobs(aconv, nsl, tp->a1);
  tp->chunks.resize(nch);
  if (held) {
    for (long m : amaxel) tp->a1_maxel = std::max(tp->a1_maxel, m);
    tp->a1_jobs.upload(aconv, c.stream);
    tp->n_a1_jobs = (int)aconv.size();
  } else {
    for (int ci = 0; ci < nch; ++ci) {
      TmaPlan::Chunk& ch = tp->chunks[ci];
      for (int gp = 0; gp < ng; ++gp) ch.a1_maxel = std::max(ch.a1_maxel, amaxel[(size_t)ci * ng + gp]);
      ch.ha1.assign(aconv.begin() + (long)job0[(size_t)ci * ng], aconv.begin() + (long)job0[(size_t)(ci + 1) * ng]);
      ch.a1.upload(ch.ha1, c.stream);
      ch.n_a1 = (int)ch.ha1.size();
    }
    cuda_check(cudaStreamSynchronize(c.stream), "sync");
    if (!tp->host_copies)
      for (auto& ch : tp->chunks) std::vector<GroupJob>().swap(ch.ha1);
  }
  // ---- left mirror: every distinct (operator, scale) referenced by Lt, all its blocks,
  // each padded to 16 rows and columns; blocks of one padded width w share one matrix of
  // w columns
  std::map<int, int> wcls;  // padded width -> class
  std::vector<int> wcls_w;
  for (const OpLayout& L : Lenv.cls)
    for (const Block& B : L.blocks)
      if (!wcls.count(pad16(B.cols))) {
        wcls[pad16(B.cols)] = (int)wcls_w.size();
        wcls_w.push_back(pad16(B.cols));
      }
  const int nwc = (int)wcls_w.size();
  std::vector<long> lrows_c(nwc, 0);
  struct MirKeyHash {
    size_t operator()(const std::pair<const double*, double>& kk) const {
      uint64_t b;
      std::memcpy(&b, &kk.second, sizeof b);
      return std::hash<uint64_t>()((uint64_t)(uintptr_t)kk.first * 0x9e3779b97f4a7c15ULL ^ b);
    }
  };
  std::unordered_map<std::pair<const double*, double>, int, MirKeyHash> lm_id;
  std::vector<std::vector<long>> mblk_row;  // per mirror, per block: row in its width class
  struct PendL {  // one block of a new mirror: source, width class, row in the class, shape
    const double* src;
    int cls;
    long crow;
    int rows, cols;
    double scale;
  };
  std::vector<PendL> lpend;
  std::vector<std::array<int, 16>> lmid((size_t)nmid);
  std::vector<std::array<char, 16>> lneg((size_t)nmid);
  for (int beta = 0; beta < nmid; ++beta)
    for (int nn = 0; nn < 16; ++nn) {
      lmid[beta][nn] = -1;
      lneg[beta][nn] = 0;
      const TRef& r = lt.ref[beta][nn];
      if (!r.p) continue;
      const double a = std::fabs(r.coef);
      const double scale = a == 1.0 ? 1.0 : r.coef;
      auto key = std::make_pair(r.p, scale);
      auto it = lm_id.find(key);
      if (it == lm_id.end()) {
        const int id = (int)mblk_row.size();
        it = lm_id.emplace(key, id).first;
        const OpLayout& L = Lenv.cls[r.cls];
        mblk_row.emplace_back(L.blocks.size());
        for (size_t b = 0; b < L.blocks.size(); ++b) {
          const Block& B = L.blocks[b];
          const int wc = wcls[pad16(B.cols)];
          mblk_row[id][b] = lrows_c[wc];
          lpend.push_back({r.p + B.off, wc, lrows_c[wc], B.rows, B.cols, scale});
          lrows_c[wc] += pad16(B.rows);
        }
      }
      lmid[beta][nn] = it->second;
      lneg[beta][nn] = (a == 1.0 && r.coef < 0) ? 1 : 0;
    }
  std::vector<long> lbase(nwc, 0);
  long ltot = 0;
  for (int wc = 0; wc < nwc; ++wc) {
    lbase[wc] = ltot;
    ltot += lrows_c[wc] * wcls_w[wc];
  }
  const long ls = std::max<long>(ltot, 8);
  tp->lmir.alloc(ls * nsl, c.stream);
  cuda_check(cudaMemsetAsync(tp->lmir.p, 0, tp->lmir.n * sizeof(__nv_bfloat16), c.stream), "memset");
  std::vector<GroupJob> lconv;
  lconv.reserve(lpend.size());
  for (const PendL& pl : lpend) {
    const int w = wcls_w[pl.cls];
    lconv.push_back({pl.src, tp->lmir.p + lbase[pl.cls] * nsl + pl.crow * 8, lrows_c[pl.cls] * 8,
                     lrows_c[pl.cls] * 8 * nsl, pl.rows, pl.cols, pl.cols, w, pl.scale});
    tp->l_maxel = std::max<long>(tp->l_maxel, (long)pl.rows * w);
  }
  check_group_jobs(lconv, nsl, tp->lmir);
  tp->l_jobs.upload(lconv, c.stream);
  tp->n_l_jobs = (int)lconv.size();
  // ---- tensor maps
  std::vector<CUtensorMap> maps;
  // every map must lie inside its buffer (a box outside the map's extent reads zeros,
  // but the extent itself is trusted by the hardware)
  struct MapInfo {
    long rows, cols;
    int box;
  };
  std::vector<MapInfo> minfo;
  // a matrix of rows x cols in the column-group layout from element off
  auto add_map = [&](const DArr<__nv_bfloat16>& buf, long off, long rows, long cols, int box_rows) {
    if (off < 0 || rows < 1 || cols < 1 || rows % 16 != 0 || cols % 16 != 0 || off % 8 != 0 ||
        (size_t)(off + nsl * rows * cols) > buf.n)
      throw Error(ST_ECUDA, "internal: tensor map outside its buffer");
    const int id = (int)maps.size();
    CUtensorMap m;
    if (!encode_slice_map(&m, buf.p + off, (uint64_t)rows, (uint64_t)cols, nsl, (uint32_t)box_rows))
      throw Error(ST_ECUDA, "cuTensorMapEncodeTiled failed");
    maps.push_back(m);
    minfo.push_back({rows, cols, box_rows});
    return id;
  };
  // Two or three slices: a term stays in the ring whole, so a block that is longer than
  // tm_term_pieces is cut into equal parts (a term each).  Stage 1: the widest N tiles whose ring
  // holds the longest part.
  // Three and two slices, ms per sigma, against whole terms with one CTA per SM and twice the ring,
  // and one 16-column copy of one slice per stage where they did not fit that either: K=16, M=2000
  // (sectors of up to 238) 67.6 and 34.8 -> 15.1 and 8.8; K=16, M=1000 (121) 4.02 and 2.68 -> 2.41
  // and 1.45; K=20, M=800 (83) 3.34 and 1.62 -> 2.72 and 1.60; K=40, M=2000 (115, three slices)
  // 47.8 -> 33.2.
  int n1max = tm_max_n(TM_MODE_STORE_BF16, nsl);
  const int n2max = tm_max_n(TM_MODE_REDUCE_F32, nsl);
  auto parts_of = [&](int kk, int limit) {
    return nsl == 1 ? 1 : (kk / TM_PIECE_COLS + limit - 1) / limit;
  };
  // columns [first, second) of part i of `parts`
  auto part_cols = [](int kk, int parts, int i) {
    const int kp = kk / TM_PIECE_COLS;
    return std::make_pair(kp * i / parts * TM_PIECE_COLS, kp * (i + 1) / parts * TM_PIECE_COLS);
  };
  if (nsl > 1) {
    int kmax = 16;
    for (int qr = 0; qr < nR; ++qr) kmax = std::max(kmax, pad16(Rb.dim[qr]));
    const int parts = parts_of(kmax, TM_TERM_PIECES), len = (kmax / TM_PIECE_COLS + parts - 1) / parts;
    while (n1max > 64 && tm_term_pieces(nsl, n1max) < len) n1max -= 16;
  }
  std::vector<std::vector<std::array<int, 3>>> nt1(ng);  // per g': (row0, width, Psi map) of the stage-1 N tiles
  std::vector<std::vector<int>> a1map(nstack, std::vector<int>(ng, -1));
  int n1wide = 16, n2wide = 16;
  for (int gp = 0; gp < ng; ++gp) {
    if (rb[gp].empty()) continue;
    const int parts = (gR[gp] + n1max - 1) / n1max;
    int r0 = 0;
    for (int p = 0; p < parts; ++p) {
      const int w = std::min(gR[gp] - r0, pad16((gR[gp] - r0 + (parts - p) - 1) / (parts - p)));
      nt1[gp].push_back({r0, w, add_map(tp->psi_b, goff[gp] * nsl, gR[gp], gC[gp], w)});
      r0 += w;
      n1wide = std::max(n1wide, w);
    }
    for (int st = 0; st < nstack; ++st)
      if (a1rows[st][gp] > 0) a1map[st][gp] = add_map(tp->a1, a1off[st][gp] * nsl, a1rows[st][gp], gC[gp], 128);
  }
  for (int ql = 0; ql < nL; ++ql) n2wide = std::max(n2wide, std::min(n2max, pad16(Lb.dim[ql])));
  const int limit1 = tm_term_pieces(nsl, n1wide), limit2 = tm_term_pieces(nsl, n2wide);
  // X^T region of (chunk, g')
  std::vector<std::vector<int>> xtmap(nch, std::vector<int>(ng, -1));
  for (int ci = 0; ci < nch; ++ci)
    for (int gp = 0; gp < ng; ++gp)
      if (xregrows[ci][gp] > 0) xtmap[ci][gp] = add_map(tp->xt, xreg[ci][gp] * nsl, xregrows[ci][gp], gR[gp], 128);
  // left mirror: per width class one map per box height
  std::vector<std::vector<int>> lmap(nwc, std::vector<int>(n2max / 16 + 1, -1));
  for (int wc = 0; wc < nwc; ++wc)
    if (lrows_c[wc] > 0)
      for (int h = 16; h <= n2max; h += 16)
        lmap[wc][h / 16] = add_map(tp->lmir, lbase[wc] * nsl, lrows_c[wc], wcls_w[wc], h);
  tp->maps.alloc(std::max<size_t>(maps.size(), 1), c.stream);
  if (!maps.empty())
    cuda_check(cudaMemcpyAsync(tp->maps.p, maps.data(), maps.size() * sizeof(CUtensorMap), cudaMemcpyHostToDevice,
                               c.stream),
               "h2d");
  if (tp->host_copies) tp->hmaps = maps;
  // ---- work lists per chunk
  std::vector<long> rowmap;
  double st1_tiles = 0, st1_steps = 0, st2_tiles = 0, st2_steps = 0, st1_fl = 0, st2_fl = 0;
  for (int ci = 0; ci < nch; ++ci) {
    TmaPlan::Chunk& ch = tp->chunks[ci];
    std::vector<TmTile> t1, t2;
    std::vector<TmTerm> m1, m2;
    std::vector<ZeroJob> zj;
    // stage 1: per g', per (chunk, mask) run, 128-row tiles x N tiles; every group fills its own
    // part of the lists
    std::vector<std::array<size_t, 3>> at1(ng + 1, std::array<size_t, 3>{0, 0, rowmap.size()});  // tiles, terms, rows
    for (int gp = 0; gp < ng; ++gp) {
      at1[gp + 1] = at1[gp];
      size_t nterm[4];  // terms of the K block of n2'
      for (int n2p = 0; n2p < 4; ++n2p) {
        const int qrp = Rb.find(gq[gp].first + LQA[n2p], gq[gp].second + LQB[n2p]);
        nterm[n2p] = qrp < 0 ? 0 : (size_t)parts_of(pad16(Rb.dim[qrp]), limit1);
      }
      for (const Run& run : runs[gp]) {
        if (run.chunk != ci) continue;
        const size_t nrow = (size_t)((run.r1 - run.r0 + 127) / 128);
        at1[gp + 1][0] += nrow * nt1[gp].size();
        for (int n2p = 0; n2p < 4; ++n2p)
          if ((run.mask >> n2p) & 1) at1[gp + 1][1] += nrow * nt1[gp].size() * nterm[n2p];
        at1[gp + 1][2] += nrow * 128;
      }
    }
    t1.resize(at1[ng][0]);
    m1.resize(at1[ng][1]);
    rowmap.resize(at1[ng][2]);
    std::vector<std::array<double, 2>> st1(ng, {0, 0});  // steps, flops
    host_parallel(ng, (long)rowmap.size() / 16, [&](long gp) {
      size_t it = at1[gp][0], im = at1[gp][1], ir = at1[gp][2];
      const std::vector<long>& dst = rowdst[stack_of(ci)][gp];
      for (const Run& run : runs[gp]) {
        if (run.chunk != ci) continue;
        for (long r0 = run.r0; r0 < run.r1; r0 += 128) {
          const long moff = (long)ir;
          for (long i = 0; i < 128; ++i) rowmap[ir++] = r0 + i < run.r1 ? dst[(size_t)(r0 + i)] : -1;
          for (const auto& nt : nt1[gp]) {
            TmTile tl{};
            tl.t0 = (int)im;
            int ksum = 0;
            for (int n2p = 0; n2p < 4; ++n2p) {
              if (!((run.mask >> n2p) & 1)) continue;
              // the K block of n2': the column block (n2', qr') of g'
              const int qrp = Rb.find(gq[gp].first + LQA[n2p], gq[gp].second + LQB[n2p]);
              const int coff = cpos[qrp * 4 + n2p][1];
              const int kk = pad16(Rb.dim[qrp]);
              const int parts = parts_of(kk, limit1);
              for (int p = 0; p < parts; ++p) {
                const auto cols = part_cols(kk, parts, p);
                m1[im++] = {a1map[stack_of(ci)][gp], nt[2], coff + cols.first, (int)r0, coff + cols.first, nt[0],
                            cols.second - cols.first, nsl << 4};
              }
              ksum += kk * npair;
              st1[gp][0] += (kk + 63) / 64 * npair;
            }
            tl.t1 = (int)im;
            tl.nseg = 1;
            tl.xbase = xreg[ci][gp] * nsl;
            tl.xrows = xregrows[ci][gp];
            tl.n = nt[1];
            tl.m_valid = 128;
            tl.ldo = gR[gp];
            tl.out_off = nt[0];
            tl.rowmap_off = moff;
            t1[it++] = tl;
            st1[gp][1] += 2.0 * 128 * nt[1] * ksum;
          }
        }
      }
    });
    for (const auto& v : st1) {
      st1_steps += v[0];
      st1_fl += v[1];
    }
    // X^T rows of this chunk that stage 1 does not write: zero them before the chunk
    // (with one chunk the buffer is zero from the start)
    if (nch > 1) {
      std::vector<std::vector<ZeroJob>> zg(ng);
      const int b0 = chunks[ci].first, b1 = chunks[ci].second;
      host_parallel(ng, (long)(b1 - b0) * ng * 4, [&](long gp) {
        std::vector<char> written((size_t)(b1 - b0) * 4 * nR, 0);  // [beta][n2][qr]
        auto at = [&](int beta, int n2, int qr) { return ((size_t)(beta - b0) * 4 + n2) * nR + qr; };
        // the row blocks are sorted by chunk
        auto x = std::lower_bound(rb[gp].begin(), rb[gp].end(), ci,
                                  [&](const RowBlk& a, int c2) { return chunk_of[a.beta] < c2; });
        for (; x != rb[gp].end() && chunk_of[x->beta] == ci; ++x) written[at(x->beta, x->n2, x->qr)] = 1;
        for (int beta = b0; beta < b1; ++beta) {
          if (!xhas[(size_t)beta * ng + gp]) continue;
          const int g = gout[(size_t)beta * ng + gp];
          for (const auto& cb : gcol[g]) {
            if (written[at(beta, cb[0], cb[1])]) continue;
            // the block's rows in every column group
            const long r0 = xrow[(size_t)beta * ng + gp] + cb[2], rows = xregrows[ci][gp];
            zg[gp].push_back({tp->xt.p + xreg[ci][gp] * nsl + r0 * 8, (long)pad16(Rb.dim[cb[1]]) * 8, rows * 8, nsl,
                              gR[gp] / 8, rows * 8 * nsl});
          }
        }
      });
      for (const auto& z : zg) zj.insert(zj.end(), z.begin(), z.end());
    }
    // stage 2: per output block (g, (ql, n1) column block, N part), 128-row tiles, terms
    // over the chunk's bond states; long term lists cut into parts (split-K)
    struct Pending {
      TmTile tl;
      std::vector<TmTerm> terms;
    };
    std::vector<std::vector<Pending>> pend(ng);
    std::vector<long> gsteps(ng, 0);
    host_parallel(ng, (long)nmid * ng, [&](long g) {
      for (const auto& rbk : grow[g]) {
        const int ql = rbk[0], n1 = rbk[1];
        const int dql = Lb.dim[ql];
        for (int c0 = 0; c0 < pad16(dql); c0 += n2max) {
          const int nw = std::min(n2max, pad16(dql) - c0);
          // the block's terms for the first row tile; other row tiles shift the X^T row
          std::vector<TmTerm> base;
          for (int beta = chunks[ci].first; beta < chunks[ci].second; ++beta) {
            const int gp = gin[(size_t)beta * ng + g];
            if (gp < 0 || !xhas[(size_t)beta * ng + gp]) continue;
            for (int n1p = 0; n1p < 4; ++n1p) {
              const TRef& r = lt.ref[beta][n1 * 4 + n1p];
              if (!r.p) continue;
              const OpLayout& Lay = Lenv.cls[r.cls];
              const int qlp = Lb.find(Lb.qa[ql] - Lay.da, Lb.qb[ql] - Lay.db);
              if (qlp < 0) continue;
              const int bl = Lay.blk_of_col[qlp];
              if (bl < 0 || Lay.blocks[bl].rs != ql) continue;
              const auto rpp = rpos[qlp * 4 + n1p];
              if (rpp[0] != gp) continue;
              const int mid_ = lmid[beta][n1 * 4 + n1p];
              const int wc = wcls.at(pad16(Lb.dim[qlp]));
              const int kk = pad16(Lb.dim[qlp]), parts = parts_of(kk, limit2);
              for (int p = 0; p < parts; ++p) {
                const auto cols = part_cols(kk, parts, p);
                base.push_back({xtmap[ci][gp], lmap[wc][nw / 16], rpp[1] + cols.first, (int)xrow[(size_t)beta * ng + gp],
                                cols.first, (int)(mblk_row[mid_][bl] + c0), cols.second - cols.first,
                                (int)lneg[beta][n1 * 4 + n1p]});
              }
            }
          }
          if (base.empty()) continue;
          for (TmTerm& t : base) t.neg |= nsl << 4;
          long steps = 0;  // products
          for (const TmTerm& t : base) steps += (long)t.k / TM_PIECE_COLS * npair;
          for (int r0 = 0; r0 < gC[g]; r0 += 128) {
            Pending pd;
            pd.tl = TmTile{};
            pd.tl.n = nw;
            pd.tl.m_valid = std::min(128, gC[g] - r0);
            pd.tl.ldo = gR[g];
            pd.tl.out_off = sgoff[g] + (long)r0 * gR[g] + rbk[2] + c0;
            pd.terms = base;
            for (TmTerm& t : pd.terms) t.ay += r0;
            gsteps[g] += steps;
            pend[g].push_back(std::move(pd));
          }
        }
      }
    });
    const long total_steps = std::accumulate(gsteps.begin(), gsteps.end(), 0L);
    const long target = c.split_tps > 0 ? std::max<long>(1, total_steps / std::max<long>(1, std::lround(c.split_tps * 152)))
                                        : std::numeric_limits<long>::max();
    std::vector<Pending> all;
    for (auto& pg : pend) std::move(pg.begin(), pg.end(), std::back_inserter(all));
    for (Pending& pd : all) {
      long acc = 0;
      size_t t0 = 0;
      for (size_t t = 0; t < pd.terms.size(); ++t) {
        acc += (long)pd.terms[t].k / TM_PIECE_COLS * npair;
        if (acc >= target || t + 1 == pd.terms.size()) {
          TmTile tl = pd.tl;
          tl.t0 = (int)m2.size();
          long ks = 0;
          for (size_t u = t0; u <= t; ++u) {
            m2.push_back(pd.terms[u]);
            ks += (long)pd.terms[u].k * npair;
          }
          tl.t1 = (int)m2.size();
          if (ks / TM_PIECE_COLS > (1L << 30)) throw Error(ST_ECUDA, "internal: stage-2 tile too long");
          t2.push_back(tl);
          st2_steps += (double)((ks + 63) / 64);
          st2_fl += 2.0 * 128 * tl.n * ks;
          t0 = t + 1;
          acc = 0;
        }
      }
    }
    longest_first(t1, m1);
    longest_first(t2, m2);
    // the copy lists of both launches (stage 2: sets every tile's stages and segments);
    // their pieces follow from the terms checked below
    ch.l1.plan(TM_MODE_STORE_BF16, nsl, t1, m1, c.stream);
    ch.l2.plan(TM_MODE_REDUCE_F32, nsl, t2, m2, c.stream);
    st1_tiles += (double)t1.size();
    st2_tiles += (double)t2.size();
    // every access of the kernels checked against its buffer before anything runs:
    // operand boxes (their coordinates, alignment and widths), the rows stage 1 stores
    // through the row map and the blocks stage 2 reduces into
    auto check_terms = [&](const std::vector<TmTile>& tt, const std::vector<TmTerm>& mm, int nmax) {
      host_parallel((long)(tt.size() + 255) / 256, (long)mm.size(), [&](long blk) {
        for (size_t ti = (size_t)blk * 256; ti < std::min(tt.size(), (size_t)(blk + 1) * 256); ++ti) {
          const TmTile& tl = tt[ti];
          if (tl.n < 16 || tl.n > nmax || tl.n % 16 || tl.t0 < 0 || tl.t1 <= tl.t0 || tl.t1 > (int)mm.size())
            throw Error(ST_ECUDA, "internal: malformed TMA tile");
          for (int t = tl.t0; t < tl.t1; ++t) {
            const TmTerm& m = mm[t];
            if (((m.neg >> 4) & 15) != nsl || m.amap < 0 || m.amap >= (int)minfo.size() || m.bmap < 0 ||
                m.bmap >= (int)minfo.size() || minfo[m.amap].box != 128 || minfo[m.bmap].box != tl.n || m.k < 16 ||
                m.k % 16 || m.ax % 8 || m.bx % 8 || m.ay % 16 || m.by % 16 || m.ax < 0 || m.bx < 0 || m.ay < 0 ||
                m.by < 0 || m.ay >= minfo[m.amap].rows || m.by >= minfo[m.bmap].rows ||
                m.ax + m.k > minfo[m.amap].cols || m.bx + m.k > minfo[m.bmap].cols)
              throw Error(ST_ECUDA, "internal: malformed TMA term");
          }
        }
      });
    };
    check_terms(t1, m1, n1max);
    check_terms(t2, m2, n2max);
    // stage-1 stores: every row inside its region, every region (all slices) inside X
    for (const long d : rowmap)
      if (d < -1) throw Error(ST_ECUDA, "internal: stage-1 row map");
    host_parallel((long)(t1.size() + 255) / 256, (long)t1.size() * 16, [&](long blk) {
      for (size_t ti = (size_t)blk * 256; ti < std::min(t1.size(), (size_t)(blk + 1) * 256); ++ti) {
        const TmTile& tl = t1[ti];
        if (tl.rowmap_off < 0 || tl.rowmap_off + 128 > (long)rowmap.size() || tl.out_off < 0 || tl.out_off % 8 ||
            tl.ldo % 8 || tl.out_off + tl.n > tl.ldo || tl.xbase < 0 || tl.xbase % 8 || tl.xrows < 1 ||
            (size_t)(tl.xbase + nsl * tl.xrows * tl.ldo) > tp->xt.n)
          throw Error(ST_ECUDA, "internal: stage-1 row map, columns or region out of range");
        for (int r = 0; r < 128; ++r)
          if (rowmap[(size_t)(tl.rowmap_off + r)] >= tl.xrows)
            throw Error(ST_ECUDA, "internal: stage-1 row outside its X region");
      }
    });
    for (const TmTile& tl : t2) {
      long prod = 0;
      for (int t = tl.t0; t < tl.t1; ++t) prod += (long)m2[(size_t)t].k / TM_PIECE_COLS * npair;
      if (tl.pad < 1 || tl.nseg != (int)((prod + TM_SEG_PRODUCTS - 1) / TM_SEG_PRODUCTS))
        throw Error(ST_ECUDA, "internal: stage-2 stage or segment count");
    }

    for (const TmTile& tl : t2)
      if (tl.m_valid < 1 || tl.m_valid > 128 || tl.out_off < 0 || tl.out_off % 4 || tl.ldo % 4 ||
          tl.out_off + (long)(tl.m_valid - 1) * tl.ldo + tl.n > tp->sig_total)
        throw Error(ST_ECUDA, "internal: stage-2 reduction outside sigma^T");
    for (const ZeroJob& z : zj)
      if (z.p < tp->xt.p || z.p + (long)(z.nsl - 1) * z.stride + (z.reps - 1) * z.pitch + z.n > tp->xt.p + tp->xt.n)
        throw Error(ST_ECUDA, "internal: zero job outside X");
    ch.t1.upload(t1, c.stream);
    ch.m1.upload(m1, c.stream);
    ch.n1 = (int)t1.size();
    ch.t2.upload(t2, c.stream);
    ch.m2.upload(m2, c.stream);
    ch.n2 = (int)t2.size();
    ch.l1.fill(TM_MODE_STORE_BF16, nsl, ch.t1.p, ch.n1, ch.m1.p, c.stream);
    ch.l2.fill(TM_MODE_REDUCE_F32, nsl, ch.t2.p, ch.n2, ch.m2.p, c.stream);
    ch.nz = (int)zj.size();
    for (const ZeroJob& z : zj) ch.zmax = std::max(ch.zmax, z.n);
    ch.z.upload(zj, c.stream);
    cuda_check(cudaStreamSynchronize(c.stream), "sync");
    if (tp->host_copies) {
      ch.ht1.swap(t1);
      ch.ht2.swap(t2);
      ch.hm1.swap(m1);
      ch.hm2.swap(m2);
      ch.hz.swap(zj);
    }
  }
  tp->rowmap.upload(rowmap, c.stream);
  if (tp->host_copies) tp->hrowmap = rowmap;
  // the operator stacks depend only on the environments: filled once per plan if all are held
  if (tp->n_a1_jobs) launch_conv_groups(tp->a1_jobs, tp->n_a1_jobs, nsl, tp->a1_maxel, c.stream);
  if (tp->n_l_jobs) launch_conv_groups(tp->l_jobs, tp->n_l_jobs, nsl, tp->l_maxel, c.stream);
  tp->err.alloc(1, c.stream);
  cuda_check(cudaMemsetAsync(tp->err.p, 0, sizeof(int), c.stream), "memset");
  cuda_check(cudaStreamSynchronize(c.stream), "sync");
  tp->stats[0] = st1_tiles;
  tp->stats[1] = st1_steps;
  tp->stats[2] = st2_tiles;
  tp->stats[3] = st2_steps;
  tp->stats[4] = st1_fl;
  tp->stats[5] = st2_fl;
  tp->stats[6] = (double)maxchunk * 2;
  tp->stats[7] = (double)a1tot * 2;
  tp->stats[8] = nch;
  plan.flops = flops.get();
}

void run_tma_sigma(Context& c, SigmaPlan& plan, const double* x, double* y) {
  TmaPlan& tp = *plan.tm;
  // the conversions read x and write y themselves (their jobs are made for plan.in and plan.out)
  if (tp.n_psi_jobs) launch_conv_groups(tp.psi_jobs, tp.n_psi_jobs, tp.nsl, tp.psi_maxel, c.stream, x - plan.in.p);
  cuda_check(cudaMemsetAsync(tp.sig_t.p, 0, tp.sig_total * sizeof(float), c.stream), "memset");
  for (auto& ch : tp.chunks) {
    if (ch.n_a1) launch_conv_groups(ch.a1, ch.n_a1, tp.nsl, ch.a1_maxel, c.stream);
    if (ch.nz) launch_zero(ch.z.p, ch.nz, ch.zmax, c.stream);
    cuda_check(launch_gemm_slices(TM_MODE_STORE_BF16, tp.nsl, ch.t1.p, ch.n1, tp.maps.p, tp.rowmap.p, tp.xt.p, tp.err.p,
                                  c.stream, ch.l1.dev()),
               "tma stage 1");
    cuda_check(launch_gemm_slices(TM_MODE_REDUCE_F32, tp.nsl, ch.t2.p, ch.n2, tp.maps.p, nullptr, tp.sig_t.p, tp.err.p,
                                  c.stream, ch.l2.dev()),
               "tma stage 2");
  }
  if (tp.n_sig_jobs) launch_unconv(tp.sig_jobs.p, tp.n_sig_jobs, tp.sig_maxel, c.stream, y - plan.out.p);
}

int plan_error(Context& c, SigmaPlan& plan) {
  int h = 0;
  int* p = plan.tm ? plan.tm->err.p : nullptr;
  if (!p) return 0;
  cuda_check(cudaMemcpyAsync(&h, p, sizeof(int), cudaMemcpyDeviceToHost, c.stream), "d2h");
  cuda_check(cudaStreamSynchronize(c.stream), "sync");
  return h;
}

// ---------------------------------------------------------------- environment update on the tensor cores

namespace {

// transposed FP64 block -> nsl BF16 slices: dst[j * ldd + i] = slices of scale * src[i * lds + j]
// for i < rows, j < cols; zeros for rows <= i < wrows (the padded contraction columns)
struct ConvTJob {
  const double* src;
  __nv_bfloat16* dst;
  long slice_stride;
  int rows, cols, lds, ldd, nsl, wrows;
  double scale;
};

__global__ void convt_kernel(const ConvTJob* __restrict__ jobs) {
  const ConvTJob jb = jobs[blockIdx.y];
  const long n = (long)jb.cols * jb.wrows;
  for (long e = (long)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += (long)gridDim.x * blockDim.x) {
    const int j = (int)(e / jb.wrows), i = (int)(e % jb.wrows);
    double v = i < jb.rows ? jb.scale * jb.src[(long)i * jb.lds + j] : 0.0;
    __nv_bfloat16* d = jb.dst + (long)j * jb.ldd + i;
    for (int s = 0; s < jb.nsl; ++s) {
      const __nv_bfloat16 h = __double2bfloat16(v);
      d[s * jb.slice_stride] = h;
      v -= (double)__bfloat162float(h);
    }
  }
}

__global__ void f32_to_f64_kernel(const float* __restrict__ src, double* __restrict__ dst, long n) {
  for (long e = (long)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += (long)gridDim.x * blockDim.x)
    dst[e] = (double)src[e];
}

}  // namespace

// L_{k+1}[beta] = sum (A^{n1})^T Lt_beta^{n1 n1'} A^{n1'} (left, Eqs. leftrenorm / prenormdec) or
// R_k[beta] = sum B^{n2} Rt_beta^{n2 n2'} (B^{n2'})^T (right), both stages as tensor-core
// grouped GEMMs with every operand in three BF16 slices (six products, FP32 accumulation):
//   left : stage 1 T^T_beta[n1][j, ql] = sum_{n1'} At^{n1'}[j, ql'] Lt^{n1 n1'}[ql, ql']   (At = A^T per block)
//          stage 2 L'[qa, qa']       = sum_{n1} At^{n1}[qa, ql] T^T_beta[n1][qa', ql]
//   right: stage 1 T_beta[n2][j, qr] = sum_{n2'} B^{n2'}[j, qr'] Rt^{n2 n2'}[qr, qr']
//          stage 2 R'[qb, qb']       = sum_{n2} B^{n2}[qb, qr] T_beta[n2][qb', qr]
// The intermediates are BF16 slices of the FP32 results; the new operators are
// accumulated in FP32 and stored in FP64.
void env_update_tc(Context& c, Tilde& t, const SiteT& A, int site, Env& out, bool left) {
  constexpr int NSL = 3;
  const auto& st = left ? c.mpo.bonds[site + 1] : c.mpo.bonds[site];
  const Bond& Lb = A.L;
  const Bond& Rb = A.R;
  Env& env = *t.env;
  const Bond& ob = left ? Rb : Lb;  // bond of the new operators
  env_alloc(c, out, ob, st);
  const int no = ob.nsec();
  // ---- site-tensor mirror: left: At per block [d(qr) x pad8(d(ql))]; right: [d(ql) x pad8(d(qr))]
  std::vector<long> soff(A.blocks.size());
  long stot = 0;
  for (size_t b = 0; b < A.blocks.size(); ++b) {
    const Block& B = A.blocks[b];
    soff[b] = stot;
    stot += left ? (long)B.cols * pad8(B.rows) : (long)B.rows * pad8(B.cols);
  }
  const long ss = std::max<long>(stot, 8);
  DArr<__nv_bfloat16> smir;
  smir.alloc((size_t)ss * NSL, c.stream);
  {
    if (left) {
      std::vector<ConvTJob> jobs;
      long mx = 0;
      for (size_t b = 0; b < A.blocks.size(); ++b) {
        const Block& B = A.blocks[b];
        jobs.push_back({A.d.p + B.off, smir.p + soff[b], ss, B.rows, B.cols, B.cols, pad8(B.rows), NSL, pad8(B.rows),
                        1.0});
        mx = std::max<long>(mx, (long)B.cols * pad8(B.rows));
      }
      DArr<ConvTJob> dj;
      dj.upload(jobs, c.stream);
      for (int o0 = 0; o0 < (int)jobs.size(); o0 += 65535) {
        const int nj = std::min(65535, (int)jobs.size() - o0);
        const long g = std::min<long>(std::max<long>(1, (mx + 255) / 256), 64);
        convt_kernel<<<dim3((unsigned)g, nj), 256, 0, c.stream>>>(dj.p + o0);
        count_launches(1);
      }
      cuda_check(cudaGetLastError(), "convt launch");
      cuda_check(cudaStreamSynchronize(c.stream), "sync");
    } else {
      std::vector<ConvJob> jobs;
      long mx = 0;
      for (size_t b = 0; b < A.blocks.size(); ++b) {
        const Block& B = A.blocks[b];
        jobs.push_back({A.d.p + B.off, smir.p + soff[b], ss, B.rows, B.cols, B.cols, pad8(B.cols), NSL, 1.0,
                        pad8(B.cols)});
        mx = std::max<long>(mx, (long)B.rows * pad8(B.cols));
      }
      DArr<ConvJob> dj;
      dj.upload(jobs, c.stream);
      if (!jobs.empty()) launch_conv(dj, (int)jobs.size(), mx, c.stream);
      cuda_check(cudaStreamSynchronize(c.stream), "sync");
    }
  }
  // ---- W-contracted operator mirror: every distinct (operator, scale), all blocks,
  // row-major with leading dimension pad8(cols)
  std::vector<std::vector<long>> boff(env.cls.size());
  std::vector<long> bsz(env.cls.size());
  for (size_t i = 0; i < env.cls.size(); ++i) boff[i] = padded_offsets(env.cls[i], &bsz[i]);
  struct KeyHash {
    size_t operator()(const std::pair<const double*, double>& kk) const {
      uint64_t b;
      std::memcpy(&b, &kk.second, sizeof b);
      return std::hash<uint64_t>()((uint64_t)(uintptr_t)kk.first * 0x9e3779b97f4a7c15ULL ^ b);
    }
  };
  std::unordered_map<std::pair<const double*, double>, long, KeyHash> moff;
  std::vector<std::array<long, 16>> mref(st.size());
  std::vector<std::array<char, 16>> mneg(st.size());
  long mtot = 0;
  std::vector<std::pair<const TRef*, long>> created;
  for (size_t beta = 0; beta < st.size(); ++beta)
    for (int nn = 0; nn < 16; ++nn) {
      mref[beta][nn] = -1;
      mneg[beta][nn] = 0;
      const TRef& r = t.ref[beta][nn];
      if (!r.p) continue;
      const double a = std::fabs(r.coef);
      const double scale = a == 1.0 ? 1.0 : r.coef;
      auto key = std::make_pair(r.p, scale);
      auto it = moff.find(key);
      if (it == moff.end()) {
        it = moff.emplace(key, mtot).first;
        created.push_back({&r, mtot});
        mtot += bsz[r.cls];
      }
      mref[beta][nn] = it->second;
      mneg[beta][nn] = (a == 1.0 && r.coef < 0) ? 1 : 0;
    }
  const long ms_ = std::max<long>(mtot, 8);
  DArr<__nv_bfloat16> omir;
  omir.alloc((size_t)ms_ * NSL, c.stream);
  {
    std::vector<ConvJob> jobs;
    long mx = 0;
    for (const auto& cr : created) {
      const TRef& r = *cr.first;
      const double a = std::fabs(r.coef);
      const double scale = a == 1.0 ? 1.0 : r.coef;
      const OpLayout& L = env.cls[r.cls];
      for (size_t b = 0; b < L.blocks.size(); ++b) {
        const Block& B = L.blocks[b];
        jobs.push_back({r.p + B.off, omir.p + cr.second + boff[r.cls][b], ms_, B.rows, B.cols, B.cols, pad8(B.cols),
                        NSL, scale, pad8(B.cols)});
        mx = std::max<long>(mx, (long)B.rows * pad8(B.cols));
      }
    }
    DArr<ConvJob> dj;
    dj.upload(jobs, c.stream);
    if (!jobs.empty()) launch_conv(dj, (int)jobs.size(), mx, c.stream);
    cuda_check(cudaStreamSynchronize(c.stream), "sync");
  }
  // ---- FP32 staging of the new operators (same layout as their FP64 data)
  std::vector<DArr<float>> f32(out.cls.size());
  for (size_t ci = 0; ci < out.cls.size(); ++ci) {
    f32[ci].alloc(std::max<size_t>(out.data[ci].n, 1), c.stream);
    cuda_check(cudaMemsetAsync(f32[ci].p, 0, f32[ci].n * sizeof(float), c.stream), "memset");
  }
  auto f32_op = [&](int beta) {
    return f32[out.st_cls[beta]].p + (size_t)out.st_slot[beta] * out.cls[out.st_cls[beta]].nnz;
  };
  // ---- the intermediate blocks per bond state: left (n1, j): d(j) x pad8(d(ql));
  // right (n2, j): d(j) x pad8(d(qr))
  const Bond& ib = left ? Lb : Rb;  // bond of the contracted index of stage 1
  auto inner_of = [&](int beta, int n, int j) -> int {
    // left: ql with ql + q(n1) + dQ_beta = qr_j; right: qr with qr = ql_j + dQ + q(n2)
    if (left) return Lb.find(Rb.qa[j] + st[beta].dna - LQA[n], Rb.qb[j] + st[beta].dnb - LQB[n]);
    return Rb.find(Lb.qa[j] + st[beta].dna + LQA[n], Lb.qb[j] + st[beta].dnb + LQB[n]);
  };
  std::vector<size_t> tsz(st.size(), 0);
  for (size_t beta = 0; beta < st.size(); ++beta)
    for (int n = 0; n < 4; ++n)
      for (int j = 0; j < no; ++j) {
        const int q = inner_of((int)beta, n, j);
        if (q >= 0) tsz[beta] += (size_t)ob.dim[j] * pad8(ib.dim[q]);
      }
  const size_t budget = std::max<size_t>(1, (size_t)c.chunk_budget_mb * (1u << 20) / (2 * NSL));
  for (size_t b0 = 0; b0 < st.size();) {
    size_t b1 = b0, tot = 0;
    while (b1 < st.size() && (b1 == b0 || tot + tsz[b1] <= budget)) tot += tsz[b1++];
    const long ts = std::max<long>((long)tot, 8);
    DArr<__nv_bfloat16> T;
    T.alloc((size_t)ts * NSL, c.stream);
    cuda_check(cudaMemsetAsync(T.p, 0, T.n * sizeof(__nv_bfloat16), c.stream), "memset");
    TcBuilder g1, g2;
    size_t toff = 0;
    double fl = 0;
    for (size_t beta = b0; beta < b1; ++beta) {
      std::vector<long> tpos((size_t)4 * no, -1);
      for (int n = 0; n < 4; ++n)
        for (int j = 0; j < no; ++j) {
          const int q = inner_of((int)beta, n, j);
          if (q < 0) continue;
          const int m = ob.dim[j], nn = ib.dim[q];
          TcTask tk{};
          tk.Cb = T.p + toff;
          tk.slice_stride = ts;
          tk.ldcb = pad8(nn);
          tk.m = m;
          tk.n = nn;
          tk.nslices = NSL;
          g1.begin(tk);
          for (int np = 0; np < 4; ++np) {
            const int slot = n * 4 + np;
            const TRef& r = t.ref[beta][slot];
            if (!r.p) continue;
            const OpLayout& Lay = env.cls[r.cls];
            int qp, bl, sb;
            if (left) {
              qp = Lb.find(Lb.qa[q] - Lay.da, Lb.qb[q] - Lay.db);  // ql'
              if (qp < 0) continue;
              bl = Lay.blk_of_col[qp];
              if (bl < 0 || Lay.blocks[bl].rs != q) continue;
              sb = A.blk(qp, np);
              if (sb < 0 || A.blocks[sb].cs != j) continue;
            } else {
              qp = Rb.find(Lb.qa[j] + LQA[np], Lb.qb[j] + LQB[np]);  // qr'
              if (qp < 0) continue;
              bl = Lay.blk_of_col[qp];
              if (bl < 0 || Lay.blocks[bl].rs != q) continue;
              sb = A.blk(j, np);
              if (sb < 0 || A.blocks[sb].cs != qp) continue;
            }
            const int kk = ib.dim[qp];
            g1.term(smir.p + soff[sb], ss, pad8(kk), omir.p + mref[beta][slot] + boff[r.cls][bl], ms_, pad8(kk), kk,
                    mneg[beta][slot] != 0, NSL);
            fl += 2.0 * m * nn * kk;
          }
          if (g1.end()) {
            tpos[(size_t)n * no + j] = (long)toff;
            toff += (size_t)m * pad8(nn);
          }
        }
      const OpLayout& Lo = out.lay((int)beta);
      float* obase = f32_op((int)beta);
      for (const Block& B : Lo.blocks) {
        TcTask tk{};
        tk.C = obase + B.off;
        tk.ldc = B.cols;
        tk.m = B.rows;
        tk.n = B.cols;
        g2.begin(tk);
        for (int n = 0; n < 4; ++n) {
          int q, sb;
          if (left) {
            q = Lb.find(Rb.qa[B.rs] - LQA[n], Rb.qb[B.rs] - LQB[n]);  // ql of A^{n}[ql, qa]
            if (q < 0) continue;
            sb = A.blk(q, n);
            if (sb < 0 || A.blocks[sb].cs != B.rs) continue;
          } else {
            q = Rb.find(Lb.qa[B.rs] + LQA[n], Lb.qb[B.rs] + LQB[n]);  // qr of B^{n}[qb, qr]
            if (q < 0) continue;
            sb = A.blk(B.rs, n);
            if (sb < 0 || A.blocks[sb].cs != q) continue;
          }
          const long tp = tpos[(size_t)n * no + B.cs];
          if (tp < 0) continue;
          const int kk = ib.dim[q];
          g2.term(smir.p + soff[sb], ss, pad8(kk), T.p + tp, ts, pad8(kk), kk, false, NSL);
          fl += 2.0 * B.rows * B.cols * kk;
        }
        g2.end();
      }
    }
    c.other_flops_total += fl;
    DArr<int> err;
    err.alloc(1, c.stream);
    cuda_check(cudaMemsetAsync(err.p, 0, sizeof(int), c.stream), "memset");
    DArr<TcTile> t1, t2;
    DArr<TcTask> k1, k2;
    DArr<TcTerm> m1, m2;
    t1.upload(g1.tiles, c.stream);
    k1.upload(g1.tasks, c.stream);
    m1.upload(g1.terms, c.stream);
    t2.upload(g2.tiles, c.stream);
    k2.upload(g2.tasks, c.stream);
    m2.upload(g2.terms, c.stream);
    cuda_check(launch_gemm_bf16_tc(t1.p, (int)g1.tiles.size(), k1.p, m1.p, err.p, c.stream, NSL), "tc env stage 1");
    cuda_check(launch_gemm_bf16_tc(t2.p, (int)g2.tiles.size(), k2.p, m2.p, err.p, c.stream, NSL), "tc env stage 2");
    int h = 0;
    cuda_check(cudaMemcpyAsync(&h, err.p, sizeof(int), cudaMemcpyDeviceToHost, c.stream), "d2h");
    cuda_check(cudaStreamSynchronize(c.stream), "sync");
    if (h) throw Error(ST_ETIMEOUT, "tensor-core GEMM: a bounded wait ran out");
    b0 = b1;
  }
  for (size_t ci = 0; ci < out.cls.size(); ++ci) {
    const long n = (long)out.data[ci].n;
    if (n <= 0) continue;
    f32_to_f64_kernel<<<(unsigned)std::min<long>((n + 255) / 256, 152 * 16), 256, 0, c.stream>>>(f32[ci].p,
                                                                                                  out.data[ci].p, n);
    count_launches(1);
  }
  cuda_check(cudaGetLastError(), "f32 to f64");
  cuda_check(cudaStreamSynchronize(c.stream), "sync");
}

// ---------------------------------------------------------------- exact environment update

// Environment update (Eqs. leftrenorm/rightrenorm, prenormmatrix/prenormdec) on the
// tensor cores with FP64-level results: every FP64 block is scaled by a power of two and
// split into TM_EXACT_SLICES integer slices of 7 bits, exact in BF16; the products of two
// slices summed over a block's K (<= 128 columns, products <= 2^14) are exact integers in
// the FP32 accumulators; pairs of slices of one level i + j share a weight and accumulate
// together (still exact), and the levels are added with their powers of two in two-float
// (hi + lo) registers and stored in FP64.  Dropped pairs (i + j >= slices) and the
// remainder of the splitting are below 2^-42 of each block's largest element.
//   left : E1  T^T_beta[n1][j, ql] = sum_{n1'} At^{n1'}[j, ql'] Lt^{n1 n1'}[ql, ql']
//          E2  L'[qa, qa']        = sum_{n1} At^{n1}[qa, ql] T^T_beta[n1][qa', ql]
//   right: E1  T_beta[n2][j, qr]  = sum_{n2'} B^{n2'}[j, qr'] Rt^{n2 n2'}[qr, qr']
//          E2  R'[qb, qb']        = sum_{n2} B^{n2}[qb, qr] T_beta[n2][qb', qr]
constexpr int TM_EXACT_SLICES = 6;

namespace {

// matrices of one padded width (K dimension) holding blocks stacked by rows
struct WidthClasses {
  std::map<int, int> cls;  // width -> class
  std::vector<int> w;
  std::vector<long> rows, base;
  int of(int width) {
    auto it = cls.find(width);
    if (it != cls.end()) return it->second;
    const int c = (int)w.size();
    cls[width] = c;
    w.push_back(width);
    rows.push_back(0);
    base.push_back(0);
    return c;
  }
  long place(int c, int nrows) {  // row offset of a new block of nrows rows (padded to 16)
    const long r = rows[c];
    rows[c] += pad16(nrows);
    return r;
  }
  long finish() {
    long t = 0;
    for (size_t c = 0; c < w.size(); ++c) {
      base[c] = t;
      t += rows[c] * w[c];
    }
    return std::max<long>(t, 8);
  }
};

}  // namespace

void env_update_exact(Context& c, Tilde& t, const SiteT& A, int site, Env& out, bool left) {
  constexpr int NSL = TM_EXACT_SLICES;
  const auto& st = left ? c.mpo.bonds[site + 1] : c.mpo.bonds[site];
  const Bond& Lb = A.L;
  const Bond& Rb = A.R;
  Env& env = *t.env;
  const Bond& ob = left ? Rb : Lb;  // bond of the new operators
  const Bond& ib = left ? Lb : Rb;  // bond of the contracted index
  env_alloc(c, out, ob, st);
  const int no = ob.nsec();
  const int nmax = tm_max_n(TM_MODE_EXACT_F64, 1);
  std::vector<SplitJob> split1;  // site and operator blocks
  int nexpo = 0;
  // ---- site tensor: left At blocks [d(qr) x d(ql)], right B blocks [d(ql) x d(qr)]; K = columns
  WidthClasses sc;
  std::vector<int> s_cls(A.blocks.size()), s_exp(A.blocks.size());
  std::vector<long> s_row(A.blocks.size());
  for (size_t b = 0; b < A.blocks.size(); ++b) {
    const Block& B = A.blocks[b];
    const int rows = left ? B.cols : B.rows, kdim = left ? B.rows : B.cols;
    s_cls[b] = sc.of(pad16(kdim));
    s_row[b] = sc.place(s_cls[b], rows);
    s_exp[b] = nexpo++;
  }
  const long ss = sc.finish();
  DArr<__nv_bfloat16> smir;
  smir.alloc((size_t)ss * NSL, c.stream);
  cuda_check(cudaMemsetAsync(smir.p, 0, smir.n * sizeof(__nv_bfloat16), c.stream), "memset");
  for (size_t b = 0; b < A.blocks.size(); ++b) {
    const Block& B = A.blocks[b];
    const int w = sc.w[s_cls[b]];
    split1.push_back({A.d.p + B.off, smir.p + sc.base[s_cls[b]] + s_row[b] * w, ss, B.rows, B.cols, B.cols, w,
                      left ? B.cols : pad16(B.cols), left ? 1 : 0, s_exp[b], 1.0});
  }
  // ---- W-contracted operators: every distinct (operator, coefficient), all blocks; K = columns
  WidthClasses oc;
  struct KeyHash {
    size_t operator()(const std::pair<const double*, double>& kk) const {
      uint64_t b;
      std::memcpy(&b, &kk.second, sizeof b);
      return std::hash<uint64_t>()((uint64_t)(uintptr_t)kk.first * 0x9e3779b97f4a7c15ULL ^ b);
    }
  };
  std::unordered_map<std::pair<const double*, double>, int, KeyHash> mid_of;
  std::vector<std::vector<long>> m_row;  // per mirror, per block
  std::vector<std::vector<int>> m_exp;
  std::vector<int> m_cls_of_ref;
  struct PendO {
    const double* src;
    int cls;
    long row;
    int rows, cols, ex;
    double coef;
  };
  std::vector<PendO> opend;
  std::vector<std::array<int, 16>> mref(st.size());
  for (size_t beta = 0; beta < st.size(); ++beta)
    for (int nn = 0; nn < 16; ++nn) {
      mref[beta][nn] = -1;
      const TRef& r = t.ref[beta][nn];
      if (!r.p) continue;
      auto key = std::make_pair(r.p, r.coef);
      auto it = mid_of.find(key);
      if (it == mid_of.end()) {
        const int id = (int)m_row.size();
        it = mid_of.emplace(key, id).first;
        const OpLayout& L = env.cls[r.cls];
        m_row.emplace_back(L.blocks.size());
        m_exp.emplace_back(L.blocks.size());
        for (size_t b = 0; b < L.blocks.size(); ++b) {
          const Block& B = L.blocks[b];
          const int cl = oc.of(pad16(B.cols));
          m_row[id][b] = oc.place(cl, B.rows);
          m_exp[id][b] = nexpo++;
          opend.push_back({r.p + B.off, cl, m_row[id][b], B.rows, B.cols, m_exp[id][b], r.coef});
        }
      }
      mref[beta][nn] = it->second;
    }
  const long os = oc.finish();
  DArr<__nv_bfloat16> omir;
  omir.alloc((size_t)os * NSL, c.stream);
  cuda_check(cudaMemsetAsync(omir.p, 0, omir.n * sizeof(__nv_bfloat16), c.stream), "memset");
  for (const PendO& po : opend) {
    const int w = oc.w[po.cls];
    split1.push_back({po.src, omir.p + oc.base[po.cls] + po.row * w, os, po.rows, po.cols, po.cols, w, po.cols, 0,
                      po.ex, po.coef});
  }
  // ---- intermediate T blocks (FP64) per (beta, n, j): d(j) x d(q) with q the inner sector
  auto inner_of = [&](size_t beta, int n, int j) -> int {
    if (left) return Lb.find(Rb.qa[j] + st[beta].dna - LQA[n], Rb.qb[j] + st[beta].dnb - LQB[n]);
    return Rb.find(Lb.qa[j] + st[beta].dna + LQA[n], Lb.qb[j] + st[beta].dnb + LQB[n]);
  };
  // the source terms (site block, mirror, operator block) of the T block (beta, n, j)
  auto sources = [&](size_t beta, int n, int j, int q, std::vector<std::array<int, 3>>& src, double& fl) {
    src.clear();
    for (int np = 0; np < 4; ++np) {
      const int slot = n * 4 + np;
      const TRef& r = t.ref[beta][slot];
      if (!r.p) continue;
      const OpLayout& Lay = env.cls[r.cls];
      int qp, bl, sb;
      if (left) {
        qp = Lb.find(Lb.qa[q] - Lay.da, Lb.qb[q] - Lay.db);
        if (qp < 0) continue;
        bl = Lay.blk_of_col[qp];
        if (bl < 0 || Lay.blocks[bl].rs != q) continue;
        sb = A.blk(qp, np);
        if (sb < 0 || A.blocks[sb].cs != j) continue;
      } else {
        qp = Rb.find(Lb.qa[j] + LQA[np], Lb.qb[j] + LQB[np]);
        if (qp < 0) continue;
        bl = Lay.blk_of_col[qp];
        if (bl < 0 || Lay.blocks[bl].rs != q) continue;
        sb = A.blk(j, np);
        if (sb < 0 || A.blocks[sb].cs != qp) continue;
      }
      src.push_back({sb, mref[beta][slot], bl});
      fl += 2.0 * ob.dim[j] * ib.dim[q] * ib.dim[qp];
    }
  };
  // chunks of bond states whose T blocks (FP64 + slices, 18 bytes per element) fit the budget
  std::vector<size_t> tsz(st.size(), 0);
  for (size_t beta = 0; beta < st.size(); ++beta)
    for (int n = 0; n < 4; ++n)
      for (int j = 0; j < no; ++j) {
        const int q = inner_of(beta, n, j);
        if (q >= 0) tsz[beta] += (size_t)pad16(ob.dim[j]) * pad16(ib.dim[q]);
      }
  const size_t budget = std::max<size_t>(1, (size_t)c.chunk_budget_mb * (1u << 20) / (8 + 2 * NSL));
  // split of the site and operator blocks (shared by all chunks)
  const int nexpo_fixed = nexpo;
  int max_texp = 0;
  for (size_t b0 = 0, b1; b0 < st.size(); b0 = b1) {
    size_t tot = 0;
    for (b1 = b0; b1 < st.size() && (b1 == b0 || tot + tsz[b1] <= budget); ++b1) tot += tsz[b1];
    int cnt = 0;
    for (size_t beta = b0; beta < b1; ++beta)
      for (int n = 0; n < 4; ++n)
        for (int j = 0; j < no; ++j) cnt += inner_of(beta, n, j) >= 0;
    max_texp = std::max(max_texp, cnt);
  }
  DArr<int> expo;
  expo.alloc(std::max(nexpo_fixed + max_texp, 1), c.stream);
  DArr<int> err;
  err.alloc(1, c.stream);
  cuda_check(cudaMemsetAsync(err.p, 0, sizeof(int), c.stream), "memset");
  DArr<SplitJob> dj1;
  dj1.upload(split1, c.stream);
  for (const SplitJob& j : split1)
    if (j.rows < 1 || j.cols < 1 || j.expo < 0 || j.expo >= nexpo_fixed) throw Error(ST_ECUDA, "internal: split job");
  cuda_check(launch_split_exact(dj1.p, (int)split1.size(), NSL, expo.p, c.stream), "exact split");
  // tensor maps of the site and operator classes (per slice; operators per box height)
  std::vector<CUtensorMap> maps;
  auto add_map = [&](const DArr<__nv_bfloat16>& buf, long off, long stride, long rows, int w, int box) {
    const int first = (int)maps.size();
    for (int sl = 0; sl < NSL; ++sl) {
      const long o = off + sl * stride;
      if (rows < 1 || o < 0 || o % 8 || (size_t)(o + rows * w) > buf.n)
        throw Error(ST_ECUDA, "internal: tensor map outside its buffer");
      CUtensorMap m;
      if (!encode_bf16_map(&m, buf.p + o, (uint64_t)rows, (uint64_t)w, (uint64_t)w, (uint32_t)box))
        throw Error(ST_ECUDA, "cuTensorMapEncodeTiled failed");
      maps.push_back(m);
    }
    return first;
  };
  std::vector<int> smap(sc.w.size(), -1);
  for (size_t k = 0; k < sc.w.size(); ++k)
    if (sc.rows[k] > 0) smap[k] = add_map(smir, sc.base[k], ss, sc.rows[k], sc.w[k], 128);
  std::vector<std::vector<int>> omap(oc.w.size(), std::vector<int>(nmax / 16 + 1, -1));
  for (size_t k = 0; k < oc.w.size(); ++k)
    if (oc.rows[k] > 0)
      for (int h = 16; h <= nmax; h += 16) omap[k][h / 16] = add_map(omir, oc.base[k], os, oc.rows[k], oc.w[k], h);
  const size_t nfixed_maps = maps.size();
  double fl = 0;
  std::vector<std::array<int, 3>> src;
  for (size_t b0 = 0, b1; b0 < st.size(); b0 = b1) {
    size_t tot = 0;
    for (b1 = b0; b1 < st.size() && (b1 == b0 || tot + tsz[b1] <= budget); ++b1) tot += tsz[b1];
    maps.resize(nfixed_maps);
    // T layout of this chunk: FP64 blocks, their slices by width class, their exponents
    const size_t nb = b1 - b0;
    std::vector<long> tpos(nb * 4 * no, -1), t_row(nb * 4 * no, -1);
    std::vector<int> t_cls(nb * 4 * no, -1), t_exp(nb * 4 * no, -1);
    WidthClasses tcw;
    long ttot = 0;
    int nte = nexpo_fixed;
    struct E1 {
      size_t tix;
      int r0, c0, m_valid, nvalid, cols;
      size_t s0, s1;  // range in srcs
    };
    std::vector<E1> e1x;
    std::vector<std::array<int, 3>> srcs;
    for (size_t beta = b0; beta < b1; ++beta)
      for (int n = 0; n < 4; ++n)
        for (int j = 0; j < no; ++j) {
          const int q = inner_of(beta, n, j);
          if (q < 0) continue;
          sources(beta, n, j, q, src, fl);
          if (src.empty()) continue;
          const size_t tix = ((beta - b0) * 4 + n) * no + j;
          const int rows = ob.dim[j], cols = ib.dim[q];
          tpos[tix] = ttot;
          ttot += (long)rows * cols;
          t_cls[tix] = tcw.of(pad16(cols));
          t_row[tix] = tcw.place(t_cls[tix], rows);
          t_exp[tix] = nte++;
          const size_t s0 = srcs.size();
          srcs.insert(srcs.end(), src.begin(), src.end());
          for (int r0 = 0; r0 < rows; r0 += 128)
            for (int c0 = 0; c0 < cols; c0 += nmax)
              e1x.push_back({tix, r0, c0, std::min(128, rows - r0), std::min(nmax, cols - c0), cols, s0, srcs.size()});
        }
    const long ts = tcw.finish();
    DArr<double> T64;
    T64.alloc(std::max<long>(ttot, 1), c.stream);
    DArr<__nv_bfloat16> tmir;
    tmir.alloc((size_t)ts * NSL, c.stream);
    cuda_check(cudaMemsetAsync(tmir.p, 0, tmir.n * sizeof(__nv_bfloat16), c.stream), "memset");
    std::vector<std::vector<int>> tmap(tcw.w.size(), std::vector<int>(nmax / 16 + 1, -1));
    for (size_t k = 0; k < tcw.w.size(); ++k)
      if (tcw.rows[k] > 0)
        for (int h = 16; h <= nmax; h += 16) tmap[k][h / 16] = add_map(tmir, tcw.base[k], ts, tcw.rows[k], tcw.w[k], h);
    // E1 tiles: T block (rows, <= 64 columns) per tile; contractions cut into <= 128 columns
    std::vector<TmTile> e1t;
    std::vector<TmTerm> e1m;
    for (const E1& x : e1x) {
      TmTile tl{};
      tl.t0 = (int)e1m.size();
      tl.m_valid = x.m_valid;
      tl.nvalid = x.nvalid;
      tl.n = pad16(x.nvalid);
      for (size_t si = x.s0; si < x.s1; ++si) {
        const auto& sr = srcs[si];
        const Block& SB = A.blocks[sr[0]];
        const int kdim = left ? SB.rows : SB.cols;
        for (int kc = 0; kc < pad16(kdim); kc += 128)
          e1m.push_back({smap[s_cls[sr[0]]], omap[oc.cls[pad16(kdim)]][tl.n / 16], kc, (int)(s_row[sr[0]] + x.r0), kc,
                         (int)(m_row[sr[1]][sr[2]] + x.c0), std::min(128, pad16(kdim) - kc), NSL << 4, s_exp[sr[0]],
                         m_exp[sr[1]][sr[2]]});
      }
      tl.t1 = (int)e1m.size();
      tl.ldo = x.cols;
      tl.out_off = tpos[x.tix] + (long)x.r0 * x.cols + x.c0;
      e1t.push_back(tl);
    }
    // split of this chunk's T blocks
    std::vector<SplitJob> split2;
    for (size_t tix = 0; tix < tpos.size(); ++tix) {
      if (tpos[tix] < 0) continue;
      const int j = (int)(tix % no), n = (int)((tix / no) % 4);
      const size_t beta = b0 + tix / ((size_t)4 * no);
      const int rows = ob.dim[j], cols = ib.dim[inner_of(beta, n, j)];
      const int w = tcw.w[t_cls[tix]];
      split2.push_back({T64.p + tpos[tix], tmir.p + tcw.base[t_cls[tix]] + t_row[tix] * w, ts, rows, cols, cols, w,
                        pad16(cols), 0, t_exp[tix], 1.0});
    }
    // E2 tiles: every block of every new operator of the chunk, per output class
    std::vector<std::vector<TmTile>> e2t(out.cls.size());
    std::vector<TmTerm> e2m;
    std::vector<std::array<int, 2>> s2;
    for (size_t beta = b0; beta < b1; ++beta) {
      const OpLayout& Lo = out.lay((int)beta);
      const int oc_ = out.st_cls[(int)beta];
      const long obase = (long)(out.op((int)beta) - out.data[oc_].p);
      for (const Block& B : Lo.blocks) {
        s2.clear();
        for (int n = 0; n < 4; ++n) {
          int q, sb;
          if (left) {
            q = Lb.find(Rb.qa[B.rs] - LQA[n], Rb.qb[B.rs] - LQB[n]);
            if (q < 0) continue;
            sb = A.blk(q, n);
            if (sb < 0 || A.blocks[sb].cs != B.rs) continue;
          } else {
            q = Rb.find(Lb.qa[B.rs] + LQA[n], Lb.qb[B.rs] + LQB[n]);
            if (q < 0) continue;
            sb = A.blk(B.rs, n);
            if (sb < 0 || A.blocks[sb].cs != q) continue;
          }
          const size_t tix = ((beta - b0) * 4 + n) * no + B.cs;
          if (tpos[tix] < 0) continue;
          s2.push_back({sb, (int)tix});
          fl += 2.0 * B.rows * B.cols * ib.dim[q];
        }
        if (s2.empty()) continue;
        for (int r0 = 0; r0 < B.rows; r0 += 128)
          for (int c0 = 0; c0 < B.cols; c0 += nmax) {
            TmTile tl{};
            tl.t0 = (int)e2m.size();
            tl.m_valid = std::min(128, B.rows - r0);
            tl.nvalid = std::min(nmax, B.cols - c0);
            tl.n = pad16(tl.nvalid);
            for (const auto& sr : s2) {
              const Block& SB = A.blocks[sr[0]];
              const int kdim = left ? SB.rows : SB.cols;
              for (int kc = 0; kc < pad16(kdim); kc += 128)
                e2m.push_back({smap[s_cls[sr[0]]], tmap[t_cls[(size_t)sr[1]]][tl.n / 16], kc, (int)(s_row[sr[0]] + r0),
                               kc, (int)(t_row[(size_t)sr[1]] + c0), std::min(128, pad16(kdim) - kc), NSL << 4,
                               s_exp[sr[0]], t_exp[(size_t)sr[1]]});
            }
            tl.t1 = (int)e2m.size();
            tl.ldo = B.cols;
            tl.out_off = obase + B.off + (long)r0 * B.cols + c0;
            e2t[(size_t)oc_].push_back(tl);
          }
      }
    }
    // bounds of every output, term and split job before anything runs
    for (const TmTile& tl : e1t)
      if (tl.out_off < 0 || tl.out_off + (long)(tl.m_valid - 1) * tl.ldo + tl.nvalid > (long)T64.n || tl.n > nmax ||
          tl.nvalid > tl.n || tl.t1 <= tl.t0)
        throw Error(ST_ECUDA, "internal: exact stage-1 tile");
    for (size_t ci = 0; ci < e2t.size(); ++ci)
      for (const TmTile& tl : e2t[ci])
        if (tl.out_off < 0 || (size_t)(tl.out_off + (long)(tl.m_valid - 1) * tl.ldo + tl.nvalid) > out.data[ci].n ||
            tl.n > nmax || tl.nvalid > tl.n || tl.t1 <= tl.t0)
          throw Error(ST_ECUDA, "internal: exact stage-2 tile");
    auto check_m = [&](const std::vector<TmTerm>& mm) {
      for (const TmTerm& m : mm)
        if (m.amap < 0 || m.amap + NSL > (int)maps.size() || m.bmap < 0 || m.bmap + NSL > (int)maps.size() ||
            m.k < 16 || m.k % 16 || m.k > 128 || m.ax % 16 || m.ea < 0 || m.ea >= nte || m.eb < 0 || m.eb >= nte ||
            ((m.neg >> 4) & 15) != NSL)
          throw Error(ST_ECUDA, "internal: exact term");
    };
    check_m(e1m);
    check_m(e2m);
    for (const SplitJob& j : split2)
      if (j.rows < 1 || j.cols < 1 || j.expo < nexpo_fixed || j.expo >= nte) throw Error(ST_ECUDA, "internal: split job");
    // run: E1, split T, E2 (one launch per output class of the new operators)
    DArr<CUtensorMap> dmaps;
    dmaps.upload(maps, c.stream);
    DArr<TmTile> d1t;
    DArr<TmTerm> d1m, d2m;
    // copy lists of every launch; each piece reads through one of this update's maps
    // copy lists of every launch (their pieces follow from the terms checked above)
    TmaPlan::Lists dl1;
    dl1.plan(TM_MODE_EXACT_F64, 1, e1t, e1m, c.stream);
    d1t.upload(e1t, c.stream);
    d1m.upload(e1m, c.stream);
    dl1.fill(TM_MODE_EXACT_F64, 1, d1t.p, (int)e1t.size(), d1m.p, c.stream);
    cuda_check(launch_gemm_exact(d1t.p, (int)e1t.size(), d1m.p, dmaps.p, T64.p, err.p, c.stream, dl1.dev(), expo.p),
               "exact stage 1");
    DArr<SplitJob> dj2;
    dj2.upload(split2, c.stream);
    cuda_check(launch_split_exact(dj2.p, (int)split2.size(), NSL, expo.p, c.stream), "exact split of T");
    d2m.upload(e2m, c.stream);
    std::vector<DArr<TmTile>> d2t(out.cls.size());
    std::vector<TmaPlan::Lists> dl2(out.cls.size());
    for (size_t ci = 0; ci < out.cls.size(); ++ci) {
      if (e2t[ci].empty()) continue;
      dl2[ci].plan(TM_MODE_EXACT_F64, 1, e2t[ci], e2m, c.stream);
      d2t[ci].upload(e2t[ci], c.stream);
      dl2[ci].fill(TM_MODE_EXACT_F64, 1, d2t[ci].p, (int)e2t[ci].size(), d2m.p, c.stream);
      cuda_check(launch_gemm_exact(d2t[ci].p, (int)e2t[ci].size(), d2m.p, dmaps.p, out.data[ci].p, err.p, c.stream,
                                   dl2[ci].dev(), expo.p),
                 "exact stage 2");
    }
    // the host lists and the chunk's buffers must outlive the launches
    cuda_check(cudaStreamSynchronize(c.stream), "sync");
  }
  c.other_flops_total += fl;
  int h = 0;
  cuda_check(cudaMemcpyAsync(&h, err.p, sizeof(int), cudaMemcpyDeviceToHost, c.stream), "d2h");
  cuda_check(cudaStreamSynchronize(c.stream), "sync");
  if (h) throw Error(ST_ETIMEOUT, "tensor-core GEMM: a bounded wait ran out");
}

// ---------------------------------------------------------------- batched sigma

// Several independent two-site problems (each prepared in a tensor-core precision
// on the same device) fused into one launch per stage and chunk: the tile and term lists, tensor
// maps and row maps are concatenated, so one persistent kernel walks the tiles of
// every problem (one launch per slice count where the problems differ in it).  Optionally the
// whole sequence (conversions, stage launches, gathers) is captured once in a CUDA graph and
// replayed.  (Eight problems, three slices, device time batched and one by one: K 12-20, M 64-256
// 1.03 and 1.20 ms; K 16-32, M 362-992 17.4 and 18.2 ms.)
struct BatchPlan {
  std::vector<Context*> ctx;
  cudaStream_t stream = nullptr;
  struct Launch {
    int nsl = 1, n1 = 0, n2 = 0, nz = 0, n_a1 = 0;
    long zmax = 0, a1_maxel = 0;
    DArr<TmTile> t1, t2;
    DArr<TmTerm> m1, m2;
    TmaPlan::Lists l1, l2;
    DArr<ZeroJob> z;
    DArr<GroupJob> a1;
    void *out1 = nullptr, *out2 = nullptr;  // what the tiles' offsets count from
  };
  std::vector<Launch> launches;  // chunk by chunk
  DArr<CUtensorMap> maps;
  DArr<long> rowmap;
  DArr<GroupJob> conv[3];  // by slice count
  DArr<UnconvJob> unconv;
  int nconv[3] = {0, 0, 0}, nunconv = 0;
  long conv_maxel = 0, unconv_maxel = 0;
  DArr<int> err;
  cudaGraph_t graph = nullptr;
  cudaGraphExec_t exec = nullptr;
  long graph_launches = 0, graph_tc_launches = 0;  // kernels in one replay of the graph
  double flops = 0;
  ~BatchPlan() {
    if (exec) cudaGraphExecDestroy(exec);
    if (graph) cudaGraphDestroy(graph);
  }
};

// Chunk ch of the problems with nsl slices, in groups that share a launch per stage.  With two or
// three slices a launch's ring follows from its widest tile and has to hold its longest term, which
// may come from different problems: a problem joins the first group whose ring then still does.
static std::vector<std::vector<size_t>> batch_groups(const BatchPlan& b, size_t ch, int nsl) {
  struct Need {
    int n[2] = {16, 16}, k[2] = {16, 16};  // widest tile and longest term of the stages
  };
  std::vector<std::vector<size_t>> groups;
  std::vector<Need> needs;
  for (size_t p = 0; p < b.ctx.size(); ++p) {
    const TmaPlan& tp = *b.ctx[p]->plan.tm;
    if (tp.nsl != nsl || ch >= tp.chunks.size()) continue;
    const TmaPlan::Chunk& c = tp.chunks[ch];
    Need own;
    for (const TmTile& t : c.ht1) own.n[0] = std::max(own.n[0], t.n);
    for (const TmTile& t : c.ht2) own.n[1] = std::max(own.n[1], t.n);
    for (const TmTerm& m : c.hm1) own.k[0] = std::max(own.k[0], m.k);
    for (const TmTerm& m : c.hm2) own.k[1] = std::max(own.k[1], m.k);
    size_t g = 0;
    for (; g < groups.size(); ++g) {
      Need both = needs[g];
      bool fits = true;
      for (int i = 0; i < 2; ++i) {
        both.n[i] = std::max(both.n[i], own.n[i]);
        both.k[i] = std::max(both.k[i], own.k[i]);
        fits = fits && (nsl == 1 || both.k[i] / TM_PIECE_COLS <= tm_term_pieces(nsl, both.n[i]));
      }
      if (!fits) continue;
      needs[g] = both;
      break;
    }
    if (g == groups.size()) {
      groups.emplace_back();
      needs.push_back(own);
    }
    groups[g].push_back(p);
  }
  return groups;
}

// chunk ch of the problems `group` (of nsl slices) as one launch per stage; map0, row0: every problem's
// first tensor map and row-map entry in the concatenated arrays
static void batch_launch(BatchPlan& b, size_t ch, int nsl, const std::vector<size_t>& group,
                         const std::vector<int>& map0, const std::vector<long>& row0) {
  std::vector<TmTile> t1, t2;
  std::vector<TmTerm> m1, m2;
  std::vector<ZeroJob> zj;
  std::vector<GroupJob> aj;
  BatchPlan::Launch L;
  L.nsl = nsl;
  auto add = [&](std::vector<TmTile>& tiles, std::vector<TmTerm>& terms, const std::vector<TmTile>& pt,
                 const std::vector<TmTerm>& pm, int map, auto&& rebase) {
    const int t0 = (int)terms.size();
    for (TmTile t : pt) {
      t.t0 += t0;
      t.t1 += t0;
      rebase(t);
      tiles.push_back(t);
    }
    for (TmTerm m : pm) {
      m.amap += map;
      m.bmap += map;
      terms.push_back(m);
    }
  };
  for (size_t p : group) {
    const TmaPlan& tp = *b.ctx[p]->plan.tm;
    const TmaPlan::Chunk& c = tp.chunks[ch];
    if (!L.out1) {
      L.out1 = tp.xt.p;
      L.out2 = tp.sig_t.p;
    }
    const long dx = ((intptr_t)tp.xt.p - (intptr_t)L.out1) / (long)sizeof(__nv_bfloat16);
    const long ds = ((intptr_t)tp.sig_t.p - (intptr_t)L.out2) / (long)sizeof(float);
    add(t1, m1, c.ht1, c.hm1, map0[p], [&](TmTile& t) {
      t.rowmap_off += row0[p];
      t.xbase += dx;
    });
    add(t2, m2, c.ht2, c.hm2, map0[p], [&](TmTile& t) { t.out_off += ds; });
    zj.insert(zj.end(), c.hz.begin(), c.hz.end());
    L.zmax = std::max(L.zmax, c.zmax);
    aj.insert(aj.end(), c.ha1.begin(), c.ha1.end());
    L.a1_maxel = std::max(L.a1_maxel, c.a1_maxel);
  }
  if (t1.empty() && t2.empty()) return;
  longest_first(t1, m1);
  longest_first(t2, m2);
  L.l1.plan(TM_MODE_STORE_BF16, nsl, t1, m1, b.stream);
  L.l2.plan(TM_MODE_REDUCE_F32, nsl, t2, m2, b.stream);
  L.n1 = (int)t1.size();
  L.n2 = (int)t2.size();
  L.nz = (int)zj.size();
  L.t1.upload(t1, b.stream);
  L.m1.upload(m1, b.stream);
  L.t2.upload(t2, b.stream);
  L.m2.upload(m2, b.stream);
  L.z.upload(zj, b.stream);
  L.n_a1 = (int)aj.size();
  L.a1.upload(aj, b.stream);
  L.l1.fill(TM_MODE_STORE_BF16, nsl, L.t1.p, L.n1, L.m1.p, b.stream);
  L.l2.fill(TM_MODE_REDUCE_F32, nsl, L.t2.p, L.n2, L.m2.p, b.stream);
  cuda_check(cudaStreamSynchronize(b.stream), "sync");
  b.launches.push_back(std::move(L));
}

BatchPlan* batch_create(const std::vector<Context*>& ctxs) {
  std::unique_ptr<BatchPlan, void (*)(BatchPlan*)> b(new BatchPlan(), batch_free);
  b->ctx = ctxs;
  b->stream = ctxs[0]->stream;
  size_t nch = 0;
  std::vector<GroupJob> cj[3];
  std::vector<UnconvJob> uj;
  std::vector<CUtensorMap> maps;
  std::vector<long> rowmap;
  std::vector<int> map0;
  std::vector<long> row0;
  for (Context* c : ctxs) {
    if (c->prepared < 0 || !c->plan.tm || c->plan.tm->precision > 3)
      throw Error(ST_ESTATE, "batched sigma: every context must be prepared in precision 1, 2 or 3");
    const TmaPlan& tp = *c->plan.tm;
    if (!tp.host_copies) throw Error(ST_ESTATE, "batched sigma: plan was built without host copies");
    nch = std::max(nch, tp.chunks.size());
    cj[tp.nsl - 1].insert(cj[tp.nsl - 1].end(), tp.h_psi_jobs.begin(), tp.h_psi_jobs.end());
    uj.insert(uj.end(), tp.h_sig_jobs.begin(), tp.h_sig_jobs.end());
    map0.push_back((int)maps.size());
    row0.push_back((long)rowmap.size());
    maps.insert(maps.end(), tp.hmaps.begin(), tp.hmaps.end());
    rowmap.insert(rowmap.end(), tp.hrowmap.begin(), tp.hrowmap.end());
    b->conv_maxel = std::max(b->conv_maxel, tp.psi_maxel);
    b->unconv_maxel = std::max(b->unconv_maxel, tp.sig_maxel);
    b->flops += c->plan.flops;
  }
  b->maps.upload(maps, b->stream);
  b->rowmap.upload(rowmap, b->stream);
  for (size_t ch = 0; ch < nch; ++ch)
    for (int nsl = 1; nsl <= 3; ++nsl)
      for (const auto& group : batch_groups(*b, ch, nsl)) batch_launch(*b, ch, nsl, group, map0, row0);
  for (int i = 0; i < 3; ++i) {
    b->conv[i].upload(cj[i], b->stream);
    b->nconv[i] = (int)cj[i].size();
  }
  b->unconv.upload(uj, b->stream);
  b->nunconv = (int)uj.size();
  b->err.alloc(1, b->stream);
  cuda_check(cudaMemsetAsync(b->err.p, 0, sizeof(int), b->stream), "memset");
  cuda_check(cudaStreamSynchronize(b->stream), "sync");
  return b.release();
}

void batch_free(BatchPlan* b) {
  if (b && b->stream) cudaStreamSynchronize(b->stream);
  delete b;
}
double batch_flops(const BatchPlan* b) { return b->flops; }

// the device work of one batched sigma (plan.in -> plan.out of every problem)
static void batch_enqueue(BatchPlan& b) {
  cudaStream_t s = b.stream;
  for (Context* c : b.ctx) {
    TmaPlan& tp = *c->plan.tm;
    cuda_check(cudaMemsetAsync(tp.sig_t.p, 0, tp.sig_total * sizeof(float), s), "memset");
  }
  for (int i = 0; i < 3; ++i)
    if (b.nconv[i]) launch_conv_groups(b.conv[i], b.nconv[i], i + 1, b.conv_maxel, s);
  for (const BatchPlan::Launch& L : b.launches) {
    if (L.n_a1) launch_conv_groups(L.a1, L.n_a1, L.nsl, L.a1_maxel, s);
    if (L.nz) launch_zero(L.z.p, L.nz, L.zmax, s);
    cuda_check(launch_gemm_slices(TM_MODE_STORE_BF16, L.nsl, L.t1.p, L.n1, b.maps.p, b.rowmap.p, L.out1, b.err.p, s,
                                  L.l1.dev()),
               "batch stage 1");
    cuda_check(launch_gemm_slices(TM_MODE_REDUCE_F32, L.nsl, L.t2.p, L.n2, b.maps.p, nullptr, L.out2, b.err.p, s,
                                  L.l2.dev()),
               "batch stage 2");
  }
  if (b.nunconv) launch_unconv(b.unconv.p, b.nunconv, b.unconv_maxel, s);
}

float batch_sigma(BatchPlan& b, const double* const* psi, double* const* sigma, bool use_graph) {
  cudaStream_t s = b.stream;
  for (size_t p = 0; p < b.ctx.size(); ++p) {
    SigmaPlan& pl = b.ctx[p]->plan;
    cuda_check(cudaMemcpyAsync(pl.in.p, psi[p], pl.psi.nnz * sizeof(double), cudaMemcpyDeviceToDevice, s), "d2d");
  }
  cudaEvent_t e0, e1;
  cuda_check(cudaEventCreate(&e0), "event");
  cuda_check(cudaEventCreate(&e1), "event");
  cuda_check(cudaEventRecord(e0, s), "record");
  if (use_graph && b.exec) {
    cuda_check(cudaGraphLaunch(b.exec, s), "graph launch");
    count_launches(b.graph_launches);
    count_tc_launches(b.graph_tc_launches);
  } else {
    batch_enqueue(b);
  }
  cuda_check(cudaEventRecord(e1, s), "record");
  if (use_graph && !b.exec) {
    // captured after one eager pass (which set up every launch attribute); the
    // captured work does not run now, later calls replay it
    const long l0 = launch_count(), t0 = tc_launch_count();
    cuda_check(cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal), "begin capture");
    batch_enqueue(b);
    cuda_check(cudaStreamEndCapture(s, &b.graph), "end capture");
    // captured launches run only when the graph is replayed: count them there
    b.graph_launches = launch_count() - l0;
    b.graph_tc_launches = tc_launch_count() - t0;
    count_launches(-b.graph_launches);
    count_tc_launches(-b.graph_tc_launches);
    cuda_check(cudaGraphInstantiate(&b.exec, b.graph, 0), "graph instantiate");
  }
  for (size_t p = 0; p < b.ctx.size(); ++p) {
    SigmaPlan& pl = b.ctx[p]->plan;
    cuda_check(cudaMemcpyAsync(sigma[p], pl.out.p, pl.psi.nnz * sizeof(double), cudaMemcpyDeviceToDevice, s), "d2d");
  }
  cuda_check(cudaEventSynchronize(e1), "sync");
  float ms = 0;
  cudaEventElapsedTime(&ms, e0, e1);
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  int h = 0;
  cuda_check(cudaMemcpy(&h, b.err.p, sizeof(int), cudaMemcpyDeviceToHost), "d2h");
  if (h) throw Error(ST_ETIMEOUT, "tensor-core GEMM: a bounded wait ran out");
  cuda_check(cudaStreamSynchronize(s), "sync");
  return ms;
}


// ---------------------------------------------------------------- blocking sums on the tensor cores

// out_i = sum_j coef_ij Op_j for the operators Op_j of one class (Sec. "Efficient
// implementation of expectation values": the W contraction with the renormalised
// operators) as one GEMM per class: A = the class's operators transposed into BF16
// slices (element-major, operator index contiguous), B = the coefficient matrix in BF16
// slices, FP32 accumulation, the result gathered into the FP64 outputs.  Three slices
// carry ~24 significant bits, so the sums have about FP32 accuracy.
void combos_tc(Context& c, Env& env, const std::vector<ComboOut>& outs, const std::vector<ComboTerm>& terms,
               const std::vector<int>& out_cls) {
  const int nsl = 3;
  DArr<int> err;
  err.alloc(1, c.stream);
  cuda_check(cudaMemsetAsync(err.p, 0, sizeof(int), c.stream), "memset");
  std::vector<std::vector<size_t>> by_cls(env.cls.size());
  for (size_t i = 0; i < outs.size(); ++i) by_cls[(size_t)out_cls[i]].push_back(i);
  for (size_t cls = 0; cls < env.cls.size(); ++cls) {
    const std::vector<size_t>& mine = by_cls[cls];
    if (mine.empty()) continue;
    const long nnz = env.cls[cls].nnz;
    const int K = env.nslot[cls];
    const int Kp = pad8(K);
    const int S = (int)mine.size();
    if (nnz <= 0 || K <= 0) continue;
    if (nnz > (long)std::numeric_limits<int>::max())
      throw Error(ST_EINVAL, "tensor-core blocking sums: operator class too large");
    const double* base = env.data[cls].p;
    // A: operators transposed, [nnz x Kp] per slice (padding columns zero)
    DArr<__nv_bfloat16> at, bt;
    at.alloc((size_t)nnz * Kp * nsl, c.stream);
    cuda_check(cudaMemsetAsync(at.p, 0, at.n * sizeof(__nv_bfloat16), c.stream), "memset");
    std::vector<ConvJob> jobs;
    jobs.reserve((size_t)K + 1);
    for (int j = 0; j < K; ++j)
      jobs.push_back({base + (long)j * nnz, at.p + j, nnz * Kp, (int)nnz, 1, 1, Kp, nsl, 1.0, 1});
    // B: coefficients [S x Kp] (a repeated operator in one sum adds up)
    std::vector<double> coef((size_t)S * Kp, 0.0);
    for (int sidx = 0; sidx < S; ++sidx) {
      const ComboOut& o = outs[mine[(size_t)sidx]];
      for (int t = o.t0; t < o.t1; ++t) {
        const long d = (long)(terms[(size_t)t].in - base);
        if (d < 0 || d % nnz != 0 || d / nnz >= K)
          throw Error(ST_ECUDA, "internal: blocking-sum term outside its operator class");
        coef[(size_t)sidx * Kp + (size_t)(d / nnz)] += terms[(size_t)t].coef;
      }
    }
    DArr<double> coef_d;
    coef_d.upload(coef, c.stream);
    bt.alloc((size_t)S * Kp * nsl, c.stream);
    jobs.push_back({coef_d.p, bt.p, (long)S * Kp, S, Kp, Kp, Kp, nsl, 1.0, Kp});
    {
      DArr<ConvJob> dj;
      dj.upload(jobs, c.stream);
      launch_conv(dj, (int)jobs.size(), std::max<long>(nnz, (long)S * Kp), c.stream);
    }
    // C^T [S x nnz] in FP32: element (e, i) of the product goes to ct[i * nnz + e]
    DArr<float> ct;
    ct.alloc((size_t)S * nnz, c.stream);
    TcBuilder g;
    TcTask task{};
    task.C = ct.p;
    task.ldc = (int)nnz;
    task.m = (int)nnz;
    task.n = S;
    task.beta = 0;
    task.trans = 1;
    g.begin(task);
    g.term(at.p, nnz * Kp, Kp, bt.p, (long)S * Kp, Kp, K, false, nsl);
    g.end();
    DArr<TcTile> d_tiles;
    DArr<TcTask> d_tasks;
    DArr<TcTerm> d_terms;
    d_tiles.upload(g.tiles, c.stream);
    d_tasks.upload(g.tasks, c.stream);
    d_terms.upload(g.terms, c.stream);
    cuda_check(launch_gemm_bf16_tc(d_tiles.p, (int)g.tiles.size(), d_tasks.p, d_terms.p, err.p, c.stream, nsl),
               "tc blocking sums");
    // gather into the FP64 outputs (a plain copy: one column per job)
    std::vector<UnconvJob> uj;
    uj.reserve((size_t)S);
    for (int sidx = 0; sidx < S; ++sidx)
      uj.push_back({ct.p + (long)sidx * nnz, outs[mine[(size_t)sidx]].out, (int)nnz, 1, 1});
    DArr<UnconvJob> du;
    du.upload(uj, c.stream);
    launch_unconv(du.p, (int)uj.size(), nnz, c.stream);
    cuda_check(cudaStreamSynchronize(c.stream), "sync");
  }
  int h = 0;
  cuda_check(cudaMemcpy(&h, err.p, sizeof(int), cudaMemcpyDeviceToHost), "d2h");
  if (h) throw Error(ST_ETIMEOUT, "tensor-core GEMM: a bounded wait ran out");
}

// ---------------------------------------------------------------- autotuner

TuneChoice autotune_plans(const std::vector<Context*>& ctxs, const std::vector<double>& splits,
                          const std::vector<int>& budgets, int reps, std::vector<double>& ms) {
  if (ctxs.empty() || splits.empty() || budgets.empty() || reps <= 0)
    throw Error(ST_EINVAL, "autotune: empty problem or candidate list");
  for (int b : budgets)
    if (b <= 0) throw Error(ST_EINVAL, "autotune: chunk budgets must be positive");
  const bool batched = ctxs.size() > 1;
  for (Context* c : ctxs) {
    if (c->prepared < 0 || !c->plan.tm || c->plan.tm->precision > 3)
      throw Error(ST_ESTATE, "autotune: every context must be prepared in precision 1, 2 or 3");
    if (batched && !c->keep_host_plans)
      throw Error(ST_ESTATE, "autotune: tuning a batch needs host copies of the plans (keep_host_plans)");
  }
  // inputs and outputs of the timed calls: zero vectors (the time does not depend on
  // the values), sized for the prepared problems, whose layouts no candidate changes
  std::vector<DArr<double>> in(ctxs.size()), out(ctxs.size());
  std::vector<const double*> pin(ctxs.size());
  std::vector<double*> pout(ctxs.size());
  for (size_t i = 0; i < ctxs.size(); ++i) {
    Context& c = *ctxs[i];
    const size_t n = std::max<size_t>(c.plan.psi.nnz, 1);
    in[i].alloc(n, c.stream);
    out[i].alloc(n, c.stream);
    cuda_check(cudaMemsetAsync(in[i].p, 0, n * sizeof(double), c.stream), "memset");
    cuda_check(cudaStreamSynchronize(c.stream), "sync");
    pin[i] = in[i].p;
    pout[i] = out[i].p;
  }
  auto rebuild = [&](double split, int budget) {
    for (Context* c : ctxs) {
      c->split_tps = split;
      c->chunk_budget_mb = budget;
      build_sigma_plan(*c, c->lt, c->rt, c->prepared, c->plan);
      cuda_check(cudaStreamSynchronize(c->stream), "sync");
    }
  };
  ms.assign(splits.size() * budgets.size(), 0.0);
  size_t best = 0;
  // on an error the contexts get their parameters back and must be prepared again
  std::vector<std::pair<double, int>> saved;
  for (Context* c : ctxs) saved.emplace_back(c->split_tps, c->chunk_budget_mb);
  try {
    for (size_t i = 0; i < splits.size(); ++i)
      for (size_t j = 0; j < budgets.size(); ++j) {
        rebuild(splits[i], budgets[j]);
        double t = 0;
        if (batched) {
          std::unique_ptr<BatchPlan, void (*)(BatchPlan*)> b(batch_create(ctxs), batch_free);
          batch_sigma(*b, pin.data(), pout.data(), true);  // eager pass, then the graph capture
          batch_sigma(*b, pin.data(), pout.data(), true);  // first replay
          for (int r = 0; r < reps; ++r) t += batch_sigma(*b, pin.data(), pout.data(), true);
        } else {
          Context& c = *ctxs[0];
          run_sigma(c, c.plan, pin[0], pout[0]);  // warm-up
          cuda_check(cudaEventRecord(c.ev0, c.stream), "record");
          for (int r = 0; r < reps; ++r) run_sigma(c, c.plan, pin[0], pout[0]);
          cuda_check(cudaEventRecord(c.ev1, c.stream), "record");
          cuda_check(cudaEventSynchronize(c.ev1), "sync");
          if (plan_error(c, c.plan)) throw Error(ST_ETIMEOUT, "tensor-core GEMM: a bounded wait ran out");
          float e = 0;
          cuda_check(cudaEventElapsedTime(&e, c.ev0, c.ev1), "elapsed");
          t = e;
        }
        const size_t at = i * budgets.size() + j;
        ms[at] = t / reps;
        if (ms[at] < ms[best]) best = at;
      }
    const TuneChoice choice{splits[best / budgets.size()], budgets[best % budgets.size()]};
    rebuild(choice.split_tps, choice.budget_mb);
    return choice;
  } catch (...) {
    for (size_t i = 0; i < ctxs.size(); ++i) {
      ctxs[i]->split_tps = saved[i].first;
      ctxs[i]->chunk_budget_mb = saved[i].second;
      ctxs[i]->prepared = -1;
    }
    throw;
  }
}

}  // namespace gbdmrg
