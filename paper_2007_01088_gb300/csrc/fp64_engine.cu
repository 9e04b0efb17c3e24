// FP64 multi-term contraction engine.
//
// One launch runs a list of jobs; each job is a batched multi-term contraction
//   C[b][m][n] (op)= sum_terms sum_k A_t[b][m][k] * B_t[b][n][k]
// over strided two-level operand views (cc3::Opnd), with three epilogues:
// plain store, FP64 atomic accumulation (cross-triple sums of the residual)
// and the triples denominator tau = (C + acc) / (w - eps^{abc}_{ijk}).
//
// On this GPU the FP64 pipe retires ~2 DFMA per clock per SM (about 1 TFLOP/s
// for the chip), so an FP64 contraction is compute bound at any practical
// tile size; the tile is sized for DFMA latency hiding (16 independent
// accumulators per thread), not for bandwidth.  What is left to lose is work on
// padding and idle SMs: a tile skips the row and column groups of 16 (64 in
// the thin tile) that lie outside its job (nv = 48 fills 9 of the 16 groups of
// a 64 x 64 tile, a job of 16 columns a quarter of them), and launches of few
// tiles are split over K when their jobs accumulate (upload_plan).
#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>
#include <vector>

#include "cc3_internal.h"
#include "fx128.cuh"

namespace cc3 {

__device__ __forceinline__ long long rowoff(int m, int m_in, long long s1,
                                            long long s0) {
  return (long long)(m / m_in) * s1 + (long long)(m % m_in) * s0;
}

// acc += the products of the first im of a thread's TM rows and jn of its TN
// columns over kn values of K.  One body per (im, jn), found by descent from
// (IM, JN): a multiply-add under a predicate takes its turn in the FP64 pipe
// even where it is off, so that a tile of one column group in four took as long
// as a full one.  no=6 nv=48 FP64 residual 8.54 -> 7.31 ms; dressing of the integrals
// at no=16 nv=128: columns of 16 0.82 -> 0.23 ms, K = 16 2.85 -> 1.89 ms per vector.
template <int BM, int BN, int TM, int TN, int IM, int JN>
__device__ __forceinline__ void products(int im, int jn, int kn, const double *a0, const double *b0,
                                         double (&acc)[TM][TN]) {
  if constexpr (IM > 1) {
    if (im < IM) return products<BM, BN, TM, TN, IM - 1, JN>(im, jn, kn, a0, b0, acc);
  }
  if constexpr (JN > 1) {
    if (jn < JN) return products<BM, BN, TM, TN, IM, JN - 1>(im, jn, kn, a0, b0, acc);
  }
#pragma unroll 4
  for (int kk = 0; kk < kn; ++kk) {
    double a[IM], b[JN];
#pragma unroll
    for (int i = 0; i < IM; ++i) a[i] = a0[kk * (BM + 1) + i * (BM / TM)];
#pragma unroll
    for (int j = 0; j < JN; ++j) b[j] = b0[kk * (BN + 1) + j * (BN / TN)];
#pragma unroll
    for (int i = 0; i < IM; ++i)
#pragma unroll
      for (int j = 0; j < JN; ++j) acc[i][j] = fma(a[i], b[j], acc[i][j]);
  }
}

template <int BM, int BN, int TM, int TN, int BK>
__global__ void __launch_bounds__(256)
fp64_engine_kernel(const Job *__restrict__ jobs, int njobs,
                   const Term *__restrict__ terms, PtrTable P) {
  static_assert((BM / TM) * (BN / TN) == 256, "256 threads");
  // one double of padding per row: the loads below store along kk
  __shared__ double sA[BK][BM + 1];
  __shared__ double sB[BK][BN + 1];
  const long long cta = blockIdx.x;
  int lo = 0, hi = njobs - 1;
  while (lo < hi) {
    int mid = (lo + hi + 1) >> 1;
    if (jobs[mid].tile_base <= cta) lo = mid; else hi = mid - 1;
  }
  const Job &J = jobs[lo];
  long long local = cta - J.tile_base;
  const int per_batch = J.tiles_m * J.tiles_n * J.ksplit;
  const int bi = (int)(local / per_batch);
  int r = (int)(local % per_batch);
  const int ks = r % J.ksplit;
  r /= J.ksplit;
  const int tn = r % J.tiles_n, tm = r / J.tiles_n;
  const int m0 = tm * BM, n0 = tn * BN;
  const int M = J.M, N = J.N, Nm = J.Nm;

  constexpr int NTX = BN / TN;
  const int tid = threadIdx.x;
  const int tx = tid % NTX, ty = tid / NTX;
  // groups of rows / columns of this tile that its job reaches, and the rows
  // and columns to load for them
  constexpr int GM = BM / TM, GN = NTX;
  const int im = min(TM, (M - m0 + GM - 1) / GM), jn = min(TN, (N - n0 + GN - 1) / GN);
  const int lm = im * GM, ln = jn * GN;
  double acc[TM][TN];
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN; ++j) acc[i][j] = 0.0;

  for (int t = 0; t < J.nterm; ++t) {
    const Term &T = terms[J.term0 + t];
    const int K = T.K;
    int kchunk = (K + J.ksplit - 1) / J.ksplit;
    kchunk = (kchunk + BK - 1) / BK * BK;
    const int kbeg = ks * kchunk;
    const int kend = min(K, kbeg + kchunk);
    if (kbeg >= kend) continue;
    const double *Ab = P.p[T.A.buf] + T.A.off + (long long)bi * T.A.sb;
    const double *Bb = P.p[T.B.buf] + T.B.off + (long long)bi * T.B.sb;
    const double *Btb = P.p[T.Bt.buf] + T.Bt.off + (long long)bi * T.Bt.sb;
    for (int k0 = kbeg; k0 < kend; k0 += BK) {
      for (int e = tid; e < lm * BK; e += 256) {
        const int mm = e / BK, kk = e % BK;
        const int m = m0 + mm, k = k0 + kk;
        double v = 0.0;
        if (m < M && k < kend)
          v = Ab[rowoff(m, T.A.m_in, T.A.sm1, T.A.sm0) +
                 rowoff(k, T.A.k_in, T.A.sk1, T.A.sk0)];
        sA[kk][mm] = T.A.neg ? -v : v;
      }
      for (int e = tid; e < ln * BK; e += 256) {
        const int nn = e / BK, kk = e % BK;
        const int n = n0 + nn, k = k0 + kk;
        double v = 0.0;
        if (n < N && k < kend) {
          if (n < Nm) {
            v = Bb[rowoff(n, T.B.m_in, T.B.sm1, T.B.sm0) +
                   rowoff(k, T.B.k_in, T.B.sk1, T.B.sk0)];
            if (T.B.neg) v = -v;
          } else {
            const int nt = n - Nm;
            v = Btb[rowoff(nt, T.Bt.m_in, T.Bt.sm1, T.Bt.sm0) +
                    rowoff(k, T.Bt.k_in, T.Bt.sk1, T.Bt.sk0)];
            if (T.Bt.neg) v = -v;
          }
        }
        sB[kk][nn] = v;
      }
      __syncthreads();
      const int kn = min(BK, kend - k0);  // the occupied sums are short
      products<BM, BN, TM, TN, TM, TN>(im, jn, kn, &sA[0][ty], &sB[0][tx], acc);
      __syncthreads();
    }
  }

  // epilogue
#pragma unroll
  for (int i = 0; i < TM; ++i) {
    const int m = m0 + ty + i * (BM / TM);
    if (m >= M) continue;
#pragma unroll
    for (int j = 0; j < TN; ++j) {
      const int n = n0 + tx + j * NTX;
      if (n >= N) continue;
      const OutD &C = (n < Nm) ? J.C : J.Ct;
      const int nc = (n < Nm) ? n : n - Nm;
      double *dst = P.p[C.buf] + C.off + (long long)bi * C.sb +
                    rowoff(m, C.m_in, C.sm1, C.sm0) +
                    rowoff(nc, C.n_in, C.sn1, C.sn0);
      const double v = acc[i][j];
      if (J.mode == EPI_STORE) {
        *dst = v;
      } else if (J.mode == EPI_ATOMIC) {
        unsigned long long *fx = P.fx[C.buf];
        if (fx)
          fx_add(fx + 2 * (dst - P.p[C.buf]), v);
        else
          atomicAdd(dst, v);
      } else {  // EPI_TAU: m = c, n = a * nv + b
        const double *ev = P.p[B_EPSV];
        const int nvv = C.n_in;
        const double eps = ev[m] + ev[nc / nvv] + ev[nc % nvv] - J.eo;
        *dst = (*dst + v) / (J.w - eps);
      }
    }
  }
}

// Splits the accumulating jobs of a launch over K so that its work spreads
// over FILL tiles (eight per SM): a chunk of K is the launch's total K x tiles
// over FILL, at least 64.  Launches of many tiles keep their jobs whole.
// sigma1's Cholesky contraction at no=9 nv=81 (an 81 x 9 output over K =
// 21,870: 3 tiles) took 9 ms on 3 SMs.  Four tiles per SM, many of them of five
// on some: no=6 nv=48 FP64 residual 7.29 ms for 6.97, the left transformation's
// thin launches at no=9 nv=81 2.12 ms for 1.71; 16 per SM take as long as 8.  FILL
// is a constant (152 SMs), not the device's count: with reproducible sums the
// parts decide the bits.
static long long split_small_launch(std::vector<Job> &jobs, const std::vector<Term> &terms) {
  constexpr double FILL = 1216.0;
  double work = 0.0;
  auto length = [&](const Job &j) {  // K of a tile: of all its terms
    long long k = 0;
    for (int t = 0; t < j.nterm; ++t) k += terms[j.term0 + t].K;
    return k;
  };
  for (const Job &j : jobs) work += (double)length(j) * j.tiles_m * j.tiles_n * j.batch;
  const int chunk = (int)std::min(1e9, std::max(64.0, work / FILL));
  long long tiles = 0;
  for (Job &j : jobs) {
    if (j.mode == EPI_ATOMIC)
      j.ksplit = (int)std::max<long long>(j.ksplit, (length(j) + chunk - 1) / chunk);
    j.tile_base = tiles;
    tiles += (long long)j.batch * j.tiles_m * j.tiles_n * j.ksplit;
  }
  return tiles;
}

int upload_plan(const Plan &p, DevPlan *d, cudaStream_t s) {
  free_plan(d);
  std::vector<Job> jobs = p.jobs;
  d->njobs = (int)jobs.size();
  d->tiles = split_small_launch(jobs, p.terms);
  if (d->njobs == 0) return CC3_OK;
  // one allocation: the jobs, then the terms
  const size_t jb = (sizeof(Job) * jobs.size() + 15) / 16 * 16, tb = sizeof(Term) * p.terms.size();
  std::vector<char> host(jb + tb);
  std::memcpy(host.data(), jobs.data(), sizeof(Job) * jobs.size());
  if (tb) std::memcpy(host.data() + jb, p.terms.data(), tb);
  char *base = nullptr;
  if (dev_malloc(&base, jb + tb + sizeof(Term)) != cudaSuccess) {
    cudaGetLastError();
    return CC3_ERR_OOM;
  }
  d->jobs = reinterpret_cast<Job *>(base);
  d->terms = reinterpret_cast<Term *>(base + jb);
  return dev_upload(base, host.data(), host.size(), s);
}

void free_plan(DevPlan *d) {
  if (d->jobs) dev_free(d->jobs);
  d->jobs = nullptr;
  d->terms = nullptr;
  d->njobs = 0;
  d->tiles = 0;
}

int launch_plan(const DevPlan &d, const PtrTable &ptrs, cudaStream_t s,
                long long *launches) {
  if (d.njobs == 0 || d.tiles == 0) return CC3_OK;
  if (d.tiles > 0x7fffffffLL) return CC3_ERR_ARG;
  dim3 grid((unsigned)d.tiles);
  if (d.tile_kind == 0)
    fp64_engine_kernel<64, 64, 4, 4, 16><<<grid, 256, 0, s>>>(d.jobs, d.njobs,
                                                               d.terms, ptrs);
  else
    fp64_engine_kernel<256, 4, 4, 1, 16><<<grid, 256, 0, s>>>(d.jobs, d.njobs,
                                                              d.terms, ptrs);
  if (launches) ++*launches;
  return cudaGetLastError() == cudaSuccess ? CC3_OK : CC3_ERR_CUDA;
}

}  // namespace cc3
