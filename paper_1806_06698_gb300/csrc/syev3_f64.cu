// syev3_f64.cu -- FP64 batched 3x3 symmetric eigensolver for sm_103a.
//
// GB300 executes 1.68 FP64 lanes per SM per clock (1/64 of FP32), so the
// kernel keeps the work off the FP64 pipe: a matrix whose entries are of
// similar size is solved by the method of C. F. Borges (arXiv 1806.06698) in
// FP32 and refined to FP64 accuracy in 62-bit fixed point on the integer
// pipes (solve_fx.cuh); a diagonal one only needs sorting.  The others --
// graded or structured entries, three close eigenvalues -- take the method
// in FP64 (solve_f64.cuh), whose cost is the FP64 pipe's:
//  * one matrix per thread; tiles of kTPB packed records arrive by 1-D bulk
//    copy (TMA) into shared memory, double-buffered on two mbarriers, and a
//    full tile's results leave their staging rows by bulk copy (2^22 mixed
//    matrices 500 us, 522 with 16-byte stores by all threads);
//  * matrices left to the FP64 path are gathered from tile to tile and solved
//    kTPB at a time, so that each of the SM's FP64 units works on full warps
//    while the SM's other CTA is in the integer part;
//  * there, a matrix whose couplings are far below every gap of its diagonal
//    takes second-order perturbation (33 FP64 operations); for the others both
//    shifted roots are located in FP32, moved right of the root by a bound on
//    the FP32 error and finished by one FP64 Borges-Gragg step and the paper's
//    stopping test; the roots that do not pass are compacted with warp ballots
//    and finished by the full FP64 iteration.
//
// Measured (ncu, 2^21 well-separated matrices): 2240 thread instructions per
// matrix, issue slots 54 % used, the integer and FMA pipes each about 52 %,
// the FP64 pipe 9 %; no one unit is full, more resident warps change nothing
// (24 per SM instead of 16: 3 % slower), so the instruction count is what is
// left.  2^24 mixed matrices (10 % of them near-diagonal, on the FP64 path):
// 1.98 ms, against 6.37 ms when every matrix took the FP64 path (FP64 pipe 83 %
// busy); eigenvalues only, 10^6: 111 us against 294.

#include <atomic>
#include <cmath>
#include <cstdint>

#include "common.cuh"
#include "internal.h"
#include "serve_tile.cuh"
#include "solve_f64.cuh"
#include "solve_fx.cuh"

namespace syev3 {
namespace {

using namespace f64;

__device__ unsigned g_flags;     // kFlagWaitTimeout when a bulk-copy wait ran out

// Order of doubles as integers (not NaN; -0 as +0).
__device__ __forceinline__ int64_t order_key(const double x) {
  const int64_t b = __double_as_longlong(x);
  return is_zero(x) ? 0 : (b ^ (int64_t)((uint64_t)(b >> 63) >> 1));
}

// Places in ascending order (equal keys in the order given).
__device__ __forceinline__ void ranks(const int64_t k0, const int64_t k1, const int64_t k2, int rk[3]) {
  rk[0] = (int)(k1 < k0) + (int)(k2 < k0);
  rk[1] = (int)(k0 <= k1) + (int)(k2 < k1);
  rk[2] = (int)(k0 <= k2) + (int)(k1 <= k2);
}

// Eigenpairs of an exactly diagonal matrix: the entries and unit vectors, in
// the order of the arrow reduction (the larger of a11 and a22 first, then the
// other, a33 last); rk as in fx::solve.
__device__ __forceinline__ void diagonal(const double a[6], double l[3], double U[9], int rk[3]) {
  const int64_t p = order_key(a[0]), q = order_key(a[1]), k2 = order_key(a[2]);
  const bool keep = p >= q;
  const int64_t k0 = keep ? p : q, k1 = keep ? q : p;
  l[0] = keep ? a[0] : a[1];
  l[1] = keep ? a[1] : a[0];
  l[2] = a[2];
  U[0] = U[4] = keep ? 1.0 : 0.0;
  U[1] = U[3] = keep ? 0.0 : 1.0;
  U[2] = U[5] = U[6] = U[7] = 0.0;
  U[8] = 1.0;
  ranks(k0, k1, k2, rk);
}

// kVectors = false: eigenvalues only (U_out is NULL).
// kServe: the serving build.  The tiles are those of the device-resident
// work list `list` (A, n, lam_out and U_out are unused): runs of matrices of
// many requests, each tile with its own input and output rows, solved as one
// ragged batch.  A tile whose input is not 16-byte aligned is loaded with
// plain loads.  The production build (kServe = false) compiles this out.
// kTPB: matrices per tile and threads per CTA.
template <int kTPB, bool kServe>
struct Shared {
  alignas(16) double in[2][kTPB * 6];
  // Staging of a tile's results (eigenvalues, then eigenvectors); between
  // tiles, the work list of roots left for the full FP64 iteration: up to two
  // per matrix of an FP64 pass.
  static constexpr int kH = 2 * kTPB;
  struct Roots {
    double x[kH], ab[kH], b1[kH], b2[kH], g[kH];
    bool capped[kH];
  };
  union {
    alignas(16) double out[kTPB * 12];
    Roots hard;
  };
  // Matrices left to the FP64 path: fewer than kTPB from earlier tiles and
  // this tile's; their records and where their results go (the index in the
  // batch; serving: the addresses of the rows).
  static constexpr int kL = 2 * kTPB;
  double rec[6][kL];
  int64_t at[kL];
  double* at_U[kServe ? kL : 1];
  TileRef<double> ref[kServe ? 2 : 1];  // serving build: the tile of each buffer
  alignas(8) uint64_t bar[2];
  int n_left, n_hard;
};

// The FP64 path for the list's last P matrices, one per thread; the whole CTA
// calls it.  Not inlined: its registers would cost the integer part resident
// warps.
template <int kTPB, bool kVectors, bool kServe>
__device__ __noinline__ void fp64_pass(Shared<kTPB, kServe>& S, const int n_left, const int P, double* lam_out,
                                       double* U_out, unsigned long long* counters) {
  const int tid = threadIdx.x, lane_id = tid & 31;
  const unsigned lt_mask = (1u << lane_id) - 1u;
  Lane L;
  L.cls = kIdle;
  const int at = n_left - P + tid;
  // A result goes straight to memory (over what the tile's write-back put
  // there, ordered by the barriers in between).
  auto put = [&](const double lam[3], const double U[9], const int rk[3]) {
    const int64_t row = S.at[at];
    double* dl = kServe ? reinterpret_cast<double*>((uintptr_t)row) : lam_out + row * 3;
    double* dU = kServe ? S.at_U[kServe ? at : 0] : (U_out != nullptr ? U_out + row * 9 : nullptr);
#pragma unroll
    for (int k = 0; k < 3; ++k) dl[rk[k]] = lam[k];
    if (kVectors && dU != nullptr) {
#pragma unroll
      for (int k = 0; k < 3; ++k)
#pragma unroll
        for (int i = 0; i < 3; ++i) dU[i * 3 + rk[k]] = U[i * 3 + k];
    }
  };
  if (tid < P) {
    const double a[6] = {S.rec[0][at], S.rec[1][at], S.rec[2][at], S.rec[3][at], S.rec[4][at], S.rec[5][at]};
    double as[6], lam[3], U[9];
    int e = 0, rk[3];
    f64::prescale(a, as, e);  // (every listed matrix is finite)
    if (weakly_coupled(as, lam, U)) {
      ranks(order_key(lam[0]), order_key(lam[1]), order_key(lam[2]), rk);
#pragma unroll
      for (int k = 0; k < 3; ++k) lam[k] = mul_pow2(lam[k], e);
      put(lam, U, rk);
    } else {
      L = make_lane<false>(a);
    }
  }
  // FP32 seeds, then one FP64 step and the stopping test.  Problem 0 is mu
  // (A - a1 I), problem 1 is nu (P(a2 I - A)P: spikes swapped), Sec. 1.2.
  const bool reduced = (L.cls == kReduced);
  double root[2] = {0.0, 0.0};
  bool hard[2] = {false, false};
  double ab = 0.0, pb1[2] = {0.0, 0.0}, pb2[2] = {0.0, 0.0}, pg[2] = {0.0, 0.0};
  if (reduced) {
    ab = L.a1 - L.a2;
    const double bb1 = L.b1 * L.b1, bb2 = L.b2 * L.b2;
    pb1[0] = bb1; pb2[0] = bb2; pg[0] = L.g - L.a1;
    pb1[1] = bb2; pb2[1] = bb1; pg[1] = L.a2 - L.g;
    // FP32 can carry the problem when its data are normal FP32 numbers
    // with room for the products formed from them: spikes^2 >= 2^-120
    // (a tiny spike gives a root near its own size, 1/x^2 terms up to
    // ~2^120) and abar >= 2^-100.  An FP32 value that still underflows only
    // makes the FP64 step more cautious or sends the root to the full
    // iteration; acceptance is always the FP64 stopping test.
    const bool fp32_ok = hi_mag(bb1) >= hi_pow2(-120) && hi_mag(bb2) >= hi_pow2(-120) &&
                         hi_mag(ab) >= hi_pow2(-100);  // (all three >= 0)
    float sd[2] = {0.f, 0.f};
    double pc[2] = {0.0, 0.0}, pK[2] = {0.0, 0.0};
    const float fab = d2f_rn(ab), fb1[2] = {d2f_rn(pb1[0]), d2f_rn(pb1[1])}, fb2[2] = {d2f_rn(pb2[0]), d2f_rn(pb2[1])};
    if (fp32_ok) {
      const double rab = rcp64(ab);
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        pc[k] = pb2[k] * rab;
        pK[k] = -pg[k] - pc[k];
      }
      const float fg[2] = {d2f_rn(pg[0]), d2f_rn(pg[1])};
      const float fc[2] = {d2f_rn(pc[0]), d2f_rn(pc[1])}, fK[2] = {d2f_rn(pK[0]), d2f_rn(pK[1])};
      seed32x2(fab, fb1, fb2, fg, fc, fK, sd);
    }
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      double x = f2d_exact(sd[k]);
      int st = 2;
      // 2^-900 <= x <= 2^100 (x >= 0): the range finish64 assumes.
      if (hi_mag(x) >= hi_pow2(-900) && dbits(x) <= dbits(0x1p+100))
        st = finish64(ab, pb1[k], pb2[k], pg[k], pc[k], pK[k], fab, fb1[k], fb2[k], x);
      root[k] = (st == 2) ? 0.0 : x;  // 0: restart from Eq. (7)
      hard[k] = (st != 0);
    }
  }
  // Compact the unfinished roots and finish them with every lane of the
  // CTA available.
  int slot[2] = {-1, -1};
  {
    const unsigned m0 = __ballot_sync(0xffffffffu, hard[0]);
    const unsigned m1 = __ballot_sync(0xffffffffu, hard[1]);
    const int total = __popc(m0) + __popc(m1);
    int wbase = 0;
    if (lane_id == 0 && total) wbase = atomicAdd(&S.n_hard, total);
    wbase = __shfl_sync(0xffffffffu, wbase, 0);
    if (hard[0]) slot[0] = wbase + __popc(m0 & lt_mask);
    if (hard[1]) slot[1] = wbase + __popc(m0) + __popc(m1 & lt_mask);
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      if (slot[k] >= 0) {
        S.hard.x[slot[k]] = root[k];
        S.hard.ab[slot[k]] = ab;
        S.hard.b1[slot[k]] = pb1[k];
        S.hard.b2[slot[k]] = pb2[k];
        S.hard.g[slot[k]] = pg[k];
      }
    }
  }
  __syncthreads();
  const int n_hard = S.n_hard;
  for (int i = tid; i < n_hard; i += kTPB) {
    bool cp;
    int steps;
    S.hard.x[i] = zero_bg_full(S.hard.ab[i], S.hard.b1[i], S.hard.b2[i], S.hard.g[i], S.hard.x[i], cp, steps);
    S.hard.capped[i] = cp;
  }
  __syncthreads();
  bool capped = false;
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    if (slot[k] >= 0) {
      root[k] = S.hard.x[slot[k]];
      capped |= S.hard.capped[slot[k]];
    }
  }
  if (L.cls != kIdle) {
    double lam[3], U[9];
    const int rk[3] = {0, 1, 2};
    if (kVectors)
      finish_lane(L, root[0], root[1], lam, U);
    else
      finish_values(L, root[0], root[1], lam);
    put(lam, U, rk);
  }
  if (counters != nullptr) {
    const unsigned cm = __ballot_sync(0xffffffffu, capped);
    if (lane_id == 0 && cm) atomicAdd(&counters[0], (unsigned long long)__popc(cm));
  }
  __syncthreads();  // the list's records have been read
  if (tid == 0) {
    S.n_left = n_left - P;
    S.n_hard = 0;
  }
}

template <int kTPB, bool kBulkIn, bool kVectors, bool kServe = false>
__global__ void __launch_bounds__(kTPB, 512 / kTPB) k_syev3_f64(const double* __restrict__ A, int64_t n,
                                                              double* __restrict__ lam_out,
                                                              double* __restrict__ U_out,
                                                              unsigned long long* __restrict__ counters,
                                                              const ServeList* __restrict__ list) {
  static_assert(!kServe || (kBulkIn && kVectors && kTPB == kServeTile), "the serving build is bulk, vectors, its tiles");
  extern __shared__ __align__(16) unsigned char s_raw[];
  auto& S = *reinterpret_cast<Shared<kTPB, kServe>*>(s_raw);
  double* const s_lam = S.out;
  double* const s_U = S.out + kTPB * 3;

  const int tid = threadIdx.x, lane_id = tid & 31;
  const unsigned lt_mask = (1u << lane_id) - 1u;
  const int64_t n_tiles = kServe ? list->n_tiles : (n + kTPB - 1) / kTPB;
  bool want_U = (U_out != nullptr);
  bool vec_lam = ((reinterpret_cast<uintptr_t>(lam_out) & 15) == 0);
  bool vec_U = want_U && ((reinterpret_cast<uintptr_t>(U_out) & 15) == 0);
  int64_t cursor = 0;  // serving build: item cursor of the tiles this CTA issues (thread 0)

  if (tid == 0) {
    S.n_left = 0;
    S.n_hard = 0;
    if (kBulkIn) {
      mbar_init(&S.bar[0], 1);
      mbar_init(&S.bar[1], 1);
      fence_mbar_init();
    }
  }
  __syncthreads();

  auto issue = [&](int64_t tile, int buf) {
    if constexpr (kServe) {
      const TileRef<double> r = serve_tile<double>(list, tile, cursor);
      S.ref[buf] = r;
      if (reinterpret_cast<uintptr_t>(r.src) & 15) {  // plain loads after the wait
        mbar_arrive(&S.bar[buf]);
        return;
      }
      const uint32_t bytes = (uint32_t)r.cnt * 48u;
      mbar_arrive_expect_tx(&S.bar[buf], bytes);
      bulk_g2s(S.in[buf], r.src, bytes, &S.bar[buf]);
      return;
    }
    const int64_t base = tile * kTPB;
    const int cnt = (int)((n - base) < kTPB ? (n - base) : kTPB);
    const uint32_t bytes = (uint32_t)cnt * 48u;  // 48 = 3 * 16: always a multiple of 16
    mbar_arrive_expect_tx(&S.bar[buf], bytes);
    bulk_g2s(S.in[buf], A + base * 6, bytes, &S.bar[buf]);
  };

  uint32_t phases = 0u;  // bit b: parity of the next completion of S.bar[b]
  int buf = 0;
  int64_t tile = blockIdx.x;
  if (kBulkIn && tid == 0 && tile < n_tiles) issue(tile, 0);

  for (;; tile += gridDim.x, buf ^= 1) {
    const bool flush = (tile >= n_tiles);  // the CTA's last turn: solve what is left in the list
    if (flush) {
      __syncthreads();  // the last FP64 pass has set S.n_left
    } else {
      const int64_t base = tile * kTPB;
      int cnt = (int)((n - base) < kTPB ? (n - base) : kTPB);
      double* lam_tile = lam_out + base * 3;
      double* U_tile = want_U ? U_out + base * 9 : nullptr;
      const int64_t next = tile + gridDim.x;
      if (tid == 0) bulk_read_wait();  // the last tile's rows have left the staging area
      if (kBulkIn) {
        if (tid == 0 && next < n_tiles) issue(next, buf ^ 1);
        const bool ok = mbar_wait(&S.bar[buf], (phases >> buf) & 1u);
        if (__syncthreads_or(!ok)) {
          // Lost wait (CTA-uniform decision): flag it, give the copies in
          // flight a second bounded chance to land so that no write into
          // shared memory outlives the CTA, and stop.
          if (tid == 0) atomicOr(&g_flags, kFlagWaitTimeout);
          mbar_wait(&S.bar[buf], (phases >> buf) & 1u);
          if (next < n_tiles) mbar_wait(&S.bar[buf ^ 1], (phases >> (buf ^ 1)) & 1u);
          return;
        }
        phases ^= 1u << buf;
        if constexpr (kServe) {
          const TileRef<double> r = S.ref[buf];
          cnt = r.cnt;
          lam_tile = r.lam;
          U_tile = r.U;
          want_U = (r.U != nullptr);
          vec_lam = ((reinterpret_cast<uintptr_t>(r.lam) & 15) == 0);
          vec_U = want_U && ((reinterpret_cast<uintptr_t>(r.U) & 15) == 0);
          if (reinterpret_cast<uintptr_t>(r.src) & 15) {
            for (int i = tid; i < cnt * 6; i += kTPB) S.in[buf][i] = r.src[i];
            __syncthreads();
          }
        }
      } else {
        __syncthreads();  // the previous tile's records and staging have been read
        for (int i = tid; i < cnt * 6; i += kTPB) S.in[buf][i] = A[base * 6 + i];
        __syncthreads();
      }

      bool left = false, nonfinite = false;
      double a_in[6];
      if (tid < cnt) {
        const double2* src = reinterpret_cast<const double2*>(&S.in[buf][tid * 6]);
        const double2 p0 = src[0], p1 = src[1], p2 = src[2];
        a_in[0] = p0.x; a_in[1] = p0.y; a_in[2] = p1.x; a_in[3] = p1.y; a_in[4] = p2.x; a_in[5] = p2.y;
        double l[3], U[9];
        int rk[3] = {0, 1, 2};
        const fx::Fixed F = fx::fixed_of<true>(a_in);
        if (!F.finite) {
          nonfinite = true;
          const double qnan = __longlong_as_double(0x7ff8000000000000LL);
#pragma unroll
          for (int k = 0; k < 3; ++k) l[k] = qnan;
#pragma unroll
          for (int k = 0; k < 9; ++k) U[k] = qnan;
        } else if (F.diagonal) {
          diagonal(a_in, l, U, rk);
        } else if (F.similar && fx::solve<kVectors, true>(F, &S.in[buf][tid * 6], l, U, rk)) {
          if (kVectors) {
#pragma unroll
            for (int k = 0; k < 3; ++k) fx::sign_rule(U, k);
          }
        } else {
          left = true;
        }
        if (!left) {
#pragma unroll
          for (int k = 0; k < 3; ++k) s_lam[tid * 3 + rk[k]] = l[k];
          if (kVectors) {
#pragma unroll
            for (int k = 0; k < 3; ++k)
#pragma unroll
              for (int i = 0; i < 3; ++i) s_U[tid * 9 + i * 3 + rk[k]] = U[i * 3 + k];
          }
        }
      }
      const unsigned ml = __ballot_sync(0xffffffffu, left);
      int lb = 0;
      if (lane_id == 0 && ml) lb = atomicAdd(&S.n_left, __popc(ml));
      lb = __shfl_sync(0xffffffffu, lb, 0);
      if (left) {
        const int slot = lb + __popc(ml & lt_mask);
#pragma unroll
        for (int i = 0; i < 6; ++i) S.rec[i][slot] = a_in[i];
        if constexpr (kServe) {
          S.at[slot] = (int64_t)reinterpret_cast<uintptr_t>(lam_tile + tid * 3);
          S.at_U[slot] = want_U ? U_tile + tid * 9 : nullptr;
        } else {
          S.at[slot] = base + tid;
        }
      }
      if (counters != nullptr) {
        const unsigned nf = __ballot_sync(0xffffffffu, nonfinite);
        if (lane_id == 0 && nf) atomicAdd(&counters[1], (unsigned long long)__popc(nf));
      }
      fence_async_shared();
      __syncthreads();

      // A full, aligned tile's rows leave by bulk copy; the staging area is
      // written again only after thread 0 has seen it read (above, before the
      // next tile's barrier).  The rows of matrices in the list receive their
      // results later.
      if (cnt == kTPB && vec_lam && (!want_U || vec_U)) {
        if (tid == 0) {
          bulk_s2g(lam_tile, s_lam, kTPB * 24);
          if (kVectors && want_U) bulk_s2g(U_tile, s_U, kTPB * 72);
        }
      } else {
        auto store = [&](double* dst, const double* src, const int m, const bool vec) {
          const int m2 = vec ? m / 2 : 0;
          for (int i = tid; i < m2; i += kTPB)
            reinterpret_cast<double2*>(dst)[i] = reinterpret_cast<const double2*>(src)[i];
          for (int i = 2 * m2 + tid; i < m; i += kTPB) dst[i] = src[i];
        };
        store(lam_tile, s_lam, cnt * 3, vec_lam);
        if (kVectors && want_U) store(U_tile, s_U, cnt * 9, vec_U);
      }
    }
    const int n_left = S.n_left;  // (stable: between the barrier above and the next tile's)
    const int P = flush ? min(n_left, kTPB) : (n_left >= kTPB ? kTPB : 0);
    if (P == 0) {
      if (flush) break;
      continue;
    }
    if (tid == 0) bulk_write_wait();  // the rows below are written after the tiles' own
    __syncthreads();  // the staging area has been read; it takes the root list now

    fp64_pass<kTPB, kVectors, kServe>(S, n_left, P, lam_out, U_out, counters);
    if (flush) break;  // at most kTPB - 1 were left by then
  }
  if (tid == 0) bulk_read_wait();
}

// Matrices per tile of a batch.  The integer part is 40 KB of straight-line
// code, so warps of one scheduler share instruction fetches only when they
// run in step: with 2 CTAs of 256 threads "no instruction" stalls fall from
// 1.7 to 0.4 cycles per issue against 4 CTAs of 128 (2^22 mixed matrices:
// 679 against 774 us; 512 threads 729, 192 x 3 771, 320 x 2 673 but slower on
// well-separated ones).  While every tile of 64 is resident at once (77824
// matrices) they are that small: the FP64 units of all SMs then share the
// matrices left to the FP64 path, which with tiles of 256 kept a quarter of the
// SMs busy (4096 tridiagonal matrices 20.4 -> 12.9 us), and the integer part
// gains from fewer warps per SM too (well-separated spectra: 4096 7.0 -> 6.0 us,
// 65000 19.8 -> 17.8; 10^5 in tiles of 64 would gain nothing more).
constexpr int kTile = 256, kTileSmall = 64;
constexpr int kMaxDevices = 64;

cudaError_t device_and_sms(int* dev, int* sms) {
  const cudaError_t e = cudaGetDevice(dev);
  return e != cudaSuccess ? e : cudaDeviceGetAttribute(sms, cudaDevAttrMultiProcessorCount, *dev);
}

// Resident CTAs per SM; raises the kernel's shared-memory limit the first
// time it is asked for on a device.
template <int kTPB, bool kBulkIn, bool kVectors, bool kServe>
cudaError_t blocks_per_sm_f64(int dev, int* per_sm) {
  constexpr auto kernel = k_syev3_f64<kTPB, kBulkIn, kVectors, kServe>;
  constexpr size_t bytes = sizeof(Shared<kTPB, kServe>);
  static std::atomic<int> cached[kMaxDevices];
  const bool keep = dev >= 0 && dev < kMaxDevices;
  int v = keep ? cached[dev].load(std::memory_order_acquire) : 0;
  if (v == 0) {
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&v, kernel, kTPB, bytes);
    if (e != cudaSuccess) return e;
    if (v < 1) v = 1;
    if (keep) cached[dev].store(v, std::memory_order_release);
  }
  *per_sm = v;
  return cudaSuccess;
}

template <int kTPB, bool kBulkIn, bool kVectors, bool kServe>
cudaError_t launch_f64_t(const double* A, int64_t n, double* lam, double* U, unsigned long long* counters,
                         const ServeList* list, cudaStream_t stream) {
  int dev = 0, sms = 0, per_sm = 0;
  cudaError_t e = device_and_sms(&dev, &sms);
  if (e != cudaSuccess) return e;
  e = blocks_per_sm_f64<kTPB, kBulkIn, kVectors, kServe>(dev, &per_sm);
  if (e != cudaSuccess) return e;
  // Serving: the list's length is known only on the device; a resident grid,
  // whose CTAs without a tile exit at once.
  const int64_t resident = (int64_t)sms * per_sm, n_tiles = kServe ? resident : (n + kTPB - 1) / kTPB;
  const int grid = (int)(n_tiles < resident ? n_tiles : resident);
  k_syev3_f64<kTPB, kBulkIn, kVectors, kServe>
      <<<grid, kTPB, sizeof(Shared<kTPB, kServe>), stream>>>(A, n, lam, U, counters, list);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_f64_serve(const ServeList* list, unsigned long long* counters, cudaStream_t stream) {
  return launch_f64_t<kServeTile, true, true, true>(nullptr, 0, nullptr, nullptr, counters, list, stream);
}

cudaError_t launch_f64(const double* A, int64_t n, double* lam, double* U, unsigned long long* counters,
                       cudaStream_t stream) {
  if (n <= 0) return cudaSuccess;
  const bool bulk = (reinterpret_cast<uintptr_t>(A) & 15) == 0;
  int dev = 0, sms = 0;
  const cudaError_t e = device_and_sms(&dev, &sms);
  if (e != cudaSuccess) return e;
  if (n <= (int64_t)sms * (512 / kTileSmall) * kTileSmall) {  // (one wave: the kernel's launch bounds)
    if (bulk && U == nullptr) return launch_f64_t<kTileSmall, true, false, false>(A, n, lam, U, counters, nullptr, stream);
    if (bulk) return launch_f64_t<kTileSmall, true, true, false>(A, n, lam, U, counters, nullptr, stream);
    return launch_f64_t<kTileSmall, false, true, false>(A, n, lam, U, counters, nullptr, stream);
  }
  if (bulk && U == nullptr) return launch_f64_t<kTile, true, false, false>(A, n, lam, U, counters, nullptr, stream);
  if (bulk) return launch_f64_t<kTile, true, true, false>(A, n, lam, U, counters, nullptr, stream);
  return launch_f64_t<kTile, false, true, false>(A, n, lam, U, counters, nullptr, stream);
}

// The failure path of the bounded waits, exercised: one thread waits on an
// mbarrier that nothing completes (no copy is issued, nothing arrives), so
// the wait runs out after kWaitLimitNs and the timeout bit is recorded, as a
// lost bulk copy would record it.
__global__ void k_wait_selftest() {
  __shared__ alignas(8) uint64_t bar;
  if (threadIdx.x == 0) {
    mbar_init(&bar, 1);
    if (!mbar_wait(&bar, 0)) atomicOr(&g_flags, kFlagWaitTimeout);
  }
}

cudaError_t launch_wait_selftest(cudaStream_t stream) {
  k_wait_selftest<<<1, 32, 0, stream>>>();
  return cudaGetLastError();
}

cudaError_t take_flags_f64(unsigned* flags) {
  unsigned v = 0, zero = 0;
  cudaError_t e = cudaMemcpyFromSymbol(&v, g_flags, sizeof(v));
  if (e != cudaSuccess) return e;
  e = cudaMemcpyToSymbol(g_flags, &zero, sizeof(zero));
  *flags |= v;
  return e;
}

}  // namespace syev3
