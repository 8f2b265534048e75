// Eighth-generation FP32 middle pass: generation 2's two-step register
// transform with each column tile's inputs staged by ONE tiled bulk tensor
// copy (TMA, cp.async.bulk.tensor.2d) per tile.
//
// A middle-pass tile is W = 16 adjacent columns k2 of one axis-0 plane k0,
// over its n1 rows (Y[k0][0..n1)[k2..k2+16): n1 rows of 128 bytes, M2 x 8
// bytes apart).  Generation 2 loads them straight from HBM at the start of
// the tile (the load latency shows as long-scoreboard stalls); generation 3
// stages them with per-thread cp.async copies (extra instructions, and bank
// conflicts in its staging layout).  Here thread 0 issues one 2-D tensor copy
// of the whole n1 x 16 box into shared memory, laid out [row][column] as the
// plain loads would read it, with completion counted in bytes on an mbarrier;
// the copy of the next tile is issued as soon as every thread has taken the
// current one out of the staging buffer, and runs under the rest of the
// current tile's work.  The arithmetic is generation 2's, so the results are
// bit-equal to it.
//
// The R2C and C2R passes along axis 0 are staged the same way (k8_r2c_ax0,
// k8_c2r_ax0 below).
//
// The copies need a tensor map per solve of the launch (host-encoded per
// launch, passed in a __grid_constant__ parameter: NJ maps, NJ = 1 for a
// single solve or kMaxJobs for a launch of several).  Every wait on the
// mbarrier is bounded (kWaitLimitCycles); a CTA whose wait gives up ORs
// kWaitTimeout into jobs.fault, waits (bounded) for its copy in flight and
// returns, the decision taken CTA-wide at the barrier that ends step A.
#pragma once
#include <cuda.h>

#include "mbar.cuh"
#include "passes2.cuh"

namespace fsa {

// 2-D tiled copy global -> shared of the box at element coordinates (x, y)
// of the tensor map; x * 8 bytes is a multiple of 16 (x = W c, W = 16 or 8).
__device__ __forceinline__ void tma_load_2d(void* dst, const CUtensorMap* map, int x, int y,
                                            unsigned long long* bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], "
      "[%4];\n" ::"r"(smem_u32(dst)),
      "l"(reinterpret_cast<unsigned long long>(map)), "r"(x), "r"(y), "r"(smem_u32(bar))
      : "memory");
}

// The tensor maps of a launch's solves (128 bytes each, 64-byte aligned).
template <int NJ> struct TmapSet {
  CUtensorMap m[NJ];
};

// Shared memory: the exchange tile (M x W complex), the staged input box
// (n1 = M/2 rows x W columns), the mbarrier.
template <class P> struct Geo8 {
  static constexpr int W = Geo2<P>::W;
  static constexpr int NT = Geo2<P>::NT;
  static constexpr int XCH = P::M * W * 8;
  static constexpr int STG = (P::M / 2) * W * 8;
  static constexpr int BAR = XCH + STG;
  static constexpr int SMEM = BAR + 16;
  static_assert(W == 16 && XCH % 16 == 0 && STG % 16 == 0, "box of 16 columns, 16-byte aligned staging");
};

// ymap.m[j]: Y of solve j as a 2-D tensor of 8-byte elements, dims
// {M2, planes * n1}, box {16, n1}.  SHARED: every solve of the launch has the
// same spectrum (densities of one plan); a CTA then takes one column tile for
// `run` solves in turn and loads the tile's spectrum values once.
template <class P, int NJ, bool SHARED = false>
__global__ void __launch_bounds__(Geo2<P>::NT, Geo2<P>::MINB_MID)
    k8_col_mid(const Jobs jobs, int M2, int planes, int run, const __grid_constant__ TmapSet<NJ> ymap) {
  using V = float2;
  using G = Geo8<P>;
  constexpr int M = P::M, n = M / 2, W = G::W, R2 = P::R2;
  extern __shared__ __align__(16) unsigned char smraw[];
  V* sm = reinterpret_cast<V*>(smraw);
  const V* stg = reinterpret_cast<const V*>(smraw + G::XCH);
  unsigned long long* bar = reinterpret_cast<unsigned long long*>(smraw + G::BAR);
  const int l = threadIdx.x % W, u = mid_u<P>(threadIdx.x);
  const int tpp = M2 / W;  // column tiles per plane
  const long long tpj = (long long)tpp * planes;  // tiles per solve
  const long long K = jobs.count;
  const long long total = tpj * K;
  const int n2 = M2 / 2;
  // work item -> (solve, tile of the solve), walked from the last item to
  // the first; SHARED orders the solves innermost and a CTA takes the K
  // items of one tile in a row
  auto phys = [&](long long it) -> long long { return kMidReverse ? total - 1 - it : it; };
  auto job_of = [&](long long it) -> long long { return SHARED ? phys(it) % K : phys(it) / tpj; };
  auto lt_of = [&](long long it) -> long long { return SHARED ? phys(it) / K : phys(it) % tpj; };
  auto next_of = [&](long long it) -> long long {
    if constexpr (SHARED) return it % run + 1 < run ? it + 1 : (it / run + gridDim.x) * run;
    else return it + gridDim.x;
  };
  const long long first = SHARED ? (long long)blockIdx.x * run : (long long)blockIdx.x;
  auto issue = [&](long long it) {  // thread 0
    const long long lt = lt_of(it);
    fence_proxy_async_smem();
    mbar_arrive_expect_tx(bar, (unsigned)G::STG);
    tma_load_2d(smraw + G::XCH, &ymap.m[job_of(it)], (int)(lt % tpp) * W, (int)(lt / tpp) * n, bar);
  };
  if (threadIdx.x == 0) {
    mbar_init(bar, 1);
    fence_mbar_init();
  }
  __syncthreads();
  if (threadIdx.x == 0 && first < total) issue(first);
  MidSpec<P> sp;
  int k = 0;
  for (long long it = first; it < total; it = next_of(it), ++k) {
    const long long lt = lt_of(it);
    const Job& jb = jobs.j[job_of(it)];
    const int k0 = (int)(lt / tpp);
    const int k2 = (int)(lt % tpp) * W + l;
    V* __restrict__ col = static_cast<V*>(jb.out) + (long long)k0 * n * M2 + k2;
    const float* __restrict__ srow =
        static_cast<const float*>(jb.S) + (long long)k0 * (n + 1) * (n2 + 1) + min(k2, M2 - k2);
    const bool late = !mbar_wait(bar, k & 1);
    stepA_fwd<P, V, true>(
        u,
        [&](int t, int r) {
          const int p = t + R2 * r;
          return p < n ? stg[p * W + l] : czero<V>();
        },
        [&](int q, int t, V v) { sm[(q * R2 + t) * W + l] = v; });
    if (__syncthreads_or(late)) {
      if (threadIdx.x == 0) {
        if (jobs.fault) atomicOr(jobs.fault, kWaitTimeout);
        mbar_wait(bar, k & 1);  // the copy still in flight
      }
      __syncthreads();
      return;
    }
    // every thread has taken the tile out of the staging buffer: the next one
    if (threadIdx.x == 0 && next_of(it) < total) issue(next_of(it));
    // SHARED: the first solve of the tile this CTA takes in turn loads the spectrum
    if (!SHARED || it % run == 0) mid_load<P>(sp, srow, u, true, n2 + 1);
    V b[R2];
#pragma unroll
    for (int t = 0; t < R2; ++t) b[t] = sm[(u * R2 + t) * W + l];
    rfft<R2, true>(b);
    mid_multiply<P, kMulSpectrum>(b, sp, u, jb, k0, k2, M2, true);
    stepB_inv<P, V>(u, b, [&](int q, int t, V v) { sm[(q * R2 + t) * W + l] = v; });
    __syncthreads();
    stepA_inv<P, V, true>(
        u, [&](int q, int t) { return sm[(q * R2 + t) * W + l]; },
        [&](int t, int r, V v) {
          const int p = t + R2 * r;
          if (p < n) col[(long long)p * M2] = v;
        });
    __syncthreads();
  }
}

// ------------------------------------------- middle pass, long lines --
// Lengths 768 and 1024: W = 8 columns (64-byte rows, the box in two copies), so
// that two CTAs fit an SM (16 columns would leave one), the twiddles in
// shared memory, and the tiles handed out dynamically (TileQueue).  Measured
// on the FP32 solve's middle pass: 384^3 0.903 -> 0.748 ms, 512^3 1.862 ->
// 1.836 ms (the tuner's earlier picks).  At length 512 the same measured
// slower than k8_col_mid (0.204 against 0.177 ms at 256^3; with 16 columns
// 0.205; with k8_col_mid's fixed tiles but shared or constant-memory twiddles
// 0.195 and 0.191): there the shared-memory pipe is as busy as the FP32 pipes,
// and thread 0's extra work per tile shows.  Results agree with generation
// 2's within round-off, not bit for bit.
//
// The two halves of a warp hold mirrored u: 2w, 2w + 1 | R1 - 2w, R1 - 2w - 1
// (warp 0: 0, 1 | R1/2, R1 - 1), so that k1 and M - k1 take one spectrum load
// and a shuffle; the two u (or t) of a half-warp differ by an odd number and
// exchange rows q are R2 + 1 entries apart, so its accesses fill both 64-byte
// halves of the banks.
template <class P> struct Geo8W {
  static constexpr int W = 8;
  static constexpr int NT = W * P::T;
  static constexpr int PITCH = P::R2 + 1;
  static constexpr int XCH = P::R1 * PITCH * W * 8;
  static constexpr int STG = (P::M / 2) * W * 8;
  static constexpr int BAR = XCH + STG;
  static constexpr int Q = BAR + 16;
  static constexpr int TW = Q + (int)sizeof(TileQueue);  // the length's twiddles
  static constexpr int SMEM = TW + P::M * 8;
  static constexpr int MINB = 512 / NT;
  static constexpr int BOXROWS = P::M / 2 > 256 ? P::M / 4 : P::M / 2;  // rows per tensor copy (at most 256)
  static_assert(P::R1 % 4 == 0 && P::R2 % 2 == 0 && XCH % 128 == 0, "paired halves, aligned staging");
};
template <class P> __device__ __forceinline__ int mid8_u(int tid) {
  constexpr int R1 = P::R1;
  const int a = 2 * (tid >> 5) + ((tid >> 3) & 1);
  return (tid & 16) == 0 ? a : (a == 0 ? R1 / 2 : R1 - a);
}
// The spectrum values of a thread's k1 = u + R1 s < M/2 (s < R2/2), and of the
// Nyquist index for u = 0; mid8_apply takes those of s >= R2/2 from the mirror.
template <class P> struct Mid8Spec {
  float v[P::R2 / 2 + 1];
};
template <class P>
__device__ __forceinline__ void mid8_load(Mid8Spec<P>& sp, const float* __restrict__ srow, int u, int st) {
  constexpr int R1 = P::R1, H = P::R2 / 2;
  const float* lo = srow + u * st;
#pragma unroll
  for (int s = 0; s < H; ++s) sp.v[s] = __ldg(lo + (R1 * s) * st);
  sp.v[H] = u == 0 ? __ldg(srow + (P::M / 2) * st) : 0.f;
}
template <class P> __device__ __forceinline__ void mid8_apply(float2* b, const Mid8Spec<P>& sp, int u) {
  constexpr int R1 = P::R1, R2 = P::R2, H = R2 / 2;
#pragma unroll
  for (int s = 0; s < H; ++s) b[s] = cscale(b[s], sp.v[s]);
  const bool w0 = threadIdx.x < 32;
  sfor<H, R2>([&](auto sc) {
    constexpr int s = decltype(sc)::value;
    float a = __shfl_xor_sync(0xffffffffu, sp.v[R2 - 1 - s], 16);
    if (w0) a = u == 0 ? sp.v[s == H ? H : R2 - s] : (u == R1 / 2 ? sp.v[R2 - 1 - s] : a);
    b[s] = cscale(b[s], a);
  });
}

// ymap.m[j]: Y of solve j as a 2-D tensor of 8-byte elements, dims
// {M2, planes * n1}, box {W, BOXROWS}.  SHARED: every solve of the launch has
// the same spectrum (densities of one plan); a CTA then takes one column tile
// for all solves in turn and loads the tile's spectrum values once.  Grid: one
// CTA per tile (SHARED: per tile of one solve), handed out by the queue.
template <class P, int NJ, bool SHARED = false>
__global__ void __launch_bounds__(Geo8W<P>::NT, Geo8W<P>::MINB)
    k8w_col_mid(const Jobs jobs, int M2, int planes, int, const __grid_constant__ TmapSet<NJ> ymap) {
  using V = float2;
  using G = Geo8W<P>;
  constexpr int M = P::M, n = M / 2, W = G::W, R2 = P::R2, PITCH = G::PITCH;
  extern __shared__ __align__(128) unsigned char smraw[];
  V* sm = reinterpret_cast<V*>(smraw);
  const V* stg = reinterpret_cast<const V*>(smraw + G::XCH);
  unsigned long long* bar = reinterpret_cast<unsigned long long*>(smraw + G::BAR);
  TileQueue* tq = reinterpret_cast<TileQueue*>(smraw + G::Q);
  const int l = threadIdx.x % W, u = mid8_u<P>(threadIdx.x);
  const int tpp = M2 / W;  // column tiles per plane
  const unsigned tpj = (unsigned)tpp * planes;  // tiles per solve (all of them fit 31 bits)
  const int K = jobs.count;
  const int n2 = M2 / 2;
  // tile number -> (solve, tile of the solve), walked from the last to the first
  auto phys = [&](int it) -> unsigned {
    const unsigned total = SHARED ? tpj : tpj * K;
    return kMidReverse ? total - 1 - it : it;
  };
  auto issue = [&](int it, int job) {  // thread 0
    const unsigned ph = phys(it), lt = SHARED ? ph : ph % tpj;
    const CUtensorMap* map = &ymap.m[SHARED ? job : (int)(ph / tpj)];
    const int x = (int)(lt % tpp) * W, y = (int)(lt / tpp) * n;
    fence_proxy_async_smem();
    mbar_arrive_expect_tx(bar, (unsigned)G::STG);
#pragma unroll
    for (int r = 0; r < n; r += G::BOXROWS) tma_load_2d(smraw + G::XCH + r * W * 8, map, x, y + r, bar);
  };
  if (threadIdx.x == 0) {
    mbar_init(bar, 1);
    tile_queue_init(tq);
    issue(blockIdx.x, 0);
  }
  const TwShared tw{reinterpret_cast<const float2*>(smraw + G::TW)};
  tw_copy<M>(reinterpret_cast<float2*>(smraw + G::TW));
  __syncthreads();
  Mid8Spec<P> sp;
  int job = 0;
  unsigned par = 0, qpar = 0;
  for (int it = blockIdx.x; it >= 0; par ^= 1) {
    const unsigned ph = phys(it), lt = SHARED ? ph : ph % tpj;
    const Job& jb = jobs.j[SHARED ? job : (int)(ph / tpj)];
    const int k0 = (int)(lt / tpp);
    const int k2 = (int)(lt % tpp) * W + l;
    V* __restrict__ col = static_cast<V*>(jb.out) + (long long)k0 * n * M2 + k2;
    const float* __restrict__ srow =
        static_cast<const float*>(jb.S) + (long long)k0 * (n + 1) * (n2 + 1) + min(k2, M2 - k2);
    const bool late = !mbar_wait(bar, par);
    stepA_fwd<P, V, true>(
        u,
        [&](int t, int r) {
          const int p = t + R2 * r;
          return p < n ? stg[p * W + l] : czero<V>();
        },
        [&](int q, int t, V v) { sm[(q * PITCH + t) * W + l] = v; }, tw);
    if (__syncthreads_or(late)) {
      if (threadIdx.x == 0) {
        if (jobs.fault) atomicOr(jobs.fault, kWaitTimeout);
        // the copy and the answer still in flight; a CTA that gives up leaves
        // its tile and one it was granted undone, which the fault word says
        mbar_wait(bar, par);
        mbar_wait(&tq->bar, qpar);
      }
      __syncthreads();
      return;
    }
    // every thread has taken the tile out of the staging buffer: the next one
    const bool more = SHARED && job + 1 < K;
    if (threadIdx.x == 0) {
      if (more) {
        issue(it, job + 1);
      } else {
        tile_answer(tq, qpar, jobs.fault);
        if (tq->next >= 0) {
          issue(tq->next, 0);
          tile_request(tq);
        }
      }
    }
    // SHARED: the first solve of the tile this CTA takes in turn loads the spectrum
    if (!SHARED || job == 0) mid8_load<P>(sp, srow, u, n2 + 1);
    V b[R2];
#pragma unroll
    for (int t = 0; t < R2; ++t) b[t] = sm[(u * PITCH + t) * W + l];
    rfft<R2, true>(b);
    mid8_apply<P>(b, sp, u);
    stepB_inv<P, V>(u, b, [&](int q, int t, V v) { sm[(q * PITCH + t) * W + l] = v; }, tw);
    __syncthreads();
    if (more) {
      ++job;
    } else {
      it = tq->next;
      job = 0;
      qpar ^= 1;
    }
    stepA_inv<P, V, true>(
        u, [&](int q, int t) { return sm[(q * PITCH + t) * W + l]; },
        [&](int t, int r, V v) {
          const int p = t + R2 * r;
          if (p < n) col[(long long)p * M2] = v;
        });
    __syncthreads();
  }
}

// The pad + R2C pass along axis 0 (pass 1) with the same staging: a tile is
// 2W = 32 (16) adjacent real columns c of rho over its n0 rows (rows C floats
// apart), carried as W complex lines (columns c, c + 1 as one complex
// value), staged by one 2-D tensor copy of the n0 x 2W box ([row][column],
// 8 W bytes a row).  rmap.m[j]: rho of solve j as a 2-D tensor of 4-byte
// elements, dims {C, n0}, box {2W, BOXROWS}; columns past C read as zero.
// Lengths 768 and 1024 take 8 lines (16 real columns, 64-byte rows) so that
// two CTAs fit an SM, with exchange rows of R2 + 1 entries (as the middle
// pass): 384^3 0.212 -> 0.135 ms, 512^3 0.416 -> 0.282 (0.313 with the
// twiddles read from HBM's table instead of shared memory).
template <class P> struct Geo8R {
  static constexpr int W = P::M <= 512 ? 16 : 8;
  static constexpr int NT = W * P::T;
  static constexpr int PITCH = W == 16 ? P::R2 : P::R2 + 1;
  static constexpr int XCH = P::R1 * PITCH * W * 8;
  static constexpr int STG = (P::M / 2) * 2 * W * 4;
  static constexpr int BAR = XCH + STG;
  static constexpr int TW = BAR + 16;  // the length's twiddles
  static constexpr int SMEM = TW + P::M * 8;
  static constexpr int MINB = NT <= 256 ? 2 : 1;
  static constexpr int BOXROWS = P::M / 2 > 256 ? P::M / 4 : P::M / 2;
  static_assert(XCH % 128 == 0 && STG % 16 == 0, "aligned staging");
};

template <class P, int NJ>
__global__ void __launch_bounds__(Geo8R<P>::NT, Geo8R<P>::MINB)
    k8_r2c_ax0(const Jobs jobs, long long C, const __grid_constant__ TmapSet<NJ> rmap) {
  using V = float2;
  using G = Geo8R<P>;
  constexpr int M = P::M, n = M / 2, K = M / 2 + 1, W = G::W, R1 = P::R1, R2 = P::R2, PITCH = G::PITCH;
  extern __shared__ __align__(16) unsigned char smraw[];
  V* sm = reinterpret_cast<V*>(smraw);
  const V* stg = reinterpret_cast<const V*>(smraw + G::XCH);  // [row][W complex]
  unsigned long long* bar = reinterpret_cast<unsigned long long*>(smraw + G::BAR);
  const int l = threadIdx.x % W, u = threadIdx.x / W;
  const long long tpj = (C + 2 * W - 1) / (2 * W);  // tiles per solve
  const long long total = tpj * jobs.count;
  auto issue = [&](long long tile) {  // thread 0
    fence_proxy_async_smem();
    mbar_arrive_expect_tx(bar, (unsigned)G::STG);
#pragma unroll
    for (int r = 0; r < n; r += G::BOXROWS)
      tma_load_2d(smraw + G::XCH + r * W * 8, &rmap.m[tile / tpj], (int)((tile % tpj) * 2 * W), r, bar);
  };
  if (threadIdx.x == 0) {
    mbar_init(bar, 1);
    fence_mbar_init();
  }
  const TwShared tw{reinterpret_cast<const float2*>(smraw + G::TW)};
  tw_copy<M>(reinterpret_cast<float2*>(smraw + G::TW));
  __syncthreads();
  if (threadIdx.x == 0 && blockIdx.x < total) issue(blockIdx.x);
  int k = 0;
  for (long long tile = blockIdx.x; tile < total; tile += gridDim.x, ++k) {
    V* __restrict__ X = static_cast<V*>(jobs.j[tile / tpj].out);
    const long long c = (tile % tpj) * (2 * W) + 2 * l;
    const bool ok = c < C;
    const bool late = !mbar_wait(bar, k & 1);
    stepA_fwd<P, V, true>(
        u,
        [&](int t, int r) {
          const int p = t + R2 * r;
          return p < n ? stg[p * W + l] : czero<V>();
        },
        [&](int q, int t, V v) { sm[(q * PITCH + t) * W + l] = v; }, tw);
    if (__syncthreads_or(late)) {
      if (threadIdx.x == 0) {
        if (jobs.fault) atomicOr(jobs.fault, kWaitTimeout);
        mbar_wait(bar, k & 1);  // the copy still in flight
      }
      __syncthreads();
      return;
    }
    if (threadIdx.x == 0 && tile + gridDim.x < total) issue(tile + gridDim.x);
    V b[R2];
#pragma unroll
    for (int t = 0; t < R2; ++t) b[t] = sm[(u * PITCH + t) * W + l];
    rfft<R2, true>(b);
    __syncthreads();
#pragma unroll
    for (int s = 0; s < R2; ++s) sm[(u + R1 * s) * W + l] = b[s];
    __syncthreads();
    // Z = DFT(a + i b): A[k] = (Z[k] + conj Z[M-k]) / 2, B[k] = (Z[k] - conj Z[M-k]) / 2i
    for (int kk = u; kk < K; kk += P::T) {
      const V zk = sm[kk * W + l];
      const V zm = sm[((M - kk) % M) * W + l];
      if (ok) {
        *reinterpret_cast<float4*>(X + (long long)kk * C + c) =
            make_float4(0.5f * (zk.x + zm.x), 0.5f * (zk.y - zm.y), 0.5f * (zk.y + zm.y), 0.5f * (zm.x - zk.x));
      }
    }
    __syncthreads();
  }
}

// The C2R pass along axis 0 + crop (pass 5) with the same staging.  Its
// tile reads all K0 = n0 + 1 rows of X (the half spectrum: rows k <= n0
// directly, k > n0 from their mirror M - k), 2 x W8 complex columns a row; at
// W = 16 the staged box and the exchange tile would take 130 KB and leave one
// CTA per SM, so this pass runs W8 = 8 complex lines (16 real columns) per
// CTA of 128 threads: a 258-row box of 128-byte rows (two copies of 129 rows,
// 33 KB; the last row lies past X and reads as zero) and a 32 KB exchange
// tile, three CTAs per SM.  xmap.m[j]: X of solve j as a 2-D tensor of
// 8-byte elements, dims {C, K0}, box {2W, BOX}.
// Lengths 768 and 1024 take W = 4 lines (64-byte rows, two or three boxes),
// again three CTAs per SM.
template <class P> struct Geo8C {
  static constexpr int W = P::M <= 512 ? 8 : 4;
  static constexpr int NT = W * P::T;
  // K0 = M/2 + 1 rows as equal boxes of at most 256 rows, their bytes a
  // multiple of 128; rows past X read as zero
  static constexpr int K0 = P::M / 2 + 1;
  static constexpr int NBOX = K0 > 512 ? 3 : 2;
  static constexpr int BOX = (K0 + NBOX - 1) / NBOX + (W == 4 ? (K0 + NBOX - 1) / NBOX % 2 : 0);
  static constexpr int ROWS = NBOX * BOX;
  static constexpr int PITCH = W == 8 ? P::R2 : P::R2 + 1;
  static constexpr int XCH = P::R1 * PITCH * W * 8;
  static constexpr int STG = ROWS * 2 * W * 8;
  static constexpr int BAR = XCH + STG;
  static constexpr int TW = BAR + 16;  // the length's twiddles
  static constexpr int SMEM = TW + P::M * 8;
  static_assert(BOX <= 256 && XCH % 128 == 0 && BOX * 2 * W * 8 % 128 == 0, "boxes of at most 256 rows");
};

template <class P, int NJ>
__global__ void __launch_bounds__(Geo8C<P>::NT, 3)
    k8_c2r_ax0(const Jobs jobs, long long C, const __grid_constant__ TmapSet<NJ> xmap) {
  using V = float2;
  using G = Geo8C<P>;
  constexpr int M = P::M, n = M / 2, W = G::W, R1 = P::R1, R2 = P::R2, PITCH = G::PITCH;
  extern __shared__ __align__(16) unsigned char smraw[];
  V* sm = reinterpret_cast<V*>(smraw);
  const float4* stg = reinterpret_cast<const float4*>(smraw + G::XCH);  // [row][W column pairs]
  unsigned long long* bar = reinterpret_cast<unsigned long long*>(smraw + G::BAR);
  const int l = threadIdx.x % W, u = threadIdx.x / W;
  const long long tpj = (C + 2 * W - 1) / (2 * W);  // tiles per solve
  const long long total = tpj * jobs.count;
  auto issue = [&](long long tile) {  // thread 0
    const CUtensorMap* map = &xmap.m[tile / tpj];
    const int x = (int)((tile % tpj) * 2 * W);
    fence_proxy_async_smem();
    mbar_arrive_expect_tx(bar, (unsigned)G::STG);
#pragma unroll
    for (int k = 0; k < G::NBOX; ++k)
      tma_load_2d(smraw + G::XCH + k * (G::STG / G::NBOX), map, x, k * G::BOX, bar);
  };
  if (threadIdx.x == 0) {
    mbar_init(bar, 1);
    fence_mbar_init();
  }
  const TwShared tw{reinterpret_cast<const float2*>(smraw + G::TW)};
  tw_copy<M>(reinterpret_cast<float2*>(smraw + G::TW));
  __syncthreads();
  if (threadIdx.x == 0 && blockIdx.x < total) issue(blockIdx.x);
  int it = 0;
  for (long long tile = blockIdx.x; tile < total; tile += gridDim.x, ++it) {
    float* __restrict__ phi = static_cast<float*>(jobs.j[tile / tpj].out);
    const long long c = (tile % tpj) * (2 * W) + 2 * l;
    const bool ok = c < C;
    const bool late = !mbar_wait(bar, it & 1);
    // Z[k] = A[k] + i B[k] with A, B Hermitian: rebuild k > n from M - k
    V b[R2];
#pragma unroll
    for (int s = 0; s < R2; ++s) {
      const int k = u + R1 * s;
      const bool lo = k <= n;
      const float4 ab = stg[(lo ? k : M - k) * W + l];
      b[s] = lo ? mk(ab.x - ab.w, ab.y + ab.z) : mk(ab.x + ab.w, ab.z - ab.y);
    }
    if (__syncthreads_or(late)) {
      if (threadIdx.x == 0) {
        if (jobs.fault) atomicOr(jobs.fault, kWaitTimeout);
        mbar_wait(bar, it & 1);  // the copies still in flight
      }
      __syncthreads();
      return;
    }
    // every thread holds its inputs: the next tile's copies run under this one
    if (threadIdx.x == 0 && tile + gridDim.x < total) issue(tile + gridDim.x);
    stepB_inv<P, V>(u, b, [&](int q, int t, V v) { sm[(q * PITCH + t) * W + l] = v; }, tw);
    __syncthreads();
    stepA_inv<P, V, true>(
        u, [&](int q, int t) { return sm[(q * PITCH + t) * W + l]; },
        [&](int t, int r, V v) {
          const int p = t + R2 * r;
          if (p < n && ok) *reinterpret_cast<V*>(phi + (long long)p * C + c) = v;
        });
    __syncthreads();
  }
}

}  // namespace fsa
