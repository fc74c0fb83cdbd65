// Sparse runs, restart by restart: a CTA owns R restarts of the whole graph and runs many iterations
// of Algorithm 1 on them without leaving the SM.
//
// The restarts are independent, so the only thing an iteration shares between SMs in the row-wise
// kernels (k_csr.cu) is an artefact of splitting the rows over them: every iteration there reads
// and writes all of x and y through L2 or HBM and ends at a kernel boundary.  Here a CTA keeps, for
// its R restarts, x^t and x^{t+1} of every vertex in shared memory (two FP32 buffers that swap) and
// y and c' in the registers of the thread that owns the vertex; an iteration gathers neighbours from
// shared memory and ends at one __syncthreads.  Evaluations (candidate bits, exact integer
// objective, best record) stay in the CTA too, so a run of T iterations is ceil(T / 4096) launches
// and no graph replay.  State is read from and written back to global memory once per launch.
//
// Same arithmetic in the same order as k_csr: each row's neighbours are summed in ascending column
// order with FP32 fused multiply-adds, from the FP32 x or (BF16 / E4M3 weights) from x rounded to
// BF16, so iterates and records are bit-identical to every other form.
//
// Structure: vertices are placed by descending degree (stable) at positions 0, 1, ..; 32 consecutive
// positions form a slice, one lane each.  Warp w owns slices w, w + 32, ... and walks one stream of
// 16-byte groups: four neighbours of each lane's row, an entry holding the neighbour's place and its
// weight (see ENT_W), rows padded to whole
// groups of the longest of their slice with weight 0.  The stream is read from shared memory when it fits beside x, else
// through L1 / L2, two groups ahead of its use.
//
// What bounds it: shared-memory wavefronts of the gathers (a random graph's 32 4-byte gathers meet
// about 3.5 bank conflicts deep) and the latency of the streams from L2, not HBM or the launch.
// Measured per iteration against the row-wise kernels, evaluations every 10 included: Max-Cut ER
// n = 2,000, B = 256 5.4 -> 2.44 us; 100 x 100 torus, B = 512 16.0 -> 9.4 us; 4-regular n = 20,000,
// B = 512 38.6 -> 33.4 us.
#include <algorithm>
#include <cstring>

#include "sbo_internal.h"

namespace sbo {
namespace {

constexpr int RST_THREADS = 1024;
constexpr int RST_SPARE = 2;   // groups a warp reads ahead of their use
constexpr int RST_WARPS = RST_THREADS / 32;
constexpr size_t RST_SMEM_MAX = 225 * 1024;   // dynamic; the static arrays take up to 1.2 KB of the 227

struct RestartParams {
  EpiArgs a;
  const uint4* ent;              // group streams (global)
  const uint32_t* wstart;        // [33] first group (of 32 uint4) of each warp's stream, and the end
  const uint8_t* ngroups;        // [slices] groups of each slice
  const float* cpp;              // [positions] c' by position (0 beyond n)
  const int64_t* cpp64;
  float *X, *Y;                  // state [unit][position][R] (unit: R restarts)
  uint8_t* best;                 // bits of the best candidates [unit][position], bit r of a byte: restart r
  unsigned int* sched;           // chunks > 1: [ticket, abort, chunks finished per unit]
  int slices, ent_in_smem, units, chunks, chunk_len;
  int64_t t0, K, T, e0;          // iterations t0 + 1 .. t0 + iters; evaluate at multiples of K and at T
  int iters;
  long long *bestF, *bestT, *evalF, *trace, *n_evals, *t_last;
  long long trace_cap, t_last_new, n_evals_new;
  uint64_t timeout_ns;
};

// Evaluation points among iterations 1 .. t (multiples of K, and T).
__device__ __forceinline__ int64_t evals_upto(int64_t t, int64_t K, int64_t T) {
  return t / K + (T > 0 && T <= t && T % K != 0 ? 1 : 0);
}

// State vectors of one position: R consecutive floats, through L2 (another SM may have written them).
template <int R>
__device__ __forceinline__ void ld_state(const float* p, float (&v)[R]) {
  if (R == 1) {
    v[0] = __ldcg(p);
  } else if (R == 2) {
    const float2 t = __ldcg(reinterpret_cast<const float2*>(p));
    v[0] = t.x; v[R - 1] = t.y;
  } else {
    const float4 t = __ldcg(reinterpret_cast<const float4*>(p));
    v[0] = t.x; v[1 % R] = t.y; v[2 % R] = t.z; v[3 % R] = t.w;
  }
}
template <int R>
__device__ __forceinline__ void st_vec(float* p, const float (&v)[R]) {
  if (R == 1) *p = v[0];
  else if (R == 2) *reinterpret_cast<float2*>(p) = make_float2(v[0], v[R - 1]);
  else *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1 % R], v[2 % R], v[3 % R]);
}

// An entry of the streams: the neighbour's position, shifted so that masking gives the byte offset of
// its x in a buffer of `base` restarts per position, and the weight's top 15 bits (sign, exponent and 6
// bits of mantissa: every |w| <= 127, even ones to 254, and so on).
constexpr uint32_t ENT_W = 0xfffe0000u;
template <int R>
__device__ __forceinline__ uint32_t entry_offset(uint32_t e, int base) {   // byte offset for R restarts
  const uint32_t o = e & ~ENT_W;
  if (R == 1) return base == 1 ? o : o >> 1;
  return R == 2 ? o : o << 1;
}

// The four neighbours of one group: their x as the contraction sees it (BF16: rounded to nearest, two
// values per conversion), added in order.
template <int R, bool BF16, int BASE>
__device__ __forceinline__ void gather4(const float* xc, const uint4& c, float (&acc)[R]) {
  const uint32_t e[4] = {c.x, c.y, c.z, c.w};
  float v[4][R];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const char* p = reinterpret_cast<const char*>(xc) + entry_offset<R>(e[k], BASE);
    if (R == 1) {
      v[k][0] = *reinterpret_cast<const float*>(p);
    } else if (R == 2) {
      const float2 t = *reinterpret_cast<const float2*>(p);
      v[k][0] = t.x; v[k][R - 1] = t.y;
    } else {
      const float4 t = *reinterpret_cast<const float4*>(p);
      v[k][0] = t.x; v[k][1 % R] = t.y; v[k][2 % R] = t.z; v[k][3 % R] = t.w;
    }
  }
  if (BF16) {
#pragma unroll
    for (int j = 0; j < 4 * R; j += 2) {
      const __nv_bfloat162 h = __floats2bfloat162_rn(v[j / R][j % R], v[(j + 1) / R][(j + 1) % R]);
      v[j / R][j % R] = __low2float(h);
      v[(j + 1) / R][(j + 1) % R] = __high2float(h);
    }
  }
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const float w = __uint_as_float(e[k] & ENT_W);
#pragma unroll
    for (int r = 0; r < R; ++r) acc[r] = fmaf(w, v[k][r], acc[r]);
  }
}

template <int R>
__device__ __forceinline__ void add_bits(const uint8_t* bb, uint32_t e, int shift, float (&acc)[R]) {
  const float w = __uint_as_float(e & ENT_W);
  const uint32_t m = bb[(e & ~ENT_W) >> shift];
#pragma unroll
  for (int r = 0; r < R; ++r) acc[r] += ((m >> r) & 1u) ? w : 0.0f;
}

// One iteration's work on one vertex after its neighbour sums: update of R restarts.
template <int R>
__device__ __forceinline__ void update(const EpiArgs& a, const float* xc, float* xn, const float (&acc)[R], float cp,
                                       float (&y)[R]) {
  float xo[R], xv[R];
  if (R == 1) {
    xo[0] = *xc;
  } else if (R == 2) {
    const float2 t = *reinterpret_cast<const float2*>(xc);
    xo[0] = t.x; xo[R - 1] = t.y;
  } else {
    const float4 t = *reinterpret_cast<const float4*>(xc);
    xo[0] = t.x; xo[1 % R] = t.y; xo[2 % R] = t.z; xo[3 % R] = t.w;
  }
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const float x = xo[r];
    const float gx = g_val(x, G_QUAD);
    const float d = acc[r] + cp + y[r] * g_der(x, G_QUAD);
    // pdbo_update (common.cuh) with the projection as a saturation: the same value
    const bool stagnating = fabsf(x - 0.5f) <= a.delta && fabsf(d) <= a.grad_tol && y[r] <= 0.0f;
    xv[r] = __saturatef(x - a.alpha * d);
    if (stagnating) xv[r] = x <= 0.5f ? 0.5f - a.delta : 0.5f + a.delta;
    y[r] = y[r] + a.beta * gx;
  }
  st_vec<R>(xn, xv);
}

// Q: slices per warp at most (y and c' of a thread's vertices live in registers: Q R + Q, or Q R + Q / 2
// with c' packed as BF16 pairs when PACK).  R: restarts per CTA.  ONE: every row has at most four
// neighbours (one group per slice).
template <int Q, int R, bool BF16, bool ONE, bool PACK>
__global__ void __launch_bounds__(RST_THREADS, 1) k_csr_restart(const __grid_constant__ RestartParams P) {
  extern __shared__ __align__(16) uint8_t smem[];
  const int npos = P.slices * 32;
  float* xs = reinterpret_cast<float*>(smem);                          // [2][npos][R]
  uint4* ent_s = reinterpret_cast<uint4*>(xs + 2 * (size_t)npos * R);  // group streams (when they fit)
  const uint32_t groups = P.wstart[RST_WARPS];
  const size_t ent_bytes = P.ent_in_smem ? ((size_t)groups + RST_SPARE) * 32 * sizeof(uint4) : 0;
  uint8_t* bb = reinterpret_cast<uint8_t*>(ent_s) + ent_bytes;         // candidate bits, one per restart
  uint8_t* best = bb + npos;                                           // bits of the best candidates
  uint8_t* ngr = best + npos;                                          // groups of each slice
  __shared__ long long red[RST_WARPS][R];
  __shared__ long long s_bestF[R], s_bestT[R];
  __shared__ uint32_t s_improved, s_any;
  __shared__ int s_ticket;

  const EpiArgs& a = P.a;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int n = a.n;
  const int p0 = warp * 32 + lane;   // this thread's vertices: positions p0, p0 + RST_THREADS, ..
  constexpr int BASE = Q > 10 ? 1 : 2;            // restarts per position the entries are scaled for
  const int shift = BASE == 1 ? 2 : 3;            // entry offset -> position

  if (P.ent_in_smem)
    for (uint32_t k = threadIdx.x; k < (groups + RST_SPARE) * 32; k += RST_THREADS) ent_s[k] = P.ent[k];
  for (int k = threadIdx.x; k < P.slices; k += RST_THREADS) ngr[k] = P.ngroups[k];
  constexpr int AHEAD = ONE ? RST_SPARE : 1;      // groups in flight per warp
  const uint32_t stream0 = P.wstart[warp] * 32 + lane;
  constexpr int NC = PACK ? (Q + 1) / 2 : Q;
  float cps[PACK ? 1 : NC];
  uint32_t cpk[PACK ? NC : 1];
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    const float c = warp + q * RST_WARPS < P.slices ? P.cpp[p0 + q * RST_THREADS] : 0.0f;
    if (!PACK) cps[PACK ? 0 : q] = c;
    else if (q & 1) cpk[PACK ? q / 2 : 0] |= __float_as_uint(c) & 0xffff0000u;
    else cpk[PACK ? q / 2 : 0] = __float_as_uint(c) >> 16;
  }

  // Work: (chunk of iterations, unit) pairs.  With one chunk a CTA runs its unit; with more, CTAs
  // take tickets in order (all units' first chunk, then all second ones, ..) and a chunk starts once
  // its unit's previous one is finished, which a CTA with an earlier ticket is running or has done.
  for (;;) {
    int u = (int)blockIdx.x, c = 0;
    if (P.chunks > 1) {
      if (threadIdx.x == 0) {
        int t = (int)atomicAdd(P.sched, 1u);
        if (t >= P.units * P.chunks) {
          t = -1;
        } else if (t >= P.units) {
          const uint64_t deadline = globaltimer_ns() + P.timeout_ns;
          const unsigned int* done = P.sched + 2 + t % P.units;
          while (ld_acquire_gpu(done) < (unsigned)(t / P.units)) {
            if (ld_acquire_gpu(P.sched + 1) != 0u || globaltimer_ns() > deadline) {
              atomicOr(a.err, ERR_TIMEOUT);
              atomicExch(P.sched + 1, 1u);   // ends every other CTA's waits too
              t = -1;
              break;
            }
            __nanosleep(200);
          }
        }
        s_ticket = t;
      }
      __syncthreads();
      const int t = s_ticket;
      if (t < 0) return;
      u = t % P.units;
      c = t / P.units;
    }
    const int r0 = u * R;
    const int nlive = min(R, a.B - r0);
    const int64_t t0 = P.t0 + (int64_t)c * P.chunk_len;
    const int iters = min(P.chunk_len, P.iters - c * P.chunk_len);
    float* Xu = P.X + (size_t)u * npos * R;
    float* Yu = P.Y + (size_t)u * npos * R;

    if (threadIdx.x < R) {
      const bool live = (int)threadIdx.x < nlive;
      s_bestF[threadIdx.x] = live ? __ldcg(&P.bestF[r0 + threadIdx.x]) : 0;
      s_bestT[threadIdx.x] = live ? __ldcg(&P.bestT[r0 + threadIdx.x]) : 0;
    }
    if (threadIdx.x == 0) s_any = 0u;
    float y[Q][R];
#pragma unroll
    for (int q = 0; q < Q; ++q) {
#pragma unroll
      for (int r = 0; r < R; ++r) y[q][r] = 0.0f;
      if (warp + q * RST_WARPS < P.slices) {
        const int p = p0 + q * RST_THREADS;
        float x[R];
        ld_state<R>(Xu + (size_t)p * R, x);
        ld_state<R>(Yu + (size_t)p * R, y[q]);
        st_vec<R>(xs + p * R, x);
      }
    }
    __syncthreads();

    // iterations to the next evaluation point
    auto until_eval = [&](int64_t t) {
      int64_t next = (t / P.K + 1) * P.K;
      if (P.T > t && P.T < next) next = P.T;
      return (int)min(next - t, (int64_t)1 << 30);
    };
    int left = until_eval(t0);
    const float* xc = xs;
    float* xn = xs + (size_t)npos * R;
    for (int it = 1; it <= iters; ++it) {
      const uint4* st = (P.ent_in_smem ? ent_s : P.ent) + stream0;
      uint4 nx[AHEAD];   // groups read ahead (the streams end in RST_SPARE spare groups)
#pragma unroll
      for (int d = 0; d < AHEAD; ++d, st += 32) nx[d] = *st;
#pragma unroll
      for (int q = 0; q < Q; ++q) {
        if (warp + q * RST_WARPS >= P.slices) break;   // no later slice either
        const int p = p0 + q * RST_THREADS;
        float acc[R];
#pragma unroll
        for (int r = 0; r < R; ++r) acc[r] = 0.0f;
        const int ng = ONE ? 1 : ngr[warp + q * RST_WARPS];
        for (int g = 0; g < ng; ++g) {
          const uint4 e = nx[0];
#pragma unroll
          for (int d = 0; d + 1 < AHEAD; ++d) nx[d] = nx[d + 1];
          nx[AHEAD - 1] = *st;
          st += 32;
          gather4<R, BF16, BASE>(xc, e, acc);
        }
        const float cp = !PACK ? cps[PACK ? 0 : q]
                               : __uint_as_float((q & 1) ? cpk[PACK ? q / 2 : 0] & 0xffff0000u : cpk[PACK ? q / 2 : 0] << 16);
        update<R>(a, xc + p * R, xn + p * R, acc, cp, y[q]);
      }
      {
        float* t = const_cast<float*>(xc);
        xc = xn;
        xn = t;
      }
      __syncthreads();
      if (--left != 0) continue;

      // candidates b = [x > 1/2]
      for (int p = p0; p < npos; p += RST_THREADS) {
        uint32_t m = 0u;
#pragma unroll
        for (int r = 0; r < R; ++r) m |= (xc[p * R + r] > 0.5f ? 1u : 0u) << r;
        bb[p] = (uint8_t)m;
      }
      __syncthreads();
      // exact objective of the candidates: 2F = sum_i b_i ((A b)_i + 2 c'_i); (A b)_i is an exact
      // integer in FP32 because every row sum of |A| is below 2^24
      long long f2[R];
#pragma unroll
      for (int r = 0; r < R; ++r) f2[r] = 0;
      const int64_t t = t0 + it;
      left = until_eval(t);
      st = (P.ent_in_smem ? ent_s : P.ent) + stream0;
      for (int s = warp; s < P.slices; s += RST_WARPS) {
        const int ng = ONE ? 1 : ngr[s];
        const int p = s * 32 + lane;
        float acc[R];
#pragma unroll
        for (int r = 0; r < R; ++r) acc[r] = 0.0f;
        for (int g = 0; g < ng; ++g, st += 32) {
          const uint4 e = *st;   // entries beyond a row's length are padding (weight 0)
          add_bits<R>(bb, e.x, shift, acc);
          add_bits<R>(bb, e.y, shift, acc);
          add_bits<R>(bb, e.z, shift, acc);
          add_bits<R>(bb, e.w, shift, acc);
        }
        if (p < n) {
          const uint32_t m = bb[p];
          const long long c2 = 2 * (long long)P.cpp64[p];
#pragma unroll
          for (int r = 0; r < R; ++r)
            if ((m >> r) & 1u) f2[r] += (long long)acc[r] + c2;
        }
      }
#pragma unroll
      for (int r = 0; r < R; ++r) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) f2[r] += __shfl_xor_sync(0xffffffffu, f2[r], o);
        if (lane == 0) red[warp][r] = f2[r];
      }
      if (threadIdx.x == 0) s_improved = 0u;
      __syncthreads();
      if (threadIdx.x < R) {
        const int r = threadIdx.x;
        long long sum = 0;
#pragma unroll 4
        for (int w = 0; w < RST_WARPS; ++w) sum += red[w][r];
        if (r < nlive) {
          const long long F = sum / 2;
          if (F < s_bestF[r]) {   // strict: equal values keep the earliest t
            s_bestF[r] = F;
            s_bestT[r] = t;
            atomicOr(&s_improved, 1u << r);
          }
          P.evalF[r0 + r] = F;
          const int64_t e_idx = P.e0 + evals_upto(t, P.K, P.T) - evals_upto(P.t0, P.K, P.T) - 1;
          if (e_idx < P.trace_cap) atomicMin(&P.trace[e_idx], F);
        }
      }
      __syncthreads();
      const uint32_t imp = s_improved;
      if (imp) {
        for (int p = p0; p < npos; p += RST_THREADS) best[p] = (uint8_t)((best[p] & ~imp) | (bb[p] & imp));
        if (threadIdx.x == 0) s_any |= imp;
      }
    }
    __syncthreads();

    // write back: x and y, and the best records that changed
    const uint32_t any = s_any;
#pragma unroll
    for (int q = 0; q < Q; ++q) {
      if (warp + q * RST_WARPS >= P.slices) break;
      const int p = p0 + q * RST_THREADS;
      float x[R];
#pragma unroll
      for (int r = 0; r < R; ++r) x[r] = xc[p * R + r];
      st_vec<R>(Xu + (size_t)p * R, x);
      st_vec<R>(Yu + (size_t)p * R, y[q]);
    }
    if (any) {
      uint8_t* bu = P.best + (size_t)u * npos;
      for (int p = p0; p < npos; p += RST_THREADS) bu[p] = (uint8_t)((__ldcg(bu + p) & ~any) | (best[p] & any));
    }
    if ((int)threadIdx.x < nlive && ((any >> threadIdx.x) & 1u)) {
      P.bestF[r0 + threadIdx.x] = s_bestF[threadIdx.x];
      P.bestT[r0 + threadIdx.x] = s_bestT[threadIdx.x];
    }
    if (u == 0 && c == P.chunks - 1 && threadIdx.x == 0) {
      *P.n_evals = P.n_evals_new;
      *P.t_last = P.t_last_new;
    }
    if (P.chunks == 1) return;
    __threadfence();
    __syncthreads();   // every thread's stores before the count that publishes them
    if (threadIdx.x == 0) red_release_gpu_add(P.sched + 2 + u, 1u);
  }
}

// x^0 and y^0 in the unit layout: from the caller ([r][i], values checked as in k_init_state) or from
// SplitMix64 and ybar; positions and restarts beyond the problem are zero.
__global__ void k_restart_init(int n, int npos, int B, int R, const int32_t* __restrict__ perm, uint64_t seed,
                               float ybar, const float* __restrict__ x0, const float* __restrict__ y0, float* X,
                               float* Y, uint32_t* err) {
  const int64_t per = (int64_t)npos * R, total = per * ((B + R - 1) / R);
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t r = e / per * R + e % R;
    const int p = (int)(e % per / R);
    float x = 0.0f, y = 0.0f;
    if (p < n && r < B) {
      const int64_t i = perm[p];
      x = x0 ? x0[r * n + i] : uniform24(seed, (uint64_t)r, (uint64_t)i);
      if (!(x >= 0.0f && x <= 1.0f)) {  // also rejects NaN
        atomicOr(err, ERR_BOUNDS);
        x = 0.5f;
      }
      y = y0 ? y0[r * n + i] : ybar;
    }
    X[e] = x;
    Y[e] = y;
  }
}

// [B][n] copy of a state array in the unit layout (read-back); pos: position of a vertex.
__global__ void k_restart_gather(const float* __restrict__ src, const int32_t* __restrict__ pos, int n, int npos, int B,
                                 int R, float* dst) {
  for (int64_t r = blockIdx.y; r < B; r += gridDim.y) {
    const float* s = src + (r / R) * npos * R + r % R;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
      dst[r * n + i] = s[(int64_t)pos[i] * R];
  }
}
__global__ void k_restart_best_row(const uint8_t* __restrict__ best, const int32_t* __restrict__ pos, int n, int npos,
                                   int R, int64_t r, uint8_t* dst) {
  const uint8_t* b = best + (r / R) * npos;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
    dst[i] = (b[pos[i]] >> (r % R)) & 1u;
}

// Between the unit layout and the row-wise kernels' variable-major one ([i ld + r]), 32 positions x 32
// restarts at a time through shared memory.  to_rows: x into the operand (and the FP32 master), y, and
// the best bits as bytes; else back.
template <bool TO_ROWS>
__global__ void __launch_bounds__(256) k_restart_convert(RestartLayout L) {
  __shared__ float tx[32][33], ty[32][33];
  __shared__ uint8_t tb[32][33];
  const int lx = threadIdx.x & 31, ly = threadIdx.x >> 5;
  const int64_t r0 = (int64_t)blockIdx.y * 32;
  for (int p0 = (int)blockIdx.x * 32; p0 < L.npos; p0 += (int)gridDim.x * 32) {
    __syncthreads();
    for (int k = ly; k < 32; k += 8) {
      if (TO_ROWS) {   // lanes along positions
        const int64_t r = r0 + k;
        const int p = p0 + lx;
        if (r < L.B && p < L.n) {
          const size_t at = ((size_t)(r / L.R) * L.npos + p) * L.R + r % L.R;
          tx[k][lx] = L.X[at];
          ty[k][lx] = L.Y[at];
          tb[k][lx] = (L.best[(size_t)(r / L.R) * L.npos + p] >> (r % L.R)) & 1u;
        }
      } else {         // lanes along restarts
        const int64_t r = r0 + lx;
        const int p = p0 + k;
        tx[lx][k] = ty[lx][k] = 0.0f;
        tb[lx][k] = 0;
        if (r < L.B && p < L.n) {
          const int64_t idx = (int64_t)L.perm[p] * L.ld + r;
          tx[lx][k] = L.Xm ? L.Xm[idx] : static_cast<const float*>(L.Xop)[idx];
          ty[lx][k] = L.Yrows[idx];
          tb[lx][k] = L.bestBits[idx];
        }
      }
    }
    __syncthreads();
    for (int k = ly; k < 32; k += 8) {
      if (TO_ROWS) {
        const int64_t r = r0 + lx;
        const int p = p0 + k;
        if (r < L.B && p < L.n) {
          const int64_t idx = (int64_t)L.perm[p] * L.ld + r;
          op_store(L.Xop, idx, tx[lx][k], L.op_type);
          if (L.Xm) L.Xm[idx] = tx[lx][k];
          L.Yrows[idx] = ty[lx][k];
          L.bestBits[idx] = tb[lx][k];
        }
      } else {
        const int64_t r = r0 + k;
        const int p = p0 + lx;
        if (r < (int64_t)(L.B + L.R - 1) / L.R * L.R && p < L.npos) {
          const size_t at = ((size_t)(r / L.R) * L.npos + p) * L.R + r % L.R;
          L.X[at] = tx[k][lx];
          L.Y[at] = ty[k][lx];
          if (r % L.R == 0) {
            uint32_t m = 0u;
            for (int q = 0; q < L.R; ++q) m |= (uint32_t)tb[k + q][lx] << q;   // R divides 32
            L.best[(size_t)(r / L.R) * L.npos + p] = (uint8_t)m;
          }
        }
      }
    }
  }
}

using RestartKernel = void (*)(RestartParams);

template <int Q, int R, bool PACK>
RestartKernel kernel_of(bool bf16, bool one) {
  if (one) return bf16 ? (RestartKernel)k_csr_restart<Q, R, true, true, PACK> : (RestartKernel)k_csr_restart<Q, R, false, true, PACK>;
  return bf16 ? (RestartKernel)k_csr_restart<Q, R, true, false, PACK> : (RestartKernel)k_csr_restart<Q, R, false, false, PACK>;
}

// Instantiations: slices per warp up to Q with R restarts, in 64 registers per thread.
RestartKernel pick_kernel(const CsrRestartShape& sh, int R, bool bf16) {
  const int q = (sh.slices + RST_WARPS - 1) / RST_WARPS;
  const bool one = sh.max_groups <= 1;
  switch (R) {
    case 1:
      if (q <= 3) return kernel_of<3, 1, false>(bf16, one);
      if (q <= 10) return kernel_of<10, 1, false>(bf16, one);
      return q <= 20 && sh.cp_bf16 ? kernel_of<20, 1, true>(bf16, one) : nullptr;
    case 2: return q <= 3 ? kernel_of<3, 2, false>(bf16, one) : q <= 10 ? kernel_of<10, 2, false>(bf16, one) : nullptr;
    case 4: return q <= 5 ? kernel_of<5, 4, false>(bf16, one) : nullptr;
    default: return nullptr;
  }
}

size_t smem_bytes(const CsrRestartShape& sh, int R, bool ent) {
  const size_t npos = (size_t)sh.slices * 32;
  return 8 * npos * R + 2 * npos + (size_t)sh.slices + 16 + (ent ? ((size_t)sh.groups + RST_SPARE) * 512 : 0);
}

}  // namespace

// Lanes within the slices, chosen against bank conflicts.  The 32 gathers of one neighbour slot of a
// slice fall on the banks of their vertices' lanes (position mod 32); which 32 vertices they are
// depends on the slices only, so a vertex may move within its slice freely.  One greedy pass over the
// vertices gives each the free lane of its slice that adds least to the squares of the bank loads of
// the gathers it takes part in, its own lane where that is as good (a torus in natural order has no
// conflicts and stays as it is).  Two restarts per CTA (graphs up to 10,240 vertices) gather 8 bytes
// per lane in two half warps over 16 pairs of banks: there the vertices move within half slices.
// Random 4-regular graph: 3.51 -> 2.05 wavefronts per 4-byte gather (n = 20,000, 3 ms of host time),
// 6.15 -> 4.10 per 8-byte gather (n = 10,000, 1 ms).
static void place_lanes(int64_t n, const int32_t* rp, const int32_t* col, std::vector<int32_t>& perm,
                 std::vector<int32_t>& pos) {
  const int BK = n > 10 * RST_THREADS ? 32 : 16;
  const int64_t slices = (n + 31) / 32;
  std::vector<int64_t> first((size_t)slices + 1, 0);   // gather sets (neighbour slots) before each slice
  for (int64_t s = 0; s < slices; ++s) {
    const int32_t i = perm[(size_t)s * 32];             // by descending degree: the longest row
    first[(size_t)s + 1] = first[(size_t)s] + (rp[i + 1] - rp[i]);
  }
  std::vector<uint8_t> load((size_t)first[(size_t)slices] * 32, 0);   // vertices per (set, half, bank)
  std::vector<int32_t> at((size_t)n + 1, 0);
  std::vector<int64_t> occ((size_t)rp[n]);              // sets a vertex is gathered in
  for (int32_t e = 0; e < rp[n]; ++e) ++at[(size_t)col[e] + 1];
  for (int64_t i = 0; i < n; ++i) at[(size_t)i + 1] += at[(size_t)i];
  {
    std::vector<int32_t> next(at.begin(), at.end() - 1);
    for (int64_t p = 0; p < n; ++p) {
      const int32_t i = perm[(size_t)p];
      const int64_t half = (p % 32) / BK * BK;
      for (int k = 0; k < rp[i + 1] - rp[i]; ++k)
        occ[(size_t)next[(size_t)col[rp[i] + k]]++] = (first[(size_t)(p / 32)] + k) * 32 + half;
    }
  }
  for (int64_t p0 = 0; p0 < n; p0 += BK) {
    const int cnt = (int)std::min<int64_t>(BK, n - p0);
    int32_t v[32];
    for (int l = 0; l < cnt; ++l) v[l] = perm[(size_t)(p0 + l)];
    uint32_t free_lanes = cnt == 32 ? 0xffffffffu : (1u << cnt) - 1u;
    for (int l = 0; l < cnt; ++l) {
      uint32_t cost[32] = {};
      for (int32_t o = at[(size_t)v[l]]; o < at[(size_t)v[l] + 1]; ++o) {
        const uint8_t* L = &load[(size_t)occ[(size_t)o]];
        for (int b = 0; b < BK; ++b) cost[b] += (uint32_t)L[b] * L[b];
      }
      int best = (free_lanes >> l) & 1u ? l : -1;
      for (int b = 0; b < cnt; ++b)
        if (((free_lanes >> b) & 1u) && (best < 0 || cost[b] < cost[best])) best = b;
      free_lanes &= ~(1u << best);
      perm[(size_t)(p0 + best)] = v[l];
      pos[(size_t)v[l]] = (int32_t)(p0 + best);
      for (int32_t o = at[(size_t)v[l]]; o < at[(size_t)v[l] + 1]; ++o) ++load[(size_t)occ[(size_t)o] + best];
    }
  }
}

bool csr_restart_build(int64_t n, const int32_t* rp, const int32_t* col, const int64_t* val, const int64_t* cp,
                       CsrRestartHost* out) {
  if (n < 1 || n > 20 * RST_THREADS) return false;
  int maxd = 0;
  for (int64_t i = 0; i < n; ++i) maxd = std::max(maxd, rp[i + 1] - rp[i]);
  if (maxd > CSR_RESTART_MAX_DEG) return false;
  for (int64_t e = 0; e < rp[n]; ++e) {   // the weight must fit an entry's top 15 bits exactly
    const float w = (float)val[e];
    uint32_t bits;
    std::memcpy(&bits, &w, 4);
    if ((int64_t)w != val[e] || (bits & ~ENT_W)) return false;
  }
  // positions by descending degree, equal degrees in vertex order
  const int slices = (int)((n + 31) / 32);
  const int shift = n > 10 * RST_THREADS ? 2 : 3;   // see k_csr_restart: BASE
  std::vector<int32_t> first((size_t)maxd + 2, 0), perm((size_t)n), pos((size_t)n);
  for (int64_t i = 0; i < n; ++i) ++first[(size_t)(maxd - (rp[i + 1] - rp[i])) + 1];
  for (int d = 0; d <= maxd; ++d) first[(size_t)d + 1] += first[(size_t)d];
  for (int64_t i = 0; i < n; ++i) {
    const int32_t p = first[(size_t)(maxd - (rp[i + 1] - rp[i]))]++;
    perm[(size_t)p] = (int32_t)i;
    pos[(size_t)i] = p;
  }
  place_lanes(n, rp, col, perm, pos);
  out->ngroups.assign((size_t)slices, 0);
  // The kernel's ONE form walks exactly one group per slice, so with no row above four neighbours slices of isolated vertices hold one (padding) too.
  for (int s = 0; s < slices; ++s) {
    int width = 0;
    for (int64_t p = (int64_t)s * 32; p < std::min<int64_t>(n, (int64_t)(s + 1) * 32); ++p)
      width = std::max(width, rp[perm[(size_t)p] + 1] - rp[perm[(size_t)p]]);
    out->ngroups[(size_t)s] = (uint8_t)std::max((width + 3) / 4, maxd <= 4 ? 1 : 0);
  }
  uint32_t groups = 0;
  out->wstart.assign(RST_WARPS + 1, 0);
  for (int w = 0; w < RST_WARPS; ++w) {
    out->wstart[(size_t)w] = groups;
    for (int s = w; s < slices; s += RST_WARPS) groups += out->ngroups[(size_t)s];
  }
  out->wstart[RST_WARPS] = groups;
  out->ent.assign(((size_t)groups + RST_SPARE) * 128, 0u);
  for (int w = 0; w < RST_WARPS; ++w) {
    size_t g = out->wstart[(size_t)w];
    for (int s = w; s < slices; s += RST_WARPS) {
      const int gr = out->ngroups[(size_t)s];
      for (int l = 0; l < 32; ++l) {
        const int64_t p = (int64_t)s * 32 + l;
        const int64_t i = p < n ? perm[(size_t)p] : -1;
        const int deg = i >= 0 ? rp[i + 1] - rp[i] : 0;
        for (int k = 0; k < 4 * gr; ++k) {
          uint32_t e = (uint32_t)p << shift;   // padding gathers its own position with weight 0
          if (k < deg) {
            const float w32 = (float)val[rp[i] + k];
            uint32_t bits;
            std::memcpy(&bits, &w32, 4);
            e = bits | (uint32_t)pos[(size_t)col[rp[i] + k]] << shift;
          }
          out->ent[(g + (size_t)(k / 4)) * 128 + (size_t)l * 4 + (k & 3)] = e;
        }
      }
      g += (size_t)gr;
    }
  }
  out->perm = std::move(perm);
  out->pos = std::move(pos);
  out->cpp.assign((size_t)slices * 32, 0.0f);
  out->cpp64.assign((size_t)slices * 32, 0);
  for (int64_t p = 0; p < n; ++p) {
    out->cpp64[(size_t)p] = cp[out->perm[(size_t)p]];
    const float c = (float)out->cpp64[(size_t)p];
    out->cpp[(size_t)p] = c;
    uint32_t bits;
    std::memcpy(&bits, &c, 4);
    if (bits & 0xffffu) out->shape.cp_bf16 = false;
  }
  out->shape.slices = slices;
  out->shape.groups = groups;
  out->shape.max_groups = std::max(1, (maxd + 3) / 4);
  return true;
}

bool csr_restart_fits(const CsrRestartShape& sh, int R) {
  return pick_kernel(sh, R, false) != nullptr && smem_bytes(sh, R, false) <= RST_SMEM_MAX;
}

// Units (CTAs' worth of restarts) run side by side at once, and how many chunks the iterations are cut
// into so that the last round of units leaves no SM idle: with u units on c CTAs, k chunks take
// ceil(u k / c) chunk times, each a chunk's iterations and about one iteration's time for the load and
// write-back of the state (4-regular graph n = 20,000, B = 512: 4 rounds -> 3.4).
static int chunks_for(int units, int ctas, int iters) {
  if (units <= ctas || units % ctas == 0) return 1;
  int best = 1;
  double best_cost = 0.0;
  for (int k = 1; k <= 16 && iters / k >= 16; ++k) {
    const double cost = (double)(((int64_t)units * k + ctas - 1) / ctas) * ((iters + k - 1) / k + 1.0);
    if (k == 1 || cost < best_cost) { best = k; best_cost = cost; }
  }
  return best;
}

int csr_restart_pick(const CsrRestartShape& sh, int B, int sms) {
  int best = 0;
  double best_cost = 0.0;
  for (int R : {1, 2, 4}) {
    if (!csr_restart_fits(sh, R)) continue;
    const int units = (B + R - 1) / R;
    const double cost = std::max(1.0, (double)units / sms) * (1.0 + R);
    if (best == 0 || cost < best_cost) { best = R; best_cost = cost; }
  }
  return best;
}

size_t csr_restart_positions(const CsrRestartShape& sh) { return (size_t)sh.slices * 32; }

cudaError_t launch_csr_restart(const CsrRestartDev& d, const EpiArgs& a, int op_type, const CsrRestartRun& run, int R,
                               int sms, cudaStream_t s) {
  RestartKernel k = pick_kernel(d.shape, R, op_type == OP_BF16);
  if (!k || run.iters < 1) return cudaErrorInvalidValue;
  RestartParams P;
  std::memset(&P, 0, sizeof(P));
  P.a = a;
  P.ent = reinterpret_cast<const uint4*>(d.ent);
  P.wstart = d.wstart;
  P.ngroups = d.ngroups;
  P.cpp = d.cpp;
  P.cpp64 = d.cpp64;
  P.X = run.X;
  P.Y = run.Y;
  P.best = run.best;
  P.sched = run.sched;
  P.slices = d.shape.slices;
  P.ent_in_smem = smem_bytes(d.shape, R, true) <= RST_SMEM_MAX;
  P.units = (a.B + R - 1) / R;
  P.t0 = run.t0;
  P.K = run.K;
  P.T = run.T;
  P.e0 = run.e0;
  P.iters = run.iters;
  P.bestF = run.bestF;
  P.bestT = run.bestT;
  P.evalF = run.evalF;
  P.trace = run.trace;
  P.trace_cap = run.trace_cap;
  P.n_evals = run.n_evals;
  P.t_last = run.t_last;
  P.n_evals_new = run.n_evals_new;
  P.t_last_new = run.t_last_new;
  P.timeout_ns = run.timeout_ns;
  P.chunks = chunks_for(P.units, sms, run.iters);   // one CTA per SM: 1,024 threads of 64 registers
  P.chunk_len = (run.iters + P.chunks - 1) / P.chunks;
  P.chunks = (run.iters + P.chunk_len - 1) / P.chunk_len;   // none empty
  const size_t sm = smem_bytes(d.shape, R, P.ent_in_smem != 0);
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)RST_SMEM_MAX);
  if (e != cudaSuccess) return e;
  if (P.chunks > 1 && (e = cudaMemsetAsync(run.sched, 0, sizeof(unsigned int) * (2 + P.units), s)) != cudaSuccess) return e;
  k<<<(unsigned)(P.chunks > 1 ? std::min(P.units, sms) : P.units), RST_THREADS, sm, s>>>(P);
  return cudaGetLastError();
}

cudaError_t launch_restart_init(const CsrRestartDev& d, int n, int B, int R, uint64_t seed, float ybar, const float* x0,
                                const float* y0, float* X, float* Y, uint32_t* err, cudaStream_t s) {
  const int npos = d.shape.slices * 32;
  const int64_t total = (int64_t)npos * R * ((B + R - 1) / R);
  k_restart_init<<<(unsigned)std::min<int64_t>((total + 255) / 256, 152 * 32), 256, 0, s>>>(n, npos, B, R, d.perm, seed,
                                                                                            ybar, x0, y0, X, Y, err);
  return cudaGetLastError();
}

cudaError_t launch_restart_gather(const CsrRestartDev& d, const float* src, int n, int B, int R, float* dst,
                                  cudaStream_t s) {
  const dim3 grid((unsigned)std::min((n + 255) / 256, 64), (unsigned)std::min(B, 65535));
  k_restart_gather<<<grid, 256, 0, s>>>(src, d.pos, n, d.shape.slices * 32, B, R, dst);
  return cudaGetLastError();
}

cudaError_t launch_restart_best_row(const CsrRestartDev& d, const uint8_t* best, int n, int R, int64_t r, uint8_t* dst,
                                    cudaStream_t s) {
  k_restart_best_row<<<(unsigned)std::min((n + 255) / 256, 304), 256, 0, s>>>(best, d.pos, n, d.shape.slices * 32, R, r,
                                                                              dst);
  return cudaGetLastError();
}

cudaError_t launch_restart_convert(const CsrRestartDev& d, RestartLayout L, bool to_rows, cudaStream_t s) {
  L.npos = d.shape.slices * 32;
  L.perm = d.perm;
  const dim3 grid((unsigned)std::min(d.shape.slices, 1024), (unsigned)((L.B + 31) / 32));
  if (to_rows) k_restart_convert<true><<<grid, 256, 0, s>>>(L);
  else k_restart_convert<false><<<grid, 256, 0, s>>>(L);
  return cudaGetLastError();
}

}  // namespace sbo
