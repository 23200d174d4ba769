// FP32 block products for 4-function atoms (the mixed-precision path).
//
// Same contraction as spgemm.cu (C_ij = sum_k op(A)_ik op(B)_kj over the triple
// list of the output block, k ascending), laid out for 4 x 4 blocks:
//   * complex: eight lanes own one output block, lane (r, h) the elements
//     (r, 2h) and (r, 2h + 1); per triple a lane reads row r of A and its two
//     columns of B (rows, conjugated, of a daggered B) with 16-byte loads, so the
//     lanes of an item read the same two 128-byte lines, and does 8 complex
//     multiply-adds; the next triple's blocks load under the current one.  What
//     bounds it is the L1 path of these loads: six instructions of four items'
//     lines each for four triples (one lane per item, as the real kernel has it,
//     reads 32 lines an instruction); 1728 atoms x 3 kicks, r = 8 A: M 1.28 -> 0.97 ms,
//     K' 0.90 -> 0.64 ms;
//   * real: one lane owns one output block and reads whole blocks (one 64-byte
//     half line each);
//   * every element's sum runs over k and the block's inner index in ascending
//     order in either layout;
//   * global-load latency is hidden by occupancy, not by staging: a 4 x 4 block is
//     too small for a shared-memory pipeline to pay;
//   * epilogues are fused: Taylor accumulation into U, store, add, and the
//     delta-form sandwich K' = K + M + W dU^dagger with the mirror and the
//     hermitian diagonal block.
#include <algorithm>

#include "rt_internal.cuh"

namespace rt {

namespace f32b4 {

constexpr int NE = 16;
constexpr int THREADS = 256;

__device__ __forceinline__ void load_block(const float* __restrict__ p, float (&v)[NE]) {
  const float4* q = reinterpret_cast<const float4*>(p);
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const float4 f = q[k];
    v[4 * k] = f.x;
    v[4 * k + 1] = f.y;
    v[4 * k + 2] = f.z;
    v[4 * k + 3] = f.w;
  }
}
__device__ __forceinline__ void load_block(const float2* __restrict__ p, float2 (&v)[NE]) {
  const float4* q = reinterpret_cast<const float4*>(p);
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const float4 f = q[k];
    v[2 * k] = make_float2(f.x, f.y);
    v[2 * k + 1] = make_float2(f.z, f.w);
  }
}
__device__ __forceinline__ void store_block(float* p, const float (&v)[NE]) {
  float4* q = reinterpret_cast<float4*>(p);
#pragma unroll
  for (int k = 0; k < 4; ++k) q[k] = make_float4(v[4 * k], v[4 * k + 1], v[4 * k + 2], v[4 * k + 3]);
}
__device__ __forceinline__ void store_block(float2* p, const float2 (&v)[NE]) {
  float4* q = reinterpret_cast<float4*>(p);
#pragma unroll
  for (int k = 0; k < 8; ++k) q[k] = make_float4(v[2 * k].x, v[2 * k].y, v[2 * k + 1].x, v[2 * k + 1].y);
}

__device__ __forceinline__ float2 fma_v(float2 a, float2 b, float2 c) {
  c.x = fmaf(a.x, b.x, c.x);
  c.x = fmaf(-a.y, b.y, c.x);
  c.y = fmaf(a.x, b.y, c.y);
  c.y = fmaf(a.y, b.x, c.y);
  return c;
}
__device__ __forceinline__ float2 conj_v(float2 a) { return make_float2(a.x, -a.y); }
template <int EPI>
__device__ __forceinline__ void r4_item(const GemmArgs& g, int64_t item) {
  const float* __restrict__ A = static_cast<const float*>(g.A);
  const float* __restrict__ B = static_cast<const float*>(g.B);
  float acc[NE];
#pragma unroll
  for (int e = 0; e < NE; ++e) acc[e] = 0.f;
  const int64_t t0 = g.ptr[item], t1 = g.ptr[item + 1];
  for (int64_t t = t0; t < t1; ++t) {
    const int2 ab = g.ab[t];
    float a[NE], b[NE];
    load_block(A + (int64_t)ab.x * NE, a);
    load_block(B + (int64_t)ab.y * NE, b);
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        float v = acc[r * 4 + c];
#pragma unroll
        for (int m = 0; m < 4; ++m) v = fmaf(a[r * 4 + m], b[m * 4 + c], v);
        acc[r * 4 + c] = v;
      }
  }
  const int q = g.item_blk[item];
  if constexpr (EPI == EPI_STORE) {
    store_block(static_cast<float*>(g.C) + (int64_t)q * NE, acc);
  } else if constexpr (EPI == EPI_ADD) {
    float* C = static_cast<float*>(g.C) + (int64_t)q * NE;
    float old[NE];
    load_block(C, old);
#pragma unroll
    for (int e = 0; e < NE; ++e) acc[e] = old[e] + acc[e];
    store_block(C, acc);
  } else if constexpr (EPI == EPI_STORE_ACC) {
    // real power T^n stored (unless C is null); coef * T^n added to complex U
    if (g.C) store_block(static_cast<float*>(g.C) + (int64_t)q * NE, acc);
    const int uq = g.umap ? g.umap[q] : q;
    if (uq >= 0) {
      float2* U = static_cast<float2*>(g.U) + (int64_t)uq * NE;
      float2 u[NE];
      load_block(U, u);
      const float cf = (float)g.coef;
#pragma unroll
      for (int e = 0; e < NE; ++e) {
        if (g.coef_imag) u[e].y += cf * acc[e];
        else u[e].x += cf * acc[e];
      }
      store_block(U, u);
    }
  }
}

// The blocks of one triple that a complex lane multiplies: row r of A; of B the
// columns 2h, 2h + 1 (b[m] = B(m, 2h..2h+1)), or, daggered, its rows 2h and 2h + 1
// (b[2 c .. 2 c + 1] = row 2h + c).
struct C4 {
  float4 a[2], b[4];
};
template <bool BDAG>
__device__ __forceinline__ void c4_load(C4& v, const float2* __restrict__ A, const float2* __restrict__ B, int2 ab,
                                        int r, int h) {
  const float4* pa = reinterpret_cast<const float4*>(A + (int64_t)ab.x * NE) + 2 * r;
  const float4* pb = reinterpret_cast<const float4*>(B + (int64_t)ab.y * NE) + (BDAG ? 4 * h : h);
  v.a[0] = pa[0];
  v.a[1] = pa[1];
#pragma unroll
  for (int m = 0; m < 4; ++m) v.b[m] = pb[BDAG ? m : 2 * m];
}
__device__ __forceinline__ float2 lo2(float4 v) { return make_float2(v.x, v.y); }
__device__ __forceinline__ float2 hi2(float4 v) { return make_float2(v.z, v.w); }

// One complex item by the eight lanes of a group (gl = 2 r + h); every lane of
// the warp comes here, `on` only those with an item.
template <bool BDAG, int EPI>
__device__ __forceinline__ void c4_item(const GemmArgs& g, int64_t item, bool on, int gl) {
  const int r = gl >> 1, h = gl & 1;
  const float2* __restrict__ A = static_cast<const float2*>(g.A);
  const float2* __restrict__ B = static_cast<const float2*>(g.B);
  float2 acc[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
  const int64_t t0 = on ? g.ptr[item] : 0;
  const int nt = on ? (int)(g.ptr[item + 1] - t0) : 0;
  const int2* __restrict__ ab = g.ab + t0;
  if (nt > 0) {
    C4 cur, nxt;
    c4_load<BDAG>(cur, A, B, ab[0], r, h);
    int2 p = ab[nt > 1 ? 1 : 0];
    for (int t = 0; t < nt; ++t) {
      c4_load<BDAG>(nxt, A, B, p, r, h);  // triple t + 1 (after the last: the last again, unused)
      p = ab[t + 2 < nt ? t + 2 : nt - 1];
      const float2 a[4] = {lo2(cur.a[0]), hi2(cur.a[0]), lo2(cur.a[1]), hi2(cur.a[1])};
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        float2 v = acc[c];
#pragma unroll
        for (int m = 0; m < 4; ++m) {
          const float4 w = BDAG ? cur.b[2 * c + (m >> 1)] : cur.b[m];
          const float2 b = (BDAG ? (m & 1) : c) ? hi2(w) : lo2(w);
          v = fma_v(a[m], BDAG ? conj_v(b) : b, v);
        }
        acc[c] = v;
      }
      cur = nxt;
    }
  }
  const int q = on ? g.item_blk[item] : 0;
  const int64_t e0 = (int64_t)q * NE + 4 * r + 2 * h;  // this lane's two elements
  if constexpr (EPI == EPI_STORE) {
    if (!on) return;
    *reinterpret_cast<float4*>(static_cast<float2*>(g.C) + e0) = make_float4(acc[0].x, acc[0].y, acc[1].x, acc[1].y);
    // delta form: also W = dK + M in FP32 (dK in FP64 through the map from
    // this pattern to dK's; -1 = no dK block), one rounding per element
    if (g.base) {
      const int kq = g.add_map ? g.add_map[q] : q;
      float2 w[2];
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        double2 kv = make_double2(0.0, 0.0);
        if (kq >= 0) kv = static_cast<const double2*>(g.base)[(int64_t)kq * NE + 4 * r + 2 * h + c];
        w[c] = make_float2((float)((double)acc[c].x + kv.x), (float)((double)acc[c].y + kv.y));
      }
      *reinterpret_cast<float4*>(static_cast<float2*>(g.U) + e0) = make_float4(w[0].x, w[0].y, w[1].x, w[1].y);
    }
  } else if constexpr (EPI == EPI_ADD) {
    if (!on) return;
    float4* C = reinterpret_cast<float4*>(static_cast<float2*>(g.C) + e0);
    const float4 old = *C;
    *C = make_float4(old.x + acc[0].x, old.y + acc[0].y, old.z + acc[1].x, old.w + acc[1].y);
  } else if constexpr (EPI == EPI_DELTA_SANDWICH) {
    // K'_ij = K_ij (+ R_ij) + M_ij + acc for j >= i (K in FP64); mirror; hermitian diagonal
    const int i = on ? g.rowidx[q] : 0, j = on ? g.colidx[q] : 1;
    double2* __restrict__ K = static_cast<double2*>(g.C);
    double2 val[2] = {make_double2(0.0, 0.0), make_double2(0.0, 0.0)};
    if (on) {
      const double2* __restrict__ base = static_cast<const double2*>(g.base) + e0;
      const int aq = g.add_map ? g.add_map[q] : q;
      float4 mv = make_float4(0.f, 0.f, 0.f, 0.f);
      if (aq >= 0)
        mv = *reinterpret_cast<const float4*>(static_cast<const float2*>(g.addend) + (int64_t)aq * NE + 4 * r + 2 * h);
      // reference split: R = U K_ref U^dagger - K_ref (FP64) joins the base, or
      // R(E) = sum_p E^p B_p at this step's field, by Horner here
      const double2* __restrict__ R = g.base2 ? static_cast<const double2*>(g.base2) + e0 : nullptr;
      const double E = g.rpoly ? *g.poly_E : 0.0;
      const int deg = E == 0.0 ? 0 : g.rdeg;  // R(0) = B_0
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        double2 kv = base[c];
        if (R) {
          kv = make_double2(kv.x + R[c].x, kv.y + R[c].y);
        } else if (g.rpoly) {
          double2 rv = g.rpoly[deg][e0 + c];
          for (int p = deg - 1; p >= 0; --p) {
            const double2 cp = g.rpoly[p][e0 + c];
            rv = make_double2(fma(rv.x, E, cp.x), fma(rv.y, E, cp.y));
          }
          kv = make_double2(kv.x + rv.x, kv.y + rv.y);
        }
        const float2 m = c ? hi2(mv) : lo2(mv);
        val[c] = make_double2(kv.x + ((double)m.x + (double)acc[c].x), kv.y + ((double)m.y + (double)acc[c].y));
      }
      if (i != j) {
        const int64_t qt = (int64_t)g.tmap[q] * NE;
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          const int64_t et = qt + (2 * h + c) * 4 + r;
          K[e0 + c] = val[c];
          K[et] = make_double2(val[c].x, -val[c].y);
          if (g.kf32) {
            float2* __restrict__ Kf = static_cast<float2*>(g.kf32);
            Kf[e0 + c] = make_float2((float)val[c].x, (float)val[c].y);
            Kf[et] = make_float2((float)val[c].x, (float)-val[c].y);
          }
        }
      }
    }
    // diagonal blocks: element (c, r) lies in lane 2 c + (r >> 1) of the group, its slot r & 1
    // (every lane of the warp takes part in the exchange)
    double herm = 0.0;
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      const int from = ((threadIdx.x & 31) & ~7) + 2 * (2 * h + c) + (r >> 1);
      const double x0 = __shfl_sync(0xffffffffu, val[0].x, from), y0 = __shfl_sync(0xffffffffu, val[0].y, from);
      const double x1 = __shfl_sync(0xffffffffu, val[1].x, from), y1 = __shfl_sync(0xffffffffu, val[1].y, from);
      if (on && i == j) {
        const double2 t = (r & 1) ? make_double2(x1, y1) : make_double2(x0, y0);
        const double dr = val[c].x - t.x, di = val[c].y + t.y;
        herm = fmax(herm, sqrt(dr * dr + di * di));
        const double2 w = make_double2(0.5 * (val[c].x + t.x), 0.5 * (val[c].y - t.y));
        K[e0 + c] = w;
        if (g.kf32) static_cast<float2*>(g.kf32)[e0 + c] = make_float2((float)w.x, (float)w.y);
      }
    }
    if (on && i == j && g.herm_max) atomicMax(g.herm_max, (unsigned long long)__double_as_longlong(herm));
  }
}

// Items by lane (real) or by groups of eight lanes (complex); a persistent launch
// (g.persistent) walks items with a grid-wide stride, and a grouped launch (g.grp)
// takes item i as item gitems[i].y of the product described by grp[gitems[i].x].
template <int EPI>
__global__ void __launch_bounds__(THREADS, 2) k_gemm4_r32(const __grid_constant__ GemmArgs g) {
  const int64_t item = (int64_t)blockIdx.x * THREADS + threadIdx.x;
  if (item < g.n_items) r4_item<EPI>(g, item);
}

constexpr int C_ITEMS = THREADS / 8;  // complex items of a CTA
constexpr int C_CTAS = 3;             // CTAs per SM (85 registers)
template <bool BDAG, int EPI>
__global__ void __launch_bounds__(THREADS, C_CTAS) k_gemm4_f32(const __grid_constant__ GemmArgs g) {
  const int gl = threadIdx.x & 7;
  const int64_t stride = g.persistent ? (int64_t)gridDim.x * C_ITEMS : g.n_items;
  // whole warps stay together: a warp leaves when its first item lies past the end
  const int64_t first = (int64_t)blockIdx.x * C_ITEMS + (threadIdx.x >> 5) * 4;
  for (int64_t w = first; w < g.n_items; w += stride) {
    const int64_t item = w + ((threadIdx.x & 31) >> 3);
    const bool on = item < g.n_items;
    const int2 gi = g.grp ? g.gitems[on ? item : w] : make_int2(0, 0);
    c4_item<BDAG, EPI>(g.grp ? g.grp[gi.x] : g, g.grp ? (int64_t)gi.y : item, on, gl);
  }
}

template <int EPI>
void launch_real(const GemmArgs& g, cudaStream_t st) {
  const int64_t grid = (g.n_items + THREADS - 1) / THREADS;
  RT_REQUIRE(grid < (1ll << 31), RT_EINTERNAL, "grid too large");
  k_gemm4_r32<EPI><<<(unsigned)grid, THREADS, 0, st>>>(g);
  RT_CUDA_CHECK(cudaGetLastError());
}

template <bool BDAG, int EPI>
void launch_one(const GemmArgs& g, cudaStream_t st) {
  int64_t grid = (g.n_items + C_ITEMS - 1) / C_ITEMS;
  if (g.persistent) {
    int dev = 0, sms = 0;
    RT_CUDA_CHECK(cudaGetDevice(&dev));
    RT_CUDA_CHECK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    grid = std::min<int64_t>(grid, (int64_t)sms * C_CTAS);
  }
  RT_REQUIRE(grid < (1ll << 31), RT_EINTERNAL, "grid too large");
  k_gemm4_f32<BDAG, EPI><<<(unsigned)grid, THREADS, 0, st>>>(g);
  RT_CUDA_CHECK(cudaGetLastError());
}

}  // namespace f32b4

// Launches the FP32 kernels for 4-function blocks; false if the variant is
// not one of theirs (the generic kernel then runs it).
bool launch_gemm4_f32(bool cplx, bool a_dag, bool b_dag, Epilogue epi, const GemmArgs& g, cudaStream_t st) {
  using namespace f32b4;
  RT_REQUIRE(!(g.grp || g.persistent) || cplx, RT_EINTERNAL, "grouped and persistent launches are complex products");
  RT_REQUIRE(!g.base || (cplx && !b_dag && epi == EPI_STORE) || epi == EPI_DELTA_SANDWICH, RT_EINTERNAL,
             "W = dK + M comes with the complex store epilogue");
  if (a_dag) return false;
  if (g.n_items == 0) return true;
  if (!cplx) {
    if (b_dag) return false;
    if (epi == EPI_STORE) return launch_real<EPI_STORE>(g, st), true;
    if (epi == EPI_STORE_ACC) return launch_real<EPI_STORE_ACC>(g, st), true;
    if (epi == EPI_ADD) return launch_real<EPI_ADD>(g, st), true;
    return false;
  }
  if (!b_dag) {
    if (epi == EPI_STORE) return launch_one<false, EPI_STORE>(g, st), true;
    if (epi == EPI_ADD) return launch_one<false, EPI_ADD>(g, st), true;
    return false;
  }
  if (epi == EPI_STORE) return launch_one<true, EPI_STORE>(g, st), true;
  if (epi == EPI_DELTA_SANDWICH) return launch_one<true, EPI_DELTA_SANDWICH>(g, st), true;
  return false;
}

}  // namespace rt
