// adjoint.cu -- hand-written reverse-mode derivative of the batched forward model (the paper
// has no gradient path; this serves gradient-based samplers and Fisher matrices).
//
// Forward (recalled):  K_l(v) = sum_m w_ml sigma_m(P_l, T_l; v) + rho_l R(v)
//                              + sum_q c_ql sigma_q(T_l; v) + kappa c_l          (Sec. 4.4, 8.1)
//                      tau_j(v) = sum_{l>=j} DL[j][l] K_l(v)                     (Sec. 4)
//                      D(v) = (R_p/R_s)^2 + sum_j a_j (1 - e^{-tau_j(v)})        (Sec. 4)
//                      D_bin,k = sum_v w_kv D(v) / sum_v w_kv                    (Sec. 4.5)
// Backward, given G_bin = dL/dD_bin (chi^2: 2 (D_bin - obs) / sigma^2):
//   G_D(v)    = sum_k G_bin,k w_kv / sum w_k                    (k_gd)
//   G_tau_j   = G_D a_j e^{-tau_j};  G_a_j = sum_v G_D (1 - e^{-tau_j})
//   G_K_l(v)  = sum_{j<=l} DL[j][l] G_tau_j(v);  G_DL[j][l] = sum_v G_tau_j(v) K_l(v)
//   per layer: sum_v G_K sigma_m, sum_v G_K dsigma_m/dT, sum_v G_K sigma_R,s, CIA alike,
//              sum_v G_K                                          (k_adjoint_tile, FP32:
//              K is the forward's, read back from the workspace's K buffer, the batch taken in
//              runs of items that fit it; or, when asked for, recomputed from the tables with
//              the opacity kernel's per-cell sums and per-layer FMAs, so bit for bit; tau
//              is recomputed; with mixed precision the cross-sections come from the FP16
//              log10 tables, decoded on the fly, and the forward runs the mixed path)
//   then, per atmosphere (FP64 sums; the path-length terms in FP32 from double-float
//   altitudes): path lengths and annulus weights -> radii, the hydrostatic recursion,
//   densities, chemistry, temperature nodes, R_p and the cloud top (k_adjoint_item).  Tile partial sums are added in a fixed order: results are
//   deterministic.
#include <algorithm>
#include <cmath>
#include <cstddef>
#include <cuda_fp16.h>
#include <type_traits>
#include "tma.h"
#include "sum3.h"
#include "tr_internal.h"

namespace tr {
namespace {

constexpr int kAT = 64;           // wavenumbers per adjoint CTA (2 per lane)
constexpr int kAThreads = 256;
constexpr int kAWarps = kAThreads / 32;
constexpr int kRT = 8;            // rays (or layers) per register tile
constexpr int kItemThreads = 256;    // half over layers, half over radii
constexpr int kItemHalf = kItemThreads / 2;

// Float index of element (row, c) of the [rows][kAT] K and G_tau tiles: a row's 16-byte chunks
// are XOR-swizzled by row / 4, so the G_DL blocks' float4 reads of rows 4 apart (one per
// thread) fall in different banks; a lane's float2 stays inside one chunk.
__device__ __forceinline__ int tix(int row, int c) {
  return row * kAT + ((((c >> 2) ^ (row >> 2)) & (kAT / 4 - 1)) << 2) + (c & 3);
}

// Jacobian rows done by one launch of each backward kernel: row r is bin first_bin + r, its slots
// [slot0[r], slot0[r + 1]) hold the wavenumber tiles from tile0[r] on.
constexpr int kMaxRows = 256;        // bins of a gradient or Jacobian
struct RowGroup {
  int n_rows, first_bin;
  int slot0[kMaxRows + 1];
  int tile0[kMaxRows];
};

struct AdjParams {
  FwdParams f;                    // tables and item buffers; wn_begin / wn_count = binned range
  const double* inv_dt;           // [n_t - 1]
  const double* inv_dtc;          // [n_t_cia - 1]
  const float* gd;                // [B][n_in] dL/dD at the native wavenumbers of the range
  int n_in, tiles, n_feat;        // tiles: slots per item of the partial sums
  int first_slot;                 // of the launch (the partial sums' pointers are its slot 0's)
  unsigned ray_mask;              // species with Rayleigh cross-sections that are not all zero
  float* part_a;                  // [B][tiles][npad]
  float* part_dl;                 // [B][tiles][npad][npad]  (ray j, shell l), j <= l
  float* part_f;                  // [B][tiles][max_layers][n_feat]
  float* part_rp;                 // [B][tiles]  sum_v G_D
  const float* kstore;            // the forward's K of the items, or NULL: recompute
  long long kcols;                // columns of a K row in kstore
  // rows.n_rows == 0: one gradient, slot = wavenumber tile, dL/dD from gd.  Else a group of
  // Jacobian rows: dL/dD of a row's slots from its bin's weights (its row of dD_bin/dtheta)
  RowGroup rows;
  const int* t_ptr; const int* t_bin; const double* t_w;   // the bins' transpose (BinsDev)
};

__device__ __forceinline__ float4 as_float4(int4 v) {
  return make_float4(__int_as_float(v.x), __int_as_float(v.y), __int_as_float(v.z),
                     __int_as_float(v.w));
}
// kLayer* flags of a layer descriptor from its third 16 bytes (k_cloud, cloud, pad_s + flags +
// pad_c, pad_f): the flags byte is byte 10 of the 16
__device__ __forceinline__ unsigned d_flags(int4 v) { return ((unsigned)v.z >> 16) & 0xffu; }
static_assert(offsetof(LayerDesc, flags) == 42 && offsetof(LayerDesc, tp) == 20,
              "layer descriptor offsets the header loads assume");

// Packed FP32 pairs beyond ffma2 and fma2 (sm_100 and later): pack2(lo, hi) forms the pair, unpack2
// returns its halves; add2, sub2 and mul2 act on each half, rounded as the scalar operation
// would be.
__device__ __forceinline__ unsigned long long pack2(float lo, float hi) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ float2 unpack2(unsigned long long v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}
__device__ __forceinline__ unsigned long long add2(unsigned long long a, unsigned long long b) {
  unsigned long long r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ unsigned long long sub2(unsigned long long a, unsigned long long b) {
  unsigned long long r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ unsigned long long mul2(unsigned long long a, unsigned long long b) {
  unsigned long long r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}

__device__ __forceinline__ float2 ldg2(const float* p) {
  return __ldg(reinterpret_cast<const float2*>(p));
}

constexpr float kLog2Of10a = 3.32192809488736234787f;

// Two adjacent cross-sections of molecule m at element offset `off` of its table: the FP32
// table, or (F16) the FP16 log10 table decoded, sigma = 10^(h + c_m) by the hardware 2^x.
template <bool F16>
__device__ __forceinline__ float2 sig2(const FwdParams& p, int m, size_t off) {
  if constexpr (F16) {
    const __half2 h = __ldg(reinterpret_cast<const __half2*>(
        reinterpret_cast<const __half*>(p.logsig16) + off));
    const float2 f = __half22float2(h);
    const float c = p.logsig_off[m];
    float a, b;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(a) : "f"((f.x + c) * kLog2Of10a));
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(b) : "f"((f.y + c) * kLog2Of10a));
    return make_float2(a, b);
  } else {
    return ldg2(p.sigma + off);
  }
}

// The same pair as loaded, so that it can be fetched ahead of its use, and its packed value.
template <bool F16>
using SigRaw = std::conditional_t<F16, unsigned, unsigned long long>;
template <bool F16>
__device__ __forceinline__ SigRaw<F16> sig_fetch(const FwdParams& p, size_t off) {
  if constexpr (F16)
    return __ldg(reinterpret_cast<const unsigned*>(reinterpret_cast<const __half*>(p.logsig16) + off));
  else
    return __ldg(reinterpret_cast<const unsigned long long*>(p.sigma + off));
}
template <bool F16>
__device__ __forceinline__ unsigned long long sig_value(SigRaw<F16> v, float c) {
  if constexpr (F16) {
    const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&v));
    float a, b;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(a) : "f"((f.x + c) * kLog2Of10a));
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(b) : "f"((f.y + c) * kLog2Of10a));
    return pack2(a, b);
  } else {
    return v;
  }
}

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// The layer-independent Rayleigh sum sum_s c_s sigma_R,s at wavenumbers w2, w2+1 (zone 0).
__device__ __forceinline__ float2 rayleigh_sum2(const FwdParams& p, int b, int w2) {
  float2 ray = make_float2(0.f, 0.f);
  if (p.ray) {
    const float* rc = p.buf.rayc + (size_t)b * kMaxZones * TR_MAX_SPECIES;   // zone 0
    for (int s = 0; s < p.n_species; ++s) {
      const float c = rc[s];
      if (c != 0.f) {
        const float2 v = ldg2(p.ray + (size_t)s * p.wn_pad + w2);
        ray.x = fmaf(c, v.x, ray.x); ray.y = fmaf(c, v.y, ray.y);
      }
    }
  }
  return ray;
}

// A warp sums the features of its tile's kRT layers two at a time: kRedRows = 2 kRT rows of one
// term per lane.  The pitch (floats) keeps rows 8-byte aligned and 2 banks apart: the lanes' writes
// along a row and the reads of 16 bytes of each row (two wavefronts) do not conflict.
constexpr int kRedPitch = 34, kRedRows = 2 * kRT;
constexpr int kHdr = 12;    // floats of a layer's header: tt, tt, tp, tp, 1/dT, 1/dT, cell, CIA bracket, ttc, 1/dTc

// Dynamic shared memory of a CTA that leaves room for three on an SM (228 KB less 1 KB and the
// rounding of each): up to 101 layers
constexpr size_t kThreeCtaSmem = (228u * 1024u) / 3 - 1024u - 128u;

// Shared memory of a tile.  The path lengths are the packed rows of ItemBuffers::dlp (row l
// holds rays 0 .. pad8(l+1)-1, zero for j > l); the G_K phase may read up to kRT - 1 rows past
// layer N's, inside the arrays that follow, for layers that it does not use.
struct AdjSmem {
  int npad, kt_rows, n_act, n_ray;
  __host__ __device__ AdjSmem(int max_layers, int na, int nr)
      : npad(pad8(max_layers)), kt_rows(max_layers), n_act(na), n_ray(nr) {}
  // a warp's feature buffers: term rows, layer headers, sums.  They reuse the K tile's space (K
  // is not read after the G_DL phase) when they fit there, else follow the other buffers
  __host__ __device__ size_t red_floats() const { return kRedRows * kRedPitch + kHdr * kRT + (size_t)((kRT * n_act + 3) & ~3); }
  __host__ __device__ bool red_in_kt() const { return kAWarps * red_floats() <= (size_t)kt_rows * kAT; }
  __host__ __device__ size_t dl_floats() const { return dlp_offset(kt_rows); }
  // the tile's Rayleigh rows (layer-independent) are staged once: n_ray x kAT floats
  __host__ __device__ size_t floats() const {
    return (size_t)kt_rows * kAT + dl_floats() + npad + (size_t)npad * kAT + kAT +
           (size_t)n_ray * kAT + (red_in_kt() ? 0 : kAWarps * red_floats());
  }
};

// One CTA per (item, 64-wavenumber tile); grid (items, tiles).  Bound by instruction latency: the
// three contractions (FP32 FMAs) are a third of the instructions, the feature sums most of the rest,
// and a warp waits 5 to 9 cycles between two of them.  So the design is for warps in flight and
// few instructions: the path lengths once, packed (21 KB at 100 layers instead of 43), so that
// three CTAs share an SM (1.62 ms against 1.81 with two; 1,024 atmospheres of 100 layers, 15 tiles,
// 5 absorbers); each absorber's corner rows alone in registers, 80 a thread, fetched one run of
// layers ahead; eight layers' terms of two features summed by all 32 lanes at once; and loops kept
// rolled for the instruction cache.  Before (one layer at a time, all absorbers' rows in 128
// registers, two CTAs): 2.12 ms; 320 atmospheres of 296 tiles with CIA 15.6 ms, now 11.4.
// RECOMP: K recomputed from the tables (a.kstore is NULL) or read from the forward's buffer;
// instantiated separately, so each form's registers are allocated for its own K phase.
template <bool F16, bool RECOMP, int CTAS>
__global__ void __launch_bounds__(kAThreads, CTAS)
k_adjoint_tile(AdjParams a) {
  extern __shared__ __align__(16) float smem[];
  __shared__ __align__(8) uint64_t bar;
  const FwdParams& p = a.f;
  // items fastest: the CTAs in flight share one tile's table rows in L2 (320 atmospheres on tables
  // of 200,000 wavenumbers: 11.4 ms against 12.1 with the tiles fastest)
  const int b = blockIdx.x, tile = blockIdx.y;            // tile: slot of the launch
  const bool jac = a.rows.n_rows > 0;
  const int slot = a.first_slot + tile;
  int row = 0;                                          // the last row whose slots begin at or before
  for (int hi = a.rows.n_rows; row + 1 < hi;) {
    const int mid = (row + hi) >> 1;
    if (a.rows.slot0[mid] <= slot) row = mid; else hi = mid;
  }
  const int wtile = jac ? a.rows.tile0[row] + slot - a.rows.slot0[row] : slot;   // wavenumber tile
  const int jac_bin = jac ? a.rows.first_bin + row : -1;
  const int N = p.buf.items[b].n_layers;
  if (N == 0) return;                                   // the item kernel zeroes its gradient
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int n_ray = __popc(a.ray_mask), n_zero = p.n_species - n_ray, n_act = a.n_feat - n_zero;
  const AdjSmem sp(p.max_layers, n_act, n_ray);
  const int npad = sp.npad;
  float* Kt = smem;                                     // [max_layers][kAT]
  float* DLT = Kt + (size_t)sp.kt_rows * kAT;           // path lengths (AdjSmem)
  float* a_s = DLT + sp.dl_floats();                    // [npad]
  float* Gt = a_s + npad;                               // [npad][kAT]  G_tau
  float* gd_s = Gt + (size_t)npad * kAT;                // [kAT]
  float* ray_s = gd_s + kAT;                            // [n_ray][kAT] Rayleigh rows
  float* red = (sp.red_in_kt() ? Kt : ray_s + (size_t)n_ray * kAT) + warp * sp.red_floats();
  const int w_first = wn_first(p.wn_begin) + wtile * kAT;

  if (threadIdx.x == 0) { mbar_init(&bar, 1); mbar_fence_init(); }
  __syncthreads();
  if (threadIdx.x == 0) {
    const uint32_t dl_bytes = (uint32_t)(sizeof(float) * (size_t)dlp_offset(N));
    mbar_arrive_expect_tx(&bar, dl_bytes + (uint32_t)(sizeof(float) * npad));
    bulk_g2s(DLT, p.buf.dlp + (size_t)b * dlp_offset(p.max_layers), dl_bytes, &bar);
    bulk_g2s(a_s, p.buf.aj + (size_t)b * npad, (uint32_t)(sizeof(float) * npad), &bar);
  }
  for (int i = threadIdx.x; i < kAT; i += kAThreads) {
    const int w = w_first + i;
    float g = 0.f;
    if (w >= p.wn_begin && w < p.wn_begin + a.n_in) {
      const int k = w - p.wn_begin;
      if (jac_bin < 0) {
        g = a.gd[(size_t)b * a.n_in + k];
      } else {                                          // dD_bin,jac_bin / dD at w
        for (int e = a.t_ptr[k]; e < a.t_ptr[k + 1]; ++e)
          if (a.t_bin[e] == jac_bin) g = (float)a.t_w[e];
      }
    }
    gd_s[i] = g;
  }
  if (p.ray) {                                          // the Rayleigh rows of this tile
    for (int i = threadIdx.x; i < n_ray * kAT; i += kAThreads) {
      const int r = i / kAT, c = i - r * kAT, w = w_first + c;
      unsigned m = a.ray_mask;                          // its r-th species
      for (int q = 0; q < r; ++q) m &= m - 1u;
      ray_s[i] = w < p.wn_pad ? __ldg(p.ray + (size_t)(__ffs(m) - 1) * p.wn_pad + w) : 0.f;
    }
  }
  // ---- K tile: the forward's, or recomputed
  const int w2 = w_first + 2 * lane;
  const bool in_row = w2 < p.wn_pad;
  const LayerDesc* LD = p.buf.layers + (size_t)b * p.max_layers;
  if constexpr (!RECOMP) {
    const float* ks = a.kstore + k_index(b, (long long)wtile * kAT + 2 * lane, 0, a.kcols, p.max_layers);
    for (int l = warp; l < N; l += kAWarps)
      *reinterpret_cast<float2*>(Kt + tix(l, 2 * lane)) =
          __ldg(reinterpret_cast<const float2*>(ks + (size_t)l * kKTile));
  } else {
    // K recomputed with the opacity kernel's arithmetic, so that it equals the stored K bit
    // for bit: per (P, T) cell the molecule sums us_c = sum_m (x_m / x_max) sigma_m,c and per
    // CIA bracket the pair sums uc_t = sum_q (y_q / y_max) sigma_q,t, in species order; per
    // layer kc + rho sigma_R + sum_c w_c us_c + sum_t y_t uc_t with the layer's coefficients
    // (Sec. 5, Sec. 8.1).  Each warp takes a contiguous run of layers, reads their brackets
    // and coefficients 32 layers per warp-wide load, and gathers a cell's corner rows only
    // when the cell changes (consecutive layers share it).
    const float2 ray = in_row ? rayleigh_sum2(p, b, w2) : make_float2(0.f, 0.f);
    const float* ox = p.buf.opx + (size_t)b * kMaxZones * kOpxStride;     // zone 0 weights
    const float4* opb = p.buf.op + (size_t)b * p.max_layers * 2;
    const size_t slab_t = (size_t)p.wn_pad, slab_p = (size_t)p.n_t * p.wn_pad;
    const int wq = in_row ? w2 : 0;
    const int per = (N + kAWarps - 1) / kAWarps;
    const int lb = min(N, warp * per), le = min(N, lb + per);
    int c_ip = -1, c_it = -1, c_itc = -1;
    float us[4][2] = {}, uc[2][2] = {};
    for (int l0 = lb; l0 < le; l0 += 32) {
      const int li = l0 + lane;
      int4 h = make_int4(0, 0, 0, 0);
      float4 ha = make_float4(0.f, 0.f, 0.f, 0.f), hb = ha;
      if (li < le) {
        h = __ldg(reinterpret_cast<const int4*>(LD + li));      // ip, it, itc, zone
        ha = __ldg(opb + 2 * li);
        hb = __ldg(opb + 2 * li + 1);
      }
      const int n_here = min(32, le - l0);
      for (int i = 0; i < n_here; ++i) {
        const int ip = __shfl_sync(0xffffffffu, h.x, i), it = __shfl_sync(0xffffffffu, h.y, i);
        const int itc = __shfl_sync(0xffffffffu, h.z, i);
        if (ip != c_ip || it != c_it) {                  // a new cell (warp-uniform)
          const size_t o0 = ((size_t)ip * p.n_t + it) * p.wn_pad + wq;
#pragma unroll
          for (int c = 0; c < 4; ++c) us[c][0] = us[c][1] = 0.f;
#pragma unroll
          for (int m = 0; m < TR_MAX_MOL; ++m) {
            if (m < p.n_mol) {
              const float xm = __ldg(ox + m);
              const size_t om = o0 + (size_t)m * p.n_p * slab_p;
              const float2 v0 = sig2<F16>(p, m, om), v1 = sig2<F16>(p, m, om + slab_t),
                           v2 = sig2<F16>(p, m, om + slab_p),
                           v3 = sig2<F16>(p, m, om + slab_p + slab_t);
              us[0][0] = fmaf(xm, v0.x, us[0][0]); us[0][1] = fmaf(xm, v0.y, us[0][1]);
              us[1][0] = fmaf(xm, v1.x, us[1][0]); us[1][1] = fmaf(xm, v1.y, us[1][1]);
              us[2][0] = fmaf(xm, v2.x, us[2][0]); us[2][1] = fmaf(xm, v2.y, us[2][1]);
              us[3][0] = fmaf(xm, v3.x, us[3][0]); us[3][1] = fmaf(xm, v3.y, us[3][1]);
            }
          }
          c_ip = ip; c_it = it;
        }
        if (p.n_cia > 0 && itc != c_itc) {              // a new CIA bracket (warp-uniform)
          uc[0][0] = uc[0][1] = uc[1][0] = uc[1][1] = 0.f;
#pragma unroll
          for (int q = 0; q < TR_MAX_CIA; ++q) {
            if (q < p.n_cia) {
              const float yq = __ldg(ox + TR_MAX_MOL + q);
              const float* bq = p.cia + ((size_t)q * p.n_t_cia + itc) * p.wn_pad + wq;
              const float2 c0 = ldg2(bq), c1 = ldg2(bq + p.wn_pad);
              uc[0][0] = fmaf(yq, c0.x, uc[0][0]); uc[0][1] = fmaf(yq, c0.y, uc[0][1]);
              uc[1][0] = fmaf(yq, c1.x, uc[1][0]); uc[1][1] = fmaf(yq, c1.y, uc[1][1]);
            }
          }
          c_itc = itc;
        }
        const float w0 = __shfl_sync(0xffffffffu, ha.x, i), w1 = __shfl_sync(0xffffffffu, ha.y, i);
        const float wc2 = __shfl_sync(0xffffffffu, ha.z, i), w3 = __shfl_sync(0xffffffffu, ha.w, i);
        const float y0 = __shfl_sync(0xffffffffu, hb.x, i), y1 = __shfl_sync(0xffffffffu, hb.y, i);
        const float rho = __shfl_sync(0xffffffffu, hb.z, i), kc = __shfl_sync(0xffffffffu, hb.w, i);
        float k0 = fmaf(rho, ray.x, kc), k1 = fmaf(rho, ray.y, kc);
        k0 = fmaf(w0, us[0][0], k0); k1 = fmaf(w0, us[0][1], k1);
        k0 = fmaf(w1, us[1][0], k0); k1 = fmaf(w1, us[1][1], k1);
        k0 = fmaf(wc2, us[2][0], k0); k1 = fmaf(wc2, us[2][1], k1);
        k0 = fmaf(w3, us[3][0], k0); k1 = fmaf(w3, us[3][1], k1);
        k0 = fmaf(y0, uc[0][0], k0); k1 = fmaf(y0, uc[0][1], k1);
        k0 = fmaf(y1, uc[1][0], k0); k1 = fmaf(y1, uc[1][1], k1);
        *reinterpret_cast<float2*>(Kt + tix(l0 + i, 2 * lane)) =
            in_row ? make_float2(k0, k1) : make_float2(0.f, 0.f);
      }
    }
  }
  const bool ok = __syncthreads_and(mbar_wait_bounded(&bar, 0, p.dev_err, TR_DEVERR_TIMEOUT));
  if (!ok) { mbar_wait_bounded(&bar, 0, nullptr, 0); return; }
  // this lane's float2 in row l of the swizzled tiles: chunk lane / 2 of 16, XORed with row / 4
  const int lane_c = 2 * (lane & 1);
  auto lane_col = [&](int row) { return ((((lane >> 1) ^ (row >> 2)) & (kAT / 4 - 1)) << 2) + lane_c; };

  const size_t item_tile = (size_t)b * a.tiles + tile;
  // ---- tau, G_tau = G_D a_j e^-tau, G_a_j = sum_v G_D (1 - e^-tau)
  const float2 g2 = *reinterpret_cast<const float2*>(gd_s + 2 * lane);
  const int n_rt = (N + kRT - 1) / kRT;
  for (int round = 0;; ++round) {
    const int pos = (round & 1) ? (kAWarps - 1 - warp) : warp;
    const int rt = round * kAWarps + pos;
    if (rt >= n_rt) break;
    const int j0 = rt * kRT;
    // packed FP32 pairs: rays (2r, 2r+1) at the lane's two wavenumbers
    unsigned long long acc2[kRT / 2][2];
#pragma unroll
    for (int r = 0; r < kRT / 2; ++r) acc2[r][0] = acc2[r][1] = 0ull;
    auto tau_row = [&](const float* kr, const float* dr) {
      const float2 kv = *reinterpret_cast<const float2*>(kr);
      const ulonglong2 d0 = *reinterpret_cast<const ulonglong2*>(dr);
      const ulonglong2 d1 = *reinterpret_cast<const ulonglong2*>(dr + 4);
      const unsigned long long dv[4] = {d0.x, d0.y, d1.x, d1.y};
      const unsigned long long k0 = pack_dup(kv.x), k1 = pack_dup(kv.y);
#pragma unroll
      for (int r = 0; r < kRT / 2; ++r) { ffma2(acc2[r][0], dv[r], k0); ffma2(acc2[r][1], dv[r], k1); }
    };
    // four rows share the swizzle and the row length (l a multiple of 4)
    for (int l = j0; l < N; l += 4) {
      const float* kr = Kt + l * kAT + lane_col(l);
      const int pitch = pad8(l + 1);
      const float* dr = DLT + dlp_offset(l) + j0;
      if (l + 4 <= N) {
#pragma unroll
        for (int u = 0; u < 4; ++u) tau_row(kr + u * kAT, dr + u * pitch);
      } else {
#pragma unroll 1
        for (int u = 0; l + u < N; ++u) tau_row(kr + u * kAT, dr + u * pitch);
      }
    }
    float acc[kRT][2];
#pragma unroll
    for (int r = 0; r < kRT / 2; ++r)
#pragma unroll
      for (int c = 0; c < 2; ++c)
        asm("mov.b64 {%0, %1}, %2;" : "=f"(acc[2 * r][c]), "=f"(acc[2 * r + 1][c]) : "l"(acc2[r][c]));
    float ga[kRT];
#pragma unroll
    for (int r = 0; r < kRT; ++r) {
      const int j = j0 + r;
      const float aj = a_s[j];
      const float e0 = __expf(-acc[r][0]), e1 = __expf(-acc[r][1]);
      *reinterpret_cast<float2*>(Gt + tix(j, 2 * lane)) = make_float2(g2.x * aj * e0, g2.y * aj * e1);
      ga[r] = g2.x * (1.f - e0) + g2.y * (1.f - e1);
    }
    // the eight rays' sums over the warp, halving the rays as the lanes pair up (16, 8, 4 apart,
    // then 2 and 1): lane 4r ends with the sum of ray r
#pragma unroll
    for (int o = 16, n = kRT / 2; o >= 4; o >>= 1, n >>= 1) {
      const bool up = lane & o;
#pragma unroll
      for (int r = 0; r < n; ++r) {
        const float mine = up ? ga[r + n] : ga[r], other = up ? ga[r] : ga[r + n];
        ga[r] = mine + __shfl_xor_sync(0xffffffffu, other, o);
      }
    }
    ga[0] += __shfl_xor_sync(0xffffffffu, ga[0], 2);
    ga[0] += __shfl_xor_sync(0xffffffffu, ga[0], 1);
    if (!(lane & 3)) a.part_a[item_tile * npad + j0 + (lane >> 2)] = ga[0];
  }
  for (int j = N + threadIdx.x; j < npad; j += kAThreads) {
    for (int c = 0; c < kAT; ++c) Gt[(size_t)j * kAT + c] = 0.f;
    a.part_a[item_tile * npad + j] = 0.f;
  }
  if (warp == 0) {
    const float s = warp_sum(g2.x + g2.y);
    if (lane == 0) a.part_rp[item_tile] = s;
  }
  __syncthreads();

  // ---- G_DL[j][l] = sum_v G_tau_j(v) K_l(v), j <= l, 4 x 4 blocks
  {
    const int nb = (N + 3) / 4;
    const int n_pairs = nb * (nb + 1) / 2;
    float* pdl = a.part_dl + item_tile * (size_t)npad * npad;
    for (int pi = threadIdx.x; pi < n_pairs; pi += kAThreads) {
      int lb = (int)((sqrtf(8.f * pi + 1.f) - 1.f) * 0.5f);
      while (lb * (lb + 1) / 2 > pi) --lb;
      while ((lb + 1) * (lb + 2) / 2 <= pi) ++lb;
      const int jb = pi - lb * (lb + 1) / 2;
      const int j0 = 4 * jb, l0 = 4 * lb;
      // packed FP32 pairs: acc2[x][y] holds the even- and odd-wavenumber halves of the sum
      unsigned long long acc2[4][4];
#pragma unroll
      for (int x = 0; x < 4; ++x) acc2[x][0] = acc2[x][1] = acc2[x][2] = acc2[x][3] = 0ull;
#pragma unroll 2
      for (int c = 0; c < kAT; c += 4) {
        ulonglong2 g[4], k[4];
#pragma unroll
        for (int x = 0; x < 4; ++x) {
          g[x] = *reinterpret_cast<const ulonglong2*>(Gt + tix(j0 + x, c));
          k[x] = (l0 + x < N) ? *reinterpret_cast<const ulonglong2*>(Kt + tix(l0 + x, c))
                              : make_ulonglong2(0ull, 0ull);
        }
#pragma unroll
        for (int x = 0; x < 4; ++x)
#pragma unroll
          for (int y = 0; y < 4; ++y) {
            ffma2(acc2[x][y], g[x].x, k[y].x);
            ffma2(acc2[x][y], g[x].y, k[y].y);
          }
      }
      // whole 16-byte rows: the entries with l < j or l >= N are not read
#pragma unroll
      for (int x = 0; x < 4; ++x) {
        float v[4];
#pragma unroll
        for (int y = 0; y < 4; ++y) {
          const float2 e = unpack2(acc2[x][y]);
          v[y] = j0 + x <= l0 + y && l0 + y < N ? e.x + e.y : 0.f;
        }
        if (j0 + x < N)
          *reinterpret_cast<float4*>(pdl + (size_t)(j0 + x) * npad + l0) = make_float4(v[0], v[1], v[2], v[3]);
      }
    }
  }

  // ---- G_K_l(v) = sum_{j<=l} DL[j][l] G_tau_j(v) over 8-layer tiles, then per-layer sums
  if (sp.red_in_kt()) __syncthreads();                  // every warp is done reading K
  const int n_lt = (N + kRT - 1) / kRT;
  const int nm = p.n_mol, nq = p.n_cia;
  // columns of the sums: the features without the species that have no Rayleigh cross-sections,
  // whose sums are zero
  const int f_dS = nm, f_R = 2 * nm, f_C = 2 * nm + n_ray, f_dC = f_C + nq, f_K = f_dC + nq;
  auto column_of = [&](int f) -> int {                  // feature f's column, or -1: zero
    if (f < 2 * nm) return f;
    const int sp_i = f - 2 * nm;
    if (sp_i >= p.n_species) return f - n_zero;
    return (a.ray_mask >> sp_i) & 1u ? f_R + __popc(a.ray_mask & ((1u << sp_i) - 1u)) : -1;
  };
  float* hd = red + kRedRows * kRedPitch;               // [kRT][kHdr]
  float* sums = hd + kHdr * kRT;                        // [kRT][n_act]
  const size_t slab_t = (size_t)p.wn_pad, slab_p = (size_t)p.n_t * p.wn_pad;
  const int wq = in_row ? w2 : 0;
  // a tile's cost grows with its layer index (the contraction runs over j <= l), so the warps
  // take the tiles from the top down, in a snake over the warps: the largest tiles first, then
  // the smallest ones to the warps that took the smaller of the large ones
  for (int round = 0;; ++round) {
    const int pos = (round & 1) ? (kAWarps - 1 - warp) : warp;
    const int kt = round * kAWarps + pos;
    if (kt >= n_lt) break;
    const int lt = n_lt - 1 - kt;
    const int l0 = lt * kRT, nr = min(kRT, N - l0);
    // the tile's layer headers (brackets, weights and reciprocal T spacings), lane r holding
    // layer l0 + r's: loaded before the contraction so that their latency overlaps it
    int cell = 0, itc = 0;
    float tp = 0.f, tt = 0.f, ttc = 0.f, idt = 0.f, idc = 0.f;
    if (lane < nr) {
      const int4* dd = reinterpret_cast<const int4*>(LD + l0 + lane);
      const int4 hb = __ldg(dd);                         // ip, it, itc
      const float4 hw = as_float4(__ldg(dd + 1));        // rho, tp, tt, ttc
      const unsigned fl = d_flags(__ldg(dd + 2));
      cell = hb.x * p.n_t + hb.y; itc = hb.z;
      tp = hw.y; tt = hw.z; ttc = hw.w;
      idt = (fl & kLayerTClamp) ? 0.f : (float)a.inv_dt[hb.y];
      idc = (nq > 0 && !(fl & kLayerTcClamp)) ? (float)a.inv_dtc[hb.z] : 0.f;
    }
    float acc[kRT][2];
    {
#pragma unroll
      for (int r = 0; r < kRT; ++r) acc[r][0] = acc[r][1] = 0.f;
      // rows l0 .. l0 + 7 of the packed path lengths have one length; four rays at a time (one
      // 16-byte load a row; they share the swizzle).  Rays beyond N: both factors are zero
      const int pitch = l0 + kRT;
      const float* dr = DLT + dlp_offset(l0);
      const int jmax = min(N, l0 + kRT);
      for (int j = 0; j < jmax; j += 4) {
        float4 d[kRT];
#pragma unroll
        for (int r = 0; r < kRT; ++r) d[r] = *reinterpret_cast<const float4*>(dr + r * pitch + j);
        const float* gr = Gt + j * kAT + lane_col(j);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const float2 g = *reinterpret_cast<const float2*>(gr + u * kAT);
#pragma unroll
          for (int r = 0; r < kRT; ++r) {
            const float dl = u == 0 ? d[r].x : u == 1 ? d[r].y : u == 2 ? d[r].z : d[r].w;
            acc[r][0] = fmaf(dl, g.x, acc[r][0]);
            acc[r][1] = fmaf(dl, g.y, acc[r][1]);
          }
        }
      }
    }
    if (!in_row) {
#pragma unroll
      for (int r = 0; r < kRT; ++r) acc[r][0] = acc[r][1] = 0.f;
    }
    // layers where the (P, T) cell and the CIA bracket change: runs of layers share their rows
    const int cell_b = __shfl_up_sync(0xffffffffu, cell, 1), itc_b = __shfl_up_sync(0xffffffffu, itc, 1);
    const unsigned chg = __ballot_sync(0xffffffffu, lane < nr && (lane == 0 || cell != cell_b));
    const unsigned chc = __ballot_sync(0xffffffffu, lane < nr && (lane == 0 || itc != itc_b));
    if (lane < nr) {
      float* h = hd + kHdr * lane;
      *reinterpret_cast<float4*>(h) = make_float4(tt, tt, tp, tp);
      *reinterpret_cast<float4*>(h + 4) = make_float4(idt, idt, __int_as_float(cell), __int_as_float(itc));
      *reinterpret_cast<float2*>(h + 8) = make_float2(ttc, idc);
    }
    __syncwarp();
    // the sums of columns fa and fb (rows 2r and 2r + 1 hold layer r's terms of each): lanes 2i
    // and 2i + 1 add row i's terms 0, 1 and 2, 3 mod 4 as chains in lane order
    auto reduce = [&](int fa, int fb) {
      __syncwarp();
      const unsigned long long* row = reinterpret_cast<const unsigned long long*>(
          red + (lane >> 1) * kRedPitch + 2 * (lane & 1));
      unsigned long long t = 0ull;
#pragma unroll
      for (int k = 0; k < 8; ++k) t = add2(t, row[2 * k]);
      const float2 u = unpack2(t);
      float v = u.x + u.y;
      v += __shfl_xor_sync(0xffffffffu, v, 1);
      const int f = lane & 2 ? fb : fa;
      if (!(lane & 1) && f >= 0) sums[(lane >> 2) * n_act + f] = v;
      __syncwarp();                                      // the rows are free again
    };
    // absorbers, one at a time: the rows of the next run's (or the next absorber's first) cell
    // are fetched while a run's layers are done
    SigRaw<F16> nx[4];
    auto fetch = [&](int m, int r) {
      const size_t o = ((size_t)m * p.n_p * p.n_t + __float_as_int(hd[kHdr * r + 6])) * slab_t + wq;
      nx[0] = sig_fetch<F16>(p, o);
      nx[1] = sig_fetch<F16>(p, o + slab_t);
      nx[2] = sig_fetch<F16>(p, o + slab_p);
      nx[3] = sig_fetch<F16>(p, o + slab_p + slab_t);
    };
    if (nm > 0) fetch(0, 0);
    const unsigned long long one2 = pack_dup(1.f);
    // The layers four at a time in a loop: unrolled over all eight, the kernel's code outgrew the
    // instruction cache (26% of the issue slots were lost to it).
    for (int m = 0; m < nm; ++m) {
      const float c = F16 ? p.logsig_off[m] : 0.f;
      // of the current cell, (v, v + 1) pairs: sigma at the lower T and its step to the upper, at
      // the lower and the upper pressure
      unsigned long long s0 = 0ull, d0 = 0ull, s1 = 0ull, d1 = 0ull;
#pragma unroll 1
      for (int rh = 0; rh < kRT; rh += kRT / 2) {
#pragma unroll
        for (int q = 0; q < kRT / 2; ++q) {
          const int r = rh + q;
          if (r >= nr) break;
          const float gk0 = rh ? acc[q + kRT / 2][0] : acc[q][0], gk1 = rh ? acc[q + kRT / 2][1] : acc[q][1];
          if ((chg >> r) & 1u) {
            s0 = sig_value<F16>(nx[0], c);
            d0 = sub2(sig_value<F16>(nx[1], c), s0);
            s1 = sig_value<F16>(nx[2], c);
            d1 = sub2(sig_value<F16>(nx[3], c), s1);
            const unsigned later = chg & ~((2u << r) - 1u);
            const int mn = later ? m : m + 1;
            if (mn < nm) fetch(mn, later ? __ffs(later) - 1 : 0);
          }
          const float* h = hd + kHdr * r;
          const ulonglong2 t = *reinterpret_cast<const ulonglong2*>(h);          // (tt, tt), (tp, tp)
          const unsigned long long idt2 = *reinterpret_cast<const unsigned long long*>(h + 4);
          // sigma(T) at both pressures, then sigma(P); d sigma / dT of the same bracket
          const unsigned long long a1 = fma2(d0, t.x, s0), a2 = fma2(d1, t.x, s1);
          const float2 sg = unpack2(fma2(sub2(a2, a1), t.y, a1));
          const float2 dt = unpack2(mul2(fma2(d0, sub2(one2, t.y), mul2(d1, t.y)), idt2));
          red[2 * r * kRedPitch + lane] = fmaf(gk0, sg.x, gk1 * sg.y);
          red[(2 * r + 1) * kRedPitch + lane] = fmaf(gk0, dt.x, gk1 * dt.y);
        }
      }
      reduce(m, f_dS + m);
    }
    if (nq > 0) {
      // CIA pairs alike: two rows of the bracket
      float2 nc[2];
      auto fetch_c = [&](int q, int r) {
        const float* bq = p.cia + ((size_t)q * p.n_t_cia + __float_as_int(hd[kHdr * r + 7])) * p.wn_pad + wq;
        nc[0] = ldg2(bq);
        nc[1] = ldg2(bq + p.wn_pad);
      };
      fetch_c(0, 0);
#pragma unroll 1
      for (int q = 0; q < nq; ++q) {
        float2 c0 = make_float2(0.f, 0.f), c1 = c0;
#pragma unroll 1
        for (int rh = 0; rh < kRT; rh += kRT / 2) {
#pragma unroll
          for (int i = 0; i < kRT / 2; ++i) {
            const int r = rh + i;
            if (r >= nr) break;
            const float gk0 = rh ? acc[i + kRT / 2][0] : acc[i][0], gk1 = rh ? acc[i + kRT / 2][1] : acc[i][1];
            if ((chc >> r) & 1u) {
              c0 = nc[0]; c1 = nc[1];
              const unsigned later = chc & ~((2u << r) - 1u);
              const int qn = later ? q : q + 1;
              if (qn < nq) fetch_c(qn, later ? __ffs(later) - 1 : 0);
            }
            const float2 h = *reinterpret_cast<const float2*>(hd + kHdr * r + 8);   // ttc, 1/dTc
            const float sg0 = c0.x + (c1.x - c0.x) * h.x, sg1 = c0.y + (c1.y - c0.y) * h.x;
            red[2 * r * kRedPitch + lane] = gk0 * sg0 + gk1 * sg1;
            red[(2 * r + 1) * kRedPitch + lane] = gk0 * (c1.x - c0.x) * h.y + gk1 * (c1.y - c0.y) * h.y;
          }
        }
        reduce(f_C + q, f_dC + q);
      }
    }
    // Rayleigh species and, last, the plain sum
#pragma unroll 1
    for (int i = 0; i <= n_ray; i += 2) {
#pragma unroll 1
      for (int h = 0; h < 2; ++h) {
        if (i + h < n_ray) {
          const float2 v = *reinterpret_cast<const float2*>(ray_s + (i + h) * kAT + 2 * lane);
#pragma unroll
          for (int r = 0; r < kRT; ++r) red[(2 * r + h) * kRedPitch + lane] = acc[r][0] * v.x + acc[r][1] * v.y;
        } else if (i + h == n_ray) {
#pragma unroll
          for (int r = 0; r < kRT; ++r) red[(2 * r + h) * kRedPitch + lane] = acc[r][0] + acc[r][1];
        }
      }
      reduce(i < n_ray ? f_R + i : f_K, i + 1 < n_ray ? f_R + i + 1 : i + 1 == n_ray ? f_K : -1);
    }
    float* pf = a.part_f + (item_tile * p.max_layers + l0) * a.n_feat;
    for (int f = lane; f < a.n_feat; f += 32) {
      const int col = column_of(f);
      for (int r = 0; r < nr; ++r) pf[r * a.n_feat + f] = col >= 0 ? sums[r * n_act + col] : 0.f;
    }
    __syncwarp();                                        // headers and sums are free for the next tile
  }
}

// dL/dD at native wavenumbers of the binned range (blockIdx.y: a run of kGdRun of them), and chi^2
// (chi^2 mode) per item.  Latency-bound: the bins' terms are taken in parallel (one thread's
// serial sum with a division per bin held the kernel at 33 us whatever the batch).
constexpr int kGdThreads = 256, kGdRun = 2048;
__global__ void __launch_bounds__(kGdThreads)
k_gd(BinsDev bd, int B, const double* __restrict__ binned, const double* __restrict__ obs,
     const double* __restrict__ sig, const double* __restrict__ gbin,
     const ItemGeom* __restrict__ items, double* __restrict__ chi2, float* __restrict__ gd, int n_in) {
  __shared__ double gb[256];
  __shared__ double red[kGdThreads / 32];
  const int b = blockIdx.x, t = threadIdx.x;
  const bool valid = items[b].status == TR_OK;
  const double* Db = binned + (size_t)b * bd.n_bin;
  double c = 0.0;
  if (t < bd.n_bin) {                                   // at most 256 bins
    double g = 0.0;
    if (gbin) {
      if (valid) g = gbin[(size_t)b * bd.n_bin + t];
    } else {
      const double d = Db[t] - obs[t], s = sig[t], r = d / s;
      if (valid) g = 2.0 * d / (s * s);
      c = r * r;
    }
    gb[t] = g;
  }
  __syncthreads();
  const int i1 = min(n_in, (int)(blockIdx.y + 1) * kGdRun);
  for (int i = blockIdx.y * kGdRun + t; i < i1; i += kGdThreads) {
    double g = 0.0;
    for (int e = bd.t_ptr[i]; e < bd.t_ptr[i + 1]; ++e) g += gb[bd.t_bin[e]] * bd.t_w[e];
    gd[(size_t)b * n_in + i] = (float)g;
  }
  if (chi2 && !gbin && blockIdx.y == 0) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
    if ((t & 31) == 0) red[t >> 5] = c;
    __syncthreads();
    if (t == 0) {
      for (int k = 1; k < (min(bd.n_bin, kGdThreads) + 31) / 32; ++k) c += red[k];
      chi2[b] = valid ? c : INFINITY;
    }
  }
}

// Sum of the wavenumber tiles' partial sums of one array [B][tiles][M] into its tile-0 slot,
// in tile order (deterministic), compensated (Kahan) so the FP32 sum of hundreds of tiles
// keeps about FP32 rounding; blockIdx.y picks the array.  Consecutive threads take
// consecutive elements, so every tile's row is read coalesced.  An array with tri > 0 is a
// [tri][tri] matrix of which only the entries (j, l) with l >= j are written and read (the
// G_DL partial sums): a warp whose 32 entries all lie below the diagonal skips them (a
// whole warp, so that the warps' long tile loops do not diverge; B tri^2 is a multiple of
// 64, so a warp's lanes leave the grid-stride loop together).
struct TileSumArgs {
  float* arr[4];
  long long m[4];
  int tri[4];
  int slots;                      // slots per item
  RowGroup rows;                  // n_rows == 0: one row of all slots
};
__global__ void k_adjoint_sum(TileSumArgs ts, int B) {
  const int r = blockIdx.z;
  const int s0 = ts.rows.n_rows > 0 ? ts.rows.slot0[r] : 0;
  const int tiles = (ts.rows.n_rows > 0 ? ts.rows.slot0[r + 1] : ts.slots) - s0;
  if (tiles < 2) return;
  float* arr = ts.arr[blockIdx.y];
  const long long M = ts.m[blockIdx.y];
  const int tri = ts.tri[blockIdx.y];
  const long long n = (long long)B * M;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x) {
    const long long b = i / M, m = i - b * M;
    if (tri > 0 && __all_sync(0xffffffffu, (int)m % tri < (int)m / tri)) continue;   // l < j
    float* row = arr + ((size_t)b * ts.slots + s0) * M + m;
    float s = row[0], c = 0.f;
    auto add = [&](int t) {
      const float y = __fsub_rn(row[(size_t)t * M], c);
      const float u = __fadd_rn(s, y);
      c = __fsub_rn(__fsub_rn(u, s), y);
      s = u;
    };
    int t = 1;                                          // eight tiles' loads in flight
    for (; t + 8 <= tiles; t += 8) {
#pragma unroll
      for (int k = 0; k < 8; ++k) add(t + k);
    }
#pragma unroll 4
    for (; t < tiles; ++t) add(t);
    row[0] = s;
  }
}

// Sums of the wavenumber tiles' partial sums into the row's first slot, in tile
// order and compensated as below, four consecutive elements a thread (of G_DL the groups that reach
// the diagonal or lie above it, which alone are read afterwards), 16 bytes a tile, no division by
// the array sizes.  For launches of several waves of such threads: 15 tiles of 1,024 items 123 us
// (135 by the kernel below), the few tiles of each of 50 Jacobian rows of 128 items 88 us (221).
// With fewer items the threads are too few: 58 tiles of 8 items 21 us (10), 296 tiles of two runs
// of 160 items 798 us (639).
struct TileSum4Args {
  float *dl, *a, *f, *rp;
  int npad, n_f, slots;           // slots per item
  RowGroup rows;                  // n_rows == 0: one row of all slots
};
constexpr int kSumThreads = 256;
constexpr long long kSum4Threads = 1 << 20;            // about four waves of the GPU's threads
__device__ __forceinline__ float kahan(float s, float& c, float v) {
  const float y = __fsub_rn(v, c);
  const float u = __fadd_rn(s, y);
  c = __fsub_rn(__fsub_rn(u, s), y);
  return u;
}
__device__ __forceinline__ void sum_tiles4(float* p, size_t stride, int tiles) {
  float4 s = *reinterpret_cast<const float4*>(p), c = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 4
  for (int t = 1; t < tiles; ++t) {
    const float4 v = *reinterpret_cast<const float4*>(p + t * stride);
    s.x = kahan(s.x, c.x, v.x); s.y = kahan(s.y, c.y, v.y);
    s.z = kahan(s.z, c.z, v.z); s.w = kahan(s.w, c.w, v.w);
  }
  *reinterpret_cast<float4*>(p) = s;
}
__device__ __forceinline__ void sum_tiles1(float* p, size_t stride, int tiles) {
  float s = *p, c = 0.f;
#pragma unroll 4
  for (int t = 1; t < tiles; ++t) s = kahan(s, c, p[t * stride]);
  *p = s;
}
__host__ __device__ inline int sum_units(int npad, int n_f) {
  return npad * npad / 4 + npad / 4 + (n_f % 4 == 0 ? n_f / 4 : n_f) + 1;
}
__global__ void __launch_bounds__(kSumThreads) k_adjoint_sum4(TileSum4Args ts) {
  const int b = blockIdx.y, r = blockIdx.z, npad = ts.npad;
  const int s0 = ts.rows.n_rows > 0 ? ts.rows.slot0[r] : 0;
  const int tiles = (ts.rows.n_rows > 0 ? ts.rows.slot0[r + 1] : ts.slots) - s0;
  if (tiles < 2) return;
  const size_t slot = (size_t)b * ts.slots + s0;
  const int q = npad / 4;                               // groups of a G_DL row
  int u = blockIdx.x * kSumThreads + threadIdx.x;
  if (u < npad * q) {
    const int j = u / q, l = 4 * (u - j * q);
    const size_t m = (size_t)npad * npad;
    if (l + 3 >= j) sum_tiles4(ts.dl + slot * m + 4 * (size_t)u, m, tiles);
    return;
  }
  u -= npad * q;
  if (u < q) return sum_tiles4(ts.a + slot * npad + 4 * u, npad, tiles);
  u -= q;
  const bool by4 = ts.n_f % 4 == 0;                     // else a slot's features are not 16-byte aligned
  const int n_f = by4 ? ts.n_f / 4 : ts.n_f;
  if (u < n_f) {
    float* f = ts.f + slot * ts.n_f;
    return by4 ? sum_tiles4(f + 4 * u, ts.n_f, tiles) : sum_tiles1(f + u, ts.n_f, tiles);
  }
  if (u == n_f) sum_tiles1(ts.rp + slot, 1, tiles);
}

struct ItemParams {
  GeomParams gp;
  const double* theta; int n_theta;
  ItemBuffers buf;
  // partial sums [B][slots][...], each row's in its first slot (k_adjoint_sum)
  const float* part_a; const float* part_dl; const float* part_f; const float* part_rp;
  int slots, n_feat;
  double* grad;                   // item b, row r: n_theta values at grad + b * item_stride + r * n_theta
  long long item_stride;
  RowGroup rows;                  // n_rows == 0: one row in slot 0
};

// (ah + al) - (bh + bl) to FP32 working precision (Knuth's TwoSum on the leading parts).
__device__ __forceinline__ float diff_df(float ah, float al, float bh, float bl) {
  const float s = __fsub_rn(ah, bh);
  const float bb = __fsub_rn(s, ah);
  const float e = __fadd_rn(__fsub_rn(ah, __fsub_rn(s, bb)), __fsub_rn(-bh, bb));
  return __fadd_rn(s, __fadd_rn(e, __fsub_rn(al, bl)));
}

// Values of the CTA sums: species, cloud top, d/dcz, d/dR_p, temperature nodes.
constexpr int kItemRed = TR_MAX_SPECIES + 1 + 2 + TR_MAX_TNODES;

// Dynamic shared memory of k_adjoint_item for a maximum layer count: FP64 per-layer arrays, the
// CTA sums' terms, the altitudes and radii, the G_DL matrix (pitch npad + 1: its rows and columns
// are both read without bank conflicts) and the features.
struct ItemSmem {
  int NM, npad, n_feat, n_val;
  __host__ __device__ ItemSmem(int nm, int nf, int nv) : NM(nm), npad(pad8(nm)), n_feat(nf), n_val(nv) {}
  __host__ __device__ size_t bytes() const {
    return sizeof(double) * (5 * (size_t)NM + 1 + (size_t)n_val * kItemHalf) +
           sizeof(float2) * ((size_t)NM + 1) +
           sizeof(float) * ((size_t)NM + 1 + (size_t)npad * (npad + 1) + (size_t)NM * n_feat) +
           sizeof(int) * (size_t)NM + 16;
  }
};

// One CTA per (atmosphere, row).  GB300 runs FP64 at a small fraction of its FP32 rate and with
// long latency (the SM completes one FP64 warp instruction per 19 cycles, a dependent one takes
// about 140), so the kernel is bound by its FP64 instructions in large batches and by their
// chains in small ones.  Four warps take the layers' terms in FP64 while the other four take the
// O(N^2) path-length sensitivities, FP32 terms (from double-float altitudes, as the forward path
// lengths) added to FP64 accuracy without an FP64 instruction (sum3.h); the backward hydrostatic
// recursion is a scan of its linear steps, and a warp adds each of the CTA's sums.  The G_DL
// matrix and the features are staged in shared memory by coalesced reads (gathered from L2 by one
// thread per radius they held the kernel at 112 us whatever the batch).  100 layers, 5 absorbers:
// 8 atmospheres 114 -> 37 us, 1,024 193 -> 141 us, 50 rows of 128 atmospheres 5.58 -> 0.72 ms (of
// which the third part of the sums, without which they keep 48 bits, 0, 3 and 19 us).
__global__ void __launch_bounds__(kItemThreads)
k_adjoint_item(ItemParams ip) {
  extern __shared__ double dsm[];
  __shared__ double s_X[TR_MAX_SPECIES], s_sum[kItemRed];
  __shared__ double s_c[4];                            // cz, delta, mu, sum G_D
  const GeomParams& gp = ip.gp;
  const int b = blockIdx.x, t = threadIdx.x, warp = t >> 5, lane = t & 31;
  const int row = blockIdx.y, slot = ip.rows.n_rows > 0 ? ip.rows.slot0[row] : 0;
  const int nth = ip.n_theta;
  double* grad = ip.grad + (size_t)b * ip.item_stride + (size_t)row * nth;
  const ItemGeom ig = ip.buf.items[b];
  if (ig.status != TR_OK || ig.n_layers == 0) {
    for (int k = t; k < nth; k += kItemThreads) grad[k] = 0.0;
    return;
  }
  const int N = ig.n_layers, NM = gp.max_layers, npad = ip.buf.npad, pitch = npad + 1;
  const double* th = ip.theta + (size_t)b * nth;
  const double* z = ip.buf.z + (size_t)b * (NM + 1);
  const double* T = ip.buf.tl + (size_t)b * NM;
  const LayerDesc* LD = ip.buf.layers + (size_t)b * NM;
  const int nm = gp.n_mol, nq = gp.n_cia, ns = gp.n_species, ntn = gp.n_tnodes;
  const int n_val = ns + 3 + ntn;                      // values of the CTA sums in use
  double* Gr = dsm;                 // [N + 1]
  double* GT = Gr + (NM + 1);       // [N]
  double* Ga = GT + NM;             // [N]
  double* fac = Ga + NM;            // [N] dr_{l+1} / dr_l of the recursion
  double* wn = fac + NM;            // [N] weight of node k_l + 1 in T_l
  double* val = wn + NM;            // [n_val][kItemHalf]
  float2* zs = reinterpret_cast<float2*>(val + (size_t)n_val * kItemHalf);   // [N + 1]
  float* rs = reinterpret_cast<float*>(zs + NM + 1);   // [N + 1]
  float* G = rs + NM + 1;                              // [N][pitch] G_DL, zero beyond the diagonal
  float* Fs = G + (size_t)npad * pitch;                // [N][n_feat]
  int* kn = reinterpret_cast<int*>(Fs + (size_t)NM * ip.n_feat);   // [N] node segment of layer l
  const double rp = ig.r_p;
  const double inv_rs2 = gp.inv_rs2;
  const double ln10 = 2.302585092994046;
  const size_t ps = (size_t)b * ip.slots + slot;

  // ---- staging; meanwhile warp 0 takes the chemistry (as the profile kernel computes it) and the
  //      constants of the recursion
  {
    const float* g = ip.part_dl + ps * npad * npad;
    for (int j = warp; j < N; j += kItemThreads / 32)
      for (int l = lane; l < N; l += 32) G[j * pitch + l] = l >= j ? __ldg(g + (size_t)j * npad + l) : 0.f;
    const float* f = ip.part_f + ps * NM * ip.n_feat;
    for (int i = t; i < N * ip.n_feat; i += kItemThreads) Fs[i] = __ldg(f + i);
    const float* pa = ip.part_a + ps * npad;
    for (int j = t; j < N; j += kItemThreads) Ga[j] = (double)__ldg(pa + j);
    for (int k = t; k <= N; k += kItemThreads) {
      const double zk = z[k];
      const float h = (float)zk;
      zs[k] = make_float2(h, (float)(zk - (double)h));
      rs[k] = (float)(rp + zk);
    }
  }
  if (warp == 0) {
    if (lane < nm) s_X[lane] = exp10(th[lane]);
    __syncwarp();
    double sumx = 0.0, mu = 0.0;
    for (int m = 0; m < nm; ++m) { sumx += s_X[m]; mu = fma(s_X[m], gp.mass[m], mu); }
    const double rem = 1.0 - sumx;
    if (lane >= nm && lane < ns) s_X[lane] = gp.fill[lane] * rem;
    if (lane == 0) {
      mu = fma(rem, gp.fill_mass, mu);
      const double delta = (gp.ln_pmax - gp.ln_pmin) / N;
      s_c[0] = (kKB * delta) / (mu * gp.amu_g_mp);
      s_c[1] = delta;
      s_c[2] = mu;
      s_c[3] = (double)__ldg(ip.part_rp + ps);
    }
  }
  __syncthreads();
  const double cz = s_c[0], delta = s_c[1], mu = s_c[2];

  // ---- radii from path lengths and annulus weights
  //      DL[j][l] = 2 (s(l+1,j) - s(l,j)), s(k,j) = sqrt(r_k^2 - r_j^2):
  //      ds(k,j)/dr_k = r_k / s,  ds(k,j)/dr_j = -r_j / s;  r_k^2 - r_j^2 = (z_k - z_j)(r_k + r_j)
  //      with z_k - z_j from the double-float altitudes; each term in FP32, sums to FP64
  const double dln = (gp.ln_pmin - gp.ln_pmax) / N;
  const int f_dS = nm, f_R = 2 * nm, f_C = 2 * nm + ns, f_dC = f_C + nq, f_K = f_dC + nq;
  double acc[TR_MAX_SPECIES + 3];                   // species, cloud top, d/dcz, d/dR_p
#pragma unroll
  for (int i = 0; i < TR_MAX_SPECIES + 3; ++i) acc[i] = 0.0;
  if (t >= kItemHalf) {
    for (int k = t - kItemHalf; k <= N; k += kItemHalf) {
      const float2 zk = zs[k];
      const float rk = rs[k];
      // two terms at a time; no guards in the loops, so that they unroll (with a guard on the second
      // term 40 us for 8 atmospheres instead of 38, 50 rows of 128 atmospheres 0.75 ms instead of 0.72)
      const double paths = sum_fp32_terms([&](auto add) {
        auto outer = [&](int j) {                   // k as the outer radius of s(k, j), j < k
          const float gs = 2.f * (G[j * pitch + k - 1] - (k < N ? G[j * pitch + k] : 0.f));
          const float2 zj = zs[j];
          const float s2 = diff_df(zk.x, zk.y, zj.x, zj.y) * (rk + rs[j]);
          return gs != 0.f ? gs * rk * rsqrtf(s2) : 0.f;
        };
        int j = 0;
#pragma unroll 4
        for (; j + 1 < k; j += 2) add(outer(j), outer(j + 1));
        if (j < k) add(outer(j), 0.f);
        auto ray = [&](int u, float dg) {           // k as the ray of s(u, k), u > k
          const float gs = 2.f * dg;
          const float2 zu = zs[u];
          const float s2 = diff_df(zu.x, zu.y, zk.x, zk.y) * (rs[u] + rk);
          return gs != 0.f ? -(gs * rk * rsqrtf(s2)) : 0.f;
        };
        float g0 = k < N ? G[k * pitch + k] : 0.f;  // G[k][u - 1]
        int u = k + 1;
#pragma unroll 4
        for (; u < N; u += 2) {
          const float g1 = G[k * pitch + u], g2 = u + 1 < N ? G[k * pitch + u + 1] : 0.f;
          add(ray(u, g0 - g1), ray(u + 1, g1 - g2));
          g0 = g2;
        }
        if (u == N) add(ray(u, g0), 0.f);
      });
      // a_j = (r_{j+1}^2 - r_j^2) / R_s^2
      const double ga = ((k >= 1 ? Ga[k - 1] : 0.0) - (k < N ? Ga[k] : 0.0));
      Gr[k] = fma(ga * 2.0 * (rp + z[k]), inv_rs2, paths);
    }
  } else {
    // ---- per layer: opacity weights, densities, cloud; recursion factors; T-node weights
    for (int l = t; l < N; l += kItemHalf) {
      const LayerDesc& d = LD[l];
      const float* F = Fs + l * ip.n_feat;
      const double lnp0 = fma((double)l, dln, gp.ln_pmax), lnp1 = fma((double)(l + 1), dln, gp.ln_pmax);
      const double lnp = 0.5 * (lnp0 + lnp1);
      const double Tl = T[l], inv_t = 1.0 / Tl;
      const double rho = (exp(lnp) * gp.inv_kb) * inv_t;
      double gT = 0.0, grho = 0.0;
      if (!(d.flags & kLayerMolZero)) {
        double gt = 0.0;
#pragma unroll
        for (int m = 0; m < TR_MAX_MOL; ++m)
          if (m < nm) {
            const double f = F[m], x = s_X[m];
            grho = fma(f, x, grho);
            acc[m] = fma(f, rho, acc[m]);
            gt = fma(x, (double)F[f_dS + m], gt);
          }
        gT = rho * gt;
      }
      if (gp.has_ray) {
#pragma unroll
        for (int s = 0; s < TR_MAX_SPECIES; ++s)
          if (s < ns && F[f_R + s] != 0.f) {         // species without Rayleigh: exact zeros
            const double R = F[f_R + s] * gp.ray_scale[s];
            grho = fma(R, s_X[s], grho);
            acc[s] = fma(R, rho, acc[s]);
          }
      }
      if (nq > 0 && !(d.flags & kLayerCiaZero)) {
        for (int q = 0; q < nq; ++q) {
          const double C = F[f_C + q] * gp.cia_scale[q], dC = F[f_dC + q] * gp.cia_scale[q];
          const double xa = s_X[gp.cia_a[q]], xb = s_X[gp.cia_b[q]];
          const double xx = rho * xa * xb, cr = C * rho * rho;
          gT = fma(rho * xx, dC, gT);
          grho = fma(C * 2.0, xx, grho);
#pragma unroll
          for (int s = 0; s < TR_MAX_SPECIES; ++s) {   // no indexed access to the sums
            if (s == gp.cia_a[q]) acc[s] = fma(cr, xb, acc[s]);
            if (s == gp.cia_b[q]) acc[s] = fma(cr, xa, acc[s]);
          }
        }
      }
      GT[l] = fma(-grho * rho, inv_t, gT);
      if (gp.cloud_mode == TR_CLOUD_FRACTIONAL) {
        // c_l = clamp((min(ln p_l, ln P_bot) - max(ln P_top, ln p_{l+1})) / Delta, 0, 1)
        const double ln_top = th[nm + ntn + 1] * ln10;
        const double hi = fmin(lnp0, gp.ln_cbot);
        const double cf = hi - fmax(ln_top, lnp1);
        if (cf > 0.0 && cf < delta && ln_top > lnp1)
          acc[TR_MAX_SPECIES] += gp.kappa_cloud * F[f_K] * (-ln10 / delta);
      }
      // dr_{l+1}/dr_l: 1 + 2 cz T_l r_l (altitude-dependent gravity), 1 (constant)
      fac[l] = gp.gravity_mode == TR_GRAV_CONST ? 1.0 : fma(2.0 * cz * Tl, rp + z[l], 1.0);
      // temperature nodes: T_l linear in log10 P between nodes, clamped beyond them
      int kseg = 0;
      double f = 0.0;
      if (ntn > 1) {
        const double x = lnp * 0.43429448190325182765;
        if (x >= gp.tnode_log10p[0]) { kseg = 0; f = 0.0; }
        else if (x <= gp.tnode_log10p[ntn - 1]) { kseg = ntn - 2; f = 1.0; }
        else {
          while (!(gp.tnode_log10p[kseg] >= x && x >= gp.tnode_log10p[kseg + 1])) ++kseg;
          f = (x - gp.tnode_log10p[kseg]) * gp.inv_dlog10p[kseg];
        }
      }
      kn[l] = kseg;
      wn[l] = f;
    }
  }
  __syncthreads();

  // ---- hydrostatic recursion, backwards (r_{l+1} = r_l + cz T_l r_l^2): G_r of r_l is g_l = g_{l+1}
  //      fac_l + Gr_l from g_N = Gr_N, a scan of linear maps g -> a g + c over the layers from the
  //      top: each lane of warp 0 composes its run of layers, the lanes' maps are scanned, and the
  //      run is replayed from the lane's entry value
  if (warp == 0) {
    const int per = (N + 31) / 32;
    const int top = N - lane * per, bot = max(0, top - per);   // layers top - 1 .. bot
    double a = 1.0, c = 0.0;
    for (int l = top - 1; l >= bot; --l) {
      a *= fac[l];
      c = fma(c, fac[l], Gr[l]);
    }
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {              // maps of lanes 0 .. lane, in that order
      const double pa = __shfl_up_sync(0xffffffffu, a, o), pc = __shfl_up_sync(0xffffffffu, c, o);
      if (lane >= o) { c = fma(pc, a, c); a *= pa; }
    }
    const double gN = Gr[N];
    double g = fma(gN, a, c);                       // g at this lane's lowest radius
    g = __shfl_up_sync(0xffffffffu, g, 1);
    if (lane == 0) g = gN;
    for (int l = top - 1; l >= bot; --l) {
      g = fma(g, fac[l], Gr[l]);
      Gr[l] = g;
    }
  }
  __syncthreads();
  // per layer, with G_r of r_{l+1}: dT_l and dcz (and, for constant gravity, dR_p) terms;
  // then the CTA sums of the mixing-ratio, cloud, cz, R_p and node terms
  if (t < kItemHalf) {
    double gnode[TR_MAX_TNODES];
#pragma unroll
    for (int k = 0; k < TR_MAX_TNODES; ++k) gnode[k] = 0.0;
    for (int l = t; l < N; l += kItemHalf) {
      const double g1 = Gr[l + 1];
      const double rl = gp.gravity_mode == TR_GRAV_CONST ? rp : rp + z[l];
      const double gr2 = g1 * rl * rl, Tl = T[l];
      const double gT = fma(gr2, cz, GT[l]);
      acc[TR_MAX_SPECIES + 1] = fma(gr2, Tl, acc[TR_MAX_SPECIES + 1]);   // d/dcz
      if (gp.gravity_mode == TR_GRAV_CONST)
        acc[TR_MAX_SPECIES + 2] += g1 * 2.0 * cz * Tl * rp;            // d/dR_p, direct
      if (ntn == 1) {
        gnode[0] += gT;
      } else {
        const double hi = gT * wn[l], lo = gT - hi;
        const int k0 = kn[l];
#pragma unroll
        for (int k = 0; k < TR_MAX_TNODES; ++k) {
          if (k == k0) gnode[k] += lo;
          if (k == k0 + 1) gnode[k] += hi;
        }
      }
    }
#pragma unroll
    for (int s = 0; s < TR_MAX_SPECIES; ++s) if (s < ns) val[s * kItemHalf + t] = acc[s];
#pragma unroll
    for (int k = 0; k < 3; ++k) val[(ns + k) * kItemHalf + t] = acc[TR_MAX_SPECIES + k];
#pragma unroll
    for (int k = 0; k < TR_MAX_TNODES; ++k) if (k < ntn) val[(ns + 3 + k) * kItemHalf + t] = gnode[k];
  }
  __syncthreads();
  for (int v = warp; v < n_val; v += kItemThreads / 32) {
    double s = 0.0;
#pragma unroll
    for (int k = 0; k < kItemHalf / 32; ++k) s += val[v * kItemHalf + 32 * k + lane];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) s_sum[v] = s;
  }
  __syncthreads();
  if (warp == 0) {
    const double glp_sum = s_sum[ns], gcz = s_sum[ns + 1], grp_dir = s_sum[ns + 2];
    const double gmu = gcz * (-cz / mu);
    // chemistry: X_m = 10^theta_m, fill gases f (1 - sum X), mu = sum X_s m_s
    double sum_fill = 0.0;
    for (int f = nm; f < ns; ++f) sum_fill += gp.fill[f] * (s_sum[f] + gmu * gp.mass[f]);
    if (lane < nm) grad[lane] = (s_sum[lane] + gmu * gp.mass[lane] - sum_fill) * s_X[lane] * ln10;
    if (lane < ntn) grad[nm + lane] = s_sum[ns + 3 + lane];
    if (lane == 0) {
      const double g_rp = Gr[0] + grp_dir + s_c[3] * 2.0 * rp * inv_rs2;
      grad[nm + ntn] = g_rp * kRJup;
      grad[nm + ntn + 1] = glp_sum;
    }
  }
}

}  // namespace

size_t adjoint_extra_bytes(const tr_tables* t, const tr_batch_desc* d, const tr_bins* bins, int B) {
  if (!t || !d || !bins) return 0;
  const int n_in = bins->dev.i1 - bins->dev.i0;
  const int tiles = (bins->dev.i1 - wn_first(bins->dev.i0) + kAT - 1) / kAT;
  const int npad = pad8(d->max_layers);
  const int n_feat = 2 * t->n_mol + t->n_species + 2 * t->n_cia + 1;
  auto al = [](size_t x) { return (x + 255) / 256 * 256; };
  size_t s = 0;
  s += al(sizeof(float) * (size_t)B * n_in);                               // gd
  s += al(sizeof(float) * (size_t)B * tiles * npad);                       // part_a
  s += al(sizeof(float) * (size_t)B * tiles * npad * npad);                // part_dl
  s += al(sizeof(float) * (size_t)B * tiles * d->max_layers * n_feat);     // part_f
  s += al(sizeof(float) * (size_t)B * tiles);                              // part_rp
  s += al(sizeof(double) * (size_t)B * bins->dev.n_bin);                   // binned scratch
  return s;
}

}  // namespace tr

using namespace tr;

extern "C" int tr_adjoint_transit(tr_ctx* ctx, const tr_tables* t, const tr_batch_desc* d, int B,
                                  const double* d_theta, const int32_t* d_nlayers,
                                  const tr_bins* bins, const double* d_obs,
                                  const double* d_sigma_obs, const double* d_gbin,
                                  double* d_chi2, double* d_grad, double* d_jac, double* d_binned,
                                  int32_t* d_status, int precision, int recompute_k, void* ws,
                                  size_t ws_bytes, void* stream) {
  if (!ctx || !t || !d || !bins || !d_theta || B < 0)
    return set_error(ctx, TR_ERR_ARG, "null argument");
  if (!d_grad && !d_jac) return set_error(ctx, TR_ERR_ARG, "neither d_grad nor d_jac given");
  if (B > TR_MAX_BATCH) return set_error(ctx, TR_ERR_ARG, "batch larger than TR_MAX_BATCH");
  const bool chi2_mode = d_grad && !d_gbin;
  if (chi2_mode && (!d_obs || !d_sigma_obs || !d_chi2))
    return set_error(ctx, TR_ERR_ARG, "chi^2 mode needs obs, sigma_obs and chi2");
  if (precision != TR_PREC_FP32 && precision != TR_PREC_MIXED)
    return set_error(ctx, TR_ERR_ARG, "unknown precision");
  const bool mixed = precision == TR_PREC_MIXED;
  if (!mixed && !t->d_sigma && t->n_mol > 0)
    return set_error(ctx, TR_ERR_UNSUPPORTED, "tables were loaded without FP32 storage");
  if (mixed && !t->d_logsig16 && t->n_mol > 0)
    return set_error(ctx, TR_ERR_UNSUPPORTED, "tables were loaded without FP16 log10 storage");
  if (bins->dev.n_bin > kMaxRows) return set_error(ctx, TR_ERR_ARG, "the adjoint supports at most 256 bins");
  if (t->interp_mode != TR_INTERP_LINEAR)
    return set_error(ctx, TR_ERR_UNSUPPORTED, "the adjoint implements the linear temperature scheme");
  if (d->t_profile != TR_TPROF_NPOINT || d->gas_mode != TR_GAS_CONSTANT)
    return set_error(ctx, TR_ERR_UNSUPPORTED,
                     "the adjoint implements the N-point temperature profile and constant "
                     "mixing ratios");
  if (B == 0) return TR_OK;
  cudaSetDevice(ctx->device);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const int n_in = bins->dev.i1 - bins->dev.i0;
  const size_t fwd = forward_workspace_bytes(B, d->max_layers, n_in);
  auto al256 = [](size_t x) { return (x + 255) / 256 * 256; };
  // [forward item buffers + depths][K buffer][path-length tiles][adjoint buffers]
  const size_t kb = al256(forward_kbuf_bytes(B, d->max_layers, bins->dev.i0, n_in));
  const size_t db = al256(dl_tile_bytes(B, d->max_layers, precision));
  const size_t need = fwd + kb + db + adjoint_extra_bytes(t, d, bins, B);
  ItemBuffers buf; double* depth = nullptr; char* extra = nullptr;
  // the altitudes and path lengths on a second branch beside the first opacity kernel
  Fork fk;
  Fork* fork = fork_ready(ctx, &fk, s) ? &fk : nullptr;
  int rc = prepare_batch(ctx, t, d, n_in, need, B, d_theta, d_nlayers, d_status, ws, ws_bytes,
                         s, &buf, &depth, &extra, fork);
  if (rc != TR_OK) return rc;
  float* kbuf = reinterpret_cast<float*>(extra);
  void* dl16 = db > 0 ? extra + kb : nullptr;
  extra += kb + db;
  // The batch in runs of as many items as the K buffer holds (equal runs): the forward, in the
  // two-stage form (the configuration tuned for this shape's forward, if any), leaves their K in
  // kbuf and the backward passes read it.  recompute_k == 1: the whole batch at once, K formed
  // again from the tables by the tile kernel.  (Recomputing K where the batch outgrows the
  // buffer, which this replaces, cost 65 us a tile against 50: 320 atmospheres of 18,905
  // wavenumbers and 100 layers took 23.2 ms, in two runs 18.2.)  The binned spectrum is needed
  // only for chi^2 or when asked for: otherwise (vector-Jacobian products, Jacobian) only the
  // opacity stage runs, and not even that when the backward recomputes K.
  const bool use_kstore = recompute_k != 1;
  const bool need_binned = chi2_mode || d_binned;
  const int fit = use_kstore ? forward_chunk_items(B, d->max_layers, bins->dev.i0, n_in) : B;
  const int n_runs = (B + fit - 1) / fit, run = (B + n_runs - 1) / n_runs;
  const auto it = ctx->tuned.find(batch_shape_key(t, d, B, bins, false, precision));
  ForwardChoice fc = it != ctx->tuned.end() ? it->second : ForwardChoice{kFormTwoStage, 0, 0, 0};
  fc.form = kFormTwoStage;
  const int tiles = (bins->dev.i1 - wn_first(bins->dev.i0) + kAT - 1) / kAT;
  const int npad = pad8(d->max_layers);
  const int n_feat = 2 * t->n_mol + t->n_species + 2 * t->n_cia + 1;
  const int nth = t->n_mol + d->n_tnodes + 2;
  auto al = [](size_t x) { return (x + 255) / 256 * 256; };
  char* e = extra;
  float* gd = reinterpret_cast<float*>(e); e += al(sizeof(float) * (size_t)B * n_in);
  float* part_a = reinterpret_cast<float*>(e); e += al(sizeof(float) * (size_t)B * tiles * npad);
  float* part_dl = reinterpret_cast<float*>(e); e += al(sizeof(float) * (size_t)B * tiles * npad * npad);
  float* part_f = reinterpret_cast<float*>(e); e += al(sizeof(float) * (size_t)B * tiles * d->max_layers * n_feat);
  float* part_rp = reinterpret_cast<float*>(e); e += al(sizeof(float) * (size_t)B * tiles);
  double* binned = d_binned ? d_binned : reinterpret_cast<double*>(e);
  cudaError_t err = cudaSuccess;
  AdjParams ap{};
  ap.f.sigma = t->d_sigma; ap.f.n_mol = t->n_mol; ap.f.n_p = t->n_p; ap.f.n_t = t->n_t;
  ap.f.wn_pad = t->wn_pad; ap.f.cia = t->d_cia; ap.f.n_cia = t->n_cia; ap.f.n_t_cia = t->n_t_cia;
  ap.f.ray = t->has_ray ? t->d_ray : nullptr; ap.f.n_species = t->n_species;
  ap.f.max_layers = d->max_layers; ap.f.wn_begin = bins->dev.i0;
  ap.f.wn_count = n_in; ap.f.dev_err = ctx->dev_err;
  if (mixed) {
    ap.f.logsig16 = t->d_logsig16;
    for (int m = 0; m < t->n_mol; ++m) ap.f.logsig_off[m] = t->logsig_offset[m];
  }
  ap.inv_dt = t->d_inv_dt; ap.inv_dtc = t->d_inv_dtc; ap.gd = gd; ap.n_in = n_in;
  ap.n_feat = n_feat;
  ap.kstore = use_kstore ? kbuf : nullptr;
  ap.kcols = forward_kcols(bins->dev.i0, n_in);
  ap.t_ptr = bins->dev.t_ptr; ap.t_bin = bins->dev.t_bin; ap.t_w = bins->dev.t_w;
  ap.ray_mask = t->has_ray ? t->ray_mask : 0u;
  const int n_ray = __builtin_popcount(ap.ray_mask), n_act = n_feat - (t->n_species - n_ray);
  const size_t smem = sizeof(float) * AdjSmem(d->max_layers, n_act, n_ray).floats();
  // three CTAs per SM (80 registers a thread) where their shared memory fits: 1.62 ms against 1.81
  // (k_adjoint_tile)
  const bool three = smem <= kThreeCtaSmem;
  void (*kern)(AdjParams) =
      use_kstore ? (mixed ? (three ? k_adjoint_tile<true, false, 3> : k_adjoint_tile<true, false, 2>)
                          : (three ? k_adjoint_tile<false, false, 3> : k_adjoint_tile<false, false, 2>))
                 : (mixed ? k_adjoint_tile<true, true, 2> : k_adjoint_tile<false, true, 2>);
  err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (err != cudaSuccess) return set_error(ctx, TR_ERR_CUDA, std::string("adjoint tile kernel: ") + cudaGetErrorString(err));
  int dev = 0, n_sm = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
  ItemParams itp{};
  itp.gp = batch_geom_params(t, d); itp.n_theta = nth;
  itp.part_a = part_a; itp.part_dl = part_dl; itp.part_f = part_f; itp.part_rp = part_rp;
  itp.n_feat = n_feat;
  const size_t smem_i = ItemSmem(d->max_layers, n_feat, t->n_species + 3 + d->n_tnodes).bytes();
  err = cudaFuncSetAttribute(k_adjoint_item, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_i);
  if (err != cudaSuccess) return set_error(ctx, TR_ERR_CUDA, std::string("adjoint item kernel: ") + cudaGetErrorString(err));

  // One backward pass over `slots` wavenumber tiles per item: the tile kernel's partial sums,
  // their GPU-wide sum into each row's first slot, and the per-atmosphere kernel writing item b's
  // row r at grad + b * stride + r * nth.  No rows: one gradient with dL/dD from gd.
  auto backward = [&](int bc, const RowGroup& rows, int slots, double* grad,
                      long long stride) -> int {
    const int n_rows = std::max(rows.n_rows, 1);
    ap.rows = rows; ap.tiles = slots;
    {
      KernelTimer kt(ctx, "k_adjoint_tile", s);
      // a range of more than 4 million wavenumbers has more tiles than the grid's second dimension
      constexpr int kMaxY = 65535;
      for (int s0 = 0; s0 < slots && err == cudaSuccess; s0 += kMaxY) {
        ap.first_slot = s0;
        ap.part_a = part_a + (size_t)s0 * npad;
        ap.part_dl = part_dl + (size_t)s0 * npad * npad;
        ap.part_f = part_f + (size_t)s0 * d->max_layers * n_feat;
        ap.part_rp = part_rp + s0;
        kern<<<dim3(bc, std::min(slots - s0, kMaxY)), kAThreads, smem, s>>>(ap);
        err = cudaGetLastError();
      }
    }
    if (err != cudaSuccess) return set_error(ctx, TR_ERR_CUDA, std::string("adjoint tile kernel: ") + cudaGetErrorString(err));
    if (slots > n_rows) {
      // the tiles' partial sums into the rows' first slots by a GPU-wide pass, so the
      // per-atmosphere kernel reads one set of sums
      KernelTimer kt(ctx, "k_adjoint_sum", s);
      const int n_f = d->max_layers * n_feat, units = sum_units(npad, n_f);
      if ((long long)bc * n_rows * units >= kSum4Threads) {
        TileSum4Args ts{};
        ts.dl = part_dl; ts.a = part_a; ts.f = part_f; ts.rp = part_rp;
        ts.npad = npad; ts.n_f = n_f; ts.slots = slots; ts.rows = rows;
        k_adjoint_sum4<<<dim3((units + kSumThreads - 1) / kSumThreads, bc, n_rows), kSumThreads, 0, s>>>(ts);
      } else {
        TileSumArgs ts{};
        ts.arr[0] = part_a;  ts.m[0] = npad;
        ts.arr[1] = part_dl; ts.m[1] = (long long)npad * npad; ts.tri[1] = npad;
        ts.arr[2] = part_f;  ts.m[2] = (long long)d->max_layers * n_feat;
        ts.arr[3] = part_rp; ts.m[3] = 1;
        ts.slots = slots; ts.rows = rows;
        const long long most = (long long)bc * npad * npad;
        const int gx = (int)std::max<long long>(1, std::min<long long>((most + 255) / 256, 8LL * n_sm));
        k_adjoint_sum<<<dim3(gx, 4, n_rows), 256, 0, s>>>(ts, bc);
      }
      err = cudaGetLastError();
      if (err != cudaSuccess) return set_error(ctx, TR_ERR_CUDA, std::string("adjoint sum kernel: ") + cudaGetErrorString(err));
    }
    itp.rows = rows; itp.slots = slots; itp.grad = grad; itp.item_stride = stride;
    {
      KernelTimer kt(ctx, "k_adjoint_item", s);
      k_adjoint_item<<<dim3(bc, n_rows), kItemThreads, smem_i, s>>>(itp);
      err = cudaGetLastError();
    }
    if (err != cudaSuccess) return set_error(ctx, TR_ERR_CUDA, std::string("adjoint item kernel: ") + cudaGetErrorString(err));
    return TR_OK;
  };
  for (int b0 = 0; b0 < B; b0 += run) {
    const int bc = std::min(run, B - b0);
    const ItemBuffers rb = items_from(buf, b0, d->max_layers);
    double* out = depth + (size_t)b0 * n_in;
    double* bin_out = binned + (size_t)b0 * bins->dev.n_bin;
    if (need_binned || use_kstore) {
      rc = run_forward(ctx, t, d->max_layers, rb, bc, bins->dev.i0, n_in, out, n_in, precision, s,
                       kbuf, dl16, &fc, /*opacity_only=*/!need_binned, fork);
      join_fork(ctx, fork, s);
      if (rc != TR_OK) return rc;
    } else {
      err = fork_start(ctx, fork, s, false);
      if (err != cudaSuccess) return set_error(ctx, TR_ERR_CUDA, cudaGetErrorString(err));
    }
    if (need_binned) {
      KernelTimer kt(ctx, "k_bin", s);
      err = launch_bin(bins->dev, bc, out, n_in, bins->dev.i0, bin_out, s);
    }
    if (err == cudaSuccess && d_grad) {
      KernelTimer kt(ctx, "k_gd", s);
      k_gd<<<dim3(bc, (n_in + kGdRun - 1) / kGdRun), kGdThreads, 0, s>>>(
          bins->dev, bc, bin_out, d_obs, d_sigma_obs,
          d_gbin ? d_gbin + (size_t)b0 * bins->dev.n_bin : nullptr, rb.items,
          (d_gbin || !d_chi2) ? nullptr : d_chi2 + b0, gd, n_in);
      err = cudaGetLastError();
    }
    if (err != cudaSuccess) return set_error(ctx, TR_ERR_CUDA, cudaGetErrorString(err));
    ap.f.buf = rb; itp.buf = rb; itp.theta = d_theta + (size_t)b0 * nth;
    if (d_grad) {
      RowGroup one;
      one.n_rows = 0; one.first_bin = 0;
      rc = backward(bc, one, tiles, d_grad + (size_t)b0 * nth, nth);
      if (rc != TR_OK) return rc;
    }
    if (!d_jac) continue;
    double* jac = d_jac + (size_t)b0 * bins->dev.n_bin * nth;
    // row k of dD_bin/dtheta: dL/dD is bin k's normalised weights, which vanish outside the
    // bin's native range, so a row covers only the tiles of that range.  The rows go in groups
    // of as many as the partial sums' space for one gradient (`tiles` slots per item) holds, one
    // launch of each kernel per group: a launch per row left the GPU with one row's CTAs (128
    // atmospheres, 50 bins of about 19 wavenumbers: 7.86 ms a call, in groups 2.3 ms).  Rows are
    // described by their first tiles, so that a group can hold bins of any width (two atmospheres,
    // four bins of about 19,000 wavenumbers: 0.71 ms a call with a launch per row, 0.33 in groups).
    const int base = wn_first(bins->dev.i0);
    const int n_bin = bins->dev.n_bin;
    auto first_tile = [&](int k) { return (bins->bin_lo[k] - base) / kAT; };
    auto n_tiles = [&](int k) { return (bins->bin_hi[k] - 1 - base) / kAT + 1 - first_tile(k); };
    for (int k = 0; k < n_bin;) {
      RowGroup g;
      g.n_rows = 0; g.first_bin = k; g.slot0[0] = 0;
      // at least one row: no bin has more tiles than the range
      for (; k < n_bin && g.slot0[g.n_rows] + n_tiles(k) <= tiles; ++k, ++g.n_rows) {
        g.tile0[g.n_rows] = first_tile(k);
        g.slot0[g.n_rows + 1] = g.slot0[g.n_rows] + n_tiles(k);
      }
      rc = backward(bc, g, g.slot0[g.n_rows], jac + (size_t)g.first_bin * nth, (long long)n_bin * nth);
      if (rc != TR_OK) return rc;
    }
  }
  return TR_OK;
}
