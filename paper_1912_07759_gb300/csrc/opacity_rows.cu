// opacity_rows.cu -- opacity K[layer, wn] of the two-stage form with the linear temperature
// scheme (Sec. 5, Sec. 8.1), both table precisions.
//
// A warp takes one unit (item, layer block, 256 consecutive wavenumbers; eight per lane) and
// walks the layers upwards.  The CTA first turns the layers' brackets into a list of row
// operations (shared memory): an operation brings two table rows of every molecule and at most
// one CIA row, and says which of the four corner sums
//   us[c] = sum_m (x_m / x_max) sigma_m,c,   c = (P_i,T_j) (P_i,T_j+1) (P_i+1,T_j) (P_i+1,T_j+1)
// they replace and which old sums move: when the layers go from one (P, T) cell to a
// neighbouring one, two of the four sums are those of the old cell, so a step across a cell
// edge loads two rows, and a diagonal step or a jump takes two operations.  The rows come by
// TMA boxes (two T rows at one P, or two P rows at one T, of all molecules) into a ring of
// stages of the warp's own: a column is used by one lane only, so no other warp is involved; the
// warp waits for an operation's rows, forms the sums, refills the stage and writes the layers up
// to the next operation:
//   K = kappa_cloud + rho sigma_R + sum_c (rho x_max w_c) us[c] + sum_T (rho^2 y_max w_T) uc[T].
//
// What bounds it: the bytes from L2 into the SMs.  The ring kernel it replaced loaded all four rows
// of a cell for every run of layers (36 runs an atmosphere at 22 x 27 tables, 24 rows each with two
// CIA pairs); row operations need 40 of 12 rows.  Measured, 100 layers x 200,000 wavenumbers, 5
// absorbers: one atmosphere 73 -> 66 us (293 MB of method bytes: 4.4 TB/s), 64 atmospheres 4.17 ->
// 1.83 ms (13 TB/s from L2 and 2.8 TB/s of K written), FP16 tables 32 atmospheres 2.55 -> 1.25 ms
// (half the bytes; the 2^x decode and its conversions share the bound); 4,096 atmospheres of
// 50-150 layers over 945 wavenumbers with 2 absorbers 0.92 -> 0.51 ms.  Rows loaded straight into
// registers (no shared memory) took 2.08 ms for the 64 atmospheres.  Operands of the packed FMAs
// are kept twice in shared memory: duplicating them in registers cost two moves each.
#include <algorithm>
#include "opacity.h"

namespace tr {
namespace {

constexpr int kRowWarps = 2;                        // warps (neighbouring tiles) per CTA
constexpr int kRowCtas = 6;                         // CTAs per SM the registers are held to
constexpr int kRowMaxStages = 8;
constexpr int kRowTW = kRowTile;                    // wavenumbers per warp
static_assert(kRowTW % 128 == 0, "lanes take groups of four wavenumbers, 128 apart");

// One row operation: x = the first row's P index | T index << 16, y = layer it precedes | kind <<
// 8 | CIA kind << 11 | new zone << 14 | CIA row << 16 | zone << 26.
enum { kOpNone = 0, kOpPDown, kOpTUp, kOpTDown, kOpSet01, kOpSet23 };
enum { kCiaNone = 0, kCiaUp, kCiaDown, kCiaSet0, kCiaSet1 };
__device__ __forceinline__ unsigned op_y(int l, int kind, int ck, int newz, int crow, int zone) {
  return (unsigned)(l | (kind << 8) | (ck << 11) | (newz << 14) | (crow << 16)) |
         ((unsigned)zone << 26);
}

// The operations of layers [l_begin, l_end) of item b, in layer order, into ops[] (at most two
// per layer, then one that carries l_end); returns their number without the last.
__device__ int build_ops(const FwdParams& p, int b, int l_begin, int l_end, int lane, uint2* ops) {
  const bool has_mol = p.n_mol > 0, has_cia = p.n_cia > 0, zoned = p.buf.zoned != 0;
  const LayerDesc* L = p.buf.layers + (size_t)b * p.max_layers;
  int n = 0;
  int4 carry = make_int4(0, 0, 0, 0);
  for (int l0 = l_begin; l0 < l_end; l0 += 32) {
    const int li = l0 + lane;
    const bool valid = li < l_end;
    const int4 h = valid ? __ldg(reinterpret_cast<const int4*>(L + li)) : make_int4(0, 0, 0, 0);
    int4 q;                                         // the layer below
    q.x = __shfl_up_sync(0xffffffffu, h.x, 1);
    q.y = __shfl_up_sync(0xffffffffu, h.y, 1);
    q.z = __shfl_up_sync(0xffffffffu, h.z, 1);
    q.w = __shfl_up_sync(0xffffffffu, h.w, 1);
    if (lane == 0) q = carry;
    carry.x = __shfl_sync(0xffffffffu, h.x, 31);
    carry.y = __shfl_sync(0xffffffffu, h.y, 31);
    carry.z = __shfl_sync(0xffffffffu, h.z, 31);
    carry.w = __shfl_sync(0xffffffffu, h.w, 31);
    const bool first = li == l_begin;
    const bool newz = zoned && (first || h.w != q.w);
    const bool all = first || newz;                 // every sum is formed anew
    const int dp = h.x - q.x, dt = h.y - q.y, dc = h.z - q.z;
    int k0 = kOpNone, k1 = kOpNone;                 // kinds and first rows of the operations
    int ip0 = h.x, it0 = h.y, ip1 = h.x, it1 = h.y;
    if (has_mol && (all || dp != 0 || dt != 0)) {
      if (all || dp > 0 || dp < -1 || dt > 1 || dt < -1) {
        k0 = kOpSet01; k1 = kOpSet23; ip1 = h.x + 1;
      } else {
        const int kt = dt > 0 ? kOpTUp : kOpTDown, tt = dt > 0 ? h.y + 1 : h.y;
        if (dp == 0) { k0 = kt; it0 = tt; }
        else {                                      // the P step at the old T bracket first
          k0 = kOpPDown; it0 = q.y;
          if (dt != 0) { k1 = kt; it1 = tt; }
        }
      }
    }
    int c0 = kCiaNone, c1 = kCiaNone, row0 = 0;
    const int row1 = h.z + 1;
    if (has_cia && (all || dc != 0)) {
      if (!all && dc == 1) { c0 = kCiaUp; row0 = h.z + 1; }
      else if (!all && dc == -1) { c0 = kCiaDown; row0 = h.z; }
      else { c0 = kCiaSet0; c1 = kCiaSet1; row0 = h.z; }
    }
    const bool two = k1 != kOpNone || c1 != kCiaNone;
    const bool any = valid && (all || k0 != kOpNone || c0 != kCiaNone);
    const int mine = any ? (two ? 2 : 1) : 0;
    const unsigned m1 = __ballot_sync(0xffffffffu, mine >= 1);
    const unsigned m2 = __ballot_sync(0xffffffffu, mine == 2);
    const unsigned below = (1u << lane) - 1u;
    const int at = n + __popc(m1 & below) + __popc(m2 & below);
    if (mine >= 1)
      ops[at] = make_uint2((unsigned)(ip0 | (it0 << 16)), op_y(li, k0, c0, newz ? 1 : 0, row0, h.w & 31));
    if (mine == 2)
      ops[at + 1] = make_uint2((unsigned)(ip1 | (it1 << 16)), op_y(li, k1, c1, 0, row1, h.w & 31));
    n += __popc(m1) + __popc(m2);
  }
  if (lane == 0) ops[n] = make_uint2(0u, op_y(l_end, kOpNone, kCiaNone, 0, 0, 0));
  __syncwarp();
  return n;
}

// Two adjacent wavenumbers of a staged table row (FP32, or FP16 log10 sigma decoded) as a packed
// FP32 pair: columns 4 lane + 128 g + {0, 1} and {2, 3} of the tile in lo and hi.
template <bool F16>
__device__ __forceinline__ void row_pairs(const unsigned char* row, int g, int lane, float off,
                                          unsigned long long& lo, unsigned long long& hi) {
  if constexpr (F16) {
    const uint2 r = *reinterpret_cast<const uint2*>(row + 256 * g + 8 * lane);
    const float2 a = __half22float2(*reinterpret_cast<const __half2*>(&r.x));
    const float2 c = __half22float2(*reinterpret_cast<const __half2*>(&r.y));
    asm("mov.b64 %0, {%1, %2};" : "=l"(lo) : "f"(ex2_fast((a.x + off) * kLog2Of10)),
                                             "f"(ex2_fast((a.y + off) * kLog2Of10)));
    asm("mov.b64 %0, {%1, %2};" : "=l"(hi) : "f"(ex2_fast((c.x + off) * kLog2Of10)),
                                             "f"(ex2_fast((c.y + off) * kLog2Of10)));
  } else {
    const ulonglong2 r = *reinterpret_cast<const ulonglong2*>(row + 512 * g + 16 * lane);
    lo = r.x;
    hi = r.y;
  }
}

// Bytes of a ring stage: two rows of every molecule, one of every CIA pair.
struct RowStage {
  unsigned mol, cia, bytes;
  __host__ __device__ RowStage(int n_mol, int n_cia, bool f16)
      : mol((unsigned)(2 * n_mol * kRowTW * (f16 ? 2 : 4))), cia((unsigned)(n_cia * kRowTW * 4)),
        bytes((mol + cia + 127u) & ~127u) {}
};

// NMOL absorbers (ANY: at most NMOL, p.n_mol of them) and NCIA pairs (ANY: at most NCIA; else
// NCIA or none).
template <int NMOL, int NCIA, bool ANY, bool F16>
__global__ void __launch_bounds__(32 * kRowWarps, kRowCtas)
k_opacity_rows(FwdParams p, const __grid_constant__ CUtensorMap tm_t,
               const __grid_constant__ CUtensorMap tm_p, const __grid_constant__ CUtensorMap tm_c,
               float* __restrict__ kbuf, long long kcols, int Bc, int n_groups, int n_lb,
               int lb_size, int n_stages) {
  extern __shared__ unsigned char row_raw[];
  __shared__ __align__(8) uint64_t full[kRowWarps][kRowMaxStages];
  __shared__ int n_ops_s;
  pdl_trigger();                                    // the contraction may launch (it waits)
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const OpUnit o = op_unit(p, blockIdx.x, Bc, n_lb, lb_size);   // o.tile: a group of tiles
  if (o.l_begin >= o.l_end) return;
  const int b = p.b_off + o.bc;
  const RowStage plan(p.n_mol, p.n_cia, F16);
  unsigned char* base = reinterpret_cast<unsigned char*>(
      (reinterpret_cast<uintptr_t>(row_raw) + 127) & ~(uintptr_t)127);
  unsigned char* ring = base + (size_t)warp * n_stages * plan.bytes;
  const float4* cf = reinterpret_cast<float4*>(base + (size_t)kRowWarps * n_stages * plan.bytes);
  uint2* ops = reinterpret_cast<uint2*>(const_cast<float4*>(cf) + 4 * lb_size);

  // the CTA's layer coefficients (last warp) and row operations (first warp)
  if (warp == kRowWarps - 1) {
    const float4* src = p.buf.op + ((size_t)b * p.max_layers + o.l_begin) * 2;
    for (int i = lane; i < 2 * (o.l_end - o.l_begin); i += 32) {
      const float4 v = __ldg(src + i);                // each twice: operands of the packed FMAs
      const_cast<float4*>(cf)[2 * i] = make_float4(v.x, v.x, v.y, v.y);
      const_cast<float4*>(cf)[2 * i + 1] = make_float4(v.z, v.z, v.w, v.w);
    }
  }
  if (warp == 0) {
    const int n = build_ops(p, b, o.l_begin, o.l_end, lane, ops);
    if (lane == 0) n_ops_s = n;
  }
  const int tile0 = (o.tile * kRowWarps + warp) * kRowTW;   // first column of this warp's tile
  const int x0 = wn_first(p.wn_begin) + tile0;
  const bool active = tile0 < kcols;
  if (lane == 0) {
    for (int i = 0; i < n_stages; ++i) mbar_init(&full[warp][i], 1);
    mbar_fence_init();
  }
  // packed FP32 pairs throughout: each half is rounded as fmaf would
  constexpr int G = kRowTW / 128, V2 = 2 * G;       // groups of four wavenumbers; pairs per lane
  unsigned long long us[4][V2] = {}, uc[2][V2] = {}, ray[V2];
  float xm[NMOL], yq[NCIA];
  auto weights = [&](int zone) {
    item_weights<NMOL, NCIA>(p, b, zone, xm, yq);
#pragma unroll
    for (int i = 0; i < V2; ++i) ray[i] = 0ull;
    if (p.ray) {                                    // species order, as rayleigh2
      const float* rc = p.buf.rayc + ((size_t)b * kMaxZones + zone) * TR_MAX_SPECIES;
#pragma unroll 2
      for (int sp = 0; sp < p.n_species; ++sp) {
        const unsigned long long c = pack_dup(__ldg(rc + sp));
#pragma unroll
        for (int g = 0; g < G; ++g) {
          const int w = x0 + 128 * g + 4 * lane;
          if (w < p.wn_pad) {
            const ulonglong2 r = __ldg(reinterpret_cast<const ulonglong2*>(p.ray + (size_t)sp * p.wn_pad + w));
            ffma2(ray[2 * g], c, r.x);
            ffma2(ray[2 * g + 1], c, r.y);
          }
        }
      }
    }
  };
  if (active) weights(p.buf.zoned ? (int)__ldg(&p.buf.layers[(size_t)b * p.max_layers + o.l_begin].zone) : 0);
  __syncthreads();
  if (!active) return;
  const int n_ops = n_ops_s;

  // lane 0 starts the loads of operation k into its stage
  auto issue = [&](int k) {
    const uint2 op = ops[k];
    const int st = k % n_stages;
    unsigned char* sb = ring + (size_t)st * plan.bytes;
    const unsigned kind = (op.y >> 8) & 7u, ck = (op.y >> 11) & 7u;
    mbar_arrive_expect_tx(&full[warp][st], (kind ? plan.mol : 0u) + (ck ? plan.cia : 0u));
    if (kind) {
      tma_load_4d(sb, (kind == kOpTUp || kind == kOpTDown) ? &tm_p : &tm_t, x0, (int)(op.x >> 16),
                  (int)(op.x & 0xffffu), 0, &full[warp][st]);
    }
    if (ck) tma_load_3d(sb + plan.mol, &tm_c, x0, (int)((op.y >> 16) & 0x3ffu), 0, &full[warp][st]);
  };
  if (lane == 0)
    for (int k = 0; k < n_stages && k < n_ops; ++k) issue(k);

  bool in_row[G];
#pragma unroll
  for (int g = 0; g < G; ++g) in_row[g] = x0 + 128 * g + 4 * lane < p.wn_pad;
  const bool whole = x0 + kRowTW <= p.wn_pad;       // no column beyond the rows
  float* dst = kbuf + k_index(o.bc, tile0, o.l_begin, kcols, p.max_layers) + 4 * lane;
  const size_t g_step = (size_t)p.max_layers * kKTile;      // to the next 128 wavenumbers
  const int g_store = (int)min((long long)G, (kcols - tile0) / 128);

  int st = 0;
  unsigned par = 0;
  for (int k = 0; k < n_ops; ++k) {
    const uint2 op = ops[k];
    if (!__all_sync(0xffffffffu, mbar_wait_bounded(&full[warp][st], par, p.dev_err, TR_DEVERR_TIMEOUT))) {
      // give up; the copies in flight land before the CTA may exit (bounded)
      for (int d = 0; d < n_stages && k + d < n_ops; ++d)
        mbar_wait_bounded(&full[warp][(k + d) % n_stages], ((k + d) / n_stages) & 1, nullptr, 0);
      return;
    }
    if ((op.y >> 14) & 1u) weights((int)(op.y >> 26));   // another chemistry zone (two-layer gases)
    const unsigned kind = (op.y >> 8) & 7u, ck = (op.y >> 11) & 7u;
    const unsigned char* sb = ring + (size_t)st * plan.bytes;
    // the sums of the two rows of every molecule, in the species order of every caller, into d0
    // and d1
    auto sums = [&](unsigned long long (&d0)[V2], unsigned long long (&d1)[V2]) {
#pragma unroll
      for (int i = 0; i < V2; ++i) d0[i] = d1[i] = 0ull;
#pragma unroll
      for (int m = 0; m < NMOL; ++m)
        if (!ANY || m < p.n_mol) {
          const float off = F16 ? p.logsig_off[m] : 0.f;
          const unsigned long long x = pack_dup(xm[m]);
          const unsigned char* ra = sb + (size_t)(2 * m) * kRowTW * (F16 ? 2 : 4);
          const unsigned char* rb = ra + kRowTW * (F16 ? 2 : 4);
#pragma unroll
          for (int g = 0; g < G; ++g) {
            unsigned long long lo, hi;
            row_pairs<F16>(ra, g, lane, off, lo, hi);
            ffma2(d0[2 * g], x, lo);
            ffma2(d0[2 * g + 1], x, hi);
            row_pairs<F16>(rb, g, lane, off, lo, hi);
            ffma2(d1[2 * g], x, lo);
            ffma2(d1[2 * g + 1], x, hi);
          }
        }
    };
    auto move = [&](unsigned long long (&d)[V2], const unsigned long long (&from)[V2]) {
#pragma unroll
      for (int i = 0; i < V2; ++i) d[i] = from[i];
    };
    // a P step down moves the lower P's sums to the upper corners, a T step the sums of one T
    // to the other side of the bracket
    switch (kind) {
      case kOpPDown: move(us[2], us[0]); move(us[3], us[1]); sums(us[0], us[1]); break;
      case kOpTUp: move(us[0], us[1]); move(us[2], us[3]); sums(us[1], us[3]); break;
      case kOpTDown: move(us[1], us[0]); move(us[3], us[2]); sums(us[0], us[2]); break;
      case kOpSet01: sums(us[0], us[1]); break;
      case kOpSet23: sums(us[2], us[3]); break;
      default: break;
    }
    if (ck) {
      unsigned long long s[V2] = {};
#pragma unroll
      for (int q = 0; q < NCIA; ++q)
        if (!ANY || q < p.n_cia) {
          const unsigned long long x = pack_dup(yq[q]);
#pragma unroll
          for (int g = 0; g < G; ++g) {
            unsigned long long lo, hi;
            row_pairs<false>(sb + plan.mol + (size_t)q * kRowTW * 4, g, lane, 0.f, lo, hi);
            ffma2(s[2 * g], x, lo);
            ffma2(s[2 * g + 1], x, hi);
          }
        }
#pragma unroll
      for (int i = 0; i < V2; ++i) {
        if (ck == kCiaUp) uc[0][i] = uc[1][i];
        if (ck == kCiaDown) uc[1][i] = uc[0][i];
        if (ck == kCiaUp || ck == kCiaSet1) uc[1][i] = s[i];
        else uc[0][i] = s[i];
      }
    }
    __syncwarp();                                   // every lane has read the stage
    if (lane == 0 && k + n_stages < n_ops) issue(k + n_stages);
    if (++st == n_stages) { st = 0; par ^= 1u; }

    // the layers up to the next operation, all of one cell
#pragma unroll 1
    for (int n = (int)(ops[k + 1].y & 0xffu) - (int)(op.y & 0xffu); n > 0; --n) {
      const ulonglong2* c = reinterpret_cast<const ulonglong2*>(cf);
      const ulonglong2 w01 = c[0], w23 = c[1], y01 = c[2], rk = c[3];
      cf += 4;
      unsigned long long kk[V2];
#pragma unroll
      for (int i = 0; i < V2; ++i) {
        kk[i] = fma2(rk.x, ray[i], rk.y);
        ffma2(kk[i], w01.x, us[0][i]);
        ffma2(kk[i], w01.y, us[1][i]);
        ffma2(kk[i], w23.x, us[2][i]);
        ffma2(kk[i], w23.y, us[3][i]);
        ffma2(kk[i], y01.x, uc[0][i]);
        ffma2(kk[i], y01.y, uc[1][i]);
      }
      if (!whole) {
#pragma unroll
        for (int g = 0; g < G; ++g)
          if (!in_row[g]) kk[2 * g] = kk[2 * g + 1] = 0ull;
      }
#pragma unroll
      for (int g = 0; g < G; ++g)
        if (g < g_store) {
          const float2 lo = *reinterpret_cast<const float2*>(&kk[2 * g]), hi = *reinterpret_cast<const float2*>(&kk[2 * g + 1]);
          __stcs(reinterpret_cast<float4*>(dst + g_step * g), make_float4(lo.x, lo.y, hi.x, hi.y));
        }
      dst += kKTile;
    }
  }
}

template <int NMOL, int NCIA, bool ANY, bool F16>
cudaError_t launch_t(const FwdParams& p, const RowMaps& tm, int Bc, float* kbuf, long long kcols,
                     int cap, cudaStream_t s) {
  auto kern = k_opacity_rows<NMOL, NCIA, ANY, F16>;
  const int tiles = (int)((kcols + kRowTW - 1) / kRowTW), groups = (tiles + kRowWarps - 1) / kRowWarps;
  const RowStage plan(p.n_mol, p.n_cia, F16);
  constexpr unsigned kSm = 227u * 1024u, kCta = 1024u + 256u;   // per SM; runtime and static
  int n_sm = 1, dev = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
  const long long units0 = (long long)Bc * groups;
  const int n_lb = opacity_layer_blocks(units0, 4LL * std::max(n_sm, 1), p.max_layers);
  const int lb_size = (p.max_layers + n_lb - 1) / n_lb;
  const long long ctas = units0 * n_lb;
  if (ctas > 0x7fffffffLL) return cudaErrorInvalidValue;
  const unsigned list = (unsigned)(64 * lb_size + 8 * (2 * lb_size + 1)) + 128u;
  const unsigned ring1 = kRowWarps * plan.bytes;                // one stage of every warp
  // As many CTAs as fit with one stage per warp (at most what the registers allow, or the
  // caller's cap), then the deepest rings that fit them.  Warps count for more than depth: 64
  // full-size atmospheres take 1.83 ms with 12 warps of one stage, 2.23 ms with 8 of two and
  // 2.63 ms with 6 of two (a stage is refilled while the layers after its operation are formed).
  const int most = cap > 0 ? std::min(cap, kRowCtas) : kRowCtas;
  long long per_sm = std::max<long long>(1, std::min<long long>(most, kSm / (ring1 + list + kCta)));
  per_sm = std::min(per_sm, std::max<long long>(1, (ctas + n_sm - 1) / n_sm));
  int stages = ring1 > 0 ? (int)(((long long)kSm / per_sm - kCta - list) / ring1) : 1;
  stages = std::max(1, std::min(stages, kRowMaxStages));
  unsigned smem = (unsigned)stages * ring1 + list;
  if (cap > 0) smem = std::max(smem, kSm / (cap + 1) + 1u);     // no more than cap CTAs per SM
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  kern<<<(unsigned)ctas, 32 * kRowWarps, smem, s>>>(p, *tm.t_pair, *tm.p_pair, *tm.cia, kbuf, kcols,
                                                    Bc, groups, n_lb, lb_size, stages);
  return cudaGetLastError();
}

template <bool F16>
cudaError_t launch_f(const FwdParams& p, const RowMaps& tm, int Bc, float* kbuf, long long kcols,
                     int cap, cudaStream_t s) {
  static_assert(TR_MAX_MOL == 8 && TR_MAX_CIA == 4, "opacity instantiations cover the limits");
  if (p.n_cia == 0 || p.n_cia == 2) {
    switch (p.n_mol) {
      case 1: return launch_t<1, 2, false, F16>(p, tm, Bc, kbuf, kcols, cap, s);
      case 2: return launch_t<2, 2, false, F16>(p, tm, Bc, kbuf, kcols, cap, s);
      case 3: return launch_t<3, 2, false, F16>(p, tm, Bc, kbuf, kcols, cap, s);
      case 4: return launch_t<4, 2, false, F16>(p, tm, Bc, kbuf, kcols, cap, s);
      case 5: return launch_t<5, 2, false, F16>(p, tm, Bc, kbuf, kcols, cap, s);
      default: break;
    }
  }
  return launch_t<8, 4, true, F16>(p, tm, Bc, kbuf, kcols, cap, s);
}

}  // namespace

cudaError_t launch_opacity_rows(const FwdParams& p, const RowMaps& tm, int Bc, float* kbuf,
                                long long kcols, int cap, cudaStream_t s) {
  static_assert(TR_MAX_LAYERS < 256, "operation fields");
  return p.logsig16 ? launch_f<true>(p, tm, Bc, kbuf, kcols, cap, s)
                    : launch_f<false>(p, tm, Bc, kbuf, kcols, cap, s);
}

}  // namespace tr
