// tc_fp32.cu -- the FP32 path's slant optical depth tau[ray, wn] = sum_{l >= j} DL[j][l] K[l][wn]
// (Sec. 4, eqs. tot_opt_dpth, opt_dpth) on the 5th-generation tensor cores as three TF32
// products (3xTF32), and the transit depth D = (R_p/R_s)^2 + sum_j a_j (1 - e^-tau_j) (Sec. 4).
// Every FP32 operand x is split exactly into hi = x with its 13 low mantissa bits cleared (a
// TF32 value) and lo = x - hi, and tau = K_hi DL_hi + K_hi DL_lo + K_lo DL_hi is accumulated in
// FP32 in tensor memory.  The dropped K_lo DL_lo term and the TF32 rounding of the lo parts
// each stay below 2^-20 of a product, the size of FP32 accumulation error over the column.
//
// k_contract_tc: persistent, one CTA per SM over a contiguous range of (item, 128-wn) units.
// A unit's layers are taken as two halves (the top half first): each half is a job of its own
// for the loads, the splitters and the MMA, so the loads of later halves, the split of one half
// and the MMAs of the one before overlap.
// The kernel is instantiated per padded layer count, so the MMA issue and split loops are
// unrolled with constant operands: issued from a runtime loop, the MMAs went at about half the
// rate (the issuing thread, not the tensor pipe, set the pace).
// Warp roles, every hand-over through an mbarrier:
//   * warp 8 (producer): TMA loads of a half's FP32 K rows [KP / 2 layers][128 wn] (boxes of 8
//     rows of the opacity kernel's K buffer) into a ring of up to eight half-unit stages;
//   * warps 0-3 and 10-13 (splitters; thread = TMEM lane = one wavenumber of the unit; the first
//     four take the top halves, the others the bottom halves, side by side): per half, each
//     thread splits its wavenumber's K values of the half's layers (zero at and beyond N) and
//     stores K_hi and K_lo into its half's TMEM buffer (the MMA's A operand, column = layer);
//     when the item changes (once every MMA of the previous unit is done), one thread
//     bulk-copies the item's path-length tiles DL_hi / DL_lo (built once per item by k_dl_tf32)
//     into shared memory;
//   * warp 9 (one thread): per half, for its 8-layer slices from the top down, three MMAs
//     D[128 x N_ks] (+)= A[128 x 8] B[N_ks x 8]^T, N_ks the rays the slice reaches (DL = 0 for
//     rays above a layer), into the unit's one of two TMEM accumulators; a commit frees the
//     half buffer, one after the bottom half hands the accumulator to the epilogue;
//   * warps 4-7 (epilogue): tau from TMEM -> sum_j a_j (1 - e^-tau_j) -> FP64 depth.
// What sets the pace, 100 layers x 200,000 wavenumbers (10.3 units of 112 x 128 an SM; K read at
// the copy bandwidth would take 11.8 us): 30.6 us an atmosphere in batches of 64 at first, 27.7
// with the path-length tiles cut to the rays each slice reaches (57 KB instead of 100), which
// makes room for six half-unit stages (two whole-unit stages were refilled a unit late), 21.0 with
// the MMA thread elected by elect.sync and its descriptors moved by constants (the issuing
// thread's operand moves took about 100 cycles an MMA, the tensor pipe 32), 19.0 with the halves
// split side by side (the split alone took 3,000 cycles a unit, mostly waits), 18.8 with the
// epilogue's TMEM loads one step ahead.  One atmosphere: 42.6 -> 28.6 us.  Left: without the
// epilogue 14.3 (its exponentials share the SM with the split), without the MMAs 16.2.  Two CTAs
// per SM with 32-layer chunks took 23.3; a second epilogue group 22.2 (spills).
// All waits are bounded; on a timeout every role stops, in-flight copies and MMAs are waited
// for (bounded) and the TMEM is released before the CTA exits.
#include <algorithm>
#include "tma.h"
#include "tr_internal.h"
#include "umma.h"

namespace tr {
namespace {

constexpr int kTM = 128;                  // wavenumbers per unit = MMA M = TMEM lanes
constexpr int kTEpi0 = 4;                 // epilogue warps 4..7
constexpr int kTProd = 8;
constexpr int kTMma = 9;
constexpr int kTSplit1 = 10;              // splitters: warps 0..3 and 10..13
constexpr int kTSplitters = 4;            // warps per half: 0..3 the top halves, 10..13 the bottom
constexpr int kTThreads = 32 * (kTSplit1 + 4);
constexpr int kTMaxKP = 112;              // layers (padded to 16) the kernel takes
// TMEM columns: half buffer h at 128 h (K_hi at + 0, K_lo at + 64, KP / 2 columns each);
// accumulators at 256 and 384 (NP columns)
constexpr uint32_t kColHalf = 128, kColLo = 64, kColD0 = 256, kColD1 = 384, kTmemCols = 512;

__host__ __device__ inline int pad16i(int n) { return (n + 15) & ~15; }

// Rays slice ks (layers 8 ks .. 8 ks + 7) reaches: j <= 8 ks + 7, rounded up to the MMA's N step
// of 16; slices 2 m and 2 m + 1 both 16 (m + 1).  A slice's path-length tile is its rays x 8
// layers in K-major core matrices (8 rays x 4 layers, 128 bytes): ray group g, layer half c at
// 128 (2 g + c).  Core matrices before slice ks: dl_cores(ks).
__host__ __device__ constexpr int dl_cores(int ks) {
  return 4 * (ks / 2) * (ks / 2 + 1) + (ks & 1) * 4 * (ks / 2 + 1);
}

constexpr int kTMaxStages = 8;
struct TcLayout {
  uint32_t stage, dl_bytes, dl, aj, total;
  int stages;
  __host__ __device__ TcLayout(int KP) {
    stage = (uint32_t)(KP / 2) * kTM * 4;                 // FP32 K rows of a half [KP / 2][128]
    dl_bytes = (uint32_t)dl_cores(KP / 8) * 128u;         // DL_hi; DL_lo follows
    const uint32_t rest = 2 * dl_bytes + 2u * kTM * 4 + 128u;   // + alignment slack
    constexpr uint32_t kDyn = 227u * 1024u - 256u;        // less the static shared memory
    stages = (int)((kDyn - rest) / stage);
    if (stages > kTMaxStages) stages = kTMaxStages;
    dl = (uint32_t)stages * stage;
    aj = dl + 2 * dl_bytes;
    total = dl + rest;
  }
};

// x with the 13 low mantissa bits cleared: exactly a TF32 value, whatever rounding the tensor
// core applies to its inputs
__device__ __forceinline__ float tf32_hi(float x) {
  return __uint_as_float(__float_as_uint(x) & 0xFFFFE000u);
}

// The path-length tiles of every item, the MMA's B operand: tiles[b][0] = DL_hi, [b][1] =
// DL_lo, each the slices' core matrices (see dl_cores; row j % 8, column l % 4), zero for j > l and
// outside the item's N layers.  Grid (core matrices / 4, B items): a warp writes one core
// matrix per store (lane = (ray, layer) of it, one value each) from four 32-byte row segments
// of the geometry kernel's layer-major DL.
__global__ void __launch_bounds__(128)
k_dl_tf32(ItemBuffers buf, int max_layers, int n_cm, float* __restrict__ tiles) {
  pdl_wait();                                               // the path lengths are written
  const int b = blockIdx.y;
  const int q = 4 * blockIdx.x + (threadIdx.x >> 5);        // core matrix of this warp
  if (q >= n_cm) return;
  int m = 0;                                                // its pair of slices
  while (4 * (m + 1) * (m + 2) <= q) ++m;
  int rem = q - 4 * m * (m + 1);
  const int odd = rem >= 4 * (m + 1) ? 1 : 0;
  rem -= odd * 4 * (m + 1);
  const int lane = threadIdx.x & 31, r = lane >> 2, c = lane & 3;
  const int j = 8 * (rem >> 1) + r, l = 8 * (2 * m + odd) + 4 * (rem & 1) + c;
  const int N = buf.items[b].n_layers;
  const float* dlt = buf.dlt + (size_t)b * max_layers * buf.npad;
  const float x = (l < N && j <= l) ? dlt[(size_t)l * buf.npad + j] : 0.f;
  const float h = tf32_hi(x);
  float* hi = tiles + ((size_t)b * 2 * n_cm + q) * 32;
  hi[lane] = h;                                             // row r, column c: 4 r + c = lane
  hi[(size_t)n_cm * 32 + lane] = x - h;
}

// Barrier over `threads` threads (named barrier `id`) that also returns whether any of them
// passed pred = true: the warps of one role take the same stop decision.
__device__ __forceinline__ bool tc_sync_or(int id, int threads, bool pred) {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.u32 p, %1, 0;\n\t"
      "barrier.red.or.pred q, %2, %3, p;\n\t"
      "selp.u32 %0, 1, 0, q;\n\t}"
      : "=r"(r) : "r"((uint32_t)pred), "r"(id), "r"(threads) : "memory");
  return r != 0;
}

// Instantiated per padded layer count KP (16 .. 112): the MMA issue loop and the split loop are
// unrolled with constant operands (a runtime loop issued the MMAs at about half the rate).
template <int KP>
__global__ void __launch_bounds__(kTThreads, 1)
k_contract_tc(FwdParams p, const __grid_constant__ CUtensorMap tm_k, int Bc, int n_tiles,
              const float* __restrict__ tiles) {
  constexpr int NP = KP;                    // rays (padded) = layers (padded)
  extern __shared__ __align__(128) uint8_t tsm_raw[];
  __shared__ __align__(8) uint64_t sfull[kTMaxStages], sempty[kTMaxStages], hfull[2], hfree[2],
      accfull[2], accempty[2], dlfull;
  __shared__ uint32_t tmem_base;
  __shared__ int abort_flag;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(tsm_raw) + 127) &
                                             ~(uintptr_t)127);
  const TcLayout lay(KP);
  const int S = lay.stages;
  uint8_t* B_hi = base + lay.dl;
  uint8_t* B_lo = B_hi + lay.dl_bytes;
  float* ep_aj = reinterpret_cast<float*>(base + lay.aj);      // [2][128], epilogue's copy
  const long long units = (long long)Bc * n_tiles;
  const long long per = (units + gridDim.x - 1) / gridDim.x;
  const long long u_begin = (long long)blockIdx.x * per;
  const long long u_end = u_begin + per < units ? u_begin + per : units;
  const int n_units = u_end > u_begin ? (int)(u_end - u_begin) : 0;
  const int wbase = wn_first(p.wn_begin);
  constexpr int HL = KP / 2;                // layers of a half (a multiple of 8)

  if (warp == 0) tmem_alloc(&tmem_base, kTmemCols);
  if (tid == 0) {
    for (int i = 0; i < S; ++i) { mbar_init(&sfull[i], 1); mbar_init(&sempty[i], kTSplitters); }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&hfull[i], kTSplitters); mbar_init(&hfree[i], 1);
      mbar_init(&accfull[i], 1); mbar_init(&accempty[i], 4);
    }
    mbar_init(&dlfull, 1);
    abort_flag = 0;
    mbar_fence_init();
  }
  tcgen05_fence_before();
  __syncthreads();
  tcgen05_fence_after();
  const uint32_t tmem = tmem_base;
  // launched as a dependent of the opacity kernel: only the set-up above overlaps its tail
  pdl_wait();                                   // K and the path-length tiles are written

  if (warp == kTProd) {
    // ---------------- producer
    if (lane == 0) {
      // half job h = 2k + (1 - hh): the rows of half hh (top half first) of unit k
      const int n_jobs = 2 * n_units;
      int h = 0, st = 0, q = 0;
      for (; h < n_jobs; ++h) {
        const long long u = u_begin + (h >> 1);
        const int row0 = (int)u * p.max_layers + ((h & 1) ? 0 : HL);   // u = bc n_tiles + tile
        const bool ok = q == 0 ||
                        mbar_wait_bounded(&sempty[st], (q - 1) & 1, p.dev_err, TR_DEVERR_TIMEOUT);
        if (!ok || *(volatile int*)&abort_flag) { atomicExch(&abort_flag, 1); break; }
        uint8_t* sb = base + (size_t)st * lay.stage;
        mbar_arrive_expect_tx(&sfull[st], lay.stage);
        for (int i = 0; i < HL / 8; ++i)
          tma_load_2d(sb + (size_t)i * 8 * kTM * 4, &tm_k, 0, row0 + i * 8, &sfull[st]);
        if (++st == S) { st = 0; ++q; }
      }
      for (int i = 0; i < S && i < h; ++i) {      // every copy issued has landed
        const int hl = h - 1 - i;
        mbar_wait_bounded(&sfull[hl % S], (hl / S) & 1, nullptr, 0);
      }
    }
  } else if (warp < kTEpi0 || warp >= kTSplit1) {
    // ---------------- splitters: thread v = wavenumber row v of the unit = TMEM lane v
    const int v = 32 * (warp & 3) + lane;          // 0 .. 127
    const uint32_t lane_base = (uint32_t)(32 * (warp & 3)) << 16;
    const int hb = warp >= kTSplit1 ? 1 : 0;       // half job parity: 0 top halves, 1 bottom
    const int l0 = hb ? 0 : HL;                    // the half's first layer
    const bool lead = tid == 32 * kTSplit1;        // copies the items' path-length tiles
    int dl_item = -1, dl_issued = 0;
    int st = hb, sq = 0;                           // stage of half job 2k + hb
    while (st >= S) { st -= S; ++sq; }
    for (int k = 0; k < n_units; ++k) {
      const long long u = u_begin + k;
      const int b = p.b_off + (int)(u / n_tiles);
      const int N = __ldg(&p.buf.items[b].n_layers);
      // half job 2k + hb: the MMAs of half job 2k - 2 + hb are done with its half buffer
      bool hok = (k == 0 || mbar_wait_bounded(&hfree[hb], (k - 1) & 1, p.dev_err, TR_DEVERR_TIMEOUT)) &&
                 !*(volatile int*)&abort_flag;
      // when the item changes, its path-length tiles replace the old ones once every MMA of unit
      // k - 1 is done: the commit of its bottom half, just waited for by the bottom halves'
      // splitters, completes after all of them.  The MMA thread waits for the copy
      if (lead && hok && b != dl_item) {
        const char* src = reinterpret_cast<const char*>(tiles) + (size_t)b * 2 * lay.dl_bytes;
        mbar_arrive_expect_tx(&dlfull, 2u * lay.dl_bytes);
        bulk_g2s(B_hi, src, lay.dl_bytes, &dlfull);
        bulk_g2s(B_lo, src + lay.dl_bytes, lay.dl_bytes, &dlfull);
        ++dl_issued;
        dl_item = b;
      }
      __syncwarp();
      // its K rows have landed
      hok = hok && mbar_wait_bounded(&sfull[st], sq & 1, p.dev_err, TR_DEVERR_TIMEOUT);
      if (!__all_sync(0xffffffffu, hok)) { if (lane == 0) atomicExch(&abort_flag, 1); break; }
      tcgen05_fence_after();
      const float* kf = reinterpret_cast<const float*>(base + (size_t)st * lay.stage);
      const uint32_t col = tmem + lane_base + kColHalf * hb;
      const int n_half = N - l0;                     // layers of the half below the item's top
#pragma unroll
      for (int g = 0; g < HL / 8; ++g) {
        uint32_t hi[8], lo[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const int l = 8 * g + i;
          const float x = l < n_half ? kf[l * kTM + v] : 0.f;
          const float hv = tf32_hi(x);
          hi[i] = __float_as_uint(hv);
          lo[i] = __float_as_uint(x - hv);
        }
        tmem_st8(col + 8 * g, hi);
        tmem_st8(col + kColLo + 8 * g, lo);
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&sempty[st]);      // this warp's reads of the stage are done
      st += 2;
      while (st >= S) { st -= S; ++sq; }
      tmem_st_wait();
      tcgen05_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&hfull[hb]);       // this warp's rows of the half are written
    }
    // the last tile copy has landed before the CTA may exit (the MMA thread observes every copy
    // but the last one when the CTA stops early)
    if (dl_issued > 0) mbar_wait_bounded(&dlfull, (dl_issued - 1) & 1, nullptr, 0);
  } else if (warp == kTMma) {
    // ---------------- MMA issue (one thread)
    if (elect_one()) {
      const uint64_t dh0 = umma_smem_desc(smem_addr(B_hi), 128, 256);
      const uint64_t dl0 = umma_smem_desc(smem_addr(B_lo), 128, 256);
      uint64_t* last = nullptr;                     // the last commit issued and its phase
      int last_par = 0, dl_item = -1, dl_copies = 0;
      bool stop = false;
      for (int k = 0; k < n_units && !stop; ++k) {
        const int a = k & 1, q = k >> 1;
        const int b = p.b_off + (int)((u_begin + k) / n_tiles);
        bool ok = q == 0 ||
                  mbar_wait_bounded(&accempty[a], (q - 1) & 1, p.dev_err, TR_DEVERR_TIMEOUT);
        // a new item's path-length tiles have landed (the splitters copy them at the item's
        // first unit, after every MMA of the previous unit is done)
        if (ok && b != dl_item) {
          ok = mbar_wait_bounded(&dlfull, dl_copies & 1, p.dev_err, TR_DEVERR_TIMEOUT);
          ++dl_copies;
          dl_item = b;
        }
        if (!ok) { atomicExch(&abort_flag, 1); break; }
        const uint32_t d = tmem + (a ? kColD1 : kColD0);
        bool first = true;
#pragma unroll
        for (int hh = 1; hh >= 0; --hh) {
          const int h = 2 * k + (1 - hh), hb = h & 1, hq = h >> 1;
          ok = mbar_wait_bounded(&hfull[hb], hq & 1, p.dev_err, TR_DEVERR_TIMEOUT) &&
               !*(volatile int*)&abort_flag;
          if (!ok) { atomicExch(&abort_flag, 1); stop = true; break; }
          tcgen05_fence_after();
          const uint32_t ah = tmem + kColHalf * hb, al = ah + kColLo;
#pragma unroll
          for (int i = HL / 8 - 1; i >= 0; --i) {
            const int ks = hh * (HL / 8) + i;        // the slice's 8 layers: 8 ks .. 8 ks + 7
            // the rays slice ks reaches: j <= 8 ks + 7, rounded up to the MMA's N step of 16
            const int n = min(NP, pad16i(8 * ks + 8));
            const uint32_t idesc = umma_idesc_tf32_f32(kTM, n);
            const uint64_t koff = (uint64_t)dl_cores(ks) * (128 / 16);
            const uint64_t dh = dh0 + koff, dlo = dl0 + koff;
            umma_tf32_ta(d, ah + 8 * i, dh, idesc, first ? 0u : 1u);
            umma_tf32_ta(d, ah + 8 * i, dlo, idesc, 1u);
            umma_tf32_ta(d, al + 8 * i, dh, idesc, 1u);
            first = false;
          }
          umma_commit(&hfree[hb]);                  // the half buffer is free
          last = &hfree[hb];
          last_par = hq & 1;
        }
        if (!stop) umma_commit(&accfull[a]);        // the accumulator is ready
      }
      // the MMAs issued are complete before the CTA may release the TMEM (the last commit
      // issued completes after all of them)
      if (last) mbar_wait_bounded(last, (uint32_t)last_par, nullptr, 0);
    }
  } else {
    // ---------------- epilogue: thread = TMEM lane = wavenumber row
    const int row = 32 * (warp & 3) + lane;
    const uint32_t lane_base = (uint32_t)(32 * (warp & 3)) << 16;
    for (int k = 0; k < n_units; ++k) {
      const long long u = u_begin + k;
      const int bc = (int)(u / n_tiles), tile = (int)(u % n_tiles);
      const int b = p.b_off + bc;
      const ItemGeom ig = p.buf.items[b];
      const int a = k & 1;
      float* aj = ep_aj + a * kTM;
      if (row < NP) aj[row] = row < p.buf.npad ? __ldg(p.buf.aj + (size_t)b * p.buf.npad + row) : 0.f;
      const bool ok = mbar_wait_bounded(&accfull[a], (k >> 1) & 1, p.dev_err, TR_DEVERR_TIMEOUT) &&
                      !*(volatile int*)&abort_flag;
      // aj of this unit in place; all epilogue warps stop together on a failed wait
      if (tc_sync_or(2, 128, !ok)) { if (lane == 0) atomicExch(&abort_flag, 1); break; }
      tcgen05_fence_after();
      const uint32_t taddr = tmem + lane_base + (a ? kColD1 : kColD0);
      // 16 columns are read while the 16 before are summed
      float part = 0.f;
      uint32_t t[2][16];
      tmem_ld16_nowait(taddr, t[0]);
#pragma unroll
      for (int c0 = 0; c0 < NP; c0 += 16) {
        uint32_t* tau = t[(c0 / 16) & 1];
        tmem_ld_wait16(tau);
        if (c0 + 16 < NP) tmem_ld16_nowait(taddr + (uint32_t)(c0 + 16), t[(c0 / 16 + 1) & 1]);
#pragma unroll
        for (int i = 0; i < 16; i += 4) {
          const float4 w = *reinterpret_cast<const float4*>(aj + c0 + i);
          part = fmaf(w.x, 1.f - __expf(-__uint_as_float(tau[i])), part);
          part = fmaf(w.y, 1.f - __expf(-__uint_as_float(tau[i + 1])), part);
          part = fmaf(w.z, 1.f - __expf(-__uint_as_float(tau[i + 2])), part);
          part = fmaf(w.w, 1.f - __expf(-__uint_as_float(tau[i + 3])), part);
        }
      }
      tcgen05_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&accempty[a]);     // this warp's TMEM lanes are read
      const int w = wbase + tile * kTM + row;
      if (w >= p.wn_begin && w < p.wn_begin + p.wn_count)
        p.out[(long long)b * p.out_stride + (w - p.wn_begin)] =
            ig.n_layers > 0 ? ig.rp2_rs2 + (double)part : 0.0;
    }
  }
  tcgen05_fence_before();
  __syncthreads();
  if (warp == 0) tmem_dealloc(tmem, kTmemCols);
}

}  // namespace

size_t tc_dl_bytes(int B, int max_layers) {
  if (!tc_contract_fits(max_layers)) return 0;
  return 2 * (size_t)B * TcLayout(pad16i(max_layers)).dl_bytes;
}

cudaError_t launch_dl_tf32(const ItemBuffers& buf, int B, int max_layers, void* tiles,
                           cudaStream_t s) {
  if (B <= 0) return cudaSuccess;
  if (!tc_contract_fits(max_layers)) return cudaErrorInvalidValue;
  const int n_cm = dl_cores(pad16i(max_layers) / 8);
  if (B < kFewAtmospheres)                                  // as k_pathlen before it
    return launch_dependent(k_dl_tf32, dim3((n_cm + 3) / 4, B), dim3(128), 0, s, buf, max_layers,
                            n_cm, static_cast<float*>(tiles));
  k_dl_tf32<<<dim3((n_cm + 3) / 4, B), 128, 0, s>>>(buf, max_layers, n_cm,
                                                    static_cast<float*>(tiles));
  return cudaGetLastError();
}

bool tc_contract_fits(int max_layers) {
  const int KP = pad16i(max_layers);
  return max_layers >= 1 && KP <= kTMaxKP;
}

cudaError_t launch_contract_tc(const FwdParams& p, int Bc, const float* kbuf, const void* tiles,
                               cudaStream_t s) {
  if (Bc <= 0 || p.wn_count <= 0) return cudaSuccess;
  if (!tc_contract_fits(p.max_layers)) return cudaErrorInvalidValue;
  const int KP = pad16i(p.max_layers);
  const int w_first = wn_first(p.wn_begin);
  if (!tiles) return cudaErrorInvalidValue;
  const int tiles_w = (p.wn_begin + p.wn_count - w_first + kTM - 1) / kTM;
  CUtensorMap tm{};
  if (!encode_2d_f32(&tm, kbuf, kTM, (unsigned long long)Bc * tiles_w * p.max_layers, kTM * 4, kTM,
                     8))
    return cudaErrorInvalidValue;
  const uint32_t smem = TcLayout(KP).total;
  void (*kern)(FwdParams, CUtensorMap, int, int, const float*) = nullptr;
  switch (KP) {
    case 16: kern = k_contract_tc<16>; break;
    case 32: kern = k_contract_tc<32>; break;
    case 48: kern = k_contract_tc<48>; break;
    case 64: kern = k_contract_tc<64>; break;
    case 80: kern = k_contract_tc<80>; break;
    case 96: kern = k_contract_tc<96>; break;
    case 112: kern = k_contract_tc<112>; break;
    default: return cudaErrorInvalidValue;
  }
  static_assert(kTMaxKP == 112, "one instantiation per padded layer count");
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)smem);
  if (e != cudaSuccess) return e;
  int dev = 0, n_sm = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
  const long long units = (long long)Bc * tiles_w;
  const int grid = (int)std::min<long long>(units, (long long)std::max(n_sm, 1));
  return launch_dependent(kern, dim3(grid), dim3(kTThreads), smem, s, p, tm, Bc, tiles_w,
                          static_cast<const float*>(tiles));
}

}  // namespace tr
