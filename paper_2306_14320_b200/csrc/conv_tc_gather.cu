// im2win-based convolution (Algorithm 2) on the sm_100a tensor cores: the GATHER kernel, for problems that leave
// most of the chip idle in the other kernels and for filter sizes that none of them is specialised on.
//
// The contraction  O[p, j] = sum_k A[p][k] * F[j][k],  p = (i, m, n), k = (r, u, v), is cut into
//   128 output positions x NT filters x one of Z slices of the reduction
// per CTA.  An element of A lies at  base(p) + off(k)  in the source -- the untransformed input or the im2win tensor
// alike -- so any filter size, stride, channel and filter count is the same code: sixteen warps load their elements
// from global memory (lane = position: neighbouring lanes read neighbouring columns, and the Fh*Fw readings of an
// element meet in L1), convert, and write 16-byte pieces into a ring of K-major 128-byte-swizzled operand tiles; the
// filter's native rows take the same way, so no copy of the filter is made.  One warp issues tcgen05.mma (A and B
// from shared memory, accumulator in TMEM).  The Z slices of a tile are one thread-block cluster: each CTA leaves its
// partial tile in its shared memory, and every CTA of the cluster adds one Z-th of the columns from all of them
// (distributed shared memory, fixed order) and stores it.  One launch, no zeroed output, no atomics, same bits on
// every call.
//
// What bounds it: at small sizes the latency of one pass (launch, prologue, two trips to L2, epilogue); on large
// problems the loads (128 x 64 elements per 64 steps of the reduction, one 128-byte line or two per warp instruction;
// 0.8 us per stage and CTA, BF16).  The kernel with window tables and filter tiles built from the im2win tensor that
// served general filter sizes before: 2-12 x slower on every shape tried (B200: 3x4, 64 images of 64x56x56, K = 128,
// BF16 651 -> 229 us; 2x3, 16 of 32x60x60, K = 256, TF32 78 -> 40 us; 12x12 stride 4, 2 of 8x33x33, K = 24, TF32
// 110 -> 9 us).  Every wait is bounded (status word + common teardown on expiry).
#include <cuda.h>

#include <type_traits>

#include "common.cuh"
#include "ptx_sm100.cuh"
#include "strip_common.cuh"

namespace im2win {
namespace {

using namespace stripc;

constexpr int kGW = 16;                      // gather warps (and, afterwards, epilogue warps)
constexpr int kGThreads = (kGW + 1) * 32;    // + the MMA-issuing warp (the MMAs issued by a gather warp: 25-45 % slower stages)
constexpr int kGStages = 6;
constexpr int kGMaxZ = 16;                   // cluster size (above 8: non-portable)
constexpr int kBK = 64;                      // reduction elements per stage

struct GParams {
  const float* src;
  const float* f;
  float* out;
  int32_t* status;
  int32_t K, Wo;
  int64_t HoWo, Kg, Mtot;
  int64_t plane, row_mul, col_mul, u_mul, v_mul;  // source elements from one channel, output row, output column, filter row, filter column to the next
  int64_t img;                                    // source elements per image
  int32_t FF, Fw, Fh;
  int32_t NT, n_ntiles, Z;                        // filters per tile; reduction slices (cluster size)
  int64_t KS;                                     // reduction elements per slice
  int32_t SB;                                     // stages
  int32_t nhwc, vec;                              // vec: filter rows are whole 16-byte units
  int32_t wait_early;                             // the source may be written by the preceding kernel in the stream
  uint32_t idesc, tmem_cols, stage_bytes, off_bar;
};

struct GBars {
  uint64_t full[kGStages], empty[kGStages], acc;
};

__device__ __forceinline__ float lds_cluster_f32(uint32_t a) {
  float v;
  asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(a) : "memory");
  return v;
}

// NBT: 16-byte filter pieces per thread, operand block and stage (64 filters each).
// IX: type of positions, reduction indices and source offsets (64 bits: tensors of 2^31 elements and more).
template <bool BF16, int NBT, typename IX>
__global__ void __launch_bounds__(kGThreads, 1) conv_tc_gather_kernel(const GParams P) {
  constexpr int EPC = BF16 ? 8 : 4;    // reduction elements per 16-byte piece
  constexpr int SUB = BF16 ? 1 : 2;    // 128-byte operand rows per stage
  constexpr int BKS = kBK / SUB;       // reduction elements per operand row
  // Two register sets up to 128 filters: the next stage's loads are in flight while this one's values are stored.  (65 to 128
  // filters: 36 bytes a thread of it, TF32 60, spill at the 96 registers that 17 warps of one CTA leave.)
  constexpr bool AHEAD = NBT <= 2;
  using UX = typename std::make_unsigned<IX>::type;

  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint8_t* const smem = smem_raw + ((1024u - (ptx::smem_u32(smem_raw) & 1023u)) & 1023u);
  GBars* const bars = reinterpret_cast<GBars*>(smem + P.off_bar);
  SMisc* const misc = reinterpret_cast<SMisc*>(smem + P.off_bar + sizeof(GBars));
  const uint32_t sm0 = ptx::smem_u32(smem);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  const uint32_t z = P.Z > 1 ? cluster_ctarank() : 0u;
  const uint32_t unit = blockIdx.x / (uint32_t)P.Z;
  const uint32_t tile = unit / (uint32_t)P.n_ntiles;
  const int32_t n0 = (int32_t)(unit - tile * (uint32_t)P.n_ntiles) * P.NT;
  const IX HoWo = (IX)P.HoWo, Mtot = (IX)P.Mtot;
  const IX kbeg = (IX)z * (IX)P.KS, kend = min(kbeg + (IX)P.KS, (IX)P.Kg);
  const int32_t nst = (int32_t)((kend - kbeg + kBK - 1) / kBK);

  if (threadIdx.x == 0) {
    for (int i = 0; i < kGStages; ++i) {
      ptx::mbar_init(ptx::smem_u32(&bars->full[i]), kGW);
      ptx::mbar_init(ptx::smem_u32(&bars->empty[i]), 1);
    }
    ptx::mbar_init(ptx::smem_u32(&bars->acc), 1);
    ptx::fence_mbar_init();
    misc->abort = 0;
  }
  if (warp == kGW) {
    ptx::tmem_alloc(ptx::smem_u32(&misc->tmem_base), P.tmem_cols);
    ptx::tmem_relinquish();
  }
  const uint32_t a_bytes = SUB * 16384u;
  const uint32_t bar_full0 = ptx::smem_u32(&bars->full[0]), bar_empty0 = ptx::smem_u32(&bars->empty[0]);
  // (launched as a programmatic dependent: after a kernel that lets its dependents start early, the source and the
  // output are touched only once that grid has completed -- unless it is this call's own transform, which neither
  // writes what is read here nor reads what is written, and is only waited for before the end)
  if (P.wait_early) asm volatile("griddepcontrol.wait;" ::: "memory");

  bool ok = true;
  if (warp < kGW) {
    // ================================================================ GATHER: global memory -> operand tiles
    const int q = warp & 7;            // this warp's 16-byte column of the operand rows
    const int pg0 = (warp >> 3) * 2;   // and its two groups of 32 positions
    const float* base[2];
    uint32_t adst[2];
#pragma unroll
    for (int g = 0; g < 2; ++g) {
      // (positions past the end repeat the last one: their rows are computed and dropped)
      const int row = (pg0 + g) * 32 + lane;
      const UX p = min((UX)tile * 128u + (UX)row, (UX)Mtot - 1u);
      const UX i = p / (UX)HoWo, pq = p - i * (UX)HoWo;
      const UX m = pq / (UX)P.Wo, n = pq - m * (UX)P.Wo;
      base[g] = P.src + (int64_t)i * P.img + (int64_t)m * P.row_mul + (int64_t)n * P.col_mul;
      adst[g] = (uint32_t)((row >> 3) * 1024 + (row & 7) * 128 + ((q ^ (row & 7)) << 4));
    }
    // lane e < EPC walks off(k) for element e of the pieces: k = (r, u, v) advances by 64 per stage
    IX kr[SUB];
    int32_t ku[SUB], kv[SUB];
    const IX plane = (IX)P.plane, u_mul = (IX)P.u_mul, v_mul = (IX)P.v_mul;
    const int32_t dr = kBK / P.FF, dw = kBK - dr * P.FF, du = dw / P.Fw, dv = dw - du * P.Fw;
#pragma unroll
    for (int sb = 0; sb < SUB; ++sb) {
      const IX k = kbeg + sb * BKS + q * EPC + (lane & (EPC - 1));
      kr[sb] = k / P.FF;
      const int32_t w = (int32_t)(k - kr[sb] * P.FF);
      ku[sb] = w / P.Fw;
      kv[sb] = w - ku[sb] * P.Fw;
    }
    const int32_t tid = (int32_t)threadIdx.x;  // < 512
    const float* frow[NBT];
    bool fuse[NBT], frok[NBT];
    uint32_t fdst[NBT];
#pragma unroll
    for (int t = 0; t < NBT; ++t) {
      const int32_t idx = tid + t * (kGW * 32);
      const int32_t j = idx >> 3, c = idx & 7;
      fuse[t] = idx < P.NT * 8;
      frok[t] = fuse[t] && n0 + j < P.K;
      frow[t] = P.f + (frok[t] ? (int64_t)(n0 + j) * P.Kg : 0);
      fdst[t] = a_bytes + (uint32_t)((j >> 3) * 1024 + (j & 7) * 128 + ((c ^ (j & 7)) << 4));
    }
    const int32_t fk0 = (tid & 7) * EPC;

    struct Regs {
      float a[SUB][2][EPC];
      float b[SUB][NBT][EPC];
    };
    auto load = [&](int32_t it, Regs& R) {
#pragma unroll
      for (int sb = 0; sb < SUB; ++sb) {
        const IX k0 = kbeg + (IX)it * kBK + sb * BKS;
        const IX ka = k0 + q * EPC;
        const bool mine = ka + (lane & (EPC - 1)) < kend;
        const IX off = mine ? kr[sb] * plane + ku[sb] * u_mul + kv[sb] * v_mul : 0;
        kv[sb] += dv; ku[sb] += du; kr[sb] += dr;
        if (kv[sb] >= P.Fw) { kv[sb] -= P.Fw; ++ku[sb]; }
        if (ku[sb] >= P.Fh) { ku[sb] -= P.Fh; ++kr[sb]; }
#pragma unroll
        for (int e = 0; e < EPC; ++e) {
          const IX o = __shfl_sync(0xffffffffu, off, e);
          R.a[sb][0][e] = __ldg(base[0] + o);
          R.a[sb][1][e] = __ldg(base[1] + o);
        }
        if (ka + EPC > kend) {  // the slice ends inside this piece: zeros behind it
#pragma unroll
          for (int e = 0; e < EPC; ++e)
            if (ka + e >= kend) { R.a[sb][0][e] = 0.f; R.a[sb][1][e] = 0.f; }
        }
#pragma unroll
        for (int t = 0; t < NBT; ++t) {
          const IX kb = k0 + fk0;
          if (frok[t] && P.vec && kb + EPC <= kend) {
#pragma unroll
            for (int e = 0; e < EPC; e += 4) {
              const float4 w = __ldg(reinterpret_cast<const float4*>(frow[t] + kb + e));
              R.b[sb][t][e] = w.x; R.b[sb][t][e + 1] = w.y; R.b[sb][t][e + 2] = w.z; R.b[sb][t][e + 3] = w.w;
            }
          } else {
#pragma unroll
            for (int e = 0; e < EPC; ++e) R.b[sb][t][e] = (frok[t] && kb + e < kend) ? __ldg(frow[t] + kb + e) : 0.f;
          }
        }
      }
    };
    auto piece = [&](uint32_t dst, const float (&x)[EPC]) {
      if constexpr (BF16)
        sts_v4(dst, ptx::pack_bf16x2(x[0], x[1]), ptx::pack_bf16x2(x[2], x[3]), ptx::pack_bf16x2(x[4], x[5]), ptx::pack_bf16x2(x[6], x[7]));
      else
        sts_v4(dst, __float_as_uint(x[0]), __float_as_uint(x[1]), __float_as_uint(x[2]), __float_as_uint(x[3]));
    };
    Ring er;
    auto store = [&](const Regs& R) -> bool {
      if (!wait_bar_warp(P, misc, bar_empty0 + (uint32_t)er.idx * 8u, er.phase ^ 1u, DEV_TIMEOUT_A_EMPTY)) return false;
      const uint32_t stage = sm0 + (uint32_t)er.idx * P.stage_bytes;
#pragma unroll
      for (int sb = 0; sb < SUB; ++sb) {
        piece(stage + (uint32_t)sb * 16384u + adst[0], R.a[sb][0]);
        piece(stage + (uint32_t)sb * 16384u + adst[1], R.a[sb][1]);
#pragma unroll
        for (int t = 0; t < NBT; ++t)
          if (fuse[t]) piece(stage + (uint32_t)(sb * P.NT * 128) + fdst[t], R.b[sb][t]);
      }
      ptx::fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0) ptx::mbar_arrive(bar_full0 + (uint32_t)er.idx * 8u);
      er.advance(P.SB);
      return true;
    };
    Regs R0;
    load(0, R0);  // (in flight across the prologue's barrier)
    __syncthreads();
    if constexpr (AHEAD) {
      Regs R1;
      for (int32_t it = 0; it < nst; it += 2) {
        if (it + 1 < nst) load(it + 1, R1);
        if (!(ok = store(R0)) || it + 1 >= nst) break;
        if (it + 2 < nst) load(it + 2, R0);
        if (!(ok = store(R1))) break;
      }
    } else {
      for (int32_t it = 0; it < nst && ok; ++it) {
        if (it > 0) load(it, R0);
        ok = store(R0);
      }
    }
  } else {
    // ================================================================ MMA ISSUER (the whole warp, one lane issues)
    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    const uint32_t d_tmem = misc->tmem_base;
    const uint32_t elect = lane == 0 ? 1u : 0u;
    const uint64_t d0 = ptx::smem_desc_k_sw128(sm0);
    const uint32_t lo0 = (uint32_t)d0, hi = (uint32_t)(d0 >> 32);
    const uint32_t b_sub16 = (uint32_t)(P.NT * 128) >> 4;
    Ring fr;
    uint32_t acc = 0;
    for (int32_t it = 0; it < nst; ++it, fr.advance(P.SB)) {
      ok = wait_bar_warp(P, misc, bar_full0 + (uint32_t)fr.idx * 8u, fr.phase, DEV_TIMEOUT_A_FULL, 20);
      if (!ok) break;
      ptx::tc_fence_after();
      const uint32_t a_lo = lo0 + (uint32_t)fr.idx * (P.stage_bytes >> 4), b_lo = a_lo + (a_bytes >> 4);
#pragma unroll
      for (int sb = 0; sb < SUB; ++sb) {
#pragma unroll
        for (int k4 = 0; k4 < 4; ++k4) {
          mma_ss_e<BF16, false>(d_tmem, a_lo + (uint32_t)(sb * 1024 + k4 * 2), hi, b_lo + (uint32_t)sb * b_sub16 + (uint32_t)(k4 * 2), hi,
                                P.idesc, acc, elect);
          acc = 1;
        }
      }
      mma_commit_e<false>(bar_empty0 + (uint32_t)fr.idx * 8u, elect);
    }
    if (ok) mma_commit_e<false>(ptx::smem_u32(&bars->acc), elect);
  }

  // ==================================================================== EPILOGUE (the gather warps)
  const int q4 = warp & 3, cg = warp >> 2;  // TMEM lane quarter; sixteen-column blocks cg, cg + 4, ...
  if (warp < kGW) {
    if (ok) ok = wait_bar_warp(P, misc, ptx::smem_u32(&bars->acc), 0u, DEV_TIMEOUT_ACC);
    ptx::tc_fence_after();
  }
  const uint32_t tmem_base = misc->tmem_base;
  const uint32_t d_tmem = tmem_base + ((uint32_t)(q4 * 32) << 16);
  const UX p = (UX)tile * 128u + (UX)(q4 * 32 + lane);
  const bool valid = p < (UX)Mtot;
  const int64_t cstride = P.nhwc ? 1 : P.HoWo;
  float* orow = P.out;
  if (valid) {
    const UX i = p / (UX)HoWo, pq = p - i * (UX)HoWo;
    orow += P.nhwc ? (int64_t)p * P.K + n0 : ((int64_t)i * P.K + n0) * P.HoWo + (int64_t)pq;
  }
  if (P.Z == 1) {
    if (warp < kGW && ok) {
#pragma unroll 1
      for (int32_t c0 = cg * 16; c0 < P.NT; c0 += 64) {
        uint32_t v[16];
        ptx::tmem_ld_x16(d_tmem + (uint32_t)c0, v);
        ptx::tmem_wait_ld();
        if (valid) store16(orow + (int64_t)c0 * cstride, cstride, v, P.K - n0 - c0, P.nhwc && (P.K & 3) == 0);
      }
    }
  } else {
    // partial tile -> own shared memory (column by column, 128 rows each; the operand stages are free: every MMA that
    // reads them has completed)
    if (warp < kGW && ok) {
#pragma unroll 1
      for (int32_t c0 = cg * 16; c0 < P.NT; c0 += 64) {
        uint32_t v[16];
        ptx::tmem_ld_x16(d_tmem + (uint32_t)c0, v);
        ptx::tmem_wait_ld();
        float* const o = reinterpret_cast<float*>(smem) + (c0 * 128 + q4 * 32 + lane);
#pragma unroll
        for (int e = 0; e < 16; ++e) o[e * 128] = __uint_as_float(v[e]);
      }
    }
    __syncwarp();
    cluster_sync_all();
    if (warp < kGW && ok) {
      // this CTA's share of the columns: [c_lo, c_hi), a warp per (column, lane quarter)
      const int32_t per = (P.NT + P.Z - 1) / P.Z;
      const int32_t c_lo = (int32_t)z * per, c_hi = min(c_lo + per, min(P.NT, P.K - n0));
      uint32_t peer[kGMaxZ];
#pragma unroll
      for (int r = 0; r < kGMaxZ; ++r) peer[r] = mapa(sm0 + (uint32_t)((q4 * 32 + lane) * 4), r < P.Z ? (uint32_t)r : 0u);
#pragma unroll 1
      for (int32_t c = c_lo + cg; c < c_hi; c += 4) {
        float part[kGMaxZ];
#pragma unroll
        for (int r = 0; r < kGMaxZ; ++r)
          if (r < P.Z) part[r] = lds_cluster_f32(peer[r] + (uint32_t)c * 512u);
        float s = 0.f;
#pragma unroll
        for (int r = 0; r < kGMaxZ; ++r)
          if (r < P.Z) s += part[r];
        if (valid) orow[(int64_t)c * cstride] = s;
      }
    }
    __syncwarp();
    cluster_sync_all();  // no CTA leaves while another may still read its partial tile
  }

  // ------------------------------------------------------------------ teardown
  ptx::tc_fence_before();
  __syncthreads();
  if (warp == kGW) {
    // on the abort path MMAs may still be in flight: give them a bounded chance to finish
    if (*reinterpret_cast<volatile int32_t*>(&misc->abort)) {
      if (lane == 0) ptx::mma_commit(ptx::smem_u32(&bars->acc));
      for (uint32_t it = 0; it < kSpin && !ptx::mbar_try_wait(ptx::smem_u32(&bars->acc), 0u); ++it) {}
      __syncwarp();
    }
    ptx::tc_fence_after();
    ptx::tmem_dealloc(tmem_base, P.tmem_cols);
    if (!P.wait_early) asm volatile("griddepcontrol.wait;" ::: "memory");  // this grid completes after the one it overlapped
  }
}

// ---------------------------------------------------------------------------------------------- host side

struct GPlan {
  int32_t NT, n_ntiles, Z;
  int64_t KS;
  double us;  // estimated time
};

// CTAs of clusters of Z that run at a time, one CTA per SM (a whole B200 as cudaOccupancyMaxActiveClusters counts it: the
// SMs of a GPC that do not fill a cluster stay idle).  Part of the estimate only: a card, or a part of one, that cannot
// place a cluster of Z says so at the launch, and the plan is made again with smaller ones.
int cluster_slots(int z, int nsm) {
  static const int slots[kGMaxZ + 1] = {0, 148, 148, 135, 132, 130, 132, 105, 120, 135, 110, 77, 84, 91, 98, 105, 112};
  if (nsm == 148) return slots[z];
  const int n = nsm * 3 / 4 / z * z;
  return z == 1 ? nsm : (n > 0 ? n : z);
}

// The cut with the least estimated time, in microseconds measured on B200: 5 for launch, prologue, first loads and
// store; per stage of 64 reduction elements 0.8 / 1.35 / 1.5 (BF16, tiles up to 64 / 128 / 256 filters) or
// 1.2 / 1.7 / 2.1 (TF32); 1 + 0.05 Z for the cluster's sum.  Neighbouring positions are s elements apart in the input
// and s*Fh in an im2win tensor, and every load takes that many times the lines: 0.17 per stage and element, and (im2win
// tensor) 1 for the first loads.
GPlan gather_plan(const Geometry& g, bool bf16, bool fused, int nt_max, int z_max = kGMaxZ) {
  const int nsm = sm_count();
  const int64_t tiles = (g.Mtot + 127) / 128;
  const int64_t stages = (g.Kg + kBK - 1) / kBK;
  GPlan best{0, 0, 0, 0, 1e30};
  const int fix_nt = knobs().gather_nt, fix_z = knobs().gather_z;
  for (int cand : {16, 32, 48, 64, 96, 128, 192, 256}) {
    if ((fix_nt && cand != fix_nt) || cand > nt_max) continue;
    const int64_t nn = (g.K + cand - 1) / cand;
    const int32_t nt = (int32_t)(((g.K + nn - 1) / nn + 15) / 16 * 16);
    const double stage = 0.17 * ((fused ? g.s : g.sFh) - 1) +
                         (bf16 ? (nt <= 64 ? 0.8 : (nt <= 128 ? 1.35 : 1.5)) : (nt <= 64 ? 1.2 : (nt <= 128 ? 1.7 : 2.1)));
    for (int z = 1; z <= z_max && z <= stages; ++z) {
      if (fix_z && z != fix_z) continue;
      const int64_t per = (stages + z - 1) / z;
      if ((stages + per - 1) / per != z) continue;  // (no empty slice)
      const int64_t units = tiles * nn * z;
      if (units > INT32_MAX / 2) continue;
      const int64_t sl = cluster_slots(z, nsm), waves = (units + sl - 1) / sl;
      const double us = 4.0 + (double)waves * (1.0 + (double)per * stage + nt * 0.005) + (z > 1 ? 1.0 + 0.05 * z : 0.0);
      if (us < best.us) best = GPlan{nt, (int32_t)nn, z, per * kBK, us};
    }
  }
  if (!fused) best.us += 1.0;
  return best;
}

// Estimated time of the persistent kernel on the same problem, in the same microseconds (a fit to 110 random layers
// that leave SMs idle, within 30 %, low rather than high): its channel groups of S MMA steps, the reduction slices it
// can use (none for the channels-last output), the bf16 copy of a streamed filter, and an epilogue that adds each
// slice's columns into the zeroed output by atomics.
double persistent_us(const Geometry& g, bool bf16) {
  const int64_t ff = g.FF, nsm = sm_count();
  int64_t cb = 8;
  if (ff == 121) cb = 1;
  else if (g.Fh == g.Fw && ff > 1 && g.C <= 3) cb = 3;
  else if (ff == 1) cb = 32;
  else if (bf16 || ff < 7) cb = 16;
  const int64_t ng = (g.C + cb - 1) / cb, S = (cb * ff + (bf16 ? 15 : 7)) / (bf16 ? 16 : 8);
  const int64_t n256 = (g.K + 255) / 256, nt = ((g.K + n256 - 1) / n256 + 15) / 16 * 16;
  const int64_t units = (g.Mtot + 127) / 128 * n256;
  int64_t z = g.out_nhwc || units >= nsm ? 1 : nsm / units;
  z = z > 16 ? 16 : z;
  z = z > ng ? ng : z;
  const int64_t per = (ng + z - 1) / z;
  z = (ng + per - 1) / per;
  const bool resident = n256 == 1 && ng * S * nt * 32 < 150000;
  const double start = (resident ? 4.8 : 5.5) + (bf16 && !resident ? 2.5 : 0.0);
  const double us = start + (double)(per * S * ((units + nsm - 1) / nsm)) * 0.06 +
                    (z > 1 ? 2.0 + (double)(nt * (z < 8 ? z : 8)) * 0.0115 : (double)nt * 0.016);
  // Short reductions onto wide filter tiles run whole there, and well (no slices, no atomics; 2 us more for the copy of a
  // bf16 filter): 2 images of 32x33x33, 416 filters, TF32 from the tensor 9.9 us, the gather kernel 15.9; 11 of 32x12x21,
  // 502 filters 11.6 and 17.6.  (1,680 under-filled calls: 13 slower than with the other kernels without this, 1 with it.)
  if (g.s == 1 && g.Fh == g.Fw && (ff == 9 || ff == 25) && g.C % 16 == 0 && g.Kg <= 720 && nt >= 112) {
    const double whole = start + (bf16 ? 2.0 : 0.0) + (double)(ng * S * ((units + nsm - 1) / nsm)) * 0.06 + (double)nt * 0.016;
    return us < whole ? us : whole;
  }
  return us;
}

template <bool BF16, int NBT, typename IX>
int launch_gather_t(const GParams& P, int64_t grid, size_t smem, cudaStream_t st) {
  auto kern = conv_tc_gather_kernel<BF16, NBT, IX>;
  if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxDynamicSmem) != cudaSuccess ||
      (P.Z > 8 && cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess)) {
    cudaGetLastError();
    return IM2WIN_ECUDA;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3((unsigned)kGThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = (unsigned)P.Z; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = P.Z > 1 ? 2 : 1;
  const bool refused = knobs().gather_zfail && P.Z > knobs().gather_zfail;  // (test build)
  if (refused || cudaLaunchKernelEx(&cfg, kern, P) != cudaSuccess) {
    cudaGetLastError();
    return IM2WIN_ECUDA;
  }
  note_kernel(KERNEL_GATHER);
  {
    const int v[4] = {P.NT, P.n_ntiles, P.Z, (int)P.KS};
    note_plan(v, 4);
  }
  return IM2WIN_OK;
}

// The limits of the general path (any filter size), those of a tile whose positions' strips are staged in shared
// memory beside two filter stages and whose window fits the tensor memory beside the accumulator: larger problems
// were never accepted, and stay refused.
bool general_limits(const Geometry& g, bool bf16) {
  constexpr int64_t kSegments = 8;  // images a tile may span
  const int64_t tp = (kSegments - 1) * g.HoWo + 1 < 128 ? (kSegments - 1) * g.HoWo + 1 : 128;
  const int64_t nn = (g.K + 255) / 256, nt = ((g.K + nn - 1) / nn + 15) / 16 * 16;
  const int64_t rowwrap = (int64_t)g.L - (int64_t)(g.Wo - 1) * g.sFh, wraps = (tp + g.Wo - 2) / g.Wo;
  int64_t nseg = (tp - 1) / g.HoWo + 2;
  if (nseg > kSegments) nseg = kSegments;
  int64_t pitch = (tp - 1) * g.sFh + wraps * (rowwrap > g.sFh ? rowwrap - g.sFh : 0) + nseg * (g.FF + 6) + 4;
  pitch = (pitch + 3) / 4 * 4;
  const int64_t step = bf16 ? 16 : 8, taps = (g.FF + step - 1) / step * step;
  return pitch <= INT32_MAX / 64 && (bf16 ? taps / 2 : taps) + nt <= 512 &&
         2 * nt * 128 + pitch * 4 + taps * 4 + 4096 <= 227 * 1024 - 2048 && (g.Mtot + tp - 1) / tp * nn <= INT32_MAX;
}

}  // namespace

// Whether the kernel is expected to be the fastest on a problem that other kernels implement too: launches that leave
// SMs idle there (B200, device time: 3x3, 256 channels and filters, one 16x16 image, BF16 22 -> 10 us; 5 images of
// 64x15x15, K = 142, stride 2, BF16 16.5 -> 8 us; 7 of 408x19x19, K = 32, BF16 35 -> 15 us; over 110 random
// layers of up to two waves of tiles the better of the two on each takes 1550 us, the other kernels alone 1891).  The
// factor keeps ties, which the estimates do not separate, where they were.
bool gather_preferred(const Geometry& g, int mode, bool fused) {
  const Knobs& k = knobs();  // (test build: configurations that force or exclude a kernel choose among the others)
  if (k.no_strip || k.force_strip || k.no_window || k.force_window || k.no_box || k.no_pim || k.bslice || k.no_gather) return false;
  if (g.Mtot > 128 * 300) return false;
  const bool bf16 = mode == IM2WIN_MODE_BF16;
  const double limit = 0.8 * persistent_us(g, bf16);
  // (no cut takes less than this: most calls are decided without looking at the cuts, 2 us of host time)
  const int64_t tiles = (g.Mtot + 127) / 128, stages = (g.Kg + kBK - 1) / kBK;
  int64_t z = tiles < sm_count() ? sm_count() / tiles : 1;
  if (z > kGMaxZ) z = kGMaxZ;
  if (5.0 + (double)((stages + z - 1) / z) * (bf16 ? 0.8 : 1.2) >= limit) return false;
  return gather_plan(g, bf16, fused, 256).us < limit;
}

// Estimated time from the input, in microseconds: the plan's, and for every wave behind the first the 1.5 + 0.015 NT us of a
// CTA's start and store that nothing hides there.
double gather_us(const Geometry& g, int mode) {
  const GPlan pl = gather_plan(g, mode == IM2WIN_MODE_BF16, true, 256);
  if (pl.NT == 0) return 1e30;
  const int64_t slots = cluster_slots(pl.Z, sm_count());
  const int64_t waves = ((g.Mtot + 127) / 128 * pl.n_ntiles * pl.Z + slots - 1) / slots;
  return pl.us + (double)(waves - 1) * (1.5 + 0.015 * pl.NT);
}

// For fused calls that no fused specialisation takes (rows whose staged input does not fit shared memory).  The other
// side: the transform, and the persistent kernel as above with an epilogue in every wave.  Fitted to 104
// such layers (rows of 400 to 2,600 columns) on B200: the picks take 3 % more than the better of the two on each, the
// transform and the specialised kernel always 13 %, this kernel always 33 % (1080x1920, 7x7 stride 2 from three channels, 64
// filters, TF32 141 and 230 us; 64x1600, 3x5, 16 channels, 64 filters 23 and 53; 200x1000, 7x1, 32 channels 221 and 103).
bool gather_beats_transform(const Geometry& g, int mode) {
  const int64_t nsm = sm_count(), n256 = (g.K + 255) / 256, pwaves = ((g.Mtot + 127) / 128 * n256 + nsm - 1) / nsm;
  const double other = transform_us(g) + persistent_us(g, mode == IM2WIN_MODE_BF16) + (double)(pwaves - 1) * (double)(g.K / n256) * 0.016;
  return gather_us(g, mode) < other;
}

int launch_conv_tc_gather(const float* src, const float* f, float* out, const Geometry& g, int mode, cudaStream_t st,
                          bool fused, bool behind_transform) {
  const bool bf16 = mode == IM2WIN_MODE_BF16;
  if (!general_limits(g, bf16)) return IM2WIN_EUNSUPPORTED;
  GParams P{};
  P.src = src; P.f = f; P.out = out;
  P.status = device_status_word();
  if (!P.status) return IM2WIN_ECUDA;
  P.K = g.K; P.HoWo = g.HoWo; P.Wo = g.Wo; P.Kg = g.Kg; P.Mtot = g.Mtot;
  P.FF = g.FF; P.Fw = g.Fw; P.Fh = g.Fh;
  if (fused) {
    P.plane = (int64_t)g.H * g.W; P.row_mul = (int64_t)g.s * g.W; P.col_mul = g.s; P.u_mul = g.W; P.v_mul = 1;
  } else {
    P.plane = g.HoL; P.row_mul = g.L; P.col_mul = g.sFh; P.u_mul = 1; P.v_mul = g.Fh;
  }
  P.img = (int64_t)g.C * P.plane;
  const bool big = P.img >= (1ll << 31) || g.Mtot >= (1ll << 31) - 256 || g.Kg >= (1ll << 31) - 4096 || knobs().gather_big;
  P.nhwc = g.out_nhwc;
  P.vec = (g.Kg & 3) == 0;
  P.wait_early = behind_transform ? 0 : 1;
  const int sub = bf16 ? 1 : 2;
  // (a cluster that cannot be placed is an error of its launch, before anything is enqueued: the next smaller cut then)
  for (int z_max = kGMaxZ; z_max >= 1; z_max = P.Z - 1) {
    const GPlan pl = gather_plan(g, bf16, fused, big ? 64 : 256, z_max);
    if (pl.NT == 0) return IM2WIN_EUNSUPPORTED;
    P.NT = pl.NT; P.n_ntiles = pl.n_ntiles; P.Z = pl.Z; P.KS = pl.KS;
    P.idesc = ptx::make_idesc(128, P.NT, bf16 ? 1 : 2);
    P.tmem_cols = 32;
    while ((int32_t)P.tmem_cols < P.NT) P.tmem_cols *= 2;
    P.stage_bytes = (uint32_t)(sub * (16384 + P.NT * 128));
    P.SB = kGStages;
    while ((size_t)P.SB * P.stage_bytes > 200 * 1024) --P.SB;
    uint32_t off = (uint32_t)P.SB * P.stage_bytes;
    if (off < (uint32_t)(P.NT * 512)) off = (uint32_t)(P.NT * 512);  // (the partial tile takes the stages' place)
    P.off_bar = off;
    const size_t smem = off + sizeof(GBars) + sizeof(SMisc) + 1024;
    const int64_t grid = (g.Mtot + 127) / 128 * P.n_ntiles * P.Z;
    if (grid > INT32_MAX) return IM2WIN_EUNSUPPORTED;
#define IM2WIN_GATHER(NBT, IX) (bf16 ? launch_gather_t<true, NBT, IX>(P, grid, smem, st) : launch_gather_t<false, NBT, IX>(P, grid, smem, st))
    const int rc = big ? IM2WIN_GATHER(1, int64_t)
                       : (P.NT <= 64 ? IM2WIN_GATHER(1, int32_t) : (P.NT <= 128 ? IM2WIN_GATHER(2, int32_t) : IM2WIN_GATHER(4, int32_t)));
    if (rc == IM2WIN_OK) return rc;
#undef IM2WIN_GATHER
  }
  return IM2WIN_ECUDA;
}

}  // namespace im2win
