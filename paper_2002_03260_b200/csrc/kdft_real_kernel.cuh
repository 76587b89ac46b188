// One KDFT axis with nodes (or a length without a folded form) and fp16 pieces, as a product with a REAL matrix.
//
// Take frequencies about their centre: k = c +- k', c = (N-1)/2, k' = p + 1/2, p < N/2 (N even).  With nodes t_j on the input,
//     y[c +- k'] = sum_j exp(s*2*pi*i*(c +- k')*t_j) x_j = C_p +- s*i*S_p,
//     C_p = sum_j cos(2*pi*k'*t_j) z_j,  S_p = sum_j sin(2*pi*k'*t_j) z_j,  z_j = exp(s*2*pi*i*c*t_j) x_j:
// one real N x N matrix acts on the real and on the imaginary parts alike: half the multiplications of the complex
// matrix and half its table.  Two forms:
//   FORM 1 (nodes on the input; solve for nodes on the output): z = phase * x, D = R z, y[c +- k'] = C +- s*i*S.
//   FORM 2 (nodes on the output; solve for nodes on the input): u_p = x[c+k'] + x[c-k'], v_p = s*i*(x[c+k'] - x[c-k']),
//          y_k = phase_k * (R [u; v])_k.
// A lane of the tile is the real or the imaginary part of a line (lanes 2l and 2l+1: line l of the tile's 64); the phase and
// the pair sums are taken while the data is split, the recombination of the two lanes while it is stored (one exchange
// per output value).
//
// Pipeline as in kdft_kernel.cuh: TMA producer, split warps that write the operand to tensor memory, one MMA issuer,
// eight epilogue warps that cut the accumulation chain every `chunk_kb` stages.  The raw data of a stage (64 reals of the
// contraction) arrives as halves with a barrier pair of their own.
//
// Bound: the instructions of the split and epilogue warps (tensor pipe a third busy at 256 points).  Nodes on all axes of 256^3,
// the reduction included: 405-414 us with the complex matrix; in this form 246 us back to back on one input and 271 us on
// changing inputs (nodes on the output 259 us); a pass 100 to 127 -> 68 us.  Two table stages and five half stages of raw data
// against three and two: 281 and 287 us before the epilogue was shortened.
#pragma once
#include "kdft_f16_kernel.cuh"

namespace dft3d {

constexpr int kRealLines = 64;                             // lines per tile
constexpr int kRealStagesB = 2;                            // table stages in shared memory
constexpr int kRealHalves = 5;                             // half stages of raw data in shared memory
constexpr int kRealBytesHalf = kF16BytesStageA / 2;
constexpr int kRealPhaseBytes = 2 * 32 * 8;                // FORM 1: phases of a half, one set per lane kind
constexpr size_t kKdftRealSmemBytes =
    size_t(kRealStagesB) * kBytesStageB + size_t(kRealHalves) * (kRealBytesHalf + kRealPhaseBytes) + 1024 + 512;

// FORM 1: the powers of two in the three sets of phases (ordinary data, data near the top and near the bottom of the range)
constexpr int kRealPhaseSets = 3;
__host__ __device__ constexpr int real_phase_up(int set) { return set == 1 ? -32 : (set == 2 ? 64 : 0); }

struct KdftRealParams {
  int n, bn, n_tiles, chunk_kb;         // table columns per tile; chunk_kb counts 64-real stages
  long long m_tiles, rows, batches, C;
  int lpb, bpt;                         // lines of one batch in a tile, batches per tile
  long long c_tiles;
  const float* phase;                   // FORM 1: [kRealPhaseSets][lane kind][n padded to 64] pairs (a, b): z = re*a + im*b;
                                        // FORM 2: (re, im) per k
  int phase_pitch;                      // FORM 1: n padded to 64
  float sign;
  float* out;
  unsigned int* status;
  float out_mul;
  const unsigned int* amax_in;
  unsigned int* amax_out;
  WaitControl wc;
};

struct KdftRealShared {
  uint64_t b_full[kRealStagesB], b_empty[kRealStagesB];
  uint64_t a_full[kRealHalves], a_empty[kRealHalves];
  uint64_t t_full[kStagesT], t_empty[kStagesT];
  uint64_t acc_full, acc_empty;
  uint32_t tmem_base;
  volatile int abort_flag;
  long long wait_limit;
};

// single-thread wait (producer, MMA issuer)
#define DFT3D_WAIT(bar, parity, code)                               \
  if (!bounded_wait((bar), (parity), &sh.abort_flag, sh.wait_limit)) {             \
    sh.abort_flag = 1;                                              \
    atomicCAS(p.status, 0u, (unsigned)(code));                      \
    goto role_done;                                                 \
  }
// whole-warp wait: the warp leaves together, so the .sync.aligned tensor-memory
// instructions that follow are never executed by a partial warp
#define DFT3D_WAIT_WARP(bar, parity, code)                                              \
  if (!__all_sync(0xffffffffu, bounded_wait((bar), (parity), &sh.abort_flag, sh.wait_limit) ? 1 : 0)) { \
    sh.abort_flag = 1;                                                                  \
    atomicCAS(p.status, 0u, (unsigned)(code));                                          \
    goto role_done;                                                                     \
  }

template <int MODE, int FORM>
__global__ void __launch_bounds__(kKdftThreads, 1)
kdft_real_axis_kernel(const __grid_constant__ CUtensorMap map_data, const __grid_constant__ CUtensorMap map_w,
                      const KdftRealParams p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = ptx::align_1024(smem_raw);
  uint8_t* smem_b = smem;
  uint8_t* smem_a = smem + size_t(kRealStagesB) * kBytesStageB;
  uint8_t* smem_ph = smem_a + size_t(kRealHalves) * kRealBytesHalf;   // [half][lane kind][32] pairs of floats
  KdftRealShared& sh = *reinterpret_cast<KdftRealShared*>(smem_ph + kRealHalves * kRealPhaseBytes);

  const int tid = threadIdx.x;
  const int warp = tid >> 5;
  const int lane = tid & 31;

  ptx::griddep_launch();
  if (tid == 0) {
    for (int i = 0; i < kRealStagesB; ++i) { ptx::mbar_init(&sh.b_full[i], 1); ptx::mbar_init(&sh.b_empty[i], 1); }
    for (int i = 0; i < kRealHalves; ++i) { ptx::mbar_init(&sh.a_full[i], 1); ptx::mbar_init(&sh.a_empty[i], 4); }
    for (int i = 0; i < kStagesT; ++i) { ptx::mbar_init(&sh.t_full[i], 4); ptx::mbar_init(&sh.t_empty[i], 1); }
    ptx::mbar_init(&sh.acc_full, 1);
    ptx::mbar_init(&sh.acc_empty, kEpilogueWarps);
    sh.abort_flag = 0;
    sh.wait_limit = p.wc.limit_clocks > 0 ? p.wc.limit_clocks : kDefaultWaitClocks;
    ptx::fence_mbar_init();
  }
  if (warp == 1) {
    ptx::tmem_alloc(&sh.tmem_base, kTmemCols);
    ptx::tmem_relinquish();
  }
  if (warp == 0 && lane == 0) {
    ptx::prefetch_tensormap(&map_data);
    ptx::prefetch_tensormap(&map_w);
  }
  ptx::griddep_wait();
  ptx::tc_fence_before();
  __syncthreads();
  ptx::tc_fence_after();
  const uint32_t tmem = sh.tmem_base;

  const long long total_tiles = p.m_tiles * p.n_tiles;
  const int num_kb = (p.n + kF16BlockK - 1) / kF16BlockK;   // a ragged last stage is zero-filled by TMA on both operands
  const uint32_t bytes_b = 2u * uint32_t(p.bn) * 128u;            // two pieces, bn rows of 64 halves

  // power-of-two scale that brings the largest input magnitude into [2^13, 2^14): fp16 pieces then neither
  // overflow nor lose more than fp16's own subnormal floor (2^-25 of a scaled unit) on small entries
  // FORM 1 multiplies by the phase before it scales.  Data near either end of the float range takes phases that bring it
  // towards the middle (`up`: powers of two, tables of their own), so that neither the two products overflow together
  // nor their bits fall below the subnormal numbers.
  float in_scale = 1.0f, out_mul1 = p.out_mul, out_mul2 = 1.0f;
  const float* phase = p.phase;
  {
    const float a = __uint_as_float(*p.amax_in);
    if (a > 0.0f) {                      // never an infinity: the reduction and the epilogues leave those out
      // FORM 2: below 2^-113 the scale stops growing (2^126 is the largest power of two that is safe to multiply by);
      // nothing is lost: the sums of such data are multiples of 2^-149, i.e. of 2^-23 after scaling, which the two pieces hold
      const int e = FORM == 1 ? ilogbf(a) : max(ilogbf(a), -113);
      int up = 0;
      if (FORM == 1 && e > 100) { up = real_phase_up(1); phase += 4 * p.phase_pitch; }
      if (FORM == 1 && e < -60) { up = real_phase_up(2); phase += 8 * p.phase_pitch; }
      in_scale = ldexpf(1.0f, 13 - e - up);
      out_mul1 = ldexpf(p.out_mul, -up);
      out_mul2 = ldexpf(1.0f, e - 13 + up);
    }
  }

  if (warp < 4) {
    // warp group 0: producer and MMA issuer need few registers; hand the rest to the epilogue
    ptx::setmaxnreg_dec<DFT3D_REGS_WG0>();
    if (warp == 0) {
      // ------------------------------------------------------------ TMA producer
      if (lane == 0 && !p.wc.silent_producer) {
        uint32_t ib = 0, ia = 0;   // running stage counters
        for (long long t = blockIdx.x; t < total_tiles; t += gridDim.x) {
          const long long mt = t / p.n_tiles;
          const int nt = int(t % p.n_tiles);
          int ax = 0, ay = 0, az = 0;
          if (MODE == KDFT_CONTIG) {
            ay = int(mt * kRealLines);
          } else {
            const long long ct = mt % p.c_tiles;
            const long long bt = mt / p.c_tiles;
            ax = int(ct * p.lpb * 2);
            az = int(bt * p.bpt);
          }
          for (int kb = 0; kb < num_kb; ++kb) {
            {
              const uint32_t s = ib % kRealStagesB, ph = (ib / kRealStagesB) & 1;
              DFT3D_WAIT(&sh.b_empty[s], ph ^ 1, 0x101);
              ptx::mbar_arrive_expect_tx(&sh.b_full[s], bytes_b);
              ptx::tma_load_3d(smem_b + size_t(s) * kBytesStageB, &map_w, &sh.b_full[s], kb * kF16BlockK, nt * p.bn, 0);
              ++ib;
            }
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              const uint32_t s = ia % kRealHalves, ph = (ia / kRealHalves) & 1;
              DFT3D_WAIT(&sh.a_empty[s], ph ^ 1, 0x102);
              ptx::mbar_arrive_expect_tx(&sh.a_full[s], kRealBytesHalf + (FORM == 1 ? kRealPhaseBytes : 0));
              uint8_t* dst = smem_a + size_t(s) * kRealBytesHalf;
              if (FORM == 1) {             // 32 points of 64 lines and their phases
                const int j0 = kb * kF16BlockK + 32 * h;
                if (MODE == KDFT_CONTIG) {
                  ptx::tma_load_2d(dst, &map_data, &sh.a_full[s], 2 * j0, ay);
                  ptx::tma_load_2d(dst + kRealBytesHalf / 2, &map_data, &sh.a_full[s], 2 * j0 + 32, ay);
                } else {
                  ptx::tma_load_3d(dst, &map_data, &sh.a_full[s], ax, j0, az);
                }
                for (int c = 0; c < 2; ++c)
                  ptx::bulk_load(smem_ph + s * kRealPhaseBytes + c * (kRealPhaseBytes / 2),
                                 phase + 2 * (size_t(c) * p.phase_pitch + j0), kRealPhaseBytes / 2, &sh.a_full[s]);
              } else {                     // 16 pairs: the points left of the centre, then those right of it
                const int p0 = kb * (kF16BlockK / 2) + 16 * h, left = p.n / 2 - 16 - p0, right = p.n / 2 + p0;
                if (MODE == KDFT_CONTIG) {
                  ptx::tma_load_2d(dst, &map_data, &sh.a_full[s], 2 * left, ay);
                  ptx::tma_load_2d(dst + kRealBytesHalf / 2, &map_data, &sh.a_full[s], 2 * right, ay);
                } else {
                  ptx::tma_load_3d(dst, &map_data, &sh.a_full[s], ax, left, az);
                  ptx::tma_load_3d(dst + kRealBytesHalf / 2, &map_data, &sh.a_full[s], ax, right, az);
                }
              }
              ++ia;
            }
          }
        }
      }
    } else if (warp == 1) {
      // ------------------------------------------------------------ MMA issuer
      if (lane == 0) {
        const uint32_t idesc = ptx::make_idesc_f16(kTileM, p.bn);
        uint32_t ib = 0, it = 0, chunk_count = 0;
        for (long long t = blockIdx.x; t < total_tiles; t += gridDim.x) {
          for (int kb = 0; kb < num_kb; ++kb) {
            const bool chunk_first = (kb % p.chunk_kb) == 0;
            if (chunk_first) {
              // the tensor-core accumulator restarts from zero every chunk (see the epilogue)
              DFT3D_WAIT(&sh.acc_empty, (chunk_count & 1) ^ 1, 0x201);
              ptx::tc_fence_after();
            }
            const uint32_t sb = ib % kRealStagesB, phb = (ib / kRealStagesB) & 1;
            const uint32_t st = it % kStagesT, pht = (it / kStagesT) & 1;
            DFT3D_WAIT(&sh.b_full[sb], phb, 0x202);
            DFT3D_WAIT(&sh.t_full[st], pht, 0x203);
            ptx::tc_fence_after();
            const uint32_t b_hi = ptx::smem_u32(smem_b + size_t(sb) * kBytesStageB);
            const uint32_t b_lo = b_hi + uint32_t(p.bn) * 128u;
            const uint32_t a_hi = tmem + kAccCols + st * 64;
            const uint32_t a_lo = a_hi + 32;
#pragma unroll
            for (int k = 0; k < kF16BlockK / 16; ++k) {   // K = 16 per MMA: 8 packed columns of A, 32 bytes of each B row
              const uint64_t dhi = ptx::make_kmajor_sw128_desc(b_hi + k * 32);
              const uint64_t dlo = ptx::make_kmajor_sw128_desc(b_lo + k * 32);
              ptx::mma_f16_ts(tmem, a_hi + k * 8, dhi, idesc, (k != 0 || !chunk_first) ? 1u : 0u);
              ptx::mma_f16_ts(tmem, a_lo + k * 8, dhi, idesc, 1);
              ptx::mma_f16_ts(tmem, a_hi + k * 8, dlo, idesc, 1);
            }
            ptx::tc_commit(&sh.b_empty[sb]);
            ptx::tc_commit(&sh.t_empty[st]);
            ++ib;
            ++it;
            if ((kb + 1) % p.chunk_kb == 0 || kb + 1 == num_kb) {
              ptx::tc_commit(&sh.acc_full);
              ++chunk_count;
            }
          }
        }
      }
    }
  } else if (warp < 8) {
    // ------------------------------------------------------------ split: smem -> (hi, lo) -> tensor memory
    ptx::setmaxnreg_dec<DFT3D_REGS_SPLIT>();
    const int q = warp & 3;                 // lane quarter this warp may touch in tensor memory
    const int m = q * 32 + lane;            // lane of the tile
    const uint32_t lane_addr = tmem + (uint32_t(q * 32) << 16);
    const int line = m >> 1, comp = m & 1;
    // STRIDED: complex index of this lane's line in row 0 of a box (FORM 1: 32 rows per half, FORM 2: two boxes of 16)
    const int col = MODE == KDFT_STRIDED ? (line / p.lpb) * (FORM == 1 ? 32 : 16) * p.lpb + line % p.lpb : 0;
    // FORM 2: s*i*d has the real part -s*Im d and the imaginary part s*Re d.  The real lane takes (Re u, -s*Im d) from (re, im) of
    // the two points, the imaginary lane (s*Re d, Im u).
    const float ds = comp ? p.sign * in_scale : -p.sign * in_scale;
    const uint64_t scale2 = FORM == 1 ? pack2(in_scale, in_scale) : (comp ? pack2(ds, in_scale) : pack2(in_scale, ds));
    const uint64_t scale_l = comp ? pack2(-ds, in_scale) : pack2(in_scale, -ds);
    const uint32_t order = comp ? 0x1032u : 0x3210u;
    uint32_t ia = 0, it = 0;
    for (long long t = blockIdx.x; t < total_tiles; t += gridDim.x) {
      for (int kb = 0; kb < num_kb; ++kb) {
        const uint32_t st = it % kStagesT, pht = (it / kStagesT) & 1;
        uint32_t ph[32], pl[32];                 // 64 scaled values as fp16 pairs: hi pieces, lo pieces
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const uint32_t sa = ia % kRealHalves, pha = (ia / kRealHalves) & 1;
          DFT3D_WAIT_WARP(&sh.a_full[sa], pha, 0x301);
          const uint8_t* stage = smem_a + size_t(sa) * kRealBytesHalf;
          // the pieces of this half's 32 operand values of the lane, two at a time
          if (FORM == 1) {
            const float4* phases = reinterpret_cast<const float4*>(smem_ph + sa * kRealPhaseBytes + comp * (kRealPhaseBytes / 2));
#pragma unroll
            for (int c = 0; c < 16; ++c) {         // points 2c and 2c+1
              float4 x;
              if (MODE == KDFT_CONTIG) {
                x = reinterpret_cast<const float4*>(stage + (c >> 3) * (kRealBytesHalf / 2) + line * 128)[(c & 7) ^ (line & 7)];
              } else {
                const float2* at = reinterpret_cast<const float2*>(stage) + col + 2 * c * p.lpb;
                const float2 x0 = at[0], x1 = at[p.lpb];
                x = make_float4(x0.x, x0.y, x1.x, x1.y);
              }
              const float4 f = phases[c];
              split_half2(mul2(pack2(fmaf(x.x, f.x, x.y * f.y), fmaf(x.z, f.z, x.w * f.w)), scale2), ph[h * 16 + c], pl[h * 16 + c]);
            }
          } else {
#pragma unroll
            for (int c = 0; c < 16; ++c) {         // pair c: point 15 - c of the left box, point c of the right one
              const uint8_t *l, *r;
              if (MODE == KDFT_CONTIG) {
                const uint8_t* row = stage + line * 128;
                l = row + ((((15 - c) >> 1) ^ (line & 7)) << 4) + ((15 - c) & 1) * 8;
                r = row + kRealBytesHalf / 2 + (((c >> 1) ^ (line & 7)) << 4) + (c & 1) * 8;
              } else {
                l = stage + 8 * (col + (15 - c) * p.lpb);
                r = stage + kRealBytesHalf / 2 + 8 * (col + c * p.lpb);
              }
              // (u, v), the other way round in the imaginary lane; scaled before they are added: a sum of two floats may be none.
              // Whole points in one load each (nodes on the output, 256^3: 259 us; with 4-byte loads in the lane's order 276 us)
              uint32_t hi, lo;
              split_half2(fma2(*reinterpret_cast<const uint64_t*>(l), scale_l, mul2(*reinterpret_cast<const uint64_t*>(r), scale2)), hi, lo);
              ph[h * 16 + c] = __byte_perm(hi, 0, order);
              pl[h * 16 + c] = __byte_perm(lo, 0, order);
            }
          }
          // the half is refilled by TMA (async proxy): order this thread's reads before that write
          ptx::fence_proxy_async_smem();
          __syncwarp();
          if (lane == 0) ptx::mbar_arrive(&sh.a_empty[sa]);
          ++ia;
        }
        DFT3D_WAIT_WARP(&sh.t_empty[st], pht ^ 1, 0x302);
        ptx::tc_fence_after();
        ptx::tmem_st_32x32(lane_addr + kAccCols + st * 64, ph);
        ptx::tmem_st_32x32(lane_addr + kAccCols + st * 64 + 32, pl);
        ptx::tc_wait_st();
        ptx::tc_fence_before();
        __syncwarp();
        if (lane == 0) ptx::mbar_arrive(&sh.t_full[st]);
        ++it;
      }
    }
  } else {
    // ------------------------------------------------------------ epilogue (8 warps)
    // The tensor core adds into its fp32 accumulator with truncation, a bias that grows with the
    // number of MMAs chained on one accumulator.  So the chain is cut every `chunk_kb` stages: the
    // partial sum is pulled into registers and summed there in round-to-nearest fp32, and the tensor
    // core restarts from zero.
    ptx::setmaxnreg_inc<DFT3D_REGS_EPI>();
    const int q = warp & 3;
    const int half = (warp - 8) >> 2;        // which 128 columns of the 256-wide accumulator
    const int m = q * 32 + lane;
    const int line = m >> 1, comp = m & 1;
    const float tau = comp ? 1.0f : -1.0f;   // i*w has the real part -Im w and the imaginary part Re w
    // One factor where neither a sum (below 2^38) nor its share in the recombination can leave the normal numbers, else
    // the table's (2^-10 and the like) before the recombination and the scale of the data after it: a result that is a float
    // is reached from either end of the range.
    const float both = out_mul1 * out_mul2;
    const bool one_step = both > 1e-26f && both < 1e26f;
    const float mul = one_step ? both : out_mul1, taum = tau * mul;
    const int width = ((p.bn + 1) / 2 + 31) / 32 * 32;       // columns of the first of the two halves, at most 128
    const uint32_t lane_addr = tmem + (uint32_t(q * 32) << 16) + half * width;
    const int chunks_per_tile = (num_kb + p.chunk_kb - 1) / p.chunk_kb;
    uint32_t chunk_count = 0;
    for (long long t = blockIdx.x; t < total_tiles; t += gridDim.x) {
      const long long mt = t / p.n_tiles;
      const int nt = int(t % p.n_tiles);
      const int c0 = nt * p.bn + half * width;   // first table column held by this thread
      const int ncols = min(half ? p.bn - width : width, p.n - c0);   // how many of them (none or negative: none)
      float acc[128];
      for (int c = 0; c < chunks_per_tile; ++c, ++chunk_count) {
        DFT3D_WAIT_WARP(&sh.acc_full, chunk_count & 1, 0x401);
        ptx::tc_fence_after();
#pragma unroll
        for (int g = 0; g < 4; ++g) {
          if (32 * g < ncols) {
            uint32_t v[32];
            ptx::tmem_ld_32x32(lane_addr + g * 32, v);
            ptx::tc_wait_ld();
            if (c == 0) {
#pragma unroll
              for (int i = 0; i < 32; ++i) acc[g * 32 + i] = __uint_as_float(v[i]);
            } else {
#pragma unroll
              for (int i = 0; i < 32; ++i) acc[g * 32 + i] += __uint_as_float(v[i]);
            }
          }
        }
        ptx::tc_fence_before();
        __syncwarp();
        if (lane == 0) ptx::mbar_arrive(&sh.acc_empty);
      }
      // ---- undo the scales, recombine the lanes of a line, note the largest magnitude for the next pass, store
      float amax = 0.0f;
      if (ncols > 0) {
        if (FORM == 1) {                       // columns (C_p, S_p) -> outputs N/2 + p and N/2 - 1 - p
          const float st = p.sign * taum;
#pragma unroll
          for (int i = 0; i < 64; ++i) {
            if (i / 16 * 32 >= ncols) break;
            const float other = __shfl_xor_sync(0xffffffffu, acc[2 * i + 1], 1), c = acc[2 * i] * mul;
            acc[2 * i] = fmaf(st, other, c);
            acc[2 * i + 1] = fmaf(-st, other, c);
          }
        } else {
          const float4* ph = reinterpret_cast<const float4*>(p.phase) + c0 / 2;   // padded to whole tiles
#pragma unroll
          for (int i = 0; i < 64; ++i) {
            if (i / 16 * 32 >= ncols) break;
            const float4 f = __ldg(ph + i);
            const float o0 = __shfl_xor_sync(0xffffffffu, acc[2 * i], 1), o1 = __shfl_xor_sync(0xffffffffu, acc[2 * i + 1], 1);
            acc[2 * i] = fmaf(acc[2 * i] * mul, f.x, o0 * taum * f.y);
            acc[2 * i + 1] = fmaf(acc[2 * i + 1] * mul, f.z, o1 * taum * f.w);
          }
        }
        if (!one_step) {
#pragma unroll
          for (int i = 0; i < 128; ++i) acc[i] *= out_mul2;
        }
        long long base, step = 1;              // complex index of the line's first point, distance of its points
        bool live;
        if (MODE == KDFT_CONTIG) {
          const long long row = mt * kRealLines + line;
          live = row < p.rows;
          base = row * p.n;
        } else {
          const long long batch = (mt / p.c_tiles) * p.bpt + line / p.lpb, cc = (mt % p.c_tiles) * p.lpb + line % p.lpb;
          live = batch < p.batches && cc < p.C;
          base = batch * p.n * p.C + cc;
          step = p.C;
        }
        if (MODE == KDFT_STRIDED) {
          if (live) {
            // FORM 1: two ends that move apart; FORM 2: neighbouring outputs
            const long long hop = 2 * step * (FORM == 1 ? 1 : 2);
            float* up = p.out + 2 * (base + (FORM == 1 ? p.n / 2 + c0 / 2 : c0) * step) + comp;
            float* down = p.out + 2 * (base + (FORM == 1 ? p.n / 2 - 1 - c0 / 2 : c0 + 1) * step) + comp;
            const int count = ncols / 2;
            if (count >= 64) {
#pragma unroll
              for (int i = 0; i < 64; ++i) {
                *up = acc[2 * i];
                *down = acc[2 * i + 1];
                amax = fmaxf(amax, fmaxf(fabsf(acc[2 * i]), fabsf(acc[2 * i + 1])));
                up += hop;
                down += FORM == 1 ? -hop : hop;
              }
            } else {
#pragma unroll
              for (int i = 0; i < 64; ++i)
                if (i < count) {
                  *up = acc[2 * i];
                  *down = acc[2 * i + 1];
                  amax = fmaxf(amax, fmaxf(fabsf(acc[2 * i]), fabsf(acc[2 * i + 1])));
                  up += hop;
                  down += FORM == 1 ? -hop : hop;
                }
            }
          }
        } else {
          // the two lanes of a line swap values so that each holds whole complex numbers: 16-byte stores
          float* dst = p.out + 2 * base;
#pragma unroll
          for (int g = 0; g < 16; ++g) {
            if (8 * g >= ncols) break;
#pragma unroll
            for (int side = 0; side < 2; ++side) {
              // four outputs in ascending order, own part of each: this lane keeps w[2*comp], w[2*comp+1]
              float w[4];
              int e;                            // index of the first of the four
              bool ok;
              if (FORM == 1) {
                const int p0 = c0 / 2 + 4 * g;
#pragma unroll
                for (int i = 0; i < 4; ++i) w[i] = side == 0 ? acc[2 * (4 * g + i)] : acc[2 * (4 * g + 3 - i) + 1];
                e = side == 0 ? p.n / 2 + p0 : p.n / 2 - 4 - p0;
                ok = side == 0 ? p0 + 2 * comp < (c0 + ncols) / 2 : p0 + 2 - 2 * comp < (c0 + ncols) / 2;
              } else {
#pragma unroll
                for (int i = 0; i < 4; ++i) w[i] = acc[8 * g + 4 * side + i];
                e = c0 + 8 * g + 4 * side;
                ok = e + 2 * comp < c0 + ncols;
              }
              const float r0 = __shfl_xor_sync(0xffffffffu, comp ? w[0] : w[2], 1);
              const float r1 = __shfl_xor_sync(0xffffffffu, comp ? w[1] : w[3], 1);
              if (live && ok) {
                *reinterpret_cast<float4*>(dst + 2 * (e + 2 * comp)) =
                    comp ? make_float4(r0, w[2], r1, w[3]) : make_float4(w[0], r0, w[1], r1);
                amax = fmaxf(amax, comp ? fmaxf(fmaxf(fabsf(r0), fabsf(w[2])), fmaxf(fabsf(r1), fabsf(w[3])))
                                        : fmaxf(fmaxf(fabsf(r0), fabsf(w[0])), fmaxf(fabsf(r1), fabsf(w[1]))));
              }
            }
          }
        }
        amax = finite_magnitude(amax);
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, o));
      if (lane == 0 && amax > 0.0f) atomicMax(p.amax_out, __float_as_uint(amax));
    }
  }

role_done:
  if (warp == 0 && lane == 0 && sh.abort_flag) {
    // give loads that were already issued a bounded chance to land before the CTA goes away
    const long long t0 = clock64();
    while (clock64() - t0 < 2000000LL) { }
  }
  ptx::tc_fence_before();
  __syncthreads();
  if (warp == 1) ptx::tmem_dealloc(tmem, kTmemCols);
}

#undef DFT3D_WAIT
#undef DFT3D_WAIT_WARP

}  // namespace dft3d
