// Chains of dependent symmetric products on the 5th-generation tensor cores: the whole
// Fermi-operator recursion of a pass (about 70 products of matrices of one to six 128-row tiles per
// subgraph) in one persistent launch.
//
// Tasks are (product, subgraph, upper 128x128 tile); a CTA takes every gridDim.x-th task.  Product k of a
// subgraph starts when product k - 1 of that subgraph is complete (a counter per subgraph, released by
// the epilogue warps and acquired by the producer), so subgraphs run through the recursion
// independently of each other.  The launch is cooperative: every CTA is resident, a task only waits for
// tasks before it in the common order, and every wait is bounded.
//
// Storage inside a chain: operands as split planes in the blocked layout of common.cuh, upper tiles only;
// FP32 masters (addends of later epilogues) in tile order: tile (tm, tn) is 64 KB at
// (tm * T + tn) * 64 KB, in which epilogue warp w's float4 j of lane l sits at ((w * 8 + j) * 32 + l) * 16.
// That is the order tcgen05.ld delivers the accumulators in (a lane holds a row), so masters move
// with coalesced 512-byte accesses and no transposition.
//
// What bounds it: a 128x128 tile with 512 inner columns takes 96 MMAs in the two-plane form (3.1 us at the tensor
// rate), 512 KB of operands into the SM (4 us at 64 bytes a cycle) and about 1.8 us of hand-over between the
// MMAs, the drain and the next tile, since the four accumulators fill TMEM; the epilogue (4 to 9 us with two
// addends) runs beside them.  Hence three full operand stages (192 KB; two and a half left the MMAs waiting 10%
// longer), sixteen epilogue warps, tiles handed over in shared memory, both operands of a diagonal tile of
// a square read once, and the K steps past the last valid column left out.  N = 256 instructions over [hi | lo]
// and collector reuse of A measured no gain.
// Measured (GB300): 281 subgraphs of about 506 orbitals, 60 products of ten doublings: 198 us a product (185
// TFLOP/s of n^3, a third of it per tensor product) against 276 us launched one by one with row-major
// masters; three planes 264 against about 430 us; three subgraphs of 192 orbitals 9.8 against 15 us.
#include "chain.cuh"

namespace sedacs {

namespace {

// Epilogue warps: four per TMEM lane quadrant (warp & 3), each with a quarter (warp >> 2) of the
// tile's columns; then one producer and one MMA warp.
constexpr int kEW = 16;
constexpr int kProdW = kEW, kMmaW = kEW + 1;
constexpr int kThreads = 32 * (kEW + 2);
constexpr int kSlabBytes = 4096;                    // 32 rows x 64 columns of one plane
constexpr int kReady = 16;                          // ring of tasks (more than can be in flight)

// Operand ring: a unit holds the planes of one operand's 128 x 64 block (32 or 48 KB), two units a k-block.  Slabs:
// for each of the eight warp pairs 4 KB, first the landing place of the leading addend columns, then the
// source of the planes' bulk stores.
template <int P>
struct Cfg {
  static constexpr int kUnits = P == 2 ? 6 : 4;
  static constexpr int kUnitBytes = P * kBlkBytes;
  static constexpr int kBars = kUnits / 2;          // k-blocks in the ring, each with a full and an empty barrier
  static constexpr int kSlabTotal = 8 * kSlabBytes;
  static constexpr int kPre = 2;       // float4 columns of each addend landing in the slabs
  static constexpr int kSmem = kUnits * kUnitBytes + kSlabTotal + 1024 + 1024;
};

// TMEM columns: hi * hi of k-block kb goes to accumulator kb % 3 (fewer rounding steps per accumulator),
// the corrections to the fourth.
constexpr uint32_t kCorr = 384;

__device__ __forceinline__ unsigned ld_acquire(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void red_release(unsigned* p, unsigned v) {
  asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async;" ::: "memory"); }
__device__ __forceinline__ void bulk_s2g(void* dst, const void* src, uint32_t bytes) {
  asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst), "r"(smem_u32(src)), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void bulk_prefetch(const void* src, uint32_t bytes) {
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

// 32 columns of this warp's 32 TMEM lanes; the caller waits (tcgen05.wait::ld).
__device__ __forceinline__ void tmem_ld32_nowait(uint32_t taddr, uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
      "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]),
        "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]),
        "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]),
        "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr)
      : "memory");
}
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// A task as the producer hands it to the other roles (shared memory, read after its ready barrier).
struct alignas(16) Task {
  long long el;
  int mat, op;
  short tm, tn;
  int n_pad, n_real, last;                          // last: 1 ends the sequence
};

// The task sequence of a CTA: windows of subgraphs one after the other, within a window product by
// product over its tiles.  The tile of the next task is loaded one task ahead.
struct Tasks {
  const ChainTile* tiles;
  const int* win;
  int n_win, n_ops, w, w0, wn, pos;
  int4 t0, t1;
  int next_op;                                      // -1: no further task
  __device__ __forceinline__ Tasks(const ChainParams& p)
      : tiles(p.tiles), win(p.win), n_win(p.n_win), n_ops(p.n_ops), w(0), w0(0), wn(0), pos((int)blockIdx.x) {
    window();
    fetch();
  }
  __device__ __forceinline__ void window() {
    if (w < n_win) {
      w0 = __ldg(win + w);
      wn = __ldg(win + w + 1) - w0;
    }
  }
  __device__ __forceinline__ void fetch() {
    while (w < n_win && pos >= wn * n_ops) {
      pos -= wn * n_ops;
      ++w;
      window();
    }
    next_op = -1;
    if (w >= n_win) return;
    next_op = pos / wn;
    const int4* t = reinterpret_cast<const int4*>(tiles + (w0 + pos - next_op * wn));
    t0 = __ldg(t);
    t1 = __ldg(t + 1);
    pos += (int)gridDim.x;
  }
  __device__ __forceinline__ Task task() const {
    Task t;
    t.el = (long long)(((unsigned long long)(unsigned)t0.y << 32) | (unsigned)t0.x);
    t.mat = t0.z;
    t.op = next_op;
    t.tm = (short)t0.w;
    t.tn = (short)t1.x;
    t.n_pad = t1.y;
    t.n_real = t1.z;
    t.last = next_op < 0;
    return t;
  }
};

// Four consecutive values as planes, two words of each plane at word i.
template <int P>
__device__ __forceinline__ void pack(const float (&x)[4], uint32_t (&d)[P][16], int i) {
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    float a = x[2 * h], b = x[2 * h + 1];
    if (P == 2) {
      const __half2 hi = __floats2half2_rn(a, b);
      const float2 f = __half22float2(hi);
      const __half2 lo = __floats2half2_rn((a - f.x) * kF16LoScale, (b - f.y) * kF16LoScale);
      d[0][i + h] = *reinterpret_cast<const uint32_t*>(&hi);
      d[1][i + h] = *reinterpret_cast<const uint32_t*>(&lo);
    } else {
#pragma unroll
      for (int pl = 0; pl < P; ++pl) {
        const __nv_bfloat162 y = __floats2bfloat162_rn(a, b);
        const float2 f = __bfloat1622float2(y);
        d[pl][i + h] = *reinterpret_cast<const uint32_t*>(&y);
        a -= f.x;
        b -= f.y;
      }
    }
  }
}

template <int P>
__global__ void __launch_bounds__(kThreads, 1) product_chain(const __grid_constant__ ChainParams p) {
  using C = Cfg<P>;
  if (*reinterpret_cast<volatile int*>(p.err) & kErrTimeout) return;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* slabs = smem + C::kUnits * C::kUnitBytes;
  uint64_t* full = reinterpret_cast<uint64_t*>(slabs + C::kSlabTotal);
  uint64_t* empty = full + C::kBars;
  uint64_t* accf = empty + C::kBars;
  uint64_t* acce = accf + 1;                        // drained: [0] accumulator 0 and corrections, [1], [2]
  uint64_t* ready = acce + 3;                       // the products before a task are complete
  uint64_t* addf = ready + kReady;                  // per warp pair: leading addend columns have landed
  uint64_t* pairb = addf + 8;                       // the two warps of a pair meet
  Task* tasks = reinterpret_cast<Task*>((reinterpret_cast<uintptr_t>(pairb + 8) + 15) & ~uintptr_t(15));
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(tasks + kReady);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    for (int s = 0; s < C::kBars; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    mbar_init(accf, 1);
    for (int j = 0; j < 3; ++j) mbar_init(&acce[j], kEW);
    for (int j = 0; j < kReady; ++j) mbar_init(&ready[j], 1);
    for (int j = 0; j < 8; ++j) {
      mbar_init(&addf[j], 1);
      mbar_init(&pairb[j], 2);
    }
    fence_mbar_init();
  }
  if (warp == 0) {
    tmem_alloc(tmem_slot, 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  bool ok = true;

  if (warp == kProdW) {
    // K-block k of the CTA's sequence has its operands in units 2k and 2k + 1 of the ring and barriers k % kBars.
    // Lane = plane * 2 + half copies its plane of each operand: one 16 KB block (half 0), or the two 8 KB halves
    // of a transposed one.
    const int pl = lane >> 1, half = lane & 1;
    const bool copies = lane < 2 * P;
    const long long my_plane = pl * p.plane;
    const int my_dst = pl * kBlkBytes + half * (kBlkBytes / 2);
    int k = 0, ti = 0;                                  // k-blocks filled, tasks begun
    Tasks ts(p);
    while (true) {
      const Task t = ts.task();
      const bool end = ts.next_op < 0;
      if (!end) ts.fetch();
      const int op = end ? 0 : t.op;
      const ChainOp& o = p.op[op];
      const int T = t.n_pad >> 7;
      if (op > 0) {
        if (lane == 0) {
          const unsigned target = (unsigned)(op * (T * (T + 1) / 2) * kEW);
          const long long t0 = clock64();
          while (ld_acquire(p.done + t.mat) < target)
            if (clock64() - t0 > kWaitLimitCycles) { ok = false; break; }
        }
        if (!__all_sync(0xffffffffu, ok)) { ok = false; break; }
        fence_proxy_async();
      }
      if (lane == 0) {
        tasks[ti & (kReady - 1)] = t;
        mbar_arrive(&ready[ti & (kReady - 1)]);
      }
      ++ti;
      if (end) break;
      if (lane == 0) {
        // the epilogue's addends on their way into L2
        const long long mt = t.el * 4 + ((long long)(t.tm * T + t.tn) << 16);
        if (o.c1 >= 0) bulk_prefetch(p.arena + o.c1 + mt, 65536);
        if (o.c2 >= 0) bulk_prefetch(p.arena + o.c2 + mt, 65536);
      }
      const uint8_t* A = p.arena + o.a + t.el * 2 + my_plane;
      const uint8_t* B = p.arena + o.b + t.el * 2 + my_plane;
      const bool one = o.a == o.b && t.tm == t.tn;      // both operands are the same blocks
      const int nkb = t.n_pad >> 6, kb_end = (t.n_real + 63) >> 6;
      // operand rows r, columns kb: the stored block, or left of the diagonal the rows kb of the stored tile
      // (kb / 2, r), read as its transpose
      auto block = [&](const uint8_t* src, int r, int kb) -> const uint8_t* {
        return (kb >> 1) < r ? src + ((long long)(kb >> 1) * nkb + 2 * r + half) * kBlkBytes + (kb & 1) * (kBlkBytes / 2)
                             : src + ((long long)r * nkb + kb) * kBlkBytes;
      };
      auto copy = [&](uint8_t* dst, const uint8_t* src, int r, int kb, uint64_t* bar) {
        const bool tr = (kb >> 1) < r;
        if (copies && (tr || half == 0)) bulk_g2s(dst, block(src, r, kb), tr ? kBlkBytes / 2 : kBlkBytes, bar);
      };
      for (int kb = 0; kb < kb_end; ++kb, ++k) {
        const int s = k % C::kBars;
        uint8_t* ua = smem + (2 * k) % C::kUnits * C::kUnitBytes + my_dst;
        uint8_t* ub = smem + (2 * k + 1) % C::kUnits * C::kUnitBytes + my_dst;
        // both units were last used by k-block k - kBars
        if (k >= C::kBars) ok = mbar_wait(&empty[s], (uint32_t)((k / C::kBars - 1) & 1));
        if (!__all_sync(0xffffffffu, ok)) { ok = false; break; }
        if (lane == 0) mbar_arrive_expect_tx(&full[s], one ? C::kUnitBytes : 2 * C::kUnitBytes);
        __syncwarp();
        copy(ua, A, t.tm, kb, &full[s]);
        if (one) continue;
        copy(ub, B, t.tn, kb, &full[s]);
      }
      if (!ok) break;
    }
    // the last copies have landed before shared memory is released
    for (int q = k - 1; q >= 0 && q >= k - C::kBars; --q) mbar_wait(&full[q % C::kBars], (uint32_t)((q / C::kBars) & 1));
  } else if (warp == kMmaW) {
    if (lane == 0) {
      constexpr uint32_t id0 = P == 2 ? idesc_f16_f32(128, 128) : idesc_bf16_f32(128, 128);
      constexpr uint64_t kPl = kBlkBytes >> 4;          // a plane further in a descriptor's address field
      const uint64_t dk = smem_desc_sw128(0), dmn = smem_desc_sw128_mn(0, kBlkBytes / 2);
      const uint32_t ring = smem_u32(smem) >> 4, corr = tmem + kCorr;
      int k = 0, ti = 0;
      while (ok) {
        if (!mbar_wait(&ready[ti & (kReady - 1)], (uint32_t)((ti / kReady) & 1))) { ok = false; break; }
        const Task t = tasks[ti & (kReady - 1)];
        if (t.last) break;
        const bool one = p.op[t.op].a == p.op[t.op].b && t.tm == t.tn;
        const int kb_end = (t.n_real + 63) >> 6;
        const uint32_t prev = (uint32_t)((ti - 1) & 1);
        auto wait_part = [&](int j) -> bool { return ti == 0 || mbar_wait(&acce[j], prev); };
        if (!wait_part(0)) { ok = false; break; }
        tc_fence_after();
        uint32_t acc = tmem;                            // accumulator kb % 3
        for (int kb = 0; kb < kb_end; ++kb, ++k) {
          const int s = k % C::kBars, ua = (2 * k) % C::kUnits, ub = one ? ua : (2 * k + 1) % C::kUnits;
          if (kb == 1 || kb == 2) {
            if (!wait_part(kb)) { ok = false; break; }
          }
          if (!mbar_wait(&full[s], (uint32_t)((k / C::kBars) & 1))) { ok = false; break; }
          tc_fence_after();
          const bool a_t = (kb >> 1) < t.tm, b_t = (kb >> 1) < t.tn;
          const uint32_t id = id0 | (a_t ? kIdescTransA : 0u) | (b_t ? kIdescTransB : 0u);
          const uint64_t sta = a_t ? 128 : 2, stb = b_t ? 128 : 2;      // one K step further
          uint64_t a0 = (a_t ? dmn : dk) + ring + (uint32_t)(ua * (C::kUnitBytes >> 4));
          uint64_t b0 = (b_t ? dmn : dk) + ring + (uint32_t)(ub * (C::kUnitBytes >> 4));
          // K steps that hold valid columns (the others would add zeros)
          const int ksteps = min(4, (t.n_real - kb * 64 + 15) >> 4);
#pragma unroll
          for (int kk = 0; kk < 4; ++kk) {
            if (kk >= ksteps) break;
            tc_mma_bf16(acc, a0, b0, id, (kb > 2 || kk != 0) ? 1u : 0u);
            tc_mma_bf16(corr, a0, b0 + kPl, id, (kb | kk) != 0 ? 1u : 0u);
            tc_mma_bf16(corr, a0 + kPl, b0, id, 1u);
            if (P == 3) {
              tc_mma_bf16(corr, a0, b0 + 2 * kPl, id, 1u);
              tc_mma_bf16(corr, a0 + kPl, b0 + kPl, id, 1u);
              tc_mma_bf16(corr, a0 + 2 * kPl, b0, id, 1u);
            }
            a0 += sta;
            b0 += stb;
          }
          acc = acc == tmem + 256 ? tmem : acc + 128;
          tc_commit(&empty[s]);
        }
        if (ok && kb_end < 2 && !wait_part(1)) ok = false;
        if (ok && kb_end < 3 && !wait_part(2)) ok = false;
        if (!ok) break;
        tc_commit(accf);
        ++ti;
      }
    }
  } else {
    // ---- epilogue warps: lane = row of the quadrant, 32 columns --------------------------------
    const int qd = warp & 3, cq = warp >> 2;
    const int pair = qd * 2 + (cq >> 1);
    uint8_t* slab = slabs + pair * kSlabBytes;
    const bool elect = (cq & 1) == 0 && lane == 0;      // issues the pair's copies
    const int row_sw = lane & 7, ch0 = (cq & 1) * 4;
    const uint32_t t_row = tmem + ((uint32_t)(qd * 32) << 16) + (uint32_t)(cq * 32);
    // this warp's leading addend columns in the slab: kPre x 512 bytes of C1, then of C2
    const float4* pre = reinterpret_cast<const float4*>(slab + (cq & 1) * (kSlabBytes / 2)) + lane;
    int ti = 0, n_add = 0, n_meet = 0;
    auto meet = [&] {
      __syncwarp();
      if (lane == 0) mbar_arrive(&pairb[pair]);
      if (!mbar_wait(&pairb[pair], (uint32_t)(n_meet & 1))) ok = false;
      ++n_meet;
    };
    while (true) {
      if (!__all_sync(0xffffffffu, mbar_wait(&ready[ti & (kReady - 1)], (uint32_t)((ti / kReady) & 1)) && ok)) {
        ok = false;
        break;
      }
      const Task t = tasks[ti & (kReady - 1)];
      if (t.last) break;
      const ChainOp& o = p.op[t.op];
      const int T = t.n_pad >> 7, kb_end = (t.n_real + 63) >> 6;
      // a master's tile, from this lane's first float4
      const long long mt = t.el * 4 + ((long long)(t.tm * T + t.tn) << 16) + ((warp * 8) * 32 + lane) * 16;
      const bool has1 = o.c1 >= 0, has2 = o.c2 >= 0;
      const bool dual = P == 2 && o.out2 >= 0;          // (the three-plane form has no two-output product)
      if (elect) {
        // the slabs are free once the last task's stores have read them
        asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
        if (has1 && !dual) {
          constexpr uint32_t nb = C::kPre * 512;
          mbar_arrive_expect_tx(&addf[pair], (has2 ? 4 : 2) * nb);
          for (int h = 0; h < 2; ++h) {                 // this warp and its neighbour (warp + 4)
            uint8_t* d = slab + h * (kSlabBytes / 2);
            const long long at = mt + h * (4 * 8 * 512);
            bulk_g2s(d, p.arena + o.c1 + at, nb, &addf[pair]);
            if (has2) bulk_g2s(d + nb, p.arena + o.c2 + at, nb, &addf[pair]);
          }
        }
      }
      // (the warp leaves together where a wait gave up in any lane)
      if (!__all_sync(0xffffffffu, mbar_wait(accf, (uint32_t)(ti & 1)) && ok)) { ok = false; break; }
      tc_fence_after();
      auto release = [&](int j) {
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&acce[j]);
      };
      float v[32];
      {
        uint32_t r0[32], r1[32];
        tmem_ld32_nowait(t_row, r0);
        tmem_ld32_nowait(t_row + kCorr, r1);
        tmem_wait_ld();
        release(0);
#pragma unroll
        for (int j = 0; j < 32; ++j)
          v[j] = P == 2 ? fmaf(__uint_as_float(r1[j]), kF16LoInv, __uint_as_float(r0[j]))
                        : __uint_as_float(r0[j]) + __uint_as_float(r1[j]);
      }
#pragma unroll
      for (int part = 1; part < 3; ++part) {
        if (kb_end > part) {
          uint32_t r0[32];
          tmem_ld32_nowait(t_row + 128 * part, r0);
          tmem_wait_ld();
          release(part);
#pragma unroll
          for (int j = 0; j < 32; ++j) v[j] += __uint_as_float(r0[j]);
        } else {
          release(part);
        }
      }

      const int row = t.tm * 128 + qd * 32 + lane, col = t.tn * 128 + cq * 32;
      // tiles on the diagonal or with padding take the general path
      const bool special = t.tm == t.tn || (t.tn + 1) * 128 > t.n_real;
      const float beta = t.tm == t.tn ? o.beta : 0.f, g1 = o.g1, g2 = o.g2;
      uint32_t u[P][16];
      // planes of this warp's 32 x 32 values into the slabs it shares with its neighbour, and from there to
      // each block's 4 KB in one bulk copy
      const long long pt = t.el * 2 + ((long long)t.tm * (t.n_pad >> 6) + t.tn * 2 + (cq >> 1)) * kBlkBytes + qd * kSlabBytes;
      auto put = [&](long long dst, bool first) {
#pragma unroll
        for (int p0 = 0; p0 < P; ++p0) {
          if (elect && (p0 > 0 || !first)) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
          meet();
#pragma unroll
          for (int i = 0; i < 4; ++i)
            *reinterpret_cast<uint4*>(slab + lane * 128 + (((ch0 + i) ^ row_sw) << 4)) =
                make_uint4(u[p0][4 * i], u[p0][4 * i + 1], u[p0][4 * i + 2], u[p0][4 * i + 3]);
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
          meet();
          if (elect) {
            bulk_s2g(p.arena + dst + p0 * p.plane + pt, slab, kSlabBytes);
            asm volatile("cp.async.bulk.commit_group;" ::: "memory");
          }
        }
      };
      // x = alpha v + beta I + g1 C1 + g2 C2, zero off the valid block: four columns from float4 j4
      auto column4 = [&](int j4, float alpha, const float4& a, const float4& b, bool sp, float4* om) {
        const float av[4] = {a.x, a.y, a.z, a.w}, bv[4] = {b.x, b.y, b.z, b.w};
        float x[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const int j = 4 * j4 + e;
          x[e] = fmaf(alpha, v[j], sp && row == col + j ? beta : 0.f);
          x[e] = fmaf(g2, bv[e], fmaf(g1, av[e], x[e]));
          if (sp && (row >= t.n_real || col + j >= t.n_real)) x[e] = 0.f;
        }
        if (om) __stcg(om + j4 * 32, make_float4(x[0], x[1], x[2], x[3]));
        pack<P>(x, u, 2 * j4);
      };
      const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
      const float4* c1 = reinterpret_cast<const float4*>(p.arena + o.c1 + mt);
      const float4* c2 = reinterpret_cast<const float4*>(p.arena + o.c2 + mt);
      if (dual) {
        // the first output alpha v, then the second with its addends from L2
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          float x[4];
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            x[e] = o.alpha * v[4 * i + e];
            if (special && (row >= t.n_real || col + 4 * i + e >= t.n_real)) x[e] = 0.f;
          }
          pack<P>(x, u, 2 * i);
        }
        put(o.out, true);
#pragma unroll
        for (int h = 0; h < 4; ++h) {
          float4 a[2], b[2];
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            a[i] = __ldcg(c1 + (2 * h + i) * 32);
            b[i] = __ldcg(c2 + (2 * h + i) * 32);
          }
#pragma unroll
          for (int i = 0; i < 2; ++i) column4(2 * h + i, o.alpha2, a[i], b[i], special, nullptr);
        }
        put(o.out2, false);
      } else {
        const float alpha = o.alpha;
        float4* om = o.outm >= 0 ? reinterpret_cast<float4*>(p.arena + o.outm + mt) : nullptr;
        auto combine = [&](bool sp) {
          if (!has1) {
#pragma unroll
            for (int i = 0; i < 8; ++i) column4(i, alpha, zero, zero, sp, om);
            return;
          }
          // the later columns straight from L2: two in flight while the leading ones are combined from the slab
          constexpr int K = C::kPre;
          float4 a[2], b[2];
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            a[i] = __ldcg(c1 + (K + i) * 32);
            b[i] = has2 ? __ldcg(c2 + (K + i) * 32) : zero;
          }
          if (!mbar_wait(&addf[pair], (uint32_t)(n_add & 1))) ok = false;
#pragma unroll
          for (int i = 0; i < K; ++i) column4(i, alpha, pre[i * 32], has2 ? pre[(K + i) * 32] : zero, sp, om);
#pragma unroll
          for (int h = K; h < 8; h += 2) {
#pragma unroll
            for (int i = 0; i < 2; ++i) column4(h + i, alpha, a[i], b[i], sp, om);
            if (h + 2 < 8) {
#pragma unroll
              for (int i = 0; i < 2; ++i) {
                a[i] = __ldcg(c1 + (h + 2 + i) * 32);
                b[i] = has2 ? __ldcg(c2 + (h + 2 + i) * 32) : zero;
              }
            }
          }
        };
        if (special) combine(true);
        else combine(false);
        if (has1) ++n_add;
        put(o.out, true);
      }
      ++ti;
      if (p.n_ops > 1) {
        // this warp's part of the tile is in memory: masters by its lanes, planes by the elected lane's copies
        __syncwarp();
        if (lane == 0) {
          if (elect) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
          fence_proxy_async();
          red_release(p.done + t.mat, 1u);
        }
        __syncwarp();
      }
    }
    if (elect) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    tmem_dealloc(tmem, 512);
  }
  if (!ok) atomicOr(p.err, kErrTimeout);
}

cudaError_t sm_count(int* sms) {
  int dev = 0;
  const cudaError_t e = cudaGetDevice(&dev);
  return e ? e : cudaDeviceGetAttribute(sms, cudaDevAttrMultiProcessorCount, dev);
}

template <int P>
cudaError_t launch(const ChainParams& p, int n_work, cudaStream_t s) {
  cudaError_t e;
  int sms = 0;
  if ((e = sm_count(&sms))) return e;
  if ((e = cudaFuncSetAttribute(product_chain<P>, cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg<P>::kSmem))) return e;
  void* args[] = {const_cast<ChainParams*>(&p)};
  const dim3 grid(n_work < sms ? n_work : sms);
  return cudaLaunchCooperativeKernel(reinterpret_cast<const void*>(product_chain<P>), grid, dim3(kThreads), args,
                                     (size_t)Cfg<P>::kSmem, s);
}

}  // namespace

// Three tiles per SM: a subgraph's next product then starts when the last one's tiles have been two rounds in
// flight, and the window's matrices (about 260 MB) are partly still in L2.  Measured for 3,415 tiles: windows of
// 152 tiles 319 us a product, 228: 249, 304: 202, 380: 196, 456: 198, 608: 206, one window: 222.
cudaError_t chain_window_tiles(int* tiles) {
  int sms = 0;
  const cudaError_t e = sm_count(&sms);
  *tiles = 3 * sms;
  return e;
}

cudaError_t launch_chain(const ChainParams& p, int planes, int n_work, int n_sub, cudaStream_t s) {
  if (n_work <= 0 || p.n_ops <= 0) return cudaSuccess;
  if (p.n_ops > 1) {
    const cudaError_t e = cudaMemsetAsync(p.done, 0, sizeof(unsigned) * n_sub, s);
    if (e) return e;
  }
  return planes == 2 ? launch<2>(p, n_work, s) : launch<3>(p, n_work, s);
}

}  // namespace sedacs
