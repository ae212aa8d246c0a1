// Restrict + forward/back substitution of Eq. (pmlij) over the symmetric tile storage
// (HD_SYMMETRIC): only the upper 16 x 16 tiles of every complex symmetric S_j^{-1} are
// stored and streamed, and a tile (I, J), I < J, serves twice, y_I += T v_J and
// y_J += T^T v_I.
//
// Order of the sum.  The tiles lie column by column and are taken in segments of up to
// three tiles of one column J (one tile in complex FP64 where no box is wider than 64; SymMap in
// hd_internal.cuh), the segments in SYM_GROUPS groups.  One warp takes a segment: each lane holds 2 x 4 entries of every tile in
// registers and forms both products from that one read; the column products T^T v_I add up
// over the segment, the row products T v_J are summed tile by tile, and the 16 sums of each
// go to a slot of their own in shared memory.  One thread per output then adds, group by
// group, the row slots (J ascending) and the column slots (segments ascending), and the
// group sums in order.  That order depends on the widths of the boxes alone: a launch may spread
// the groups over K CTAs of a cluster, over P sets of warps, and may run one or several
// right-hand sides per CTA, with bitwise the same result.
//
// What bounds it.  Many boxes: HBM (every tile twice per application).  Few boxes: the
// chain of 2 rows - 1 dependent steps per box, so the box is spread over K CTAs (each
// streams and multiplies 1/K of the tiles; one exchange of group sums per step, st.async
// into the other CTAs' shared memory) and the operands of the next step are loaded while
// this one runs.  Several right-hand sides: instruction issue, hence the packed FP32 FMAs
// (fma.rn.f32x2): with a = (re, im) of the stored entry and the vector entry b held as
// (br, br, bi, bi), the sums of a * (br, br) and of a * (bi, bi) need two packed FMAs per
// complex product and no operand shuffling; re and im are formed once per sum.
//
// Measured per application (substitution and sum, one CTA per box and tile per warp before): c64, 128^2 in 4
// boxes 0.80 -> 0.23 ms; 1003^2 in 64 boxes 2.83 -> 0.58 ms (4.6 TB/s); 2048^2 in 256 boxes 3.28 ->
// 1.82 ms; 4096^2 in 1024 boxes 8.20 -> 6.95 ms (7.1 TB/s); four sources at 2048^2 6.07 -> 4.54 ms;
// c128, 1024^2 in 64 boxes 14.3 -> 7.3 ms; narrow boxes in hd_sym_shape.cuh.
//
// A producer warp (one lane per set) streams the tiles by bulk copies into an mbarrier
// ring, ahead across steps: a stage is one round of a set, a segment for each of its warps.
// Every wait is bounded: on timeout ST_TIMEOUT is flagged, every warp runs on to the end,
// and the producer waits for its copies still in flight before the CTA exits.
//
// Hazards of the cluster form.  Received group sums sit in two buffers (even and odd
// steps): a CTA sends step t + 2 only after it has every sum of step t + 1, which the
// receiver sent after it was done with step t.  A thread that gave up a wait leaves its vector
// work, and with it the exchange (it would run ahead of that bound, and of what an mbarrier can
// count), so the other CTAs give up too.  Row j of the staging buffer is written by
// one CTA and read by all in the back substitution: a release / acquire pair at cluster
// scope (barrier `turn`) separates the two sweeps, and x_j replaces w_j one step late, when
// the other CTAs' sums of the step after prove that they have used w_j.
#include <algorithm>
#include <type_traits>

#include "hd_internal.cuh"
#include "hd_sym_shape.cuh"
#include "hd_tc.cuh"

namespace hd {

namespace {

constexpr int TB = 16, TE = TB * TB;

// ---------------------------------------------------------------- cluster and ring helpers
__device__ __forceinline__ void bulk_in(void *dst, const void *src, uint32_t bytes, uint64_t *bar) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(tc::su32(bar)), "r"(bytes) : "memory");
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   tc::su32(dst)),
               "l"(src), "r"(bytes), "r"(tc::su32(bar))
               : "memory");
}
__device__ __forceinline__ void bar_arrive(uint64_t *bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(tc::su32(bar)) : "memory");
}
__device__ __forceinline__ uint32_t cluster_map(const void *p, uint32_t rank) {
  uint32_t a;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(tc::su32(p)), "r"(rank));
  return a;
}
__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_sync_all() {
  __syncwarp();
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_send(uint32_t dst, float2 v, uint32_t bar) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v2.b32 [%0], {%1, %2}, [%3];" ::"r"(dst),
               "r"(__float_as_uint(v.x)), "r"(__float_as_uint(v.y)), "r"(bar)
               : "memory");
}
__device__ __forceinline__ void cluster_send(uint32_t dst, double2 v, uint32_t bar) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v2.b64 [%0], {%1, %2}, [%3];" ::"r"(dst),
               "l"(__double_as_longlong(v.x)), "l"(__double_as_longlong(v.y)), "r"(bar)
               : "memory");
}
// About a millisecond: a thousand times what a store into another CTA's shared memory takes.
__device__ __forceinline__ void settle() {
  for (const long long t0 = clock64(); clock64() - t0 < 2000000;) {}
}
// Bounded wait with acquire semantics at cluster scope (the phase is completed by other CTAs).
__device__ __forceinline__ bool wait_cluster(uint64_t *bar, uint32_t parity, volatile int *abort_flag) {
  for (uint32_t it = 0; it < tc::kWaitLimit; ++it) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(tc::su32(bar)), "r"(parity)
        : "memory");
    if (ok) return true;
    if ((it & 255u) == 255u && *abort_flag) return false;
  }
  return false;
}

// ---------------------------------------------------------------- arithmetic
// Complex FP32: sums of products a b kept as A = sum a br, B = sum a bi (componentwise on a).
// Complex FP64, bound by the FP64 pipe: re and im summed directly (no additions at the end).
template <typename R> struct Ops;
template <> struct Ops<float> {
  using Ent = unsigned long long;   // (re, im) of a stored entry in one 64-bit register
  struct Vec { unsigned long long x, y; };   // (br, br), (bi, bi)
  struct Acc { unsigned long long a, b; };
  static __device__ __forceinline__ Acc zero() { return Acc{0ull, 0ull}; }
  static __device__ __forceinline__ unsigned long long pack(float x, float y) {
    unsigned long long r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x), "f"(y));
    return r;
  }
  static __device__ __forceinline__ float2 unpack(unsigned long long v) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
  }
  static __device__ __forceinline__ void mac(Acc &c, Ent a, const Vec &v) {
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(c.a) : "l"(a), "l"(v.x));
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(c.b) : "l"(a), "l"(v.y));
  }
  static __device__ __forceinline__ float2 value(const Acc &c) {
    const float2 a = unpack(c.a), b = unpack(c.b);
    return make_float2(add_rn(a.x, -b.y), add_rn(a.y, b.x));
  }
  static __device__ __forceinline__ Vec vec(float x, float y) { return Vec{pack(x, x), pack(y, y)}; }
  // two consecutive vector entries (16-byte aligned)
  static __device__ __forceinline__ void load2(const float2 *p, Vec &u, Vec &v) {
    const float4 t = *reinterpret_cast<const float4 *>(p);
    u = vec(t.x, t.y);
    v = vec(t.z, t.w);
  }
};
template <> struct Ops<double> {
  using Ent = double2;
  using Vec = double2;
  struct Acc { double2 c; };
  static __device__ __forceinline__ Acc zero() { return Acc{make_double2(0.0, 0.0)}; }
  static __device__ __forceinline__ void mac(Acc &s, Ent a, const Vec &v) { s.c = cfma(a, v, s.c); }
  static __device__ __forceinline__ double2 value(const Acc &s) { return s.c; }
  static __device__ __forceinline__ void load2(const double2 *p, Vec &u, Vec &v) {
    u = p[0];
    v = p[1];
  }
};

// A lane's entries of a tile (sym_pos in hd_internal.cuh): t[q][e] = T[2 rg + e][4 cg + q].
__device__ __forceinline__ void load_tile(const float2 *tile, int lane, unsigned long long (&t)[4][2]) {
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const ulonglong2 v = reinterpret_cast<const ulonglong2 *>(tile)[q * 32 + lane];
    t[q][0] = v.x;
    t[q][1] = v.y;
  }
}
template <typename H> __device__ __forceinline__ void load_tile16(const H *tile, int lane, unsigned long long (&t)[4][2]) {
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const uint2 v = reinterpret_cast<const uint2 *>(tile)[q * 32 + lane];
    const float2 a = load_c<float2>(*reinterpret_cast<const H *>(&v.x)), b = load_c<float2>(*reinterpret_cast<const H *>(&v.y));
    t[q][0] = Ops<float>::pack(a.x, a.y);
    t[q][1] = Ops<float>::pack(b.x, b.y);
  }
}
__device__ __forceinline__ void load_tile(const __half2 *tile, int lane, unsigned long long (&t)[4][2]) { load_tile16(tile, lane, t); }
__device__ __forceinline__ void load_tile(const __nv_bfloat162 *tile, int lane, unsigned long long (&t)[4][2]) { load_tile16(tile, lane, t); }
__device__ __forceinline__ void load_tile(const double2 *tile, int lane, double2 (&t)[4][2]) {
#pragma unroll
  for (int q = 0; q < 4; ++q)
#pragma unroll
    for (int e = 0; e < 2; ++e) t[q][e] = tile[(q * 2 + e) * 32 + lane];
}

// Halves of two values exchanged between lanes l and l ^ x: the lane with `up` keeps b, the
// other a, each plus the partner's copy.
template <typename R> __device__ __forceinline__ R fold(R a, R b, bool up, int x) {
  const R send = up ? a : b, keep = up ? b : a;
  return add_rn(keep, __shfl_xor_sync(0xffffffffu, send, x));
}
// Row sums of a tile: r[e] of row 2 rg + e, over the lanes cg = lane >> 3; the lane's scalar
// goes to place row_place(lane) of the 16 complex row sums.
template <typename T> __device__ __forceinline__ decltype(T::x) reduce_rows(const T (&r)[2], int lane) {
  const bool b4 = (lane & 16) != 0, b3 = (lane & 8) != 0;
  const auto x = fold(r[0].x, r[1].x, b4, 16);
  const auto y = fold(r[0].y, r[1].y, b4, 16);
  return fold(x, y, b3, 8);
}
__device__ __forceinline__ int row_place(int lane) { return 4 * (lane & 7) + ((lane >> 3) & 2) + ((lane >> 3) & 1); }
// Column sums: c[q] of column 4 cg + q, over the lanes rg = lane & 7; the lane's scalar goes
// to place `lane` of the 16 complex column sums.
template <typename T> __device__ __forceinline__ decltype(T::x) reduce_cols(const T (&c)[4], int lane) {
  const bool b2 = (lane & 4) != 0, b1 = (lane & 2) != 0, b0 = (lane & 1) != 0;
  const auto x0 = fold(c[0].x, c[2].x, b2, 4), y0 = fold(c[0].y, c[2].y, b2, 4);
  const auto x1 = fold(c[1].x, c[3].x, b2, 4), y1 = fold(c[1].y, c[3].y, b2, 4);
  const auto x = fold(x0, x1, b1, 2), y = fold(y0, y1, b1, 2);
  return fold(x, y, b0, 1);
}

// ---------------------------------------------------------------- launch shape
// Warps of a set, a segment each per round (SW): 7 in complex FP32 (two sets and a producer make
// 15 warps, which leaves 128 registers a thread), 8 in complex FP64, whose products keep the four
// FP64 pipes of the SM equally busy only if the warps divide by four, 3 in the small form.
constexpr int MAXTERM = 8;               // sums of one output in one group (boxes up to 256 wide)

// Rounds of a group of n segments, at most `spr` (<= the set's warps) a round; round c takes the segments
// n c / rounds .. n (c + 1) / rounds.
__host__ __device__ __forceinline__ int sym_rounds(int n, int spr) { return (n + spr - 1) / spr; }

// Tiles of the largest round (one ring stage) of any box up to mt tiles wide: a narrower box
// may have fewer rounds, and so larger ones.
static int sym_stage_tiles(int mt, int spr, int seg) {
  int most = 1;
  for (int t = 1; t <= mt; ++t) {
    const SymMap map(16 * t, seg);
    for (int g = 0; g < SYM_GROUPS; ++g) {
      const int b = map.group_start(g), n = map.group_start(g + 1) - b, nr = sym_rounds(n, spr);
      for (int c = 0; c < nr; ++c)
        most = std::max(most, map.first_tile(b + n * (c + 1) / nr) - map.first_tile(b + n * c / nr));
    }
  }
  return most;
}

// ring [P][NS][ST tiles] | vs [NR][mp] T | slots [NR][nt + nseg + 1][32] R (row sums by
// tile, column sums by segment, a zero slot) | pb [2][groups][NR][mp] T (K > 1) |
// terms [groups][mt][MAXTERM] | rounds, items (below) | barriers: full, empty [P][NS], xbar [2], turn | abort.
struct SymSmem {
  size_t vs, slots, pb, terms, rounds, items, bars, total;
  int nslot, maxround;
};
template <typename R, typename S>
__host__ __device__ inline SymSmem sym_smem(int ns, int stage_tiles, int spr, int mp, int K, int P, int nr, int sw, int seg) {
  const SymMap map(mp, seg);
  SymSmem L;
  L.nslot = map.nt + map.nseg + 1;
  L.maxround = sym_rounds(map.base + (map.rem > 0), spr) * (SYM_GROUPS / (K * P));   // rounds of a set per step
  L.vs = (size_t)P * ns * stage_tiles * TE * sizeof(S);
  L.slots = L.vs + (size_t)nr * mp * 2 * sizeof(R);
  L.pb = L.slots + (size_t)nr * L.nslot * 32 * sizeof(R);
  L.terms = L.pb + (K > 1 ? 2 * (size_t)SYM_GROUPS * nr * mp * 2 * sizeof(R) : 0);
  L.rounds = L.terms + (size_t)SYM_GROUPS * map.mt * MAXTERM * sizeof(uint16_t);
  L.items = L.rounds + (size_t)P * (L.maxround + 1) * sizeof(uint32_t);
  L.bars = (L.items + (size_t)P * L.maxround * sw * sizeof(uint32_t) + 15) & ~(size_t)15;
  L.total = L.bars + (2 * (size_t)P * ns + 3) * sizeof(uint64_t) + 16;
  return L;
}

}  // namespace

// One cluster of K CTAs per (box, NR right-hand sides); the P sets of a CTA walk
// SYM_GROUPS / (K P) groups each, one after another.  The vector work of a step is spread
// over VG groups of warps, NR / VG right-hand sides each.
template <typename R, typename S, int K, int P, int NR, int VG, int SW, int PER_SM>
__global__ void __launch_bounds__((P * SW + 1) * 32, PER_SM)
k_subst_sym(const SubDev *__restrict__ subs, const C<R> *__restrict__ poolr,
            const S *__restrict__ factor, const double2 *__restrict__ rg, int NX, int64_t vec_stride,
            C<R> *__restrict__ staging, int64_t stg_stride, int nrhs, int NS, int ST, int SPR, int seg_tiles, int mpmax, int32_t *status) {
  using T = C<R>;
  using O = Ops<R>;
  using Vec = typename O::Vec;
  using Acc = typename O::Acc;
  constexpr int PW = P * SW, CT = PW * 32;
  constexpr bool SMALL = PER_SM > 2;
  constexpr int NV = NR / VG;                          // right-hand sides of a vector thread
  constexpr int GPC = SYM_GROUPS / K, GPS = GPC / P;   // groups per CTA and per set
  extern __shared__ __align__(128) unsigned char smem_raw[];
  const SubDev s = subs[blockIdx.y];
  const int m = s.ex, rows = s.ey;
  const int SEG = sizeof(R) == 4 ? 3 : seg_tiles;   // (a constant where it can be)
  const SymMap map(m, SEG);
  const int mt = map.mt, nt = map.nt;
  const uint32_t rank = K > 1 ? cluster_rank() : 0u;
  const int r0 = (int)(blockIdx.x / K) * NR;
  const int nq = SMALL ? min(NR, nrhs - r0) : NR;   // right-hand sides to form products for
  const SymSmem L = sym_smem<R, S>(NS, ST, SPR, mpmax, K, P, NR, SW, SEG);
  S *ring = reinterpret_cast<S *>(smem_raw);
  T *vs = reinterpret_cast<T *>(smem_raw + L.vs);
  R *slots = reinterpret_cast<R *>(smem_raw + L.slots);
  T *pb = reinterpret_cast<T *>(smem_raw + L.pb);
  uint16_t *terms = reinterpret_cast<uint16_t *>(smem_raw + L.terms);     // [group][A][MAXTERM] slots of the sum, x 32
  uint32_t *rounds = reinterpret_cast<uint32_t *>(smem_raw + L.rounds);   // [set][round] first tile | tiles << 16 (0: end)
  uint32_t *items = reinterpret_cast<uint32_t *>(smem_raw + L.items);     // [set][round][warp], packed as below
  uint64_t *full = reinterpret_cast<uint64_t *>(smem_raw + L.bars);
  uint64_t *empty = full + P * NS;
  uint64_t *xbar = empty + P * NS;
  uint64_t *turn = xbar + 2;
  volatile int *abort_flag = reinterpret_cast<volatile int *>(turn + 1);
  const int qstride = L.nslot * 32;   // slots of one right-hand side
  int warp = threadIdx.x >> 5;
  if constexpr (SMALL && sizeof(R) == 8) {
    // (FP64 runs at the rate of each quarter of the SM: the roles turn with the CTA's place on the SM, or
    // the producers and the longest segments of its CTAs would meet on one quarter)
    if (threadIdx.x == 0) {
      uint32_t w;
      asm volatile("mov.u32 %0, %%warpid;" : "=r"(w));
      abort_flag[1] = (int)(w >> 2);
    }
    __syncthreads();
    warp = (warp + abort_flag[1]) % (PW + 1);
  }
  const int lane = threadIdx.x & 31, tid = warp * 32 + lane;
  if (tid == 0) {
    for (int q = 0; q < P * NS; ++q) {
      tc::bar_init(&full[q], 1);
      tc::bar_init(&empty[q], SW);
    }
    tc::bar_init(&xbar[0], 1);
    tc::bar_init(&xbar[1], 1);
    tc::bar_init(turn, K);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  // The schedule of a step, the same in every step.  Round c of a set: its tiles, consecutive
  // in memory (one ring stage).  Item of a warp in a round: segment (I0, J) of n tiles (0: none),
  // its first tile `at` in the stage, I0 | J << 5 | n << 10 | at << 12 | segment << 17.
  // segments s0 .. s1 - 1 of round c of a set (false: the set has fewer rounds)
  auto round_of = [&](int set, int c, int &s0, int &s1) {
    for (int g = (int)rank * GPC + set * GPS; g < (int)rank * GPC + (set + 1) * GPS; ++g) {
      const int b = map.group_start(g), n = map.group_start(g + 1) - b, nr = sym_rounds(n, SPR);
      if (c < nr) {
        s0 = b + n * c / nr;
        s1 = b + n * (c + 1) / nr;
        return true;
      }
      c -= nr;
    }
    return false;
  };
  auto make_item = [&](int seg, int t0) {
    int I, J;
    map.segment(seg, I, J);
    return (uint32_t)I | (uint32_t)J << 5 | (uint32_t)min(SEG, J - I + 1) << 10 |
           (uint32_t)(J * (J + 1) / 2 + I - t0) << 12 | (uint32_t)seg << 17;
  };
  for (int i = tid; i < P * (L.maxround + 1); i += CT + 32) {
    const int set = i / (L.maxround + 1), c = i - set * (L.maxround + 1);
    int s0, s1;
    uint32_t v = 0;
    if (round_of(set, c, s0, s1)) {
      const int t0 = map.first_tile(s0);
      v = (uint32_t)t0 | (uint32_t)(map.first_tile(s1) - t0) << 16;
    }
    rounds[i] = v;
  }
  if constexpr (K == 1 && (SMALL || sizeof(R) == 8 || NR > 1)) {
    // bound by arithmetic: a segment goes to the free warp of the round whose quarter of the SM
    // (warp % 4) has the fewest products so far (lane = warp; the busiest quarter then has 2 to
    // 10 % more than the mean, up to 55 % when they are dealt out in order: 14.7 -> 13.5 ms per
    // complex FP64 application of 144 boxes)
    if (warp == 0) {
      uint32_t load = 0;
      for (int c = 0; c < L.maxround; ++c)
        for (int set = 0; set < P; ++set) {
          bool open = lane / SW == set && lane < PW;
          int s0 = 0, s1 = 0;
          round_of(set, c, s0, s1);
          const int t0 = s0 < s1 ? map.first_tile(s0) : 0;
          for (int seg = s0; seg < s1; ++seg) {
            const uint32_t item = make_item(seg, t0), n = item >> 10 & 3u;
            const bool diag = (item & 31u) + n > (item >> 5 & 31u);
            const uint32_t to = __reduce_min_sync(0xffffffffu, open ? load << 5 | (uint32_t)lane : 0xffffffffu) & 31u;
            if ((uint32_t)lane == to) {
              items[(set * L.maxround + c) * SW + lane - set * SW] = item;
              open = false;
            }
            if (((uint32_t)lane & 3u) == (to & 3u)) load += 8u * n - (diag ? 4u : 0u) + 1u;
          }
          if (open) items[(set * L.maxround + c) * SW + lane - set * SW] = 0;
        }
    }
  } else {
    for (int i = tid; i < P * L.maxround * SW; i += CT + 32) {
      const int set = i / (L.maxround * SW), c = i / SW - set * L.maxround;
      const int k = (i + 3 * c + set) % SW;   // (rounds with fewer segments leave other warps out)
      int s0, s1;
      items[i] = round_of(set, c, s0, s1) && s0 + k < s1 ? make_item(s0 + k, map.first_tile(s0)) : 0u;
    }
  }
  for (int i = tid; i < SYM_GROUPS * mt; i += CT + 32) {
    const int g = i / mt, A = i - g * mt;
    int n = 0;
    for (int J = A; J < mt; ++J)
      if (map.group_of(map.col_seg(J) + (SEG == 1 ? A : A / 3)) == g) terms[i * MAXTERM + n++] = (uint16_t)((J * (J + 1) / 2 + A) * 32);
    for (int k = 0; SEG * k < A; ++k)
      if (map.group_of(map.col_seg(A) + k) == g) terms[i * MAXTERM + n++] = (uint16_t)((nt + map.col_seg(A) + k) * 32);
    for (; n < MAXTERM; ++n) terms[i * MAXTERM + n] = (uint16_t)((nt + map.nseg) * 32);
  }
  for (int i = tid; i < NR * 32; i += CT + 32) slots[(i >> 5) * qstride + (nt + map.nseg) * 32 + (i & 31)] = (R)0;
  if (SMALL)   // (the sums of those that do not exist)
    for (int i = nq * qstride + tid; i < NR * qstride; i += CT + 32) slots[i] = (R)0;
  if (K > 1) cluster_sync_all();   // barriers ready in every CTA before the first remote store
  else __syncthreads();

  const int nsteps = 2 * rows - 1;

  if (warp == PW) {
    // ---------------- producer warp: lane p streams the rounds of set p in use order
    if (lane < P) {
      uint64_t *pf = full + lane * NS, *pe = empty + lane * NS;
      S *pr = ring + (size_t)lane * NS * ST * TE;
      const uint32_t *rd = rounds + lane * (L.maxround + 1);
      const S *Fs = factor + s.foff;
      int issued = 0, slot = 0;
      uint32_t ph = 0;
      bool ok = true;
      for (int st = 0; st < nsteps && ok; ++st) {
        const int j = st < rows ? st : 2 * rows - 2 - st;
        const S *blk = Fs + (int64_t)j * nt * TE;
        for (int c = 0; rd[c]; ++c) {
          if (!tc::bar_wait(&pe[slot], ph ^ 1u, abort_flag)) { ok = false; break; }
          bulk_in(pr + (size_t)slot * ST * TE, blk + (rd[c] & 0xFFFFu) * TE,
                  (rd[c] >> 16) * (uint32_t)(TE * sizeof(S)), &pf[slot]);
          ++issued;
          if (++slot == NS) { slot = 0; ph ^= 1u; }
        }
      }
      if (!ok) {
        *abort_flag = 1;
        atomicOr(status, ST_TIMEOUT);
      }
      // no copy may still be landing in shared memory when the CTA exits
      tc::ring_drain(pf, issued, NS);
    }
  } else {
    // ---------------- consumer warps; thread a < m of vector group vg owns output a of the
    //                  right-hand sides q0 .. q0 + NV - 1 of the CTA
    const int vspan = (mpmax + 31) & ~31;   // VG vspan <= CT
    const int vg = VG > 1 && tid >= vspan ? 1 : 0;
    const int a = tid - vg * vspan, A = a >> 4, q0 = vg * NV;
    const int gx = s.ex0 + a;
    bool vec = a < m;   // has vector work (until a wait fails)
    const bool ownx = vec && gx >= s.ox0 && gx < s.ox1;
    const bool writer = vec && (K == 1 || (uint32_t)((a >> 5) % K) == rank);
    const int nlive = nrhs - r0 - q0;   // right-hand sides q < nlive exist
    const T *ia2f = poolr + s.aoff + 2 * m + 1 + rows;
    T a1 = mk<T>(0, 0);
    if (vec) a1 = poolr[s.aoff + a];
    uint32_t peer_pb[K], peer_bar[K];   // this thread's slot of group sum rank * GPC, and xbar[0], in the other CTAs
#pragma unroll
    for (int d = 1; d < K; ++d) {
      const uint32_t peer = (rank + (uint32_t)d) % (uint32_t)K;
      peer_pb[d] = cluster_map(pb + ((size_t)rank * GPC * NR + q0) * mpmax + a, peer);
      peer_bar[d] = cluster_map(xbar, peer);
    }
    bool ok = true;
    auto fail = [&]() {
      ok = false;
      if (K > 1) vec = false;
      *abort_flag = 1;
      atomicOr(status, ST_TIMEOUT);
    };
    const double2 *rga = rg + (int64_t)(r0 + q0) * vec_stride + (int64_t)s.ey0 * NX + gx;
    T *stga = staging + (int64_t)(r0 + q0) * stg_stride + s.soff + a;
    // rho_j of the owned part (zero elsewhere)
    auto load_rho = [&](int j, double2 (&v)[NV]) {
      const int gy = s.ey0 + j;
      const bool own = ownx && gy >= s.oy0 && gy < s.oy1;
#pragma unroll
      for (int q = 0; q < NV; ++q) {
        v[q] = make_double2(0.0, 0.0);
        if (own && q < nlive) v[q] = rga[q * vec_stride + (int64_t)j * NX];
      }
    };
    if (a < mt * TB) {   // the first step's vector, rho_0
      double2 v[NV];
      load_rho(0, v);
#pragma unroll
      for (int q = 0; q < NV; ++q) vs[(q0 + q) * mpmax + a] = vec ? mk<T>(from_d<R>(v[q].x), from_d<R>(v[q].y)) : mk<T>(0, 0);
    }
    T x[NV];   // K > 1: x_{j+1}, not yet written out
#pragma unroll
    for (int q = 0; q < NV; ++q) x[q] = mk<T>(0, 0);
    const int set = warp / SW, ws = warp - set * SW;
    uint64_t *sf = full + set * NS, *se = empty + set * NS;
    const S *sring = ring + (size_t)set * NS * ST * TE;
    const uint32_t *myitems = items + set * L.maxround * SW + ws;
    const uint32_t *rd = rounds + set * (L.maxround + 1);
    const int rplace = row_place(lane);
    const T *vsr = vs + 2 * (lane & 7), *vsc = vs + 4 * (lane >> 3);
    int slot = 0;
    uint32_t ph = 0;
    for (int st = 0; st < nsteps; ++st) {
      const bool fwd = st < rows;
      const int j = fwd ? st : 2 * rows - 2 - st;
      asm volatile("bar.sync 1, %0;" ::"n"(CT) : "memory");   // vs complete; the sums of the last step are read
      if (K > 1 && rows > 1) {
        if (st == rows - 1 && tid == 0) {   // this CTA's part of w_0 .. w_{rows-2} is in the staging buffer
          asm volatile("fence.acq_rel.cluster;" ::: "memory");
          for (uint32_t p = 0; p < (uint32_t)K; ++p)
            asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_map(turn, p)) : "memory");
        }
        if (st == rows && vec && ok && !wait_cluster(turn, 0, abort_flag)) fail();
      }
      // operands of the step's end, in flight while the products run: rho_{j+1} or w_j, and the
      // next step's coupling L_{j+1} or U_{j-1}
      double2 nrho[NV];
      T nstg[NV], ncf = mk<T>(0, 0);
      if (vec) {
        if (st + 1 < nsteps) ncf = ia2f[st + 1 < rows ? j + 1 : j];
        if (st + 1 < rows) load_rho(j + 1, nrho);
        if (!fwd)
#pragma unroll
          for (int q = 0; q < NV; ++q)
            if (q < nlive) nstg[q] = __ldcg(stga + q * stg_stride + (int64_t)j * m);
      }
      // products of this warp's segments
#pragma unroll 1
      for (int c = 0; rd[c]; ++c) {
        const uint32_t item = myitems[c * SW];
        if (ok && !(K > 1 ? tc::bar_spin(&sf[slot], ph, abort_flag) : tc::bar_wait(&sf[slot], ph, abort_flag))) fail();
        if (item) {
          const int I0 = (int)(item & 31u), J = (int)(item >> 5 & 31u), n = (int)(item >> 10 & 3u);
          const int at = (int)(item >> 12 & 31u), seg = (int)(item >> 17);
          const S *tile = sring + (slot * ST + at) * TE;
          R *rowslot = slots + (J * (J + 1) / 2 + I0) * 32 + rplace, *colslot = slots + (nt + seg) * 32 + lane;
          // N tiles, the last one on the diagonal (which serves its rows only) or not
          auto products = [&](auto N_, auto diag_) {
            constexpr int N = decltype(N_)::value;
            constexpr bool DIAG = decltype(diag_)::value;
            // all tiles in registers, or one at a time (complex FP64; small CTAs with several right-hand
            // sides, whose 128 registers would spill: 576 boxes of 48, two sources 0.293 -> 0.25 ms)
            constexpr bool HOLD = sizeof(R) == 4 && !(SMALL && NR > 1);
            typename O::Ent t[HOLD ? N : 1][4][2];
            if (HOLD)
#pragma unroll
              for (int k = 0; k < N; ++k) load_tile(tile + k * TE, lane, t[k]);
#pragma unroll 1
            for (int q = 0; q < nq; ++q) {
              const T *vr = vsr + q * mpmax + I0 * TB, *vc = vsc + q * mpmax + J * TB;
              Vec vJ[4];
              O::load2(vc, vJ[0], vJ[1]);
              O::load2(vc + 2, vJ[2], vJ[3]);
              Acc cacc[4];
#pragma unroll
              for (int c4 = 0; c4 < 4; ++c4) cacc[c4] = O::zero();
              T rv[N][2];
#pragma unroll
              for (int k = 0; k < N; ++k) {
                if (!HOLD) load_tile(tile + k * TE, lane, t[0]);
                const auto &tk = t[HOLD ? k : 0];
                Acc r0a = O::zero(), r1a = O::zero();
#pragma unroll
                for (int c4 = 0; c4 < 4; ++c4) {
                  O::mac(r0a, tk[c4][0], vJ[c4]);
                  O::mac(r1a, tk[c4][1], vJ[c4]);
                }
                if (!DIAG || k + 1 < N) {
                  Vec v0, v1;
                  O::load2(vr + k * TB, v0, v1);
#pragma unroll
                  for (int c4 = 0; c4 < 4; ++c4) {
                    O::mac(cacc[c4], tk[c4][0], v0);
                    O::mac(cacc[c4], tk[c4][1], v1);
                  }
                }
                rv[k][0] = O::value(r0a);
                rv[k][1] = O::value(r1a);
              }
              R out[N];
#pragma unroll
              for (int k = 0; k < N; ++k) out[k] = reduce_rows(rv[k], lane);
              constexpr bool COLS = !DIAG || N > 1;   // (a diagonal tile on its own has no column sums)
              R oc = (R)0;
              if constexpr (COLS) {
                const T cv[4] = {O::value(cacc[0]), O::value(cacc[1]), O::value(cacc[2]), O::value(cacc[3])};
                oc = reduce_cols(cv, lane);
              }
#pragma unroll
              for (int k = 0; k < N; ++k) rowslot[q * qstride + k * 32] = out[k];
              if constexpr (COLS) colslot[q * qstride] = oc;
            }
          };
          using One = std::integral_constant<int, 1>;
          using Two = std::integral_constant<int, 2>;
          using Three = std::integral_constant<int, 3>;
          if (n == 3 && I0 + 2 < J) products(Three{}, std::false_type{});
          else if (n == 3) products(Three{}, std::true_type{});
          else if (sizeof(R) == 8 && n == 1 && I0 < J) products(One{}, std::false_type{});
          else if (n == 2) products(Two{}, std::true_type{});
          else products(One{}, std::true_type{});
        }
        // every value read from the stage has been used: the next copy may land
        __syncwarp();
        if (lane == 0) bar_arrive(&se[slot]);
        if (++slot == NS) { slot = 0; ph ^= 1u; }
      }
      asm volatile("bar.sync 1, %0;" ::"n"(CT) : "memory");   // every slot of this CTA's groups is written
      if (vec) {
        const int par = st & 1;
        T p[GPC][NV];   // the CTA's group sums
#pragma unroll
        for (int gi = 0; gi < GPC; ++gi) {
          const uint4 id = *reinterpret_cast<const uint4 *>(terms + (((int)rank * GPC + gi) * mt + A) * MAXTERM);
          const R *sl = slots + q0 * qstride + 2 * (a & 15);
          auto at = [&](uint32_t i, int q) { return *reinterpret_cast<const T *>(sl + q * qstride + i); };
          if constexpr (sizeof(R) == 4) {   // all loads first, the missing terms zero
#pragma unroll
            for (int q = 0; q < NV; ++q) {
              const T x0 = at(id.x & 0xFFFFu, q), x1 = at(id.x >> 16, q), x2 = at(id.y & 0xFFFFu, q), x3 = at(id.y >> 16, q);
              p[gi][q] = cadd(cadd(cadd(x0, x1), x2), x3);
            }
            if ((id.z & 0xFFFFu) != (uint32_t)(nt + map.nseg) * 32u)
#pragma unroll
              for (int q = 0; q < NV; ++q) {
                const T x0 = at(id.z & 0xFFFFu, q), x1 = at(id.z >> 16, q), x2 = at(id.w & 0xFFFFu, q), x3 = at(id.w >> 16, q);
                p[gi][q] = cadd(cadd(cadd(cadd(p[gi][q], x0), x1), x2), x3);
              }
          } else {                          // no addition that is not needed: the FP64 pipe is the bound
            const uint32_t w4[4] = {id.x, id.y, id.z, id.w};
#pragma unroll
            for (int q = 0; q < NV; ++q) p[gi][q] = at(id.x & 0xFFFFu, q);
#pragma unroll
            for (int i = 1; i < MAXTERM; ++i) {
              const uint32_t t = w4[i / 2] >> (16 * (i & 1)) & 0xFFFFu;
              if (t == (uint32_t)(nt + map.nseg) * 32u) break;
#pragma unroll
              for (int q = 0; q < NV; ++q) p[gi][q] = cadd(p[gi][q], at(t, q));
            }
          }
#pragma unroll
          for (int q = 0; q < NV; ++q)
#pragma unroll
            for (int d = 1; d < K; ++d)
              cluster_send(peer_pb[d] + (uint32_t)(((par * SYM_GROUPS + gi) * NR + q) * mpmax * (int)sizeof(T)),
                           p[gi][q], peer_bar[d] + (uint32_t)par * 8u);
        }
        if (K > 1 && tid == 0)
          asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(tc::su32(&xbar[par])),
                       "r"((uint32_t)((SYM_GROUPS - GPC) * NR * m * (int)sizeof(T)))
                       : "memory");
        const T ca = cmul(a1, ncf);   // entry a of the next step's L_{j+1} or U_{j-1}
        T rho[NV];
#pragma unroll
        for (int q = 0; q < NV; ++q)
          if (st + 1 < rows) rho[q] = mk<T>(from_d<R>(nrho[q].x), from_d<R>(nrho[q].y));
        if (K > 1 && ok && !wait_cluster(&xbar[par], (uint32_t)((st >> 1) & 1), abort_flag)) fail();
#pragma unroll
        for (int q = 0; q < NV; ++q) {
          T y = mk<T>(0, 0);
#pragma unroll
          for (int g = 0; g < SYM_GROUPS; ++g) {
            T t = mk<T>(0, 0);
            if (K == 1) {
              t = p[g % GPC][q];
            } else if (g / GPC == (int)rank) {
#pragma unroll
              for (int gi = 0; gi < GPC; ++gi)
                if (g % GPC == gi) t = p[gi][q];
            } else {
              t = pb[((size_t)(par * SYM_GROUPS + g) * NR + q0 + q) * mpmax + a];
            }
            y = g == 0 ? t : cadd(y, t);
          }
          const bool out = writer && q < nlive;
          T *stg = stga + q * stg_stride + (int64_t)j * m;
          if (fwd) {
            if (out) *stg = y;                                    // w_j
            vs[(q0 + q) * mpmax + a] = st + 1 < rows ? cfms(ca, y, rho[q])   // rho_{j+1} - L_{j+1} w_j
                                              : cmul(ca, y);          // U x_{rows-1}
          } else {
            // x_{j+1} goes out one step late: every CTA's sums of this step used w_{j+1}
            if (K > 1 && out && st > rows) stg[m] = x[q];
            const T xj = csub(nstg[q], y);
            if (K > 1) x[q] = xj;
            else if (out) *stg = xj;
            vs[(q0 + q) * mpmax + a] = cmul(ca, xj);                     // U_{j-1} x_j
          }
        }
      }
    }
    if (K > 1 && writer && rows > 1)
#pragma unroll
      for (int q = 0; q < NV; ++q)
        if (q < nlive) stga[q * stg_stride] = x[q];   // x_0
  }
  if (K > 1) {
    cluster_sync_all();   // no CTA leaves while another may still write into its shared memory
    // st.async is not ordered by the barrier.  Where no wait failed, every sum sent here has been
    // waited for; else some may still be on their way, and the CTA stays until they have landed
    if (*abort_flag) settle();
  }
}

// ---------------------------------------------------------------- launch
static int sm_count() {
  int dev = 0, sms = 152;
  if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return sms;
}

template <typename R> static const C<R> *lpool_of(const hd_ctx *ctx);
template <> const float2 *lpool_of<float>(const hd_ctx *ctx) { return ctx->d_lpoolf; }
template <> const double2 *lpool_of<double>(const hd_ctx *ctx) { return ctx->d_lpool; }

// Tiles of a segment in a launch whose widest box has mp rows: three, and one in complex FP64
// up to 64, where a step would wait for one warp's 192 FP64 instructions at 64 cycles each (4 boxes of
// 48 0.68 -> 0.38 ms, of 64 1.04 -> 0.58; at 96 the sums of so many column slots cost more: 1.64 -> 1.80).
template <typename R> static int sym_segment(int mp) { return sizeof(R) == 8 && mp <= 64 ? 1 : 3; }

template <typename R, typename S, int K, int P, int NR, int VG, int SW, int PER_SM>
static cudaError_t launch_sym(hd_ctx *ctx, const double2 *r, int nrhs, int64_t vec_stride, void *staging,
                              int64_t stg_stride, cudaStream_t st, int *depth) {
  using T = C<R>;
  const int mpmax = (ctx->max_m + TB - 1) / TB * TB;
  const int groups = (nrhs + NR - 1) / NR;
  int dev = 0, optin = 0, sm = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev);
  if (e != cudaSuccess) return e;
  if (PER_SM > 1) optin = std::min(optin, sm / PER_SM - 1024);   // (1 KB of every CTA's is the system's)
  // the ring takes what is left, two stages at least where a round of every warp allows it (large
  // CTAs of complex FP64, bound by their arithmetic: one), else fewer warps per round
  const int seg = sym_segment<R>(mpmax);
  int spr = SW, stiles = 0, ns = 0;
  for (; spr >= 1; --spr) {
    stiles = sym_stage_tiles(mpmax / TB, spr, seg);
    const size_t fixed = sym_smem<R, S>(0, stiles, spr, mpmax, K, P, NR, SW, seg).total;
    const size_t stage = (size_t)P * (stiles * TE * sizeof(S) + 2 * sizeof(uint64_t));
    ns = fixed < (size_t)optin ? (int)std::min<size_t>(16, ((size_t)optin - fixed) / stage) : 0;
    if (ns >= (PER_SM > 2 ? (spr > 1 ? 2 : 1) : (sizeof(R) == 4 && spr > 3 ? 2 : 1))) break;
  }
  if (spr < 1) return cudaErrorInvalidValue;
  if (depth) { *depth = ns; return cudaSuccess; }   // (asked for the ring's stages only)
  if (ctx->tune_ns > 0 && nrhs == 1) ns = std::min(ns, ctx->tune_ns);   // (what was tuned)
  const size_t smem = sym_smem<R, S>(ns, stiles, spr, mpmax, K, P, NR, SW, seg).total;
  auto kern = k_subst_sym<R, S, K, P, NR, VG, SW, PER_SM>;
  if ((e = allow_smem(kern, smem)) != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(groups * K), (unsigned)ctx->nsub);   // a box's source groups side by side share its factor reads in L2
  cfg.blockDim = dim3(P * SW * 32 + 32);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = K;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = K > 1 ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kern, (const SubDev *)ctx->d_subs, lpool_of<R>(ctx),
                            reinterpret_cast<const S *>(ctx->factor), r, ctx->NX, vec_stride,
                            reinterpret_cast<T *>(staging), stg_stride, nrhs, ns, stiles, spr, seg, mpmax, ctx->d_status);
}

static SymPick sym_pick(const hd_ctx *ctx, int nrhs) {
  return ctx->prec == HD_C128 ? sym_pick64(ctx->max_m, ctx->nsub, nrhs, sm_count())
                              : sym_pick32(ctx->max_m, ctx->nsub, nrhs, sm_count());
}

// Consumer threads of a single-source launch (what the autotuner reports).
int subst_sym_threads(const hd_ctx *ctx) {
  const SymPick p = sym_pick(ctx, 1);
  return p.P * p.SW * 32;
}

static cudaError_t launch_sym64(hd_ctx *ctx, const SymPick &p, const double2 *r, int nrhs, int64_t vs, void *stg, int64_t ss,
                                cudaStream_t st, int *depth) {
  using R = double;
  using S = double2;
  if (p.per_sm == 3) return launch_sym<R, S, 1, 1, 1, 1, 4, 3>(ctx, r, nrhs, vs, stg, ss, st, depth);
  if (p.per_sm > 2) return launch_sym<R, S, 1, 1, 1, 1, 3, 4>(ctx, r, nrhs, vs, stg, ss, st, depth);
  if (p.K == 4) return launch_sym<R, S, 4, 1, 1, 1, 8, 1>(ctx, r, nrhs, vs, stg, ss, st, depth);
  if (p.K == 2) return launch_sym<R, S, 2, 1, 1, 1, 8, 1>(ctx, r, nrhs, vs, stg, ss, st, depth);
  return p.per_sm == 2 ? launch_sym<R, S, 1, 1, 1, 1, 8, 2>(ctx, r, nrhs, vs, stg, ss, st, depth)
                       : launch_sym<R, S, 1, 1, 1, 1, 8, 1>(ctx, r, nrhs, vs, stg, ss, st, depth);
}

template <typename S, int NR>
static cudaError_t launch_sym32(hd_ctx *ctx, const SymPick &p, const double2 *r, int nrhs, int64_t vs, void *stg, int64_t ss,
                                cudaStream_t st, int *depth) {
  using R = float;
  constexpr int VG = NR > 1 ? 2 : 1;   // two sets have threads for two groups of vectors, if the box is no wider than one
  const bool wide = ctx->max_m > 224;
  if (p.per_sm > 2) return launch_sym<R, S, 1, 1, NR, 1, 3, 4>(ctx, r, nrhs, vs, stg, ss, st, depth);
  if (p.K == 4) return launch_sym<R, S, 4, 1, NR, 1, 7, 1>(ctx, r, nrhs, vs, stg, ss, st, depth);
  if (p.K == 2)
    return wide ? launch_sym<R, S, 2, 2, NR, 1, 7, 1>(ctx, r, nrhs, vs, stg, ss, st, depth)
                : launch_sym<R, S, 2, 2, NR, VG, 7, 1>(ctx, r, nrhs, vs, stg, ss, st, depth);
  return wide ? launch_sym<R, S, 1, 2, NR, 1, 7, 1>(ctx, r, nrhs, vs, stg, ss, st, depth)
              : launch_sym<R, S, 1, 2, NR, VG, 7, 1>(ctx, r, nrhs, vs, stg, ss, st, depth);
}
template <typename S>
static cudaError_t launch_sym_nr(hd_ctx *ctx, const SymPick &p, const double2 *r, int nrhs, int64_t vs, void *stg, int64_t ss,
                                 cudaStream_t st, int *depth) {
  return p.NR == 4   ? launch_sym32<S, 4>(ctx, p, r, nrhs, vs, stg, ss, st, depth)
         : p.NR == 2 ? launch_sym32<S, 2>(ctx, p, r, nrhs, vs, stg, ss, st, depth)
                     : launch_sym32<S, 1>(ctx, p, r, nrhs, vs, stg, ss, st, depth);
}

static cudaError_t launch_pick(hd_ctx *ctx, const double2 *r, int nrhs, int64_t vec_stride, void *staging, int64_t stg_stride,
                               cudaStream_t st, int *depth) {
  const SymPick p = sym_pick(ctx, nrhs);
  switch (ctx->prec) {
    case HD_C64: return launch_sym_nr<float2>(ctx, p, r, nrhs, vec_stride, staging, stg_stride, st, depth);
    case HD_C64_H: return launch_sym_nr<__half2>(ctx, p, r, nrhs, vec_stride, staging, stg_stride, st, depth);
    case HD_C64_B: return launch_sym_nr<__nv_bfloat162>(ctx, p, r, nrhs, vec_stride, staging, stg_stride, st, depth);
    default: return launch_sym64(ctx, p, r, nrhs, vec_stride, staging, stg_stride, st, depth);
  }
}

cudaError_t launch_subst_sym(hd_ctx *ctx, const double2 *r, int nrhs, int64_t vec_stride, void *staging,
                             int64_t stg_stride, cudaStream_t st) {
  return launch_pick(ctx, r, nrhs, vec_stride, staging, stg_stride, st, nullptr);
}

// Ring stages of a single-source launch: the most the autotuner has to choose from.
int subst_sym_stages(hd_ctx *ctx) {
  int depth = 0;
  return launch_pick(ctx, nullptr, 1, 0, nullptr, 0, nullptr, &depth) == cudaSuccess ? depth : 0;
}

}  // namespace hd
