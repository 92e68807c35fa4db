// uf_stripe.cu -- the Striped UniFrac accumulation (paper Sec. 2-3, Figs. 1-3).
//
// For every branch e of a launch, stripe s and sample k the paper adds
// f(emb_e[k], emb_e[(k + s + 1) mod n]) * length_e into the stripe buffer.
// Here the per-branch term is rewritten (exact algebra; the finalize kernel
// states it per method):
//   |u - v| = u + v - 2 min(u, v),  [a xor b] = a + b - 2 ab,  [a or b] = a + b - ab,
// so with x = l * u (l * presence for unweighted) every weighted and
// unweighted numerator and denominator follows from the diagonal
// D[k] = sum_e x_e[k] and, per cell, either
//   M[s][k] = sum_e min(x_e[k], x_e[k + s + 1])        (min form) or
//   A[s][k] = sum_e |x_e[k] - x_e[k + s + 1]|          (abs form).
// One min-form update is one FMNMX (ALU pipe, half rate) plus half an FADD2;
// one abs-form update is half an FSUB2 plus one FADD (FMA pipe).  The FP32
// kernel gives stripes 1, 3, 5 and 7 of every 8 the abs form so the two pipes
// share the load (odd micro-tile rows read their partner pairs at even,
// register-pair aligned offsets).  The FP64 path's rows are 64-bit fixed
// point, and its kernel (k_stripe_u64) adds R = sum max(x_j - x_k, 0) in
// integers, A = 2 R + D_k - D_j: GB300 has 2 FP64 lanes per clock per SM but
// 64 integer ones, and integer sums are exact, so the only rounding is that
// of a row's value to the grid, and no difference of two sums cancels.  Where
// that grid is too coarse for some sample's branches (grid_need) the rows are
// FP64 values, all in the abs form.  Generalized UniFrac keeps two
// accumulators, den = sum l s^a and, FP32, Q = sum l min(u, v) s^(a-1) with
// num = den - 2Q or, FP64, N = sum l |u - v| s^(a-1) = num.
//
// Work is split into units (row chunk of up to a.chunk branches, tile of
// TILE_S stripes x TILE_K samples).  Persistent CTAs take units from a global
// counter, chunk-major, so the CTAs in flight read the same rows and those
// rows stay in L2.  Per unit, stages of rows (FP32: 16 rows, two stages;
// FP64: 8 rows, three stages) of the u window [k0, k0 + TILE_K) and the
// partner window [k0 + s0, k0 + s0 + TILE_K + TILE_S) go to shared memory by
// 16-byte cp.async while the previous stage is computed, and each thread
// updates an RD x RK register micro-tile.  Shared rows are XOR-swizzled in
// 16-byte units so the per-thread 16-byte reads are free of bank conflicts.
//
// Precision (the kernels on FP32 and FP64 rows).  Register partials over
// B1 = 64 branches are summed into a
// second level kept in shared memory in the path's own precision (FP32 for
// the paper's fp32 mode, Sec. 4, FP64 otherwise); at the end of the unit that
// level is scaled by 2^F and rounded once to an int64 fixed-point value (FP64:
// two words, the second holding the remainder at 2^-32 of the first's step),
// which is added atomically into the int64 accumulator.  Integer addition is
// exact and order-free, so chunks may land in any order and the result is
// still deterministic; every cell (and the diagonal) runs the same FP32 /
// FP64 operation sequence within a unit, so two identical samples give
// bitwise equal accumulators and a distance of exactly 0 (an abs-form cell
// adds |x - x| = 0 exactly).
// F is chosen by the host from an upper bound B on any accumulated value so
// that 2 B 2^F <= 2^61.
#include <algorithm>
#include <cfloat>
#include <type_traits>

#include "uf_device.cuh"

namespace ufg {

namespace {

// Threads of a CTA: TX (stripe) x TX (sample), TX = 16 or, for small problems,
// 8 (tiles of a quarter of the cells: less padding and more units in flight).
constexpr int B1 = 64;        // inner partial length (branches)

// Shared rows are stored in 16-byte units with unit j placed at
// j ^ ((j >> 3) & MASK), MASK = (bytes a thread reads per 8-sample run) / 16 - 1.
// Eight threads that read the same unit offset q of consecutive 8-sample runs
// (any starting run) then hit eight distinct 16-byte bank groups.
template <typename T>
__host__ __device__ constexpr int swz(int elem) {
  constexpr int VEC = 16 / sizeof(T);
  constexpr int MASK = 8 * sizeof(T) / 16 - 1;
  const int j = elem / VEC;
  return (j ^ ((j >> 3) & MASK)) * VEC + elem % VEC;
}

template <typename T, int RD, int RK, int NACC, int TX>
struct Geo {
  static constexpr int NT = TX * TX;
  // branch rows per pipeline stage and cp.async stages: FP32 16 rows in two
  // stages (half the block barriers of 8-row stages), FP64 8 rows in three
  static constexpr int RB = sizeof(T) == 4 ? 16 : 8;
  static constexpr int NSTAGE = sizeof(T) == 4 ? 2 : 3;
  static constexpr int TS = TX * RD;             // stripes per tile
  static constexpr int TK = TX * RK;             // samples per tile
  static constexpr int VEC = 16 / sizeof(T);     // elements per 16-byte copy
  static constexpr int UW = TK;                  // u window
  static constexpr int VW = TK + TS;             // partner window (needs TK + TS - 1, shifted by one)
  static constexpr int ROW = UW + VW;            // both parts are multiples of 128 bytes
  static constexpr int STAGE = RB * ROW + RB;    // + the rows' lengths (keeps 16-byte alignment)
  static constexpr int UCH = UW / VEC, VCH = VW / VEC, CH = UCH + VCH;
  static constexpr int NV = (RD + RK + VEC - 1) / VEC;  // partner vectors per thread
  // second level per thread and cell, in the path's precision
  using Mid = T;
  static constexpr size_t SMEM =
      (size_t)NSTAGE * STAGE * sizeof(T) + (size_t)NACC * RD * RK * NT * sizeof(Mid);
};

__device__ __forceinline__ void cp_async16(void *smem, const void *gmem) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory"); }

// a - b on a register pair (one packed FP32 subtract)
__device__ __forceinline__ float2 fsub2(float2 a, float2 b) {
  unsigned long long ra, rb, rr;
  asm("mov.b64 %0, {%1, %2};" : "=l"(ra) : "f"(a.x), "f"(a.y));
  asm("mov.b64 %0, {%1, %2};" : "=l"(rb) : "f"(b.x), "f"(b.y));
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(rr) : "l"(ra), "l"(rb));
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(rr));
  return r;
}

struct Unit {
  int r0, r1;       // branch rows
  int k0, s0;       // tile origin: first sample, first stripe
  int n, s_lo, s_hi;
  int64_t x_col;    // the table's first column in an embedding row
  int64_t m_off;    // the table's first accumulator cell
};

// Table holding tile number tt of the batch (tables in order of tile0).
__device__ __forceinline__ int table_of_tile(const TabDesc *tabs, int n_tabs, int tt) {
  int lo = 0, hi = n_tabs - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (tabs[mid].tile0 <= tt) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

// Next work unit for this CTA: chunk-major over (row chunk, tile of any table).
__device__ __forceinline__ bool next_unit(const StripeArgs &a, int tile_s, int tile_k, int *s_unit,
                                          Unit *u) {
  __syncthreads();  // everyone is done with the previous unit's shared data
  if (threadIdx.x == 0) *s_unit = atomicAdd(a.counter, 1);
  __syncthreads();
  const int id = *s_unit;
  const int n_chunks = (a.rows + a.chunk - 1) / a.chunk;
  if (id >= n_chunks * a.n_tiles) return false;
  const int c = id / a.n_tiles, tt = id - c * a.n_tiles;
  const TabDesc &tb = a.tabs[a.n_tabs == 1 ? 0 : table_of_tile(a.tabs, a.n_tabs, tt)];
  const int t = tt - tb.tile0;
  // bands of kband sample tiles: all stripe tiles of a band, then the next band
  const int n_st = tb.m_hi - tb.m_lo + 1;
  const int kb = max(1, min(tb.kband, tb.n_ktiles));
  const int band = t / (kb * n_st), within = t - band * (kb * n_st);
  const int width = min(kb, tb.n_ktiles - band * kb);
  const int kt = band * kb + within % width, st = within / width;
  u->r0 = c * a.chunk;
  u->r1 = min(a.rows, u->r0 + a.chunk);
  u->k0 = kt * tile_k;
  u->s0 = (tb.m_lo + st) * tile_s;
  u->n = tb.n;
  u->s_lo = tb.s_lo;
  u->s_hi = tb.s_hi;
  u->x_col = tb.x_col;
  u->m_off = tb.m_off;
  return true;
}

// Stage loader: G::RB branch rows [e0, e0 + G::RB) of the u window (columns from
// ucol) and the partner window (columns from vcol).
template <typename T, int RD, int RK, int NACC, int TX, bool LEN>
__device__ __forceinline__ void load_stage(T *stage, const StripeArgs &a, int e0, int e_end, int64_t ucol,
                                           int64_t vcol) {
  using G = Geo<T, RD, RK, NACC, TX>;
  const T *X = (const T *)a.X;
  for (int c = threadIdx.x; c < G::RB * G::CH; c += G::NT) {
    const int r = c / G::CH, q = c - r * G::CH;
    T *row = stage + r * G::ROW;
    const int e = e0 + r;
    T *dst;
    int64_t src;
    if (q < G::UCH) {
      dst = row + swz<T>(q * G::VEC);
      src = ucol + q * G::VEC;
    } else {
      const int qv = q - G::UCH;
      dst = row + G::UW + swz<T>(qv * G::VEC);
      src = vcol + qv * G::VEC;
    }
    if (e < e_end) {
      cp_async16(dst, X + (int64_t)e * a.pitch + src);
    } else {
      // rows past the unit: zero, or for FP32 proportions the embedding's
      // 1e-30 floor (their length is 0, so they add nothing either way)
      const T pad = (LEN && sizeof(T) == 4) ? T(1e-30f) : T(0);
#pragma unroll
      for (int i = 0; i < G::VEC; i++) dst[i] = pad;
    }
  }
  if (LEN && threadIdx.x < G::RB) {
    const int e = e0 + threadIdx.x;
    stage[G::RB * G::ROW + threadIdx.x] = e < e_end ? (T)a.len[e] : T(0);
  }
}

// Add one thread's second-level cells (fixed point) into the accumulator.
template <typename T, int RD, int RK, int TX, typename Mid>
__device__ __forceinline__ void commit_cells(unsigned long long *M, const Mid *mid, const StripeArgs &a,
                                             const Unit &U, int s_base, int k_base) {
#pragma unroll
  for (int i = 0; i < RD; i++) {
    const int s = s_base + i;
    if (s < U.s_lo || s > U.s_hi) continue;
    unsigned long long *row = M + U.m_off + (int64_t)(s - U.s_lo) * U.n;
#pragma unroll
    for (int j = 0; j < RK; j++) {
      const int k = k_base + j;
      if (k < U.n) {
        const Fx2 q = to_fixed2(mid[(i * RK + j) * (TX * TX) + threadIdx.x], a.scale);
        atomicAdd(row + k, (unsigned long long)q.hi);
        if constexpr (sizeof(T) == 8) atomicAdd(row + k + a.m_lo_off, (unsigned long long)q.lo);
      }
    }
  }
}

// ---- weighted / unweighted on FP32 and FP64 rows ----
// rows i of the micro-tile with bit i of ABSM clear: M += min(x_k, x_j);
// with it set: A += |x_k - x_j| (FP64: every row)
template <typename T, int RD, int RK, int TX, unsigned ABSM, int MINB>
__global__ void __launch_bounds__(TX *TX, MINB) k_stripe_min(const StripeArgs a) {
  using G = Geo<T, RD, RK, 1, TX>;
  constexpr int NT = G::NT;
  using Mid = typename G::Mid;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T *stg = reinterpret_cast<T *>(smem_raw);
  Mid *mid = reinterpret_cast<Mid *>(smem_raw + (size_t)G::NSTAGE * G::STAGE * sizeof(T));
  __shared__ int s_unit;
  const int tk = threadIdx.x % TX, ts = threadIdx.x / TX;
  const int w0 = RK * tk + RD * ts;  // partner window of this thread, used from w0 + 1
  Unit U;
  while (next_unit(a, G::TS, G::TK, &s_unit, &U)) {
#pragma unroll
    for (int c = 0; c < RD * RK; c++) mid[c * NT + threadIdx.x] = Mid(0);
    const int nst = (U.r1 - U.r0 + G::RB - 1) / G::RB;
#pragma unroll
    for (int p = 0; p < G::NSTAGE - 1; p++) {
      if (p < nst) load_stage<T, RD, RK, 1, TX, false>(stg + p * G::STAGE, a, U.r0 + p * G::RB, U.r1, U.x_col + U.k0,
                                        U.x_col + U.k0 + U.s0);
      cp_async_commit();
    }
    T acc[RD][RK];
#pragma unroll
    for (int i = 0; i < RD; i++)
#pragma unroll
      for (int j = 0; j < RK; j++) acc[i][j] = T(0);
    int in_sub = 0;
    for (int it = 0; it < nst; it++) {
      cp_async_wait<G::NSTAGE - 2>();
      __syncthreads();
      {
        const int nx = it + G::NSTAGE - 1;
        if (nx < nst)
          load_stage<T, RD, RK, 1, TX, false>(stg + (nx % G::NSTAGE) * G::STAGE, a, U.r0 + nx * G::RB, U.r1,
                                          U.x_col + U.k0, U.x_col + U.k0 + U.s0);
        cp_async_commit();
      }
      const T *stage = stg + (it % G::NSTAGE) * G::STAGE;
      // the whole stage unrolled: 3 % faster than two rows per iteration in
      // a micro-benchmark of the FP32 kernel (fewer loop and address
      // instructions, more freedom to interleave the ALU and FMA pipes)
#pragma unroll
      for (int r = 0; r < G::RB; r++) {
        const T *urow = stage + r * G::ROW;
        const T *vrow = urow + G::UW;
        T u[RK], v[G::NV * G::VEC];
#pragma unroll
        for (int q = 0; q < RK / G::VEC; q++)
          *reinterpret_cast<uint4 *>(&u[q * G::VEC]) =
              *reinterpret_cast<const uint4 *>(urow + swz<T>(RK * tk + q * G::VEC));
#pragma unroll
        for (int q = 0; q < G::NV; q++)
          *reinterpret_cast<uint4 *>(&v[q * G::VEC]) =
              *reinterpret_cast<const uint4 *>(vrow + swz<T>(w0 + q * G::VEC));
        if constexpr (sizeof(T) == 8) {
          // two FP64 instructions per update on 2 lanes per clock per SM bound
          // it: 2.58e11 updates/s on 2,048 samples (k_stripe_u64 3.61e12)
          static_assert(ABSM == FP64_ABS_ROW_MASK);
#pragma unroll
          for (int i = 0; i < RD; i++)
#pragma unroll
            for (int j = 0; j < RK; j++) acc[i][j] += fabs(u[j] - v[i + j + 1]);
        } else {
#pragma unroll
          for (int i = 0; i < RD; i++)
#pragma unroll
            for (int j = 0; j < RK; j += 2) {
              if (!((ABSM >> i) & 1u)) {  // two mins, one paired add
                float2 a2 = make_float2(acc[i][j], acc[i][j + 1]);
                const float2 m2 = make_float2(fminf(u[j], v[i + j + 1]), fminf(u[j + 1], v[i + j + 2]));
                a2 = __fadd2_rn(a2, m2);
                acc[i][j] = a2.x;
                acc[i][j + 1] = a2.y;
              } else {  // one paired difference, one paired add of absolute values
                const float2 d2 = fsub2(make_float2(u[j], u[j + 1]), make_float2(v[i + j + 1], v[i + j + 2]));
                float2 a2 = make_float2(acc[i][j], acc[i][j + 1]);
                a2 = __fadd2_rn(a2, make_float2(fabsf(d2.x), fabsf(d2.y)));
                acc[i][j] = a2.x;
                acc[i][j + 1] = a2.y;
              }
            }
        }
      }
      in_sub += G::RB;
      if (in_sub == B1 || it == nst - 1) {
#pragma unroll
        for (int i = 0; i < RD; i++)
#pragma unroll
          for (int j = 0; j < RK; j++) {
            mid[(i * RK + j) * NT + threadIdx.x] += acc[i][j];
            acc[i][j] = T(0);
          }
        in_sub = 0;
      }
    }
    cp_async_wait<0>();
    commit_cells<T, RD, RK, TX>(a.M, mid, a, U, U.s0 + RD * ts, U.k0 + RK * tk);
  }
}

// ---- weighted / unweighted, FP64 on 64-bit fixed-point rows ----
// c += max(v - u, 0) for u, v < 2^63: a 64-bit difference, a test of its sign
// and a predicated 64-bit add, 5 integer instructions.
__device__ __forceinline__ void add_relu(unsigned long long &c, unsigned long long u, unsigned long long v) {
  asm("{\n .reg .pred p;\n .reg .u32 u0, u1, v0, v1, c0, c1, d0, d1;\n"
      " mov.b64 {u0, u1}, %1;\n mov.b64 {v0, v1}, %2;\n mov.b64 {c0, c1}, %0;\n"
      " sub.cc.u32 d0, v0, u0;\n subc.u32 d1, v1, u1;\n setp.ge.s32 p, d1, 0;\n"
      " @p add.cc.u32 c0, c0, d0;\n @p addc.u32 c1, c1, d1;\n mov.b64 %0, {c0, c1};\n}\n"
      : "+l"(c)
      : "l"(u), "l"(v));
}

// Integer pipe bound: 5 instructions per update at 64 lanes per clock per SM
// is 12.8 updates per clock; in a loop over resident rows this form reaches
// 14.7 (some of the adds issue elsewhere), the 64-bit min 12.6, the FP64 form
// |u - v| 0.8.  The sums stay in registers for the whole unit (they are exact,
// so there is no second level) and go to the two-word accumulators at its end.
template <int RD, int RK, int TX, int MINB>
__global__ void __launch_bounds__(TX *TX, MINB) k_stripe_u64(const StripeArgs a) {
  using T = unsigned long long;
  using G = Geo<T, RD, RK, 0, TX>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T *stg = reinterpret_cast<T *>(smem_raw);
  __shared__ int s_unit;
  const int tk = threadIdx.x % TX, ts = threadIdx.x / TX;
  const int w0 = RK * tk + RD * ts;
  Unit U;
  while (next_unit(a, G::TS, G::TK, &s_unit, &U)) {
    const int nst = (U.r1 - U.r0 + G::RB - 1) / G::RB;
#pragma unroll
    for (int p = 0; p < G::NSTAGE - 1; p++) {
      if (p < nst) load_stage<T, RD, RK, 0, TX, false>(stg + p * G::STAGE, a, U.r0 + p * G::RB, U.r1, U.x_col + U.k0,
                                        U.x_col + U.k0 + U.s0);
      cp_async_commit();
    }
    T acc[RD][RK];
#pragma unroll
    for (int i = 0; i < RD; i++)
#pragma unroll
      for (int j = 0; j < RK; j++) acc[i][j] = 0;
    for (int it = 0; it < nst; it++) {
      cp_async_wait<G::NSTAGE - 2>();
      __syncthreads();
      {
        const int nx = it + G::NSTAGE - 1;
        if (nx < nst)
          load_stage<T, RD, RK, 0, TX, false>(stg + (nx % G::NSTAGE) * G::STAGE, a, U.r0 + nx * G::RB, U.r1,
                                          U.x_col + U.k0, U.x_col + U.k0 + U.s0);
        cp_async_commit();
      }
      const T *stage = stg + (it % G::NSTAGE) * G::STAGE;
#pragma unroll 2
      for (int r = 0; r < G::RB; r++) {
        const T *urow = stage + r * G::ROW;
        const T *vrow = urow + G::UW;
        T u[RK], v[G::NV * G::VEC];
#pragma unroll
        for (int q = 0; q < RK / G::VEC; q++)
          *reinterpret_cast<uint4 *>(&u[q * G::VEC]) =
              *reinterpret_cast<const uint4 *>(urow + swz<T>(RK * tk + q * G::VEC));
#pragma unroll
        for (int q = 0; q < G::NV; q++)
          *reinterpret_cast<uint4 *>(&v[q * G::VEC]) =
              *reinterpret_cast<const uint4 *>(vrow + swz<T>(w0 + q * G::VEC));
#pragma unroll
        for (int i = 0; i < RD; i++)
#pragma unroll
          for (int j = 0; j < RK; j++) add_relu(acc[i][j], u[j], v[i + j + 1]);
      }
    }
    cp_async_wait<0>();
    // 2 R as hi (units of 2^-F) and lo (2^-(F+32)) words
    const unsigned long long mask = (1ull << a.x_shift) - 1ull;
#pragma unroll
    for (int i = 0; i < RD; i++) {
      const int s = U.s0 + RD * ts + i;
      if (s < U.s_lo || s > U.s_hi) continue;
      unsigned long long *row = a.M + U.m_off + (int64_t)(s - U.s_lo) * U.n;
#pragma unroll
      for (int j = 0; j < RK; j++) {
        const int k = U.k0 + RK * tk + j;
        if (k >= U.n || acc[i][j] == 0) continue;
        atomicAdd(row + k, (acc[i][j] >> a.x_shift) << 1);
        atomicAdd(row + k + a.m_lo_off, (acc[i][j] & mask) << (33 - a.x_shift));
      }
    }
  }
}

// ---- generalized: den += l s w and, FP32, Q += l min(u, v) w or, FP64,
//      N += l |u - v| w, with w = s^(alpha - 1) ----
template <typename T, int RD, int RK, int TX, int MODE, int MINB>
__global__ void __launch_bounds__(TX *TX, MINB) k_stripe_gen(const StripeArgs a) {
  using G = Geo<T, RD, RK, 2, TX>;
  constexpr int NT = G::NT;
  using Mid = typename G::Mid;
  constexpr bool F32 = sizeof(T) == 4;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T *stg = reinterpret_cast<T *>(smem_raw);
  Mid *midd = reinterpret_cast<Mid *>(smem_raw + (size_t)G::NSTAGE * G::STAGE * sizeof(T));
  Mid *midq = midd + RD * RK * NT;
  __shared__ int s_unit;
  const int tk = threadIdx.x % TX, ts = threadIdx.x / TX;
  const int w0 = RK * tk + RD * ts;
  const T am1 = (T)(a.alpha - 1.0);
  Unit U;
  while (next_unit(a, G::TS, G::TK, &s_unit, &U)) {
#pragma unroll
    for (int c = 0; c < RD * RK; c++) midd[c * NT + threadIdx.x] = midq[c * NT + threadIdx.x] = Mid(0);
    const int nst = (U.r1 - U.r0 + G::RB - 1) / G::RB;
#pragma unroll
    for (int p = 0; p < G::NSTAGE - 1; p++) {
      if (p < nst) load_stage<T, RD, RK, 2, TX, true>(stg + p * G::STAGE, a, U.r0 + p * G::RB, U.r1, U.x_col + U.k0,
                                       U.x_col + U.k0 + U.s0);
      cp_async_commit();
    }
    T accd[RD][RK], accq[RD][RK];
#pragma unroll
    for (int i = 0; i < RD; i++)
#pragma unroll
      for (int j = 0; j < RK; j++) accd[i][j] = accq[i][j] = T(0);
    int in_sub = 0;
    for (int it = 0; it < nst; it++) {
      cp_async_wait<G::NSTAGE - 2>();
      __syncthreads();
      {
        const int nx = it + G::NSTAGE - 1;
        if (nx < nst)
          load_stage<T, RD, RK, 2, TX, true>(stg + (nx % G::NSTAGE) * G::STAGE, a, U.r0 + nx * G::RB, U.r1,
                                         U.x_col + U.k0, U.x_col + U.k0 + U.s0);
        cp_async_commit();
      }
      const T *stage = stg + (it % G::NSTAGE) * G::STAGE;
#pragma unroll 1
      for (int r = 0; r < G::RB; r++) {
        const T *urow = stage + r * G::ROW;
        const T *vrow = urow + G::UW;
        const T l = stage[G::RB * G::ROW + r];
        T u[RK], v[G::NV * G::VEC];
#pragma unroll
        for (int q = 0; q < RK / G::VEC; q++)
          *reinterpret_cast<uint4 *>(&u[q * G::VEC]) =
              *reinterpret_cast<const uint4 *>(urow + swz<T>(RK * tk + q * G::VEC));
#pragma unroll
        for (int q = 0; q < G::NV; q++)
          *reinterpret_cast<uint4 *>(&v[q * G::VEC]) =
              *reinterpret_cast<const uint4 *>(vrow + swz<T>(w0 + q * G::VEC));
        if constexpr (F32) {
          // pairs of cells per f32x2 instruction; the embedding keeps every
          // proportion >= 1e-30 (an offset no nonzero FP32 proportion can see),
          // so s > 0: for alpha = 1/2 an absent pair adds l sqrt(2e-30) to den
          // and exactly half of that to Q (net 0 to num), for other alpha its
          // term is zeroed explicitly
          const float2 l2 = make_float2(l, l);
#pragma unroll
          for (int i = 0; i < RD; i++)
#pragma unroll
            for (int j = 0; j < RK; j += 2) {
              const float2 uu = make_float2(u[j], u[j + 1]);
              const float2 vv = make_float2(v[i + j + 1], v[i + j + 2]);
              const float2 s2 = __fadd2_rn(uu, vv);
              float2 r2 = make_float2(sfu_pow<MODE>(s2.x, am1), sfu_pow<MODE>(s2.y, am1));
              if (MODE == 1) {  // s^(alpha-1) of an absent pair (s = 2e-30) must not count
                r2.x = s2.x > 4e-30f ? r2.x : 0.f;
                r2.y = s2.y > 4e-30f ? r2.y : 0.f;
              }
              const float2 w2 = __fmul2_rn(l2, r2);
              const float2 m2 = make_float2(fminf(uu.x, vv.x), fminf(uu.y, vv.y));
              float2 d2 = make_float2(accd[i][j], accd[i][j + 1]);
              float2 q2 = make_float2(accq[i][j], accq[i][j + 1]);
              d2 = __ffma2_rn(s2, w2, d2);
              q2 = __ffma2_rn(m2, w2, q2);
              accd[i][j] = d2.x;
              accd[i][j + 1] = d2.y;
              accq[i][j] = q2.x;
              accq[i][j + 1] = q2.y;
            }
        } else {
#pragma unroll
          for (int i = 0; i < RD; i++)
#pragma unroll
            for (int j = 0; j < RK; j++) {
              const T uu = u[j], vv = v[i + j + 1];
              const T s = uu + vv;
              T w = l * gen_pow<T, MODE>(s, am1);
              if (MODE == 1) w = s > T(0) ? w : T(0);
              accd[i][j] = fma(s, w, accd[i][j]);
              accq[i][j] = fma(fabs(uu - vv), w, accq[i][j]);
            }
        }
      }
      in_sub += G::RB;
      if (in_sub == B1 || it == nst - 1) {
#pragma unroll
        for (int i = 0; i < RD; i++)
#pragma unroll
          for (int j = 0; j < RK; j++) {
            const int c = (i * RK + j) * NT + threadIdx.x;
            midd[c] += accd[i][j];
            midq[c] += accq[i][j];
            accd[i][j] = accq[i][j] = T(0);
          }
        in_sub = 0;
      }
    }
    cp_async_wait<0>();
    commit_cells<T, RD, RK, TX>(a.M, midd, a, U, U.s0 + RD * ts, U.k0 + RK * tk);
    commit_cells<T, RD, RK, TX>(a.M2, midq, a, U, U.s0 + RD * ts, U.k0 + RK * tk);
  }
}

// ---- variance-adjusted weighted (Chang, Luan & Sun 2011):
//      den += w (u + v), N += w |u - v|, w = 1 / sqrt((c_k + c_j)(r_k + r_j))
//      with u = l p the length-scaled proportions, c the counts below the
//      branch and r = T - c, and w = 0 where either factor is 0 ----
// Rows hold three planes (u, c, r) of `pitch` elements each.  A stage carries
// RB rows of all three planes; the micro-tile is RD x RK with two
// accumulators per cell.
template <typename T, int RD, int RK, int TX>
struct GeoV {
  static constexpr int NT = TX * TX;
  static constexpr int RB = sizeof(T) == 4 ? 8 : 4;  // rows per stage
  static constexpr int NSTAGE = 2;
  static constexpr int NPL = 3;                       // planes: u, c, r
  static constexpr int TS = TX * RD, TK = TX * RK;
  static constexpr int VEC = 16 / sizeof(T);
  static constexpr int UW = TK, VW = TK + TS, ROW = UW + VW;
  static constexpr int STAGE = RB * NPL * ROW;  // rows past the unit are zero (w = 0)
  static constexpr int UCH = UW / VEC, VCH = VW / VEC, CH = UCH + VCH;
  static constexpr int NV = (RD + RK + VEC - 1) / VEC;
  static constexpr size_t SMEM = (size_t)NSTAGE * STAGE * sizeof(T) + (size_t)2 * RD * RK * NT * sizeof(T);
  // Shared-memory position of row element `elem`.  A quarter-warp reads eight
  // 16-byte chunks: consecutive ones for FP32 (RK = 4 floats per chunk), which
  // hit eight distinct bank groups unswizzled (the swizzle of the 8 x 8 tile
  // would put two of them on one group whenever the run starts at an odd
  // chunk); every second one for FP64, which the swizzle spreads.
  static __device__ __forceinline__ int at(int elem) { return sizeof(T) == 4 ? elem : swz<T>(elem); }
};

template <typename T, int RD, int RK, int TX>
__device__ __forceinline__ void load_stage_vaw(T *stage, const StripeArgs &a, int e0, int e_end, int64_t ucol,
                                               int64_t vcol) {
  using G = GeoV<T, RD, RK, TX>;
  const T *X = (const T *)a.X;
  for (int c = threadIdx.x; c < G::RB * G::NPL * G::CH; c += G::NT) {
    const int rp = c / G::CH, q = c - rp * G::CH;  // rp = row * NPL + plane
    const int r = rp / G::NPL, pl = rp - r * G::NPL;
    T *row = stage + rp * G::ROW;
    const int e = e0 + r;
    T *dst;
    int64_t src;
    if (q < G::UCH) {
      dst = row + G::at(q * G::VEC);
      src = ucol + q * G::VEC;
    } else {
      const int qv = q - G::UCH;
      dst = row + G::UW + G::at(qv * G::VEC);
      src = vcol + qv * G::VEC;
    }
    if (e < e_end) {
      cp_async16(dst, X + ((int64_t)e * G::NPL + pl) * a.pitch + src);
    } else {
#pragma unroll
      for (int i = 0; i < G::VEC; i++) dst[i] = T(0);
    }
  }
}

template <typename T>
__device__ __forceinline__ T vaw_weight(T prod);
template <>
__device__ __forceinline__ float vaw_weight<float>(float prod) {
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(prod));
  return prod > 0.f ? r : 0.f;
}
template <>
__device__ __forceinline__ double vaw_weight<double>(double prod) {
  return prod > 0.0 ? rsqrt(prod) : 0.0;
}

template <typename T, int RD, int RK, int TX, int MINB>
__global__ void __launch_bounds__(TX *TX, MINB) k_stripe_vaw(const StripeArgs a) {
  using G = GeoV<T, RD, RK, TX>;
  constexpr int NT = G::NT;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T *stg = reinterpret_cast<T *>(smem_raw);
  T *midd = reinterpret_cast<T *>(smem_raw + (size_t)G::NSTAGE * G::STAGE * sizeof(T));
  T *midn = midd + RD * RK * NT;
  __shared__ int s_unit;
  const int tk = threadIdx.x % TX, ts = threadIdx.x / TX;
  const int w0 = RK * tk + RD * ts;
  Unit U;
  while (next_unit(a, G::TS, G::TK, &s_unit, &U)) {
#pragma unroll
    for (int c = 0; c < RD * RK; c++) midd[c * NT + threadIdx.x] = midn[c * NT + threadIdx.x] = T(0);
    const int nst = (U.r1 - U.r0 + G::RB - 1) / G::RB;
    if (nst > 0)
      load_stage_vaw<T, RD, RK, TX>(stg, a, U.r0, U.r1, U.x_col + U.k0, U.x_col + U.k0 + U.s0);
    cp_async_commit();
    T accd[RD][RK], accn[RD][RK];
#pragma unroll
    for (int i = 0; i < RD; i++)
#pragma unroll
      for (int j = 0; j < RK; j++) accd[i][j] = accn[i][j] = T(0);
    int in_sub = 0;
    for (int it = 0; it < nst; it++) {
      cp_async_wait<0>();
      __syncthreads();
      if (it + 1 < nst)
        load_stage_vaw<T, RD, RK, TX>(stg + ((it + 1) % G::NSTAGE) * G::STAGE, a, U.r0 + (it + 1) * G::RB, U.r1,
                                  U.x_col + U.k0, U.x_col + U.k0 + U.s0);
      cp_async_commit();
      const T *stage = stg + (it % G::NSTAGE) * G::STAGE;
#pragma unroll 1
      for (int r = 0; r < G::RB; r++) {
        T u[3][RK], v[3][G::NV * G::VEC];
#pragma unroll
        for (int pl = 0; pl < 3; pl++) {
          const T *urow = stage + (r * G::NPL + pl) * G::ROW;
          const T *vrow = urow + G::UW;
#pragma unroll
          for (int q = 0; q < RK / G::VEC; q++)
            *reinterpret_cast<uint4 *>(&u[pl][q * G::VEC]) =
                *reinterpret_cast<const uint4 *>(urow + G::at(RK * tk + q * G::VEC));
#pragma unroll
          for (int q = 0; q < G::NV; q++)
            *reinterpret_cast<uint4 *>(&v[pl][q * G::VEC]) =
                *reinterpret_cast<const uint4 *>(vrow + G::at(w0 + q * G::VEC));
        }
        if constexpr (sizeof(T) == 4) {
          // pairs of cells per f32x2 instruction (the weight's reciprocal
          // square roots stay scalar, on the SFU)
#pragma unroll
          for (int i = 0; i < RD; i++)
#pragma unroll
            for (int j = 0; j < RK; j += 2) {
              const float2 uu = make_float2(u[0][j], u[0][j + 1]);
              const float2 vv = make_float2(v[0][i + j + 1], v[0][i + j + 2]);
              // the two samples' counts below the branch, and the rest of their totals
              const float2 mv = __fadd2_rn(make_float2(u[1][j], u[1][j + 1]),
                                           make_float2(v[1][i + j + 1], v[1][i + j + 2]));
              const float2 rest = __fadd2_rn(make_float2(u[2][j], u[2][j + 1]),
                                             make_float2(v[2][i + j + 1], v[2][i + j + 2]));
              const float2 prod = __fmul2_rn(mv, rest);
              const float2 w = make_float2(vaw_weight<float>(prod.x), vaw_weight<float>(prod.y));
              const float2 s2 = __fadd2_rn(uu, vv);
              const float2 d2 = fsub2(uu, vv);
              float2 ad = make_float2(accd[i][j], accd[i][j + 1]);
              float2 an = make_float2(accn[i][j], accn[i][j + 1]);
              ad = __ffma2_rn(s2, w, ad);
              an = __ffma2_rn(make_float2(fabsf(d2.x), fabsf(d2.y)), w, an);
              accd[i][j] = ad.x;
              accd[i][j + 1] = ad.y;
              accn[i][j] = an.x;
              accn[i][j + 1] = an.y;
            }
        } else {
#pragma unroll
          for (int i = 0; i < RD; i++)
#pragma unroll
            for (int j = 0; j < RK; j++) {
              const T uu = u[0][j], vv = v[0][i + j + 1];
              const T mv = u[1][j] + v[1][i + j + 1];  // the two samples' counts below the branch
              const T rest = u[2][j] + v[2][i + j + 1];  // and the rest of their totals
              const T w = vaw_weight<T>(mv * rest);
              accd[i][j] = fma(uu + vv, w, accd[i][j]);
              accn[i][j] = fma(fabs(uu - vv), w, accn[i][j]);
            }
        }
      }
      in_sub += G::RB;
      if (in_sub >= B1 || it == nst - 1) {
#pragma unroll
        for (int i = 0; i < RD; i++)
#pragma unroll
          for (int j = 0; j < RK; j++) {
            const int c = (i * RK + j) * NT + threadIdx.x;
            midd[c] += accd[i][j];
            midn[c] += accn[i][j];
            accd[i][j] = accn[i][j] = T(0);
          }
        in_sub = 0;
      }
    }
    cp_async_wait<0>();
    commit_cells<T, RD, RK, TX>(a.M, midd, a, U, U.s0 + RD * ts, U.k0 + RK * tk);
    commit_cells<T, RD, RK, TX>(a.M2, midn, a, U, U.s0 + RD * ts, U.k0 + RK * tk);
  }
}

// ---- diagonal: D[k] += sum_e x_e[k], with the operation sequence a stripe
//      cell in min form runs when its two columns are equal ----
// Phase 1: one partial per (B1-row sub-block, sample), summed in row order;
// sub-blocks restart at every chunk boundary, as in the stripe kernels.
// Table holding combined sample column k (tables in order of off).
__device__ __forceinline__ int table_of_col(const TabDesc *tabs, int n_tabs, int k) {
  int lo = 0, hi = n_tabs - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (tabs[mid].off <= k) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

template <typename T>
__global__ void k_diag_partial(const StripeArgs a, T *__restrict__ part) {
  const int kg = blockIdx.x * blockDim.x + threadIdx.x;
  if (kg >= a.n_cols) return;
  const TabDesc &tb = a.tabs[a.n_tabs == 1 ? 0 : table_of_col(a.tabs, a.n_tabs, kg)];
  const int64_t k = tb.x_col + (kg - tb.off);  // the sample's column in its segment
  const int sb = blockIdx.y;
  const T *X = (const T *)a.X;
  const int per_chunk = (a.chunk + B1 - 1) / B1;
  const int c = sb / per_chunk;
  const int e0 = c * a.chunk + (sb - c * per_chunk) * B1;
  const int e1 = min(min(a.rows, (c + 1) * a.chunk), e0 + B1);
  T acc = T(0);
  for (int e = e0; e < e1; e++) {
    const T x = X[(int64_t)e * a.pitch + k];
    acc += tmin<T>(x, x);
  }
  part[(int64_t)sb * a.n_cols + kg] = acc;
}

// Phase 2: a chunk's sub-block partials summed in order in the rows' precision,
// then rounded to fixed point (the stripe kernels' second level); blockIdx.y is
// the chunk, whose integers add in any order.
template <typename T>
__global__ void k_diag_reduce(const StripeArgs a, const T *__restrict__ part, int n_sb) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= a.n_cols) return;
  const int per_chunk = (a.chunk + B1 - 1) / B1;
  const int sb0 = blockIdx.y * per_chunk, sb1 = min(n_sb, sb0 + per_chunk);
  T mid = T(0);
#pragma unroll 8
  for (int sb = sb0; sb < sb1; sb++) mid += part[(int64_t)sb * a.n_cols + k];
  const Fx2 d = to_fixed2(mid, a.scale);
  atomicAdd(a.Dg + k, (unsigned long long)d.hi);
  if constexpr (sizeof(T) == 8) atomicAdd(a.Dg + k + a.d_lo_off, (unsigned long long)d.lo);
}

// FP64: the fixed-point rows' sums, each value split into its two words
// (one thread per column and DIAG_ROWS rows, integers in any order).
constexpr int DIAG_ROWS = 64;
__global__ void k_diag_u64(const StripeArgs a) {
  const int kg = blockIdx.x * blockDim.x + threadIdx.x;
  if (kg >= a.n_cols) return;
  const TabDesc &tb = a.tabs[a.n_tabs == 1 ? 0 : table_of_col(a.tabs, a.n_tabs, kg)];
  const unsigned long long *X = (const unsigned long long *)a.X + tb.x_col + (kg - tb.off);
  const int e0 = blockIdx.y * DIAG_ROWS, e1 = min(a.rows, e0 + DIAG_ROWS);
  const unsigned long long mask = (1ull << a.x_shift) - 1ull;
  unsigned long long hi = 0, lo = 0;  // lo < DIAG_ROWS * 2^32
#pragma unroll 4
  for (int e = e0; e < e1; e++) {
    const unsigned long long x = X[(int64_t)e * a.pitch];
    hi += x >> a.x_shift;
    lo += (x & mask) << (32 - a.x_shift);
  }
  if (hi) atomicAdd(a.Dg + kg, hi);
  if (lo) atomicAdd(a.Dg + kg + a.d_lo_off, lo);
}

// A persistent launch: as many CTAs as fit (or units, if fewer), after the
// unit counter is reset.
template <typename K>
cudaError_t run_units(K kernel, int threads, size_t smem, const StripeArgs &a, cudaStream_t st) {
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  int per_sm = 0, dev = 0, sms = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, smem);
  if (e != cudaSuccess) return e;
  e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  const int n_chunks = (a.rows + a.chunk - 1) / a.chunk, units = n_chunks * a.n_tiles;
  const int grid = std::max(1, std::min(units, std::max(per_sm, 1) * sms));
  e = cudaMemsetAsync(a.counter, 0, sizeof(int), st);
  if (e != cudaSuccess) return e;
  return launch_k(kernel, dim3(grid), dim3(threads), smem, st, a);
}

template <typename T, int RD, int RK, int TX, unsigned ABSM, int MINB>
cudaError_t run_min(const StripeArgs &a, cudaStream_t st) {
  return run_units(k_stripe_min<T, RD, RK, TX, ABSM, MINB>, TX * TX, Geo<T, RD, RK, 1, TX>::SMEM, a, st);
}
template <int RD, int RK, int TX, int MINB>
cudaError_t run_u64(const StripeArgs &a, cudaStream_t st) {
  return run_units(k_stripe_u64<RD, RK, TX, MINB>, TX * TX, Geo<unsigned long long, RD, RK, 0, TX>::SMEM, a, st);
}
template <typename T, int RD, int RK, int TX, int MINB>
cudaError_t run_vaw(const StripeArgs &a, cudaStream_t st) {
  return run_units(k_stripe_vaw<T, RD, RK, TX, MINB>, TX * TX, GeoV<T, RD, RK, TX>::SMEM, a, st);
}
template <typename T, int RD, int RK, int TX, int MODE, int MINB>
cudaError_t run_gen(const StripeArgs &a, cudaStream_t st) {
  return run_units(k_stripe_gen<T, RD, RK, TX, MODE, MINB>, TX * TX, Geo<T, RD, RK, 2, TX>::SMEM, a, st);
}

}  // namespace

// Shapes of (accumulator, precision): micro-tiles of the FP32 min kernel 8 x 8
// (shape 1: 4 x 8 at three CTAs per SM, 64-stripe tiles that waste fewer
// stripes of small tables), FP64 min kernel 4 x 8 (64-bit sums at two CTAs per
// SM), generalized 4 x 8 (two accumulators), variance-adjusted 4 x 4 (two
// accumulators, three planes), all on 16 x 16 threads; the last shape of each
// is the small one, 8 x 8 threads of a 4 x 8 (4 x 4) micro-tile.
int stripe_small_shape(int acc, bool fp32) { return acc == ACC_MIN && fp32 ? 2 : 1; }

void stripe_tile_shape(int acc, bool fp32, int *tile_s, int *tile_k, int shape) {
  const bool min8 = acc == ACC_MIN && fp32, small = shape == stripe_small_shape(acc, fp32);
  *tile_s = small ? 32 : (min8 && shape == 0 ? 128 : 64);
  *tile_k = acc == ACC_VAW ? (small ? 32 : 64) : (small ? 64 : 128);
}

int stripe_shapes(int acc, bool fp32, unsigned abs_mask) {
  return acc == ACC_MIN && fp32 && abs_mask != 0xFFu ? 2 : 1;
}

int stripe_chunk_rows() { return 2048; }

SmallPlan stripe_small_plan(int acc, bool fp32, bool fixed, const int *n, size_t n_tabs, int rows, int chunk,
                            int shape, bool shape_free, int sms) {
  const bool fp64 = !fp32 && !fixed;  // bound by the FP64 pipe
  auto tiles_of = [&](int sh, int64_t *cells) {
    int ts = 0, tk = 0;
    stripe_tile_shape(acc, fp32, &ts, &tk, sh);
    int64_t t = 0;
    for (size_t i = 0; i < n_tabs; i++) t += (int64_t)((n[i] / 2 + ts - 1) / ts) * ((n[i] + tk - 1) / tk);
    *cells = t * ts * tk;
    return t;
  };
  SmallPlan p{shape, chunk, false};
  int64_t cells = 0;
  int64_t tiles = tiles_of(shape, &cells);
  const int small = stripe_small_shape(acc, fp32);
  if (shape_free && shape != small) {
    // the small tiles stage twice the bytes per update; updates on FP64 rows
    // are bound by the FP64 pipe either way
    const double rate = fp64 ? 1.0 : 0.85;
    int64_t cells_s = 0;
    const int64_t tiles_s = tiles_of(small, &cells_s);
    if ((double)cells_s < rate * (double)cells) {
      p.shape = small;
      tiles = tiles_s;
    }
  }
  // units in flight: CTAs of 256 threads run two per SM (FP64 rows: one), the
  // small ones eight
  const int64_t slots = (int64_t)sms * (p.shape == small ? 8 : fp64 ? 1 : 2), want = 4 * slots;
  // kernels whose chunk is tuned are cut only where the smallest candidate
  // leaves under two waves (1,003 samples generalized, three waves of tuned
  // units: cut to four they took 2 % longer)
  const bool tuned = !fixed;
  const int64_t least = tuned ? std::min(chunk, 1024) : chunk;
  if (tiles > 0 && tiles * ((rows + least - 1) / least) < (tuned ? 2 * slots : want)) {
    // (launch_diag's sub-blocks of B1 rows restart at every chunk)
    const int step = acc == ACC_MIN && !fixed ? B1 : 16;
    const int64_t c = ((int64_t)rows * tiles / want + step) / step * step;
    p.chunk = (int)std::min<int64_t>(chunk, std::max<int64_t>(c, step));
    p.split = true;
  }
  return p;
}

cudaError_t launch_stripe_acc(int acc, bool fp32, const StripeArgs &a, cudaStream_t st) {
  if (a.rows <= 0 || a.n_tiles <= 0) return cudaSuccess;
  if (acc == ACC_MIN) {
    if (!fp32 && a.fixed) return a.shape == 1 ? run_u64<4, 8, 8, 8>(a, st) : run_u64<4, 8, 16, 2>(a, st);
    if (!fp32)
      return a.shape == 1 ? run_min<double, 4, 8, 8, FP64_ABS_ROW_MASK, 4>(a, st)
                          : run_min<double, 4, 8, 16, FP64_ABS_ROW_MASK, 1>(a, st);
    if (a.abs_mask == 0xFFu)
      return a.shape == 2 ? run_min<float, 4, 8, 8, 0xFFu, 8>(a, st) : run_min<float, 8, 8, 16, 0xFFu, 2>(a, st);
    if (a.shape == 2) return run_min<float, 4, 8, 8, FP32_ABS_ROW_MASK, 8>(a, st);
    return a.shape == 1 ? run_min<float, 4, 8, 16, FP32_ABS_ROW_MASK, 3>(a, st)
                        : run_min<float, 8, 8, 16, FP32_ABS_ROW_MASK, 2>(a, st);
  }
  const bool small = a.shape == 1;
  if (acc == ACC_VAW) {
    if (fp32) return small ? run_vaw<float, 4, 4, 8, 8>(a, st) : run_vaw<float, 4, 4, 16, 2>(a, st);
    return small ? run_vaw<double, 4, 4, 8, 4>(a, st) : run_vaw<double, 4, 4, 16, 1>(a, st);
  }
  const bool half = a.alpha == 0.5;
  if (fp32) {
    if (small) return half ? run_gen<float, 4, 8, 8, 0, 8>(a, st) : run_gen<float, 4, 8, 8, 1, 8>(a, st);
    return half ? run_gen<float, 4, 8, 16, 0, 2>(a, st) : run_gen<float, 4, 8, 16, 1, 2>(a, st);
  }
  if (small) return half ? run_gen<double, 4, 8, 8, 0, 4>(a, st) : run_gen<double, 4, 8, 8, 1, 4>(a, st);
  return half ? run_gen<double, 4, 8, 16, 0, 1>(a, st) : run_gen<double, 4, 8, 16, 1, 1>(a, st);
}

size_t diag_scratch_bytes(bool fp32, bool fixed, int rows, int n_cols) {
  if (fixed) return 0;
  // one sub-block of B1 rows after another (chunks are multiples of B1)
  const int64_t n_sb = (rows + B1 - 1) / B1;
  return (size_t)std::max<int64_t>(n_sb, 1) * n_cols * (fp32 ? 4 : 8);
}

cudaError_t launch_diag(bool fp32, const StripeArgs &a, void *scratch, cudaStream_t st) {
  if (a.rows <= 0) return cudaSuccess;
  const int gx = (a.n_cols + 127) / 128;
  if (a.fixed)
    return launch_k(k_diag_u64, dim3(gx, (a.rows + DIAG_ROWS - 1) / DIAG_ROWS), dim3(128), 0, st, a);
  const int per_chunk = (a.chunk + B1 - 1) / B1;
  const int n_chunks = (a.rows + a.chunk - 1) / a.chunk;
  const int n_sb = (n_chunks - 1) * per_chunk + ((a.rows - (n_chunks - 1) * a.chunk) + B1 - 1) / B1;
  auto both = [&](auto partial, auto reduce, auto *part) {
    const cudaError_t e = launch_k(partial, dim3(gx, n_sb), dim3(128), 0, st, a, part);
    return e != cudaSuccess ? e : launch_k(reduce, dim3(gx, n_chunks), dim3(128), 0, st, a, part, n_sb);
  };
  return fp32 ? both(k_diag_partial<float>, k_diag_reduce<float>, (float *)scratch)
              : both(k_diag_partial<double>, k_diag_reduce<double>, (double *)scratch);
}

}  // namespace ufg
