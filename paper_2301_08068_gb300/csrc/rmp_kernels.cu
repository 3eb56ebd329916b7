// rmp_kernels.cu -- sm_103a kernels of librmp: the fused raycast-RMP evaluation, the
// LiDAR scan policy and the map-build kernels.
//
// One evaluation is ONE launch: each thread generates its ray's Halton direction in
// registers (Sec. III-E, Eq. halton), marches it with an exact fixed-point DDA (Sec. III-F)
// that crosses the map free box by free box, evaluates the obstacle policy (Sec. III-C), and the block reduces the
// 9 unique terms of sum A_i and sum A_i f_i (Fig. 3's block reduce) with a compensated
// FP32 tree (or FP64).  CTA 0 sums the per-CTA partials in a fixed order and resolves Eq. (1) (FP32 Jacobi eigenvectors refined by FP64 Rayleigh
// quotients, FP64 adjugate solve at full rank), so the result is deterministic.
//
// Bit-exact steps (Halton direction, DDA, hit distance, the FP32 decisions that gate a
// ray) use explicitly rounded intrinsics (__fmul_rn, __fmaf_rn, ...) so that no
// contraction or fast-math rewrite can change them.
#include <algorithm>
#include <climits>
#include <cstddef>
#include <type_traits>

#include "rmp_internal.h"

namespace rmp {
namespace {

// ------------------------------------------------------------------ Halton directions
// Radical inverse base 2 of i, rounded to FP32 (exact for i < 2^24).
__device__ __forceinline__ float halton2(uint32_t i) {
  return __fmul_rn(__uint2float_rn(__brev(i)), 2.3283064365386963e-10f);  // * 2^-32
}

// The 16 base-3 digits of i (< 2^24 < 3^16) reversed: H(i,3) * 3^16.
template <int DIGITS>
__device__ __forceinline__ uint32_t reverse3(uint32_t i) {
  uint32_t num = 0;
#pragma unroll
  for (int k = 0; k < DIGITS; ++k) {
    const uint32_t q = i / 3u;
    num = num * 3u + (i - 3u * q);
    i = q;
  }
  return num;
}

// The reversed digits of every 5-digit number.
struct Reverse5 {
  uint8_t v[243];
  constexpr Reverse5() : v() {
    for (int i = 0; i < 243; ++i) {
      int num = 0, q = i;
      for (int k = 0; k < 5; ++k) {
        num = num * 3 + q % 3;
        q /= 3;
      }
      v[i] = (uint8_t)num;
    }
  }
};
__device__ const Reverse5 kReverse5;

// TABLE: three lookups of 5 digits and the last digit (25 instructions for 75; the batch kernel,
// which is bound by instructions and keeps the table in L1); else two halves of 8 digits whose
// chains run side by side (one evaluation, bound by latency, would wait for the table).
template <bool TABLE>
__device__ __forceinline__ uint32_t halton3_numerator(uint32_t i) {
  if (TABLE) {
    const uint32_t q1 = i / 243u, q2 = i / 59049u, q3 = i / 14348907u;
    return __ldg(&kReverse5.v[i - 243u * q1]) * 177147u +
           __ldg(&kReverse5.v[q1 - 243u * q2]) * 729u +
           __ldg(&kReverse5.v[q2 - 243u * q3]) * 3u + q3;
  }
  const uint32_t hi = i / 6561u;
  return reverse3<8>(i - 6561u * hi) * 6561u + reverse3<8>(hi);
}

// num / 3^16 (num < 3^16) correctly rounded to FP32: the quotient of num 2^s, s such that it has
// exactly 24 significant bits, from an FP32 product a few units off, set right by its exact
// remainder (within 2^28, so 32-bit arithmetic holds it); rounded to nearest on the remainder (no
// ties: 3^16 is odd).  FP64 division and a 64-bit integer division are slower on this GPU.
__device__ __forceinline__ float halton3_f32(uint32_t num) {
  if (num == 0) return 0.0f;
  constexpr uint32_t M = 43046721u;
  constexpr float rM = 1.0f / 43046721.0f;
  const int t = __clz(num) - 6;
  const int s = t + ((num << t) >= M ? 23 : 24);
  int q = __float2int_rn(__fmul_rn(__fmul_rn(__uint2float_rn(num), rM), __int_as_float((127 + s) << 23)));
  int rem = (int)((uint32_t)((unsigned long long)num << s) - (uint32_t)q * M);
  const int adj = __float2int_rn(__fmul_rn(__int2float_rn(rem), rM));
  rem -= adj * (int)M;
  q += adj + (2 * rem > (int)M ? 1 : 0) - (2 * rem < -(int)M ? 1 : 0);
  return __fmul_rn(__int2float_rn(q), __int_as_float((127 - s) << 23));
}

// cos and sin of 2*pi*v by a fixed FP32 recipe: octant q = floor(8v), fraction t,
// reduced angle a = x * RN(pi/4) (x = t, or 1 - t in odd octants), Taylor series of
// sin (through a^11) and cos (through a^12) with RN(1/n!) coefficients by Horner's rule
// with fused multiply-adds, then the octant's symmetry.
__device__ __forceinline__ void sincos_turns(float v, float& c_out, float& s_out) {
  constexpr float kPi4 = 0.78539816339744830962f;
  constexpr float f2 = 1.0f / 2.0f, f3 = 1.0f / 6.0f, f4 = 1.0f / 24.0f, f5 = 1.0f / 120.0f,
                  f6 = 1.0f / 720.0f, f7 = 1.0f / 5040.0f, f8 = 1.0f / 40320.0f,
                  f9 = 1.0f / 362880.0f, f10 = 1.0f / 3628800.0f, f11 = 1.0f / 39916800.0f,
                  f12 = 1.0f / 479001600.0f;
  const float w = __fmul_rn(v, 8.0f);
  const int q = __float2int_rz(w);
  const float t = __fsub_rn(w, __int2float_rn(q));
  const float x = (q & 1) ? __fsub_rn(1.0f, t) : t;
  const float a = __fmul_rn(x, kPi4);
  const float a2 = __fmul_rn(a, a);
  float ps = -f11;
  ps = __fmaf_rn(ps, a2, f9);
  ps = __fmaf_rn(ps, a2, -f7);
  ps = __fmaf_rn(ps, a2, f5);
  ps = __fmaf_rn(ps, a2, -f3);
  const float sa = __fmaf_rn(__fmul_rn(a2, a), ps, a);
  float pc = f12;
  pc = __fmaf_rn(pc, a2, -f10);
  pc = __fmaf_rn(pc, a2, f8);
  pc = __fmaf_rn(pc, a2, -f6);
  pc = __fmaf_rn(pc, a2, f4);
  pc = __fmaf_rn(pc, a2, -f2);
  const float ca = __fmaf_rn(a2, pc, 1.0f);
  const int o = q & 7;
  // octant o: angle = o*pi/4 + (t pi/4); odd octants measure a from the next multiple
  const bool swap = ((o + 1) & 2) != 0;          // octants 1,2,5,6: cos <-> sin
  float c = swap ? sa : ca;
  float s = swap ? ca : sa;
  if (o >= 2 && o <= 5) c = -c;                  // cos < 0 in octants 2..5
  if (o >= 4) s = -s;                            // sin < 0 in octants 4..7
  c_out = c;
  s_out = s;
}

struct Ray {
  float dir[3];
  int D[3];
};

template <bool TABLE>
__device__ __forceinline__ Ray make_ray(uint32_t i) {
  const float u = halton2(i);
  const float v = halton3_f32(halton3_numerator<TABLE>(i));
  const float z = __fsub_rn(1.0f, __fmul_rn(2.0f, u));
  const float st = __fmul_rn(2.0f, __fsqrt_rn(__fmul_rn(u, __fsub_rn(1.0f, u))));
  float c, s;
  sincos_turns(v, c, s);
  Ray r;
  r.dir[0] = __fmul_rn(st, c);
  r.dir[1] = __fmul_rn(st, s);
  r.dir[2] = z;
#pragma unroll
  for (int a = 0; a < 3; ++a) r.D[a] = __float2int_rn(__fmul_rn(r.dir[a], 16777216.0f));
  return r;
}

// ------------------------------------------------------------------ launch order
// Kernels that follow one another on a stream are launched with programmatic serialisation:
// each waits for its predecessor's completion, memory included, before it reads or writes
// anything but its parameters and constants (wait_previous), and lets its successor become
// resident once all its own CTAs have called launch_next -- after its own wait, so that no more
// than one launch is ahead, and late where CTAs waiting for the next launch would take up SMs
// unevenly (256 CTAs on the 304 to 456 places of a single evaluation: after the march; with the
// call at the start the ESDF policy of 4096 states took 27 us for 23).  The order of effects is
// the stream's; what overlaps is the launch itself and work on parameters alone: back to back,
// 1024 rays 12.4 -> 9.8 us, a batch of one state 26.5 -> 21.7 us.
// Such a kernel is resident while its predecessor still writes, so what a launch can write --
// states, counts, points, set-up records -- is read by plain loads only: the read-only path
// (__ldg, const __restrict__ parameters) is for data that does not change while the kernel runs,
// and its loads may be moved above the wait.  Maps and primitives stay on it: an upload is
// complete before any launch that uses it.
__device__ __forceinline__ void wait_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void launch_next() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// ------------------------------------------------------------------ small arithmetic
// 1 / x to an ulp or so; infinity for 0.
__device__ __forceinline__ float recip_fast(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

// x / d and x % d for x < 2^24 and a quotient below 2^19 (error of the FP32 product below 1/8):
// the product set right by its remainder.
__device__ __forceinline__ uint32_t divide24(uint32_t x, uint32_t d, uint32_t& rem) {
  int q = __float2int_rz(__uint2float_rn(x) * recip_fast(__uint2float_rn(d)));
  int r = (int)x - q * (int)d;
  if (r < 0) {
    q -= 1;
    r += (int)d;
  } else if (r >= (int)d) {
    q += 1;
    r -= (int)d;
  }
  rem = (uint32_t)r;
  return (uint32_t)q;
}

// ------------------------------------------------------------------ map access
// Index of the block's brick, or -1 where it is missing or free; `slot`: its place in the box
// field.
__device__ __forceinline__ int hash_lookup(const DevMap& m, int bx, int by, int bz,
                                           uint32_t& slot) {
  const unsigned long long key = (unsigned long long)(uint32_t)(bx + kKeyBias) |
                                 ((unsigned long long)(uint32_t)(by + kKeyBias) << 21) |
                                 ((unsigned long long)(uint32_t)(bz + kKeyBias) << 42);
  uint32_t h = (uint32_t)((key * 0x9E3779B97F4A7C15ull) >> m.hash_shift);
  for (uint32_t probe = 0; probe <= m.cap_mask; ++probe) {   // bounded: table has empties
    const unsigned long long k = __ldg(&m.table[h].key);
    if (k == key) {
      slot = __ldg(&m.table[h].box);
      return (int)__ldg(&m.table[h].slot);
    }
    if (k == kEmptyKey) return -1;
    h = (h + 1) & m.cap_mask;
  }
  return -1;
}

// ------------------------------------------------------------------ exact DDA (raycast R)
// Fixed point: P in 2^-16 voxel units, D in 2^-24 units.  N_a = distance (in P units) to the
// next boundary of axis a; the ray reaches it at t_a = N_a / |D_a|.  A voxel-by-voxel DDA
// steps the axis with the smallest t_a (exact rationals; ties go to the lowest axis); an
// axis with D_a = 0 never wins.  A voxel is entered only if N_a 2^24 <= R_fx |D_a|.
//
// The march reproduces that walk box by box.  Every voxel of an occupied block (and every
// free block) has, for each of the 8 octants of ray directions, a free box that starts at
// the voxel (block) and extends 1, 2, 4 or 8 voxels (blocks) forward along each axis,
// grown greedily at upload (box_field_kernel): a ray of that octant stays in the box until
// it crosses one of the box's three far faces, so one step of exact integer arithmetic
// takes it to the first voxel beyond.  One byte says whether the voxel is occupied and, if
// not, how far the box reaches, so the march needs neither the bricks nor a voxel walk:
// on the 40 m map a ray takes 4.2 boxes on average instead of 114 voxels, and the longest
// of a warp's 32 rays 6.8 (22 at most over 16 states), where a box of equal sides needs
// up to 60 along a wall.
//
// Reflected frame.  Axes the ray descends are mirrored (k -> ~k), so every ray climbs; the
// frame's origin is the grid's first block in that direction.  Voxel q_a, block q_a >> 3,
// voxel in its block q_a & 7; q_a and N_a grow together, one voxel and 2^16 a crossing.
constexpr int kSegContinues = 0;   // piece ended at its upper parameter bound
constexpr int kGridLog = 7;        // pieces of a ray are cut at multiples of R / 2^kGridLog

struct RayFx {
  int q0[3];                // start voxel, reflected frame
  uint32_t N0[3], A[3];     // its N_a; |D_a|
  uint32_t up;              // bit a: D_a > 0 (not mirrored); the octant of the box field
};

struct MarchState {
  int q[3];                 // voxel, reflected frame
  uint32_t N[3];
  uint32_t n_last, a_last;  // entry numerator / |D| of the current voxel (0/1 at the start)
  int ax_last;              // axis of the last step (for map exits)
};

// First block of axis a in the reflected frame's direction, as a mirrored block coordinate.
template <int LAYOUT>
__device__ __forceinline__ int frame_lo(const DevMap& m, int a, bool up) {
  if (LAYOUT != kLayoutGrid) return 0;
  return up ? m.gmin[a] : -(m.gmin[a] + m.gdim[a]);
}

__device__ __forceinline__ int unmirror(int q, int lo, bool up) {
  const int k = q + 8 * lo;
  return up ? k : ~k;
}

template <int LAYOUT>
__device__ __forceinline__ void ray_fx(const DevMap& m, const long long P[3], const int D[3],
                                       RayFx& r) {
  r.up = 0;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const bool up = D[a] > 0;
    const int k = (int)(P[a] >> 16), lo = frame_lo<LAYOUT>(m, a, up);
    r.up |= up ? 1u << a : 0u;
    r.q0[a] = (up ? k : ~k) - 8 * lo;
    r.A[a] = (uint32_t)abs(D[a]);
    const uint32_t frac = (uint32_t)P[a] & 0xffffu;
    // D_a = 0 is mirrored like a descending axis; N_a >= 1 keeps it from ever winning
    r.N0[a] = up ? 65536u - frac : (D[a] == 0 ? frac + 1u : frac);
  }
}

// Pieces of a ray.  The parameter range (0, R], R = R_fx / 2^24 voxel units, is cut at the
// points T_j = j R / 2^kGridLog; a piece covers (T_lo, T_hi] between two of them.  A crossing
// numerator n of axis a satisfies n / |D_a| <= T_j iff n 2^(24 + kGridLog) <= j R_fx |D_a|, so
// a piece's start state and its limits L_a (the crossings with t <= T_hi are those with
// N_a <= L_a) are integer functions of j.  Pieces of one ray can be marched by different
// threads at once; the ray's result is the first piece (in t) that hit or left the map, else
// the last piece.  With R_fx <= 2^30 and |D_a| <= 2^24 every product stays below 2^62.
__device__ __forceinline__ void limits_at(const RayFx& r, long long R_fx, uint32_t j, uint32_t L[3]) {
#pragma unroll
  for (int a = 0; a < 3; ++a)
    L[a] = (uint32_t)(((unsigned long long)j * (unsigned long long)R_fx * r.A[a]) >> (24 + kGridLog));
}

// State after every crossing with t <= T_j: per axis the count of boundaries N0_a + 2^16 m
// (m >= 0) within the bound; the entry of the current voxel is the latest of the axes' last
// crossings (at equal times the highest axis, which the single steps take last).
__device__ __forceinline__ void piece_start(const RayFx& r, long long R_fx, uint32_t j,
                                            MarchState& st) {
  st.n_last = 0;
  st.a_last = 1;
  st.ax_last = 0;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    st.q[a] = r.q0[a];
    st.N[a] = r.N0[a];
  }
  if (j == 0) return;
  bool any = false;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const unsigned long long X = (unsigned long long)j * (unsigned long long)R_fx * r.A[a];
    const unsigned long long Y = (unsigned long long)r.N0[a] << (24 + kGridLog);
    if (r.A[a] != 0 && X >= Y) {
      const uint32_t cnt = (uint32_t)((X - Y) >> (40 + kGridLog)) + 1;
      const uint32_t nl = r.N0[a] + ((cnt - 1) << 16);
      if (!any || (unsigned long long)nl * st.a_last >= (unsigned long long)st.n_last * r.A[a]) {
        st.n_last = nl;
        st.a_last = r.A[a];
        st.ax_last = a;
      }
      any = true;
      st.q[a] += (int)cnt;
      st.N[a] += cnt << 16;
    }
  }
}

// Crossings of axis p (numerator N, |D_p| = A) that the box step takes before the exit axis's
// face crossing F / E: #{m >= 0 : (N + 2^16 m) E < F A} (`le`: <=, when p is the lower axis, the
// tie order) = 1 + floor(num / (2^16 E)) with num = F A - N E (- 1 unless `le`), and, floors
// nesting, = 1 + floor((num >> 16) / E).  A box extends at most 64 voxels, so the quotient is at
// most 64 and num >> 16 below 2^30 in size; the quotient comes from an FP32 product (rE = 1 / E
// to an ulp or two, error below 2^-15) and is set right by its exact remainder.  No crossing
// (num >= -2^16 E, as N is at most 2^16 from the last one) gives 0; D_p = 0 is held to 0.
__device__ __forceinline__ int crossings_before(uint32_t F, uint32_t E, float rE, uint32_t N,
                                                uint32_t A, bool le) {
  const long long num = (long long)((unsigned long long)F * A) -
                        (long long)((unsigned long long)N * E) - (le ? 0 : 1);
  const int nh = (int)(num >> 16);
  int c = __float2int_rd(__int2float_rn(nh) * rE);
  const int rem = nh - c * (int)E;
  c += rem < 0 ? 0 : (rem >= (int)E ? 2 : 1);
  return max(c, 0);
}

// One block's entry for the ray's octant: bit 31 set = the block holds an occupied voxel (the
// low bits: its slot in the box field), else the log2 extents of the free box of blocks
// starting there, 2 bits per axis.  `brick`: where its occupancy bits are.
template <int LAYOUT, bool BOXES>
__device__ __forceinline__ uint32_t block_entry(const DevMap& m, const uint32_t* top,
                                                const int step[4], const int b[3], uint32_t up,
                                                const uint32_t*& brick) {
  if (LAYOUT == kLayoutGrid) {
    const int idx = b[0] * step[0] + b[1] * step[1] + b[2] * step[2];
    if (!BOXES) brick = reinterpret_cast<const uint32_t*>(m.bricks) + 16 * (size_t)(idx + step[3]);
    return __ldg(top + idx);
  }
  uint32_t slot = 0;
  const int at = hash_lookup(m, up & 1 ? b[0] : ~b[0], up & 2 ? b[1] : ~b[1],
                             up & 4 ? b[2] : ~b[2], slot);
  if (at < 0) return 0u;                            // a missing block: free, alone
  brick = reinterpret_cast<const uint32_t*>(m.bricks) + 16 * (size_t)at;
  return 0x80000000u | slot;
}

// March a piece from state st until a hit, a map exit or the limits L (returns `at_limit`; st is
// then not the piece's end, which piece_start gives in closed form when it is wanted).
// Called by all lanes of the warp (`work` false: nothing to march), which meet at every box:
// left to itself, the compiler lets lanes whose paths parted (free or occupied block, a hit)
// run on as separate groups, and a pass then costs a multiple of its ~120 instructions.
// Bound by the chain from one box to the next (a block entry, a byte of the box field, the
// exit axis by exact 64-bit comparisons, the crossing counts of the other two axes) with two
// dependent loads; the field's lines stay in L1, which holds all of the SM's 228 KB since
// nothing is staged in shared memory.  Measured against a march over symmetric free boxes of
// blocks with a voxel walk inside occupied blocks: 65536 rays on the 40 m map 54 -> 15.2 us,
// 262144 rays on the 100 m map 101.6 -> 27.7 us (whole evaluations, later changes included).
template <int KIND, int LAYOUT, bool BOXES>
__device__ __forceinline__ int march_run(const DevMap& m, MarchState& st, const RayFx& r,
                                         const uint32_t L[3], int at_limit, bool work) {
  const uint32_t* A = r.A;
  int* q = st.q;
  uint32_t* N = st.N;
  const float rA[3] = {recip_fast(__uint2float_rn(A[0])), recip_fast(__uint2float_rn(A[1])),
                       recip_fast(__uint2float_rn(A[2]))};
  int hi[3];                                        // first voxel beyond the map / the grid
  // dense: N of the map's far faces, or, for a face farther than any range, of a voxel in between
  // that no crossing within L reaches (L is at most 2^30, H stays below 2^32)
  uint32_t H[3];
  int step[4] = {0, 0, 0, 0};                       // signed brick strides and the first brick
  const uint32_t* top = m.top;
  int status = at_limit;
  bool run = work;
  if (LAYOUT == kLayoutGrid) {
    const int str[3] = {1, m.gdim[0], m.gdim[0] * m.gdim[1]};
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const bool up = (r.up >> a) & 1u;
      hi[a] = (KIND == RMP_MAP_DENSE_U8 && up) ? m.dims[a] : 8 * m.gdim[a];
      H[a] = N[a] + ((uint32_t)min(hi[a] - 1 - q[a], 2 * kMaxRangeVoxels - 1) << 16);
      step[a] = up ? str[a] : -str[a];
      step[3] += up ? 0 : (m.gdim[a] - 1) * str[a];
      // a dense map: a piece that starts outside has left the map
      if (KIND == RMP_MAP_DENSE_U8 && (q[a] >= hi[a] || q[a] < (up ? 0 : 8 * m.gdim[a] - m.dims[a]))) {
        status = RMP_RAY_MISS_EXIT;
        run = false;
      }
    }
    top += (size_t)r.up * ((size_t)str[2] * m.gdim[2]) + step[3];
  }
  const uint8_t* box = reinterpret_cast<const uint8_t*>(m.cells) + 512 * r.up;
  // every pass advances each running lane by at least one voxel
  for (uint32_t it = 0; it < 8u * (kMaxRangeVoxels + 2); ++it) {
    if (!__any_sync(0xffffffffu, run)) break;
    if (!run) continue;
    uint32_t F[3];                                  // numerators of the box's far faces
    bool inside = true;
    if (LAYOUT == kLayoutGrid && KIND != RMP_MAP_DENSE_U8)
      inside = (unsigned)q[0] < (unsigned)hi[0] && (unsigned)q[1] < (unsigned)hi[1] &&
               (unsigned)q[2] < (unsigned)hi[2];
    if (inside) {
      const int b[3] = {q[0] >> 3, q[1] >> 3, q[2] >> 3};
      const int l[3] = {q[0] & 7, q[1] & 7, q[2] & 7};
      const uint32_t* brick = nullptr;
      uint32_t e = block_entry<LAYOUT, BOXES>(m, top, step, b, r.up, brick);
      const bool occupied = (int)e < 0;
      if (occupied) {
        const uint32_t p = (uint32_t)(l[0] | (l[1] << 3) | (l[2] << 6));
        if (BOXES) {
          e = __ldg(box + 4096 * (size_t)(e & 0x7fffffffu) + p);
        } else {                                    // no box field: single voxels
          const uint32_t w = p ^ ((r.up & 1u ? 0u : 7u) | (r.up & 2u ? 0u : 56u) |
                                  (r.up & 4u ? 0u : 448u));
          e = (__ldg(brick + (w >> 5)) >> (w & 31u)) & 1u ? 0u : 64u;
        }
        if (e == 0u) {
          status = RMP_RAY_HIT;
          run = false;
        }
      }
      // extents in voxels, a block's counted from its first voxel
      const int sh = occupied ? 0 : 3, part = occupied ? 0 : 7;
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        const int ahead = (1 << (((e >> (2 * a)) & 3u) + sh)) - (l[a] & part) - 1;
        F[a] = N[a] + ((uint32_t)ahead << 16);
        if (KIND == RMP_MAP_DENSE_U8) F[a] = min(F[a], H[a]);
      }
    } else {
      // outside the grid of a hashed map: nothing ahead once it lies behind on any axis, else
      // every voxel short of it is free (at most 64 at once, see crossings_before)
      run = q[0] < hi[0] && q[1] < hi[1] && q[2] < hi[2];
      const int gap = min(max(-q[0], max(-q[1], -q[2])), 64);
#pragma unroll
      for (int a = 0; a < 3; ++a) F[a] = N[a] + ((uint32_t)(gap - 1) << 16);
    }
    // exit axis: the first face crossing (ties: the lowest axis)
    const bool y = (unsigned long long)F[1] * A[0] < (unsigned long long)F[0] * A[1];
    const uint32_t Fw = y ? F[1] : F[0], Aw = y ? A[1] : A[0];
    const bool z = (unsigned long long)F[2] * Aw < (unsigned long long)Fw * A[2];
    const uint32_t Fe = z ? F[2] : Fw, Ae = z ? A[2] : Aw;
    run = run && Fe <= (z ? L[2] : (y ? L[1] : L[0]));
    if (!run) continue;
    const float rE = z ? rA[2] : (y ? rA[1] : rA[0]);
    // the other two axes, i < j: i is x unless x exits, j is z unless z exits
    const bool x = !y && !z;
    const int ci = crossings_before(Fe, Ae, rE, x ? N[1] : N[0], x ? A[1] : A[0], !x);
    const int cj = crossings_before(Fe, Ae, rE, z ? N[1] : N[2], z ? A[1] : A[2], z);
    const int ce = (int)((Fe - (z ? N[2] : (y ? N[1] : N[0]))) >> 16) + 1;
    const int c[3] = {x ? ce : ci, x ? ci : (z ? cj : ce), z ? ce : cj};
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      q[a] += c[a];
      N[a] += (uint32_t)c[a] << 16;
    }
    st.n_last = Fe;
    st.a_last = Ae;
    st.ax_last = z ? 2 : (y ? 1 : 0);
    if (KIND == RMP_MAP_DENSE_U8 && Fe == (z ? H[2] : (y ? H[1] : H[0]))) {
      status = RMP_RAY_MISS_EXIT;                   // the exit axis stepped off the map
      run = false;
    }
  }
  return status;
}

__device__ __forceinline__ bool piece_final(int status) {
  return status == RMP_RAY_HIT || status == RMP_RAY_MISS_EXIT;
}

// Distinct 8^3 blocks whose occupancy a voxel-by-voxel march tests: the voxel path is monotone
// on each axis and blocks are convex, so this is 1 + the block changes along each axis up to
// the last tested voxel (for a map exit the voxel before the exit step; none if the ray
// starts outside the map).
__device__ __forceinline__ uint32_t blocks_tested(const RayFx& r, const MarchState& o, int status) {
  uint32_t n = 1;
  bool moved = false;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const bool left = status == RMP_RAY_MISS_EXIT && a == o.ax_last && o.q[a] > r.q0[a];
    moved = moved || o.q[a] > r.q0[a];
    n += (uint32_t)(((o.q[a] - (left ? 1 : 0)) >> 3) - (r.q0[a] >> 3));
  }
  return status == RMP_RAY_MISS_EXIT && !moved ? 0u : n;
}

__device__ __forceinline__ float entry_distance(uint32_t n, uint32_t a, float vs_f) {
  const float t = __fdiv_rn(__uint2float_rn(n), __uint2float_rn(a));
  return __fmul_rn(__fmul_rn(t, 256.0f), vs_f);
}

// ------------------------------------------------------------------ obstacle policy (Sec. III-C)
// u: unit direction towards the obstacle (r = -u points away), d: distance; the velocity
// is carried as an unevaluated FP32 pair vh + vl (= xdot to ~2^-48 relative).  Writes
// f_i (3), A_i (6 unique) and A_i f_i (3).  `active` and `in_radius` are the FP32
// decisions specified in the header; the values are FP32 except that xdot.r is a
// compensated dot product (Ogita, Rump and Oishi, "Accurate sum and dot product", 2005)
// because f_damp amplifies its rounding error by eta_damp / eps at small d, and w_r uses
// (r - d) formed exactly instead of 1 - d/r, which cancels near the radius.
__device__ __forceinline__ float dot2(const float vh[3], const float vl[3], const float r[3]) {
  float p = __fmul_rn(vh[0], r[0]);
  float e = __fmaf_rn(vh[0], r[0], -p);
#pragma unroll
  for (int a = 1; a < 3; ++a) {
    const float h = __fmul_rn(vh[a], r[a]);
    const float eh = __fmaf_rn(vh[a], r[a], -h);
    const float t = __fadd_rn(p, h);
    const float bp = __fsub_rn(t, p);
    const float es = __fadd_rn(__fsub_rn(p, __fsub_rn(t, bp)), __fsub_rn(h, bp));
    p = t;
    e = __fadd_rn(e, __fadd_rn(eh, es));
  }
  const float lo = vl[0] * r[0] + vl[1] * r[1] + vl[2] * r[2];
  return __fadd_rn(p, __fadd_rn(e, lo));
}

__device__ __forceinline__ void obstacle_policy(const EvalConsts& k, const float u[3], float d,
                                                const float vh[3], const float vl[3],
                                                bool active, bool in_radius, float f[3],
                                                float A[6], float af[3]) {
  const float r[3] = {-u[0], -u[1], -u[2]};
  const float frep = k.eta_rep * expf(-d * k.inv_nu_rep);
  const float xr = dot2(vh, vl, r);
  const float mm = active ? xr * xr : 0.0f;
  const float kd = __fdividef(k.eta_damp, d * k.inv_nu_damp + k.eps);
  const float z = kd * mm;                       // |f_damp| (|r| = 1)
  const float fr = frep + z;                     // f = (f_rep + |f_damp|) r
  f[0] = fr * r[0];
  f[1] = fr * r[1];
  f[2] = fr * r[2];
  float w = 0.0f;
  if (in_radius) {
    const float y = (__fsub_rn(k.r_hi, d) + k.r_lo) * k.inv_r;   // 1 - d/r
    const float x = d * k.inv_r;
    w = k.w_mode == 0 ? y * y : y * y * (1.0f + 2.0f * x);      // (1-x)^2 ; 1-3x^2+2x^3
  }
  const float h = z + k.c * log1pf(expf(-2.0f * k.c * z));
  const float sc = __fdividef(z, h);            // s(f_damp) = sc * r
  const float alpha = w * sc * sc;               // A = alpha r r^T
  A[0] = alpha * r[0] * r[0];
  A[1] = alpha * r[0] * r[1];
  A[2] = alpha * r[0] * r[2];
  A[3] = alpha * r[1] * r[1];
  A[4] = alpha * r[1] * r[2];
  A[5] = alpha * r[2] * r[2];
  const float rf = r[0] * f[0] + r[1] * f[1] + r[2] * f[2];
  const float g = alpha * rf;                    // A f = alpha (r.f) r
  af[0] = g * r[0];
  af[1] = g * r[1];
  af[2] = g * r[2];
}

__device__ __forceinline__ bool active32(const float v[3], const float u[3]) {
  const float dot = __fmaf_rn(v[2], u[2], __fmaf_rn(v[1], u[1], __fmul_rn(v[0], u[0])));
  return dot > 0.0f;
}

// ------------------------------------------------------------------ reduction
// Compensated FP32 accumulator: (s, c) with s + c the running sum; additions use the
// error-free TwoSum so the tree keeps about twice FP32's precision.
struct Acc32 {
  float s[9], c[9];
};

__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
  s = __fadd_rn(a, b);
  const float bp = __fsub_rn(s, a);
  e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bp)), __fsub_rn(b, bp));
}

__device__ __forceinline__ void acc_add(Acc32& acc, const float v[9]) {
#pragma unroll
  for (int q = 0; q < 9; ++q) {
    float s, e;
    two_sum(acc.s[q], v[q], s, e);
    acc.s[q] = s;
    acc.c[q] = __fadd_rn(acc.c[q], e);
  }
}

struct Acc64 {
  double s[9];
};

// Sums of one CTA handed from the block reduction to grid_finish: the 9 terms (FP64 value
// v, and for the compensated reduction also the unevaluated FP32 pair s + c it came from)
// and the hit and active counts.  In shared memory, written by lanes 0-10 of warp 0 (lane
// q < 9: term q; lanes 9, 10: the counts), which are the lanes that read them again.
struct CtaSums {
  double v[9];
  float s[9], c[9];
  unsigned u[2];
};

__device__ __forceinline__ void merge1(float& s, float& c, float s2, float c2) {
  float t, e;
  two_sum(s, s2, t, e);
  s = t;
  c = __fadd_rn(__fadd_rn(c, c2), e);
}

__device__ __forceinline__ void merge1(double& s, double s2) { s += s2; }

// Sums of the 9 terms over each group of W = 32 >> lgW lanes by the tree of a shuffle-down
// reduction (lane i takes lane i + W/2, then W/4, ...), but with the terms shared out: at each
// level a lane and its partner keep half of their terms each and merge only those, 12 merges a
// lane instead of 45 (the merges commute bit for bit, so the tree's results are the same).
// Afterwards slot j (j < WarpTerms::n) of a lane holds term first + j; n is 0 where the lane
// holds none.  Lanes 0, W, 2 W, ... hold term 0.
struct WarpTerms {
  int first, n;
};

// terms a lane holds before level j
__host__ __device__ constexpr int term_split(int j) {
  return j == 0 ? 9 : (j == 1 ? 5 : (j == 2 ? 3 : (j == 3 ? 2 : 1)));
}

__device__ __forceinline__ WarpTerms warp_terms(uint32_t lgW) {
  const uint32_t lane = threadIdx.x & 31;
  WarpTerms t{0, 9};
#pragma unroll
  for (int j = 0; j < 5; ++j) {
    const uint32_t off = 16u >> (lgW + j);
    const int h = term_split(j + 1);
    if (off == 0) continue;
    if (lane & off) {
      t.first += h;
      t.n -= h;
    } else {
      t.n = t.n < h ? t.n : h;
    }
    if (t.n < 0) t.n = 0;
  }
  return t;
}

// FP32 pairs (s, c), or FP64 values (c unused); slots 0 .. of s (and c) are left as above.
template <typename T, bool PAIR>
__device__ __forceinline__ void warp_reduce_terms(T (&s)[9], T (&c)[9], uint32_t lgW) {
  const uint32_t lane = threadIdx.x & 31;
#pragma unroll
  for (int j = 0; j < 5; ++j) {
    const uint32_t off = 16u >> (lgW + j);
    if (off == 0) continue;
    const int m = term_split(j), h = term_split(j + 1);
    const bool upper = (lane & off) != 0;
#pragma unroll
    for (int i = 0; i < 5; ++i) {
      if (i >= h) continue;
      const T s1 = h + i < m ? s[h + i < 9 ? h + i : 8] : T(0), s0 = s[i];
      const T rs = __shfl_xor_sync(0xffffffffu, upper ? s0 : s1, off);
      s[i] = upper ? s1 : s0;
      if constexpr (PAIR) {
        const T c1 = h + i < m ? c[h + i < 9 ? h + i : 8] : T(0), c0 = c[i];
        const T rc = __shfl_xor_sync(0xffffffffu, upper ? c0 : c1, off);
        c[i] = upper ? c1 : c0;
        merge1(s[i], c[i], rs, rc);
      } else {
        merge1(s[i], rs);
      }
    }
  }
}

// Block-level reduction of the per-thread accumulators and counts: the shared-out tree per warp,
// (where one of its lanes `added` anything; all sums are zero otherwise), then lane q of warp 0
// merges term q of the warps in warp order (all terms at once, not one thread walking them).
// Called by every thread of a CTA of at most 8 warps; `wide`: the FP64 values are wanted.
template <int RED>
struct BlockReduce;

template <>
struct BlockReduce<RMP_REDUCE_KAHAN32> {
  using Acc = Acc32;
  __device__ static void init(Acc& a) {
#pragma unroll
    for (int q = 0; q < 9; ++q) a.s[q] = a.c[q] = 0.0f;
  }
  __device__ static void add(Acc& a, const float v[9]) { acc_add(a, v); }
  __device__ static void reduce(Acc& a, bool added, unsigned nh, unsigned na, CtaSums& out,
                                bool wide) {
    __shared__ float sh[8][18];
    __shared__ unsigned shu[8][2];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const WarpTerms t = warp_terms(0);
    if (__any_sync(0xffffffffu, added)) warp_reduce_terms<float, true>(a.s, a.c, 0);
    nh = __reduce_add_sync(0xffffffffu, nh);
    na = __reduce_add_sync(0xffffffffu, na);
    if (t.n > 0) {
      sh[warp][t.first] = a.s[0];
      sh[warp][9 + t.first] = a.c[0];
    }
    if (lane == 0) {
      shu[warp][0] = nh;
      shu[warp][1] = na;
    }
    __syncthreads();
    if (warp == 0) {
      if (lane < 9) {
        float sw[8], cw[8];                          // all loads before the serial merges
#pragma unroll
        for (int w = 0; w < 8; ++w) {
          sw[w] = w < nw ? sh[w][lane] : 0.0f;
          cw[w] = w < nw ? sh[w][9 + lane] : 0.0f;
        }
        float s = sw[0], c = cw[0];
#pragma unroll
        for (int w = 1; w < 8; ++w)
          if (w < nw) merge1(s, c, sw[w], cw[w]);
        out.s[lane] = s;
        out.c[lane] = c;
        if (wide) out.v[lane] = (double)s + (double)c;
      } else if (lane < 11) {
        unsigned t = 0;
        for (int w = 0; w < nw; ++w) t += shu[w][lane - 9];
        out.u[lane - 9] = t;
      }
    }
  }
};

template <>
struct BlockReduce<RMP_REDUCE_FP64> {
  using Acc = Acc64;
  __device__ static void init(Acc& a) {
#pragma unroll
    for (int q = 0; q < 9; ++q) a.s[q] = 0.0;
  }
  __device__ static void add(Acc& a, const float v[9]) {
#pragma unroll
    for (int q = 0; q < 9; ++q) a.s[q] += (double)v[q];
  }
  __device__ static void reduce(Acc& a, bool added, unsigned nh, unsigned na, CtaSums& out, bool) {
    __shared__ double sh[8][9];
    __shared__ unsigned shu[8][2];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const WarpTerms t = warp_terms(0);
    if (__any_sync(0xffffffffu, added)) warp_reduce_terms<double, false>(a.s, a.s, 0);
    nh = __reduce_add_sync(0xffffffffu, nh);
    na = __reduce_add_sync(0xffffffffu, na);
    if (t.n > 0) sh[warp][t.first] = a.s[0];
    if (lane == 0) {
      shu[warp][0] = nh;
      shu[warp][1] = na;
    }
    __syncthreads();
    if (warp == 0) {
      if (lane < 9) {
        double s = sh[0][lane];
        for (int w = 1; w < nw; ++w) s += sh[w][lane];
        out.v[lane] = s;
      } else if (lane < 11) {
        unsigned t = 0;
        for (int w = 0; w < nw; ++w) t += shu[w][lane - 9];
        out.u[lane - 9] = t;
      }
    }
  }
};

// ------------------------------------------------------------------ FP64 resolve (Eq. 1)
// f = (sum A)^+ (sum A f) with eigenvalues <= 1e-12 lambda_max treated as zero.  FP64
// division and square root cost hundreds of cycles each on this GPU and every FP64
// instruction of a warp occupies the FP64 pipe for tens of cycles whatever the number of
// active lanes (measured: the resolve's stages take about 64 cycles per FP64 instruction),
// so the FP64 arithmetic is kept to what the result needs and the work is split:
//   eigenvectors by cyclic Jacobi rotations in FP32 (the matrix scaled by a power of two
//   and narrowed to FP32 by integer operations on its bit patterns), and, in another warp
//   (or another lane of the same warp), the FP64 adjugate solve adj(S) b / det(S);
//   lanes 0-2: each eigenvalue as the FP64 Rayleigh quotient v^T S v / v^T v of its FP32
//   eigenvector (second-order accurate, ~1e-14 lambda_max), with 1 / v^T v = 2 - v^T v to
//   first order (v^T v = 1 + O(1e-7)); the eigenvector components widened to FP64 by bit
//   packing (exact);
//   lane 0: the eigenvalues sorted and the rank decided by comparing order-preserving
//   integer keys of the FP64 values; full rank uses the adjugate solution, a deficient
//   rank projects b on the kept eigenvectors; writes f, eig, rank into r.

// S / 2^(E - 1023) narrowed to FP32 by truncation, E the largest biased exponent of the six
// entries (so the largest lies in [1, 2)); entries with a zero or subnormal exponent, or
// below 2^-126 of the largest, become 0.  Integer operations only.
__device__ __forceinline__ void narrow_scaled(const double* S, float a[6]) {
  int hi[6];
  unsigned lo[6];
  int emax = 0;
#pragma unroll
  for (int q = 0; q < 6; ++q) {
    hi[q] = __double2hiint(S[q]);
    lo[q] = (unsigned)__double2loint(S[q]);
    emax = max(emax, (hi[q] >> 20) & 0x7FF);
  }
#pragma unroll
  for (int q = 0; q < 6; ++q) {
    const int e = (hi[q] >> 20) & 0x7FF;
    const int fe = e - emax + 127;
    const unsigned mant = ((unsigned)(hi[q] & 0xFFFFF) << 3) | (lo[q] >> 29);
    const unsigned bits = ((unsigned)hi[q] & 0x80000000u) | ((unsigned)fe << 23) | mant;
    a[q] = (e != 0 && fe > 0) ? __uint_as_float(bits) : 0.0f;
  }
}

// An FP32 value widened to FP64 exactly by packing its bits (zero and subnormal inputs give
// zero; the eigenvector components this serves are normal or zero).
__device__ __forceinline__ double widen(float f) {
  const unsigned b = __float_as_uint(f);
  const unsigned e = (b >> 23) & 0xFFu;
  const unsigned hi = (b & 0x80000000u) | ((e + 896u) << 20) | ((b & 0x7FFFFFu) >> 3);
  return e == 0 ? 0.0 : __hiloint2double((int)hi, (int)((b & 7u) << 29));
}

// Integer key with the order of the (non-NaN) double x.
__device__ __forceinline__ long long order_key(double x) {
  const long long b = __double_as_longlong(x);
  return b >= 0 ? b : (b ^ 0x7FFFFFFFFFFFFFFFll);
}

// Eigenvectors (columns of W) of the symmetric S by FP32 Jacobi sweeps.  One thread.
__device__ __forceinline__ void jacobi_f32(const double* S, float W[3][3]) {
  float sa[6];
  narrow_scaled(S, sa);
  float a00 = sa[0], a01 = sa[1], a02 = sa[2], a11 = sa[3], a12 = sa[4], a22 = sa[5];
  for (int sweep = 0; sweep < 6; ++sweep) {
    const float off = fabsf(a01) + fabsf(a02) + fabsf(a12);
    const float dia = fabsf(a00) + fabsf(a11) + fabsf(a22);
    if (!(off > 1e-6f * dia)) break;              // FP32 accuracy; FP64 refines below
#pragma unroll
    for (int pq = 0; pq < 3; ++pq) {
      float app, aqq, apq, apo, aqo;
      if (pq == 0) { app = a00; aqq = a11; apq = a01; apo = a02; aqo = a12; }
      else if (pq == 1) { app = a00; aqq = a22; apq = a02; apo = a01; aqo = a12; }
      else { app = a11; aqq = a22; apq = a12; apo = a01; aqo = a02; }
      if (apq == 0.0f) continue;
      const float tau = __fdividef(aqq - app, 2.0f * apq);
      const float at = fabsf(tau);
      const float root = at < 1e18f ? (1.0f + at * at) * rsqrtf(1.0f + at * at) : at;
      const float tt = copysignf(__fdividef(1.0f, at + root), tau);
      const float c = rsqrtf(1.0f + tt * tt), sn = tt * c;
      const float npp = app - tt * apq, nqq = aqq + tt * apq;
      const float npo = c * apo - sn * aqo, nqo = sn * apo + c * aqo;
      const int p = pq == 2 ? 1 : 0, q = pq == 0 ? 1 : 2;
      if (pq == 0) { a00 = npp; a11 = nqq; a01 = 0.f; a02 = npo; a12 = nqo; }
      else if (pq == 1) { a00 = npp; a22 = nqq; a02 = 0.f; a01 = npo; a12 = nqo; }
      else { a11 = npp; a22 = nqq; a12 = 0.f; a01 = npo; a02 = nqo; }
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        const float vp = W[i][p], vq = W[i][q];
        W[i][p] = c * vp - sn * vq;
        W[i][q] = sn * vp + c * vq;
      }
    }
  }
}

// 1 / x in FP64 for a positive x, by Newton's iteration for the reciprocal, r <- r + r (1 - m r),
// on the mantissa m in [1, 2): two steps from the FP32 reciprocal of m truncated to FP32
// (relative error 2^-22.4 -> 2^-44.8 -> below the FP64 rounding of the steps, about one ulp),
// the exponent applied by integer operations.  Four FP64 instructions instead of a division's
// sequence; subnormal, infinite or NaN x, and results outside the normal range, take the
// division.
__device__ __forceinline__ double recip_pos(double x) {
  const long long bx = __double_as_longlong(x);
  const int ex = (int)((bx >> 52) & 0x7FF);
  const double m = __longlong_as_double((bx & 0x000FFFFFFFFFFFFFll) | 0x3FF0000000000000ll);
  const float mf = __uint_as_float(0x3F800000u | (unsigned)((bx >> 29) & 0x7FFFFF));
  double r = widen(__frcp_rn(mf));                        // in [0.5, 1]
  double e = fma(-m, r, 1.0);
  r = fma(r, e, r);
  e = fma(-m, r, 1.0);
  r = fma(r, e, r);
  const long long br = __double_as_longlong(r);
  const int er = (int)((br >> 52) & 0x7FF) - (ex - 1023);
  if (ex == 0 || ex == 2047 || er <= 0 || er >= 2047) return 1.0 / x;
  return __longlong_as_double((br & 0x000FFFFFFFFFFFFFll) | ((long long)er << 52));
}

// FP64 solve adj(S) b / det(S); ok = det > 0.  The roundings are spelled out, so that one thread
// and a warp give the same bits: a cofactor p q - r u as fma(p, q, -(r u)), the determinant as
// fma(S2, c02, fma(S1, c01, S0 c00)), a row as fma(z, b2, fma(x, b0, y b1)).
__device__ __forceinline__ double cofactor(double p, double q, double r, double u) {
  return __fma_rn(p, q, -__dmul_rn(r, u));
}
__device__ __forceinline__ double determinant(const double* S, double c00, double c01, double c02) {
  return __fma_rn(S[2], c02, __fma_rn(S[1], c01, __dmul_rn(S[0], c00)));
}
__device__ __forceinline__ double adjugate_row(double x, double y, double z, const double* b,
                                               double inv) {
  return __dmul_rn(__fma_rn(z, b[2], __fma_rn(x, b[0], __dmul_rn(y, b[1]))), inv);
}

// One thread.
__device__ __forceinline__ void adjugate_solve(const double* S, const double* b, double& fa0,
                                               double& fa1, double& fa2, int& ok) {
  const double c00 = cofactor(S[3], S[5], S[4], S[4]), c01 = cofactor(S[2], S[4], S[1], S[5]),
               c02 = cofactor(S[1], S[4], S[2], S[3]), c11 = cofactor(S[0], S[5], S[2], S[2]),
               c12 = cofactor(S[1], S[2], S[0], S[4]), c22 = cofactor(S[0], S[3], S[1], S[1]);
  const double det = determinant(S, c00, c01, c02);
  ok = det > 0.0;
  if (det > 0.0) {
    const double inv = recip_pos(det);
    fa0 = adjugate_row(c00, c01, c02, b, inv);
    fa1 = adjugate_row(c01, c11, c12, b, inv);
    fa2 = adjugate_row(c02, c12, c22, b, inv);
  }
}

// A whole warp, S and b in every lane: the cofactors on lanes 0-5, the determinant and its
// reciprocal in all of them, component i of the solution in lane i (0-2): 17 FP64 instructions
// one after the other instead of 38.
__device__ __forceinline__ double adjugate_solve_warp(const double* S, const double* b, int& ok) {
  const uint32_t t = threadIdx.x & 31;
  const double p = t == 0 ? S[3] : (t == 1 ? S[2] : (t == 2 || t == 4 ? S[1] : S[0]));
  const double q = t == 0 || t == 3 ? S[5] : (t == 1 || t == 2 ? S[4] : (t == 4 ? S[2] : S[3]));
  const double r = t == 0 ? S[4] : (t == 1 || t == 5 ? S[1] : (t == 4 ? S[0] : S[2]));
  const double u = t == 0 || t == 4 ? S[4] : (t == 1 ? S[5] : (t == 2 ? S[3] : (t == 3 ? S[2] : S[1])));
  const double c = cofactor(p, q, r, u);
  const double c00 = __shfl_sync(0xffffffffu, c, 0), c01 = __shfl_sync(0xffffffffu, c, 1),
               c02 = __shfl_sync(0xffffffffu, c, 2), c11 = __shfl_sync(0xffffffffu, c, 3),
               c12 = __shfl_sync(0xffffffffu, c, 4), c22 = __shfl_sync(0xffffffffu, c, 5);
  const double det = determinant(S, c00, c01, c02);
  ok = det > 0.0;
  if (!ok) return 0.0;
  return adjugate_row(t == 0 ? c00 : (t == 1 ? c01 : c02), t == 0 ? c01 : (t == 1 ? c11 : c12),
                      t == 0 ? c02 : (t == 1 ? c12 : c22), b, recip_pos(det));
}

// Sorted eigenpairs and rank from the FP32 eigenvectors W (valid in lane 0): lanes 0-2 take
// the FP64 Rayleigh quotients; lane 0 sorts, decides the rank, writes eig and rank into r and
// keeps in es what a rank-deficient projection needs.  Called by all 32 lanes of one warp;
// only lane 0's r and es are set.
struct EigenSet {
  float c[3][3];   // eigenvector i (ascending eigenvalues) in c[i]
  float dv[3];     // its v^T v - 1
  bool keep[3];    // eigenvalue above the rank threshold
};

// v^T v - 1 for an FP32 vector with v^T v = 1 + O(1e-7), in FP32 error-free arithmetic:
// the squares split exactly into product and FMA error, the three products summed by TwoSum,
// the sum minus 1 exact (Sterbenz), the small terms added last (error ~1e-15).
__device__ __forceinline__ float norm2_minus_one(float v0, float v1, float v2) {
  const float p0 = __fmul_rn(v0, v0), p1 = __fmul_rn(v1, v1), p2 = __fmul_rn(v2, v2);
  const float e0 = __fmaf_rn(v0, v0, -p0), e1 = __fmaf_rn(v1, v1, -p1), e2 = __fmaf_rn(v2, v2, -p2);
  float s1, r1, s2, r2;
  two_sum(p0, p1, s1, r1);
  two_sum(s1, p2, s2, r2);
  return __fadd_rn(__fsub_rn(s2, 1.0f), __fadd_rn(__fadd_rn(r1, r2), __fadd_rn(__fadd_rn(e0, e1), e2)));
}

// One thread: eig (ascending), rank and what a rank-deficient projection needs, from the
// eigenvalues, their vectors (columns of V) and v^T v - 1.
__device__ __forceinline__ void rank_eigen(const double lam[3], const float dv[3],
                                           const float V[3][3], rmp_result_t& r, EigenSet& es) {
  // ascending eigenpairs by a 3-element sorting network on the values' integer keys
  double e0 = lam[0], e1 = lam[1], e2 = lam[2];
  float d0 = dv[0], d1 = dv[1], d2 = dv[2];
  long long q0 = order_key(e0), q1 = order_key(e1), q2 = order_key(e2);
  float c0[3] = {V[0][0], V[1][0], V[2][0]}, c1[3] = {V[0][1], V[1][1], V[2][1]},
        c2[3] = {V[0][2], V[1][2], V[2][2]};
  auto swap01 = [&]() {
    const double te = e0;
    const float td = d0;
    const long long tq = q0;
    e0 = e1; d0 = d1; q0 = q1; e1 = te; d1 = td; q1 = tq;
#pragma unroll
    for (int i = 0; i < 3; ++i) { const float tc = c0[i]; c0[i] = c1[i]; c1[i] = tc; }
  };
  if (q1 < q0) swap01();
  if (q2 < q1) {
    const double te = e1;
    const float td = d1;
    const long long tq = q1;
    e1 = e2; d1 = d2; q1 = q2; e2 = te; d2 = td; q2 = tq;
#pragma unroll
    for (int i = 0; i < 3; ++i) { const float tc = c1[i]; c1[i] = c2[i]; c2[i] = tc; }
  }
  if (q1 < q0) swap01();
  // kept: lambda_max > 1e-300 and lambda > 1e-12 lambda_max
  const long long thr = order_key(1e-12 * e2);
  const bool live = q2 > order_key(1e-300);
  es.keep[0] = live && q0 > thr;
  es.keep[1] = live && q1 > thr;
  es.keep[2] = live && q2 > thr;
  r.eig[0] = e0;
  r.eig[1] = e1;
  r.eig[2] = e2;
  r.rank = (es.keep[0] ? 1u : 0u) + (es.keep[1] ? 1u : 0u) + (es.keep[2] ? 1u : 0u);
  es.dv[0] = d0;
  es.dv[1] = d1;
  es.dv[2] = d2;
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    es.c[0][i] = c0[i];
    es.c[1][i] = c1[i];
    es.c[2][i] = c2[i];
  }
}

__device__ __forceinline__ void resolve_eigen(const double* S, const float (&W)[3][3],
                                              rmp_result_t& r, EigenSet& es) {
  const int t = threadIdx.x & 31;
  float V[3][3];
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) V[i][j] = __shfl_sync(0xffffffffu, W[i][j], 0);
  // lanes 0-8: lane 3 i + c takes component c of eigenvector i (column i of V): its term
  // v_c (S v)_c in FP64; lane 3 i adds the three terms and applies 1 / v^T v = 1 - (v^T v - 1)
  // to first order.  Seven FP64 instructions per warp (every FP64 instruction holds the
  // pipe about 64 cycles whatever the active lanes).
  const int iv = t < 9 ? t / 3 : 0, c = t < 9 ? t - 3 * iv : 0;
  const float w0 = iv == 0 ? V[0][0] : (iv == 1 ? V[0][1] : V[0][2]);
  const float w1 = iv == 0 ? V[1][0] : (iv == 1 ? V[1][1] : V[1][2]);
  const float w2 = iv == 0 ? V[2][0] : (iv == 1 ? V[2][1] : V[2][2]);
  double term = 0.0;
  if (t < 9) {
    const double sc0 = c == 0 ? S[0] : (c == 1 ? S[1] : S[2]);
    const double sc1 = c == 0 ? S[1] : (c == 1 ? S[3] : S[4]);
    const double sc2 = c == 0 ? S[2] : (c == 1 ? S[4] : S[5]);
    const double u = sc0 * widen(w0) + sc1 * widen(w1) + sc2 * widen(w2);
    term = widen(c == 0 ? w0 : (c == 1 ? w1 : w2)) * u;
  }
  const double t1 = __shfl_down_sync(0xffffffffu, term, 1);
  const double t2 = __shfl_down_sync(0xffffffffu, term, 2);
  const float dv_t = norm2_minus_one(w0, w1, w2);
  double lam_t = (term + t1) + t2;
  lam_t = fma(-lam_t, widen(dv_t), lam_t);
  double lam[3];
  float dv[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    lam[i] = __shfl_sync(0xffffffffu, lam_t, 3 * i);
    dv[i] = __shfl_sync(0xffffffffu, dv_t, 3 * i);
  }
  if (t == 0) rank_eigen(lam, dv, V, r, es);
}

// f into r from the rank (resolve_eigen) and the adjugate solution: full rank takes the
// adjugate, a deficient rank projects b on the kept eigenvectors.  Lane 0 of the warp that
// ran resolve_eigen.
__device__ __forceinline__ void resolve_f(const double* b, const EigenSet& es, double fa0,
                                          double fa1, double fa2, int ok, rmp_result_t& r) {
  r.f[0] = r.f[1] = r.f[2] = 0.0;
  if (r.rank == 3 && ok) {
    r.f[0] = fa0;
    r.f[1] = fa1;
    r.f[2] = fa2;
    return;
  }
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    if (!es.keep[i]) continue;
    const float* c = es.c[i];
    const double proj = (c[0] * b[0] + c[1] * b[1] + c[2] * b[2]) / (r.eig[i] * (1.0 + widen(es.dv[i])));
    r.f[0] += proj * c[0];
    r.f[1] += proj * c[1];
    r.f[2] += proj * c[2];
  }
}

// One warp, S and b in every lane: the adjugate solve across the lanes, then lane 0's Jacobi
// sweeps and the Rayleigh quotients.  Only lane 0's r is set.
__device__ void resolve_pinv(const double* S, const double* b, rmp_result_t& r) {
  float W[3][3] = {{1.f, 0.f, 0.f}, {0.f, 1.f, 0.f}, {0.f, 0.f, 1.f}};
  int ok;
  const double f = adjugate_solve_warp(S, b, ok);
  const double fa0 = __shfl_sync(0xffffffffu, f, 0), fa1 = __shfl_sync(0xffffffffu, f, 1),
               fa2 = __shfl_sync(0xffffffffu, f, 2);
  if ((threadIdx.x & 31) == 0) jacobi_f32(S, W);
  EigenSet es;
  resolve_eigen(S, W, r, es);
  if ((threadIdx.x & 31) == 0) resolve_f(b, es, fa0, fa1, fa2, ok, r);
}

// Two warps of a CTA (threads 0-63): warp 0 runs the Jacobi sweeps and the Rayleigh
// quotients while warp 1 runs the adjugate solve; they meet at named barrier 1 only for
// the choice of f.  Called by threads 0-63 of a CTA of at least 64 threads; S, b and r in
// shared memory.
__device__ void resolve_pinv_cta(const double* S, const double* b, rmp_result_t& r) {
  __shared__ double fa_sh[3];
  __shared__ int ok_sh;
  const int t = threadIdx.x;
  if (t >= 32) {
    int ok;
    const double f = adjugate_solve_warp(S, b, ok);
    if (t < 35) fa_sh[t - 32] = f;
    if (t == 32) ok_sh = ok;
    __syncwarp();
    asm volatile("bar.sync 1, 64;" ::: "memory");
    return;
  }
  float W[3][3] = {{1.f, 0.f, 0.f}, {0.f, 1.f, 0.f}, {0.f, 0.f, 1.f}};
  if (t == 0) jacobi_f32(S, W);
  EigenSet es;
  resolve_eigen(S, W, r, es);
  __syncwarp();
  asm volatile("bar.sync 1, 64;" ::: "memory");
  if (t == 0) resolve_f(b, es, fa_sh[0], fa_sh[1], fa_sh[2], ok_sh, r);
}

// A partial in the workspace (80 bytes, one per CTA): the compensated reduction stores each
// term as its FP32 pair (s, c), the FP64 reduction as a double (CtaPartial); both end with
// the hit and active counts.  An empty slot holds 0xFF in every byte, a pattern no
// stored field takes: FP32 and FP64 arithmetic on this GPU returns its canonical NaNs
// (sign bit clear), never the all-ones word, and the counts stay far below 2^31.
struct CtaPartial32 {
  float s[9], c[9];
  unsigned n_hits, n_active;
};
static_assert(sizeof(CtaPartial32) == sizeof(CtaPartial) && sizeof(CtaPartial) == 80,
              "partials are five 16-byte words");
constexpr uint64_t kFinishWaitNs = 10000000000ull;   // CTA 0 waits at most 10 s for a slot

// Slots are written with relaxed stores at GPU scope (each field one single-copy-atomic
// access) and read back with relaxed 64-bit loads, so a reader sees every field either
// empty or complete.
__device__ __forceinline__ void st_relaxed32(void* p, uint32_t v) {
  asm volatile("st.relaxed.gpu.global.b32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ void st_relaxed64(void* p, unsigned long long v) {
  asm volatile("st.relaxed.gpu.global.b64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ void load_slot(const CtaPartial* p, uint32_t w[20]) {
  const unsigned long long* q = reinterpret_cast<const unsigned long long*>(p);
  unsigned long long v[10];
#pragma unroll
  for (int i = 0; i < 5; ++i)
    asm volatile("ld.relaxed.gpu.global.v2.b64 {%0, %1}, [%2];"
                 : "=l"(v[2 * i]), "=l"(v[2 * i + 1])
                 : "l"(q + 2 * i)
                 : "memory");
#pragma unroll
  for (int i = 0; i < 10; ++i) {
    w[2 * i] = (uint32_t)v[i];
    w[2 * i + 1] = (uint32_t)(v[i] >> 32);
  }
}
__device__ __forceinline__ void empty_slot(CtaPartial* p) {
  uint4* q = reinterpret_cast<uint4*>(p);
  const uint4 e = make_uint4(~0u, ~0u, ~0u, ~0u);
#pragma unroll
  for (int i = 0; i < 5; ++i) q[i] = e;
}
__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Storing a CTA's sums in its slot, lanes 0-10 of warp 0 one field each; the words of a
// CTA's own sums as its slot would hold them; whether a slot's words are all written; and
// starting a thread's accumulator from the words of a partial / merging one into it.
template <int RED>
struct PartialIO;

template <>
struct PartialIO<RMP_REDUCE_KAHAN32> {
  __device__ static void store(CtaPartial* slot, const CtaSums& cs, int t) {
    CtaPartial32* p = reinterpret_cast<CtaPartial32*>(slot);
    if (t < 9) {
      st_relaxed32(&p->s[t], __float_as_uint(cs.s[t]));
      st_relaxed32(&p->c[t], __float_as_uint(cs.c[t]));
    } else if (t == 9) {
      st_relaxed32(&p->n_hits, cs.u[0]);
    } else if (t == 10) {
      st_relaxed32(&p->n_active, cs.u[1]);
    }
  }
  __device__ static void words(const CtaSums& cs, uint32_t w[20]) {
#pragma unroll
    for (int q = 0; q < 9; ++q) {
      w[q] = __float_as_uint(cs.s[q]);
      w[9 + q] = __float_as_uint(cs.c[q]);
    }
    w[18] = cs.u[0];
    w[19] = cs.u[1];
  }
  __device__ static bool ready(const uint32_t w[20]) {
    bool ok = true;
#pragma unroll
    for (int i = 0; i < 20; ++i) ok = ok && w[i] != ~0u;
    return ok;
  }
  __device__ static void set(Acc32& a, const uint32_t w[20]) {
#pragma unroll
    for (int q = 0; q < 9; ++q) {
      a.s[q] = __uint_as_float(w[q]);
      a.c[q] = __uint_as_float(w[9 + q]);
    }
  }
  __device__ static void merge(Acc32& a, const uint32_t w[20]) {
#pragma unroll
    for (int q = 0; q < 9; ++q) merge1(a.s[q], a.c[q], __uint_as_float(w[q]), __uint_as_float(w[9 + q]));
  }
};

template <>
struct PartialIO<RMP_REDUCE_FP64> {
  __device__ static void store(CtaPartial* slot, const CtaSums& cs, int t) {
    if (t < 9) st_relaxed64(&slot->v[t], (unsigned long long)__double_as_longlong(cs.v[t]));
    else if (t == 9) st_relaxed32(&slot->n_hits, cs.u[0]);
    else if (t == 10) st_relaxed32(&slot->n_active, cs.u[1]);
  }
  __device__ static void words(const CtaSums& cs, uint32_t w[20]) {
#pragma unroll
    for (int q = 0; q < 9; ++q) {
      const unsigned long long b = (unsigned long long)__double_as_longlong(cs.v[q]);
      w[2 * q] = (uint32_t)b;
      w[2 * q + 1] = (uint32_t)(b >> 32);
    }
    w[18] = cs.u[0];
    w[19] = cs.u[1];
  }
  __device__ static bool ready(const uint32_t w[20]) {
    bool ok = w[18] != ~0u && w[19] != ~0u;
#pragma unroll
    for (int q = 0; q < 9; ++q) ok = ok && (w[2 * q] & w[2 * q + 1]) != ~0u;
    return ok;
  }
  __device__ static double word_pair(const uint32_t w[20], int q) {
    return __hiloint2double((int)w[2 * q + 1], (int)w[2 * q]);
  }
  __device__ static void set(Acc64& a, const uint32_t w[20]) {
#pragma unroll
    for (int q = 0; q < 9; ++q) a.s[q] = word_pair(w, q);
  }
  __device__ static void merge(Acc64& a, const uint32_t w[20]) {
#pragma unroll
    for (int q = 0; q < 9; ++q) a.s[q] += word_pair(w, q);
  }
};

// CTA 0's wait, one warp at a time: every lane with a pending slot (`ok` false) loads it
// until all of its fields are written (then its words are in w).  The warp polls as a
// whole -- it leaves the loop when every lane is done, lanes never spin on their own --
// because lanes that finished while others of their warp still spin stall for microseconds
// (measured).  Returns false when the wait passed `deadline` (global timer, ns).  Called by
// all lanes of the warp.
template <int RED>
__device__ __forceinline__ bool wait_slots(const CtaPartial* p, bool ok, uint32_t w[20],
                                           unsigned long long deadline) {
  while (!__all_sync(0xffffffffu, ok)) {
    if (!ok) {
      load_slot(p, w);
      ok = PartialIO<RED>::ready(w);
    }
    if (__any_sync(0xffffffffu, global_ns() > deadline)) return false;
  }
  return true;
}

// Grid completion, deterministic, with the partial sums streamed to CTA 0: lanes 0-10 of
// warp 0 of every other CTA store its sums in its slot and the CTA exits (no atomics, no
// fence); CTA 0, once its own rays are done, takes the slots as they fill -- thread t slot
// t, then t + blockDim, ... in order, merging each into its accumulator and emptying the
// slot -- then reduces the threads (BlockReduce) and resolves.  The summation order is
// fixed by slot index, whatever the order of arrival, and the partials of CTAs that
// finished early are read while the slowest still march: after the last partial only its
// load, the block reduction and the resolve remain.  CTA 0 never waits on a CTA that
// waits on it, so the wait ends once every CTA has run; it is bounded all the same
// (kFinishWaitNs), and a wait that expires reports RMP_ERR_TIMEOUT and marks the workspace
// poisoned (every later evaluation on it reports RMP_ERR_TIMEOUT until it is
// re-initialised).  A grid of one CTA resolves its own sums.  Called by all threads of
// every CTA after BlockReduce::reduce.
template <int RED>
__device__ void grid_finish(const CtaSums& cta, WsHeader* ws, CtaPartial* parts,
                            rmp_result_t* out, uint32_t n_rays, int status) {
  __shared__ CtaSums gsum;
  __shared__ int poison_sh;
  const int G = gridDim.x;
  const CtaSums* tot = &cta;
  int st = status;
  if (G > 1) {
    if (blockIdx.x != 0) {
      if (threadIdx.x < 32)
        PartialIO<RED>::store(parts + blockIdx.x, cta, threadIdx.x);
      return;
    }
    if (threadIdx.x == 0) poison_sh = ws->poisoned ? 1 : 0;
    __syncthreads();
    const bool poisoned = poison_sh != 0;
    typename BlockReduce<RED>::Acc acc;
    BlockReduce<RED>::init(acc);
    unsigned nh = 0, na = 0;
    bool expired = false;
    const unsigned long long deadline = global_ns() + kFinishWaitNs;
    // warp-uniform trip count: lane l of the warp takes slot base + l
    for (int base = threadIdx.x & ~31; base < G && !poisoned; base += blockDim.x) {
      const int i = base + (int)(threadIdx.x & 31);
      uint32_t w[20];
      if (i == 0) PartialIO<RED>::words(cta, w);
      if (!wait_slots<RED>(parts + i, i == 0 || i >= G, w, deadline)) {
        expired = true;
        break;
      }
      if (i >= G) continue;
      if (i > 0) empty_slot(parts + i);
      if (i == (int)threadIdx.x) PartialIO<RED>::set(acc, w);
      else PartialIO<RED>::merge(acc, w);
      nh += w[18];
      na += w[19];
    }
    BlockReduce<RED>::reduce(acc, true, nh, na, gsum, true);
    const int any_expired = __syncthreads_or(expired);
    if (poisoned || any_expired) {
      if (threadIdx.x == 0) ws->poisoned = 1;
      st = RMP_ERR_TIMEOUT;
    }
    tot = &gsum;
  }
  // lanes 0-8 hold the terms they reduced, lanes 9 and 10 the counts; the result leaves as 18
  // words of 18 lanes (one thread storing the record took 800 cycles)
  __shared__ rmp_result_t r;
  if (threadIdx.x < 9) {
    (&r.A[0])[threadIdx.x] = tot->v[threadIdx.x];      // A, then Af
  } else if (threadIdx.x < 11) {
    (&r.n_hits)[threadIdx.x - 9] = tot->u[threadIdx.x - 9];
  } else if (threadIdx.x == 11) {
    r.n_rays = n_rays;
    r.status = st;
    r.reserved = 0;
  }
  __syncthreads();
  if (threadIdx.x < 64) resolve_pinv_cta(r.A, r.Af, r);
  if (threadIdx.x < 32) {
    __syncwarp();
    if (threadIdx.x < 18)
      reinterpret_cast<unsigned long long*>(out)[threadIdx.x] =
          reinterpret_cast<const unsigned long long*>(&r)[threadIdx.x];
  }
}

static_assert(offsetof(rmp_result_t, Af) == offsetof(rmp_result_t, A) + 48 &&
                  offsetof(rmp_result_t, n_active) == offsetof(rmp_result_t, n_hits) + 4,
              "the finish writes these as arrays");

// Which state component (0-2 x, 3-5 xdot) thread t sets up, or -1: x on threads 0-2 and
// xdot on threads 32-34, two warps, so that the FP64 work of each runs in parallel.
__device__ __forceinline__ int state_component(unsigned t) {
  return t < 3 ? (int)t : ((t >= 32 && t < 35) ? (int)t - 29 : -1);
}

__device__ __forceinline__ void split_velocity(double x, CtaState& cs, int a) {
  cs.v[a] = __double2float_rn(x);
  cs.vl[a] = __double2float_rn(__dsub_rn(x, (double)cs.v[a]));
}

// Coherent ray order: thread slot j -> ray index.  Ray indices i with the same residue
// i mod M (M = 2^a 3^b) share the first a binary digits of H(i,2) and the first b ternary
// digits of H(i,3), so they point into one cell of the sphere; slots enumerate residue
// classes one after the other, so a warp covers at most two cells.  Q = n / M, R = n % M:
// classes r < R hold Q + 1 rays, the others Q.  M = 1 is the identity.
__device__ __forceinline__ uint32_t ray_of_slot(uint32_t j, uint32_t M, uint32_t Q, uint32_t R) {
  const uint32_t big = R * (Q + 1);
  const bool lo = j < big;
  uint32_t q;
  const uint32_t r = divide24(lo ? j : j - big, lo ? Q + 1 : Q, q);   // at most M <= n / 32 classes
  return (lo ? r : R + r) + M * q;
}

// ------------------------------------------------------------------ per-ray march and outputs
// One thread's segment `seg` (of S = 2^lg_segs) of the ray `ray` from position P: march the
// piece, then combine the ray's S segments -- adjacent lanes -- into the first final one
// (lowest index), else the last one.  Warp-synchronous: every lane of the warp calls it (work =
// false for lanes without a segment).  Returns the ray's status with (n, a), the entry
// crossing of its last voxel, in every lane of the group.  `rec` (nullable): where the lane
// that holds the ray's end writes its hit record.
template <int KIND, int LAYOUT, bool BOXES>
__device__ __forceinline__ int march_ray(const DevMap& m, const EvalConsts& k, const long long P[3],
                                         const Ray& ray, uint32_t seg, uint32_t lgS, bool work,
                                         uint32_t& n, uint32_t& a, rmp_ray_hit_t* rec) {
  const uint32_t S = 1u << lgS;
  const uint32_t lane = threadIdx.x & 31;
  // this lane's piece: segment seg of the ray, grid points j_lo .. j_hi
  const uint32_t j_lo = seg << (kGridLog - lgS), j_hi = (seg + 1) << (kGridLog - lgS);
  MarchState st;
  RayFx r;
  uint32_t L[3];
  ray_fx<LAYOUT>(m, P, ray.D, r);
  piece_start(r, k.R_fx, j_lo, st);
  limits_at(r, k.R_fx, j_hi, L);
  const int status = march_run<KIND, LAYOUT, BOXES>(
      m, st, r, L, seg == S - 1 ? RMP_RAY_MISS_RANGE : kSegContinues, work);
  const uint32_t ballot = __ballot_sync(0xffffffffu, work && piece_final(status));
  const uint32_t grp0 = lane & ~(S - 1);
  const uint32_t gmask = (S == 32 ? 0xffffffffu : ((1u << S) - 1u)) << grp0;
  const uint32_t fb = ballot & gmask;
  const int src = fb ? (__ffs(fb) - 1) : (int)(grp0 + S - 1);
  if (rec && work && (int)lane == src) {
    if (status == RMP_RAY_MISS_RANGE) piece_start(r, k.R_fx, 1u << kGridLog, st);   // its end
    rmp_ray_hit_t h;
    h.steps = 0;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      const bool up = (r.up >> i) & 1u;
      h.voxel[i] = unmirror(st.q[i], frame_lo<LAYOUT>(m, i, up), up);
      h.steps += (uint32_t)(st.q[i] - r.q0[i]);
    }
    h.d = st.n_last == 0 ? 0.0f : entry_distance(st.n_last, st.a_last, m.vs_f);
    h.status = (uint8_t)status;
    h.pad = 0;
    h.blocks = (uint16_t)blocks_tested(r, st, status);
    *rec = h;
  }
  n = __shfl_sync(0xffffffffu, st.n_last, src);
  a = __shfl_sync(0xffffffffu, st.a_last, src);
  return __shfl_sync(0xffffffffu, status, src);
}

// A hit (or scan point) that the robot does not approach, or beyond the policy radius, adds
// exact zeros to the sums whenever no intermediate of the policy overflows: bound on |v|^2
// prepared by the host (quiet_v2).  Its policy is then evaluated for the per-ray outputs only.
__device__ __forceinline__ bool quiet_state(const EvalConsts& k, const float v[3]) {
  return v[0] * v[0] + v[1] * v[1] + v[2] * v[2] < k.quiet_v2;
}

// The rows of (f_i, A_i), 9 floats each, of 32 consecutive points (`count` of them exist) written
// together: through `sh` (288 floats of the warp) element l + 32 i goes to lane l, so that a
// store covers whole lines, not four bytes of 32 rows (262144 points: 15.0 -> 10.2 us; the ray
// kernels, whose rows lie apart, would hold more registers for it and be slower without rows).
// Called by all lanes of the warp.
__device__ __forceinline__ void store_rows(float* rows, uint32_t count, const float f[3],
                                           const float A[6], float* sh) {
  const uint32_t lane = threadIdx.x & 31;
  float* mine = sh + 9 * lane;
  __syncwarp();
#pragma unroll
  for (int i = 0; i < 3; ++i) mine[i] = f[i];
#pragma unroll
  for (int i = 0; i < 6; ++i) mine[3 + i] = A[i];
  __syncwarp();
#pragma unroll
  for (uint32_t i = 0; i < 9; ++i) {
    const uint32_t e = lane + 32 * i;
    if (e < 9 * count) rows[e] = sh[e];
  }
}

// The ray's obstacle policy (Sec. III-C) from its end: vals = A_i (6) and A_i f_i (3), all zero
// unless it hit; counts hits and active rays; writes the optional per-ray (f_i, A_i).  Returns
// whether vals is to be added.
__device__ __forceinline__ bool ray_outputs(const DevMap& m, const EvalConsts& k, const Ray& ray,
                                            int status, uint32_t n, uint32_t a, const float v[3],
                                            const float vl[3], bool quiet, float* per, float vals[9],
                                            unsigned& n_hit, unsigned& n_act) {
  float f[3] = {0.f, 0.f, 0.f}, A[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f}, af[3] = {0.f, 0.f, 0.f};
  bool adds = false;
  if (status == RMP_RAY_HIT) {
    const float d = n == 0 ? 0.0f : entry_distance(n, a, m.vs_f);
    const bool act = active32(v, ray.dir);
    const bool inr = d < k.r_up;
    n_hit += 1;
    n_act += (act && inr) ? 1u : 0u;
    adds = (act && inr) || !quiet;
    if (adds || per) obstacle_policy(k, ray.dir, d, v, vl, act, inr, f, A, af);
  }
#pragma unroll
  for (int q = 0; q < 6; ++q) vals[q] = A[q];
  vals[6] = af[0];
  vals[7] = af[1];
  vals[8] = af[2];
  if (per) {
    per[0] = f[0]; per[1] = f[1]; per[2] = f[2];
    per[3] = A[0]; per[4] = A[1]; per[5] = A[2]; per[6] = A[3]; per[7] = A[4]; per[8] = A[5];
  }
  return adds;
}

// ------------------------------------------------------------------ fused raycast kernel
// Thread g of the launch handles segment g % S of the ray in slot g / S; the S segments of a
// ray sit in adjacent lanes, and the ray's result is the first segment (lowest index) that
// hit or left the map, else the last one -- found with a warp ballot and moved to the
// ray's first lane by shuffles.  That lane evaluates the policy and writes the outputs.
//
// BLOCK, CTAS: the register budget.  256 x 2 where the launch is one wave of 256-thread CTAs: its
// slowest warps decide, and more registers serve them better (65536 rays 15.2 us; held to 85
// registers 17.4, to 64 18.8).  128 x 6 (85 registers, 24 warps an SM) for the 128-thread CTAs of
// larger launches, which keep every SM busy: 262144 rays on the 100 m map 30.0 -> 27.7 us.
template <int KIND, int LAYOUT, int RED, bool BOXES, int BLOCK, int CTAS>
__global__ void __launch_bounds__(BLOCK, CTAS) raycast_rmp_kernel(
    DevMap m, EvalConsts k, const double* state, WsHeader* ws, CtaPartial* parts,
    rmp_result_t* out, rmp_ray_hit_t* hits, float* per_ray) {
  __shared__ CtaState cs;
  // state component of this thread: x on threads 0-2, xdot on threads 32-34 (another warp,
  // so the two FP64 chains below run side by side instead of one after the other); a synchronous
  // call's state comes quantised in the launch (its FP64 chain took 1200 cycles here)
  const int comp = state_component(threadIdx.x);
  typename BlockReduce<RED>::Acc acc;
  BlockReduce<RED>::init(acc);
  unsigned n_hit = 0, n_act = 0;
  const uint32_t lgS = k.lg_segs, S = 1u << lgS;
  const uint32_t lane = threadIdx.x & 31;
  const uint32_t total = k.n_rays << lgS;
  const uint32_t stride = gridDim.x * blockDim.x;
  uint32_t base = blockIdx.x * blockDim.x + (threadIdx.x & ~31u);
  // the first ray needs nothing of what comes before on the stream
  uint32_t ray_idx = ray_of_slot(base + lane < total ? (base + lane) >> lgS : 0, k.perm_M,
                                 k.perm_Q, k.perm_R);
  Ray ray = make_ray<false>(ray_idx + k.halton_offset);
  wait_previous();
  if (!state) {                                     // the launch carries the state, quantised
    if (threadIdx.x == 0) cs = k.cs0;
  } else if (comp >= 0 && comp < 3) {
    const double sv = state[comp];
    const double o = KIND != RMP_MAP_DENSE_U8 ? 0.0
                     : (comp == 0 ? m.origin[0] : (comp == 1 ? m.origin[1] : m.origin[2]));
    const double q = __dmul_rn(__ddiv_rn(__dsub_rn(sv, o), m.vs), 65536.0);
    // |voxel| < 2^22 keeps block keys and fixed-point products in range; NaN fails too
    const int bad = !(fabs(q) < 274877906944.0);
    cs.bad[comp] = bad;
    cs.P[comp] = bad ? 0 : __double2ll_rn(q);
  } else if (comp >= 3) {
    split_velocity(state[comp], cs, comp - 3);
  }
  __syncthreads();                                  // state ready
  const bool bad = (cs.bad[0] | cs.bad[1] | cs.bad[2]) != 0;
  const bool quiet = quiet_state(k, cs.v);
  bool first = true, added = false;
  // warp-uniform trip count: every lane takes part in each ballot / shuffle
  for (; base < total; base += stride) {
    const uint32_t g = base + lane;
    const bool active = g < total;
    const uint32_t seg = g & (S - 1);
    if (!first) {
      ray_idx = ray_of_slot(active ? (g >> lgS) : 0, k.perm_M, k.perm_Q, k.perm_R);
      ray = make_ray<false>(ray_idx + k.halton_offset);
    }
    first = false;
    const long long P[3] = {cs.P[0], cs.P[1], cs.P[2]};
    uint32_t en, ea;
    const int mstat = march_ray<KIND, LAYOUT, BOXES>(m, k, P, ray, seg, lgS, active && !bad, en, ea,
                                              hits ? hits + ray_idx : nullptr);
    if (!active || bad || seg != 0) continue;
    float vals[9];
    if (ray_outputs(m, k, ray, mstat, en, ea, cs.v, cs.vl, quiet,
                    per_ray ? per_ray + 9 * (size_t)ray_idx : nullptr, vals, n_hit, n_act)) {
      BlockReduce<RED>::add(acc, vals);
      added = true;
    }
  }
  launch_next();
  __shared__ CtaSums sums;
  BlockReduce<RED>::reduce(acc, added, n_hit, n_act, sums, gridDim.x == 1);
  grid_finish<RED>(sums, ws, parts, out, k.n_rays,
                   (cs.bad[0] | cs.bad[1] | cs.bad[2]) ? RMP_ERR_INVALID_ARG : RMP_OK);
}

// ------------------------------------------------------------------ batched evaluation
// Device form of the host's direction-cell choice, one warp per state: M = 2^a 3^b <=
// n / 32 minimising |log M - log(n / 48)| + 0.5 |log(3^b / (pi 2^a))| (cells close to
// square on the sphere).  The score is piecewise linear in b with its steeper kink where
// M = n / 48, so for a given a only the b next to that kink, b = 0 and the largest b the
// bound allows need checking; lane a checks those, the warp keeps the best (lowest a on
// ties).  Only the work schedule and the summation grouping depend on the choice.
__device__ __forceinline__ uint32_t pick_cells_warp(uint32_t n) {
  const uint32_t lane = threadIdx.x & 31;
  const float L3 = 1.5849625f, LPI = 1.6514961f;   // log2(3), log2(pi)
  const float lt = __log2f(fmaxf((float)n * (1.0f / 48.0f), 1.0f));
  const float lm = __log2f((float)n * (1.0f / 32.0f));
  float best_score = 3.0e38f;
  uint32_t best = 1;
  const int a = (int)lane;
  const bool fits = a <= 24 && (32ull << a) <= n;
  int b_max = 0;                                    // largest b with 32 2^a 3^b <= n (< 2^25)
  uint32_t m = 32u << (fits ? a : 0), pow3 = 1;     // pow3: 3^lane (lanes 0-15)
#pragma unroll
  for (int i = 0; i < 15; ++i) {
    m *= 3u;
    if (m > n) m = 0x40000000u;                     // past it for good
    b_max += m <= n ? 1 : 0;
    pow3 *= i < (int)(lane & 15u) ? 3u : 1u;
    m = m > n ? 0x15555555u : m;
  }
  const int bk = (int)floorf((lt - (float)a) / L3);
  const int bm = (int)floorf((lm - (float)a) / L3) + 1;
  const int cand[4] = {0, bk, bk + 1, bm};
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int bb = min(max(cand[i], 0), b_max);
    const uint32_t mm = __shfl_sync(0xffffffffu, pow3, bb) << (fits ? a : 0);
    const float score = fabsf((float)a + (float)bb * L3 - lt) +
                        0.5f * fabsf((float)bb * L3 - LPI - (float)a);
    if (fits && score < best_score) {
      best_score = score;
      best = mm;
    }
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    const float s2 = __shfl_down_sync(0xffffffffu, best_score, off);
    const uint32_t m2 = __shfl_down_sync(0xffffffffu, best, off);
    if (s2 < best_score) {                          // strict: the lower lane wins ties
      best_score = s2;
      best = m2;
    }
  }
  return __shfl_sync(0xffffffffu, best, 0);
}

// A state's summation segments (log2): the launch's fixed choice, or the most (up to 4) whose
// threads the persistent launch holds at once -- a function of the ray count and the launch
// shape alone, so a state's result does not depend on the other states of the batch or their
// order.
__host__ __device__ __forceinline__ uint32_t state_lg_segs(const EvalConsts& k, uint32_t n) {
  if (k.lg_segs <= 2u) return k.lg_segs;
  if (k.seg_threads == 0u) return n <= 4096u ? 2u : (n <= 16384u ? 1u : 0u);
  uint32_t lg = 2u;
  while (lg > 0u && ((unsigned long long)n << lg) > k.seg_threads) --lg;
  return lg;
}

// Segments marched per ray (log2), at most the summation's: a tuned launch marches those, the
// default the most whose threads fill half of the persistent launch over the whole batch of
// `total` rays -- beyond that, the extra segments' set-up costs more than their shorter chains
// save (256 states of 20000 rays: 1 / 2 / 4 segments 365 / 598 / 1006 us; 16 of 3125: 29.8 / 28.7 /
// 40.6; one of 16384: 25.1 / 23.5 / 24.2).
__device__ __forceinline__ uint32_t march_lg_segs(const EvalConsts& k, uint32_t lg_sum,
                                                  unsigned long long total) {
  if (k.lg_segs <= 2u) return lg_sum;
  while (lg_sum > 0u && (total << lg_sum) > k.seg_threads / 2) --lg_sum;
  return lg_sum;
}

// Sum of x over the CTA's threads (256), in every thread; sh: 8 words.
__device__ __forceinline__ uint32_t block_sum256(uint32_t x, uint32_t* sh) {
  x = __reduce_add_sync(0xffffffffu, x);
  __syncthreads();                                  // sh is no longer read
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = x;
  __syncthreads();
  uint32_t t = 0;
#pragma unroll
  for (int w = 0; w < 8; ++w) t += sh[w];
  return t;
}

// Per-state set-up of a batch, CTAs of 256 threads with a run of consecutive states each.  The
// chunks and groups before a CTA's run follow from the ray counts alone, so every CTA adds
// them up itself (4 bytes a state) instead of waiting for the others; then, 256 states at a
// time, one thread per state takes its ranges from a block scan and one warp per state
// quantises the position (lanes 0-2, FP64), splits the velocity (lanes 3-5) and chooses the
// direction cells.  The tickets and the work counter are cleared, and every state without
// rays or with an error gets its result here (chunks of an invalid state are skipped).
// Bound by one state's latency: 7.3 us for 256 states (one CTA with 8 states a warp, and cells
// picked with divisions: 46 us).
__global__ void __launch_bounds__(256) batch_prep_kernel(
    const double* states, const uint32_t* n_rays, uint32_t n_states,
    uint32_t max_rays, DevMap m, EvalConsts k, BatchHeader* hdr, BatchState* bs,
    uint32_t* sticket, uint32_t* gticket, rmp_result_t* out) {
  __shared__ uint32_t sh[8], scan[3][8];
  wait_previous();
  launch_next();
  const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t per = (n_states + gridDim.x - 1) / gridDim.x;
  const uint32_t s0 = min(blockIdx.x * per, n_states), s1 = min(s0 + per, n_states);
  // rays of the batch in units of 16, rounded up per state (32 bits hold them: a workspace takes
  // about 10 bytes a ray)
  uint32_t load = 0;
  for (uint32_t j = tid; j < n_states; j += 256)
    load += n_rays[j] <= max_rays ? (n_rays[j] + 15) / 16 : 0u;
  const unsigned long long total = 16ull * block_sum256(load, sh);
  uint32_t before_w = 0, before_p = 0, before_g = 0, all_w = 0;
  for (uint32_t j = tid; j < n_states; j += 256) {
    const uint32_t n = n_rays[j];
    if (n > max_rays) continue;
    const uint32_t lg = state_lg_segs(k, n), parts = ((n << lg) + 31) / 32;
    const uint32_t work = ((n << march_lg_segs(k, lg, total)) + 31) / 32;
    all_w += work;
    if (j < s0) {
      before_w += work;
      before_p += parts;
      before_g += (parts + kBatchGroup - 1) / kBatchGroup;
    }
  }
  before_w = block_sum256(before_w, sh);
  before_p = block_sum256(before_p, sh);
  before_g = block_sum256(before_g, sh);
  if (blockIdx.x == 0) {
    all_w = block_sum256(all_w, sh);
    if (tid == 0) {
      hdr->next_chunk = 0;
      hdr->total_chunks = all_w;
      hdr->n_states = n_states;
    }
  }
  const uint32_t first_g = before_g;
  for (uint32_t base = s0; base < s1; base += 256) {
    const uint32_t tile = min(256u, s1 - base);
    const uint32_t n = tid < tile ? n_rays[base + tid] : 0u;
    const uint32_t lg = state_lg_segs(k, n), lgs = march_lg_segs(k, lg, total);
    const uint32_t nv = n <= max_rays ? n : 0u;
    // work chunks, partials and groups of this thread's state, then their inclusive scans
    const uint32_t v[3] = {((nv << lgs) + 31) / 32, ((nv << lg) + 31) / 32,
                           (((nv << lg) + 31) / 32 + kBatchGroup - 1) / kBatchGroup};
    uint32_t inc[3] = {v[0], v[1], v[2]};
#pragma unroll
    for (int off = 1; off < 32; off <<= 1)
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, inc[i], off);
        if (lane >= (uint32_t)off) inc[i] += y;
      }
    __syncthreads();                                // the last tile's scan is no longer read
    if (lane == 31)
#pragma unroll
      for (int i = 0; i < 3; ++i) scan[i][warp] = inc[i];
    __syncthreads();
    uint32_t all[3] = {0, 0, 0};
#pragma unroll
    for (uint32_t w = 0; w < 8; ++w)
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        if (w == warp) inc[i] += all[i];
        all[i] += scan[i][w];
      }
    if (tid < tile) {
      BatchState* sp = bs + base + tid;
      sp->n_rays = n;
      sp->work0 = before_w + inc[0] - v[0];
      sp->part0 = before_p + inc[1] - v[1];
      sp->group0 = before_g + inc[2] - v[2];
      sp->lg_segs = lg | (lgs << 8);
      sticket[base + tid] = 0;
    }
    before_w += all[0];
    before_p += all[1];
    before_g += all[2];
    for (uint32_t j = warp; j < tile; j += 8) {
      const uint32_t b = base + j;
      const uint32_t nb = n_rays[b];
      const double* x = states + 6 * (size_t)b;
      BatchState* sp = bs + b;
      bool bad = false;
      if (lane < 3) {
        const double o = m.kind != RMP_MAP_DENSE_U8 ? 0.0
                         : (lane == 0 ? m.origin[0] : (lane == 1 ? m.origin[1] : m.origin[2]));
        const double q = __dmul_rn(__ddiv_rn(__dsub_rn(x[lane], o), m.vs), 65536.0);
        bad = !(fabs(q) < 274877906944.0);
        sp->P[lane] = bad ? 0 : __double2ll_rn(q);
      } else if (lane < 6) {
        const double v = x[lane];
        const float vh = __double2float_rn(v);
        sp->v[lane - 3] = vh;
        sp->vl[lane - 3] = __double2float_rn(__dsub_rn(v, (double)vh));
      }
      bad = __any_sync(0xffffffffu, bad) || nb > max_rays;
      const uint32_t M = nb >= 32 ? pick_cells_warp(nb) : 1u;
      if (lane == 0) {
        sp->status = bad ? RMP_ERR_INVALID_ARG : RMP_OK;
        sp->perm_M = M;
        sp->perm_Q = nb / M;
      }
      if (bad || nb == 0) {                         // 18 8-byte words of result
        const unsigned long long w =
            lane == 15 ? (unsigned long long)nb
                       : (lane == 17 && bad ? (unsigned long long)RMP_ERR_INVALID_ARG : 0ull);
        if (lane < 18) reinterpret_cast<unsigned long long*>(out + b)[lane] = w;
      }
    }
  }
  for (uint32_t i = first_g + tid; i < before_g; i += 256) gticket[i] = 0;
}

// Lane i's terms and counts of a chunk partial (FP32 pairs for the compensated reduction, as
// CtaPartial32) or of a group partial (FP64), read past L1: another SM wrote it.
template <bool PAIR>
__device__ __forceinline__ void load_partial(const CtaPartial* p, double v[9], unsigned& h,
                                             unsigned& a) {
  if (PAIR) {
    const uint4* q = reinterpret_cast<const uint4*>(p);
    uint32_t w[20];
#pragma unroll
    for (int i = 0; i < 5; ++i) {
      const uint4 x = __ldcg(q + i);
      w[4 * i] = x.x;
      w[4 * i + 1] = x.y;
      w[4 * i + 2] = x.z;
      w[4 * i + 3] = x.w;
    }
#pragma unroll
    for (int i = 0; i < 9; ++i)
      v[i] = (double)__uint_as_float(w[i]) + (double)__uint_as_float(w[9 + i]);
    h = w[18];
    a = w[19];
  } else {
#pragma unroll
    for (int i = 0; i < 9; ++i) v[i] = __ldcg(&p->v[i]);
    h = __ldcg(&p->n_hits);
    a = __ldcg(&p->n_active);
  }
}

// Sum of 32 lanes' FP64 terms into *p (or the lanes' slot 0, p null), counts into h, a.
__device__ __forceinline__ void warp_sum_partial(double (&v)[9], unsigned& h, unsigned& a,
                                                 CtaPartial* p) {
  const WarpTerms t = warp_terms(0);
  warp_reduce_terms<double, false>(v, v, 0);
  h = __reduce_add_sync(0xffffffffu, h);
  a = __reduce_add_sync(0xffffffffu, a);
  if (p) {
    if (t.n > 0) p->v[t.first] = v[0];
    if ((threadIdx.x & 31) == 0) {
      p->n_hits = h;
      p->n_active = a;
    }
  }
}

// Attractor policy (Sec. III-B, Eq. attractorPolicy): f_a = alpha s(goal - x) - beta xdot in FP64,
// component a in lane a (0-2).  Called by all lanes of a warp, so that the root, the exponential
// and the division are one warp instruction stream (an FP64 instruction holds the pipe about
// 64 cycles whatever the lanes).
__device__ __noinline__ double attractor(const EvalConsts& k, const double* st,
                                         const double* goal) {
  const uint32_t lane = threadIdx.x & 31, a = lane < 3 ? lane : 0;
  const double va = goal[a] - st[a];
  const double v0 = __shfl_sync(0xffffffffu, va, 0), v1 = __shfl_sync(0xffffffffu, va, 1),
               v2 = __shfl_sync(0xffffffffu, va, 2);
  const double z = sqrt(v0 * v0 + v1 * v1 + v2 * v2);
  const double h = z + k.c64 * log1p(exp(-2.0 * k.c64 * z));
  return k.att_alpha * (va / h) - k.att_beta * st[3 + a];
}

template <int KIND>
__device__ __forceinline__ bool outside(const DevMap& m, const int k[3]) {
  return KIND == RMP_MAP_DENSE_U8 &&
         ((unsigned)k[0] >= (unsigned)m.dims[0] || (unsigned)k[1] >= (unsigned)m.dims[1] ||
          (unsigned)k[2] >= (unsigned)m.dims[2]);
}

// Occupancy of voxel (kx, ky, kz) (global voxel coordinates, inside the map for dense
// maps): its bit of the block's brick.
template <int LAYOUT>
__device__ __forceinline__ bool voxel_occupied(const DevMap& m, int kx, int ky, int kz) {
  long long at;
  if (LAYOUT == kLayoutGrid) {
    const int x = (kx >> 3) - m.gmin[0], y = (ky >> 3) - m.gmin[1], z = (kz >> 3) - m.gmin[2];
    if ((unsigned)x >= (unsigned)m.gdim[0] || (unsigned)y >= (unsigned)m.gdim[1] ||
        (unsigned)z >= (unsigned)m.gdim[2])
      return false;
    at = x + (long long)m.gdim[0] * (y + (long long)m.gdim[1] * z);
  } else {
    uint32_t slot;
    at = hash_lookup(m, kx >> 3, ky >> 3, kz >> 3, slot);
    if (at < 0) return false;
  }
  const uint32_t p = (uint32_t)((kx & 7) | ((ky & 7) << 3) | ((kz & 7) << 6));
  return (__ldg(reinterpret_cast<const uint32_t*>(m.bricks) + 16 * at + (p >> 5)) >> (p & 31u)) & 1u;
}

// One control step of a point robot (Sec. IV-A closed loop): the combined policy's acceleration f
// is integrated by semi-implicit Euler in FP64, xdot' = xdot + f dt, x' = x + xdot' dt; then, in
// this order: outside a dense grid -> LEFT_MAP; the voxel of x' occupied -> COLLIDED; |x' - goal| <
// goal_tol -> REACHED; steps == max_steps -> TIMEOUT.  Every seg_steps steps the displacement since
// the last segment end is a segment, and consecutive segments A, B add 1 - acos(cos(A, B)) / pi to
// the smoothness sum.  In two parts, called by a warp with axis a in lane a (0-2; an FP64
// instruction costs the same for one lane or three): what the next evaluation waits for, and the
// rest.
struct RolloutMove {
  double x, xn, v;          // position before and after, new velocity
  long long fx;             // the new position, quantised
  bool far;                 // it is beyond the fixed-point range
};

template <int KIND>
__device__ __forceinline__ RolloutMove rollout_move(const DevMap& m, const RolloutConsts& rc,
                                                    double x, double v, double f) {
  const uint32_t lane = threadIdx.x & 31;
  RolloutMove w;
  w.x = x;
  w.v = __fma_rn(f, rc.dt, v);
  w.xn = __fma_rn(w.v, rc.dt, x);
  const double o = KIND == RMP_MAP_DENSE_U8
                       ? (lane == 1 ? m.origin[1] : (lane == 2 ? m.origin[2] : m.origin[0]))
                       : 0.0;
  const double q = __dmul_rn(__ddiv_rn(__dsub_rn(w.xn, o), m.vs), 65536.0);
  w.far = __any_sync(0xffffffffu, lane < 3 && !(fabs(q) < 274877906944.0));
  w.fx = w.far ? 0 : __double2ll_rn(q);
  return w;
}

// The step's path, segment and ending into the robot's record r.  Returns the status in lane 0.
template <int KIND, int LAYOUT>
__device__ __noinline__ uint32_t rollout_book(const DevMap& m, const RolloutConsts& rc,
                                              RolloutDev& r, double x, double xn, double goal,
                                              long long fx, bool far) {
  const uint32_t lane = threadIdx.x & 31, a = lane < 3 ? lane : 0;
  auto of = [](double v, int i) { return __shfl_sync(0xffffffffu, v, i); };
  // (v0 w0 + v1 w1) + v2 w2 of two vectors that lie across the lanes, in every lane
  auto dot3 = [&](double v, double w) {
    const double p = __dmul_rn(of(v, 0), of(w, 0));
    return __fma_rn(of(v, 2), of(w, 2), __fma_rn(of(v, 1), of(w, 1), p));
  };
  const double path = r.path_length;
  const uint32_t steps = r.steps + 1;
  const double dl = dot3(xn - x, xn - x);
  if (rc.seg_steps && steps % rc.seg_steps == 0) {
    const double seg = xn - r.seg_start[a], prev = r.prev_seg[a];
    const bool have = r.have_prev != 0;
    __syncwarp();                                   // every lane has read what lanes 0-2 write below
    if (have) {
      const double dot = dot3(prev, seg), na = dot3(prev, prev), nb = dot3(seg, seg);
      if (na > 0.0 && nb > 0.0) {
        double cs = dot / (sqrt(na) * sqrt(nb));
        cs = cs > 1.0 ? 1.0 : (cs < -1.0 ? -1.0 : cs);
        const double add = 1.0 - acos(cs) / 3.14159265358979323846;
        if (lane == 0) {
          r.smooth_sum += add;
          r.smooth_n += 1;
        }
      }
    }
    if (lane < 3) {
      r.seg_start[a] = xn;
      r.prev_seg[a] = seg;
    }
    if (lane == 0) r.have_prev = 1;
  }
  const int ka = (int)(fx >> 16);
  const int k[3] = {__shfl_sync(0xffffffffu, ka, 0), __shfl_sync(0xffffffffu, ka, 1),
                    __shfl_sync(0xffffffffu, ka, 2)};
  const double dg = dot3(xn - goal, xn - goal);
  const double len = sqrt(lane == 1 ? dg : dl);    // lane 0: the step's, lane 1: to the goal
  const double to_goal = of(len, 1);
  if (lane != 0) return 0;
  uint32_t status = RMP_ROLLOUT_RUNNING;
  if (far || (KIND == RMP_MAP_DENSE_U8 && outside<KIND>(m, k))) status = RMP_ROLLOUT_LEFT_MAP;
  else if (voxel_occupied<LAYOUT>(m, k[0], k[1], k[2])) status = RMP_ROLLOUT_COLLIDED;
  else if (to_goal < rc.goal_tol) status = RMP_ROLLOUT_REACHED;
  else if (steps >= rc.max_steps) status = RMP_ROLLOUT_TIMEOUT;
  r.path_length = path + len;
  r.steps = steps;
  r.status = status;
  return status;
}

// Running robot b's control step in device memory, f_a in lane a.  A robot that stops gets 0 rays
// from then on.
template <int KIND, int LAYOUT>
__device__ __forceinline__ void rollout_step(const DevMap& m, const RolloutArgs& g, uint32_t b,
                                             double f) {
  const uint32_t lane = threadIdx.x & 31, a = lane < 3 ? lane : 0;
  double* st = g.states + 6 * (size_t)b;
  const RolloutMove w = rollout_move<KIND>(m, g.rc, st[a], st[3 + a], f);
  if (lane < 3) {
    st[3 + a] = w.v;
    st[a] = w.xn;
  }
  const uint32_t status = rollout_book<KIND, LAYOUT>(m, g.rc, g.rs[b], w.x, w.xn,
                                                     g.goals[3 * (size_t)b + a], w.fx, w.far);
  if (lane != 0) return;
  if (status != RMP_ROLLOUT_RUNNING) g.n_rays[b] = 0;
  else if (g.running) atomicAdd(g.running, 1u);
}

// A robot whose evaluation failed stops.
__device__ __forceinline__ void rollout_fail(const RolloutArgs& g, uint32_t b) {
  g.rs[b].status = RMP_ROLLOUT_FAILED;
  g.n_rays[b] = 0;
}

// The last chunk of a group sums the group's partials into a group partial; the last group
// of a state sums the state's groups, adds the attractor (combined evaluations) and
// resolves.  Called by all 32 lanes of the warp whose chunk completed the group.  Kept
// out of line: it runs once per 32 partials, and inlined it would sit between the march
// loops in the instruction stream.  A partial's FP32 pairs become FP64 here, one partial
// per lane, not where they are stored: an FP64 instruction holds a scheduler's pipe about 64
// cycles whatever the active lanes (256 states: 17.2 M -> 1.3 M FP64 warp instructions; with the
// shared-out trees 1289 -> 1000 us).
template <int KIND, int LAYOUT, int RED>
__device__ __noinline__ void batch_group_finish(const DevMap& m, const EvalConsts& k,
                                                const RolloutArgs& step, CtaPartial* cparts,
                                                CtaPartial* gparts, uint32_t* sticket,
                                                uint32_t part0, uint32_t gi, uint32_t gsz,
                                                uint32_t n_parts, uint32_t chunks, uint32_t group0,
                                                uint32_t b,
                                                uint32_t n_b, const double* states,
                                                const double* goals, rmp_result_t* out) {
  const uint32_t lane = threadIdx.x & 31;
  // the group's partials, lane i: partial i
  __threadfence();
  double v[9] = {0., 0., 0., 0., 0., 0., 0., 0., 0.};
  unsigned th = 0, ta = 0;
  if (lane < gsz)
    load_partial<RED == RMP_REDUCE_KAHAN32>(cparts + part0 + gi * kBatchGroup + lane, v, th, ta);
  const uint32_t n_groups = (n_parts + kBatchGroup - 1) / kBatchGroup;
  warp_sum_partial(v, th, ta, n_groups > 1 ? gparts + group0 + gi : nullptr);
  if (n_groups > 1) {                               // (a single group's sums are the state's)
    __threadfence();
    __syncwarp();
    uint32_t last = 0;
    if (lane == 0) last = atomicAdd(&sticket[b], 1u) == n_groups - 1 ? 1u : 0u;
    if (!__shfl_sync(0xffffffffu, last, 0)) return;
    // last group of the state: lane i sums groups i, i + 32, ... in order, then the tree
    __threadfence();
#pragma unroll
    for (int i = 0; i < 9; ++i) v[i] = 0.0;
    th = ta = 0;
    for (uint32_t j = lane; j < n_groups; j += 32) {
      double pv2[9];
      unsigned h2, a2;
      load_partial<false>(gparts + group0 + j, pv2, h2, a2);
#pragma unroll
      for (int i = 0; i < 9; ++i) v[i] += pv2[i];
      th += h2;
      ta += a2;
    }
    warp_sum_partial(v, th, ta, nullptr);
  }
  // combined with the attractor (Eq. 1, metric I): the ray sums (or their mean, divided in the
  // lanes that hold them) plus its terms
  double mine = v[0];
  double att = 0.0;
  if (goals) {
    if (k.att_mean) mine = mine / (double)n_b;
    // the first of several chunks has left it in the record
    att = chunks > 1 ? __ldcg(&out[b].f[lane < 3 ? lane : 0])
                     : attractor(k, states + 6 * (size_t)b, goals + 3 * (size_t)b);
  }
  // every lane gets all terms back from the lanes that hold them (warp_terms(0))
  constexpr int kHolder[9] = {0, 2, 4, 8, 10, 16, 18, 20, 24};
  double tv[9];
#pragma unroll
  for (int i = 0; i < 9; ++i) tv[i] = __shfl_sync(0xffffffffu, mine, kHolder[i]);
  if (goals) {
    tv[0] += 1.0;
    tv[3] += 1.0;
    tv[5] += 1.0;
#pragma unroll
    for (int i = 0; i < 3; ++i) tv[6 + i] += __shfl_sync(0xffffffffu, att, i);
  }
  rmp_result_t r;
  resolve_pinv(tv, tv + 6, r);
  if (lane == 0) {
#pragma unroll
    for (int i = 0; i < 6; ++i) r.A[i] = tv[i];
#pragma unroll
    for (int i = 0; i < 3; ++i) r.Af[i] = tv[6 + i];
    r.n_rays = n_b;
    r.n_hits = th;
    r.n_active = ta;
    r.status = RMP_OK;
    r.reserved = 0;
    out[b] = r;
  }
  if (step.rs) {                                    // a rollout: the robot's control step follows
    const double f0 = __shfl_sync(0xffffffffu, r.f[0], 0), f1 = __shfl_sync(0xffffffffu, r.f[1], 0),
                 f2 = __shfl_sync(0xffffffffu, r.f[2], 0);
    rollout_step<KIND, LAYOUT>(m, step, b, lane == 1 ? f1 : (lane == 2 ? f2 : f0));
  }
}

// Persistent batched evaluation: every warp takes work chunks (its own index first, then from
// the work counter) until none is left; a chunk is 32 / s rays of one state (coherent ray order of
// that state), marched and evaluated as in the single-state kernel.  Each partial's 9 terms are
// summed over its lanes (compensated FP32 or FP64 tree), stored, and the partial's group and the
// state's tickets decide which warp sums a group (<= 32 partials, one per lane) and which one
// sums the state's groups and resolves it -- every sum in a fixed order, so results do not
// depend on which warp ran which chunk, nor on s.
// Register budget 64 (launch bounds 256 x 4): 32 warps per SM hide each other's latency; the
// per-state values used only after the march are read after it.
template <int KIND, int LAYOUT, int RED, bool BOXES>
__global__ void __launch_bounds__(256, 4) raycast_batch_kernel(
    const __grid_constant__ DevMap m, const __grid_constant__ EvalConsts k, BatchHeader* hdr, const BatchState* bs,
    uint32_t* sticket, uint32_t* gticket, CtaPartial* cparts, CtaPartial* gparts,
    rmp_result_t* out, rmp_ray_hit_t* hits, float* per_ray, uint32_t max_rays,
    const double* states, const double* goals, const __grid_constant__ RolloutArgs step) {
  const uint32_t lane = threadIdx.x & 31;
  wait_previous();
  launch_next();
  const uint32_t total = *(volatile const uint32_t*)&hdr->total_chunks;
  const uint32_t nst = *(volatile const uint32_t*)&hdr->n_states;
  // first chunk: the warp's index in the grid; later ones from the counter (offset by the
  // number of warps), requested as soon as a chunk starts so the atomic's latency is
  // hidden.  (Same-address atomics are serialised, several ns each: a grid-wide rush on
  // the counter at kernel start would delay every warp's first chunk.)
  const uint32_t n_warps = gridDim.x * (blockDim.x >> 5);
  uint32_t c = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  while (c < total) {
    uint32_t cn = 0xffffffffu;
    if (lane == 0 && total > n_warps) cn = n_warps + atomicAdd(&hdr->next_chunk, 1u);
    // the chunk's state: the last one whose first chunk is <= c, 32 places tested at a time
    uint32_t lo = 0, len = nst;
    while (len > 1) {
      const uint32_t by = (len + 31) / 32, at = lo + lane * by;
      const bool le = lane * by < len && bs[at].work0 <= c;   // true for lane 0
      const uint32_t last = 31 - __clz(__ballot_sync(0xffffffffu, le));
      lo += last * by;
      len = min(by, len - last * by);
    }
    const uint32_t b = lo;
    const BatchState* sp = bs + b;
    if (sp->status != RMP_OK) {              // its result is the prep kernel's
      if (step.rs && lane == 0 && c == sp->work0) rollout_fail(step, b);
      c = __shfl_sync(0xffffffffu, cn, 0);
      continue;
    }
    const long long P[3] = {sp->P[0], sp->P[1], sp->P[2]};
    const uint32_t n_b = sp->n_rays;
    const uint32_t q = c - sp->work0;
    const uint32_t lgs = sp->lg_segs >> 8, S = 1u << lgs;
    const uint32_t g = q * 32 + lane;
    const uint32_t slot = g >> lgs, seg = g & (S - 1);
    const bool active = slot < n_b;
    const uint32_t pM = sp->perm_M, pQ = sp->perm_Q;
    const uint32_t ray_idx = ray_of_slot(active ? slot : 0, pM, pQ, n_b - pQ * pM);
    const Ray ray = make_ray<true>(ray_idx + k.halton_offset);
    const size_t ro = (size_t)b * max_rays + ray_idx;
    uint32_t en, ea;
    const int mstat = march_ray<KIND, LAYOUT, BOXES>(m, k, P, ray, seg, lgs, active, en, ea,
                                              hits ? hits + ro : nullptr);
    // read after the march, so that they are not held in registers across it
    const float v[3] = {sp->v[0], sp->v[1], sp->v[2]};
    const float vl[3] = {sp->vl[0], sp->vl[1], sp->vl[2]};
    const uint32_t part0 = sp->part0, group0 = sp->group0;
    const uint32_t lg = sp->lg_segs & 255u, lgW = lg - lgs;
    float vals[9] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    unsigned nh = 0, na = 0;
    bool adds = false;
    if (active && seg == 0)
      adds = ray_outputs(m, k, ray, mstat, en, ea, v, vl, quiet_state(k, v),
                         per_ray ? per_ray + 9 * ro : nullptr, vals, nh, na);
    // without any, the partials are the zeros that vals holds
    const bool any = __any_sync(0xffffffffu, adds);
    if (!any)
#pragma unroll
      for (int i = 0; i < 9; ++i) vals[i] = 0.0f;
    // the chunk's 2^lgW partials, 32 >> lgW lanes each (a ray's other segments hold zeros)
    const uint32_t n_parts = ((n_b << lg) + 31) / 32;
    const uint32_t first = q << lgW, mine = first + (lane >> (5 - lgW));
    uint32_t cnt = nh | (na << 16);
#pragma unroll
    for (int j = 0; j < 5; ++j) {
      const uint32_t off = 16u >> (lgW + j);
      if (off) cnt += __shfl_xor_sync(0xffffffffu, cnt, off);
    }
    const WarpTerms t = warp_terms(lgW);
    CtaPartial* part = cparts + part0 + mine;
    if (RED == RMP_REDUCE_FP64) {
      double pv[9];
#pragma unroll
      for (int i = 0; i < 9; ++i) pv[i] = any ? (double)vals[i] : 0.0;
      if (any) warp_reduce_terms<double, false>(pv, pv, lgW);
      if (mine < n_parts) {
        if (t.n > 0) part->v[t.first] = pv[0];
        if (t.n > 1) part->v[t.first + 1] = pv[1];
      }
    } else {
      float cv[9] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
      if (any) warp_reduce_terms<float, true>(vals, cv, lgW);
      CtaPartial32* p = reinterpret_cast<CtaPartial32*>(part);
      if (mine < n_parts) {
        if (t.n > 0) {
          p->s[t.first] = vals[0];
          p->c[t.first] = cv[0];
        }
        if (t.n > 1) {
          p->s[t.first + 1] = vals[1];
          p->c[t.first + 1] = cv[1];
        }
      }
    }
    if (mine < n_parts && (lane & ((32u >> lgW) - 1)) == 0) {
      part->n_hits = cnt & 0xffffu;
      part->n_active = cnt >> 16;
    }
    // the warp of a state's first chunk forms its attractor as well, beside the others' marches
    // (6000 cycles of FP64 that would otherwise follow the last chunk), and leaves it in the
    // result's record until the state is resolved; its ticket orders it before that
    const uint32_t chunks = ((n_b << lgs) + 31) / 32;
    if (goals && q == 0 && chunks > 1) {
      const double att = attractor(k, states + 6 * (size_t)b, goals + 3 * (size_t)b);
      if (lane < 3) out[b].f[lane] = att;
    }
    const uint32_t gi = first / kBatchGroup;
    const uint32_t gsz = min(kBatchGroup, n_parts - gi * kBatchGroup);
    const uint32_t stored = min(1u << lgW, n_parts - first);
    uint32_t stage = 0;
    __threadfence();
    __syncwarp();
    if (lane == 0) stage = atomicAdd(&gticket[group0 + gi], stored) + stored == gsz ? 1u : 0u;
    stage = __shfl_sync(0xffffffffu, stage, 0);
    if (stage)
      batch_group_finish<KIND, LAYOUT, RED>(m, k, step, cparts, gparts, sticket, part0, gi, gsz,
                                            n_parts, chunks, group0, b, n_b, states, goals, out);
    c = __shfl_sync(0xffffffffu, cn, 0);
  }
}

// ------------------------------------------------------------------ one CTA per state
// Where states have few rays (state_per_cta, rollout_resident) a CTA evaluates one by itself: its
// partials lie in shared memory, so there is no set-up launch, ticket or fence, and a state waits
// for its own slowest warp.  Every sum is cut and ordered as in raycast_batch_kernel.
constexpr uint32_t kPartWords = 18;                 // a partial: 9 FP32 pairs or 9 doubles

// Named barriers 1 (in resolve_pinv_cta) to 4; arrival only for the warps that go on.
__device__ __forceinline__ void bar_arrive(int id, uint32_t threads) {
  asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
__device__ __forceinline__ void bar_sync(int id, uint32_t threads) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

// Chunk q of a state (a warp): its rays' segments marched and evaluated, its partials stored.
template <int KIND, int LAYOUT, int RED, bool BOXES>
__device__ __forceinline__ void state_chunk(const DevMap& m, const EvalConsts& k,
                                            const long long* Ps, const float* vs, const float* vls,
                                            const Ray& ray, uint32_t q, uint32_t n, uint32_t lg,
                                            uint32_t lgs, float* parts, rmp_ray_hit_t* hit,
                                            float* per, unsigned& nh, unsigned& na) {
  const uint32_t lane = threadIdx.x & 31, gl = q * 32 + lane, seg = gl & ((1u << lgs) - 1);
  const uint32_t lgW = lg - lgs, n_parts = ((n << lg) + 31) / 32;
  const bool active = (gl >> lgs) < n;
  const long long P[3] = {Ps[0], Ps[1], Ps[2]};
  uint32_t en, ea;
  const int mstat = march_ray<KIND, LAYOUT, BOXES>(m, k, P, ray, seg, lgs, active, en, ea, hit);
  const float v[3] = {vs[0], vs[1], vs[2]}, vl[3] = {vls[0], vls[1], vls[2]};
  float vals[9] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
  bool adds = false;
  if (active && seg == 0)
    adds = ray_outputs(m, k, ray, mstat, en, ea, v, vl, quiet_state(k, v), per, vals, nh, na);
  const bool any = __any_sync(0xffffffffu, adds);
  if (!any)
#pragma unroll
    for (int i = 0; i < 9; ++i) vals[i] = 0.0f;
  const uint32_t mine = (q << lgW) + (lane >> (5 - lgW));
  const WarpTerms t = warp_terms(lgW);
  float* part = parts + kPartWords * mine;
  if (RED == RMP_REDUCE_FP64) {
    double pv[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) pv[i] = any ? (double)vals[i] : 0.0;
    if (any) warp_reduce_terms<double, false>(pv, pv, lgW);
    double* pd = reinterpret_cast<double*>(part);
    if (mine < n_parts) {
      if (t.n > 0) pd[t.first] = pv[0];
      if (t.n > 1) pd[t.first + 1] = pv[1];
    }
  } else {
    float cv[9] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    if (any) warp_reduce_terms<float, true>(vals, cv, lgW);
    if (mine < n_parts) {
      if (t.n > 0) {
        part[t.first] = vals[0];
        part[9 + t.first] = cv[0];
      }
      if (t.n > 1) {
        part[t.first + 1] = vals[1];
        part[9 + t.first + 1] = cv[1];
      }
    }
  }
}

// s + c of an FP32 pair in FP64.  A normal value is widened by integer instructions (an FP64
// conversion holds the pipe about 64 cycles); the rare others by the conversion.  For a CTA whose
// other warps wait; where they march the integers cost more (64 states of 4096 rays packed 72 ->
// 73.5 us).
__device__ __forceinline__ double pair_sum(float s, float c) {
  auto plain = [](float f) {                        // zero or normal
    const uint32_t b = __float_as_uint(f) << 1;
    return b == 0u || (b >= 0x01000000u && b < 0xff000000u);
  };
  if (plain(s) && plain(c)) return widen(s) + widen(c);
  return (double)s + (double)c;
}

// The sums of a state from its partials, called by all warps after a barrier: a warp per group,
// then term `lane` (0-8) of the groups in those lanes of warp 0, in the order of a tree over lanes.
template <int RED>
__device__ __forceinline__ double state_sum(const float* parts, uint32_t n_parts,
                                            double (*gsum)[9]) {
  const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const uint32_t n_groups = (n_parts + kBatchGroup - 1) / kBatchGroup;
  for (uint32_t gi = warp; gi < n_groups; gi += nw) {
    const uint32_t at = gi * kBatchGroup + lane;
    const float* part = parts + kPartWords * at;
    double v[9];
#pragma unroll
    for (int i = 0; i < 9; ++i)
      v[i] = at >= n_parts ? 0.0
             : RED == RMP_REDUCE_FP64 ? reinterpret_cast<const double*>(part)[i]
                                      : pair_sum(part[i], part[9 + i]);
    warp_reduce_terms<double, false>(v, v, 0);
    const WarpTerms t = warp_terms(0);
    if (t.n > 0) gsum[gi][t.first] = v[0];
  }
  const uint32_t group_warps = min(n_groups, nw);
  if (warp > 0 && warp < group_warps) bar_arrive(2, 32 * group_warps);
  if (warp > 0) return 0.0;
  if (group_warps > 1) bar_sync(2, 32 * group_warps);
  else __syncwarp();
  double v[kStateGroups];
#pragma unroll
  for (uint32_t i = 0; i < kStateGroups; ++i) v[i] = lane < 9 && i < n_groups ? gsum[i][lane] : 0.0;
#pragma unroll
  for (uint32_t off = kStateGroups / 2; off > 0; off >>= 1)
    if (n_groups > off)
#pragma unroll
      for (uint32_t i = 0; i < off; ++i) v[i] += v[i + off];
  return v[0];
}

// A state quantised by warp 0, a component a lane (0-5); returns whether the position is unusable.
template <int KIND>
__device__ __forceinline__ bool quantise_state(const DevMap& m, double x, long long* P, float* v,
                                               float* vl) {
  const uint32_t lane = threadIdx.x & 31;
  bool bad = false;
  if (lane < 3) {
    const double o = KIND != RMP_MAP_DENSE_U8 ? 0.0
                     : (lane == 0 ? m.origin[0] : (lane == 1 ? m.origin[1] : m.origin[2]));
    const double q = __dmul_rn(__ddiv_rn(__dsub_rn(x, o), m.vs), 65536.0);
    bad = !(fabs(q) < 274877906944.0);
    P[lane] = bad ? 0 : __double2ll_rn(q);
  } else if (lane < 6) {
    const float vh = __double2float_rn(x);
    v[lane - 3] = vh;
    vl[lane - 3] = __double2float_rn(__dsub_rn(x, (double)vh));
  }
  return __any_sync(0xffffffffu, bad);
}

// Segments marched per ray (log2): a tuned launch's, else the most whose chunks `warps` warps hold
// at once, at most the summation's lg.
__host__ __device__ __forceinline__ uint32_t cta_lg_segs(const EvalConsts& k, uint32_t n,
                                                         uint32_t lg, uint32_t warps) {
  if (k.lg_segs <= 2u) return lg;
  while (lg > 0 && ((n << lg) + 31) / 32 > warps) --lg;
  return lg;
}

// A batch of few-ray states, a CTA each (see state_per_cta): set up, marched, summed and resolved
// in one launch; the last warp forms the attractor after its chunks.  Bound by that chain.
// 128 states of 256 rays with the attractor: 17.8 us (set-up and persistent grid 30); 304 of 1024:
// 43 (77).
struct StateShared {
  double S[9], att[3];
  double gsum[kStateGroups][9];
  long long P[3];
  float v[3], vl[3];
  rmp_result_t res;
  uint32_t n, cells;
  unsigned hits, active;
  int bad;
};

template <int KIND, int LAYOUT, int RED, bool BOXES>
__global__ void __launch_bounds__(1024, 1) raycast_state_kernel(
    const __grid_constant__ DevMap m, const __grid_constant__ EvalConsts k,
    const double* states, const uint32_t* n_rays, uint32_t max_rays,
    rmp_result_t* out, rmp_ray_hit_t* hits, float* per_ray, const double* goals, uint32_t most) {
  extern __shared__ __align__(16) float parts[];
  __shared__ StateShared sh;
  const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const uint32_t b = blockIdx.x;
  wait_previous();
  const double* st = states + 6 * (size_t)b;
  if (warp == 0) {
    const bool bad = quantise_state<KIND>(m, lane < 6 ? st[lane] : 0.0, sh.P, sh.v, sh.vl);
    if (lane == 0) {
      sh.bad = bad;
      sh.hits = sh.active = 0;
    }
  } else if (warp == 1) {
    const uint32_t n = n_rays[b], M = n >= 32 ? pick_cells_warp(n) : 1u;
    if (lane == 0) {
      sh.n = n;
      sh.cells = M;
    }
  }
  __syncthreads();
  const uint32_t n = sh.n;
  const bool bad = sh.bad || n > max_rays;
  if (bad || n == 0) {                              // 18 8-byte words of result
    const unsigned long long w =
        lane == 15 ? (unsigned long long)n
                   : (lane == 17 && bad ? (unsigned long long)RMP_ERR_INVALID_ARG : 0ull);
    if (threadIdx.x < 18) reinterpret_cast<unsigned long long*>(out + b)[threadIdx.x] = w;
    launch_next();
    return;
  }
  const uint32_t lg = state_lg_segs(k, n), lgs = cta_lg_segs(k, n, lg, most);
  const uint32_t n_parts = ((n << lg) + 31) / 32, chunks = ((n << lgs) + 31) / 32;
  const uint32_t M = sh.cells, Q = n / M;
  unsigned nh = 0, na = 0;
  for (uint32_t q = warp; q < chunks; q += nw) {
    const uint32_t slot = (q * 32 + lane) >> lgs;
    const uint32_t ray_idx = ray_of_slot(slot < n ? slot : 0, M, Q, n - Q * M);
    const Ray ray = make_ray<true>(ray_idx + k.halton_offset);
    const size_t ro = (size_t)b * max_rays + ray_idx;
    state_chunk<KIND, LAYOUT, RED, BOXES>(m, k, sh.P, sh.v, sh.vl, ray, q, n, lg, lgs, parts,
                                          hits ? hits + ro : nullptr,
                                          per_ray ? per_ray + 9 * ro : nullptr, nh, na);
  }
  launch_next();
  nh = __reduce_add_sync(0xffffffffu, nh);
  na = __reduce_add_sync(0xffffffffu, na);
  if (lane == 0 && nh) {
    atomicAdd(&sh.hits, nh);
    atomicAdd(&sh.active, na);
  }
  if (goals && warp == nw - 1) {
    const double att = attractor(k, st, goals + 3 * (size_t)b);
    if (lane < 3) sh.att[lane] = att;
  }
  __syncthreads();                                  // partials, counts, attractor
  double mine = state_sum<RED>(parts, n_parts, sh.gsum);
  if (warp == 0) {
    if (lane < 9) {
      if (goals) {
        if (k.att_mean) mine = mine / (double)n;
        if (lane == 0 || lane == 3 || lane == 5) mine += 1.0;
        if (lane >= 6) mine += sh.att[lane - 6];
      }
      sh.S[lane] = mine;
    }
    __syncwarp();
  }
  if (warp >= 2) return;
  bar_sync(4, 64);
  resolve_pinv_cta(sh.S, sh.S + 6, sh.res);
  if (warp == 1) return;
  if (lane < 6) sh.res.A[lane] = sh.S[lane];
  else if (lane < 9) sh.res.Af[lane - 6] = sh.S[lane];
  else if (lane == 9) {
    sh.res.n_rays = n;
    sh.res.n_hits = sh.hits;
    sh.res.n_active = sh.active;
    sh.res.status = RMP_OK;
    sh.res.reserved = 0;
  }
  __syncwarp();
  if (lane < 18)
    reinterpret_cast<unsigned long long*>(out + b)[lane] =
        reinterpret_cast<const unsigned long long*>(&sh.res)[lane];
}

// ------------------------------------------------------------------ resident rollouts
// A robot's control steps depend on its own steps alone, so one CTA takes one robot through all its
// steps: no launch, set-up, ticket or fence between steps, the robot, its ray directions (the same
// at every step) and the partials in shared memory, and a robot waits for its own slowest warp
// instead of the launch's (where this is taken: rollout_resident).  Every sum is cut and ordered as
// in raycast_batch_kernel (see state_lg_segs, batch_group_finish).
// A step: the warps march the chunks, 32 / s rays each; the last two, which have no chunk where the
// CTA has room, form the attractor and book the step before (whose ending so only decides after
// the march whether it counts); a warp per group of 32 partials sums it; warp 0 sums the groups,
// solves and moves the robot.
// Bound by that chain: the slowest of a robot's marches (13 us of 1024 rays, their mean 6) and
// the FP64 after it.
// 128 robots of 1024 rays, 48 steps: 1380 us, of which the call itself about 450 (set-up and
// evaluation launched per step: 2690); 16 robots of 64 rays 555 (1455).
struct RolloutShared {
  RolloutDev r;
  double st[6], x0[3], goal[3], att[3], S[9];       // x0: the position before the last step
  double gsum[kStateGroups][9];
  long long P[3];
  float v[3], vl[3];
  rmp_result_t res;
  uint32_t cells;
  int go, far;
};

template <int KIND, int LAYOUT, int RED, bool BOXES>
__global__ void __launch_bounds__(1024, 1) rollout_kernel(const __grid_constant__ DevMap m,
                                                          const __grid_constant__ EvalConsts k,
                                                          const __grid_constant__ RolloutArgs g,
                                                          uint32_t n, uint32_t lg, uint32_t lgs,
                                                          uint32_t steps) {
  extern __shared__ __align__(16) float dyn[];      // directions [6][n], then the partials
  __shared__ RolloutShared sh;
  const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const uint32_t b = blockIdx.x;
  const uint32_t n_parts = ((n << lg) + 31) / 32, chunks = ((n << lgs) + 31) / 32;
  float* parts = dyn + ((6 * n + 3) & ~3u);
  wait_previous();
  if (warp == 0) {
    if (lane < sizeof(RolloutDev) / 8)
      reinterpret_cast<unsigned long long*>(&sh.r)[lane] =
          reinterpret_cast<const unsigned long long*>(g.rs + b)[lane];
    const double x = lane < 6 ? g.states[6 * (size_t)b + lane] : 0.0;
    if (lane < 6) sh.st[lane] = x;
    if (lane < 3) sh.goal[lane] = g.goals[3 * (size_t)b + lane];
    const bool bad = quantise_state<KIND>(m, x, sh.P, sh.v, sh.vl);
    const uint32_t M = n >= 32 ? pick_cells_warp(n) : 1u;
    __syncwarp();
    if (lane == 0) {                                // the other warps learn of a stopped robot by go
      const bool runs = sh.r.status == RMP_ROLLOUT_RUNNING;
      if (runs && bad) g.rs[b].status = RMP_ROLLOUT_FAILED;
      sh.cells = M;
      sh.go = runs && !bad ? 1 : 0;
    }
  }
  __syncthreads();
  if (!sh.go) return;
  for (uint32_t slot = threadIdx.x; slot < n; slot += blockDim.x) {
    const uint32_t M = sh.cells, Q = n / M;
    const Ray ray = make_ray<true>(ray_of_slot(slot, M, Q, n - Q * M) + k.halton_offset);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      dyn[a * n + slot] = ray.dir[a];
      dyn[(3 + a) * n + slot] = __int_as_float(ray.D[a]);
    }
  }
  for (uint32_t step = 0;; ++step) {
    __syncthreads();                                // the state; first: the directions
    const bool last = step == steps;
    for (uint32_t q = warp; q < chunks && !last; q += nw) {
      const uint32_t at = (q * 32 + lane) >> lgs, slot = at < n ? at : 0;
      Ray ray;
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        ray.dir[a] = dyn[a * n + slot];
        ray.D[a] = __float_as_int(dyn[(3 + a) * n + slot]);
      }
      unsigned nh = 0, na = 0;
      state_chunk<KIND, LAYOUT, RED, BOXES>(m, k, sh.P, sh.v, sh.vl, ray, q, n, lg, lgs, parts,
                                            nullptr, nullptr, nh, na);
    }
    if (warp == nw - 1 && step > 0) {
      const uint32_t a = lane < 3 ? lane : 0;
      const uint32_t status = rollout_book<KIND, LAYOUT>(m, g.rc, sh.r, sh.x0[a], sh.st[a],
                                                         sh.goal[a], sh.P[a], sh.far != 0);
      if (lane == 0) sh.go = status == RMP_ROLLOUT_RUNNING;
    }
    if (warp == nw - 2 && !last) {
      const double att = attractor(k, sh.st, sh.goal);
      if (lane < 3) sh.att[lane] = att;
    }
    __syncthreads();                                // the partials, the attractor, the booking
    if (last || !sh.go) break;
    double mine = state_sum<RED>(parts, n_parts, sh.gsum);
    if (warp == 0) {
      if (lane < 9) {
        if (k.att_mean) mine = (n & (n - 1)) == 0 ? mine * g.rc.inv_rays : mine / (double)n;
        if (lane == 0 || lane == 3 || lane == 5) mine += 1.0;
        if (lane >= 6) mine += sh.att[lane - 6];
        sh.S[lane] = mine;
      }
      __syncwarp();
      // A metric I + sum A_i with entries below 1e5 has full rank beyond doubt: its eigenvalues
      // are at least 1 less the FP32 roundings of A_i (1e-6 of the entries), the threshold is 1e-12
      // of the largest.  f is then the adjugate's solution.
      int ok;
      double f = adjugate_solve_warp(sh.S, sh.S + 6, ok);
      if (!__all_sync(0xffffffffu, ok && fabs(sh.S[lane < 6 ? lane : 0]) < 1e5)) {
        resolve_pinv(sh.S, sh.S + 6, sh.res);
        __syncwarp();
        f = sh.res.f[lane < 3 ? lane : 0];
      }
      const uint32_t a = lane < 3 ? lane : 0;
      const RolloutMove w = rollout_move<KIND>(m, g.rc, sh.st[a], sh.st[3 + a], f);
      __syncwarp();
      if (lane < 3) {
        sh.x0[a] = w.x;
        sh.st[a] = w.xn;
        sh.st[3 + a] = w.v;
        sh.P[a] = w.fx;
        const float vh = __double2float_rn(w.v);
        sh.v[a] = vh;
        sh.vl[a] = __double2float_rn(__dsub_rn(w.v, (double)vh));
      }
      if (lane == 0) sh.far = w.far ? 1 : 0;
    }
  }
  if (warp == 0) {
    if (lane < sizeof(RolloutDev) / 8)
      reinterpret_cast<unsigned long long*>(g.rs + b)[lane] =
          reinterpret_cast<const unsigned long long*>(&sh.r)[lane];
    if (lane < 6) g.states[6 * (size_t)b + lane] = sh.st[lane];
    if (lane == 0 && sh.go) atomicAdd(g.running, 1u);
  }
}

// ------------------------------------------------------------------ L2 bandwidth probe
// Reads n16 uint4 words `passes` times, grid-stride, 16-byte loads cached in L2 only
// (ld.global.cg), four independent loads in flight per thread; XOR of everything read per
// CTA into checksum[blockIdx.x].
__global__ void __launch_bounds__(512) probe_l2_kernel(const uint4* __restrict__ buf, size_t n16,
                                                       uint32_t passes, uint64_t* checksum) {
  uint32_t acc = 0;
  const size_t stride = (size_t)gridDim.x * blockDim.x;
  for (uint32_t p = 0; p < passes; ++p) {
    size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    for (; i + 3 * stride < n16; i += 4 * stride) {
      const uint4 a = __ldcg(buf + i), b = __ldcg(buf + i + stride),
                  c = __ldcg(buf + i + 2 * stride), d = __ldcg(buf + i + 3 * stride);
      acc ^= a.x ^ a.y ^ a.z ^ a.w ^ b.x ^ b.y ^ b.z ^ b.w ^ c.x ^ c.y ^ c.z ^ c.w ^ d.x ^ d.y ^
             d.z ^ d.w;
    }
    for (; i < n16; i += stride) {
      const uint4 a = __ldcg(buf + i);
      acc ^= a.x ^ a.y ^ a.z ^ a.w;
    }
  }
  acc = __reduce_xor_sync(0xffffffffu, acc);
  __shared__ uint32_t warp_acc[16];
  if ((threadIdx.x & 31) == 0) warp_acc[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    uint32_t t = 0;
    for (uint32_t w = 0; w < (blockDim.x >> 5); ++w) t ^= warp_acc[w];
    checksum[blockIdx.x] = t;
  }
}

// ------------------------------------------------------------------ ESDF policy (Sec. III-D)
// Signed distance of one primitive at x, in the fixed FP64 order of the ABI's definition
// (explicitly rounded operations: no contraction may change the distance or the argmin).
__device__ __forceinline__ double esdf_prim_sdf(const rmp_primitive_t& p, const double x[3]) {
  const double q0 = __dsub_rn(x[0], p.center[0]), q1 = __dsub_rn(x[1], p.center[1]),
               q2 = __dsub_rn(x[2], p.center[2]);
  if (p.kind == RMP_PRIM_SPHERE)
    return __dsub_rn(__dsqrt_rn(__dadd_rn(__dadd_rn(__dmul_rn(q0, q0), __dmul_rn(q1, q1)),
                                          __dmul_rn(q2, q2))),
                     p.size[0]);
  const double a0 = __dsub_rn(fabs(q0), p.size[0]), a1 = __dsub_rn(fabs(q1), p.size[1]),
               a2 = __dsub_rn(fabs(q2), p.size[2]);
  const double o0 = a0 > 0.0 ? a0 : 0.0, o1 = a1 > 0.0 ? a1 : 0.0, o2 = a2 > 0.0 ? a2 : 0.0;
  const double out = __dsqrt_rn(__dadd_rn(__dadd_rn(__dmul_rn(o0, o0), __dmul_rn(o1, o1)),
                                          __dmul_rn(o2, o2)));
  double in = a0 > a1 ? a0 : a1;
  in = in > a2 ? in : a2;
  in = in < 0.0 ? in : 0.0;
  return __dadd_rn(out, in);
}

// The same distance and, if wanted, its gradient (unit, pointing away from the primitive),
// spheres and boxes in one instruction stream: both are the length of a vector o (the offset
// from the centre; its part outside the box) less a constant, and the gradient is o / |o| (the
// centre of a sphere: 0; inside a box the normal of the nearest face).
__device__ __forceinline__ double esdf_nearest(const rmp_primitive_t& p, const double x[3],
                                               double* g) {
  const bool ball = p.kind == RMP_PRIM_SPHERE;
  double q[3], a[3], o[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    q[i] = __dsub_rn(x[i], p.center[i]);
    a[i] = __dsub_rn(fabs(q[i]), p.size[i]);
    o[i] = ball ? fabs(q[i]) : (a[i] > 0.0 ? a[i] : 0.0);
  }
  const double L = __dsqrt_rn(__dadd_rn(__dadd_rn(__dmul_rn(o[0], o[0]), __dmul_rn(o[1], o[1])),
                                        __dmul_rn(o[2], o[2])));
  if (g) {
    const int k = (a[0] >= a[1] && a[0] >= a[2]) ? 0 : (a[1] >= a[2] ? 1 : 2);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      const double n = L > 0.0 ? __ddiv_rn(o[i], L) : ((!ball && i == k) ? 1.0 : 0.0);
      g[i] = q[i] < 0.0 ? -n : n;
    }
  }
  double in = a[0] > a[1] ? a[0] : a[1];
  in = in > a[2] ? in : a[2];
  in = in < 0.0 ? in : 0.0;
  return __dadd_rn(L, ball ? -p.size[0] : in);
}

// Signed distance of primitive i to FP32 precision, with a bound on its error: S adds up the
// sizes of everything the distance is formed from, and the roundings of the operands, the
// differences, the squares and the root stay below 2^-20.5 S (2^-19 is used) beside an absolute
// term for squares that underflow.  p: centre and kind (1 sphere), size and the primitive's share
// of S, infinite where FP32 squares could overflow: the bound is then infinite too.
__device__ __forceinline__ float esdf_prim_sdf32(const float4 c, const float4 h, const float x[3],
                                                 float x_sum, float& err) {
  const float q0 = x[0] - c.x, q1 = x[1] - c.y, q2 = x[2] - c.z;
  const bool ball = c.w != 0.0f;
  const float a0 = fabsf(q0) - h.x, a1 = fabsf(q1) - h.y, a2 = fabsf(q2) - h.z;
  const float o0 = ball ? q0 : fmaxf(a0, 0.0f), o1 = ball ? q1 : fmaxf(a1, 0.0f),
              o2 = ball ? q2 : fmaxf(a2, 0.0f);
  const float L = __fsqrt_rn(o0 * o0 + o1 * o1 + o2 * o2);
  const float S = x_sum + h.w;
  err = S < 1e18f ? 1.9073486328125e-6f * S + 1e-18f : INFINITY;
  return L + (ball ? -h.x : fminf(fmaxf(fmaxf(a0, a1), a2), 0.0f));
}

// Order-preserving unsigned key of a float that is not NaN, and back.
__device__ __forceinline__ uint32_t float_key(float f) {
  const uint32_t b = __float_as_uint(f);
  return b ^ ((b >> 31) ? 0xffffffffu : 0x80000000u);
}
__device__ __forceinline__ float key_float(uint32_t k) {
  return __uint_as_float(k ^ ((k >> 31) ? 0x80000000u : 0xffffffffu));
}

// The ESDF policy, G states (8, 16 or 32) a CTA.  An FP64 instruction holds a scheduler's pipe
// about 64 cycles whatever its active lanes, so the exact arithmetic runs with a state per lane:
//   1. a warp per state finds the nearest primitive (lane i: i, i + 32, ...) from FP32 distances
//      and their error bounds: it is decided when only one primitive's lower bound lies below
//      the smallest upper bound; otherwise (ties, or closer than FP32 can tell) those primitives
//      are compared by their FP64 distances, the first minimum of a sequential scan winning;
//   2. one warp evaluates the damping part of the obstacle policy of Sec. III-C on (d, gradient),
//      one its repulsion and weight, one the attractor;
//   3. one warp runs the Jacobi sweeps, another the adjugate solve; three warps take one
//      Rayleigh quotient each; the first sorts, decides the rank and writes the results.
// The warps of the serial parts rotate with the CTA and with its turn on an SM, so
// that an SM's CTAs use different schedulers' pipes.  Bound by the FP64 chain of steps 2 and 3;
// four CTAs an SM (64 registers), so that 16384 states are one wave (three: 48 us).  16384 states,
// 200 primitives: 33.6 us (one warp per state, every distance in FP64, policy in one lane: 638);
// 128 states 16 (51).
//
// ROLL: a closed loop.  The CTA takes its robots (g, in place of states and goals) through `steps`
// control steps on map m, one evaluation and a warp per robot for the step each time, while any of
// them runs; `running` counts those that still do.  128 robots, 24 steps, the call: 797 us (two
// launches a step: 917).
template <bool ROLL, int KIND, int LAYOUT>
__global__ void __launch_bounds__(256, 4) esdf_eval_kernel(
    const rmp_primitive_t* __restrict__ prims, const float4* __restrict__ prims32, uint32_t n_prims,
    EsdfConsts k, const double* states_in, const double* goals_in,
    uint32_t n_states, uint32_t G, rmp_result_t* out, double* query,
    const __grid_constant__ DevMap m, const __grid_constant__ RolloutArgs g_roll, uint32_t steps,
    uint32_t* running) {
  __shared__ uint32_t near_sh[32], act_sh[32];
  __shared__ bool bad_sh[32];
  __shared__ double P[7][32], att[3][32], fa[3][32], lam_sh[3][32];
  __shared__ float W[9][32], dv_sh[3][32];
  __shared__ int ok_sh[32];
  const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t role = (warp + blockIdx.x + blockIdx.x / k.sms) & 7u;
  constexpr uint32_t kNone = 0xffffffffu;
  // a rollout's states change from step to step
  const double* states = ROLL ? g_roll.states : states_in;
  const double* goals = ROLL ? g_roll.goals : goals_in;
  wait_previous();
  for (uint32_t base = blockIdx.x * G, step = 0; base < n_states;) {
    for (uint32_t s = warp; s < G && base + s < n_states; s += 8) {
      const double* st = states + 6 * (size_t)(base + s);
      // one component a lane: a single FP64 conversion for all of them
      const double comp = st[lane < 6 ? lane : 0];
      const float cf = __double2float_rn(comp);
      const bool bad = __any_sync(0xffffffffu, (__double2hiint(comp) & 0x7ff00000) == 0x7ff00000);
      uint32_t bi = kNone;
      if (!bad) {
        const float xf[3] = {__shfl_sync(0xffffffffu, cf, 0), __shfl_sync(0xffffffffu, cf, 1),
                             __shfl_sync(0xffffffffu, cf, 2)};
        const float x_sum = fabsf(xf[0]) + fabsf(xf[1]) + fabsf(xf[2]);
        // smallest upper bound; the two smallest lower bounds and the first one's primitive
        float up = INFINITY, lo1 = INFINITY, lo2 = INFINITY;
        uint32_t i1 = kNone;
        for (uint32_t i = lane; i < n_prims; i += 32) {
          float err;
          const float sd = esdf_prim_sdf32(__ldg(prims32 + 2 * i), __ldg(prims32 + 2 * i + 1), xf,
                                           x_sum, err);
          const bool known = err < INFINITY;
          up = fminf(up, known ? sd + err : INFINITY);
          const float lo = known ? sd - err : -INFINITY;
          if (lo < lo1 || i1 == kNone) {
            lo2 = lo1;
            lo1 = lo;
            i1 = i;
          } else {
            lo2 = fminf(lo2, lo);
          }
        }
        const float cut = key_float(__reduce_min_sync(0xffffffffu, float_key(up)));
        const bool mine = i1 != kNone && lo1 <= cut;
        const uint32_t cand = __ballot_sync(0xffffffffu, mine);
        const bool more = __any_sync(0xffffffffu, mine && lo2 <= cut);
        if (__popc(cand) == 1 && !more) {
          bi = __shfl_sync(0xffffffffu, i1, __ffs(cand) - 1);
        } else {
          const double x[3] = {st[0], st[1], st[2]};
          double best = INFINITY;
          for (uint32_t i = lane; i < n_prims; i += 32) {
            float err;
            const float sd = esdf_prim_sdf32(__ldg(prims32 + 2 * i), __ldg(prims32 + 2 * i + 1), xf,
                                             x_sum, err);
            if (err < INFINITY && !(sd - err <= cut)) continue;
            const double e = esdf_prim_sdf(prims[i], x);
            if (e < best) {                   // strict: a lane's earlier primitive wins ties
              best = e;
              bi = i;
            }
          }
#pragma unroll
          for (int off = 16; off > 0; off >>= 1) {
            const double b2 = __shfl_down_sync(0xffffffffu, best, off);
            const uint32_t i2 = __shfl_down_sync(0xffffffffu, bi, off);
            if (b2 < best || (b2 == best && i2 < bi)) {
              best = b2;
              bi = i2;
            }
          }
        }
      }
      if (lane == 0) {
        near_sh[s] = bi;
        bad_sh[s] = bad;
      }
    }
    __syncthreads();
    // a state per lane from here on
    const uint32_t b = base + lane;
    const bool mine = lane < G && b < n_states;
    const double* st = states + 6 * (size_t)(mine ? b : base);
    if ((role == 0 || role == 2) && mine) {
      const double x[3] = {st[0], st[1], st[2]};
      const uint32_t bi = near_sh[lane];
      double d = INFINITY, g[3] = {0.0, 0.0, 0.0};
      if (bi != kNone) {
        const double sd = esdf_nearest(prims[bi], x, role == 0 ? g : nullptr);
        d = sd > 0.0 ? sd : 0.0;
      }
      // obstacle policy (Sec. III-C) on the single pair (d, r = g), FP64
      if (role == 2) {
        double frep = 0.0, w = 0.0;
        if (bi != kNone) frep = k.eta_rep * exp(-d / k.nu_rep);
        if (d < k.r) {
          const double y = (k.r - d) / k.r;               // 1 - d / r, exact difference
          w = k.w_mode == 0 ? y * y : y * y * (1.0 + 2.0 * (d / k.r));
        }
        P[3][lane] = frep;
        P[4][lane] = w;
      } else {
        double z = 0.0, sc = 0.0;
        uint32_t act = 0;
        if (bi != kNone) {
          const double xr = __dadd_rn(__dadd_rn(__dmul_rn(st[3], g[0]), __dmul_rn(st[4], g[1])),
                                      __dmul_rn(st[5], g[2]));
          const bool active = xr < 0.0;
          act = (active && d < k.r) ? 1u : 0u;
          const double m = active ? xr * xr : 0.0;
          const double kd = k.eta_damp / (d / k.nu_damp + k.eps);
          z = kd * m;                                     // |f_damp|
          const double h = z + k.c * log1p(exp(-2.0 * k.c * z));
          sc = h > 0.0 ? z / h : 0.0;
        }
        P[0][lane] = g[0];
        P[1][lane] = g[1];
        P[2][lane] = g[2];
        P[5][lane] = z;
        P[6][lane] = sc;
        act_sh[lane] = act;
        if (query) {
          double* qd = query + 4 * (size_t)b;
          qd[0] = d;
          qd[1] = g[0];
          qd[2] = g[1];
          qd[3] = g[2];
        }
      }
    } else if (role == 1 && mine && goals) {               // attractor, metric I (Eq. 1)
      const double* gl = goals + 3 * (size_t)b;
      const double e0 = gl[0] - st[0], e1 = gl[1] - st[1], e2 = gl[2] - st[2];
      const double zz = sqrt(e0 * e0 + e1 * e1 + e2 * e2);
      const double hh = zz + k.c * log1p(exp(-2.0 * k.c * zz));
      att[0][lane] = k.alpha * (e0 / hh) - k.beta * st[3];
      att[1][lane] = k.alpha * (e1 / hh) - k.beta * st[4];
      att[2][lane] = k.alpha * (e2 / hh) - k.beta * st[5];
    }
    __syncthreads();
    if (!ROLL && base + gridDim.x * G >= n_states) launch_next();   // the CTA's last states
    // the sums, in the warps that need them: A = w sc^2 r r^T, f = (f_rep + z) r
    double tv[9];
    const bool bad = mine && bad_sh[lane];
    if (role < 3 && mine) {
      const double g[3] = {P[0][lane], P[1][lane], P[2][lane]};
      const double alpha_m = P[4][lane] * P[6][lane] * P[6][lane], fr = P[3][lane] + P[5][lane];
      tv[0] = alpha_m * g[0] * g[0];
      tv[1] = alpha_m * g[0] * g[1];
      tv[2] = alpha_m * g[0] * g[2];
      tv[3] = alpha_m * g[1] * g[1];
      tv[4] = alpha_m * g[1] * g[2];
      tv[5] = alpha_m * g[2] * g[2];
      const double rf = fr * ((g[0] * g[0] + g[1] * g[1]) + g[2] * g[2]);
#pragma unroll
      for (int a = 0; a < 3; ++a) tv[6 + a] = alpha_m * rf * g[a];
      if (goals && !bad) {
        tv[0] += 1.0;
        tv[3] += 1.0;
        tv[5] += 1.0;
#pragma unroll
        for (int a = 0; a < 3; ++a) tv[6 + a] += att[a][lane];
      }
    }
    if (role == 0 && mine) {
      float V[3][3] = {{1.f, 0.f, 0.f}, {0.f, 1.f, 0.f}, {0.f, 0.f, 1.f}};
      jacobi_f32(tv, V);
#pragma unroll
      for (int i = 0; i < 9; ++i) W[i][lane] = V[i / 3][i % 3];
    } else if (role == 1 && mine) {
      double f0 = 0.0, f1 = 0.0, f2 = 0.0;
      int ok = 0;
      adjugate_solve(tv, tv + 6, f0, f1, f2, ok);
      fa[0][lane] = f0;
      fa[1][lane] = f1;
      fa[2][lane] = f2;
      ok_sh[lane] = ok;
    }
    __syncthreads();
    if (role < 3 && mine) {                                // eigenvalue `role`: its quotient
      const float w0 = W[role][lane], w1 = W[3 + role][lane], w2 = W[6 + role][lane];
      const double t0 = widen(w0) * (tv[0] * widen(w0) + tv[1] * widen(w1) + tv[2] * widen(w2));
      const double t1 = widen(w1) * (tv[1] * widen(w0) + tv[3] * widen(w1) + tv[4] * widen(w2));
      const double t2 = widen(w2) * (tv[2] * widen(w0) + tv[4] * widen(w1) + tv[5] * widen(w2));
      const float dv = norm2_minus_one(w0, w1, w2);
      const double l = __dadd_rn(__dadd_rn(t0, t1), t2);
      lam_sh[role][lane] = fma(-l, widen(dv), l);
      dv_sh[role][lane] = dv;
    }
    __syncthreads();
    if (role == 0 && mine) {
      rmp_result_t r;
      const double lam[3] = {lam_sh[0][lane], lam_sh[1][lane], lam_sh[2][lane]};
      const float dv[3] = {dv_sh[0][lane], dv_sh[1][lane], dv_sh[2][lane]};
      float V[3][3];
#pragma unroll
      for (int i = 0; i < 9; ++i) V[i / 3][i % 3] = W[i][lane];
      EigenSet es;
      rank_eigen(lam, dv, V, r, es);
      resolve_f(tv + 6, es, fa[0][lane], fa[1][lane], fa[2][lane], ok_sh[lane], r);
#pragma unroll
      for (int i = 0; i < 6; ++i) r.A[i] = tv[i];
#pragma unroll
      for (int i = 0; i < 3; ++i) r.Af[i] = tv[6 + i];
      r.n_rays = 1;
      r.n_hits = near_sh[lane] != kNone ? 1u : 0u;
      r.n_active = act_sh[lane];
      r.status = bad ? RMP_ERR_INVALID_ARG : RMP_OK;
      r.reserved = 0;
      if (bad) {
        r.f[0] = r.f[1] = r.f[2] = 0.0;
        r.eig[0] = r.eig[1] = r.eig[2] = 0.0;
        r.rank = 0;
      }
      out[b] = r;
    }
    __syncthreads();                                       // the next tile reuses the arrays
    if constexpr (!ROLL) {
      base += gridDim.x * G;
    } else {
      bool runs = false;
      for (uint32_t s = warp; s < G && base + s < n_states; s += 8) {
        const uint32_t r = base + s;
        const uint32_t before = g_roll.rs[r].status;
        __syncwarp();                               // every lane has read what lane 0 may write
        if (before != RMP_ROLLOUT_RUNNING) continue;
        if (out[r].status != RMP_OK) {
          if (lane == 0) rollout_fail(g_roll, r);
        } else {
          rollout_step<KIND, LAYOUT>(m, g_roll, r, out[r].f[lane < 3 ? lane : 0]);
        }
        __syncwarp();
        const bool goes = g_roll.rs[r].status == RMP_ROLLOUT_RUNNING;
        runs = runs || goes;
        if (step + 1 == steps && goes && lane == 0) atomicAdd(running, 1u);
      }
      if (!__syncthreads_or(runs) || ++step == steps) break;
    }
  }
}

// ------------------------------------------------------------------ LiDAR scan kernel (Sec. III-G)
template <int RED>
__global__ void __launch_bounds__(256) scan_rmp_kernel(const float* pts, EvalConsts k,
                                                       const double* state,
                                                       WsHeader* ws, CtaPartial* parts,
                                                       rmp_result_t* out, float* per_ray) {
  __shared__ CtaState cs;
  __shared__ float rows[8][288];
  const int comp = state_component(threadIdx.x);
  wait_previous();
  launch_next();                                    // two CTAs an SM, with room for two more
  if (!state) {
    if (threadIdx.x == 0) cs = k.cs0;
  } else if (comp >= 0 && comp < 3) {
    cs.xf[comp] = __double2float_rn(state[comp]);
  } else if (comp >= 3) {
    split_velocity(state[comp], cs, comp - 3);
  }
  __syncthreads();
  typename BlockReduce<RED>::Acc acc;
  BlockReduce<RED>::init(acc);
  unsigned n_hit = 0, n_act = 0;
  const float v[3] = {cs.v[0], cs.v[1], cs.v[2]};
  const float vl[3] = {cs.vl[0], cs.vl[1], cs.vl[2]};
  const bool quiet = quiet_state(k, v);
  bool added = false;
  // warp-uniform trip count: the lanes write their rows together
  for (uint32_t base = blockIdx.x * blockDim.x + (threadIdx.x & ~31u); base < k.n_rays;
       base += gridDim.x * blockDim.x) {
    const uint32_t j = base + (threadIdx.x & 31);
    const bool in = j < k.n_rays;
    float q[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) q[a] = in ? __fsub_rn(pts[3 * (size_t)j + a], cs.xf[a]) : 0.0f;
    float f[3] = {0.f, 0.f, 0.f}, vals[9] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    bool valid = isfinite(q[0]) && isfinite(q[1]) && isfinite(q[2]);
    float d = 0.0f;
    if (valid) {
      d = __fsqrt_rn(__fmaf_rn(q[2], q[2], __fmaf_rn(q[1], q[1], __fmul_rn(q[0], q[0]))));
      valid = in && d > 0.0f && d >= k.min_up && d <= k.max_dn;
    }
    if (valid) {
      const float u[3] = {__fdiv_rn(q[0], d), __fdiv_rn(q[1], d), __fdiv_rn(q[2], d)};
      const bool act = active32(v, u);
      const bool inr = d < k.r_up;
      n_hit += 1;
      n_act += (act && inr) ? 1u : 0u;
      const bool adds = (act && inr) || !quiet;
      if (adds || per_ray) obstacle_policy(k, u, d, v, vl, act, inr, f, vals, vals + 6);
      if (adds) {
        BlockReduce<RED>::add(acc, vals);
        added = true;
      }
    }
    if (per_ray)
      store_rows(per_ray + 9 * (size_t)base, min(32u, k.n_rays - base), f, vals,
                 rows[threadIdx.x >> 5]);
  }
  __shared__ CtaSums sums;
  BlockReduce<RED>::reduce(acc, added, n_hit, n_act, sums, gridDim.x == 1);
  grid_finish<RED>(sums, ws, parts, out, k.n_rays, RMP_OK);
}

// ------------------------------------------------------------------ map build kernels
__device__ __forceinline__ bool brick_any(const uint4* w) {
  const uint4 a = w[0], b = w[1], c = w[2], d = w[3];
  return ((a.x | a.y | a.z | a.w) | (b.x | b.y | b.z | b.w) | (c.x | c.y | c.z | c.w) |
          (d.x | d.y | d.z | d.w)) != 0u;
}

// Dense grid -> bricks: thread per (brick, word); word w covers lz = w/2 and
// ly = 4 (w&1) .. +3, lx = 0..7.
__global__ void dense_bricks_kernel(const uint8_t* __restrict__ occ, int dx, int dy, int dz,
                                    int nbx, int nby, int nbz, uint32_t* __restrict__ bricks) {
  const size_t total = (size_t)nbx * nby * nbz * kBrickWords;
  for (size_t idx = blockIdx.x * (size_t)blockDim.x + threadIdx.x; idx < total;
       idx += (size_t)gridDim.x * blockDim.x) {
    const size_t brick = idx / kBrickWords;
    const int w = (int)(idx % kBrickWords);
    const int bx = (int)(brick % nbx), by = (int)((brick / nbx) % nby), bz = (int)(brick / ((size_t)nbx * nby));
    const int z = bz * 8 + (w >> 1);
    uint32_t word = 0;
    for (int r = 0; r < 4; ++r) {
      const int y = by * 8 + 4 * (w & 1) + r;
      for (int lx = 0; lx < 8; ++lx) {
        const int x = bx * 8 + lx;
        if (x < dx && y < dy && z < dz && occ[(size_t)x + (size_t)dx * ((size_t)y + (size_t)dy * z)] != 0)
          word |= 1u << (lx + 8 * r);
      }
    }
    bricks[idx] = word;
  }
}

// Occupied blocks get consecutive slots in the box field: slot_of[b] (~0 for a free block) and
// its inverse `list`; *count = how many there are.  The order of the slots is arbitrary; no
// result depends on it.  Hash layout: the slot goes to the block's table entry as well.
template <int LAYOUT>
__global__ void block_slots_kernel(const uint4* __restrict__ bricks, uint32_t n_bricks,
                                   const int32_t* __restrict__ keys, DevMap m, HashEntry* table,
                                   uint32_t* __restrict__ slot_of, uint32_t* __restrict__ list,
                                   uint32_t* count) {
  const uint32_t lane = threadIdx.x & 31;
  // warp-uniform trip count; one atomic per warp (same-address atomics are serialised)
  for (uint32_t b0 = blockIdx.x * blockDim.x + (threadIdx.x & ~31u); b0 < n_bricks;
       b0 += gridDim.x * blockDim.x) {
    const uint32_t b = b0 + lane;
    const bool any = b < n_bricks && brick_any(bricks + 4 * (size_t)b);
    const uint32_t mask = __ballot_sync(0xffffffffu, any);
    uint32_t first = 0;
    if (lane == 0 && mask) first = atomicAdd(count, (uint32_t)__popc(mask));
    first = __shfl_sync(0xffffffffu, first, 0);
    const uint32_t slot = any ? first + __popc(mask & ((1u << lane) - 1u)) : ~0u;
    if (any) list[slot] = b;
    if (b >= n_bricks) continue;
    if (LAYOUT == kLayoutGrid) {
      slot_of[b] = slot;
    } else if (any) {
      const unsigned long long key = pack_key(keys[3 * (size_t)b], keys[3 * (size_t)b + 1],
                                              keys[3 * (size_t)b + 2]);
      uint32_t h = (uint32_t)((key * 0x9E3779B97F4A7C15ull) >> m.hash_shift);
      for (uint32_t probe = 0; probe <= m.cap_mask; ++probe) {
        if (table[h].key == key) {
          table[h].box = slot;
          break;
        }
        h = (h + 1) & m.cap_mask;
      }
    }
  }
}

// The free boxes of the march.  One CTA takes the 8^3 cells of one brick (level 0: the voxels
// of an occupied block) or of one super-brick (level 1: 8^3 blocks of the grid) with the 8
// cells around it as 24 x 24 rows of 24 bits, and writes for each cell and octant the box
// [cell, cell + 2^e) (e in 0..3 per axis, in the octant's direction) that a greedy growth
// reaches: the axes take turns (x, y, z) doubling their extent until the doubled box would
// hold an occupied cell.  Cells beyond a map count as free (dense maps clip the boxes).
// Thread (signs of y and z, row of the centre) holds, for each pair of extents (ey, ez), the OR
// of the 2^ey x 2^ez rows ahead, built in two OR passes (z in shared memory, then y) that share
// their doubling prefixes, so that only x is left.  It grows the boxes of its row's 8 cells and
// both signs of x at once, 16 in the bits of a word: round d of turns only meets the extents
// 0 .. d + 1, 63 combinations in all.  Bound by those bit operations: 69 us for the 40 m map's
// 7846 occupied blocks (cell by cell with a shared load and a mask per test 156 us, one
// sign of x at a time 99 us).
// Level 0 stores bytes, 0 for an occupied voxel and 64 | ex | ey <<
// 2 | ez << 4 for a free one, in reflected order (see march_run), 8 octants x 512 per slot.
// Level 1 stores words in 8 octant planes: the same bits for a free block, 2^31 | slot for an
// occupied one.
struct BoxFieldArgs {
  DevMap m;
  const uint32_t* bricks;
  const int32_t* keys;        // hash layout: block keys
  const uint32_t* slot_of;    // grid layout
  const uint32_t* list;
  const uint32_t* count;
  uint32_t cap;               // slots the field has room for
  uint8_t* field;             // null: no level 0 (count > cap)
  uint32_t* top;              // grid layout: level 1
  uint32_t n_super;           // CTAs of level 1, the first ones of the grid
};

template <int LAYOUT>
__global__ void __launch_bounds__(256) box_field_kernel(BoxFieldArgs g) {
  __shared__ uint32_t words[27][16];
  __shared__ uint32_t vol[24][24];          // [z][y], bit x
  __shared__ uint32_t U[2][4][8][24];       // [sign z][ez][centre z][y]
  const DevMap& m = g.m;
  const uint32_t t = threadIdx.x;
  const bool level1 = blockIdx.x < g.n_super;
  const uint32_t n = level1 ? g.n_super : (g.field ? min(*g.count, g.cap) : 0u);
  const uint32_t stride = level1 ? g.n_super : gridDim.x - g.n_super;
  const int sx = (m.gdim[0] + 7) / 8, sy = (m.gdim[1] + 7) / 8;
  for (uint32_t i = level1 ? blockIdx.x : blockIdx.x - g.n_super; i < n; i += stride) {
    int c[3];                                // the centre's coordinates (grid or key)
    uint32_t b = i;
    __syncthreads();                         // the last brick's shared data is no longer read
    if (level1) {
      c[0] = (int)(i % (uint32_t)sx);
      c[1] = (int)(i / (uint32_t)sx % (uint32_t)sy);
      c[2] = (int)(i / ((uint32_t)sx * (uint32_t)sy));
      for (uint32_t row = t; row < 576; row += 256) {
        const int z = 8 * c[2] - 8 + (int)(row / 24), y = 8 * c[1] - 8 + (int)(row % 24);
        uint32_t bits = 0;
        if ((unsigned)z < (unsigned)m.gdim[2] && (unsigned)y < (unsigned)m.gdim[1]) {
          const uint32_t* src = g.slot_of + (size_t)m.gdim[0] * ((size_t)y + (size_t)m.gdim[1] * z);
          for (int x = 0; x < 24; ++x) {
            const int xx = 8 * c[0] - 8 + x;
            if ((unsigned)xx < (unsigned)m.gdim[0] && src[xx] != ~0u) bits |= 1u << x;
          }
        }
        vol[row / 24][row % 24] = bits;
      }
    } else {
      b = g.list[i];
      if (LAYOUT == kLayoutGrid) {
        c[0] = (int)(b % (uint32_t)m.gdim[0]);
        c[1] = (int)(b / (uint32_t)m.gdim[0] % (uint32_t)m.gdim[1]);
        c[2] = (int)(b / ((uint32_t)m.gdim[0] * (uint32_t)m.gdim[1]));
      } else {
        for (int a = 0; a < 3; ++a) c[a] = g.keys[3 * (size_t)b + a];
      }
      for (uint32_t w = t; w < 27 * 16; w += 256) {
        const int nb = (int)(w >> 4);
        const int x = c[0] + nb % 3 - 1, y = c[1] + nb / 3 % 3 - 1, z = c[2] + nb / 9 - 1;
        long long at = -1;
        if (LAYOUT == kLayoutGrid) {
          if ((unsigned)x < (unsigned)m.gdim[0] && (unsigned)y < (unsigned)m.gdim[1] &&
              (unsigned)z < (unsigned)m.gdim[2])
            at = x + (long long)m.gdim[0] * (y + (long long)m.gdim[1] * z);
        } else {
          uint32_t slot;
          at = hash_lookup(m, x, y, z, slot);
        }
        words[nb][w & 15] = at >= 0 ? __ldg(g.bricks + 16 * at + (w & 15)) : 0u;
      }
      __syncthreads();
      for (uint32_t row = t; row < 576; row += 256) {
        const uint32_t z = row / 24, y = row % 24;
        const uint32_t nb = 9 * (z >> 3) + 3 * (y >> 3), w = ((y & 7) >> 2) + 2 * (z & 7),
                       sh = 8 * (y & 3);
        vol[z][y] = ((words[nb][w] >> sh) & 0xffu) | (((words[nb + 1][w] >> sh) & 0xffu) << 8) |
                    (((words[nb + 2][w] >> sh) & 0xffu) << 16);
      }
    }
    __syncthreads();
    for (uint32_t w = t; w < 384; w += 256) {        // OR along z
      const uint32_t y = w % 24, z = w / 24 % 8, s = w / 192;
      uint32_t acc = 0;
#pragma unroll
      for (int d = 0; d < 8; ++d) {
        acc |= vol[s ? 8 + z + d : 8 + z - d][y];
        if (d == 0) U[s][0][z][y] = acc;
        else if (d == 1) U[s][1][z][y] = acc;
        else if (d == 3) U[s][2][z][y] = acc;
        else if (d == 7) U[s][3][z][y] = acc;
      }
    }
    __syncthreads();
    const uint32_t row = t & 63, z = row >> 3, y = row & 7;
    const uint32_t cs = t >> 6, sy_up = cs & 1u, sz_up = cs >> 1;
    const uint32_t yr = sy_up ? y : 7 - y, zr = sz_up ? z : 7 - z;
    // X[ey + 4 ez][ex]: bit i < 8 set if the box from cell i on holds an occupied cell, bit 16 + i
    // the same for reflected cell i, the row read backwards (the shifts carry bits of one half
    // into bits 9-15 of the other, which no cell's box reaches)
    uint32_t X[16][4];
#pragma unroll
    for (int ez = 0; ez < 4; ++ez) {                 // OR along y
      uint32_t acc = 0;
#pragma unroll
      for (int d = 0; d < 8; ++d) {
        acc |= U[sz_up][ez][z][sy_up ? 8 + y + d : 8 + y - d];
        if (d == 0 || d == 1 || d == 3 || d == 7) {
          const int w = 4 * ez + (d == 0 ? 0 : (d == 1 ? 1 : (d == 3 ? 2 : 3)));
          // 24 bits: the row from its cell 0 on; reversed, from reflected cell 0 on
          X[w][0] = ((acc >> 8) & 0xffffu) | (__brev(acc) & 0xffff0000u);
          X[w][1] = X[w][0] | X[w][0] >> 1;
          X[w][2] = X[w][1] | X[w][1] >> 2;
          X[w][3] = X[w][2] | X[w][2] >> 4;
        }
      }
    }
    // the cells whose extents are 2^0 .. 2^3 so far, per axis, and those still growing
    const uint32_t open = 0x00ff00ffu & ~X[0][0];
    uint32_t E[3][4], G[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      E[a][0] = 0x00ff00ffu;
      E[a][1] = E[a][2] = E[a][3] = 0u;
      G[a] = open;
    }
#pragma unroll
    for (int d = 0; d < 3; ++d)
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        uint32_t blocked = 0;   // the box with axis a doubled holds an occupied cell
        const int p = a == 0 ? 1 : 0, q = a == 2 ? 1 : 2;      // the other two axes
#pragma unroll
        for (int ep = 0; ep < 4; ++ep)
#pragma unroll
          for (int eq = 0; eq < 4; ++eq) {
            if (ep > (p < a ? d + 1 : d) || eq > (q < a ? d + 1 : d)) continue;
            const int ex = a == 0 ? d + 1 : ep, ey = a == 1 ? d + 1 : (a == 0 ? ep : eq),
                      ez = a == 2 ? d + 1 : eq;
            blocked |= X[ey + 4 * ez][ex] & E[p][ep] & E[q][eq];
          }
        G[a] &= ~blocked;
        E[a][d] &= ~G[a];
        E[a][d + 1] = G[a];
      }
#pragma unroll
    for (uint32_t sx_up = 0; sx_up < 2; ++sx_up) {
      const uint32_t oct = sx_up | (sy_up << 1) | (sz_up << 2);
      // bits -> bytes: cell i's bit of each of the 7 code bits to byte i
      uint32_t lo = 0, hi = 0;
#pragma unroll
      for (int j = 0; j < 7; ++j) {
        const uint32_t both = j == 6 ? open : open & (j & 1 ? E[j >> 1][2] | E[j >> 1][3]
                                                            : E[j >> 1][1] | E[j >> 1][3]);
        const uint32_t bits = sx_up ? both & 0xffu : both >> 16;
        lo |= (((bits & 15u) * 0x00204081u) & 0x01010101u) << j;
        hi |= (((bits >> 4) * 0x00204081u) & 0x01010101u) << j;
      }
      if (!level1) {
        *reinterpret_cast<uint2*>(g.field + 4096 * (size_t)i + 512 * oct + 64 * zr + 8 * yr) =
            make_uint2(lo, hi);
        continue;
      }
      const int by = 8 * c[1] + (int)y, bz = 8 * c[2] + (int)z;
      const size_t nb = (size_t)m.gdim[0] * m.gdim[1] * m.gdim[2];
      if (by >= m.gdim[1] || bz >= m.gdim[2]) continue;
      for (int xr = 0; xr < 8; ++xr) {
        const int bx = 8 * c[0] + (sx_up ? xr : 7 - xr);
        if (bx >= m.gdim[0]) continue;
        const uint32_t code = ((xr < 4 ? lo : hi) >> (8 * (xr & 3))) & 0xffu;
        const size_t at = (size_t)bx + (size_t)m.gdim[0] * ((size_t)by + (size_t)m.gdim[1] * bz);
        g.top[oct * nb + at] = code ? (code & 63u) : (0x80000000u | g.slot_of[at]);
      }
    }
  }
}

// Free distance of each 2^3 cell of the occupied bricks: the Chebyshev distance in voxels
// from the cell to the nearest occupied voxel, capped at kCellDistCap (a free cell at
// distance dv holds no voxel closer than dv to an obstacle, so every voxel of it centres a
// free box of half-width dv - 1).  One CTA per brick: the 3^3 bricks around it are loaded
// into shared memory as a 24^3 bit volume (rows of 24 x-bits), dilated by one voxel in the
// Chebyshev metric kCellDistCap - 1 times (the 3^3 maximum, one pass per dilation); a cell's
// distance is the first dilation that reaches one of its 8 voxels.  Only voxels within
// kCellDistCap - 1 of the centre brick matter, and they lie inside the volume.  Free bricks
// get 0 (never read).
static_assert(kCellDistCap == 4, "the halo of one brick covers dilations up to 3 voxels");
__global__ void __launch_bounds__(256) cell_dist_kernel(const uint32_t* __restrict__ bricks,
                                                        DevMap m, uint64_t n_bricks,
                                                        uint32_t* __restrict__ cells) {
  __shared__ uint32_t vol[2][24][24];   // [z][y], bit x
  __shared__ uint32_t words[8];
  __shared__ int occupied;
  const int t = threadIdx.x;
  const int gx = m.gdim[0], gy = m.gdim[1], gz = m.gdim[2];
  for (uint64_t b = blockIdx.x; b < n_bricks; b += gridDim.x) {
    __syncthreads();                    // the previous brick's shared data is no longer read
    if (t == 0) occupied = 0;
    if (t < 8) words[t] = 0;
    __syncthreads();
    if (t < 16 && __ldg(bricks + 16 * b + t) != 0u) occupied = 1;
    __syncthreads();
    if (!occupied) {
      if (t < 8) cells[8 * b + t] = 0u;
      continue;
    }
    const int bx = (int)(b % (uint64_t)gx);
    const int by = (int)((b / (uint64_t)gx) % (uint64_t)gy);
    const int bz = (int)(b / ((uint64_t)gx * (uint64_t)gy));
    for (int r = t; r < 576; r += blockDim.x) {
      const int zz = r / 24, yy = r - 24 * (r / 24);
      const int nz = bz + zz / 8 - 1, ny = by + yy / 8 - 1;
      const int lz = zz & 7, ly = yy & 7;
      uint32_t row = 0u;
      if ((unsigned)nz < (unsigned)gz && (unsigned)ny < (unsigned)gy) {
#pragma unroll
        for (int dx = 0; dx < 3; ++dx) {
          const int nx = bx + dx - 1;
          if ((unsigned)nx >= (unsigned)gx) continue;
          const size_t nb = (size_t)nx + (size_t)gx * ((size_t)ny + (size_t)gy * (size_t)nz);
          const uint32_t w = __ldg(bricks + 16 * nb + (ly >> 2) + 2 * lz);
          row |= ((w >> (8 * (ly & 3))) & 0xffu) << (8 * dx);
        }
      }
      vol[0][zz][yy] = row;
    }
    __syncthreads();
    // thread c < 64: cell c of the centre brick (voxels 8 + 2 (c & 3) .. +1 in x, etc.)
    const int cx = 8 + 2 * (t & 3), cy = 8 + 2 * ((t >> 2) & 3), cz = 8 + 2 * ((t >> 4) & 3);
    const uint32_t cmask = 3u << cx;
    int d = kCellDistCap;
    auto touches = [&](int buf) {
      return ((vol[buf][cz][cy] | vol[buf][cz][cy + 1] | vol[buf][cz + 1][cy] |
               vol[buf][cz + 1][cy + 1]) & cmask) != 0u;
    };
    if (t < 64 && touches(0)) d = 0;
    for (int k = 1; k < kCellDistCap; ++k) {
      const int src = (k - 1) & 1, dst = k & 1;
      for (int r = t; r < 576; r += blockDim.x) {
        const int zz = r / 24, yy = r - 24 * (r / 24);
        uint32_t acc = 0u;
#pragma unroll
        for (int dz = -1; dz <= 1; ++dz) {
#pragma unroll
          for (int dy = -1; dy <= 1; ++dy) {
            const int z2 = zz + dz, y2 = yy + dy;
            if ((unsigned)z2 < 24u && (unsigned)y2 < 24u) acc |= vol[src][z2][y2];
          }
        }
        vol[dst][zz][yy] = (acc | (acc << 1) | (acc >> 1)) & 0xffffffu;
      }
      __syncthreads();
      // the next dilation writes vol[src], whose reads ended at the barrier above, and only
      // reads vol[dst]: no second barrier is needed
      if (t < 64 && d == kCellDistCap && touches(dst)) d = k;
    }
    if (t < 64) atomicOr(&words[t >> 3], (uint32_t)d << (4 * (t & 7)));
    __syncthreads();
    if (t < 8) cells[8 * b + t] = words[t];
  }
}

// What the host asks of a hashed map's blocks before it lays the map out: info[0] |= 1 a key
// out of range, 2 a duplicate key, 4 a full table (hash_build_kernel), info[1] = blocks with an
// occupied voxel, info[2 + a] / info[5 + a] = the largest -key / key of such a block on axis a.
// Reduced over the warp and the CTA first: atomics of all threads on the same words are
// serialised (the 40 m map, 7846 occupied blocks: 4.3 us, now 3.6 us).
__global__ void __launch_bounds__(256) key_bbox_kernel(const int32_t* __restrict__ keys,
                                                       const uint4* __restrict__ bricks,
                                                       uint32_t n_blocks, int* info) {
  __shared__ int best[6];
  __shared__ unsigned total;
  const uint32_t lane = threadIdx.x & 31;
  if (threadIdx.x < 6) best[threadIdx.x] = INT_MIN;
  if (threadIdx.x == 0) total = 0;
  __syncthreads();
  int v[6] = {INT_MIN, INT_MIN, INT_MIN, INT_MIN, INT_MIN, INT_MIN};
  unsigned count = 0;
  for (uint32_t b = blockIdx.x * blockDim.x + threadIdx.x; b < n_blocks;
       b += gridDim.x * blockDim.x) {
    if (!brick_any(bricks + 4 * (size_t)b)) continue;
    count += 1;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const int k = keys[3 * (size_t)b + a];
      v[a] = max(v[a], -k);
      v[3 + a] = max(v[3 + a], k);
    }
  }
  count = __reduce_add_sync(0xffffffffu, count);
#pragma unroll
  for (int a = 0; a < 6; ++a) v[a] = __reduce_max_sync(0xffffffffu, v[a]);
  if (lane == 0 && count > 0) {
#pragma unroll
    for (int a = 0; a < 6; ++a) atomicMax(best + a, v[a]);
    atomicAdd(&total, count);
  }
  __syncthreads();
  if (threadIdx.x < 6 && total > 0) atomicMax(info + 2 + threadIdx.x, best[threadIdx.x]);
  if (threadIdx.x == 6 && total > 0) atomicAdd(reinterpret_cast<unsigned*>(info) + 1, total);
}

// Scatter the non-empty bricks of a hashed map into the grid layout.
__global__ void grid_scatter_kernel(const int32_t* __restrict__ keys, const uint4* __restrict__ bricks,
                                    uint32_t n_blocks, DevMap m, uint4* __restrict__ grid) {
  const int gx = m.gmin[0], gy = m.gmin[1], gz = m.gmin[2], dx = m.gdim[0], dy = m.gdim[1];
  for (uint32_t b = blockIdx.x * blockDim.x + threadIdx.x; b < n_blocks;
       b += gridDim.x * blockDim.x) {
    const uint4* w = bricks + 4 * (size_t)b;
    const uint4 w0 = w[0], w1 = w[1], w2 = w[2], w3 = w[3];
    const uint32_t any = w0.x | w0.y | w0.z | w0.w | w1.x | w1.y | w1.z | w1.w | w2.x | w2.y |
                         w2.z | w2.w | w3.x | w3.y | w3.z | w3.w;
    if (!any) continue;
    const int x = keys[3 * (size_t)b] - gx, y = keys[3 * (size_t)b + 1] - gy,
              z = keys[3 * (size_t)b + 2] - gz;
    const uint32_t idx = (uint32_t)x + (uint32_t)dx * ((uint32_t)y + (uint32_t)dy * (uint32_t)z);
    uint4* dst = grid + 4 * (size_t)idx;
    dst[0] = w0;
    dst[1] = w1;
    dst[2] = w2;
    dst[3] = w3;
  }
}

// TSDF blocks -> bricks: bit b of block n is tsdf[n*512 + b] <= 0 (the TSDF voxel order
// lx + 8 ly + 64 lz is the brick's bit order).  Bound by reading the TSDF once: a warp reads
// 32 consecutive voxels per load, a ballot makes them a word, 4 loads in flight (one thread
// per word, each with its own line: 23.6 us for the 40 m map's 23 MB, now 7.9 us).
__global__ void __launch_bounds__(256) tsdf_bricks_kernel(const float* __restrict__ tsdf,
                                                          uint32_t n_blocks,
                                                          uint32_t* __restrict__ bricks) {
  const uint32_t lane = threadIdx.x & 31;
  const uint32_t n_warps = gridDim.x * (blockDim.x >> 5);
  for (uint32_t b = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); b < n_blocks; b += n_warps) {
    const float* t = tsdf + 512 * (size_t)b + lane;
    uint32_t word = 0;
#pragma unroll
    for (int i = 0; i < 16; i += 4) {
      const float v0 = __ldg(t + 32 * i), v1 = __ldg(t + 32 * i + 32),
                  v2 = __ldg(t + 32 * i + 64), v3 = __ldg(t + 32 * i + 96);
      const uint32_t w0 = __ballot_sync(0xffffffffu, v0 <= 0.0f),
                     w1 = __ballot_sync(0xffffffffu, v1 <= 0.0f),
                     w2 = __ballot_sync(0xffffffffu, v2 <= 0.0f),
                     w3 = __ballot_sync(0xffffffffu, v3 <= 0.0f);
      word = lane == (uint32_t)i ? w0 : (lane == (uint32_t)i + 1 ? w1 : (lane == (uint32_t)i + 2 ? w2
             : (lane == (uint32_t)i + 3 ? w3 : word)));
    }
    if (lane < kBrickWords) bricks[kBrickWords * (size_t)b + lane] = word;
  }
}

// Insert block keys into the open-addressing table (linear probing, bounded).
// err bits: 1 key out of range, 2 duplicate key, 4 table full.
__global__ void hash_build_kernel(const int32_t* __restrict__ keys, uint32_t n_blocks,
                                  const uint4* __restrict__ bricks, HashEntry* table,
                                  uint32_t cap_mask, int hash_shift, unsigned int* err) {
  for (uint32_t b = blockIdx.x * blockDim.x + threadIdx.x; b < n_blocks;
       b += gridDim.x * blockDim.x) {
    const int bx = keys[3 * (size_t)b], by = keys[3 * (size_t)b + 1], bz = keys[3 * (size_t)b + 2];
    if (bx < -kKeyBias || bx >= kKeyBias || by < -kKeyBias || by >= kKeyBias ||
        bz < -kKeyBias || bz >= kKeyBias) {
      atomicOr(err, 1u);
      continue;
    }
    const unsigned long long key = (unsigned long long)(uint32_t)(bx + kKeyBias) |
                                   ((unsigned long long)(uint32_t)(by + kKeyBias) << 21) |
                                   ((unsigned long long)(uint32_t)(bz + kKeyBias) << 42);
    uint32_t h = (uint32_t)((key * 0x9E3779B97F4A7C15ull) >> hash_shift);
    bool done = false;
    for (uint32_t probe = 0; probe <= cap_mask; ++probe) {
      const unsigned long long prev = atomicCAS(&table[h].key, kEmptyKey, key);
      if (prev == kEmptyKey) {
        // all-free bricks read as missing
        table[h].slot = brick_any(bricks + 4 * (size_t)b) ? b : 0xFFFFFFFFu;
        done = true;
        break;
      }
      if (prev == key) {
        atomicOr(err, 2u);
        done = true;
        break;
      }
      h = (h + 1) & cap_mask;
    }
    if (!done) atomicOr(err, 4u);
  }
}

}  // namespace

// ------------------------------------------------------------------ launchers
// A launch with programmatic serialisation (see wait_previous, which every kernel launched like
// this calls).
template <class... P, class... A>
static cudaError_t launch_after_shared(void (*kernel)(P...), unsigned grid, unsigned block,
                                       size_t shared, cudaStream_t stream, A... args) {
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t c = {};
  c.gridDim = dim3(grid);
  c.blockDim = dim3(block);
  c.dynamicSmemBytes = shared;
  c.stream = stream;
  c.attrs = &attr;
  c.numAttrs = 1;
  return cudaLaunchKernelEx(&c, kernel, P(args)...);
}
template <class... P, class... A>
static cudaError_t launch_after(void (*kernel)(P...), unsigned grid, unsigned block,
                                cudaStream_t stream, A... args) {
  return launch_after_shared(kernel, grid, block, 0, stream, args...);
}

// Every kernel variant of a map and reduction: f is called with <kind, layout, reduction, box
// field present> as integral constants.
template <int V>
using Int = std::integral_constant<int, V>;

template <int KIND, int LAYOUT, class F>
static void for_reduction(const DevMap& m, int reduce_mode, F f) {
  if (reduce_mode == RMP_REDUCE_FP64) {
    if (m.cells) f(Int<KIND>(), Int<LAYOUT>(), Int<RMP_REDUCE_FP64>(), Int<1>());
    else f(Int<KIND>(), Int<LAYOUT>(), Int<RMP_REDUCE_FP64>(), Int<0>());
  } else {
    if (m.cells) f(Int<KIND>(), Int<LAYOUT>(), Int<RMP_REDUCE_KAHAN32>(), Int<1>());
    else f(Int<KIND>(), Int<LAYOUT>(), Int<RMP_REDUCE_KAHAN32>(), Int<0>());
  }
}

template <class F>
static void for_map(const DevMap& m, int reduce_mode, F f) {
  if (m.kind == RMP_MAP_DENSE_U8) for_reduction<RMP_MAP_DENSE_U8, kLayoutGrid>(m, reduce_mode, f);
  else if (m.layout == kLayoutGrid) for_reduction<RMP_MAP_HASHED_TSDF, kLayoutGrid>(m, reduce_mode, f);
  else for_reduction<RMP_MAP_HASHED_TSDF, kLayoutHash>(m, reduce_mode, f);
}

// CTAs per SM of the variant that launch_raycast runs at this CTA size.
int raycast_occupancy(const DevMap& m, int reduce_mode, int block) {
  int n = 0;
  cudaError_t e = cudaSuccess;
  for_map(m, reduce_mode, [&](auto kind, auto layout, auto red, auto boxes) {
    if (block == 256)
      e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(
          &n, raycast_rmp_kernel<kind.value, layout.value, red.value, boxes.value != 0, 256, 2>, block, 0);
    else
      e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(
          &n, raycast_rmp_kernel<kind.value, layout.value, red.value, boxes.value != 0, 128, 6>, block, 0);
  });
  return e == cudaSuccess ? n : -1;
}

cudaError_t launch_raycast(const DevMap& m, const EvalConsts& k, const double* state_dev,
                           void* ws, rmp_result_t* out_dev, rmp_ray_hit_t* hits,
                           float* per_ray, int block, int grid, cudaStream_t stream) {
  // grid_finish needs whole warps 0 and 1 (the resolve's named barrier)
  if (block != 64 && block != 128 && block != 256) return cudaErrorInvalidValue;
  WsHeader* hdr = (WsHeader*)ws;
  CtaPartial* parts = (CtaPartial*)((char*)ws + kWsHeaderBytes);
  for_map(m, k.reduce_mode, [&](auto kind, auto layout, auto red, auto boxes) {
    if (block == 256)
      launch_after(raycast_rmp_kernel<kind.value, layout.value, red.value, boxes.value != 0, 256, 2>,
                   grid, block, stream, m, k, state_dev, hdr, parts, out_dev, hits, per_ray);
    else
      launch_after(raycast_rmp_kernel<kind.value, layout.value, red.value, boxes.value != 0, 128, 6>,
                   grid, block, stream, m, k, state_dev, hdr, parts, out_dev, hits, per_ray);
  });
  return cudaGetLastError();
}

int batch_occupancy(const DevMap& m, int reduce_mode, int block) {
  int n = 0;
  cudaError_t e = cudaSuccess;
  for_map(m, reduce_mode, [&](auto kind, auto layout, auto red, auto boxes) {
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(
        &n, raycast_batch_kernel<kind.value, layout.value, red.value, boxes.value != 0>, block, 0);
  });
  return e == cudaSuccess ? n : -1;
}

cudaError_t launch_batch(const DevMap& m, const EvalConsts& k, const double* states_dev,
                         const uint32_t* n_rays_dev, uint32_t n_states, uint32_t max_rays,
                         void* ws, rmp_result_t* out_dev, rmp_ray_hit_t* hits, float* per_ray,
                         int block, int grid, cudaStream_t stream, const double* goals_dev,
                         const RolloutArgs& step) {
  const uint32_t sms = k.sms;
  if (!step.rs && state_per_cta(n_states, max_rays, sms)) {
    // warps a CTA: all of an SM's 32 for one state, fewer where CTAs share it and hide each
    // other's serial steps; segments only while every state has its place (5000 states of 64 rays:
    // 4 segments 149 us, 1 86), one warp left for the attractor (128 of 256 rays 19.9 -> 17.8)
    const uint32_t most = n_states <= sms ? 32u : (n_states <= 2 * sms ? 16u : 8u);
    const uint32_t lg = state_lg_segs(k, max_rays), parts = ((max_rays << 2) + 31) / 32;
    const uint32_t hold = n_states <= 2 * sms ? most - (goals_dev ? 1u : 0u) : 1u;
    const uint32_t chunks = ((max_rays << cta_lg_segs(k, max_rays, lg, hold)) + 31) / 32;
    const uint32_t warps = std::min(std::max(chunks + (goals_dev ? 1u : 0u), 2u), most);
    for_map(m, k.reduce_mode, [&](auto kind, auto layout, auto red, auto boxes) {
      launch_after_shared(
          raycast_state_kernel<kind.value, layout.value, red.value, boxes.value != 0>, n_states,
          32 * warps, 4 * kPartWords * parts, stream, m, k, states_dev, n_rays_dev, max_rays,
          out_dev, hits, per_ray, goals_dev, hold);
    });
    return cudaGetLastError();
  }
  const BatchLayout L = batch_layout(n_states, max_rays);
  char* w = (char*)ws;
  BatchHeader* hdr = (BatchHeader*)w;
  BatchState* bs = (BatchState*)(w + L.states);
  uint32_t* sticket = (uint32_t*)(w + L.sticket);
  uint32_t* gticket = (uint32_t*)(w + L.gticket);
  CtaPartial* cparts = (CtaPartial*)(w + L.cparts);
  CtaPartial* gparts = (CtaPartial*)(w + L.gparts);
  // 8 states a CTA (a warp each) as far as the SMs go; longer runs beyond
  const unsigned prep = n_states < 8u * sms ? (n_states + 7u) / 8u : sms;
  launch_after(batch_prep_kernel, prep, 256, stream, states_dev, n_rays_dev, n_states, max_rays, m,
               k, hdr, bs, sticket, gticket, out_dev);
  for_map(m, k.reduce_mode, [&](auto kind, auto layout, auto red, auto boxes) {
    launch_after(raycast_batch_kernel<kind.value, layout.value, red.value, boxes.value != 0>, grid,
                 block, stream, m, k, hdr, bs, sticket, gticket, cparts, gparts, out_dev, hits,
                 per_ray, max_rays, states_dev, goals_dev, step);
  });
  return cudaGetLastError();
}

// Shared memory of a resident rollout: directions and partials.
static size_t rollout_shared(uint32_t rays, uint32_t parts) {
  return 4 * (size_t)(((6 * rays + 3) & ~3u) + kPartWords * parts);
}

cudaError_t launch_rollout(const DevMap& m, const EvalConsts& k, const RolloutArgs& g, uint32_t n,
                           uint32_t steps, cudaStream_t stream) {
  // at most 32 warps a CTA; 16 where two robots share an SM and hide each other's serial steps
  const uint32_t rays = g.rc.n_rays, most = n <= k.sms ? 32u : 16u;
  const uint32_t lg = state_lg_segs(k, rays), parts = ((rays << lg) + 31) / 32;
  // two warps left for the attractor and the booking where the chunks allow (8 robots of 256 rays:
  // 4 segments, both on marching warps 18.3 us a step, 2 segments 15.8)
  const uint32_t lgs = cta_lg_segs(k, rays, lg, most - 2);
  const uint32_t groups = (parts + kBatchGroup - 1) / kBatchGroup;
  const uint32_t warps = std::min(std::max(((rays << lgs) + 31) / 32 + 2, groups), most);   // >= 3
  const size_t dyn = rollout_shared(rays, parts);
  // the limit belongs to the kernel, whichever thread or context launches it: every call sets the
  // same one, the most that any may want, so that none lowers it under another's launch
  const int limit = (int)rollout_shared(kStateRays, kStateGroups * kBatchGroup);
  cudaError_t e = cudaSuccess;
  for_map(m, k.reduce_mode, [&](auto kind, auto layout, auto red, auto boxes) {
    const auto f = rollout_kernel<kind.value, layout.value, red.value, boxes.value != 0>;
    e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, limit);
    if (e == cudaSuccess) f<<<n, 32 * warps, dyn, stream>>>(m, k, g, rays, lg, lgs, steps);
  });
  return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t launch_probe_l2(const uint4* buf, size_t n16, uint32_t passes, int grid,
                            uint64_t* checksum, cudaStream_t stream) {
  probe_l2_kernel<<<grid, 512, 0, stream>>>(buf, n16, passes, checksum);
  return cudaGetLastError();
}

// As few states a CTA as give one CTA an SM: few states wait for latency; beyond, 32, where the
// FP64 steps fill their lanes (152 SMs, 1217 states: 8 a CTA 20.1 us, 16 18.0, 32 20.5; 2432 states:
// 22.3, 18.2, 20.5).
static uint32_t esdf_states_per_cta(uint32_t n, uint32_t sms) {
  return n <= 8u * sms ? 8u : (n <= 16u * sms ? 16u : 32u);
}

cudaError_t launch_esdf_eval(const rmp_primitive_t* prims, const float4* prims32,
                             uint32_t n_prims, const EsdfConsts& k, const double* states,
                             const double* goals, uint32_t n_states, rmp_result_t* out,
                             double* query, cudaStream_t stream) {
  if (n_states == 0) return cudaSuccess;
  const uint32_t G = esdf_states_per_cta(n_states, k.sms);
  uint32_t grid = (n_states + G - 1) / G;
  if (grid > 65535) grid = 65535;                   // CTA-stride beyond
  launch_after(esdf_eval_kernel<false, 0, 0>, grid, 256, stream, prims, prims32, n_prims, k, states,
               goals, n_states, G, out, query, DevMap(), RolloutArgs(), 0u, (uint32_t*)nullptr);
  return cudaGetLastError();
}

cudaError_t launch_esdf_rollout(const rmp_primitive_t* prims, const float4* prims32,
                                uint32_t n_prims, const EsdfConsts& k, const DevMap& m,
                                const RolloutArgs& g, uint32_t n, uint32_t steps,
                                rmp_result_t* res, uint32_t* running, cudaStream_t stream) {
  const uint32_t G = esdf_states_per_cta(n, k.sms), grid = (n + G - 1) / G;
  const double* none = nullptr;
  double* query = nullptr;
  auto run = [&](auto kernel) {
    launch_after(kernel, grid, 256, stream, prims, prims32, n_prims, k, none, none, n, G, res, query,
                 m, g, steps, running);
  };
  if (m.kind == RMP_MAP_DENSE_U8) run(esdf_eval_kernel<true, RMP_MAP_DENSE_U8, kLayoutGrid>);
  else if (m.layout == kLayoutGrid) run(esdf_eval_kernel<true, RMP_MAP_HASHED_TSDF, kLayoutGrid>);
  else run(esdf_eval_kernel<true, RMP_MAP_HASHED_TSDF, kLayoutHash>);
  return cudaGetLastError();
}

cudaError_t launch_scan(const float* pts, const EvalConsts& k, const double* state_dev,
                        void* ws, rmp_result_t* out_dev, float* per_ray, int block, int grid,
                        cudaStream_t stream) {
  if (block != 64 && block != 128 && block != 256) return cudaErrorInvalidValue;  // as above
  WsHeader* hdr = (WsHeader*)ws;
  CtaPartial* parts = (CtaPartial*)((char*)ws + kWsHeaderBytes);
  if (k.reduce_mode == RMP_REDUCE_FP64)
    launch_after(scan_rmp_kernel<RMP_REDUCE_FP64>, grid, block, stream, pts, k, state_dev, hdr, parts,
                                                                 out_dev, per_ray);
  else
    launch_after(scan_rmp_kernel<RMP_REDUCE_KAHAN32>, grid, block, stream, pts, k, state_dev, hdr, parts,
                                                                    out_dev, per_ray);
  return cudaGetLastError();
}

cudaError_t launch_dense_bricks(const uint8_t* occ, const int dims[3], const int nb[3],
                                uint32_t* bricks, cudaStream_t stream) {
  const size_t total = (size_t)nb[0] * nb[1] * nb[2] * kBrickWords;
  const int grid = (int)((total + 255) / 256 < 65535 ? (total + 255) / 256 : 65535);
  dense_bricks_kernel<<<grid, 256, 0, stream>>>(occ, dims[0], dims[1], dims[2], nb[0], nb[1],
                                                nb[2], bricks);
  return cudaGetLastError();
}

static int grid_for(size_t n) { return (int)((n + 255) / 256 < 65535 ? ((n + 255) / 256 > 0 ? (n + 255) / 256 : 1) : 65535); }

cudaError_t launch_block_slots(const uint32_t* bricks, uint32_t n, const int32_t* keys,
                               const DevMap& m, HashEntry* table, uint32_t* slot_of,
                               uint32_t* list, uint32_t* count, cudaStream_t stream) {
  if (m.layout == kLayoutGrid)
    block_slots_kernel<kLayoutGrid><<<grid_for(n), 256, 0, stream>>>(
        (const uint4*)bricks, n, keys, m, table, slot_of, list, count);
  else
    block_slots_kernel<kLayoutHash><<<grid_for(n), 256, 0, stream>>>(
        (const uint4*)bricks, n, keys, m, table, slot_of, list, count);
  return cudaGetLastError();
}

cudaError_t launch_box_field(const DevMap& m, const uint32_t* bricks, const int32_t* keys,
                             const uint32_t* slot_of, const uint32_t* list, const uint32_t* count,
                             uint32_t cap, uint8_t* field, uint32_t* top, int sm_count,
                             cudaStream_t stream) {
  BoxFieldArgs g;
  g.m = m;
  g.bricks = bricks;
  g.keys = keys;
  g.slot_of = slot_of;
  g.list = list;
  g.count = count;
  g.cap = cap;
  g.field = field;
  g.top = top;
  g.n_super = 0;
  if (m.layout == kLayoutGrid)
    g.n_super = (uint32_t)((m.gdim[0] + 7) / 8) * (uint32_t)((m.gdim[1] + 7) / 8) *
                (uint32_t)((m.gdim[2] + 7) / 8);
  // level 0 strides over the occupied blocks (their number is on the device)
  const uint32_t wave = (uint32_t)sm_count * 8u;
  const uint32_t grid = g.n_super + (field ? (cap < wave ? (cap > 0 ? cap : 1u) : wave) : 0u);
  if (grid == 0) return cudaSuccess;
  if (m.layout == kLayoutGrid) box_field_kernel<kLayoutGrid><<<grid, 256, 0, stream>>>(g);
  else box_field_kernel<kLayoutHash><<<grid, 256, 0, stream>>>(g);
  return cudaGetLastError();
}

cudaError_t launch_cell_dist(const uint32_t* bricks, const DevMap& m, uint32_t* cells,
                             cudaStream_t stream) {
  const uint64_t n = (uint64_t)m.gdim[0] * m.gdim[1] * m.gdim[2];
  const uint64_t g = n < 65536u ? n : 65536u;          // grid-stride beyond
  cell_dist_kernel<<<(unsigned)(g > 0 ? g : 1), 256, 0, stream>>>(bricks, m, n, cells);
  return cudaGetLastError();
}

cudaError_t launch_key_bbox(const int32_t* keys, const uint32_t* bricks, uint32_t n_blocks,
                            int* info, cudaStream_t stream) {
  key_bbox_kernel<<<grid_for(n_blocks), 256, 0, stream>>>(keys, (const uint4*)bricks, n_blocks, info);
  return cudaGetLastError();
}

cudaError_t launch_grid_scatter(const int32_t* keys, const uint32_t* bricks, uint32_t n_blocks,
                                const DevMap& m, uint32_t* grid_bricks, cudaStream_t stream) {
  grid_scatter_kernel<<<grid_for(n_blocks), 256, 0, stream>>>(keys, (const uint4*)bricks, n_blocks,
                                                              m, (uint4*)grid_bricks);
  return cudaGetLastError();
}

cudaError_t launch_tsdf_bricks(const float* tsdf, uint32_t n_blocks, uint32_t* bricks,
                               cudaStream_t stream) {
  tsdf_bricks_kernel<<<grid_for(32 * (size_t)n_blocks), 256, 0, stream>>>(tsdf, n_blocks, bricks);
  return cudaGetLastError();
}

cudaError_t launch_hash_build(const int32_t* keys, uint32_t n_blocks, const uint32_t* bricks,
                              HashEntry* table, uint32_t cap_mask, int hash_shift,
                              unsigned int* err, cudaStream_t stream) {
  const int grid = (int)((n_blocks + 255) / 256 < 65535 ? (n_blocks + 255) / 256 : 65535);
  hash_build_kernel<<<grid > 0 ? grid : 1, 256, 0, stream>>>(keys, n_blocks, (const uint4*)bricks,
                                                             table, cap_mask, hash_shift, err);
  return cudaGetLastError();
}

}  // namespace rmp
