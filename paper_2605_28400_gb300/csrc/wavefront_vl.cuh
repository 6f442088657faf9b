// wavefront_vl.cuh — wavefront kernel with two cells of one triplet per register ("virtual
// lanes"), for scoring schemes whose sigma'' are all >= 0: scores of every alignment type, and the
// global type with traceback codes.
//
// wavefront_vl_kernel<NJ, NH>: the column-task engine of wavefront.cuh (same queue, progress flags
// and bounded waits; Eq. 1 in the shifted frame of engine.h), with each lane's NJ x 2NH tile held
// as NJ x NH registers of two 16-bit halves:
//  * Layout. The low half holds the left NH columns of the tile at slice s = t - r - 2*lc, the
//    high half the right NH columns one slice behind (s - 1). The 4 x 8 lanes thus act as 4 x 16
//    virtual lanes of NJ x NH tiles on the usual anti-diagonal skew, and every halo comes from a
//    step already finished: rows and the corner by the same packed shuffles as a plain tile, the
//    high half's left column from the low half's previous right column (one PRMT per row).
//  * Arithmetic. Each half holds M' - B + bias with -infinity near 0 (engine.h's biased form):
//    plain 32-bit adds are the two 16-bit adds, issued as multiply-adds by a runtime 1 on the FMA
//    pipe, and the maxima are unsigned 16x2 DPX operations on the ALU pipe.
//  * Range. With every sigma'' >= 0, M' is non-decreasing along each axis and adjacent cells differ
//    by at most 2*max sigma'' (follow the optimal path to the farther cell back to where it enters
//    the farther plane and copy its in-plane moves one plane lower: in-plane costs do not depend
//    on the third coordinate). From lane 0's first cell, a warp's working set reaches 22 axis steps
//    down (19 slices and the halos) and 4 NJ + 16 NH - 2 up (the block). Each warp keeps one base B
//    for its task, warp-uniform, so shuffled halos need no conversion. B starts at the larger of
//    lane 0's upper and left neighbours at slice 0 and rises with lane 0's first cell whenever that
//    is 2048 above the bias (checked every two steps). Score: bias 2^14, -infinity 0, max sigma''
//    <= 33, so every half stays in [14932, 29200) (NH = 8). The host admits the mode only then.
//  * Records by step, raw. What block (J+1, K) needs at its step u is what lanes (3, lc) of block
//    (J, K) hold at its step u + 3, half for half, and block (J, K+1) needs what lanes (r, 7) hold at
//    step u + 15. So a record row is the packed words of one producer step and the producer's base
//    (8 x (NH + 2) and 4 x 6 words), stored as they are; the consumer adds the difference of the two
//    bases, one add per two cells. (Absolute int32 records by slice cost ~30 conversions a step on
//    each side and 100 words instead of 72 for NH = 4.) The only -infinity among the stored halves
//    that is ever read is the corner on the k = 0 face, which its reader sets by itself; a lane
//    outside its slices reads nothing and gets -infinity.
//  * A step's work besides the cells is what bounds a lone warp (2 cycles per ALU instruction),
//    so it is kept short: the steps in which every lane is inside the cube run a copy without any
//    range check; residues, profile values and pieces are fetched one to three steps ahead, so no
//    load latency is left inside a step; loads and selects write plain registers (a predicated load
//    over a shuffled value, or a default value per load, costs a move each: 60 of 550 instructions).
//  * Edges of a task's sweep: the high half of a lane is inactive while the low half computes
//    slice 0 (it is reset to -infinity afterwards); the low half's extra slice a + 1 at the end is
//    computed on virtual residues and never counted.
#pragma once
#include "wavefront.cuh"

namespace trioseq {

constexpr int kVlBias = 1 << 14;
// Traceback keys (TB): a half holds 8*(M' - B) + 3 + kVlTbBias. With S = 8*max sigma'' the halves
// lie in [kVlTbBias - 44S, kVlTbBias + 2048 + 4S + 188S] (NJ = 8, NH = 4), above what an add to
// -infinity reaches (8 + 3S + 7); with max sigma'' <= 30 that is [1216, 59904].
constexpr int kVlTbBias = 11776;  // a multiple of 8

constexpr int kVlRing = 64;  // slices in the residue ring

template <int NJ, int NH>
struct VlGeom {
  static constexpr int NK = 2 * NH;                  // cell columns per lane
  static constexpr int WJ = kPR * NJ, WK = kPC * NK;
  static constexpr int RJ = vl_rec_j(NH), RK = kVlRecK;  // record row strides (ints)
  // ring slot: row words [lane column][NH], corners [lane column], column words [lane row][NJ]
  static constexpr int RC = kPC * NH, RQ = RC + kPC, SLOT = RQ + kPR * NJ;
  static constexpr int PJ16 = WJ + 8, PK16 = WK + 8;  // CS: halves per row-major profile row
  static constexpr int CVG = NJ * NH / 4;             // 16-byte groups of a lane's sigma'' tile
};

// Launch shape of a variant: 1-warp CTAs (2-warp for CS = 1), so that the CTA scheduler spreads the
// warps of a small launch over all SMs and their sub-partitions (4-warp CTAs put four tasks on one SM
// while others idle: two tasks on a sub-partition cost each 25-30% of its speed), and so that registers
// bound the resident warps in steps of one: `blocks` CTAs per SM.
// CS = 0 keeps the lane's sigma''(y,z) tile in registers; CS = 1 and 2 keep it and row-major profiles in
// shared memory (10 and 9 warps per SM).
// Two warps per sub-partition all but saturate it (32 x 64 tasks without waits: a step per 0.34 us with
// one, 0.27 with two, 0.26 with three), and a third would need the 8 x 4 tile in 168 registers: protein 1,000
// residues 0.67 -> 0.85 ms. The cap of 224 registers that `blocks` = 9 gives still leaves two; its code is the
// faster with traceback (DNA, 3,000 residues 11.3 -> 10.5 ms), the slower without (protein, 1,000 residues 0.649
// -> 0.653 ms, semi-global, where it spills, 4.09 -> 4.27, local 1,500 1.80 -> 2.20).
template <int NJ, int NH, int CS, int AT = kGlobal, bool TB = false>
struct VlLaunch {
  static constexpr int warps = CS == 1 ? 2 : 1;
  static constexpr int blocks =
      CS == 1 ? 5 : (CS == 2 ? 9 : (NH >= 8 ? 8 : (NJ >= 8 ? (TB ? 9 : 8) : 12)));
  static constexpr int regs = 65536 / (warps * 32 * blocks) / 8 * 8;
  static constexpr int max_regs = regs > 255 ? 255 : regs;
};

// Position of tile cell (pp, qq) in anti-diagonal order (diagonal pp + qq ascending, pp
// ascending within it): the order pass 2 visits the cells in, and pass 1 in reverse.
template <int NJ, int NH>
__host__ __device__ constexpr int vl_diag_index(int pp, int qq) {
  int e = 0;
  for (int dg = 0; dg < pp + qq; ++dg) {
    const int lo = dg - (NH - 1) > 0 ? dg - (NH - 1) : 0, hi = dg < NJ - 1 ? dg : NJ - 1;
    e += hi - lo + 1;
  }
  const int lo = pp + qq - (NH - 1) > 0 ? pp + qq - (NH - 1) : 0;
  return e + (pp - lo);
}

namespace {

// Record accesses: relaxed, gpu scope, each 32-bit element single-copy atomic, since a record word is
// its own readiness flag.
__device__ __forceinline__ void vl_load4(const int* w, int* v) {
  asm volatile("ld.relaxed.gpu.global.v4.s32 {%0,%1,%2,%3}, [%4];"
               : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3])
               : "l"(w)
               : "memory");
}
__device__ __forceinline__ void vl_load2(const int* w, int& x, int& y) {
  asm volatile("ld.relaxed.gpu.global.v2.s32 {%0,%1}, [%2];" : "=r"(x), "=r"(y) : "l"(w) : "memory");
}
__device__ __forceinline__ void vl_store(int* w, int a, int b, int c, int d, int* cb, int x, int y,
                                         int pr) {
  asm volatile(
      "{\n .reg .pred q;\n setp.ne.b32 q, %8, 0;\n"
      " @q st.relaxed.gpu.global.v4.s32 [%0], {%1,%2,%3,%4};\n"
      " @q st.relaxed.gpu.global.v2.s32 [%5], {%6,%7};\n}"
      ::"l"(w), "r"(a), "r"(b), "r"(c), "r"(d), "l"(cb), "r"(x), "r"(y), "r"(pr)
      : "memory");
}
__device__ __forceinline__ void vl_store(int* w, int a, int b, int c, int d, int pr) {
  asm volatile(
      "{\n .reg .pred q;\n setp.ne.b32 q, %5, 0;\n"
      " @q st.relaxed.gpu.global.v4.s32 [%0], {%1,%2,%3,%4};\n}"
      ::"l"(w), "r"(a), "r"(b), "r"(c), "r"(d), "r"(pr)
      : "memory");
}
// Predicated stores to the staging ring (32-bit shared addresses).
__device__ __forceinline__ void st_ring_row(unsigned w, int a, int b, int c, int d, int pr) {
  asm volatile(
      "{\n .reg .pred q;\n setp.ne.b32 q, %5, 0;\n @q st.shared.v4.s32 [%0], {%1,%2,%3,%4};\n}"
      ::"r"(w), "r"(a), "r"(b), "r"(c), "r"(d), "r"(pr)
      : "memory");
}
__device__ __forceinline__ void st_ring_corner(unsigned w, int a, int pr) {
  asm volatile("{\n .reg .pred q;\n setp.ne.b32 q, %2, 0;\n @q st.shared.s32 [%0], %1;\n}"
               ::"r"(w), "r"(a), "r"(pr)
               : "memory");
}
// column words: row 2e in the high half of word 2e, row 2e + 1 in that of word 2e + 1
template <int NJ>
__device__ __forceinline__ void st_ring_col(unsigned w, const int* v, int pr) {
  if constexpr (NJ == 8)
    asm volatile(
        "{\n .reg .pred q;\n setp.ne.b32 q, %9, 0;\n @q st.shared.v4.s32 [%0], {%1,%2,%3,%4};\n"
        " @q st.shared.v4.s32 [%0+16], {%5,%6,%7,%8};\n}"
        ::"r"(w), "r"(v[0] << 16), "r"(v[0]), "r"(v[1] << 16), "r"(v[1]), "r"(v[2] << 16), "r"(v[2]),
        "r"(v[3] << 16), "r"(v[3]), "r"(pr)
        : "memory");
  else
    asm volatile(
        "{\n .reg .pred q;\n setp.ne.b32 q, %5, 0;\n @q st.shared.v4.s32 [%0], {%1,%2,%3,%4};\n}"
        ::"r"(w), "r"(v[0] << 16), "r"(v[0]), "r"(v[1] << 16), "r"(v[1]), "r"(pr)
        : "memory");
}
// A lane's flag as an integer register: each use is one compare into a predicate.
__device__ __forceinline__ int vl_flag(bool b) {
  int f = b ? 1 : 0;
  asm volatile("" : "+r"(f));
  return f;
}

// N 16-bit values (N = 4 or 8) from shared memory as N/2 words
template <int N>
__device__ __forceinline__ void ld_halves(const unsigned short* p, unsigned (&v)[N / 2]) {
  if constexpr (N == 8) {
    const uint4 x = *reinterpret_cast<const uint4*>(p);
    v[0] = x.x;
    v[1] = x.y;
    v[2] = x.z;
    v[3] = x.w;
  } else {
    const uint2 x = *reinterpret_cast<const uint2*>(p);
    v[0] = x.x;
    v[1] = x.y;
  }
}

}  // namespace

// AT: the alignment type of Sec. II. Semi-global feeds its zero axes through the halo cells at
// j = -1 / k = -1 (as wavefront_kernel does, in the relative halves) and takes the best
// original-frame score over the last slices i = a, j = b, k = c. Local adds v = 0 to Eq. 1, i.e.
// M' >= -2*alpha*(i+j+k), which also gives its zero axes, as one more packed max in pass 1 (the
// floor is the same along an anti-diagonal of a half), and takes the best original-frame score
// over every cell: per step, each cell's M relative to a per-step reference is folded into a packed
// 16-bit maximum by one add-max, and the step's maximum into a 32-bit best.
//
// TB: traceback keys (global type). A half holds the key 8*M' + 3 relative to the base, so that
// every candidate's rank in Eq. 1's order comes out in its low 3 bits with few extra adds: the
// profiles carry +3 (J), +2 (K) and +1 (sigma''(y,z)), so the sums the score kernel forms anyway
// end in 6 (110), 5 (101), 4 (011) and, with a second K profile without its +2, 7 (111); 100 is
// the stored key itself (3), and 010 and 001 take -1 and -2 in an add-max in place of the score
// kernel's 3-input max. The low 3 bits of the maximum are the winning move; they are shifted into
// one code word per tile row and cleared to 3 again: 6 ALU-pipe instructions per two cells, where
// the one-pass int32 keys take 10 per cell. -infinity is 8, so the negative adds do not wrap it.
// Codes: lane l's low and high halves write the records of virtual lanes 2l and 2l + 1 (columns
// 0..NH-1 and NH..2NH-1 of its tile): at step t, words ((task * T + t) * 64 + 2l + h) * W ..,
// W = NJ*NH/8; cell (p, q) of a virtual lane is e = p*NH + q, in word e/8 at bit vl_code_bit(e).
//
// Hand-off. A record word is its own readiness flag. A task fills its record rows with kVlSentinel,
// which no packed word and no base equals, before it starts, and releases its progress word; a
// consumer acquires the progress words of its producers once, at its start, and from then on reloads a
// staged piece until none of its words is the sentinel (bounded). So a producer-consumer level lags
// by its skew and one trip through L2, and nothing is published while a task runs. Against progress
// counts published every 8 steps, same kernel: protein, 300 residues, 0.52 -> 0.25 ms; local, 1,500
// residues, 4.3 -> 1.9 ms; DNA traceback, 3,000 residues, 17.5 -> 14.5 ms.
// Measured (kernel time, this form against the int32 tiles or the earlier two-per-register kernel that
// kept absolute records by slice): DNA traceback, 1,000 residues, 1.45 -> 0.90 ms, 3,000 residues 21.7 ->
// 10.1 ms, 96 triplets of 200..600 6.2 -> 3.0 ms; protein score, 300 residues, 0.50 -> 0.19 ms, 1,000
// residues 1.74 -> 0.67 ms, 4,000 residues 28.0 (int32) and 21.7 -> 17.2 ms (3,720 GCUPS).
// A lone warp's step of 32 x 64 cells takes 0.34 us (0.61 before) in ~340 instructions, of which 200 are
// cell work at 2 cycles each on the ALU or the FMA pipe. Mixed, the two pipes do not reach 2 x 64
// instructions per SM and clock: three-register operands leave 85 (3-input max with a multiply-add) to
// 103 (add-max with one), so operand reads bind a full sub-partition; the rest of a launch is the
// chain of column tasks.
template <int NJ, int NH, int CS, int AT, bool TB>
__global__ void __launch_bounds__(VlLaunch<NJ, NH, CS, AT, TB>::warps * 32)
    __maxnreg__((VlLaunch<NJ, NH, CS, AT, TB>::max_regs)) wavefront_vl_kernel(const WaveParams p) {
  static_assert(AT == kGlobal || CS == 0, "the variant types keep sigma'' in registers");
  static_assert(!TB || (AT == kGlobal && CS == 0 && NH == 4), "traceback keys: global, NH = 4");
  using G = VlGeom<NJ, NH>;
  static_assert((NJ == 4 || NJ == 8) && (NH == 4 || NH == 8), "tile sides");
  constexpr int NK = G::NK, WJ = G::WJ, WK = G::WK;
  constexpr int NEGH = TB ? 8 : 0;      // -infinity of a half
  constexpr int NEG = NEGH * 0x10001;   // in both halves
  constexpr int BIAS = TB ? kVlTbBias : kVlBias;
  constexpr int kOffJ = TB ? 3 : 0, kOffK = TB ? 2 : 0, kOffC = TB ? 1 : 0;  // rank offsets
  // Two forms of a step, each where it is the faster (a step is bound by issue and by what the compiler lets
  // its loads share a scoreboard with, so neither is everywhere):
  // kXR: residues of S0 from a ring in shared memory instead of a global load per step. Local, protein 1,500
  // residues 2.00 -> 1.80 ms; global, 4,000 residues 17.4 -> 17.9, 1,024 semi-global triplets 4.1 -> 5.0.
  // kPK: right-column halves go to the next lane as the words the records hold, two rows each: half the
  // shuffles and selects. Protein 4,000 residues 17.4 -> 17.25 ms, 1,000 0.665 -> 0.644; DNA traceback, 3,000
  // residues 10.5 -> 11.9, local 1,500 2.00 -> 2.16.
  constexpr bool kXR = AT == kLocal && NJ == 8 && NH == 4;
  constexpr bool kPK = AT == kGlobal && !TB && CS == 0 && NJ == 8 && NH == 4;
  constexpr int NCV = kPK ? NJ / 2 : NJ;  // column words a step takes from the left lane
  constexpr int W = NJ * NK / 8;        // TB: code words per lane per step
  extern __shared__ int4 smem4[];
  int* smem = reinterpret_cast<int*>(smem4);
  const int KP = p.KP;
  const int VIRT = KP - 1;
  const int sigN = (KP * KP + 3) & ~3;
  int* sig = smem;
  const int warp = threadIdx.x >> 5;
  // opaque, so that the lane's indices stay in registers instead of being formed again in every step
  int lane = threadIdx.x & 31, r = lane >> 3, lc = lane & 7;
  asm volatile("" : "+r"(lane), "+r"(r), "+r"(lc));
  // Per warp: 16-bit profiles, the staging ring (two slots), and with CS the sigma'' tiles of the
  // warp's lanes ([group][lane][4] ints). Without CS the profile entries lie [x][lane row][lane
  // column] (J, NJ halves each, repeated per lane column) and [half][x][lane column] (K, NH
  // halves), so the 8 lanes of a 16-byte load phase read 8 distinct bank groups whatever their
  // residues (row-major rows left 36-46% of the shared-load wavefronts to bank conflicts).
  constexpr bool kPT = !CS;
  const int prof_ints =
      kPT ? KP * (kPR * kPC * NJ / 2 + kPC * NH) : KP * (G::PJ16 + G::PK16) / 2;
  const int warp_ints = prof_ints + kRing * G::SLOT + kVlRing + (CS ? 32 * 4 * G::CVG : 0);
  int* prof = smem + sigN + warp * warp_ints;
  unsigned short* profJ = reinterpret_cast<unsigned short*>(prof);
  unsigned short* profK =
      reinterpret_cast<unsigned short*>(prof + (kPT ? KP * kPR * kPC * NJ / 2 : KP * G::PJ16 / 2));
  int* ring = prof + prof_ints;
  int* xr = ring + kRing * G::SLOT;  // kXR: residues by slice
  int4* cvs = reinterpret_cast<int4*>(xr + kVlRing);  // CS only
  // this lane's profile entries: J of residue x at pJ + x * kSJ, K at pKl / pKh + x * kSK
  constexpr int kSJ = kPT ? kPR * kPC * NJ : G::PJ16, kSK = kPT ? kPC * NH : G::PK16;
  const unsigned short* pJ = profJ + (kPT ? lane * NJ : r * NJ);
  const unsigned short* pKl = profK + (kPT ? lc * NH : lc * NK);
  const unsigned short* pKh = profK + (kPT ? (KP * kPC + lc) * NH : lc * NK + NH);
  for (int e = threadIdx.x; e < KP * KP; e += blockDim.x) sig[e] = p.sig[e];
  __syncthreads();

  // Staging: item e < kPC is the row words of one lane column with its corner and base, item kPC + rr
  // the column words and base of lane row rr. The two halves of the warp (g) stage the items of an even
  // step and of the next one, so a pair of steps takes one load, one readiness check, one conversion
  // and one store; the lanes without an item of their own load another lane's again (no extra traffic,
  // no predicate).
  constexpr int kJL = kPC;
  const int g = lane >> 4, e0 = lane & 15;
  const unsigned ring_s = (unsigned)__cvta_generic_to_shared(ring);

  for (;;) {
    int task = 0;
    if (lane == 0) task = atomicAdd(p.queue, 1);
    task = __shfl_sync(kFull, task, 0);
    if (task >= p.ntasks) return;
    if (task < p.pace_n && task > 0) {  // in the test of the bounded waits alone (WaveParams)
      const int need = (int)((long long)task * p.pace_T / p.pace_n);
      bool okp = true;
      int seen = 0;
      if (lane == 0 && need > 0) okp = wait_flag(p.pace_flag, need, &seen, p.wait_ns);
      if (!__shfl_sync(kFull, okp, 0)) {
        if (lane == 0) atomicOr(p.err, 1);
        return;
      }
    }
    const Task tk = p.tasks[task];
    const TripDesc& d = p.desc[tk.trip];
    const int a = d.len[0], b = d.len[1], c = d.len[2];
    const int nJ = d.nJ, nK = d.nK, T = d.T;
    const int J = tk.J, K = tk.K;
    const int8_t* S0 = p.seq + d.s_off[0];
    const int8_t* S1 = p.seq + d.s_off[1];
    const int8_t* S2 = p.seq + d.s_off[2];
    const int j0 = J * WJ + r * NJ, k0 = K * WK + lc * NK;
    // records exist where there is a consumer: j-rows of all but the last block row, k-rows of all but the
    // last block column
    const int me = J * nK + K, mek = J * (nK - 1) + K;

    // Profiles of this block: sigma''(x, y_j) and sigma''(x, z_k); residue index 0 and beyond the
    // end are VIRT.
    __syncwarp();
    for (int e = lane; e < KP * WJ; e += 32) {
      const int x = e / WJ, jl = e - x * WJ, j = J * WJ + jl;
      const int y = (j >= 1 && j <= b) ? (int)S1[j - 1] : VIRT;
      const unsigned short v16 = (unsigned short)(sig[x * KP + y] + kOffJ);
      if (kPT) {
        const int rr = jl / NJ, pq = jl - rr * NJ;
        for (int l = 0; l < kPC; ++l) profJ[((x * kPR + rr) * kPC + l) * NJ + pq] = v16;
      } else {
        profJ[x * G::PJ16 + jl] = v16;
      }
    }
    for (int e = lane; e < KP * WK; e += 32) {
      const int x = e / WK, kl = e - x * WK, k = K * WK + kl;
      const int z = (k >= 1 && k <= c) ? (int)S2[k - 1] : VIRT;
      const unsigned short v16 = (unsigned short)(sig[x * KP + z] + kOffK);
      if (kPT) {
        const int l = kl / NK, rem = kl - l * NK, h = rem / NH, q = rem - h * NH;
        profK[((h * KP + x) * kPC + l) * NH + q] = v16;
      } else {
        profK[x * G::PK16 + kl] = v16;
      }
    }
    // sigma''(y_j, z_k) for both halves (left and right NH columns), packed, for the whole task:
    // in registers, or (CS) in shared memory in anti-diagonal order, read as the passes go
    int Cv[CS ? 1 : NJ][CS ? 1 : NH];
    {
      int yo[NJ];
#pragma unroll
      for (int pp = 0; pp < NJ; ++pp) {
        const int j = j0 + pp;
        yo[pp] = ((j >= 1 && j <= b) ? (int)S1[j - 1] : VIRT) * KP;
      }
#pragma unroll
      for (int qq = 0; qq < NH; ++qq) {
        const int kl = k0 + qq, kh = k0 + NH + qq;
        const int zl = (kl >= 1 && kl <= c) ? (int)S2[kl - 1] : VIRT;
        const int zh = (kh >= 1 && kh <= c) ? (int)S2[kh - 1] : VIRT;
#pragma unroll
        for (int pp = 0; pp < NJ; ++pp) {
          const int v = (int)__byte_perm(sig[yo[pp] + zl], sig[yo[pp] + zh], 0x5410) +
                        kOffC * 0x10001;
          if constexpr (CS) {
            const int e = vl_diag_index<NJ, NH>(pp, qq);
            reinterpret_cast<int*>(cvs + (e >> 2) * 32 + lane)[e & 3] = v;
          } else {
            Cv[pp][qq] = v;
          }
        }
      }
    }
    __syncwarp();

    // Owner of the final cell (a, b, c): its lane, half and tile cell.
    const int endK = c % WK;
    const bool owns_end = (J == b / WJ) && (K == c / WK) && (r == (b % WJ) / NJ) &&
                          (lc == endK / NK);
    const int end_p = b % NJ, end_h = (endK % NK) >= NH, end_q = (endK % NK) % NH;
    const int g2 = p.g2;  // -2*alpha per consumed residue (the frame shift)
    // Semi-global: tasks whose block holds the last row j = b or the last column k = c, and (0, 0)
    const bool last_j = AT == kSemiGlobal && J == nJ - 1, last_k = AT == kSemiGlobal && K == nK - 1;
    const bool first = AT == kSemiGlobal && J == 0 && K == 0;
    int best = kNeg;  // semi-global / local: best original-frame score of this lane's counted cells

    // TB: -1 from a launch argument (the subtraction stays a multiply-add), and the key masks as
    // registers (both in one LOP3)
    const int m1 = -p.one;
    unsigned key_mask = 0xfff8fff8u, key_low = 0x00030003u;
    if (TB) asm volatile("" : "+r"(key_mask), "+r"(key_low));
    int P[NJ][NH];
    int pk[NJ / 2];  // the right column's high halves, two rows a word
#pragma unroll
    for (int e = 0; e < NJ / 2; ++e) pk[e] = NEG;
    int rowA[NH + 1], colA[NJ], rowB[NH + 1], colB[NJ];
#pragma unroll
    for (int pp = 0; pp < NJ; ++pp) {
#pragma unroll
      for (int qq = 0; qq < NH; ++qq) P[pp][qq] = NEG;
      colA[pp] = NEG;
      colB[pp] = NEG;
    }
#pragma unroll
    for (int qq = 0; qq <= NH; ++qq) {
      rowA[qq] = NEG;
      rowB[qq] = NEG;
    }

    // Records: producer (J-1, K) of j-rows and (J, K-1) of k-rows; at step u an item comes from
    // producer row u + kPR - 1 or u + 2*kPC - 1.
    const bool has_j = J > 0, has_k = K > 0;
    // the item this lane loads: its own, or one whose producer exists
    const int it_e = has_j ? (has_k ? (e0 < kJL + kPR ? e0 : e0 - kJL - kPR) : e0 % kJL)
                           : kJL + e0 % kPR;
    const bool is_j = it_e < kJL, own = it_e == e0;
    const int it_l = is_j ? it_e : it_e - kJL;          // lane column or lane row
    const int it_delta = (is_j ? 2 * it_l : it_l) - g;  // the item's slice in pair u is u - delta
    const int it_off = is_j ? it_l * NH : 4 * it_l;
    const int it_off2 = is_j ? kPC * NH + 2 * it_l : kPR * 4 + 2 * it_l;
    const int f_j = vl_flag(has_j && own && is_j), f_k = vl_flag(has_k && own && !is_j);
    const unsigned st_w = ring_s + 4 * (g * G::SLOT + (is_j ? it_l * NH : G::RQ + it_l * NJ));
    const unsigned st_c = ring_s + 4 * (g * G::SLOT + G::RC + it_l);
    const int it_stride = is_j ? G::RJ : G::RK;
    const int* it_src =
        p.faces + (is_j ? d.oj_off + ((int64_t)(me - nK) * T + (kPR - 1) + g) * G::RJ
                        : d.ok_off + ((int64_t)(mek - 1) * T + (2 * kPC - 1) + g) * G::RK);
    const bool out_j = r == kPR - 1 && J + 1 < nJ, out_k = lc == kPC - 1 && K + 1 < nK;
    const int f_oj = vl_flag(out_j), f_ok = vl_flag(out_k);
    int* dstJ = p.faces + d.oj_off + (int64_t)me * T * G::RJ + lc * NH;
    int* dstK = p.faces + d.ok_off + (int64_t)mek * T * G::RK + r * 4;
    bool ok = true;
    uint32_t* codes = TB ? p.codes + d.code_off + (int64_t)me * T * 32 * W + lane * W : nullptr;
    // Without a producer the halo of the first lane row or column stays -infinity.
    for (int e = lane; e < kRing * G::SLOT; e += 32) ring[e] = NEG;
    // This task's rows start as the sentinel; then wait until those of its producers do.
    {
      const auto fill = [&](int* q, int64_t n) {
        int4* q4 = reinterpret_cast<int4*>(q);
        for (int64_t e = lane; e < n / 4; e += 32)
          st_relaxed_if(q4 + e, make_int4(kVlSentinel, kVlSentinel, kVlSentinel, kVlSentinel), true);
      };
      if (J + 1 < nJ) fill(p.faces + d.oj_off + (int64_t)me * T * G::RJ, (int64_t)T * G::RJ);
      if (K + 1 < nK) fill(p.faces + d.ok_off + (int64_t)mek * T * G::RK, (int64_t)T * G::RK);
      __syncwarp();
      int* prog = p.progress + d.prog_base + me;
      if (lane == 0) {
        int seen = 0;
        st_release(prog, 1);
        if (has_j) ok = wait_flag(prog - nK, 1, &seen, p.wait_ns);
        if (ok && has_k) ok = wait_flag(prog - 1, 1, &seen, p.wait_ns);
      }
      ok = __shfl_sync(kFull, ok, 0);
      __syncwarp();  // the other lanes' loads come after lane 0's acquire
    }

    // A piece: the words and (corner, base) or (base, base) of one item in pair u (steps u and u + 1,
    // u even). mul converts the words to this task's base by one multiply-add each; an item whose slice
    // is outside the cube holds -infinity and mul = 0.
    struct Piece {
      int v[NH], x, y, mul;
    };
    Piece pq;
    const bool has_any = has_j || has_k;
    const auto load = [&](int u) {
      const int* src = it_src + (int64_t)u * it_stride;
      vl_load4(src + it_off, pq.v);
      if (NH == 8) vl_load4(src + it_off + (is_j ? 4 : 0), pq.v + NH - 4);
      vl_load2(src + it_off2, pq.x, pq.y);
    };
    // `inner`: every lane's slice of both steps lies in the cube.
    auto fetch = [&](int u, bool inner) {
      if (!has_any) return;
      if (inner) {
        load(u);
      } else {
        // a row item has a producer value up to the extra slice a + 1, a column item up to a
        const int sl = u - it_delta;
        const bool valid = sl >= 0 && sl <= (is_j ? a + 1 : a);
#pragma unroll
        for (int e = 0; e < NH; ++e) pq.v[e] = NEG;
        pq.x = pq.y = NEG;
        pq.mul = 0;
        if (valid) {
          load(u);
          pq.mul = 0x10001;
        }
      }
    };
    // Reload the piece of pair u until none of its words is the sentinel (bounded).
    auto resolve = [&](int u) {
      const auto missing = [&]() {
        unsigned m = __vimax3_u32((unsigned)pq.x, (unsigned)pq.y, (unsigned)pq.v[0]);
#pragma unroll
        for (int e = 1; e + 1 < NH; e += 2)
          m = __vimax3_u32(m, (unsigned)pq.v[e], (unsigned)pq.v[e + 1]);
        return max(m, (unsigned)pq.v[NH - 1]) == (unsigned)kVlSentinel;
      };
      if (__any_sync(kFull, missing())) {
        const uint64_t t0 = global_ns();
        unsigned ns = 32;
        for (;;) {
          __nanosleep(ns);
          if (ns < 256) ns <<= 1;
          if (missing()) load(u);
          if (!__any_sync(kFull, missing())) break;
          if (__shfl_sync(kFull, (int64_t)(global_ns() - t0) > p.wait_ns ? 1 : 0, 0)) {
            ok = false;
            break;
          }
        }
      }
    };

#pragma unroll
    for (int e = 0; e < NH; ++e) pq.v[e] = 0;
    pq.x = pq.y = pq.mul = 0;
    if (ok) {
      fetch(0, false);
      resolve(0);
    }
    // The base: the larger of lane 0's upper and left neighbours at slice 0 (first word of lane
    // column 0 and of lane row 0); lane 0's first cell is at most 2*max sigma'' above it.
    int Bt = 0;
    {
      const int mine = (pq.v[0] & 0xffff) + pq.y - BIAS;
      const int mj = __shfl_sync(kFull, mine, 0), mk = __shfl_sync(kFull, mine, has_j ? kJL : 0);
      if (has_j) Bt = mj;
      if (has_k) Bt = has_j ? max(mj, mk) : mk;
      Bt &= ~7;  // a multiple of 8: the keys keep their low bits, and a stored base is no sentinel
    }
    // M'[-1][-1][-1] = 0 feeds the origin through the (1,1,1) move (low half of lane 0).
    if (J == 0 && K == 0 && lane == 0) rowB[0] = (NEG & ~0xffff) | (BIAS + (TB ? 3 : 0));
    // Semi-global zero axes in the shifted frame: M'[-1][-1][k] = g2*k feeds the k axis (move
    // (1,1,0)), M'[-1][j][-1] = g2*j the j axis (move (1,0,1)), M'[i][-1][-1] = g2*i the i axis
    // (move (0,1,1)); lane 0 starts from slice -1 (low halves; the high half's are reset). Beyond b and
    // c the axes stay at their last value, so that M' does not change along virtual residues (below).
    const auto feed = [&](int v) { return max(v + BIAS - Bt, 0); };
    if (AT == kSemiGlobal && lane == 0) {
      if (J == 0) {
#pragma unroll
        for (int qq = 0; qq <= NH; ++qq) rowB[qq] = feed(g2 * min(max(k0 + qq - 1, 0), c));
      }
      if (K == 0) {
#pragma unroll
        for (int pp = 0; pp < NJ; ++pp) colB[pp] = feed(g2 * min(j0 + pp, b));
      }
    }

    // Residues and profiles ahead of their step: at step t, xlast, xc and xq hold the residues of
    // slices s, s + 1 and s + 2, and the profile words of slice s are in registers.
    const auto residue = [&](int sl) {
      return (unsigned)(sl - 1) < (unsigned)a ? (int)__ldg(S0 + sl - 1) : VIRT;
    };
    const int s00 = -(r + 2 * lc);  // slice of this lane at step 0
    unsigned jA[NJ / 2], jB[NJ / 2], kl[NH / 2], kh[NH / 2];  // jA: even steps' slice s, jB: s - 1
    int xc = residue(s00), xq = residue(s00 + 1);
    {
      const int xm = residue(s00 - 1);
      ld_halves<NJ>(pJ + xm * kSJ, jB);
      ld_halves<NJ>(pJ + xc * kSJ, jA);
      ld_halves<NH>(pKl + xc * kSK, kl);
      ld_halves<NH>(pKh + xm * kSK, kh);
    }
    int xlast = xc;
    xc = xq;
    // kXR: the residues from slice s + 2 on come from a ring of two blocks of 32 slices (block n covers slices
    // 32n .. 32n + 31), a block being stored in the middle of the one before, when the block it replaces is
    // behind every lane.
    if constexpr (kXR) {
      xr[lane] = residue(lane);
      xr[32 + lane] = VIRT;  // the slices before 0
      __syncwarp();
    } else {
      xq = residue(s00 + 2);
    }
    const auto refill = [&](const int t) {
      if (kXR && (t & 31) == 16) xr[(t + 16 + lane) & (kVlRing - 1)] = residue(t + 16 + lane);
    };

    // One step: the halo of slice s goes into rowCur / colCur, slice s - 1 is in rowPrev / colPrev.
    // inner: every lane has 1 <= s < a, so no lane needs a range check, a reset or end-cell work,
    // and nor does the piece of step t + 2.
    // Stage the piece of pair t (two cells per word: one add converts both to this base) in ring slots
    // `slot` and `slot` + 1, and load that of pair t + 2 in its place.
    auto stage = [&](const int t, const bool inner, const int slot) -> bool {
      resolve(t);
      if (!ok) return false;
      const int db1 = pq.y - Bt, db = db1 * (inner ? 0x10001 : pq.mul);
      int w[NH];
#pragma unroll
      for (int e = 0; e < NH; ++e) w[e] = pq.v[e] + db;
      int cw = pq.x + db;
      // Lane column 0's corner is -infinity in the low half on the k = 0 face, and at the extra slice
      // a + 1 (where its producer had no left neighbour). It must not be added to: the borrow would
      // reach the high half.
      if (e0 == 0 && (K == 0 || (!inner && t + g > a)))
        cw = ((pq.x & ~0xffff) + ((inner || pq.mul) ? db1 << 16 : 0)) | NEGH;
      const unsigned o = 4 * slot * G::SLOT;
#pragma unroll
      for (int q4 = 0; q4 < NH / 4; ++q4)
        st_ring_row(st_w + o + 16 * q4, w[4 * q4], w[4 * q4 + 1], w[4 * q4 + 2], w[4 * q4 + 3], f_j);
      st_ring_corner(st_c + o, cw, f_j);
      if constexpr (kPK) st_ring_row(st_w + o, w[0], w[1], w[2], w[3], f_k);
      else st_ring_col<NJ>(st_w + o, w, f_k);
      if (inner || t + 2 < T) fetch(t + 2, inner);
      __syncwarp();
      return true;
    };
    auto step = [&](const int t, const bool inner, const int slot, unsigned (&jc)[NJ / 2],
                    unsigned (&jp)[NJ / 2], int (&rowCur)[NH + 1], const int (&rowPrev)[NH + 1],
                    int (&colCur)[NJ], const int (&colPrev)[NJ]) {
      const int s = t - r - 2 * lc;
      int A[NJ], Bq[NH];
#pragma unroll
      for (int w = 0; w < NJ / 2; ++w) {  // low half: slice s, high half: slice s - 1
        A[2 * w] = (int)__byte_perm(jc[w], jp[w], 0x5410);
        A[2 * w + 1] = (int)__byte_perm(jc[w], jp[w], 0x7632);
      }
#pragma unroll
      for (int w = 0; w < NH / 2; ++w) {
        Bq[2 * w] = (int)__byte_perm(kl[w], kh[w], 0x5410);
        Bq[2 * w + 1] = (int)__byte_perm(kl[w], kh[w], 0x7632);
      }
      // profile words of step t + 1, residue of slice s + 3
      ld_halves<NJ>(pJ + xc * kSJ, jp);
      ld_halves<NH>(pKl + xc * kSK, kl);
      ld_halves<NH>(pKh + xlast * kSK, kh);
      xlast = xc;
      if constexpr (kXR) {
        xc = xr[(s + 2) & (kVlRing - 1)];
      } else {
        xc = xq;
        xq = inner ? (int)__ldg(S0 + (s + 2)) : residue(s + 3);
      }
      // Halo of slice s from the neighbour lanes' previous step; the edge lanes take the staged
      // words instead. Column words: this row's value in the high half (kPK: two rows' values).
#pragma unroll
      for (int qq = 0; qq <= NH; ++qq)
        rowCur[qq] = __shfl_up_sync(kFull, qq == 0 ? colPrev[NJ - 1] : P[NJ - 1][qq - 1], kPC);
      int cv_[NCV], mine[NJ];
#pragma unroll
      for (int pp = 0; pp < NJ; ++pp) mine[pp] = P[pp][NH - 1];
#pragma unroll
      for (int w = 0; w < NCV; ++w) cv_[w] = __shfl_up_sync(kFull, kPK ? pk[w % (NJ / 2)] : mine[w], 1);
      {
        const int* q = ring + slot * G::SLOT;
        const int corner = q[G::RC + lc];
        rowCur[0] = r == 0 ? corner : rowCur[0];
#pragma unroll
        for (int q4 = 0; q4 < NH / 4; ++q4) {
          const int4 w = reinterpret_cast<const int4*>(q + lc * NH)[q4];
          rowCur[1 + 4 * q4] = r == 0 ? w.x : rowCur[1 + 4 * q4];
          rowCur[2 + 4 * q4] = r == 0 ? w.y : rowCur[2 + 4 * q4];
          rowCur[3 + 4 * q4] = r == 0 ? w.z : rowCur[3 + 4 * q4];
          rowCur[4 + 4 * q4] = r == 0 ? w.w : rowCur[4 + 4 * q4];
        }
#pragma unroll
        for (int p4 = 0; p4 < NCV / 4; ++p4) {
          const int4 w = reinterpret_cast<const int4*>(q + G::RQ + r * NJ)[p4];
          cv_[4 * p4] = lc == 0 ? w.x : cv_[4 * p4];
          cv_[4 * p4 + 1] = lc == 0 ? w.y : cv_[4 * p4 + 1];
          cv_[4 * p4 + 2] = lc == 0 ? w.z : cv_[4 * p4 + 2];
          cv_[4 * p4 + 3] = lc == 0 ? w.w : cv_[4 * p4 + 3];
        }
      }
#pragma unroll
      for (int pp = 0; pp < NJ; ++pp)
        colCur[pp] = (int)__byte_perm((unsigned)cv_[kPK ? pp / 2 : pp], (unsigned)mine[pp],
                                      kPK && pp % 2 == 0 ? 0x5410 : 0x5432);
      // Axis feeds. Only two kinds of halo cells are finite: those of slice -1 (each lane meets slice -1
      // once, the step before its first) and the i-axis feed M'[s][-1][-1] of lane 0 of task (0, 0);
      // every other halo cell of the first row or column stays -infinity, as staged.
      if (AT == kSemiGlobal && !inner && (J == 0 || K == 0)) {
        if (J == 0 && r == 0 && s == -1) {
#pragma unroll
          for (int qq = 0; qq <= NH; ++qq)
            rowCur[qq] = (int)(((unsigned)rowCur[qq] & 0xffff0000u) |
                               (unsigned)feed(g2 * min(k0 + qq - 1, c)));
        }
        if (K == 0 && lc == 0 && s == -1) {
#pragma unroll
          for (int pp = 0; pp < NJ; ++pp)
            colCur[pp] = (int)(((unsigned)colCur[pp] & 0xffff0000u) |
                               (unsigned)feed(g2 * min(j0 + pp, b)));
        }
      }
      if (AT == kSemiGlobal && first && lane == 0 && s >= 0)
        rowCur[0] = (int)(((unsigned)rowCur[0] & 0xffff0000u) | (unsigned)feed(g2 * s));

      const bool active = inner || (s >= 0 && s <= a + 1);
      unsigned cw[TB ? NJ : 1];  // TB: one code word per tile row, both halves
      if (active) {
        // sigma''(y, z) of tile cell (pp, qq): a register, or (CS) a shared-memory read
        const auto cv = [&](const int pp, const int qq) -> unsigned {
          if constexpr (CS) {
            const int e = vl_diag_index<NJ, NH>(pp, qq);
            return (unsigned)reinterpret_cast<const int*>(cvs + (e >> 2) * 32 + lane)[e & 3];
          } else {
            return (unsigned)Cv[pp][qq];
          }
        };
        // Local: the floor of each anti-diagonal e = pp + qq of the tile, both halves, relative
        // and clamped at 0 (a floor below the representable range cannot win: every value of
        // the working set lies above it): M' >= g2*(i+j+k) with i+j+k = s + j0 + k0 + e (low
        // half) and s - 1 + j0 + k0 + NH + e (high half).
        unsigned fl_base = 0, fl_step = 0, fl = 0;  // local: the current diagonal's floor
        if constexpr (AT == kLocal) {
          const int f0 = max(g2 * (s + j0 + k0) + BIAS - Bt, -30000);  // fits s16 with + g2*e below
          fl_base = (unsigned)(f0 & 0xffff) | ((unsigned)((f0 + g2 * (NH - 1)) & 0xffff) << 16);
          fl_step = (unsigned)g2 * 0x10001u;
        }
        int Bd[NH];  // sigma''(x, z) in the diagonal sum: without the rank offset of the 101 move
#pragma unroll
        for (int qq = 0; qq < NH; ++qq) Bd[qq] = Bq[qq] - kOffK * 0x10001;
        // Q = max{ max(Pd + A + B, Myz) + C, Pxy + A, Pxz + B, Sx, Sy, Sz }: the diagonal and the (0,1,1)
        // move share the add of C, so a register takes 4 ALU-pipe instructions (two fused add-maxima,
        // two 3-input maxima) and 2.25 multiply-adds. (With E = max{ Pd + A + B + C, ... } formed first,
        // 3.25: both pipes and the register reads bind, an SMSP does a step per 0.30 us at best.)
        // The part from the previous slice (E, X) runs one anti-diagonal ahead of the part within the
        // slice, so each fills the other's waits. ea[pp] holds A + (row above, slice s - 1) of the last
        // column done in row pp: the 110 sum of that column and the diagonal sum of the next.
        int E[NJ][NH], X[NJ][NH], Q[NJ][NH], ea[NJ];
#pragma unroll
        for (int pp = 0; pp < NJ; ++pp)
          ea[pp] = mad_lo(A[pp], p.one, pp == 0 ? rowPrev[0] : colPrev[pp - 1]);
        auto from_prev = [&](const int pp, const int qq) {
          const int Pxy = (pp == 0) ? rowPrev[qq + 1] : P[pp - 1][qq];
          const int Pxz = (qq == 0) ? colPrev[pp] : P[pp][qq - 1];
          X[pp][qq] = ea[pp];
          ea[pp] = mad_lo(A[pp], p.one, Pxy);
          const unsigned eb = (unsigned)mad_lo(Bq[qq], p.one, Pxz);
          unsigned Sx = (unsigned)P[pp][qq];
          if constexpr (AT == kLocal) Sx = __vmaxu2(Sx, fl);  // v = 0: the diagonal's floor
          E[pp][qq] = (int)__vimax3_u16x2((unsigned)ea[pp], eb, Sx);
        };
        auto in_slice = [&](const int pp, const int qq) {
          const int Myz = (pp == 0) ? rowCur[qq] : (qq == 0 ? colCur[pp - 1] : Q[pp - 1][qq - 1]);
          const int Sy = (pp == 0) ? rowCur[qq + 1] : Q[pp - 1][qq];
          const int Sz = (qq == 0) ? colCur[pp] : Q[pp][qq - 1];
          const unsigned w = __viaddmax_u16x2((unsigned)X[pp][qq], (unsigned)Bd[qq], (unsigned)Myz);
          unsigned q = __viaddmax_u16x2(w, cv(pp, qq), (unsigned)E[pp][qq]);
          if constexpr (TB) {
            q = __viaddmax_u16x2((unsigned)Sy, 0xffffffffu, q);  // rank 2
            q = __viaddmax_u16x2((unsigned)Sz, 0xfffefffeu, q);  // rank 1
            asm("lop3.b32 %0, %1, %2, %3, 0xea;"  // (q & key_mask) | key_low
                : "=r"(Q[pp][qq])
                : "r"(q), "r"(key_mask), "r"(key_low));
            const unsigned rk = (unsigned)mad_lo(Q[pp][qq], m1, (int)q);  // rank - 3 (with borrows)
            cw[pp] = qq == 0 ? rk : (unsigned)mad_lo((int)cw[pp], 16, (int)rk);
          } else {
            Q[pp][qq] = (int)__vimax3_u16x2(q, (unsigned)Sy, (unsigned)Sz);
          }
        };
#pragma unroll
        for (int dg = -1; dg < NJ + NH - 1; ++dg) {
          if constexpr (AT == kLocal) fl = __viaddmax_s16x2(fl_base, (unsigned)(dg + 1) * fl_step, 0u);
#pragma unroll
          for (int pp = 0; pp < NJ; ++pp) {
            const int qq = dg + 1 - pp;
            if (qq >= 0 && qq < NH) from_prev(pp, qq);
          }
#pragma unroll
          for (int pp = 0; pp < NJ; ++pp) {
            const int qq = dg - pp;
            if (qq >= 0 && qq < NH) in_slice(pp, qq);
          }
        }
#pragma unroll
        for (int pp = 0; pp < NJ; ++pp)
#pragma unroll
          for (int qq = 0; qq < NH; ++qq) P[pp][qq] = Q[pp][qq];
        if (!inner && s == 0) {  // the high half was at slice -1: -infinity there and in its halos
#pragma unroll
          for (int pp = 0; pp < NJ; ++pp) {
#pragma unroll
            for (int qq = 0; qq < NH; ++qq) P[pp][qq] = (P[pp][qq] & 0xffff) | (NEGH << 16);
            colCur[pp] = (colCur[pp] & 0xffff) | (NEGH << 16);
          }
#pragma unroll
          for (int qq = 0; qq <= NH; ++qq) rowCur[qq] = (rowCur[qq] & 0xffff) | (NEGH << 16);
          if (AT == kSemiGlobal && J == 0 && r == 0) {
            // the high half's halo row j = -1 at slice -1 is the k-axis feed M'[-1][-1][k]
#pragma unroll
            for (int qq = 0; qq <= NH; ++qq)
              rowCur[qq] |= feed(g2 * min(k0 + NH + qq - 1, c)) << 16;
          }
        }
      }
      if (active) {
        if constexpr (TB) {  // the codes of both virtual lanes (rows 2w and 2w + 1 in word w)
          uint32_t* dst = codes + (int64_t)t * 32 * W;
          uint32_t w[NJ];
#pragma unroll
          for (int e = 0; e < NJ; ++e) cw[e] += 0x33333333u;  // ranks: the sums of rank - 3 plus 3s
#pragma unroll
          for (int e = 0; e < NJ / 2; ++e) {
            w[e] = __byte_perm(cw[2 * e], cw[2 * e + 1], 0x5410);
            w[NJ / 2 + e] = __byte_perm(cw[2 * e], cw[2 * e + 1], 0x7632);
          }
#pragma unroll
          for (int e = 0; e < NJ / 4; ++e)
            reinterpret_cast<uint4*>(dst)[e] =
                make_uint4(w[4 * e], w[4 * e + 1], w[4 * e + 2], w[4 * e + 3]);
        }
        // Record rows of this step: the last lane row's bottom words with the corner its consumer
        // needs, the last lane column's right high halves (slice s - 1), and the base of both.
        {
          int* q = dstJ + (int64_t)t * G::RJ;
          vl_store(q, P[NJ - 1][0], P[NJ - 1][1], P[NJ - 1][2], P[NJ - 1][3],
                   q + kPC * NH - lc * NH + 2 * lc, colCur[NJ - 1], Bt, f_oj);
          if constexpr (NH == 8)
            vl_store(q + 4, P[NJ - 1][4], P[NJ - 1][5], P[NJ - 1][6], P[NJ - 1][7], f_oj);
        }
        {
          int* q = dstK + (int64_t)t * G::RK;
#pragma unroll
          for (int e = 0; e < NJ / 2; ++e)
            pk[e] = (int)__byte_perm((unsigned)P[2 * e][NH - 1], (unsigned)P[2 * e + 1][NH - 1],
                                     0x7632);
          vl_store(q, pk[0], pk[1], NJ == 8 ? pk[NJ / 2 - 2] : 0, NJ == 8 ? pk[NJ / 2 - 1] : 0, q + kPR * 4 - r * 2, Bt, Bt,
                   inner ? f_ok : (s >= 1 ? f_ok : 0));
        }
        const int ub = Bt - BIAS;  // biased half -> absolute M' (or key)
        // Original-frame scores M = M' - g2*(i+j+k). Relative to a per-step reference, D = half + 2^14 -
        // g2*d (d: the cell's offset of i+j+k from the reference cell's) equals M - mbase with
        // mbase = Bt - g2*(reference) - 2^15 and lies in (0, 2^16) by the range argument, so one unsigned
        // add-max per register folds a cell into a packed maximum.
        const unsigned g2x2 = (unsigned)g2 * 0x10001u;
        const unsigned add0 = 0x40004000u - ((unsigned)(g2 * (NH - 1)) << 16);  // high half: slice s - 1
        // the best D of the tile, d from the lane corner's i+j+k at the low half's slice. Cells of one
        // anti-diagonal share d, so they meet in 3-input maxima first.
        const auto best_of_tile = [&]() {
          unsigned acc = 0;
#pragma unroll
          for (int dg = 0; dg < NJ + NH - 1; ++dg) {
            const unsigned off = add0 - (unsigned)dg * g2x2;
            unsigned m[3] = {0u, 0u, 0u};
            int k = 0;
#pragma unroll
            for (int pp = 0; pp < NJ; ++pp) {
              const int qq = dg - pp;
              if (qq >= 0 && qq < NH) {
                m[k++] = (unsigned)P[pp][qq];
                if (k == 3) {
                  acc = __viaddmax_u16x2(__vimax3_u16x2(m[0], m[1], m[2]), off, acc);
                  k = 0;
                }
              }
            }
            if (k == 2) acc = __viaddmax_u16x2(__vmaxu2(m[0], m[1]), off, acc);
            if (k == 1) acc = __viaddmax_u16x2(m[0], off, acc);
          }
          return acc;
        };
        if constexpr (AT == kLocal) {
          // Every cell counts but the low half's extra slice a + 1 and the high half's slice -1 (a masked
          // half contributes 0, below any counted cell's D).
          const unsigned acc = best_of_tile();
          const int dlo = inner || s <= a ? (int)(acc & 0xffffu) : 0,
                    dhi = inner || s >= 1 ? (int)(acc >> 16) : 0;
          best = max(best, max(dlo, dhi) + Bt - g2 * (s + j0 + k0) - 32768);
        }
        if constexpr (AT == kSemiGlobal) {
          // The faces i = a, j = b and k = c. Along virtual residues M' does not change, so the block's
          // last row holds the values of row b and its last column those of column c, wherever b and c
          // lie in the block; cells beyond b or c only lose g2 a step more, so none needs a mask.
          if (last_j && r == kPR - 1) {
            unsigned acc = 0;
#pragma unroll
            for (int qq = 0; qq < NH; ++qq)
              acc = __viaddmax_u16x2((unsigned)P[NJ - 1][qq], add0 - (unsigned)qq * g2x2, acc);
            const int dlo = inner || s <= a ? (int)(acc & 0xffffu) : 0,
                      dhi = inner || s >= 1 ? (int)(acc >> 16) : 0;
            best = max(best, max(dlo, dhi) + Bt - g2 * (s + b + k0) - 32768);
          }
          if (last_k && lc == kPC - 1 && (inner || s >= 1)) {  // high halves, slice s - 1
            unsigned acc = 0;
#pragma unroll
            for (int pp = 0; pp < NJ; ++pp)
              acc = __viaddmax_u16x2((unsigned)P[pp][NH - 1], 0x40004000u - (unsigned)pp * g2x2, acc);
            best = max(best, (int)(acc >> 16) + Bt - g2 * (s - 1 + j0 + c) - 32768);
          }
          if (!inner && (s == a || s == a + 1)) {
            const unsigned acc = best_of_tile();
            best = max(best, (int)(s == a ? acc & 0xffffu : acc >> 16) + Bt - g2 * (s + j0 + k0) - 32768);
          }
        }
        if (AT == kGlobal && !inner && owns_end && (end_h ? s - 1 == a : s == a)) {
          unsigned v = 0;
#pragma unroll
          for (int pp = 0; pp < NJ; ++pp)
#pragma unroll
            for (int qq = 0; qq < NH; ++qq)
              if (pp == end_p && qq == end_q) v = (unsigned)P[pp][qq];
          const int h16 = end_h ? (int)(v >> 16) : (int)(v & 0xffffu);
          p.scores[d.out_idx] = (TB ? (h16 + ub) >> 3 : h16 + ub) + d.score_base;
        }
      }
    };
    // Raise the base when lane 0's first cell is 2048 above the bias (warp-uniform; after an odd
    // step, whose current halos are in rowB / colB). That cell never falls (M' grows along i).
    // max(v, d + -infinity) - d leaves -infinity as it is and borrows from no half.
    auto rebase = [&]() {
      const int ref = __shfl_sync(kFull, (int)((unsigned)P[0][0] & 0xffffu), 0);
      const int dlt = (ref - BIAS) & ~7;
      if (dlt >= 2048) {
        const unsigned m = (unsigned)dlt * 0x10001u, mn = m + NEG;
#pragma unroll
        for (int pp = 0; pp < NJ; ++pp) {
#pragma unroll
          for (int qq = 0; qq < NH; ++qq)
            P[pp][qq] = (int)(__vmaxu2((unsigned)P[pp][qq], mn) - m);
          colB[pp] = (int)(__vmaxu2((unsigned)colB[pp], mn) - m);
        }
        if constexpr (kPK) {
#pragma unroll
          for (int e = 0; e < NJ / 2; ++e) pk[e] = (int)(__vmaxu2((unsigned)pk[e], mn) - m);
        }
#pragma unroll
        for (int qq = 0; qq <= NH; ++qq) rowB[qq] = (int)(__vmaxu2((unsigned)rowB[qq], mn) - m);
        Bt += dlt;
      }
    };
    // Steps from kInner on and below a have every lane at a slice 1 <= s < a: no range checks, resets or
    // end-cell work.
    constexpr int kInner = (kPR - 1) + 2 * (kPC - 1) + 1;
    static_assert(kInner % 2 == 0, "pairs of steps");
    // A pair of steps. Longer unrolling (four steps, pieces two pairs ahead in two register sets) shortens
    // a lone warp's step by 10-20%, but its code overflows the instruction cache as soon as warps are in
    // different phases: the 300-residue protein triplet 0.19 -> 0.23 ms, 1,024 triplets 3.7 -> 4.6 ms.
    auto pair = [&](const int t, const bool inner) -> bool {
      const int slot = t & 2;
      refill(t);
      if (!stage(t, inner, slot)) return false;
      step(t, inner, slot, jA, jB, rowA, rowB, colA, colB);
      if (inner || t + 1 < T) step(t + 1, inner, slot + 1, jB, jA, rowB, rowA, colB, colA);
      rebase();
      return true;
    };
    int t = 0;
    bool running = ok;
    while (running && t < T) {
      if (t == kInner) {
        // t + 5 <= a: the residue of slice t + 4 is fetched unchecked
        for (; running && t + 5 <= a; t += 2) running = pair(t, true);
        if (!running) break;
      }
      running = pair(t, false);
      t += 2;
    }
    __syncwarp();
    if (!ok) {
      if (lane == 0) atomicOr(p.err, 1);
      return;
    }
    if (AT != kGlobal) {  // the triplet's score is the max over its tasks' lanes
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) best = max(best, __shfl_xor_sync(kFull, best, off));
      if (lane == 0) atomicMax(p.scores + d.out_idx, best);
    }
  }
}

}  // namespace trioseq
