// affine.cu — score of the exact 3-way global alignment under affine gaps (sm_103a).
//
// The model is the sum-of-pairs score with natural gap costs: each pair's induced pairwise
// alignment (columns with a gap in both of its sequences deleted) scores sigma per residue pair,
// alpha per residue against a gap, and gamma once per maximal run of gaps in one sequence. The
// paper names affine gaps as future work (Sec. VI) without a definition; this is the reading the
// oracle implements.
//
// State of an alignment prefix: per pair, the kind of its last induced column (0 both residues or
// none, 1 gap in the pair's first sequence, 2 gap in its second). Only 13 of the 27 combinations
// can follow a column: the four moves with at least two residues set all three pairs, and each
// single-residue move sets two and keeps the third (Eq. 1's moves, (pair 01, pair 02, pair 12)):
//   111 -> s (0,0,0)   110 -> a (0,2,2)   101 -> b (2,0,1)   011 -> c (1,1,0)
//   100 -> x0..x2 (2,2,k12)   010 -> y0..y2 (1,k02,2)   001 -> z0..z2 (k01,1,1)
//
// affine_kernel: the register-tiled wavefront of wavefront.cuh (column tasks, queue, boundary
// records, progress flags, staging ring) with 13 values per cell.
//  * Push form. A cell publishes, for each move out of it, the best value with the openings that
//    move adds already charged: one value per (move, state it leads to), 13 in all, each read by
//    exactly one cell. So a cell's 13 states are 13 reads (4 with a substitution score added; the
//    single-residue moves cost 0 in the shifted frame of engine.h), and its 13 outgoing values are
//    46 maxima and add-maxima over groups of states with the same number of openings, instead of
//    the 91 add-max candidates of the definition. That, with the values in registers instead of 13
//    ints per cell in memory, is what the kernel is for: it is bound by the ALU pipe (46
//    instructions per cell, or per two cells when packed).
//  * Tile. 4 x 4 cells per lane: 96 values live across slices (the moves out of slice s - 1), two
//    CTAs of 4 warps per SM. Boundary records hold the 6 values a neighbour needs per cell.
//  * PK = true: two triplets per register, one per 16-bit half, biased by 2^14 (engine.h's biased
//    packed mode; needs sigma'' >= 0). Real values lie above 2^14 - 8|gamma| (any cell is reached by
//    three gap runs, at most 6 openings, and one more move opens at most 2), -infinity is 4|gamma|,
//    so no add-max wraps below 0 and no sum carries out of a half; the host admits the mode when
//    both sides keep their distance.
//  * Measured (256 DNA triplets of 100..300 residues, 2.7e9 cells): the plane kernel 0.51 s
//    (5 GCUPS), this one 11.9 ms with one triplet per register and 6.3 ms (426 GCUPS) with two;
//    1,024 triplets 24.6 ms. 46 ALU-pipe instructions per two cells allow 846 GCUPS at 64 per SM
//    and clock; the step's other half is halo exchange, records and the adds. One triplet of 250
//    residues, bound by its chain of column tasks, takes 0.8 ms.
// affine_plane_kernel: the direct form, one CTA per triplet over anti-diagonal planes in global
// memory, for a triplet whose boundary records would not fit in memory.
#include <cuda_runtime.h>
#include <stdint.h>

#include "wavefront.cuh"

namespace trioseq {

namespace {

constexpr int kAffNeg = -(1 << 30);  // a state no prefix ends in
constexpr int kAffStates = kAffineStates;
constexpr int kAffStride = 16;       // int32 per cell in the plane buffers (13 used, 64 bytes)
constexpr int kAffThreads = 256;     // of affine_plane_kernel

// The 13 reachable states as kinds (pair 01, pair 02, pair 12); 0 both residues or none, 1 gap
// in the pair's first sequence, 2 gap in its second. Compile-time, so that with the loops over
// moves and states unrolled every state index and opening count folds to a constant and the 13
// values of a cell stay in registers.
__host__ __device__ constexpr int st_kind(int s, int pq) {
  constexpr int8_t t[kAffineStates][3] = {
      {0, 0, 0}, {0, 2, 2}, {2, 0, 1}, {1, 1, 0}, {2, 2, 0}, {2, 2, 1}, {2, 2, 2},
      {1, 0, 2}, {1, 1, 2}, {1, 2, 2}, {0, 1, 1}, {1, 1, 1}, {2, 1, 1}};
  return t[s][pq];
}

__host__ __device__ constexpr int st_index(int k01, int k02, int k12) {
  for (int s = 0; s < kAffineStates; ++s)
    if (st_kind(s, 0) == k01 && st_kind(s, 1) == k02 && st_kind(s, 2) == k12) return s;
  return 0;  // unreachable combinations never occur
}

// moves in Eq. 1's listing order: 111 110 101 011 100 010 001
__host__ __device__ constexpr int mv(int m, int q) {
  constexpr int8_t t[7][3] = {{1, 1, 1}, {1, 1, 0}, {1, 0, 1}, {0, 1, 1},
                              {1, 0, 0}, {0, 1, 0}, {0, 0, 1}};
  return t[m][q];
}

// kind a move gives the pair (p0, p1): 0 untouched (gap in both), 1 both residues, 2 gap in p0,
// 3 gap in p1
__host__ __device__ constexpr int move_kind(int m, int pq) {
  const int p0 = pq == 2 ? 1 : 0, p1 = pq == 0 ? 1 : 2;
  const int r0 = mv(m, p0), r1 = mv(m, p1);
  return (!r0 && !r1) ? 0 : ((r0 && r1) ? 1 : (r0 ? 3 : 2));
}

// new state and number of gap runs opened when move m follows state s
__host__ __device__ constexpr int next_state(int m, int s) {
  int k[3] = {0, 0, 0};
  for (int pq = 0; pq < 3; ++pq) {
    const int mk = move_kind(m, pq);
    k[pq] = mk == 0 ? st_kind(s, pq) : (mk == 1 ? 0 : mk - 1);
  }
  return st_index(k[0], k[1], k[2]);
}
__host__ __device__ constexpr int opens(int m, int s) {
  int n = 0;
  for (int pq = 0; pq < 3; ++pq) {
    const int mk = move_kind(m, pq);
    if (mk >= 2 && st_kind(s, pq) != mk - 1) ++n;
  }
  return n;
}

}  // namespace

__global__ void __launch_bounds__(kAffThreads) affine_plane_kernel(const AffinePlaneParams p) {
  __shared__ int sig[kMaxAlphabet * kMaxAlphabet];
  __shared__ int next;
  const int KP = p.KP;
  for (int e = threadIdx.x; e < KP * KP; e += blockDim.x) sig[e] = p.sub[e];
  int32_t* const base = p.planes + (int64_t)blockIdx.x * 4 * p.plane_cells * kAffStride;
  for (;;) {
    __syncthreads();
    if (threadIdx.x == 0) next = atomicAdd(p.queue, 1);
    __syncthreads();
    const int q = next;
    if (q >= p.n) return;
    const TripDesc& d = p.desc[p.tasks[q].trip];
    const int a = d.len[0], b = d.len[1], c = d.len[2];
    const int8_t* S0 = p.seq + d.s_off[0];
    const int8_t* S1 = p.seq + d.s_off[1];
    const int8_t* S2 = p.seq + d.s_off[2];
    const int C = c + 1;
    const int gap = p.gap, go = p.gap_open;
    // plane d lives in buffer d & 3; cell (j, k) at (j * C + k) * 16
    for (int dd = 0; dd <= a + b + c; ++dd) {
      int32_t* cur = base + (int64_t)(dd & 3) * p.plane_cells * kAffStride;
      const int jlo = max(0, dd - a - c), jhi = min(b, dd);
      const int64_t rows = jhi - jlo + 1;
      for (int64_t e = threadIdx.x; e < rows * C; e += blockDim.x) {
        const int j = jlo + (int)(e / C), k = (int)(e % C);
        const int i = dd - j - k;
        if (i < 0 || i > a) continue;
        int F[kAffStates];
#pragma unroll
        for (int s = 0; s < kAffStates; ++s) F[s] = kAffNeg;
        if (dd == 0) F[0] = 0;
        const int x = i > 0 ? (int)S0[i - 1] : 0, y = j > 0 ? (int)S1[j - 1] : 0,
                  z = k > 0 ? (int)S2[k - 1] : 0;
#pragma unroll
        for (int m = 0; m < 7; ++m) {
          const int di = mv(m, 0), dj = mv(m, 1), dk = mv(m, 2);
          if (dd == 0 || i < di || j < dj || k < dk) continue;
          const int4* G = reinterpret_cast<const int4*>(
              base + (int64_t)((dd - di - dj - dk) & 3) * p.plane_cells * kAffStride +
              ((int64_t)(j - dj) * C + (k - dk)) * kAffStride);
          const int4 g0 = G[0], g1 = G[1], g2 = G[2], g3 = G[3];
          const int g[16] = {g0.x, g0.y, g0.z, g0.w, g1.x, g1.y, g1.z, g1.w,
                             g2.x, g2.y, g2.z, g2.w, g3.x, g3.y, g3.z, g3.w};
          // the column's pair scores: sigma per residue pair, alpha per residue against a gap
          int fixed = 0;
          fixed += move_kind(m, 0) == 1 ? sig[x * KP + y] : (move_kind(m, 0) ? gap : 0);
          fixed += move_kind(m, 1) == 1 ? sig[x * KP + z] : (move_kind(m, 1) ? gap : 0);
          fixed += move_kind(m, 2) == 1 ? sig[y * KP + z] : (move_kind(m, 2) ? gap : 0);
#pragma unroll
          for (int s = 0; s < kAffStates; ++s) {
            const int ns = next_state(m, s);
            F[ns] = max(F[ns], g[s] + fixed + opens(m, s) * go);
          }
        }
        int4* out = reinterpret_cast<int4*>(cur + ((int64_t)j * C + k) * kAffStride);
        // a state no prefix ends in stays at the floor instead of drifting below it
        int v[16];
#pragma unroll
        for (int s = 0; s < 16; ++s) v[s] = s < kAffStates ? max(F[s], kAffNeg) : kAffNeg;
        out[0] = make_int4(v[0], v[1], v[2], v[3]);
        out[1] = make_int4(v[4], v[5], v[6], v[7]);
        out[2] = make_int4(v[8], v[9], v[10], v[11]);
        out[3] = make_int4(v[12], v[13], v[14], v[15]);
        if (i == a && j == b && k == c) {
          int best = F[0];
#pragma unroll
          for (int s = 1; s < kAffStates; ++s) best = max(best, F[s]);
          p.scores[d.out_idx] = best;
        }
      }
      __syncthreads();
    }
  }
}

// ---- the register-tiled wavefront ---------------------------------------------------------------

namespace {

constexpr int kAJ = 4, kAK = 4;                          // cells per lane
constexpr int kAWJ = kPR * kAJ, kAWK = kPC * kAK;        // cells per column task: 16 x 32
constexpr int kASegJ = 4 + 6 * kAK;   // j-record ints per lane column: corners, 6 values per cell
constexpr int kASegK = 6 * kAJ;       // k-record ints per lane row
constexpr int kASlot = kPC * kASegJ + kPR * kASegK;      // ints per ring slot
constexpr int kAPJ = kAWJ + 4, kAPK = kAWK + 4;          // padded profile rows
constexpr int kAPieces = kASlot / 4, kANPL = (kAPieces + 31) / 32;
static_assert(kAffineWJ == kAWJ && kAffineWK == kAWK, "the host cuts the plane the same way");
static_assert(kAffineRecJ == kPC * kASegJ && kAffineRecK == kPR * kASegK, "record strides");

template <bool PK>
__device__ __forceinline__ int mx2(int a, int b) {
  return PK ? (int)__vmaxu2((unsigned)a, (unsigned)b) : max(a, b);
}
template <bool PK>
__device__ __forceinline__ int mx3(int a, int b, int c) {
  return PK ? (int)__vimax3_u16x2((unsigned)a, (unsigned)b, (unsigned)c) : __vimax3_s32(a, b, c);
}
template <bool PK>  // max(a + g, c)
__device__ __forceinline__ int amx(int a, int g, int c) {
  return PK ? (int)__viaddmax_u16x2((unsigned)a, (unsigned)g, (unsigned)c)
            : __viaddmax_s32(a, g, c);
}

}  // namespace

template <bool PK>
__global__ void __launch_bounds__(kWarpsPerCta * 32, 2) affine_kernel(const AffineParams p) {
  extern __shared__ int4 smem4[];
  int* smem = reinterpret_cast<int*>(smem4);
  const int KP = p.KP, VIRT = KP - 1;
  const int sigN = (KP * KP + 3) & ~3;
  constexpr int NPROF = PK ? 2 : 1;
  int* sig = smem;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  int* profJ = smem + sigN + warp * (NPROF * KP * (kAPJ + kAPK) + kRing * kASlot);
  int* profK = profJ + KP * kAPJ;
  int* profJ1 = profK + KP * kAPK;  // packed: the high halves' triplet
  int* profK1 = profJ1 + KP * kAPJ;
  int* ring = profJ + NPROF * KP * (kAPJ + kAPK);
  for (int e = threadIdx.x; e < KP * KP; e += blockDim.x) sig[e] = p.sig[e];
  __syncthreads();
  const int r = lane >> 3, lc = lane & 7;
  const int NEG = p.neg, g1 = p.go1, g2 = p.go2;

  // staging pieces of this lane: 7 per lane column of the j-record, 6 per lane row of the k-record
  int cp_kind[kANPL], cp_delta[kANPL], cp_col[kANPL], cp_dst[kANPL];
#pragma unroll
  for (int m = 0; m < kANPL; ++m) {
    const int q = lane + 32 * m;
    constexpr int NJP = kPC * kASegJ / 4;
    cp_kind[m] = q < NJP ? 1 : (q < kAPieces ? 2 : 0);
    cp_delta[m] = q < NJP ? q / (kASegJ / 4) : (q - NJP) / (kASegK / 4);
    cp_col[m] = q < NJP ? 4 * q : 4 * (q - NJP);
    cp_dst[m] = 4 * q;
  }

  for (;;) {
    int task = 0;
    if (lane == 0) task = atomicAdd(p.queue, 1);
    task = __shfl_sync(kFull, task, 0);
    if (task >= p.ntasks) return;
    const Task tk = p.tasks[task];
    const TripDesc& d = p.desc[tk.trip];
    const TripDesc& d1 = PK ? p.desc[d.pair] : d;
    const int a = d.glen[0], b = d.glen[1], c = d.glen[2];
    const int a0 = d.len[0], b0 = d.len[1], c0 = d.len[2];
    const int a1 = d1.len[0], b1 = d1.len[1], c1 = d1.len[2];
    const int nJ = d.nJ, nK = d.nK, T = d.T;
    const int J = tk.J, K = tk.K;
    const int8_t* S0 = p.seq + d.s_off[0];
    const int8_t* S1 = p.seq + d.s_off[1];
    const int8_t* S2 = p.seq + d.s_off[2];
    const int8_t* T0 = p.seq + d1.s_off[0];
    const int8_t* T1 = p.seq + d1.s_off[1];
    const int8_t* T2 = p.seq + d1.s_off[2];
    const int j0 = J * kAWJ + r * kAJ, k0 = K * kAWK + lc * kAK;
    const int me = J * nK + K;

    // profiles of this block, as in wavefront_kernel (index 0 and beyond the end: VIRT)
    __syncwarp();
    for (int e = lane; e < KP * kAWJ; e += 32) {
      const int x = e / kAWJ, jl = e - x * kAWJ, j = J * kAWJ + jl;
      profJ[x * kAPJ + jl] = sig[x * KP + ((j >= 1 && j <= b0) ? (int)S1[j - 1] : VIRT)];
      if (PK) profJ1[x * kAPJ + jl] = sig[x * KP + ((j >= 1 && j <= b1) ? (int)T1[j - 1] : VIRT)];
    }
    for (int e = lane; e < KP * kAWK; e += 32) {
      const int x = e / kAWK, kl = e - x * kAWK, k = K * kAWK + kl;
      profK[x * kAPK + kl] = sig[x * KP + ((k >= 1 && k <= c0) ? (int)S2[k - 1] : VIRT)];
      if (PK) profK1[x * kAPK + kl] = sig[x * KP + ((k >= 1 && k <= c1) ? (int)T2[k - 1] : VIRT)];
    }
    int Cv[kAJ][kAK];
#pragma unroll
    for (int pp = 0; pp < kAJ; ++pp) {
      const int j = j0 + pp;
      const int yo = ((j >= 1 && j <= b0) ? (int)S1[j - 1] : VIRT) * KP;
      const int yo1 = PK ? ((j >= 1 && j <= b1) ? (int)T1[j - 1] : VIRT) * KP : 0;
#pragma unroll
      for (int qq = 0; qq < kAK; ++qq) {
        const int k = k0 + qq;
        Cv[pp][qq] = sig[yo + ((k >= 1 && k <= c0) ? (int)S2[k - 1] : VIRT)];
        if (PK)
          Cv[pp][qq] = (int)__byte_perm(
              Cv[pp][qq], sig[yo1 + ((k >= 1 && k <= c1) ? (int)T2[k - 1] : VIRT)], 0x5410);
      }
    }
    __syncwarp();

    // Owners of the final cells (of each half).
    const bool owns_end = J == b0 / kAWJ && K == c0 / kAWK && r == (b0 % kAWJ) / kAJ &&
                          lc == (c0 % kAWK) / kAK;
    const bool owns_end1 = PK && J == b1 / kAWJ && K == c1 / kAWK && r == (b1 % kAWJ) / kAJ &&
                           lc == (c1 % kAWK) / kAK;

    // Moves out of slice s - 1, per cell; the bottom row's and right column's moves within the
    // slice (for the lane below and the lane to the right); the halos of slice s - 1.
    int P111[kAJ][kAK], P110[kAJ][kAK], P101[kAJ][kAK], P100[3][kAJ][kAK];
    int bR011[kAK], bR010[3][kAK], rC011[kAJ], rC001[3][kAJ];
    int row111[kAK + 1], row110[kAK], col111[kAJ], col101[kAJ], cor011 = NEG;
#pragma unroll
    for (int pp = 0; pp < kAJ; ++pp) {
#pragma unroll
      for (int qq = 0; qq < kAK; ++qq) {
        P111[pp][qq] = P110[pp][qq] = P101[pp][qq] = NEG;
        P100[0][pp][qq] = P100[1][pp][qq] = P100[2][pp][qq] = NEG;
      }
      rC011[pp] = rC001[0][pp] = rC001[1][pp] = rC001[2][pp] = NEG;
      col111[pp] = col101[pp] = NEG;
    }
#pragma unroll
    for (int qq = 0; qq < kAK; ++qq) {
      bR011[qq] = bR010[0][qq] = bR010[1][qq] = bR010[2][qq] = NEG;
      row111[qq] = row110[qq] = NEG;
    }
    row111[kAK] = NEG;
    // the empty prefix: the move (1,1,1) out of cell (-1,-1,-1), value 0
    if (J == 0 && K == 0 && lane == 0) row111[0] = PK ? kBias16x2 : 0;

    const int64_t recJ = (int64_t)(a + 1) * kAffineRecJ, recK = (int64_t)(a + 1) * kAffineRecK;
    int* const faces = p.faces;
    const int* srcJ = faces + d.oj_off + (int64_t)(me - nK) * recJ;  // producer (J-1, K)
    const int* srcK = faces + d.ok_off + (int64_t)(me - 1) * recK;   // producer (J, K-1)
    int* dstJ = faces + d.oj_off + (int64_t)me * recJ + lc * kASegJ;
    int* dstK = faces + d.ok_off + (int64_t)me * recK + r * kASegK;
    const bool out_j = r == kPR - 1 && J + 1 < nJ, out_k = lc == kPC - 1 && K + 1 < nK;
    const int* progJ = p.progress + d.prog_base + (me - nK);
    const int* progK = p.progress + d.prog_base + (me - 1);
    int* progMe = p.progress + d.prog_base + me;
    int cachedJ = J > 0 ? 0 : 1 << 30, cachedK = K > 0 ? 0 : 1 << 30;  // warp-uniform
    bool ok = true;

    // Staging as in the score kernels: pieces loaded two steps ahead, parked one step ahead,
    // producers checked once per pair of steps.
    int4 pf[kANPL];
    int pf_u = -1;
    auto fetch = [&](int u, bool chk) {
      const int needJ = min(u + 1 + kPR, T), needK = min(u + 1 + kPC, T);
      if (chk && (cachedJ < needJ || cachedK < needK)) {  // warp-uniform
        bool okl = true;
        int cj = cachedJ, ck = cachedK;
        if (lane == 0) {
          if (cj < needJ) okl = wait_flag(progJ, needJ, &cj, p.wait_ns);
          if (okl && ck < needK) okl = wait_flag(progK, needK, &ck, p.wait_ns);
        }
        ok = __shfl_sync(kFull, okl, 0);
        cachedJ = __shfl_sync(kFull, cj, 0);
        cachedK = __shfl_sync(kFull, ck, 0);
        __syncwarp();
      }
      pf_u = u;
#pragma unroll
      for (int m = 0; m < kANPL; ++m) {
        const int sl = u - cp_delta[m];
        const bool have = ok && cp_kind[m] != 0 && sl >= 0 && sl <= a &&
                          (cp_kind[m] == 1 ? J > 0 : K > 0);
        const int* src = cp_kind[m] == 1 ? srcJ + (int64_t)sl * kAffineRecJ + cp_col[m]
                                         : srcK + (int64_t)sl * kAffineRecK + cp_col[m];
        pf[m] = ld_cg_if(reinterpret_cast<const int4*>(src), have, NEG);
      }
    };
    auto park = [&]() {
#pragma unroll
      for (int m = 0; m < kANPL; ++m)
        st_shared_if(reinterpret_cast<int4*>(ring + (pf_u & (kRing - 1)) * kASlot + cp_dst[m]),
                     pf[m], cp_kind[m] != 0);
    };
    fetch(0, true);
    park();
    fetch(1, false);
    // residues of S0 by slice, as in wavefront_kernel; packed: bits 0-7 and 8-15
    auto xblock = [&](int base) -> int {
      const int sl = base + lane;
      const int x0 = (sl >= 1 && sl <= a0) ? (int)__ldg(S0 + sl - 1) : VIRT;
      if (!PK) return x0;
      const int x1 = (sl >= 1 && sl <= a1) ? (int)__ldg(T0 + sl - 1) : VIRT;
      return x0 | (x1 << 8);
    };
    int xprev = PK ? (VIRT | (VIRT << 8)) : VIRT, xcur = xblock(0), xnext = xblock(32);

    int pub_in = p.TI;
    for (int t = 0; t < T; ++t) {
      const int s = t - r - lc;
      park();
      if (t + 2 < T) fetch(t + 2, (t & 1) == 0);
      if (!ok) break;
      if ((t & 31) == 0 && t > 0) {
        xprev = xcur;
        xcur = xnext;
        xnext = xblock(t + 32);
      }
      const int xa = __shfl_sync(kFull, xcur, s & 31);
      const int xb = __shfl_sync(kFull, xprev, s & 31);
      const int x = (s >= (t & ~31)) ? xa : xb;
      __syncwarp();
      // Halo of slice s: from the lane above and the lane to the left (their previous step), or
      // the staged records in the first lane row and column.
      int nrow111[kAK + 1], nrow110[kAK], row011[kAK + 1], row010[3][kAK];
      int ncol111[kAJ], ncol101[kAJ], col011[kAJ], col001[3][kAJ];
      {
        const int* sl = ring + (t & (kRing - 1)) * kASlot;
        const int4* rs = reinterpret_cast<const int4*>(sl + lc * kASegJ);
        const int4* cs = reinterpret_cast<const int4*>(sl + kPC * kASegJ + r * kASegK);
        const int4 e0 = rs[0];
        const bool top = r == 0, left = lc == 0;
        const int u0 = __shfl_up_sync(kFull, col111[kAJ - 1], kPC);
        const int u1 = __shfl_up_sync(kFull, cor011, kPC);
        nrow111[0] = top ? e0.x : u0;
        row011[0] = top ? e0.y : u1;
        const auto up4 = [&](const int4& e, const int (&src)[kAK], int* dst) {
          const int ev[4] = {e.x, e.y, e.z, e.w};
#pragma unroll
          for (int qq = 0; qq < kAK; ++qq) {
            const int v = __shfl_up_sync(kFull, src[qq], kPC);
            dst[qq] = top ? ev[qq] : v;
          }
        };
        up4(rs[1], P111[kAJ - 1], nrow111 + 1);
        up4(rs[2], P110[kAJ - 1], nrow110);
        up4(rs[3], bR011, row011 + 1);
#pragma unroll
        for (int h = 0; h < 3; ++h) up4(rs[4 + h], bR010[h], row010[h]);
        const auto left4 = [&](const int4& e, int s0, int s1, int s2, int s3, int* dst) {
          const int ev[4] = {e.x, e.y, e.z, e.w}, sv[4] = {s0, s1, s2, s3};
#pragma unroll
          for (int pp = 0; pp < kAJ; ++pp) {
            const int v = __shfl_up_sync(kFull, sv[pp], 1);
            dst[pp] = left ? ev[pp] : v;
          }
        };
        constexpr int e = kAK - 1;
        left4(cs[0], P111[0][e], P111[1][e], P111[2][e], P111[3][e], ncol111);
        left4(cs[1], P101[0][e], P101[1][e], P101[2][e], P101[3][e], ncol101);
        left4(cs[2], rC011[0], rC011[1], rC011[2], rC011[3], col011);
#pragma unroll
        for (int h = 0; h < 3; ++h)
          left4(cs[3 + h], rC001[h][0], rC001[h][1], rC001[h][2], rC001[h][3], col001[h]);
      }
      const bool active = s >= 0 && s <= a;
      if (active) {
        int A[kAJ], B[kAK];
        {
          const int xl = PK ? (x & 0xff) : x;
          const int4 va = *reinterpret_cast<const int4*>(profJ + xl * kAPJ + r * kAJ);
          const int4 vb = *reinterpret_cast<const int4*>(profK + xl * kAPK + lc * kAK);
          A[0] = va.x; A[1] = va.y; A[2] = va.z; A[3] = va.w;
          B[0] = vb.x; B[1] = vb.y; B[2] = vb.z; B[3] = vb.w;
          if (PK) {
            const int xh = x >> 8;
            const int4 wa = *reinterpret_cast<const int4*>(profJ1 + xh * kAPJ + r * kAJ);
            const int4 wb = *reinterpret_cast<const int4*>(profK1 + xh * kAPK + lc * kAK);
            const int ha[4] = {wa.x, wa.y, wa.z, wa.w}, hb[4] = {wb.x, wb.y, wb.z, wb.w};
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              A[e] = (int)__byte_perm(A[e], ha[e], 0x5410);
              B[e] = (int)__byte_perm(B[e], hb[e], 0x5410);
            }
          }
        }
        // Pass 1, backwards in place: states s, a and b of slice s from the moves out of slice
        // s - 1 (x0..x2 stay where they are: the single-residue move costs 0). The adds are
        // multiply-adds by a runtime 1, on the FMA pipe.
#pragma unroll
        for (int pp = kAJ - 1; pp >= 0; --pp)
#pragma unroll
          for (int qq = kAK - 1; qq >= 0; --qq) {
            const int f111 =
                pp == 0 ? row111[qq] : (qq == 0 ? col111[pp - 1] : P111[pp - 1][qq - 1]);
            const int f110 = pp == 0 ? row110[qq] : P110[pp - 1][qq];
            const int f101 = qq == 0 ? col101[pp] : P101[pp][qq - 1];
            P111[pp][qq] = mad_lo(Cv[pp][qq], p.one,
                                  mad_lo(B[qq], p.one, mad_lo(A[pp], p.one, f111)));
            P110[pp][qq] = mad_lo(A[pp], p.one, f110);
            P101[pp][qq] = mad_lo(B[qq], p.one, f101);
          }
        // Pass 2, forwards: states c, y and z from the moves within the slice, then the 13
        // outgoing values.
#pragma unroll
        for (int qq = 0; qq < kAK; ++qq) {
          bR011[qq] = row011[qq + 1];
#pragma unroll
          for (int h = 0; h < 3; ++h) bR010[h][qq] = row010[h][qq];
        }
#pragma unroll
        for (int pp = 0; pp < kAJ; ++pp) {
          int dg = pp == 0 ? row011[0] : col011[pp - 1];
          int z0 = col001[0][pp], z1 = col001[1][pp], z2 = col001[2][pp];
#pragma unroll
          for (int qq = 0; qq < kAK; ++qq) {
            const int fs = P111[pp][qq], fa = P110[pp][qq], fb = P101[pp][qq];
            const int fc = mad_lo(Cv[pp][qq], p.one, dg);
            const int x0 = P100[0][pp][qq], x1 = P100[1][pp][qq], x2 = P100[2][pp][qq];
            const int y0 = bR010[0][qq], y1 = bR010[1][qq], y2 = bR010[2][qq];
            dg = bR011[qq];  // the diagonal of the next column
            // groups of states by the openings each move adds (0, 1 or 2)
            const int sc = mx2<PK>(fs, fc), sb = mx2<PK>(fs, fb), sa = mx2<PK>(fs, fa);
            const int bz2 = mx2<PK>(fb, z2), z01 = mx2<PK>(z0, z1), ay2 = mx2<PK>(fa, y2);
            const int y01 = mx2<PK>(y0, y1), cz1 = mx2<PK>(fc, z1), z02 = mx2<PK>(z0, z2);
            const int ax2 = mx2<PK>(fa, x2), x01 = mx2<PK>(x0, x1), cy1 = mx2<PK>(fc, y1);
            const int y02 = mx2<PK>(y0, y2), bx1 = mx2<PK>(fb, x1), x02 = mx2<PK>(x0, x2);
            const int n110 = mx3<PK>(sc, bz2, z01), o110 = mx2<PK>(x01, y01),
                      t110 = mx2<PK>(ax2, y2);
            const int n101 = mx3<PK>(sc, ay2, y01), o101 = mx2<PK>(x02, z01),
                      t101 = mx2<PK>(bx1, z2);
            const int n011 = mx3<PK>(sb, ax2, x01), o011 = mx2<PK>(y02, z02),
                      t011 = mx2<PK>(cy1, z1);
            P111[pp][qq] = mx3<PK>(n110, o110, t110);
            P110[pp][qq] = amx<PK>(n110, g2, amx<PK>(o110, g1, t110));
            P101[pp][qq] = amx<PK>(n101, g2, amx<PK>(o101, g1, t101));
            bR011[qq] = amx<PK>(n011, g2, amx<PK>(o011, g1, t011));
            P100[0][pp][qq] = amx<PK>(sc, g2, x0);
            P100[1][pp][qq] = amx<PK>(z01, g2, amx<PK>(bz2, g1, x1));
            P100[2][pp][qq] = amx<PK>(y01, g2, amx<PK>(ay2, g1, x2));
            bR010[0][qq] = amx<PK>(sb, g2, y0);
            bR010[1][qq] = amx<PK>(z02, g2, amx<PK>(cz1, g1, y1));
            bR010[2][qq] = amx<PK>(x01, g2, amx<PK>(ax2, g1, y2));
            z0 = amx<PK>(sa, g2, z0);
            const int w1 = amx<PK>(y02, g2, amx<PK>(cy1, g1, z1));
            const int w2 = amx<PK>(x02, g2, amx<PK>(bx1, g1, z2));
            z1 = w1;
            z2 = w2;
          }
          rC011[pp] = bR011[kAK - 1];
          rC001[0][pp] = z0;
          rC001[1][pp] = z1;
          rC001[2][pp] = z2;
        }
      }
      // progress t (steps < t computed and stored), between compute and stores
      if (--pub_in == 0) {
        pub_in = p.TI;
        __syncwarp();
        if (lane == 0) st_release(progMe, t);
      }
      if (active) {
        {
          int4* q4 = reinterpret_cast<int4*>(dstJ + (int64_t)s * kAffineRecJ);
          constexpr int e = kAJ - 1;
          st_global_if(q4, make_int4(ncol111[e], col011[e], NEG, NEG), out_j);  // corners
          st_global_if(q4 + 1, make_int4(P111[e][0], P111[e][1], P111[e][2], P111[e][3]), out_j);
          st_global_if(q4 + 2, make_int4(P110[e][0], P110[e][1], P110[e][2], P110[e][3]), out_j);
          st_global_if(q4 + 3, make_int4(bR011[0], bR011[1], bR011[2], bR011[3]), out_j);
#pragma unroll
          for (int h = 0; h < 3; ++h)
            st_global_if(q4 + 4 + h,
                         make_int4(bR010[h][0], bR010[h][1], bR010[h][2], bR010[h][3]), out_j);
        }
        {
          int4* q4 = reinterpret_cast<int4*>(dstK + (int64_t)s * kAffineRecK);
          constexpr int e = kAK - 1;
          st_global_if(q4, make_int4(P111[0][e], P111[1][e], P111[2][e], P111[3][e]), out_k);
          st_global_if(q4 + 1, make_int4(P101[0][e], P101[1][e], P101[2][e], P101[3][e]), out_k);
          st_global_if(q4 + 2, make_int4(rC011[0], rC011[1], rC011[2], rC011[3]), out_k);
#pragma unroll
          for (int h = 0; h < 3; ++h)
            st_global_if(q4 + 3 + h,
                         make_int4(rC001[h][0], rC001[h][1], rC001[h][2], rC001[h][3]), out_k);
        }
        // The best over the end cell's states is its (1,1,1) value: that move opens nothing.
        if ((owns_end && s == a0) || (owns_end1 && s == a1)) {
          int v0 = 0, v1 = 0;
#pragma unroll
          for (int pp = 0; pp < kAJ; ++pp)
#pragma unroll
            for (int qq = 0; qq < kAK; ++qq) {
              if (pp == b0 % kAJ && qq == c0 % kAK) v0 = P111[pp][qq];
              if (PK && pp == b1 % kAJ && qq == c1 % kAK) v1 = P111[pp][qq];
            }
          if (owns_end && s == a0)
            p.scores[d.out_idx] = (PK ? (v0 & 0xffff) - (1 << 14) : v0) + d.score_base;
          if (owns_end1 && s == a1)
            p.scores[d1.out_idx] = (int)((unsigned)v1 >> 16) - (1 << 14) + d1.score_base;
        }
      }
      // slice s becomes the previous slice
#pragma unroll
      for (int qq = 0; qq <= kAK; ++qq) row111[qq] = nrow111[qq];
#pragma unroll
      for (int qq = 0; qq < kAK; ++qq) row110[qq] = nrow110[qq];
#pragma unroll
      for (int pp = 0; pp < kAJ; ++pp) {
        col111[pp] = ncol111[pp];
        col101[pp] = ncol101[pp];
      }
      cor011 = col011[kAJ - 1];
    }
    __syncwarp();
    if (ok && lane == 0) st_release(progMe, T);
    if (!ok) {
      if (lane == 0) atomicOr(p.err, 1);
      return;
    }
  }
}

size_t affine_smem_bytes(int KP, bool pk) {
  const size_t sigN = (size_t)((KP * KP + 3) & ~3);
  return (sigN + (size_t)kWarpsPerCta *
                     ((pk ? 2 : 1) * KP * (kAPJ + kAPK) + kRing * kASlot)) * sizeof(int);
}

namespace {
const void* affine_ptr(bool pk) {
  return pk ? reinterpret_cast<const void*>(&affine_kernel<true>)
            : reinterpret_cast<const void*>(&affine_kernel<false>);
}
}  // namespace

int affine_occupancy(bool pk, size_t smem, int* blocks_per_sm) {
  const void* k = affine_ptr(pk);
  if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) !=
      cudaSuccess)
    return -2;
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, k, kWarpsPerCta * 32,
                                                       smem) == cudaSuccess
             ? 0
             : -2;
}

int launch_affine(bool pk, const AffineParams& p, int grid, size_t smem, void* stream) {
  void* args[] = {const_cast<AffineParams*>(&p)};
  return cudaLaunchKernel(affine_ptr(pk), dim3(grid), dim3(kWarpsPerCta * 32), args, smem,
                          (cudaStream_t)stream) == cudaSuccess
             ? 0
             : -2;
}

int affine_plane_occupancy(int* blocks_per_sm) {
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, affine_plane_kernel,
                                                       kAffThreads, 0) == cudaSuccess
             ? 0
             : -2;
}

int launch_affine_plane(const AffinePlaneParams& p, int grid, void* stream) {
  affine_plane_kernel<<<grid, kAffThreads, 0, (cudaStream_t)stream>>>(p);
  return cudaGetLastError() == cudaSuccess ? 0 : -2;
}

}  // namespace trioseq
