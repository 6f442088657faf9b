// wavefront_vp.cuh — wavefront kernel with two triplets per register (global type, score only), for
// scoring schemes whose sigma'' are all >= 0.
//
// wavefront_vp_kernel<NJ, NK>: a column task of 4 NJ x 8 NK cells serves a pair of triplets on the grid of
// their maximal lengths, the first in the low 16-bit halves of every register, the second in the high
// ones. Lanes, tiles and the step order are those of wavefront.cuh (lane (r, lc) computes slice
// s = t - r - lc at step t); arithmetic, staging and hand-off those of wavefront_vl.cuh:
//  * A half holds M' + 2^14 with -infinity = 0; the host admits a pair only if max sigma'' times the
//    pair's lengths stays below 2^14, so every half stays in 0 .. 2^15 and a plain 32-bit add is the two
//    16-bit adds. Values are absolute: no base, and a staged word needs no conversion.
//  * A record row is the packed words of one producer step: 8 x (NK words), 8 corners, and 4 x NJ column
//    words. What block (J+1, K) needs at its step u, lanes (3, lc) of block (J, K) hold at step u + 3; what
//    block (J, K+1) needs, lanes (r, 7) hold at step u + 7. No packed word equals kVlSentinel, so each
//    word is its own readiness flag.
//  * The shorter triplet of a pair goes on with virtual residues (sigma'' = 0). The task that owns an end cell leaves the steps without end-cell
//    work at the shorter one's last slice.
// Measured, kernel time against the int32-record form of wavefront_kernel that took these batches before
// (progress counts, 32 x 64 tasks, four-warp CTAs): 4,096 DNA triplets of 100..300 residues 12.74 -> 11.2 ms
// (3,790 GCUPS). What bounds it is issue, operand reads and the waits of two warps per sub-partition (its
// registers allow no third; held to 168, for three, the large batch takes 10.8 ms, but ten triplets of
// 300..600 residues 0.70 instead of 0.57 ms). A step of 32 x 32 x 2 cells takes ~270 instructions. Halos through
// shared memory instead of shuffles and selects: 6% fewer instructions, but waits on more scoreboards, 13.7 ms.
#pragma once
#include "wavefront_vl.cuh"

namespace trioseq {

constexpr int kVpRing = 64;  // slices in the residue ring

template <int NJ, int NK>
struct VpGeom {
  static constexpr int WJ = kPR * NJ, WK = kPC * NK;
  static constexpr int RJ = vp_rec_j(NK), RK = vp_rec_k(NJ);  // record row strides (ints)
  // ring slot: row words [lane column][NK], corners [lane column], column words [lane row][NJ]
  static constexpr int RC = kPC * NK, RQ = RC + kPC, SLOT = RQ + kPR * NJ;
  static constexpr int NV = NJ > NK ? NJ : NK;  // words of the larger staged piece
};

// One-warp CTAs, as many per SM as their registers allow (wavefront_vl.cuh, VlLaunch).
template <int NJ, int NK>
struct VpLaunch {
  static constexpr int blocks = NJ * NK >= 64 ? 8 : (NJ * NK >= 32 ? 10 : 14);
  static constexpr int regs = 65536 / (32 * blocks) / 8 * 8;
  static constexpr int max_regs = regs > 255 ? 255 : regs;
};

// J profiles repeated per lane column ([x][lane row][lane column]) keep the eight lanes of a 16-byte load
// phase on distinct bank groups; alphabets whose repeated profiles would take residency from the SM
// (more than 28 KB a warp) read one copy per lane row.
__host__ __device__ constexpr bool vp_repeat(int KP) { return KP <= 16; }

template <int NJ, int NK>
__global__ void __launch_bounds__(32) __maxnreg__((VpLaunch<NJ, NK>::max_regs))
    wavefront_vp_kernel(const WaveParams p) {
  using G = VpGeom<NJ, NK>;
  static_assert((NJ == 4 || NJ == 8) && (NK == 4 || NK == 8), "tile sides");
  constexpr int WJ = G::WJ, WK = G::WK, NV = G::NV;
  extern __shared__ int4 smem4[];
  int* smem = reinterpret_cast<int*>(smem4);
  const int KP = p.KP, VIRT = KP - 1;
  const int sigN = (KP * KP + 3) & ~3;
  int* sig = smem;
  // opaque, so that the lane's indices stay in registers instead of being formed again in every step
  int lane = threadIdx.x & 31, r = lane >> 3, lc = lane & 7;
  asm volatile("" : "+r"(lane), "+r"(r), "+r"(lc));
  // 16-bit profiles of both triplets, then the staging ring (four slots)
  const int rep = vp_repeat(KP) ? kPC : 1;
  const int nPJ = KP * kPR * rep * NJ, nPK = KP * kPC * NK;  // halves per triplet
  unsigned short* profJ = reinterpret_cast<unsigned short*>(smem + sigN);  // [triplet]
  unsigned short* profK = profJ + 2 * nPJ;
  int* ring = smem + sigN + nPJ + nPK;
  int2* xr = reinterpret_cast<int2*>(ring + kRing * G::SLOT);
  const int sJ = kPR * rep * NJ;
  constexpr int sK = kPC * NK;
  const unsigned short* pJ = profJ + (vp_repeat(KP) ? lane : r) * NJ;
  const unsigned short* pK = profK + lc * NK;
  for (int e = lane; e < KP * KP; e += 32) sig[e] = p.sig[e];
  __syncwarp();

  // Staging items, one per lane of each half warp (wavefront_vl.cuh): e0 < 8 the row words and corner of a
  // lane column, 8..11 the column words of a lane row; g = 0 stages an even step, g = 1 the next one.
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
    const TripDesc& d1 = p.desc[d.pair];  // triplet of the high halves
    const int a = d.glen[0];
    const int a0 = d.len[0], b0 = d.len[1], c0 = d.len[2];
    const int a1 = d1.len[0], b1 = d1.len[1], c1 = d1.len[2];
    const int nJ = d.nJ, nK = d.nK, T = d.T;
    const int J = tk.J, K = tk.K;
    const int8_t* S0 = p.seq + d.s_off[0];
    const int8_t* T0 = p.seq + d1.s_off[0];
    const int j0 = J * WJ + r * NJ, k0 = K * WK + lc * NK;
    // records exist where there is a consumer: j-rows of all but the last block row, k-rows of all but the
    // last block column
    const int me = J * nK + K, mek = J * (nK - 1) + K;

    // Profiles of this block for both triplets: sigma''(x, y_j) and sigma''(x, z_k); residue index 0 and
    // beyond the end are VIRT.
    __syncwarp();
#pragma unroll 1
    for (int h = 0; h < 2; ++h) {
      const int8_t* S1 = p.seq + (h ? d1.s_off[1] : d.s_off[1]);
      const int8_t* S2 = p.seq + (h ? d1.s_off[2] : d.s_off[2]);
      const int bh = h ? b1 : b0, ch = h ? c1 : c0;
      for (int jl = lane; jl < WJ; jl += 32) {
        const int j = J * WJ + jl, rr = jl / NJ, pq = jl % NJ;
        const int y = (j >= 1 && j <= bh) ? (int)S1[j - 1] : VIRT;
        for (int x = 0; x < KP; ++x) {
          const unsigned short v16 = (unsigned short)sig[x * KP + y];
          for (int l = 0; l < rep; ++l)
            profJ[h * nPJ + ((x * kPR + rr) * rep + l) * NJ + pq] = v16;
        }
      }
      for (int kl = lane; kl < WK; kl += 32) {
        const int k = K * WK + kl;
        const int z = (k >= 1 && k <= ch) ? (int)S2[k - 1] : VIRT;
        for (int x = 0; x < KP; ++x)
          profK[h * nPK + x * sK + kl] = (unsigned short)sig[x * KP + z];
      }
    }
    // sigma''(y_j, z_k) of both triplets, packed, for the whole task
    int Cv[NJ][NK];
    {
      const int8_t* S1 = p.seq + d.s_off[1];
      const int8_t* S2 = p.seq + d.s_off[2];
      const int8_t* T1 = p.seq + d1.s_off[1];
      const int8_t* T2 = p.seq + d1.s_off[2];
      int y0[NJ], y1[NJ];
#pragma unroll
      for (int pp = 0; pp < NJ; ++pp) {
        const int j = j0 + pp;
        y0[pp] = ((j >= 1 && j <= b0) ? (int)S1[j - 1] : VIRT) * KP;
        y1[pp] = ((j >= 1 && j <= b1) ? (int)T1[j - 1] : VIRT) * KP;
      }
#pragma unroll
      for (int qq = 0; qq < NK; ++qq) {
        const int k = k0 + qq;
        const int z0 = (k >= 1 && k <= c0) ? (int)S2[k - 1] : VIRT;
        const int z1 = (k >= 1 && k <= c1) ? (int)T2[k - 1] : VIRT;
#pragma unroll
        for (int pp = 0; pp < NJ; ++pp)
          Cv[pp][qq] = (int)__byte_perm(sig[y0[pp] + z0], sig[y1[pp] + z1], 0x5410);
      }
    }
    __syncwarp();

    // Owners of the final cells of both triplets; the task that holds one leaves the unchecked steps
    // before the shorter one's last slice.
    const bool end0 = J == b0 / WJ && K == c0 / WK, end1 = J == b1 / WJ && K == c1 / WK;
    const bool owns0 = end0 && r == (b0 % WJ) / NJ && lc == (c0 % WK) / NK;
    const bool owns1 = end1 && r == (b1 % WJ) / NJ && lc == (c1 % WK) / NK;
    const int end_p0 = b0 % NJ, end_q0 = c0 % NK, end_p1 = b1 % NJ, end_q1 = c1 % NK;
    const int lim = end0 || end1 ? min(a0, a1) : a;

    int P[NJ][NK];
    int rowA[NK + 1], colA[NJ], rowB[NK + 1], colB[NJ];
#pragma unroll
    for (int pp = 0; pp < NJ; ++pp) {
#pragma unroll
      for (int qq = 0; qq < NK; ++qq) P[pp][qq] = 0;
      colA[pp] = colB[pp] = 0;
    }
#pragma unroll
    for (int qq = 0; qq <= NK; ++qq) rowA[qq] = rowB[qq] = 0;

    // Records: producer (J-1, K) of row items and (J, K-1) of column items; at step u an item comes from
    // producer row u + kPR - 1 or u + kPC - 1.
    const bool has_j = J > 0, has_k = K > 0, has_any = has_j || has_k;
    const int it_e = has_j ? (has_k ? (e0 < kPC + kPR ? e0 : e0 - kPC - kPR) : e0 % kPC)
                           : kPC + e0 % kPR;
    const bool is_j = it_e < kPC, own = it_e == e0;
    const int it_l = is_j ? it_e : it_e - kPC;  // lane column or lane row
    const int it_delta = it_l - g;              // the item's slice in pair u is u - delta
    const int it_off = it_l * (is_j ? NK : NJ);
    const int it_hi = it_off + ((is_j ? NK : NJ) == 8 ? 4 : 0);
    const int it_off2 = is_j ? kPC * NK + it_l : it_off;
    const int f_j = vl_flag(has_j && own && is_j), f_k = vl_flag(has_k && own && !is_j);
    const unsigned st_w = ring_s + 4 * (g * G::SLOT + (is_j ? it_l * NK : G::RQ + it_l * NJ));
    const unsigned st_c = ring_s + 4 * (g * G::SLOT + G::RC + it_l);
    const int it_stride = is_j ? G::RJ : G::RK;
    const int* it_src =
        p.faces + (is_j ? d.oj_off + ((int64_t)(me - nK) * T + (kPR - 1) + g) * G::RJ
                        : d.ok_off + ((int64_t)(mek - 1) * T + (kPC - 1) + g) * G::RK);
    const int f_oj = vl_flag(r == kPR - 1 && J + 1 < nJ), f_ok = vl_flag(lc == kPC - 1 && K + 1 < nK);
    int* dstJ = p.faces + d.oj_off + (int64_t)me * T * G::RJ + lc * NK;
    int* dstK = p.faces + d.ok_off + (int64_t)mek * T * G::RK + r * NJ;
    bool ok = true;
    // Without a producer the halo of the first lane row or column stays -infinity.
    for (int e = lane; e < kRing * G::SLOT; e += 32) ring[e] = 0;
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

    // A piece: the words and corner of one item in pair u (steps u and u + 1, u even); outside the cube it
    // holds -infinity.
    int pv[NV], px = 0;
#pragma unroll
    for (int e = 0; e < NV; ++e) pv[e] = 0;
    const auto load = [&](int u) {
      const int* src = it_src + (int64_t)u * it_stride;
      vl_load4(src + it_off, pv);
      if (NV == 8) vl_load4(src + it_hi, pv + NV - 4);
      asm volatile("ld.relaxed.gpu.global.s32 %0, [%1];" : "=r"(px) : "l"(src + it_off2) : "memory");
    };
    // `inner`: every lane's slice of both steps lies in the cube.
    const auto fetch = [&](int u, bool inner) {
      if (!has_any) return;
      const int sl = u - it_delta;
      if (inner) {
        load(u);
      } else {
#pragma unroll
        for (int e = 0; e < NV; ++e) pv[e] = 0;
        px = 0;
        if (sl >= 0 && sl <= a) load(u);
      }
    };
    // Reload the piece of pair u until none of its words is the sentinel (bounded).
    const auto resolve = [&](int u) {
      const auto missing = [&]() {
        unsigned m = (unsigned)px;
#pragma unroll
        for (int e = 0; e < NV; e += 2) m = __vimax3_u32(m, (unsigned)pv[e], (unsigned)pv[e + 1]);
        return m == (unsigned)kVlSentinel;
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
    if (ok) {
      fetch(0, false);
      resolve(0);
    }
    // M'[-1][-1][-1] = 0 feeds the origin through the (1,1,1) move (lane 0).
    if (J == 0 && K == 0 && lane == 0) rowB[0] = kBias16x2;

    // Residues of both triplets by slice, VIRT outside theirs, in a shared ring of two blocks of 32 slices
    // (block n covers slices 32n .. 32n + 31): stored in the middle of the block before, when the block they
    // replace is behind every lane, and loaded 32 steps earlier still. (A global load per step shares its
    // scoreboard with the record loads, so each step waited for those: 15.5 -> 11.0 ms on 4,096 triplets of
    // 100..300 residues.)
    const auto xblock = [&](int base) -> int {
      const int sl = base + lane;
      const int xa = (unsigned)(sl - 1) < (unsigned)a0 ? (int)__ldg(S0 + sl - 1) : VIRT;
      const int xb = (unsigned)(sl - 1) < (unsigned)a1 ? (int)__ldg(T0 + sl - 1) : VIRT;
      return xa | (xb << 8);
    };
    const auto xstore = [&](int base, int x) {
      xr[(base + lane) & (kVpRing - 1)] = make_int2(x & 0xff, x >> 8);
    };
    int xnext = xblock(32);
    xstore(0, xblock(0));
    xstore(32, VIRT | (VIRT << 8));  // the slices before 0
    __syncwarp();
    const auto refill = [&](const int t) {
      if ((t & 31) == 16) {
        xstore(t + 16, xnext);
        xnext = xblock(t + 48);
      }
    };
    int2 xs = xr[-(r + lc) & (kVpRing - 1)];  // residues of slice s, read in the step before

    // Stage the piece of pair t in ring slots `slot` and `slot` + 1, and load that of pair t + 2 in its place.
    const auto stage = [&](const int t, const bool inner, const int slot) -> bool {
      resolve(t);
      if (!ok) return false;
      const unsigned o = 4 * slot * G::SLOT;
#pragma unroll
      for (int e = 0; e < NK; e += 4)
        st_ring_row(st_w + o + 4 * e, pv[e], pv[e + 1], pv[e + 2], pv[e + 3], f_j);
      st_ring_corner(st_c + o, px, f_j);
#pragma unroll
      for (int e = 0; e < NJ; e += 4)
        st_ring_row(st_w + o + 4 * e, pv[e], pv[e + 1], pv[e + 2], pv[e + 3], f_k);
      if (inner || t + 2 < T) fetch(t + 2, inner);
      __syncwarp();
      return true;
    };
    // One step: the halo of slice s goes into rowCur / colCur, slice s - 1 is in rowPrev / colPrev.
    // inner: every lane has 0 <= s, and s is below every last slice that matters to this task.
    const auto step = [&](const int t, const bool inner, const int slot, int (&rowCur)[NK + 1],
                          const int (&rowPrev)[NK + 1], int (&colCur)[NJ], const int (&colPrev)[NJ]) {
      const int s = t - r - lc;
      int A[NJ], Bq[NK];
      unsigned wj0[NJ / 2], wj1[NJ / 2], wk0[NK / 2], wk1[NK / 2];
      ld_halves<NJ>(pJ + xs.x * sJ, wj0);
      ld_halves<NJ>(pJ + nPJ + xs.y * sJ, wj1);
      ld_halves<NK>(pK + xs.x * sK, wk0);
      ld_halves<NK>(pK + nPK + xs.y * sK, wk1);
#pragma unroll
      for (int w = 0; w < NJ / 2; ++w) {
        A[2 * w] = (int)__byte_perm(wj0[w], wj1[w], 0x5410);
        A[2 * w + 1] = (int)__byte_perm(wj0[w], wj1[w], 0x7632);
      }
#pragma unroll
      for (int w = 0; w < NK / 2; ++w) {
        Bq[2 * w] = (int)__byte_perm(wk0[w], wk1[w], 0x5410);
        Bq[2 * w + 1] = (int)__byte_perm(wk0[w], wk1[w], 0x7632);
      }
      xs = xr[(s + 1) & (kVpRing - 1)];
      // Halo of slice s from the neighbour lanes' previous step; the edge lanes take the staged words.
#pragma unroll
      for (int qq = 0; qq <= NK; ++qq)
        rowCur[qq] = __shfl_up_sync(kFull, qq == 0 ? colPrev[NJ - 1] : P[NJ - 1][qq - 1], kPC);
#pragma unroll
      for (int pp = 0; pp < NJ; ++pp) colCur[pp] = __shfl_up_sync(kFull, P[pp][NK - 1], 1);
      {
        const int* q = ring + slot * G::SLOT;
        const int corner = q[G::RC + lc];
        rowCur[0] = r == 0 ? corner : rowCur[0];
#pragma unroll
        for (int q4 = 0; q4 < NK / 4; ++q4) {
          const int4 w = reinterpret_cast<const int4*>(q + lc * NK)[q4];
          rowCur[1 + 4 * q4] = r == 0 ? w.x : rowCur[1 + 4 * q4];
          rowCur[2 + 4 * q4] = r == 0 ? w.y : rowCur[2 + 4 * q4];
          rowCur[3 + 4 * q4] = r == 0 ? w.z : rowCur[3 + 4 * q4];
          rowCur[4 + 4 * q4] = r == 0 ? w.w : rowCur[4 + 4 * q4];
        }
#pragma unroll
        for (int p4 = 0; p4 < NJ / 4; ++p4) {
          const int4 w = reinterpret_cast<const int4*>(q + G::RQ + r * NJ)[p4];
          colCur[4 * p4] = lc == 0 ? w.x : colCur[4 * p4];
          colCur[4 * p4 + 1] = lc == 0 ? w.y : colCur[4 * p4 + 1];
          colCur[4 * p4 + 2] = lc == 0 ? w.z : colCur[4 * p4 + 2];
          colCur[4 * p4 + 3] = lc == 0 ? w.w : colCur[4 * p4 + 3];
        }
      }
      if (inner || (s >= 0 && s <= a)) {
        // Q = max{ max(Pd + A + B, Myz) + C, Pxy + A, Pxz + B, Sx, Sy, Sz }, the part from the previous
        // slice (E, X) one anti-diagonal ahead of the part within the slice, as in wavefront_vl.cuh.
        int E[NJ][NK], X[NJ][NK], Q[NJ][NK], ea[NJ];
#pragma unroll
        for (int pp = 0; pp < NJ; ++pp)
          ea[pp] = mad_lo(A[pp], p.one, pp == 0 ? rowPrev[0] : colPrev[pp - 1]);
#pragma unroll
        for (int dg = -1; dg < NJ + NK - 1; ++dg) {
#pragma unroll
          for (int pp = 0; pp < NJ; ++pp) {
            const int qq = dg + 1 - pp;
            if (qq >= 0 && qq < NK) {
              const int Pxy = (pp == 0) ? rowPrev[qq + 1] : P[pp - 1][qq];
              const int Pxz = (qq == 0) ? colPrev[pp] : P[pp][qq - 1];
              X[pp][qq] = ea[pp];
              ea[pp] = mad_lo(A[pp], p.one, Pxy);
              const unsigned eb = (unsigned)mad_lo(Bq[qq], p.one, Pxz);
              E[pp][qq] = (int)__vimax3_u16x2((unsigned)ea[pp], eb, (unsigned)P[pp][qq]);
            }
          }
#pragma unroll
          for (int pp = 0; pp < NJ; ++pp) {
            const int qq = dg - pp;
            if (qq >= 0 && qq < NK) {
              const int Myz = (pp == 0) ? rowCur[qq] : (qq == 0 ? colCur[pp - 1] : Q[pp - 1][qq - 1]);
              const int Sy = (pp == 0) ? rowCur[qq + 1] : Q[pp - 1][qq];
              const int Sz = (qq == 0) ? colCur[pp] : Q[pp][qq - 1];
              const unsigned w =
                  __viaddmax_u16x2((unsigned)X[pp][qq], (unsigned)Bq[qq], (unsigned)Myz);
              const unsigned q =
                  __viaddmax_u16x2(w, (unsigned)Cv[pp][qq], (unsigned)E[pp][qq]);
              Q[pp][qq] = (int)__vimax3_u16x2(q, (unsigned)Sy, (unsigned)Sz);
            }
          }
        }
#pragma unroll
        for (int pp = 0; pp < NJ; ++pp)
#pragma unroll
          for (int qq = 0; qq < NK; ++qq) P[pp][qq] = Q[pp][qq];
        // Record rows of this step: the last lane row's bottom words with the corner its consumer needs,
        // the last lane column's right words.
        {
          int* q = dstJ + (int64_t)t * G::RJ;
#pragma unroll
          for (int e = 0; e < NK; e += 4)
            vl_store(q + e, P[NJ - 1][e], P[NJ - 1][e + 1], P[NJ - 1][e + 2], P[NJ - 1][e + 3], f_oj);
          st_relaxed_if(q + kPC * NK - lc * NK + lc, colCur[NJ - 1], f_oj);
        }
        {
          int* q = dstK + (int64_t)t * G::RK;
#pragma unroll
          for (int e = 0; e < NJ; e += 4)
            vl_store(q + e, P[e][NK - 1], P[e + 1][NK - 1], P[e + 2][NK - 1], P[e + 3][NK - 1], f_ok);
        }
        if (!inner && owns0 && s == a0) {
          int v = 0;
#pragma unroll
          for (int pp = 0; pp < NJ; ++pp)
#pragma unroll
            for (int qq = 0; qq < NK; ++qq)
              if (pp == end_p0 && qq == end_q0) v = P[pp][qq];
          p.scores[d.out_idx] = (v & 0xffff) - (kBias16x2 & 0xffff) + d.score_base;
        }
        if (!inner && owns1 && s == a1) {
          int v = 0;
#pragma unroll
          for (int pp = 0; pp < NJ; ++pp)
#pragma unroll
            for (int qq = 0; qq < NK; ++qq)
              if (pp == end_p1 && qq == end_q1) v = P[pp][qq];
          p.scores[d1.out_idx] = (int)((unsigned)v >> 16) - (kBias16x2 & 0xffff) + d1.score_base;
        }
      }
    };
    // From step kInner on every lane's slice is in the cube.
    constexpr int kInner = (kPR - 1) + (kPC - 1);
    static_assert(kInner % 2 == 0, "pairs of steps");
    const auto pair = [&](const int t, const bool inner) -> bool {
      const int slot = t & 2;
      refill(t);
      if (!stage(t, inner, slot)) return false;
      step(t, inner, slot, rowA, rowB, colA, colB);
      if (inner || t + 1 < T) step(t + 1, inner, slot + 1, rowB, rowA, colB, colA);
      return true;
    };
    int t = 0;
    bool running = ok;
    while (running && t < T) {
      if (t == kInner) {
        // the piece of steps t + 2 and t + 3 is fetched unchecked
        for (; running && t + 3 <= lim; t += 2) running = pair(t, true);
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
  }
}

}  // namespace trioseq
