// One sweep of Algorithm 1 (all colour steps, then the diagonal step) in
// FP32 by a group of CTAs, tile by tile instead of colour by colour.
//
// In the circle method (Section 3.2) vertices i, j >= 1 meet in the colour
// step that depends on i + j mod P alone: the sums run P, P - 2, .., 1 next
// to 2 P, 2 P - 2, .., P + 1 in the first half of a sweep and P - 1, .., 2
// next to 2 P - 1, .., P + 2 in the second; vertex 0 meets v where v would
// meet itself (i = j = v).  A pair (i, j) needs the rows i and j after their
// earlier pairs, which are (i, j') with j' > j and (i', j) with i' > i of the
// same half and side of P (and all of the other side's before or after): the
// pairs of one half and side form a triangle of a 2-D wavefront.  Cut into 32 x 32 tiles of
// vertices, a tile depends only on the tiles of a larger block sum in its
// block row and column, so tiles of equal I + J run at the same time and a
// block sits in exactly one tile at a time:
//     wave A - (I + J)        the tiles with sums <= P,  A = floor(P / 32)
//     wave A + nb - (I + J)   the tiles with sums >  P.
// A CTA owns one block of 32 rows of W (and Omega).  For a tile (I, J) the
// two owners swap the entries W_I,J and W_J,I the tile's pairs read (one
// tagged 64-bit word per thread through L2, no fence), both walk the tile's
// at most 32 colour steps in shared memory and registers (one CTA barrier
// per step, ~0.1 us, where a step through L2 took 3.3 us), and each updates
// its own rows: first the columns of its next tile, which it publishes, then
// the rest, while the words travel.  Vertex 0's row is spread over the
// owners by columns; its changes are published as words too.
//
// Every entry of W gets the same FMAs in the same order as in the colour-by-
// colour kernels (a row's changes in step order), so the iterates are theirs
// bit for bit.  FP32 only: the step's arithmetic on every warp would queue
// on the narrow FP64 pipe.
// Waits (on a partner's word) are bounded like every other wait.
#pragma once
#include "common.cuh"

namespace concord {

constexpr int kWaveB = 32;          // vertices of a block
constexpr int kWaveThreads = 512;   // 16 warps, two rows of each side per warp

__host__ __device__ inline int wave_blocks(int p) { return (p + kWaveB - 1) / kWaveB; }
__host__ __device__ inline int wave_slots(int p) { return 2 * (wave_blocks(p) + 3); }
// 64-bit words of the exchange buffer (zeroed once; tags grow).
__host__ __device__ inline size_t wave_words(int p, int nm) {
  return (size_t)nm * ((size_t)wave_blocks(p) * wave_slots(p) * kWaveThreads +
                       (size_t)wave_blocks(p) * kWaveB);
}

template <int NM>
struct WaveArgs {
  int p, P, ld;
  const float* S[NM];
  float* W[NM];
  float* Om[NM];
  const float* sdiag[NM];     // s_ii, sd_stride apart
  size_t sd_stride;
  unsigned long long* words;  // wave_words(p, NM)
  unsigned tag;               // of this sweep: larger than any before in `words`
  WaitCtl wait;
};

template <int NM>
struct WaveSmem {
  float sii[NM][kWaveB][kWaveB];     // S of the own block
  float sjj[NM][kWaveB][kWaveB];     // S of the tile's other block
  float sjn[NM][kWaveB][kWaveB];     // S of that block's rows in the next tile's columns
  float om[NM][kWaveB][kWaveB];      // Omega_I,J at the tile's start
  float d[2][NM][2][16][16];         // changes [tile parity][m][row parity][j / 2][row / 2]
  float d0[NM][kWaveB];              // changes of the pairs (0, i), diagonal tiles
  float x[2][NM][2 * kWaveB + 1];    // W entries of a step's pairs
  float sd[NM][2][kWaveB];           // diagonals of S: own block, other block
  float s0[NM][kWaveB], s0n[NM][kWaveB], si0[NM][kWaveB];  // S_0,I, S_0,next, S_I,0
  float om0[NM][kWaveB];             // Omega_0,I
  float dd[NM][kWaveB];              // diagonal changes
  float s00[NM], sd0[NM];
};

struct WaveTile {
  int J;        // other block (-1: none)
  int slot;     // exchange slot
  int lo, hi;   // sums, hi of the tile's parity; empty when hi < lo
};

// The block's v-th tile of a sweep (v counts the lower, then the upper tiles
// of the first half, then those of the second); J = -1 past the last one.
__host__ __device__ inline WaveTile wave_tile(int I, int nb, int P, int v) {
  auto min = [](int x, int y) { return x < y ? x : y; };
  auto max = [](int x, int y) { return x > y ? x : y; };
  const int A = P / kWaveB;
  const int nl = A - I + 1 > 0 ? min(A - I, nb - 1) + 1 : 0;  // lower tiles J = min(A - I, nb - 1) .. 0
  // upper tiles J = nb - 1 .. jmin: some sum 32 (I + J) + 62 >= P + 1
  const int jmin = max(0, (P + 1 - 62 + kWaveB - 1 + 64 * kWaveB) / kWaveB - 64 - I);
  const int nu = nb - jmin > 0 ? nb - jmin : 0;
  WaveTile t;
  const int half = v >= nl + nu ? 1 : 0;
  const int u = v - half * (nl + nu);
  if (u >= nl + nu) {
    t.J = -1;
    t.slot = t.lo = t.hi = 0;
    return t;
  }
  const bool lower = u < nl;
  t.J = lower ? nl - 1 - u : nb - 1 - (u - nl);
  const int w = lower ? A - (I + t.J) : A + nb - (I + t.J);
  t.slot = half * (nb + 3) + w;
  const int par = (half == 0) == lower ? 1 : 0;  // parity of the sums
  t.lo = lower ? max(1, kWaveB * (I + t.J)) : max(P + 1, kWaveB * (I + t.J));
  t.hi = min(lower ? P : 2 * P, kWaveB * (I + t.J) + 2 * kWaveB - 2);
  if ((t.hi & 1) != par) --t.hi;
  return t;
}

__device__ __forceinline__ unsigned long long wave_word(unsigned tag, float v) {
  return ((unsigned long long)tag << 32) | __float_as_uint(v);
}

// The word's value once it carries `tag`.
__device__ __forceinline__ float wave_wait(const unsigned long long* p, unsigned tag, const WaitCtl& w,
                                           int who, int step) {
  unsigned long long v = ld_relaxed_u64(p);
  if ((unsigned)(v >> 32) != tag) {
    const uint64_t t0 = globaltimer_ns();
    unsigned it = 0;
    while ((unsigned)((v = ld_relaxed_u64(p)) >> 32) != tag) {
      if ((++it & 63u) == 0) {
        if (ld_relaxed_s32(w.abort) != 0) break;
        if (globaltimer_ns() - t0 > w.timeout_ns) {
          record_timeout(w, who, step);
          break;
        }
      }
    }
  }
  return __uint_as_float((unsigned)(v & 0xffffffffull));
}

__device__ __forceinline__ void cp_async16(void* smem, const void* g) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                   (unsigned)__cvta_generic_to_shared(smem)),
               "l"(g)
               : "memory");
}

// dst = the 32 x 32 block of M (rows r0 .., below p, else zero; columns c0 ..)
__device__ __forceinline__ void wave_load(float (*dst)[kWaveB], const float* M, int r0, int c0, int p,
                                          int ld, int part) {
  const int e = (int)threadIdx.x - 256 * part;
  if (e < 0 || e >= 256) return;
  const int r = e >> 3, c = (e & 7) * 4;
  if (r0 + r < p)
    cp_async16(&dst[r][c], M + (size_t)(r0 + r) * ld + c0 + c);
  else
    *reinterpret_cast<float4*>(&dst[r][c]) = make_float4(0.f, 0.f, 0.f, 0.f);
}

// The sweep.  Ops: pair(c, om, wa, wb, nw): the new values of a pair from c_m
// = s_ii + s_jj, its old values and W_lo,hi, W_hi,lo; count(d): once per
// owned row and pair; diag(i, w, dd): row i's diagonal change from W_ii
// (stores the new diagonal).  I: the CTA's block.
template <int NM, class Ops>
__device__ void wave_sweep(const WaveArgs<NM>& a, WaveSmem<NM>& s, int I, Ops& ops) {
  constexpr unsigned FULL = 0xffffffffu;
  const int tid = (int)threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int p = a.p, P = a.P, ld = a.ld, nb = wave_blocks(p), slots = wave_slots(p);
  const int nv = ld >> 2;
  const int i0 = kWaveB * I;            // first own row
  const int ir = i0 + 2 * wid;          // this warp's own rows: ir, ir + 1
  unsigned long long* const zw = a.words + (size_t)NM * nb * slots * kWaveThreads;  // [NM][32 nb]
  auto slot_words = [&](int b, int slot, int m) {
    return a.words + (((size_t)b * slots + slot) * NM + m) * kWaveThreads;
  };
  const bool own0 = ir >= 1 && ir < p, own1 = ir + 1 < p;  // vertex 0's row is not the block's

  // ---- what stays for the whole sweep
  float Z[NM], Z0[NM];  // warp 0: W_0 in the own columns (and, block 0, in column 0)
#pragma unroll
  for (int m = 0; m < NM; ++m) {
    wave_load(s.sii[m], a.S[m], i0, i0, p, ld, m & 1);
    if (tid < kWaveB) {
      s.sd[m][0][tid] = i0 + tid < p ? a.sdiag[m][(size_t)(i0 + tid) * a.sd_stride] : 1.f;
      s.s0[m][tid] = a.S[m][i0 + tid];
      s.si0[m][tid] = i0 + tid < p ? a.S[m][(size_t)(i0 + tid) * ld] : 0.f;
      s.om0[m][tid] = a.Om[m][i0 + tid];
    }
    if (tid == 0) {
      s.s00[m] = a.S[m][0];
      s.sd0[m] = a.sdiag[m][0];
    }
    Z[m] = wid == 0 ? __ldcg(a.W[m] + i0 + lane) : 0.f;
    Z0[m] = 0.f;
  }
  int zdone = nb;  // warp 0: the changes of vertex 0's pairs in blocks >= zdone are in Z
  // Vertex 0's changes of block b into Z, in the order of their steps (v
  // downwards).  wait = false: only if all of them are there.
  auto zapply = [&](int b, bool wait) -> bool {
    float d[NM];
    const int v = kWaveB * b + lane;
    bool here = true;
#pragma unroll
    for (int m = 0; m < NM; ++m) {
      d[m] = 0.f;
      if (v >= 1 && v < p) {
        const unsigned long long* q = zw + (size_t)m * kWaveB * nb + v;
        if (wait) {
          d[m] = wave_wait(q, a.tag, a.wait, 0, P - v);
        } else {
          const unsigned long long x = ld_relaxed_u64(q);
          d[m] = __uint_as_float((unsigned)(x & 0xffffffffull));
          here = here && (unsigned)(x >> 32) == a.tag;
        }
      }
    }
    if (!__all_sync(FULL, here)) return false;
#pragma unroll
    for (int m = 0; m < NM; ++m) {
      unsigned nz = __ballot_sync(FULL, d[m] != 0.f);
      while (nz) {
        const int l = 31 - __clz(nz);
        nz &= ~(1u << l);
        const float x = __shfl_sync(FULL, d[m], l);
        const float* row = a.S[m] + (size_t)(kWaveB * b + l) * ld;
        Z[m] = fmaf(x, __ldg(row + i0 + lane), Z[m]);
      }
    }
    return true;
  };

  WaveTile t = wave_tile(I, nb, P, 0);
  float A[NM][2];  // W_I,J: own rows ir, ir + 1, column 32 J + lane
#pragma unroll
  for (int m = 0; m < NM; ++m) {
    const int c = kWaveB * t.J + lane;
    A[m][0] = own0 ? a.W[m][(size_t)ir * ld + c] : 0.f;
    A[m][1] = own1 ? a.W[m][(size_t)(ir + 1) * ld + c] : 0.f;
  }
  int Jp = -1;       // the previous tile's block (its changes not yet in the other columns)
  bool diag0 = false;  // that tile held vertex 0's pairs
  int par_p = 0;       // its sums' parity

  // The own rows' changes of tile Jp (buffer db) into every column vector
  // but the excluded blocks'.  Thread groups: row parity x half of the rows.
  auto bulk = [&](int Jb, int db, bool with0, int par, int ex0, int ex1) {
    const int g = tid >> 7, rp = g & 1, hf = g >> 1;
    const int jp = (par ^ rp) & 1;  // parity of the partners of rows of parity rp
    for (int q = tid & 127; q < nv; q += 128) {
      const int blk = q >> 3;
      if (blk == ex0 || blk == ex1) continue;
#pragma unroll
      for (int m = 0; m < NM; ++m) {
        float4 acc[8];
#pragma unroll
        for (int r = 0; r < 8; ++r) {
          const int i = i0 + 2 * (8 * hf + r) + rp;
          acc[r] = i >= 1 && i < p ? reinterpret_cast<const float4*>(a.W[m] + (size_t)i * ld)[q]
                                   : make_float4(0.f, 0.f, 0.f, 0.f);
        }
        float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
        if (with0) z = __ldg(reinterpret_cast<const float4*>(a.S[m]) + q);
        const float* dm = &s.d[db][m][rp][0][8 * hf];
#pragma unroll 4
        for (int k = 15; k >= 0; --k) {
          const int j = kWaveB * Jb + 2 * k + jp;
          const float4 d0 = *reinterpret_cast<const float4*>(dm + 16 * k);
          const float4 d1 = *reinterpret_cast<const float4*>(dm + 16 * k + 4);
          const float4 sv = j < p ? __ldg(reinterpret_cast<const float4*>(a.S[m] + (size_t)j * ld) + q)
                                  : make_float4(0.f, 0.f, 0.f, 0.f);
          const float dr[8] = {d0.x, d0.y, d0.z, d0.w, d1.x, d1.y, d1.z, d1.w};
#pragma unroll
          for (int r = 0; r < 8; ++r) {
            acc[r].x = fmaf(dr[r], sv.x, acc[r].x);
            acc[r].y = fmaf(dr[r], sv.y, acc[r].y);
            acc[r].z = fmaf(dr[r], sv.z, acc[r].z);
            acc[r].w = fmaf(dr[r], sv.w, acc[r].w);
          }
          if (with0) {  // the pair (0, i) stands where i would meet itself
#pragma unroll
            for (int r = 0; r < 8; ++r)
              if (8 * hf + r == k) {
                const float d = s.d0[m][2 * k + rp];
                acc[r].x = fmaf(d, z.x, acc[r].x);
                acc[r].y = fmaf(d, z.y, acc[r].y);
                acc[r].z = fmaf(d, z.z, acc[r].z);
                acc[r].w = fmaf(d, z.w, acc[r].w);
              }
          }
        }
#pragma unroll
        for (int r = 0; r < 8; ++r) {
          const int i = i0 + 2 * (8 * hf + r) + rp;
          if (i >= 1 && i < p) reinterpret_cast<float4*>(a.W[m] + (size_t)i * ld)[q] = acc[r];
        }
      }
    }
  };

  int v = 0;
  for (; t.J >= 0; ++v) {
    const int J = t.J, j0 = kWaveB * J, db = v & 1, par = t.hi & 1;
    const bool dt = I == J;
    const WaveTile nx = wave_tile(I, nb, P, v + 1);
    const int jr = j0 + 2 * wid;
    // ---- the tile's operands on their way; the own entries to the partner
#pragma unroll
    for (int m = 0; m < NM; ++m) {
      if (!dt) wave_load(s.sjj[m], a.S[m], j0, j0, p, ld, 0);
      wave_load(s.om[m], a.Om[m], i0, j0, p, ld, 1);
      if (nx.J >= 0) wave_load(s.sjn[m], a.S[m], j0, kWaveB * nx.J, p, ld, 0);
      if (tid < kWaveB) {
        s.sd[m][1][tid] = j0 + tid < p ? a.sdiag[m][(size_t)(j0 + tid) * a.sd_stride] : 1.f;
        if (nx.J >= 0) s.s0n[m][tid] = a.S[m][kWaveB * nx.J + tid];
      }
      reinterpret_cast<float*>(s.d[db][m])[tid] = 0.f;
      // (row parity, column) picks one of the two rows per lane
      if (!dt)
        st_relaxed_u64(slot_words(I, t.slot, m) + tid,
                       wave_word(a.tag, ((par ^ lane) & 1) ? A[m][1] : A[m][0]));
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
    // ---- the previous tile's changes into the other columns, meanwhile
    if (Jp >= 0) bulk(Jp, db ^ 1, diag0, par_p, Jp, J);
    if (wid == 0)
      while (zdone > 0 && zdone - 1 != I && zapply(zdone - 1, false)) --zdone;
    // ---- the partner's entries: W_j,i of row jr + rb, column i0 + lane
    const int rb = (par ^ lane) & 1;
    float B[NM], E[NM][2];
#pragma unroll
    for (int m = 0; m < NM; ++m) {
      B[m] = 0.f;
      if (!dt) B[m] = wave_wait(slot_words(J, t.slot, m) + tid, a.tag, a.wait, jr, t.slot);
    }
    __syncthreads();  // bulk done everywhere (W_i0 below, d[db ^ 1])
    if (dt) {
      if (wid == 0 && par == 0)
        while (zdone - 1 > I) zapply(--zdone, true);
#pragma unroll
      for (int m = 0; m < NM; ++m) {
        // W_i,0: column 0 of the own rows (block 0: lane 0 of A)
        E[m][0] = I == 0 ? __shfl_sync(FULL, A[m][0], 0) : (own0 ? a.W[m][(size_t)ir * ld] : 0.f);
        E[m][1] = I == 0 ? __shfl_sync(FULL, A[m][1], 0) : (own1 ? a.W[m][(size_t)(ir + 1) * ld] : 0.f);
        if (tid < kWaveB) s.d0[m][tid] = 0.f;
      }
    }
    // the next tile's columns of the own rows, up to the previous tile
    float N[NM][2];
#pragma unroll
    for (int m = 0; m < NM; ++m) {
      N[m][0] = N[m][1] = 0.f;
      if (nx.J >= 0 && nx.J != J) {
        const int c = kWaveB * nx.J + lane;
        N[m][0] = own0 ? a.W[m][(size_t)ir * ld + c] : 0.f;
        N[m][1] = own1 ? a.W[m][(size_t)(ir + 1) * ld + c] : 0.f;
      }
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();
    // ---- the colour steps
    int bf = 0;
    for (int sum = t.hi; sum >= t.lo; sum -= 2, bf ^= 1) {
      if (!dt) {
        const int jl0 = sum - ir - j0, jl1 = jl0 - 1;       // partners of the own rows
        const int il0 = sum - jr - i0, il1 = il0 - 1;       // partners of the other block's rows
#pragma unroll
        for (int m = 0; m < NM; ++m) {
          if (lane == jl0) s.x[bf][m][2 * wid] = A[m][0];
          if (lane == jl1) s.x[bf][m][2 * wid + 1] = A[m][1];
          if (lane == il0) s.x[bf][m][kWaveB + 2 * wid] = B[m];
          if (lane == il1) s.x[bf][m][kWaveB + 2 * wid + 1] = B[m];
        }
        __syncthreads();
        // lane & 3 picks the pair: own row 0, 1, other row 0, 1
        const int k = lane & 3;
        const int il = k < 2 ? 2 * wid + k : (k == 2 ? il0 : il1);
        const int jl = k < 2 ? (k == 0 ? jl0 : jl1) : 2 * wid + k - 2;
        const int i = i0 + il, j = j0 + jl;
        float d[NM];
#pragma unroll
        for (int m = 0; m < NM; ++m) d[m] = 0.f;
        if (((il | jl) & ~31) == 0 && i >= 1 && j >= 1 && i < p && j < p) {
          float c[NM], om[NM], wa[NM], wb[NM], nw[NM];
#pragma unroll
          for (int m = 0; m < NM; ++m) {
            const float wu = s.x[bf][m][il], wv = s.x[bf][m][kWaveB + jl];
            wa[m] = i < j ? wu : wv;
            wb[m] = i < j ? wv : wu;
            om[m] = s.om[m][il][jl];
            c[m] = s.sd[m][0][il] + s.sd[m][1][jl];
          }
          ops.pair(c, om, wa, wb, nw);
#pragma unroll
          for (int m = 0; m < NM; ++m) d[m] = nw[m] - om[m];
          if (lane < 2) {
#pragma unroll
            for (int m = 0; m < NM; ++m)
              if (d[m] != 0.f) {
                s.d[db][m][il & 1][jl >> 1][il >> 1] = d[m];
                a.Om[m][(size_t)i * ld + j] = nw[m];
              }
            ops.count(d);
          }
        }
        const int ilb = rb ? il1 : il0;
#pragma unroll
        for (int m = 0; m < NM; ++m) {
          const float e0 = __shfl_sync(FULL, d[m], 0), e1 = __shfl_sync(FULL, d[m], 1);
          const float f0 = __shfl_sync(FULL, d[m], 2), f1 = __shfl_sync(FULL, d[m], 3);
          A[m][0] = fmaf(e0, s.sjj[m][jl0 & 31][lane], A[m][0]);
          A[m][1] = fmaf(e1, s.sjj[m][jl1 & 31][lane], A[m][1]);
          B[m] = fmaf(rb ? f1 : f0, s.sii[m][ilb & 31][lane], B[m]);
        }
      } else {
        const int jl0 = sum - ir - i0, jl1 = jl0 - 1;
        const int l0 = 2 * wid, l1 = 2 * wid + 1;  // own local rows; jl == l: vertex 0
        const int vz = (sum & 1) ? -1 : (sum >> 1) - i0;  // vertex 0's partner (local)
#pragma unroll
        for (int m = 0; m < NM; ++m) {
          if (lane == (jl0 & 31) && (jl0 & ~31) == 0) s.x[bf][m][l0] = jl0 == l0 ? E[m][0] : A[m][0];
          if (lane == (jl1 & 31) && (jl1 & ~31) == 0) s.x[bf][m][l1] = jl1 == l1 ? E[m][1] : A[m][1];
          if (wid == 0 && lane == vz) s.x[bf][m][kWaveB] = Z[m];
        }
        __syncthreads();
        // lane & 3: own row 0, 1, (warp 0) vertex 0's pair
        const int k = lane & 3;
        const int il = k < 2 ? 2 * wid + k : vz;
        const int jl = k < 2 ? (k == 0 ? jl0 : jl1) : vz;
        const bool with0 = il == jl;
        const int i = i0 + il, j = with0 ? 0 : i0 + jl;
        float d[NM];
#pragma unroll
        for (int m = 0; m < NM; ++m) d[m] = 0.f;
        const bool is = k < 2 || (k == 2 && wid == 0);
        if (is && ((il | jl) & ~31) == 0 && i >= 1 && i < p && (with0 || (j >= 1 && j < p))) {
          float c[NM], om[NM], wa[NM], wb[NM], nw[NM];
#pragma unroll
          for (int m = 0; m < NM; ++m) {
            const float wu = s.x[bf][m][il], wv = s.x[bf][m][with0 ? kWaveB : jl];
            wa[m] = i < j ? wu : wv;
            wb[m] = i < j ? wv : wu;
            om[m] = with0 ? s.om0[m][il] : s.om[m][il][jl];
            c[m] = s.sd[m][0][il] + (with0 ? s.sd0[m] : s.sd[m][0][jl]);
          }
          ops.pair(c, om, wa, wb, nw);
#pragma unroll
          for (int m = 0; m < NM; ++m) d[m] = nw[m] - om[m];
          if (lane < 2) {
#pragma unroll
            for (int m = 0; m < NM; ++m)
              if (d[m] != 0.f) {
                if (with0)
                  s.d0[m][il] = d[m];
                else
                  s.d[db][m][il & 1][jl >> 1][il >> 1] = d[m];
                a.Om[m][(size_t)i * ld + j] = nw[m];
              }
            ops.count(d);
          } else if (lane == 2) {  // vertex 0's row
#pragma unroll
            for (int m = 0; m < NM; ++m) {
              if (d[m] != 0.f) a.Om[m][i] = nw[m];
              st_relaxed_u64(zw + (size_t)m * kWaveB * nb + i, wave_word(a.tag, d[m]));
            }
            ops.count(d);
          }
        }
#pragma unroll
        for (int m = 0; m < NM; ++m) {
          const float e0 = __shfl_sync(FULL, d[m], 0), e1 = __shfl_sync(FULL, d[m], 1);
          const float ez = __shfl_sync(FULL, d[m], 2);
          const float* r0 = jl0 == l0 ? s.s0[m] : s.sii[m][jl0 & 31];
          const float* r1 = jl1 == l1 ? s.s0[m] : s.sii[m][jl1 & 31];
          A[m][0] = fmaf(e0, r0[lane], A[m][0]);
          A[m][1] = fmaf(e1, r1[lane], A[m][1]);
          E[m][0] = fmaf(e0, jl0 == l0 ? s.s00[m] : s.si0[m][jl0 & 31], E[m][0]);
          E[m][1] = fmaf(e1, jl1 == l1 ? s.s00[m] : s.si0[m][jl1 & 31], E[m][1]);
          if (wid == 0) Z[m] = fmaf(ez, s.sii[m][vz & 31][lane], Z[m]);
        }
      }
    }
    __syncthreads();  // the tile's changes are in s.d
    const bool with0 = dt && par == 0;
    if (with0) zdone = I;  // vertex 0's changes of the own block are in Z
    // ---- W_I,J is final for this tile; the next tile's columns follow
    float Y[NM][2];
#pragma unroll
    for (int m = 0; m < NM; ++m) {
      const int c = j0 + lane;
      if (own0) a.W[m][(size_t)ir * ld + c] = A[m][0];
      if (own1) a.W[m][(size_t)(ir + 1) * ld + c] = A[m][1];
      Y[m][0] = nx.J == J ? A[m][0] : N[m][0];
      Y[m][1] = nx.J == J ? A[m][1] : N[m][1];
      if (nx.J >= 0 && nx.J != J) {
#pragma unroll
        for (int r = 0; r < 2; ++r) {
          const int jp = (par ^ r) & 1;
#pragma unroll 4
          for (int k = 15; k >= 0; --k) {
            Y[m][r] = fmaf(s.d[db][m][r][k][wid], s.sjn[m][2 * k + jp][lane], Y[m][r]);
            if (with0 && k == wid) Y[m][r] = fmaf(s.d0[m][2 * wid + r], s.s0n[m][lane], Y[m][r]);
          }
        }
      }
      A[m][0] = Y[m][0];
      A[m][1] = Y[m][1];
    }
    __syncthreads();  // s.sjn, s.sjj, s.om are free
    Jp = J;
    diag0 = with0;
    par_p = par;
    t = nx;
  }
  // ---- the last tile's changes; vertex 0's remaining changes
  if (Jp >= 0) bulk(Jp, (v - 1) & 1, diag0, par_p, Jp, -1);
  if (wid == 0) {
    while (zdone > 0) zapply(--zdone, true);
    if (I == 0) {  // column 0 of W_0, over all of vertex 0's changes
#pragma unroll
      for (int m = 0; m < NM; ++m) Z0[m] = __shfl_sync(FULL, Z[m], 0);
    }
  }
  __syncthreads();
  // ---- diagonal step: one lane per row (row 0: the owner of block 0)
  if (wid == 0) {
    float w[NM], dd[NM];
    const int i = i0 + lane;
#pragma unroll
    for (int m = 0; m < NM; ++m) {
      dd[m] = 0.f;
      w[m] = i == 0 ? Z0[m] : (i < p ? a.W[m][(size_t)i * ld + i] : 0.f);
    }
    if (i < p) ops.diag(i, w, dd);
#pragma unroll
    for (int m = 0; m < NM; ++m) {
      s.dd[m][lane] = i == 0 ? 0.f : dd[m];  // row 0 is updated below, by columns
      if (i == 0) st_relaxed_u64(zw + (size_t)m * kWaveB * nb, wave_word(a.tag, dd[m]));
      const float z = wave_wait(zw + (size_t)m * kWaveB * nb, a.tag, a.wait, 0, P);
      if (z != 0.f) Z[m] = fmaf(z, s.s0[m][lane], Z[m]);
      __syncwarp();
      a.W[m][i0 + lane] = Z[m];
    }
  }
  __syncthreads();
#pragma unroll
  for (int m = 0; m < NM; ++m)
    for (int r = wid; r < kWaveB; r += kWaveThreads / 32) {
      const float d = s.dd[m][r];
      if (d == 0.f || i0 + r >= p) continue;
      float4* w = reinterpret_cast<float4*>(a.W[m] + (size_t)(i0 + r) * ld);
      const float4* sr = reinterpret_cast<const float4*>(a.S[m] + (size_t)(i0 + r) * ld);
      for (int q = lane; q < nv; q += 32) {
        float4 x = w[q];
        const float4 y = __ldg(sr + q);
        x.x = fmaf(d, y.x, x.x);
        x.y = fmaf(d, y.y, x.y);
        x.z = fmaf(d, y.z, x.z);
        x.w = fmaf(d, y.w, x.w);
        w[q] = x;
      }
    }
}

}  // namespace concord
