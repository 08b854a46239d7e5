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
// two owners swap the entries W_I,J and W_J,I the tile's pairs read (tagged
// 64-bit words through L2, no fence) and both walk the tile's at most 32
// colour steps.  Two warps walk them, one per side: lane l keeps the entries
// row l of its side still has to meet, next one first; a step is a swap of
// the entries at hand, the pairs' arithmetic and the FMAs of the entries to
// come.  Eight warps bring the next tile's columns up to date with the tile's
// changes and publish them; the other six, and up to three more CTAs (a
// cluster per block), meanwhile apply the previous tile's changes to all
// other columns of the own rows and fetch the next tile's operands.  Vertex
// 0's row is spread over the owners by columns; its changes are published as
// words too.
//
// p = 1000, FP32, a tile of one matrix: 9.9 us, of which the steps 5.5, the
// wait for the partner 1.4, the next tile's columns and their publication 2.8;
// with sixteen warps walking the steps together behind a CTA barrier and then
// updating everything 22 us.  What bounds it is the chain: swap, pair, FMA of
// a step (~0.17 us), and a diagonal tile's longer steps (7 - 8 us a tile).
// 32-lambda path 293 -> 119 ms, joint solve of 9 sweeps 22.3 -> 8.2 ms.
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
constexpr int kWaveThreads = 512;
constexpr int kWaveFirst = 32 * 10;  // warps 0, 1: the steps; warps 2 .. 9: the next tile's columns,
                                     // four rows each; the rest: the other columns
constexpr int kWaveRest = kWaveThreads - kWaveFirst;
constexpr int kWaveRestWarps = kWaveRest / 32, kWaveWarps = kWaveThreads / 32;
constexpr int kWaveCluster = 4;     // CTAs of a block at most: one for the above, the others for its
                                    // other columns as well
constexpr int kWaveSkew = 20;       // row stride of the skewed blocks: 16 entries, 16-byte loads of
                                    // eight lanes on distinct banks
constexpr int kWaveWords = 512;     // words an owner publishes per tile and matrix

__host__ __device__ inline int wave_blocks(int p) { return (p + kWaveB - 1) / kWaveB; }
__host__ __device__ inline int wave_slots(int p) { return 2 * (wave_blocks(p) + 3); }
// 64-bit words of the exchange buffer (zeroed once; tags grow).
__host__ __device__ inline size_t wave_words(int p, int nm) {
  return (size_t)nm * ((size_t)wave_blocks(p) * wave_slots(p) * kWaveWords +
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

// Skewed blocks: row r's entry u is column (r - 2 (u + 1)) mod 32, what the
// row that met r meets u + 1 steps later.
template <int NM>
struct WaveSmem {
  float ti[NM][kWaveB][kWaveSkew];         // S of the own block, skewed
  float t0[NM][kWaveB][kWaveSkew];         // S_0 in the own columns, skewed as row r = r
  float tj[2][NM][kWaveB][kWaveSkew];      // S of the tile's other block [tile parity], skewed
  float a[NM][kWaveB][kWaveSkew];          // W_I,J of the tile's pairs, in step order
  float b[NM][kWaveB][kWaveSkew];          // W_J,I
  float sii[NM][kWaveB][kWaveB];           // S of the own block
  float sjn[2][NM][kWaveB][kWaveB];        // S of the other block's rows in the next tile's columns
  float spn[2][NM][kWaveB][kWaveB];        // and of the previous tile's
  float om[2][NM][kWaveB][kWaveB];         // Omega_I,J
  float rc[2][2 * NM - 1][kWaveB][kWaveB];  // reciprocals of the pairs' denominators
  float x[2][2][NM][kWaveB];               // a step's entries [parity][side]
  float d[2][NM][2][16][16];               // changes [tile parity][m][row parity][j / 2][row / 2]
  float d0[2][NM][kWaveB];                 // changes of the pairs (0, i), diagonal tiles
  float sd[2][NM][kWaveB], sdi[NM][kWaveB];  // diagonals of S: other block, own block
  float s0n[2][NM][kWaveB];                // S_0 in the next tile's columns
  float s0[NM][kWaveB], si0[NM][kWaveB];   // S_0,I, S_I,0
  float om0[NM][kWaveB];                   // Omega_0,I
  float rz[2 * NM - 1][kWaveB];            // reciprocals of the pairs (0, i)
  float e[NM][kWaveB], z[NM][kWaveB];      // W_I,0 and W_0,I of a diagonal tile
  float dd[NM][kWaveB];                    // diagonal changes
  unsigned need[2][NM][4];                 // j / 2 with changes [tile parity][m][half of rows, row parity]
  float nw0[NM][kWaveB];                   // new values of the pairs (0, i)
  float s00[NM], sd0[NM];
  WaveArgs<NM> args;                       // (in registers they would be held through the sweep)
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

// Behind the exchange words of a problem: what its launches hand on (words).
constexpr int kWaveStateWords = 32, kWaveSweepParts = 4, kWaveEvalCtas = 256, kWaveEvalParts = 8;
__host__ __device__ inline size_t wave_scratch_words(int p, int nm) {
  return wave_words(p, nm) + kWaveStateWords + (size_t)kWaveSweepParts * wave_blocks(p) +
         (size_t)kWaveEvalParts * kWaveEvalCtas;
}
template <class State>
__host__ __device__ __forceinline__ State* wave_state(unsigned long long* words, int p, int nm) {
  static_assert(sizeof(State) <= 8 * kWaveStateWords, "the state's words");
  return reinterpret_cast<State*>(words + wave_words(p, nm));
}
// per CTA of the sweep: kWaveSweepParts; per CTA of the evaluation: kWaveEvalParts
__device__ __forceinline__ double* wave_sweep_parts(unsigned long long* words, int p, int nm) {
  return reinterpret_cast<double*>(words + wave_words(p, nm) + kWaveStateWords);
}
__device__ __forceinline__ double* wave_eval_parts(unsigned long long* words, int p, int nm) {
  return wave_sweep_parts(words, p, nm) + (size_t)kWaveSweepParts * wave_blocks(p);
}

// Every thread's (largest change, count) over the CTA, by thread 0 into out.
__device__ __forceinline__ void wave_put_parts(double delta, double count, double* out) {
  __shared__ double red[kWaveThreads / 32][2];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  __syncwarp();
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const double d = __shfl_down_sync(0xffffffffu, delta, o);
    delta = d > delta || d != d ? d : delta;  // (NaN stays)
    count += __shfl_down_sync(0xffffffffu, count, o);
  }
  if (lane == 0) {
    red[wid][0] = delta;
    red[wid][1] = count;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < kWaveThreads / 32; ++w) {
      const double d = red[w][0];
      delta = d > delta || d != d ? d : delta;
      count += red[w][1];
    }
    out[0] = delta;
    out[1] = count;
  }
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

__device__ __forceinline__ void cp_async4(void* smem, const void* g) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(
                   (unsigned)__cvta_generic_to_shared(smem)),
               "l"(g)
               : "memory");
}

// dst = the 32 x 32 block of M (rows r0 .., below p, else zero; columns c0
// ..), by n threads.
__device__ __forceinline__ void wave_load(float (*dst)[kWaveB], const float* M, int r0, int c0, int p,
                                          int ld, int th, int n) {
  for (int e = th; e < 8 * kWaveB; e += n) {
    const int r = e >> 3, c = (e & 7) * 4;
    if (r0 + r < p)
      cp_async16(&dst[r][c], M + (size_t)(r0 + r) * ld + c0 + c);
    else
      *reinterpret_cast<float4*>(&dst[r][c]) = make_float4(0.f, 0.f, 0.f, 0.f);
  }
}

// The same block (its diagonal one, r0 = c0), skewed; stride 0 for ld: row r0 in every row.
__device__ __forceinline__ void wave_load_skewed(float (*dst)[kWaveSkew], const float* M, int r0,
                                                 int c0, int p, int ld, int th, int n) {
  for (int e = th; e < 16 * kWaveB; e += n) {
    const int r = e >> 4, u = e & 15;
    if (ld == 0 || r0 + r < p)
      cp_async4(&dst[r][u], M + (size_t)(r0 + r) * ld + c0 + ((r - 2 * u - 2) & 31));
    else
      dst[r][u] = 0.f;
  }
}

// (The warp as a whole: lanes that come out of a wait one by one would arrive
// for the others.)
__device__ __forceinline__ void wave_bar(int id, int threads) {
  __syncwarp();
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

__device__ __forceinline__ void wave_arrive(int id, int threads) {
  __threadfence_block();
  __syncwarp();
  asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

// The block's CTAs meet (cl of them; every thread).
__device__ __forceinline__ void wave_meet(int cl) {
  __syncwarp();
  if (cl == 1)
    wave_bar(0, kWaveThreads);
  else
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}

// The cluster's CTAs if there are the cl asked for, else one (a profiler may
// launch a cooperative grid without its clusters).
__device__ __forceinline__ int wave_cluster_size(int cl) {
  int n;
  asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(n));
  return n == cl ? cl : 1;
}

// The first CTA's word at the place of *p in shared memory.
__device__ __forceinline__ unsigned wave_peer(const void* p) {
  unsigned v;
  asm volatile(
      "{\n\t.reg .b32 r;\n\tmapa.shared::cluster.u32 r, %1, 0;\n\tld.shared::cluster.u32 %0, [r];\n\t}"
      : "=r"(v)
      : "r"((unsigned)__cvta_generic_to_shared(p))
      : "memory");
  return v;
}

// y[r] += the changes of a tile (rows 4 wid + r) times blk, the S block of
// its other side's rows: the row's changes in step order (columns
// downwards), with0: vertex 0's pair where the row would meet itself.
__device__ __forceinline__ void wave_apply(float (&y)[4], const float (*d)[16][16],
                                           const float (*blk)[kWaveB], const float* d0,
                                           const float* s0, bool with0, int par, int wid, int lane) {
#pragma unroll 4
  for (int k = 15; k >= 0; --k) {
    const float2 a = *reinterpret_cast<const float2*>(&d[0][k][2 * wid]);  // rows 0, 2
    const float2 b = *reinterpret_cast<const float2*>(&d[1][k][2 * wid]);  // rows 1, 3
    const float se = blk[2 * k + par][lane], so = blk[2 * k + (par ^ 1)][lane];
    y[0] = fmaf(a.x, se, y[0]);
    y[1] = fmaf(b.x, so, y[1]);
    y[2] = fmaf(a.y, se, y[2]);
    y[3] = fmaf(b.y, so, y[3]);
    if (with0) {
      const float z = s0[lane];
      if (k == 2 * wid) {
        y[0] = fmaf(d0[4 * wid], z, y[0]);
        y[1] = fmaf(d0[4 * wid + 1], z, y[1]);
      } else if (k == 2 * wid + 1) {
        y[2] = fmaf(d0[4 * wid + 2], z, y[2]);
        y[3] = fmaf(d0[4 * wid + 3], z, y[3]);
      }
    }
  }
}

// The own rows' changes of a tile with block Jb into every column but two
// blocks', by warp w of nw; the items of the first 64 columns by the first
// CTA's warps alone (column 0 is wanted early there).  An item is 64 columns
// of eight rows (row parity x half of the rows) of a matrix; of the rows of S
// that any of the eight needs eight are requested together, the others are
// not read.
// signal: barrier 3 hears of the first columns as soon as they are done.
template <int NM>
__device__ __forceinline__ void wave_bulk(const WaveArgs<NM>& a, const WaveSmem<NM>& s, int i0, int Jb,
                                          int db, bool with0, int par, int ex0, int ex1, int w, int nw,
                                          int nw0, int lane, bool signal) {
  const int p = a.p;
  const int nv = a.ld >> 1;
  const int n0 = 4 * NM, items = n0 * ((nv + 31) >> 5);
  for (int it = w < nw0 && w < n0 ? w : n0 + w; it < items;
       it = it >= n0 ? it + nw : (it + nw0 < n0 ? it + nw0 : n0 + w)) {
    if (signal && it >= n0) {
      wave_arrive(3, kWaveThreads);
      signal = false;
    }
    const int g = it & 3, rp = g & 1, hf = g >> 1;
    const int m = NM == 1 ? 0 : (it >> 2) % NM, q = 32 * ((it >> 2) / NM) + lane;
    const unsigned need = with0 ? 0xffffu : s.need[db][m][g];
    if (need == 0 || q >= nv || (q >> 4) == ex0 || (q >> 4) == ex1) continue;
    const int j = kWaveB * Jb + ((par ^ rp) & 1), i = i0 + 16 * hf + rp;  // every other row from there
    const float2* Sb = reinterpret_cast<const float2*>(a.S[m]) + (size_t)j * nv + q;
    float2* Wr = reinterpret_cast<float2*>(a.W[m]) + (size_t)i * nv + q;
    float2 acc[8], z = make_float2(0.f, 0.f);
#pragma unroll
    for (int r = 0; r < 8; ++r)
      acc[r] = i + 2 * r >= 1 && i + 2 * r < p ? __ldcg(Wr + 2 * r * nv) : make_float2(0.f, 0.f);
    if (with0) z = __ldg(reinterpret_cast<const float2*>(a.S[m]) + q);
    const float* dm = &s.d[db][m][rp][0][8 * hf];
#pragma unroll 1
    for (int k0 = 8; k0 >= 0; k0 -= 8) {
      float2 sv[8];
#pragma unroll
      for (int k = 7; k >= 0; --k)  // (a row past p has no change; with0 asks for every row)
        if ((need >> (k0 + k)) & 1)
          sv[k] = j + 2 * (k0 + k) < p ? __ldg(Sb + 2 * (k0 + k) * nv) : make_float2(0.f, 0.f);
#pragma unroll
      for (int k = 7; k >= 0; --k) {
        if (!((need >> (k0 + k)) & 1)) continue;
        const float4 d0 = *reinterpret_cast<const float4*>(dm + 16 * (k0 + k));
        const float4 d1 = *reinterpret_cast<const float4*>(dm + 16 * (k0 + k) + 4);
        const float dr[8] = {d0.x, d0.y, d0.z, d0.w, d1.x, d1.y, d1.z, d1.w};
#pragma unroll
        for (int r = 0; r < 8; ++r) {
          acc[r].x = fmaf(dr[r], sv[k].x, acc[r].x);
          acc[r].y = fmaf(dr[r], sv[k].y, acc[r].y);
        }
        if (with0 && k0 == 8 * hf) {  // the pair (0, i) stands where i would meet itself
          const float d = s.d0[db][m][2 * (k0 + k) + rp];
          acc[k].x = fmaf(d, z.x, acc[k].x);
          acc[k].y = fmaf(d, z.y, acc[k].y);
        }
      }
    }
#pragma unroll
    for (int r = 0; r < 8; ++r)
      if (i + 2 * r >= 1 && i + 2 * r < p) Wr[2 * r * nv] = acc[r];
  }
  if (signal) wave_arrive(3, kWaveThreads);
}

// x = lane's row of a skewed block.
__device__ __forceinline__ void wave_row(float (&x)[16], const float* row) {
#pragma unroll
  for (int u = 0; u < 16; u += 4) {
    const float4 v = *reinterpret_cast<const float4*>(row + u);
    x[u] = v.x;
    x[u + 1] = v.y;
    x[u + 2] = v.z;
    x[u + 3] = v.w;
  }
}

// x one step on, no change.
__device__ __forceinline__ void wave_turn(float (&x)[16]) {
  const float first = x[0];
#pragma unroll
  for (int u = 0; u < 15; ++u) x[u] = x[u + 1];
  x[15] = first;
}

// n / d, y the correctly rounded 1 / d: a quotient and its residual, twice.
// With y correctly rounded and the quotient within an ulp the last correction
// rounds correctly (Markstein, "Computation of elementary functions on the
// IBM RISC System/6000 processor", 1990, theorem 7), so the division, 360
// cycles of a step of 700 where its slow path is on the way, is done for a
// tile ahead (wave_reciprocals).  wave_plain: no intermediate is near the
// end of the range.
__host__ __device__ __forceinline__ bool wave_plain(float n, float d) {
  return (fabsf(n) >= 0x1p-70f || n == 0.f) && fabsf(n) <= 0x1p70f && d >= 0x1p-40f && d <= 0x1p40f;
}
__host__ __device__ __forceinline__ float wave_quotient(float n, float d, float y) {
  float q = n * y;
  q = fmaf(fmaf(-d, q, n), y, q);
  return fmaf(fmaf(-d, q, n), y, q);
}

// The lanes' j / 2 with changes, by row parity and half of the rows.
template <int NM>
__device__ __forceinline__ void wave_needs(WaveSmem<NM>& s, const unsigned (&need)[NM], int db, int lane) {
#pragma unroll
  for (int m = 0; m < NM; ++m) {
    const int g = (lane & 1) + 2 * (lane >> 4);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const unsigned v = __reduce_or_sync(0xffffffffu, g == k ? need[m] : 0u);
      if (lane == 0) s.need[db][m][k] = v;
    }
  }
}

// x = (x one step on) + d * row: entry u becomes what entry u + 1 was, and
// the one just met comes last (for a row whose first pair is yet to come it
// is the entry it meets 16 steps later).
__device__ __forceinline__ void wave_step(float (&x)[16], float d, const float* row) {
  const float first = x[0];
#pragma unroll
  for (int u = 0; u < 16; u += 4) {
    const float4 v = *reinterpret_cast<const float4*>(row + u);
    x[u] = fmaf(d, v.x, x[u + 1]);
    x[u + 1] = fmaf(d, v.y, x[u + 2]);
    x[u + 2] = fmaf(d, v.z, x[u + 3]);
    x[u + 3] = fmaf(d, v.w, u < 12 ? x[(u + 4) & 15] : first);
  }
}

// The colour steps of a tile off the diagonal, by two warps: lane l is row l
// of the own block (side 0) or of the other one (side 1).  hl, ll: the sums
// less i0 + j0.  A step: the two warps swap the entries at hand, both compute
// the pairs.  Two matrices: where none of the 32 pairs is or becomes nonzero
// (at few edges most steps) that is all; one matrix comes here when it has
// many edges, and 94% of the steps have some.
template <int NM, class Ops>
__device__ __forceinline__ void wave_chain(int p, WaveSmem<NM>& s, Ops& ops, int i0, int j0, int hl,
                                           int ll, int db, int tb, int ob, int lane, int side) {
  constexpr unsigned FULL = 0xffffffffu;
  constexpr int KD = 2 * NM - 1;
  const int own0 = side ? j0 : i0, oth0 = side ? i0 : j0;  // first rows: own side's, other side's
  const bool ok = own0 + lane >= 1 && own0 + lane < p;
  const bool lo = (i0 < j0) == (side == 0);  // the own entry is W_lo,hi
  const float* T = side ? &s.ti[0][0][0] : &s.tj[tb][0][0][0];
  const float* sdo = side ? s.sdi[0] : s.sd[tb][0];
  const int oml = side ? 1 : kWaveB, omr = side ? kWaveB : 1;  // strides of (lane, partner) in a tile
  float x[NM][16], sdl[NM], om[NM], c[NM], rc[KD];
  unsigned need[NM];
  // what the step with sum sl needs and does not wait for
  auto operands = [&](int sl) {
    const int rm = (sl - lane) & 31;
#pragma unroll
    for (int m = 0; m < NM; ++m) {
      om[m] = (&s.om[ob][m][0][0])[oml * lane + omr * rm];
      c[m] = sdl[m] + sdo[kWaveB * m + rm];
    }
#pragma unroll
    for (int k = 0; k < KD; ++k) rc[k] = (&s.rc[tb][k][0][0])[oml * lane + omr * rm];
  };
#pragma unroll
  for (int m = 0; m < NM; ++m) {
    wave_row(x[m], side ? s.b[m][lane] : s.a[m][lane]);
    sdl[m] = side ? s.sd[tb][m][lane] : s.sdi[m][lane];
    need[m] = 0;
  }
  operands(hl);
  int bf = 0;
#pragma unroll 1
  for (int sl = hl; sl >= ll; sl -= 2, bf ^= 1) {
    const int r = sl - lane, rm = r & 31;
    const bool on = ok && r == rm && oth0 + r >= 1 && oth0 + r < p;
#pragma unroll
    for (int m = 0; m < NM; ++m) s.x[bf][side][m][lane] = x[m][0];
    wave_bar(4, 64);
    float wa[NM], wb[NM], n[NM], dn[NM], y[NM], o[NM];
#pragma unroll
    for (int m = 0; m < NM; ++m) {
      const float w = s.x[bf][side ^ 1][m][rm];
      wa[m] = lo ? x[m][0] : w;
      wb[m] = lo ? w : x[m][0];
      o[m] = om[m];
    }
    ops.pair(c, rc, om, wa, wb, n, dn, y);
    operands(sl - 2);
    bool loud = false;
#pragma unroll
    for (int m = 0; m < NM; ++m) loud = loud || n[m] != 0.f || o[m] != 0.f;
    if (NM == 1 || __any_sync(FULL, loud && on)) {
      float d[NM];
      bool plain = true;
#pragma unroll
      for (int m = 0; m < NM; ++m) {
        d[m] = wave_quotient(n[m], dn[m], y[m]);
        plain = plain && wave_plain(n[m], dn[m]);
      }
      if (__any_sync(FULL, on && !plain))
#pragma unroll
        for (int m = 0; m < NM; ++m) d[m] = n[m] != 0.f ? n[m] / dn[m] : 0.f;
#pragma unroll
      for (int m = 0; m < NM; ++m) {
        const float nw = d[m];
        d[m] = on ? nw - o[m] : 0.f;
        if (on && side == 0) {
          s.d[db][m][lane & 1][r >> 1][lane >> 1] = d[m];
          s.om[ob][m][lane][r] = nw;
        }
        need[m] |= d[m] != 0.f ? 1u << (rm >> 1) : 0u;
        wave_step(x[m], d[m], T + (m * kWaveB + rm) * kWaveSkew);
      }
      if (side == 0) ops.count(d);
    } else {
#pragma unroll
      for (int m = 0; m < NM; ++m) wave_turn(x[m]);
    }
  }
  if (side == 0) wave_needs<NM>(s, need, db, lane);
}

// The colour steps of a diagonal tile: lane l is row l; with0: a row that
// would meet itself meets vertex 0, whose entries of the own columns the
// lanes hold as well.
template <int NM, class Ops>
__device__ __forceinline__ void wave_chain_diag(const WaveArgs<NM>& a, WaveSmem<NM>& s, Ops& ops, int i0,
                                                int hl, int ll, bool with0, int db, int ob, int lane) {
  constexpr unsigned FULL = 0xffffffffu;
  const int p = a.p, i = i0 + lane;
  const bool iok = i >= 1 && i < p;
  constexpr int KD = 2 * NM - 1;
  float x[NM][16], e[NM], z[NM], sdl[NM], om[NM], c[NM], rc[KD];
  unsigned need[NM];
#pragma unroll
  for (int m = 0; m < NM; ++m) {
    wave_row(x[m], s.a[m][lane]);
    e[m] = with0 ? s.e[m][lane] : 0.f;
    z[m] = with0 ? s.z[m][lane] : 0.f;
    sdl[m] = s.sdi[m][lane];
    need[m] = 0;
    if (with0) s.d0[db][m][lane] = 0.f;
  }
  // what the step with sum sl needs and does not wait for
  auto operands = [&](int sl) {
    const int rm = (sl - lane) & 31;
    const bool self = sl - lane == lane;
#pragma unroll
    for (int m = 0; m < NM; ++m) {
      om[m] = *(self ? &s.om0[m][lane] : &s.om[ob][m][lane][rm]);
      c[m] = sdl[m] + *(self ? &s.sd0[m] : &s.sdi[m][rm]);
    }
#pragma unroll
    for (int k = 0; k < KD; ++k) rc[k] = *(self ? &s.rz[k][lane] : &s.rc[db][k][lane][rm]);
  };
  operands(hl);
#pragma unroll 1
  for (int sl = hl; sl >= ll; sl -= 2) {
    const int r = sl - lane, rm = r & 31;
    const bool self = r == lane;  // even sums: with0
    const int j = self ? 0 : i0 + r;
    const bool on = iok && r == rm && (self || (j >= 1 && j < p));
    float d[NM], wa[NM], wb[NM], n[NM], dn[NM], y[NM], nw[NM], o[NM];
#pragma unroll
    for (int m = 0; m < NM; ++m) {
      const float wp = __shfl_sync(FULL, x[m][0], rm);
      const float wu = self ? e[m] : x[m][0], wv = self ? z[m] : wp;
      wa[m] = i < j ? wu : wv;
      wb[m] = i < j ? wv : wu;
      o[m] = om[m];
    }
    ops.pair(c, rc, om, wa, wb, n, dn, y);
    operands(sl - 2);
    bool loud = false;
#pragma unroll
    for (int m = 0; m < NM; ++m) loud = loud || n[m] != 0.f || o[m] != 0.f;
    if (NM == 1 || __any_sync(FULL, loud && on)) {  // (as in wave_chain)
      bool plain = true;
#pragma unroll
      for (int m = 0; m < NM; ++m) {
        nw[m] = wave_quotient(n[m], dn[m], y[m]);
        plain = plain && wave_plain(n[m], dn[m]);
      }
      if (__any_sync(FULL, on && !plain))
#pragma unroll
        for (int m = 0; m < NM; ++m) nw[m] = n[m] != 0.f ? n[m] / dn[m] : 0.f;
#pragma unroll
      for (int m = 0; m < NM; ++m) {
        d[m] = on ? nw[m] - o[m] : 0.f;
        if (on && !self) {
          s.d[db][m][lane & 1][r >> 1][lane >> 1] = d[m];
          s.om[ob][m][lane][r] = nw[m];
          need[m] |= d[m] != 0.f ? 1u << (r >> 1) : 0u;
        }
        if (on && self) {  // (to memory and the other blocks after the steps)
          s.d0[db][m][lane] = d[m];
          s.nw0[m][lane] = nw[m];
        }
      }
      ops.count(d);
      if (with0) {  // vertex 0's row
        float d0[NM];
#pragma unroll
        for (int m = 0; m < NM; ++m) d0[m] = self ? d[m] : 0.f;
        ops.count(d0);
      }
      const int vz = (sl >> 1) & 31;
      const bool zon = with0 && (sl & ~63) == 0;
#pragma unroll
      for (int m = 0; m < NM; ++m) {
        wave_step(x[m], d[m], self ? s.t0[m][lane] : s.ti[m][rm]);
        if (zon) {
          e[m] = fmaf(d[m], self ? s.s00[m] : s.si0[m][rm], e[m]);
          z[m] = fmaf(__shfl_sync(FULL, d[m], vz), s.sii[m][vz][lane], z[m]);
        }
      }
    } else {
#pragma unroll
      for (int m = 0; m < NM; ++m) wave_turn(x[m]);
    }
  }
#pragma unroll
  for (int m = 0; m < NM; ++m)
    if (with0) s.z[m][lane] = z[m];
  wave_needs<NM>(s, need, db, lane);
}

// (Named in a function of its own so that the accesses are shared ones.)
template <int NM>
__device__ __forceinline__ WaveSmem<NM>& wave_smem() {
  extern __shared__ __align__(16) unsigned char wave_dyn[];
  return *reinterpret_cast<WaveSmem<NM>*>(wave_dyn);
}

// The sweep; wave_smem().args are set.  Ops: denominators(c, dn): all a
// pair's new values may be divided by, c_m = s_ii + s_jj; pair(c, rc, om, wa,
// wb, n, dn, y): the new values n / dn of a pair from c, the denominators'
// reciprocals, its old values and W_lo,hi, W_hi,lo, y = 1 / dn out of rc
// (without branches, for lanes without a pair as well); count(d): once per owned row and pair, or with zeros; diag(args, i, w, dd): row
// i's diagonal change from W_ii (stores the new diagonal).  I: the block, rank:
// the CTA of its cl (a cluster).  One sweep per launch: in a kernel that loops over sweeps the
// compiler keeps enough beside it to spill in the colour steps (1.5x).
template <int NM, class Ops>
__device__ __forceinline__ void wave_sweep(int I, int rank, int cl, Ops& ops) {
  constexpr unsigned FULL = 0xffffffffu;
  WaveSmem<NM>& s = wave_smem<NM>();
  const WaveArgs<NM>& a = s.args;
  const int tid = (int)threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const bool chain = wid < 2;
  const bool front = !chain && tid < kWaveFirst;       // the next tile's columns
  const bool rest = tid >= kWaveFirst;                 // the other columns
  const bool zwarp = wid == kWaveThreads / 32 - 1;     // of the rest: keeps vertex 0's row, too
  const int rt = tid - kWaveFirst;
  const int p = a.p, P = a.P, ld = a.ld, nb = wave_blocks(p), slots = wave_slots(p);
  const int nv = ld >> 2;
  const int i0 = kWaveB * I;  // first own row
  const int fw = wid - 2, ft = tid - 64;  // front: warp, thread
  const int ir = i0 + 4 * fw;             // front: own rows ir .. ir + 3
  unsigned long long* const zw = a.words + (size_t)NM * nb * slots * kWaveWords;  // [NM][32 nb]
  auto slot_words = [&](int b, int slot, int m) {
    return a.words + (((size_t)b * slots + slot) * NM + m) * kWaveWords;
  };
  auto own = [&](int r) { return front && ir + r >= 1 && ir + r < p; };  // not vertex 0's row
  // the own rows' entries of column c
  auto load_rows = [&](int m, int c, float (&y)[4]) {
#pragma unroll
    for (int r = 0; r < 4; ++r) y[r] = own(r) ? __ldcg(a.W[m] + (size_t)(ir + r) * ld + c) : 0.f;
  };
  // rest: the operands of tile t (after a tile with block Jq, before nx; omb:
  // the buffer for Omega, -1: it is there) on their way
  auto fetch = [&](const WaveTile& t, int Jq, const WaveTile& nx, int tb, int omb) {
    const int j0 = kWaveB * t.J, n0 = kWaveB * nx.J;
#pragma unroll
    for (int m = 0; m < NM; ++m) {
      if (t.J != I) wave_load_skewed(s.tj[tb][m], a.S[m], j0, j0, p, ld, rt, kWaveRest);
      if (omb >= 0) wave_load(s.om[omb][m], a.Om[m], i0, j0, p, ld, rt, kWaveRest);
      if (nx.J >= 0) {
        wave_load(s.sjn[tb][m], a.S[m], j0, n0, p, ld, rt, kWaveRest);
        if (Jq >= 0) wave_load(s.spn[tb][m], a.S[m], kWaveB * Jq, n0, p, ld, rt, kWaveRest);
      }
      if (rt < kWaveB) {
        if (j0 + rt < p)
          cp_async4(&s.sd[tb][m][rt], a.sdiag[m] + (size_t)(j0 + rt) * a.sd_stride);
        else
          s.sd[tb][m][rt] = 1.f;
        if (nx.J >= 0) cp_async4(&s.s0n[tb][m][rt], a.S[m] + n0 + rt);
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  // rest: the reciprocals tile t's pairs need (divisions: after what others wait for)
  auto reciprocals = [&](const WaveTile& t, int tb) {
    const int j0 = kWaveB * t.J;
    for (int e = rt; e < kWaveB * kWaveB; e += kWaveRest) {
      const int i = i0 + e / kWaveB, j = j0 + e % kWaveB;
      float c[NM], dn[2 * NM - 1];
#pragma unroll
      for (int k = 0; k < NM; ++k)
        c[k] = i < p && j < p ? __ldg(a.sdiag[k] + (size_t)i * a.sd_stride) +
                                    __ldg(a.sdiag[k] + (size_t)j * a.sd_stride)
                              : 1.f;
      Ops::denominators(c, dn);
#pragma unroll
      for (int k = 0; k < 2 * NM - 1; ++k) (&s.rc[tb][k][0][0])[e] = 1.f / dn[k];
    }
  };
  // front: a tile's entries to the partner ((row + column) parity picks two rows per lane)
  auto publish = [&](const WaveTile& t, const float (&y)[NM][4]) {
    const int rb = (t.hi ^ lane) & 1;
#pragma unroll
    for (int m = 0; m < NM; ++m)
      st_relaxed_v2u64(slot_words(I, t.slot, m) + 2 * ft, wave_word(a.tag, rb ? y[m][1] : y[m][0]),
                       wave_word(a.tag, rb ? y[m][3] : y[m][2]));
  };

  const int nw = kWaveRestWarps + kWaveWarps * (cl - 1);  // warps for the other columns
  // The last tile's changes into the own rows, the diagonal's after them;
  // helpers take the changes from the first CTA's shared memory.
  auto copy_changes = [&](int db) {
    for (int m = 0; m < NM; ++m) {
      float* d = reinterpret_cast<float*>(s.d[db][m]);
      d[tid] = __uint_as_float(wave_peer(d + tid));
      if (tid < kWaveB) s.d0[db][m][tid] = __uint_as_float(wave_peer(&s.d0[db][m][tid]));
      if (tid < 4) s.need[db][m][tid] = wave_peer(&s.need[db][m][tid]);
    }
    wave_bar(0, kWaveThreads);
  };
  auto last = [&](int Jp, int v, bool diag0, int par_p) {
    if (Jp >= 0) {
      if (rank > 0) copy_changes((v - 1) & 1);
      wave_bulk<NM>(a, s, i0, Jp, (v - 1) & 1, diag0, par_p, -1, -1, kWaveWarps * rank + wid,
                    kWaveWarps * cl, kWaveWarps, lane, false);
    }
    wave_meet(cl);
  };
  auto diagonal = [&]() {
    wave_meet(cl);
    if (rank > 0) {
      for (int m = 0; m < NM; ++m)
        if (tid < kWaveB) s.dd[m][tid] = __uint_as_float(wave_peer(&s.dd[m][tid]));
      wave_bar(0, kWaveThreads);
    }
    for (int k = kWaveWarps * rank + wid; k < NM * kWaveB; k += kWaveWarps * cl) {
      const int m = NM == 1 ? 0 : k % NM, r = k / NM;
      const float d = s.dd[m][r];
      if (d == 0.f || i0 + r >= p) continue;
      float4* w = reinterpret_cast<float4*>(a.W[m] + (size_t)(i0 + r) * ld);
      const float4* sr = reinterpret_cast<const float4*>(a.S[m] + (size_t)(i0 + r) * ld);
      for (int q0 = lane; q0 < nv; q0 += 128) {
        float4 x[4], y[4];  // requested together
#pragma unroll
        for (int e = 0; e < 4; ++e)
          if (q0 + 32 * e < nv) {
            x[e] = __ldcg(w + q0 + 32 * e);
            y[e] = __ldg(sr + q0 + 32 * e);
          }
#pragma unroll
        for (int e = 0; e < 4; ++e)
          if (q0 + 32 * e < nv) {
            x[e].x = fmaf(d, y[e].x, x[e].x);
            x[e].y = fmaf(d, y[e].y, x[e].y);
            x[e].z = fmaf(d, y[e].z, x[e].z);
            x[e].w = fmaf(d, y[e].w, x[e].w);
            w[q0 + 32 * e] = x[e];
          }
      }
    }
    if (cl > 1) wave_meet(cl);  // (the first CTA's shared memory is read)
  };

  if (rank > 0) {  // a helper: its share of every tile's changes
    WaveTile t = wave_tile(I, nb, P, 0);
    int Jp = -1, par_p = 0, v = 0;
    bool diag0 = false;
    for (; t.J >= 0; ++v) {
      const WaveTile nx = wave_tile(I, nb, P, v + 1);
      if (Jp >= 0) {
        copy_changes((v - 1) & 1);
        wave_bulk<NM>(a, s, i0, Jp, (v - 1) & 1, diag0, par_p, t.J, nx.J,
                      kWaveRestWarps + kWaveWarps * (rank - 1) + wid, nw, kWaveRestWarps, lane, false);
      }
      diag0 = I == t.J && (t.hi & 1) == 0;
      par_p = t.hi & 1;
      Jp = t.J;
      t = nx;
      wave_meet(cl);
    }
    last(Jp, v, diag0, par_p);
    diagonal();
    return;
  }

  // ---- what stays for the whole sweep
  WaveTile t = wave_tile(I, nb, P, 0);
  WaveTile nx = wave_tile(I, nb, P, 1);  // rest: the tile after t
  if (wid == 0) {
    float c[NM], dn[2 * NM - 1];
#pragma unroll
    for (int m = 0; m < NM; ++m)
      c[m] = i0 + lane < p ? a.sdiag[m][(size_t)(i0 + lane) * a.sd_stride] + a.sdiag[m][0] : 1.f;
    Ops::denominators(c, dn);
#pragma unroll
    for (int k = 0; k < 2 * NM - 1; ++k) s.rz[k][lane] = 1.f / dn[k];
  }
  float Z[NM];  // zwarp: W_0 in the own columns
#pragma unroll
  for (int m = 0; m < NM; ++m) {
    if (rest) {
      wave_load(s.sii[m], a.S[m], i0, i0, p, ld, rt, kWaveRest);
      wave_load_skewed(s.ti[m], a.S[m], i0, i0, p, ld, rt, kWaveRest);
      wave_load_skewed(s.t0[m], a.S[m], 0, i0, p, 0, rt, kWaveRest);
    }
    if (wid == 0) {
      s.sdi[m][lane] = i0 + lane < p ? a.sdiag[m][(size_t)(i0 + lane) * a.sd_stride] : 1.f;
      s.s0[m][lane] = a.S[m][i0 + lane];
      s.si0[m][lane] = i0 + lane < p ? a.S[m][(size_t)(i0 + lane) * ld] : 0.f;
      s.om0[m][lane] = a.Om[m][i0 + lane];
      if (lane == 0) {
        s.s00[m] = a.S[m][0];
        s.sd0[m] = a.sdiag[m][0];
      }
    }
    Z[m] = zwarp ? __ldcg(a.W[m] + i0 + lane) : 0.f;
  }
  if (rest) {
    fetch(t, -1, nx, 0, 0);
    reciprocals(t, 0);
    asm volatile("cp.async.wait_group 0;" ::: "memory");
  }
  int zdone = nb;  // zwarp: the changes of vertex 0's pairs in blocks >= zdone are in Z
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
  __syncthreads();

  // Per tile: barrier 1, the steps may start; 2, they are done; 3 (with
  // vertex 0's pairs), column 0 of the own rows and Z are up to date; then
  // the block's CTAs meet.
  int Jp = -1;         // the previous tile's block (its changes are not yet in the other columns)
  bool diag0 = false;  // that tile held vertex 0's pairs
  int par_p = 0;       // its sums' parity
  int v = 0;
  if (chain) {
    int ob = 0;  // Omega's buffer
    for (; t.J >= 0; ++v) {
      const int J = t.J, j0 = kWaveB * J;
      const bool with0 = I == J && (t.hi & 1) == 0;  // the tile holds vertex 0's pairs
      if (with0) wave_bar(3, kWaveThreads);
      wave_bar(1, kWaveFirst);
      if (I == J && wid == 0)
        wave_chain_diag<NM>(a, s, ops, i0, t.hi - i0 - j0, t.lo - i0 - j0, with0, v & 1, ob, lane);
      else if (I != J)
        wave_chain<NM>(p, s, ops, i0, j0, t.hi - i0 - j0, t.lo - i0 - j0, v & 1, v & 1, ob, lane, wid);
      wave_bar(2, kWaveFirst);  // the tile's changes are in s.d
      diag0 = with0;
      par_p = t.hi & 1;
      t = wave_tile(I, nb, P, v + 1);
      if (t.J != J) ob ^= 1;
      Jp = J;
      wave_meet(cl);
    }
  } else if (front) {
    int ob = 0;
    float A[NM][4];  // W_I,J: own rows, column 32 J + lane
#pragma unroll
    for (int m = 0; m < NM; ++m) load_rows(m, kWaveB * t.J + lane, A[m]);
    if (t.J != I) publish(t, A);
    for (; t.J >= 0; ++v) {
      const int J = t.J, j0 = kWaveB * J, db = v & 1, par = t.hi & 1, hl = t.hi - i0 - j0;
      const bool dt = I == J, with0 = dt && par == 0;
      const int rb = (par ^ lane) & 1;  // rows rb, rb + 2 of a warp meet column `lane` in this tile
      // the columns go to memory (further changes: with the other columns),
      // the pairs' entries to the steps
#pragma unroll
      for (int m = 0; m < NM; ++m) {
#pragma unroll
        for (int r = 0; r < 4; ++r)
          if (own(r)) a.W[m][(size_t)(ir + r) * ld + j0 + lane] = A[m][r];
        const int l = 4 * fw + rb, u = (hl - l - lane) >> 1;
        s.a[m][l][u & 15] = rb ? A[m][1] : A[m][0];
        s.a[m][l + 2][(u - 1) & 15] = rb ? A[m][3] : A[m][2];
        float* d = reinterpret_cast<float*>(s.d[db][m]);
        d[ft] = d[ft + 256] = 0.f;
        if (!dt) {
          const unsigned long long* w = slot_words(J, t.slot, m) + 2 * ft;
          s.b[m][l][u & 15] = wave_wait(w, a.tag, a.wait, j0 + l, t.slot);
          s.b[m][l + 2][(u - 1) & 15] = wave_wait(w + 1, a.tag, a.wait, j0 + l + 2, t.slot);
        }
      }
      if (!with0) wave_bar(1, kWaveFirst);
      const WaveTile nx = wave_tile(I, nb, P, v + 1);
      // the next tile's columns with the previous tile's changes
      float N[NM][4];
      if (nx.J >= 0 && nx.J != J) {
#pragma unroll
        for (int m = 0; m < NM; ++m) load_rows(m, kWaveB * nx.J + lane, N[m]);
        if (Jp >= 0)
#pragma unroll
          for (int m = 0; m < NM; ++m)
            wave_apply(N[m], s.d[db ^ 1][m], s.spn[db][m], s.d0[db ^ 1][m], s.s0n[db][m], diag0, par_p, fw,
                       lane);
      } else {
#pragma unroll
        for (int m = 0; m < NM; ++m)
#pragma unroll
          for (int r = 0; r < 4; ++r) N[m][r] = A[m][r];
      }
      if (with0) {
        wave_bar(3, kWaveThreads);
#pragma unroll
        for (int m = 0; m < NM; ++m) {  // column 0 of the own rows: lane 0 where it is in registers
          float e[4];
          if (J != 0 && nx.J != 0) load_rows(m, 0, e);
#pragma unroll
          for (int r = 0; r < 4; ++r)
            if (lane == 0) s.e[m][4 * fw + r] = J == 0 ? A[m][r] : (nx.J == 0 ? N[m][r] : e[r]);
        }
        wave_bar(1, kWaveFirst);
      }
      wave_bar(2, kWaveFirst);
      if (nx.J >= 0) {
#pragma unroll
        for (int m = 0; m < NM; ++m) {
          wave_apply(N[m], s.d[db][m], s.sjn[db][m], s.d0[db][m], s.s0n[db][m], with0, par, fw, lane);
#pragma unroll
          for (int r = 0; r < 4; ++r) A[m][r] = N[m][r];
        }
        if (nx.J != I) publish(nx, A);
      }
      if (with0 && fw == 0 && 2 * lane >= t.lo - i0 - j0 && 2 * lane <= hl && i0 + lane >= 1 && i0 + lane < p)
#pragma unroll
        for (int m = 0; m < NM; ++m) {  // vertex 0's pairs: to its row's holders, and to memory
          const float d = s.d0[db][m][lane];
          st_relaxed_u64(zw + (size_t)m * kWaveB * nb + i0 + lane, wave_word(a.tag, d));
          if (d != 0.f)
            a.Om[m][(size_t)(i0 + lane) * ld] = a.Om[m][i0 + lane] = s.nw0[m][lane];
        }
#pragma unroll
      for (int m = 0; m < NM; ++m)  // (column 0 is kept by vertex 0's pairs)
        if ((s.need[db][m][0] | s.need[db][m][1] | s.need[db][m][2] | s.need[db][m][3]) != 0) {
#pragma unroll
          for (int r = 0; r < 4; ++r)
            if (own(r) && j0 + lane > 0)
              a.Om[m][(size_t)(ir + r) * ld + j0 + lane] = s.om[ob][m][4 * fw + r][lane];
        }
      if (nx.J != J) ob ^= 1;
      diag0 = with0;
      par_p = par;
      t = nx;
      Jp = J;
      wave_meet(cl);
    }
  } else {
    int ob = 0;
    for (; t.J >= 0; ++v) {
      const int J = t.J, db = v & 1;
      const bool with0 = I == J && (t.hi & 1) == 0;
      if (nx.J >= 0) fetch(nx, J, wave_tile(I, nb, P, v + 2), db ^ 1, nx.J == J ? -1 : ob ^ 1);
      if (zwarp && with0) {
        while (zdone - 1 > I) zapply(--zdone, true);
#pragma unroll
        for (int m = 0; m < NM; ++m) s.z[m][lane] = Z[m];
      }
      if (Jp >= 0)
        wave_bulk<NM>(a, s, i0, Jp, db ^ 1, diag0, par_p, J, nx.J, wid - kWaveFirst / 32, nw,
                      kWaveRestWarps, lane, with0);
      else if (with0)
        wave_arrive(3, kWaveThreads);
      if (nx.J >= 0) reciprocals(nx, db ^ 1);
      if (zwarp && !with0)
        while (zdone > 0 && zdone - 1 != I && zapply(zdone - 1, false)) --zdone;
      asm volatile("cp.async.wait_group 0;" ::: "memory");
      if (nx.J != J) ob ^= 1;
      diag0 = with0;
      par_p = t.hi & 1;
      t = nx;
      Jp = J;
      nx = t.J >= 0 ? wave_tile(I, nb, P, v + 2) : t;
      wave_meet(cl);
      if (with0) {
        zdone = I;  // vertex 0's changes of the own block are in Z
#pragma unroll
        for (int m = 0; m < NM; ++m)
          if (zwarp) Z[m] = s.z[m][lane];
      }
    }
  }
  // ---- the last tile's changes; vertex 0's remaining changes
  if (zwarp)
    while (zdone > 0) zapply(--zdone, true);
  last(Jp, v, diag0, par_p);
  // ---- diagonal step: one lane per row (row 0: the owner of block 0)
  if (zwarp) {
    float w[NM], dd[NM];
    const int i = i0 + lane;
#pragma unroll
    for (int m = 0; m < NM; ++m) {
      dd[m] = 0.f;
      w[m] = i == 0 ? Z[m] : (i < p ? __ldcg(a.W[m] + (size_t)i * ld + i) : 0.f);
    }
    if (i < p) ops.diag(a, i, w, dd);
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
  diagonal();
}

// CTAs per block: as many as have items, if all `blocks` clusters fit on the
// device at once.
inline cudaError_t wave_cluster(const void* fn, int blocks, int nm, int p, size_t dyn, int* cl) {
  const int items = 4 * nm * ((p + 63) / 64);
  int c = kWaveCluster;
  while (c > 1 && items <= kWaveRestWarps + kWaveWarps * (c / 2 - 1)) c /= 2;
  for (; c > 1; c /= 2) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(blocks * c);
    cfg.blockDim = dim3(kWaveThreads);
    cfg.dynamicSmemBytes = dyn;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = c;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int n = 0;
    const cudaError_t e = cudaOccupancyMaxActiveClusters(&n, fn, &cfg);
    if (e != cudaSuccess) return e;
    if (n >= blocks) break;
  }
  *cl = c;
  return cudaSuccess;
}

// One sweep: `blocks` clusters of cl CTAs, all of them resident.
template <class... P, class... A>
cudaError_t wave_launch(void (*fn)(P...), int blocks, int cl, size_t dyn, cudaStream_t st, A... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(blocks * cl);
  cfg.blockDim = dim3(kWaveThreads);
  cfg.dynamicSmemBytes = dyn;
  cfg.stream = st;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeCooperative;
  at[0].val.cooperative = 1;
  at[1].id = cudaLaunchAttributeClusterDimension;
  at[1].val.clusterDim.x = cl;
  at[1].val.clusterDim.y = at[1].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = cl > 1 ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, fn, args...);
}

}  // namespace concord
