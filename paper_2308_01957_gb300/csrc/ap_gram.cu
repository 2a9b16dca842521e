// J^T W J for the Levenberg-Marquardt step (Sec. "Optimization methods").
//
// J is never stored whole (the paper names its N_pixels x N_parameters memory
// as LM's drawback): the columns of each source are stored on that source's
// support only.
//
// Pass 1 forms the Gram matrix of every 16 x 16 image tile's free columns and
// stores it, cut into the blocks of its source pairs, into a scratch array
// where every source pair keeps its tiles' blocks one after another (offsets
// planned on the host).  Pass 2 adds each pair's blocks in a fixed order and
// writes each sum into the compressed-sparse-row J^T W J (and its mirror),
// with plain stores where no other pair adds to the same entries (a shared
// parameter, as in joint fits, makes float64 atomics necessary).  No searches
// in the CSR and one write per entry instead of one atomic per tile.
//
// Float path.  The columns come sqrt(w)-scaled in tile blocks (a column's 256
// pixels of a tile in one kilobyte, zero outside the support), so a tile is
// one bulk copy per column, without addresses, bounds or weights per pixel.
// The products are 3xTF32 warp MMAs (m16n8k8; head x tail, tail x head, head
// x head; the tail x tail term is below float32 rounding).  A warp holds the
// accumulators of the whole upper triangle (up to 96 columns: 42 MMA tiles, 168
// registers) and takes 64 of the tile's 256 pixels, so each value is read from
// shared memory and split exactly once per tile, and the A and B fragments are
// the same registers.  The four warps' 64-pixel float32 sums are joined by
// compensated additions and kept as an unevaluated pair hi + lo of floats
// (float64 conversions and additions for every entry of every tile would
// occupy the thin float64 pipe longer than the MMAs take); the pair keeps about 48
// bits of sums of float32 products.  A 48-column tile is 1152 MMAs, 2300 clocks of an
// SM at the measured 303 TFLOP/s; the kernel takes some three times that (tensor
// pipe 27 to 31 % busy on the two largest forms), because a CTA loads, multiplies
// and writes one tile after the other and two to six CTAs an SM, as many as the
// registers allow, do not cover it.  tcgen05 does not pay at these shapes: its M = 128 by
// N = C MMA reads 4 + C/32 KB of operands from shared memory for
// 128 x C x 8 products, so a 48-column tile takes some 1400 clocks of
// shared-memory bandwidth for the MMAs and 1150 more to split and store both
// halves of the operands -- no less than the warp MMAs; as built before (producer
// warps gathering columns and storing swizzled heads and tails) it took 21 700
// clocks per tile.  J^T W J of the 12 x 2048^2 joint fit (196 608 tiles, 38
// columns on average) 14.2 -> 6.1 ms, of the 1536^2 crowded field 1.43 -> 0.71 ms,
// of 64 cutouts 230 -> 84 us (5.5, 0.65 and 80 before each MMA step was summed
// outside the accumulator).
//
// Float64 path: one CTA per tile, columns gathered into shared memory, products
// on the CUDA cores, float64 blocks.
#include <algorithm>
#include <type_traits>

#include "ap_internal.cuh"

namespace ap {

// ---------------------------------------------------------------------------
// float path, pass 1
// ---------------------------------------------------------------------------
namespace {

constexpr int GT_THREADS = 128;                 // four warps of 64 pixels
constexpr uint32_t GT_WAIT_LIMIT = 1u << 16;    // mbarrier polls before giving up
// Column pitch in shared memory: 32 bytes past a multiple of 128, so that the
// eight columns x four pixel pairs of a fragment load (8 bytes a lane, half a
// warp at a time) fall on 32 different banks.
constexpr int GT_PITCH = TILE_THREADS * 4 + 32;       // whole tile (diagonal jobs)
constexpr int GT_PITCH_H = TILE_THREADS * 2 + 32;     // half a tile (off-diagonal jobs)

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ uint32_t tf32_of(float x) {
  uint32_t r;
  asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
  return r;
}

__device__ __forceinline__ void split_tf32(float x, uint32_t& hi, uint32_t& lo) {
  hi = tf32_of(x);
  lo = tf32_of(x - __uint_as_float(hi));
}

__device__ __forceinline__ void mma_tf32(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                         uint32_t b0, uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
               "{%0,%1,%2,%3};"
               : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
               : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

__device__ __forceinline__ void bulk_load(uint32_t dst, const float* src, uint32_t bytes, uint32_t mbar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "l"(src), "r"(bytes), "r"(mbar)
               : "memory");
}

__device__ __forceinline__ bool mbar_wait(uint32_t mbar, uint32_t parity) {
  for (uint32_t it = 0; it < GT_WAIT_LIMIT; ++it) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred P1;\n\tmbarrier.try_wait.parity.shared::cta.b64 P1, [%1], %2;\n\t"
        "selp.b32 %0, 1, 0, P1;\n\t}\n"
        : "=r"(done)
        : "r"(mbar), "r"(parity)
        : "memory");
    if (done) return true;
  }
  return false;
}

// one kind of fragment: 8 columns x 8 pixels, split; the lane's column is
// `gid` of the group, its pixels 2 tig and 2 tig + 1 of the step (any
// assignment of pixels to the MMA's k serves, as A and B take the same one)
struct Frag {
  uint32_t h0, h1, l0, l1;
};
__device__ __forceinline__ void frag_load(Frag& f, const unsigned char* p) {
  const float2 v = *reinterpret_cast<const float2*>(p);
  split_tf32(v.x, f.h0, f.l0);
  split_tf32(v.y, f.h1, f.l1);
}

// one 8-pixel step of NM x NN MMA tiles: A = column groups 2m, 2m + 1 of fa,
// B = group n of fb; DIAG: only n >= 2m (the upper triangle).  Up to GRP tiles
// go through the three products together, so that consecutive MMAs are
// independent; the small terms first.  The tensor core truncates when it adds
// to its accumulator, so a step starts from zero and its sum joins the running
// one by a rounded float32 addition.  Accumulating in the MMA over the 64 pixels
// left 1.9 times the error in the entries (7e-8 against 3.7e-8 rms of
// sqrt(A_pp A_qq) on a crowded 96 x 160 field) and, the truncation being biased,
// ten times the error in that field's ill-conditioned LM step; the additions
// cost 10 % of the kernel.
template <int NM, int NN, bool DIAG>
__device__ __forceinline__ void mma_step(float (&d)[NM][NN][4], const Frag* fa, const Frag* fb) {
  constexpr int GRP = 8;
#pragma unroll
  for (int m = 0; m < NM; ++m) {
    const Frag &a = fa[2 * m], &b = fa[2 * m + 1];
#pragma unroll
    for (int n0 = DIAG ? 2 * m : 0; n0 < NN; n0 += GRP) {
      float t[GRP][4];
#pragma unroll
      for (int u = 0; u < GRP; ++u) {
        t[u][0] = t[u][1] = t[u][2] = t[u][3] = 0.f;
        if (n0 + u < NN) mma_tf32(t[u], a.h0, b.h0, a.h1, b.h1, fb[n0 + u].l0, fb[n0 + u].l1);
      }
#pragma unroll
      for (int u = 0; u < GRP; ++u)
        if (n0 + u < NN) mma_tf32(t[u], a.l0, b.l0, a.l1, b.l1, fb[n0 + u].h0, fb[n0 + u].h1);
#pragma unroll
      for (int u = 0; u < GRP; ++u)
        if (n0 + u < NN) mma_tf32(t[u], a.h0, b.h0, a.h1, b.h1, fb[n0 + u].h0, fb[n0 + u].h1);
#pragma unroll
      for (int u = 0; u < GRP; ++u)
        if (n0 + u < NN)
#pragma unroll
          for (int q = 0; q < 4; ++q) d[m][n0 + u][q] += t[u][q];
    }
  }
}

// Knuth's TwoSum: hi + lo carries the exact sum up to the rounding of lo
__device__ __forceinline__ void two_sum(float& hi, float& lo, float x) {
  const float s = __fadd_rn(hi, x), bp = __fsub_rn(s, hi);
  lo = __fadd_rn(lo, __fadd_rn(__fsub_rn(hi, __fsub_rn(s, bp)), __fsub_rn(x, bp)));
  hi = s;
}

template <int NM, int NN, bool DIAG>
constexpr int gt_tiles() {
  int t = 0;
  for (int m = 0; m < NM; ++m) t += NN - (DIAG ? 2 * m : 0);
  return t;
}

// The warps' sums in shared memory (where the columns were): row block m holds
// its 16 rows over the columns right of the diagonal block, at a pitch of an
// odd multiple of 8 floats -- the float2 stores of a fragment (8 rows x 4
// pairs) and the row-wise loads are both free of bank conflicts.
template <int NN, bool DIAG>
__host__ __device__ constexpr int acc_pitch(int m) { return 8 * (NN - (DIAG ? 2 * m : 0)) + 8; }
template <int NN, bool DIAG>
__host__ __device__ constexpr int acc_block(int m) {
  return DIAG ? 128 * ((NN + 1) * m - m * (m - 1)) : 16 * m * (8 * NN + 8);
}
template <int NM, int NN, bool DIAG>
constexpr int gt_smem() {
  const int cols = DIAG ? 16 * NM * GT_PITCH : (16 * NM + 8 * NN) * GT_PITCH_H;
  const int acc = acc_block<NN, DIAG>(NM) * 4 * (GT_THREADS / 32);
  return cols > acc ? cols : acc;
}
// CTAs per SM the registers are budgeted for (the accumulators and the
// fragments live in registers: 4 per MMA tile and 4 per column group)
template <int NM, int NN, bool DIAG>
constexpr int gt_min_ctas() {
  const int regs = 4 * gt_tiles<NM, NN, DIAG>() + 4 * (DIAG ? NN : 2 * NM + NN);
  return regs > 120 ? 2 : regs > 80 ? 3 : regs > 56 ? 4 : 6;
}

constexpr int GT_STAGED_PAIRS = 256;   // pair offsets kept in shared memory (tiles of up to 22 sources)

// One CTA per job: columns [ca0, ca0 + na) against [cb0, cb0 + nb) of a tile
// (DIAG: the same columns, the upper triangle).
template <int NM, int NN, bool DIAG>
__global__ void __launch_bounds__(GT_THREADS, (gt_min_ctas<NM, NN, DIAG>())) gram_tile_kernel(
    const GramJob* __restrict__ jobs, const GramEnt* __restrict__ ents, const float* __restrict__ cbuf,
    const int64_t* __restrict__ tab_all, float2* __restrict__ scr, int* __restrict__ status) {
  constexpr int NPH = DIAG ? 1 : 2;                          // loads of the tile's pixels
  constexpr int PITCH = DIAG ? GT_PITCH : GT_PITCH_H;
  constexpr uint32_t COLBYTES = TILE_THREADS * 4 / NPH;
  constexpr int NW = GT_THREADS / 32;
  constexpr int STEPS = TILE_THREADS / 8 / NW / NPH;         // 8-pixel steps of a warp per load
  extern __shared__ __align__(128) unsigned char sm[];
  __shared__ uint64_t mbar_store;
  __shared__ int64_t s_tab[GT_STAGED_PAIRS];
  __shared__ int s_ia[16 * NM], s_ib[DIAG ? 1 : 8 * NN];     // columns: (source << 8) | (free slot << 4) | free slots
  const uint32_t mbar = smem_u32(&mbar_store);
  const GramJob job = jobs[blockIdx.x];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int gid = lane >> 2, tig = lane & 3;
  const int L = job.L;
  const int64_t* tab = tab_all + job.tab0;
  const bool staged = L * (L + 1) / 2 <= GT_STAGED_PAIRS;
  if (tid == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(mbar) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  float d[NM][NN][4];
#pragma unroll
  for (int m = 0; m < NM; ++m)
#pragma unroll
    for (int n = 0; n < NN; ++n)
#pragma unroll
      for (int q = 0; q < 4; ++q) d[m][n][q] = 0.f;
#pragma unroll 1
  for (int ph = 0; ph < NPH; ++ph) {
    if (tid == 0) {
      const uint32_t bytes = (uint32_t)(job.na + (DIAG ? 0 : job.nb)) * COLBYTES;
      asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(mbar), "r"(bytes) : "memory");
    }
    __syncthreads();   // the expected bytes are set (and the last load's columns read)
    for (int x = tid; x < L; x += GT_THREADS) {
      const GramEnt e = ents[job.e0 + x];
      const float* src = cbuf + e.off + ph * (TILE_THREADS / NPH);
      for (int f = 0; f < e.nf; ++f) {
        const int a = e.col0 + f - job.ca0, b = e.col0 + f - job.cb0;
        if (a >= 0 && a < job.na) {
          bulk_load(smem_u32(sm + a * PITCH), src + f * TILE_THREADS, COLBYTES, mbar);
          s_ia[a] = (x << 8) | (f << 4) | e.nf;
        }
        if (!DIAG && b >= 0 && b < job.nb) {
          bulk_load(smem_u32(sm + (16 * NM + b) * PITCH), src + f * TILE_THREADS, COLBYTES, mbar);
          s_ib[b] = (x << 8) | (f << 4) | e.nf;
        }
      }
    }
    if (ph == 0 && staged)
      for (int p = tid; p < L * (L + 1) / 2; p += GT_THREADS) s_tab[p] = tab[p];
    if (!__syncthreads_and(mbar_wait(mbar, ph & 1))) {
      // the copies did not arrive within the limit: an error, and one more
      // wait of the same length for those still in flight before the CTA leaves
      if (tid == 0) atomicCAS(status, 0, AP_ERR_TIMEOUT);
      mbar_wait(mbar, ph & 1);
      return;
    }
    const unsigned char* base = sm + gid * PITCH + tig * 8 + warp * STEPS * 32;
#pragma unroll(gt_tiles<NM, NN, DIAG>() <= 12 ? 2 : 1)
    for (int s = 0; s < STEPS; ++s) {
      Frag fa[DIAG ? NN : 2 * NM], fb[DIAG ? 1 : NN];
#pragma unroll
      for (int g = 0; g < (DIAG ? NN : 2 * NM); ++g) frag_load(fa[g], base + g * 8 * PITCH + s * 32);
      if constexpr (!DIAG) {
#pragma unroll
        for (int g = 0; g < NN; ++g) frag_load(fb[g], base + (16 * NM + g * 8) * PITCH + s * 32);
      }
      mma_step<NM, NN, DIAG>(d, fa, DIAG ? fa : fb);
    }
    __syncthreads();   // every warp has read the columns
  }
  constexpr int ACC = acc_block<NN, DIAG>(NM);
  float* acc = reinterpret_cast<float*>(sm);
#pragma unroll
  for (int m = 0; m < NM; ++m) {
    float* mine = acc + warp * ACC + acc_block<NN, DIAG>(m) + gid * acc_pitch<NN, DIAG>(m) + 2 * tig;
#pragma unroll
    for (int n = DIAG ? 2 * m : 0; n < NN; ++n) {
      float* q = mine + 8 * (n - (DIAG ? 2 * m : 0));
      *reinterpret_cast<float2*>(q) = make_float2(d[m][n][0], d[m][n][1]);
      *reinterpret_cast<float2*>(q + 8 * acc_pitch<NN, DIAG>(m)) = make_float2(d[m][n][2], d[m][n][3]);
    }
  }
  __syncthreads();
  // the source pairs' blocks: a warp takes every fourth row, its lanes the
  // row's columns (a run of a source's columns is a run of its pair's block)
  const int* ib_of = DIAG ? s_ia : s_ib;
#pragma unroll 1
  for (int c0 = 0; c0 < job.nb; c0 += 32) {
    const int cb = c0 + lane;
    const int ib = cb < job.nb ? ib_of[cb] : 0;
    const int b = ib >> 8, fb = (ib >> 4) & 15, mb = ib & 15;
    const int rows = DIAG ? min(job.na, c0 + 32) : job.na;
#pragma unroll 2
    for (int ca = warp; ca < rows; ca += NW) {
      const int ia = s_ia[ca], a = ia >> 8, fa = (ia >> 4) & 15, m = ca >> 4;
      if (cb < job.nb && (!DIAG || cb >= ca)) {
        const float* v =
            acc + acc_block<NN, DIAG>(m) + (ca & 15) * acc_pitch<NN, DIAG>(m) + cb - (DIAG ? 16 * m : 0);
        // the four 64-pixel sums as hi + lo
        float h0 = v[0], l0 = 0.f, h1 = v[2 * ACC], l1 = 0.f;
        two_sum(h0, l0, v[ACC]);
        two_sum(h1, l1, v[3 * ACC]);
        two_sum(h0, l0, h1);
        const int p = a * L - (a * (a - 1)) / 2 + (b - a);
        scr[(staged ? s_tab[p] : tab[p]) + fa * mb + fb] = make_float2(h0, __fadd_rn(l0, l1));
      }
    }
  }
}

template <int NM, int NN, bool DIAG>
void gt_launch(const GramJob* jobs, int n, const GramPlan& gp, const float* cbuf, int* status, cudaStream_t st) {
  gram_tile_kernel<NM, NN, DIAG><<<n, GT_THREADS, gt_smem<NM, NN, DIAG>(), st>>>(
      jobs, gp.ents, cbuf, gp.tab, reinterpret_cast<float2*>(gp.scr), status);
}

}  // namespace

// ---------------------------------------------------------------------------
// float64 path, pass 1
// ---------------------------------------------------------------------------
constexpr int GRAM64_CB = 32;   // columns of a block

__device__ __forceinline__ void ld4(const double* p, double (&v)[4]) {
  const double2 a = *reinterpret_cast<const double2*>(p);
  const double2 b = *reinterpret_cast<const double2*>(p + 2);
  v[0] = a.x; v[1] = a.y; v[2] = b.x; v[3] = b.y;
}

// Load columns [c0, c0 + cb) of the tile (in (source, slot) order) into a
// pixel-major block of row stride CP, scaled by sqrt(w) of the thread's
// pixel; returns the number loaded.  Every thread fills its own row: copies
// (cp.async, all in flight together) are issued for its in-box values, then
// awaited, then scaled.
__device__ __forceinline__ int load_columns(double* blk, int CP, int c0, int cb, const TileWork& w,
                                            const int* __restrict__ jt_src, const SourceDev* __restrict__ srcs,
                                            const double* __restrict__ dbuf, const double* __restrict__ jbuf, int i,
                                            int j, bool inside, double sw, int* colp) {
  double* myrow = blk + threadIdx.x * CP;
  int col = 0, n = 0;
  for (int e = w.e0; e < w.e1 && n < cb; ++e) {
    const SourceDev& sd = srcs[jt_src[e]];
    int nfree = 0;
#pragma unroll
    for (int k = 0; k < MAX_SLOTS; ++k) nfree += (k < sd.nslot && sd.pidx[k] >= 0);
    if (col + nfree <= c0) { col += nfree; continue; }
    const int* bx = sd.conv ? sd.sup : sd.box;
    const bool in_b = inside && i >= bx[0] && i < bx[1] && j >= bx[2] && j < bx[3];
    const int bw = bx[3] - bx[2];
    const int64_t area = (int64_t)(bx[1] - bx[0]) * bw;
    const double* base =
        (sd.conv ? jbuf + sd.j_off : dbuf + sd.d_off) + (in_b ? (int64_t)(i - bx[0]) * bw + (j - bx[2]) : 0);
    int f = 0;
#pragma unroll
    for (int k = 0; k < MAX_SLOTS; ++k) {
      if (k >= sd.nslot || sd.pidx[k] < 0) continue;
      if (col >= c0 && n < cb) {
        if (in_b)
          asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(smem_u32(myrow + n)), "l"(base + k * area)
                       : "memory");
        else
          myrow[n] = 0.0;
        // column info: local source index, free-slot index, free columns of the source
        if (threadIdx.x == 0) colp[n] = ((e - w.e0) << 8) | (f << 4) | nfree;
        ++n;
      }
      ++f;
      ++col;
    }
  }
  for (int c = n; c < ((n + 15) & ~15) && c < CP; ++c) myrow[c] = 0.0;
  asm volatile("cp.async.wait_all;" ::: "memory");
  for (int c = 0; c < n; ++c) myrow[c] *= sw;
  return n;
}

// Gram of column block A (na columns) with column block B (nb_ columns) of
// the tile, stored into the pair blocks (pairs of the L tile sources are
// numbered row-major over a <= b); diag = the blocks are the same.
__device__ void gram_pair(const double* ja, const double* jb, int CP, int na, int nbc, bool diag, const int* colpa,
                          const int* colpb, int L, const int64_t* __restrict__ tab, double* __restrict__ scr) {
  const int tid = threadIdx.x;
  const int ba = (na + 3) >> 2, bb = (nbc + 3) >> 2;   // 4-column sub-blocks
  const int npb = diag ? ba * (ba + 1) / 2 : ba * bb;
  int NS = 4;
  while (NS < 32 && npb * NS * 2 <= TILE_THREADS) NS <<= 1;
  const int total = npb * NS;
  const int seglen = TILE_THREADS / NS;
  for (int base_idx = 0; base_idx < total; base_idx += TILE_THREADS) {
    const int idx = base_idx + tid;
    const bool active = idx < total;
    const int pb = active ? idx / NS : 0;
    const int seg = idx % NS;
    int A, B;
    if (diag) {
      A = 0;
      int rem = pb;
      while (rem >= ba - A) { rem -= ba - A; ++A; }
      B = A + rem;
    } else {
      A = pb / bb;
      B = pb - A * bb;
    }
    double acc[4][4];
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int b = 0; b < 4; ++b) acc[a][b] = 0.0;
    if (active) {
      const double* pa = ja + 4 * A;
      const double* pbp = jb + 4 * B;
      for (int t = seg * seglen; t < (seg + 1) * seglen; ++t) {
        double va[4], vb[4];
        ld4(pa + t * CP, va);
        ld4(pbp + t * CP, vb);
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
          for (int b = 0; b < 4; ++b) acc[a][b] += va[a] * vb[b];
      }
    }
    for (int o = NS >> 1; o > 0; o >>= 1)
#pragma unroll
      for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) acc[a][b] += __shfl_xor_sync(0xffffffffu, acc[a][b], o);
    if (!active || seg != 0) continue;
#pragma unroll
    for (int a = 0; a < 4; ++a) {
#pragma unroll
      for (int b = 0; b < 4; ++b) {
        const int ca = 4 * A + a, cb = 4 * B + b;
        if (ca >= na || cb >= nbc || (diag && cb < ca)) continue;
        const int ia = colpa[ca], ib = colpb[cb];
        const int la = ia >> 8, fa = (ia >> 4) & 15, lb = ib >> 8, fb = (ib >> 4) & 15, mb = ib & 15;
        scr[tab[la * L - (la * (la - 1)) / 2 + (lb - la)] + fa * mb + fb] = acc[a][b];
      }
    }
  }
}

// One CTA per image tile.  The tile's C columns are processed in blocks of
// cb: block I is loaded once, then paired with every block J >= I (the Gram
// is symmetric), so any number of columns fits in two shared blocks.
__global__ void __launch_bounds__(TILE_THREADS) gram_f64_kernel(
    const TileWork* __restrict__ work, const int* __restrict__ jt_src, const SourceDev* __restrict__ srcs,
    const ImageDev* __restrict__ imgs, const double* __restrict__ dbuf, const double* __restrict__ jbuf,
    const int64_t* __restrict__ tab0, const int64_t* __restrict__ tab_all, double* __restrict__ scr, int t_first,
    int cb, int two_blocks) {
  const int CP = cb + 4;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  double* blk0 = reinterpret_cast<double*>(smem_raw);
  double* blk1 = blk0 + TILE_THREADS * CP;
  int* colp0 = reinterpret_cast<int*>(blk0 + (two_blocks ? 2 : 1) * TILE_THREADS * CP);
  int* colp1 = colp0 + CP;
  const int tile = t_first + blockIdx.x;
  const TileWork w = work[tile];
  const ImageDev& im = imgs[w.image];
  const int tid = threadIdx.x;
  const int i = w.r0 + tid / TILE, j = w.c0 + tid % TILE;
  const bool inside = i < im.H && j < im.W;
  double sw = 0.0;
  if (inside) {
    const size_t o = (size_t)i * im.W + j;
    const float var = im.var[o];
    if ((im.mask == nullptr || im.mask[o] == 0) && var > 0.f && isfinite(var)) sw = sqrt(1.0 / (double)var);
  }
  // total free columns of the tile
  int C = 0;
  for (int e = w.e0; e < w.e1; ++e) {
    const SourceDev& sd = srcs[jt_src[e]];
    for (int k = 0; k < sd.nslot; ++k) C += sd.pidx[k] >= 0;
  }
  const int nblk = (C + cb - 1) / cb;
  const int L = w.e1 - w.e0;
  const int64_t* tab = tab_all + tab0[tile];
  for (int I = 0; I < nblk; ++I) {
    __syncthreads();
    const int na = load_columns(blk0, CP, I * cb, cb, w, jt_src, srcs, dbuf, jbuf, i, j, inside, sw, colp0);
    __syncthreads();
    gram_pair(blk0, blk0, CP, na, na, true, colp0, colp0, L, tab, scr);
    for (int J = I + 1; J < nblk; ++J) {
      __syncthreads();
      const int nb_ = load_columns(blk1, CP, J * cb, cb, w, jt_src, srcs, dbuf, jbuf, i, j, inside, sw, colp1);
      __syncthreads();
      gram_pair(blk0, blk1, CP, na, nb_, false, colp0, colp1, L, tab, scr);
    }
  }
}

static size_t gram64_smem(int cb, int two) {
  const int CP = cb + 4;
  return (size_t)(two ? 2 : 1) * TILE_THREADS * CP * sizeof(double) + (size_t)2 * CP * sizeof(int);
}

// ---------------------------------------------------------------------------
// pass 2: the pairs' sums over their tiles.  A pair's blocks lie one after
// another (entry fastest), so consecutive threads read consecutive values:
// thread t takes entry t mod ne of tiles t / ne, t / ne + T, ...  Each thread
// sums hi + lo compensated (float path) or in float64, the threads of an entry
// are joined in float64 in a fixed order (deterministic).
// ---------------------------------------------------------------------------
template <typename V> struct TileSum;
template <> struct TileSum<float2> {
  float hi = 0.f, lo = 0.f;
  __device__ __forceinline__ void add(float2 v) {
    two_sum(hi, lo, v.x);
    lo = __fadd_rn(lo, v.y);
  }
  __device__ __forceinline__ double get() const { return (double)hi + (double)lo; }
};
template <> struct TileSum<double> {
  double s = 0.0;
  __device__ __forceinline__ void add(double v) { s += v; }
  __device__ __forceinline__ double get() const { return s; }
};

// entry values src[k ne], k = k0, k0 + step, ... below cnt: eight loads in flight
template <typename V>
__device__ __forceinline__ double tile_sum(const V* __restrict__ src, int ne, int k0, int step, int cnt) {
  TileSum<V> acc;
  int k = k0;
  for (; k + 7 * step < cnt; k += 8 * step) {
    V v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) v[u] = src[(int64_t)(k + u * step) * ne];
#pragma unroll
    for (int u = 0; u < 8; ++u) acc.add(v[u]);
  }
  V v[8];
#pragma unroll
  for (int u = 0; u < 7; ++u)
    if (k + u * step < cnt) v[u] = src[(int64_t)(k + u * step) * ne];
#pragma unroll
  for (int u = 0; u < 7; ++u)
    if (k + u * step < cnt) acc.add(v[u]);
  return acc.get();
}

// A float sum that left float32's range (of tile entries up to 3.4e38 each; an
// infinite or NaN hi stays one) is taken again in float64, which holds it.
__device__ __forceinline__ double in_range(const double* __restrict__, int, int, int, double s) { return s; }
__device__ __forceinline__ double in_range(const float2* __restrict__ src, int ne, int k0, int cnt, double s) {
  if ((__double2hiint(s) & 0x7ff00000) != 0x7ff00000) return s;
  s = 0.0;
#pragma unroll 1
  for (int k = k0; k < cnt; ++k) s += (double)src[(int64_t)k * ne].x + (double)src[(int64_t)k * ne].y;
  return s;
}

struct EntryPos {
  int64_t ab, ba;   // in the CSR values: the entry's and its mirror's (-1: not stored)
};
__device__ __forceinline__ EntryPos entry_pos(const GramPair& gp, const int64_t* __restrict__ pos, int e) {
  return EntryPos{pos[gp.pos + 2 * e], pos[gp.pos + 2 * e + 1]};
}
__device__ __forceinline__ void gram_write(const GramPair& gp, EntryPos at, double s, double* __restrict__ vals) {
  if (at.ab < 0) return;   // below the diagonal of a source's own block
  if (gp.excl) {
    vals[at.ab] = s;
    if (at.ba >= 0) vals[at.ba] = s;
  } else {
    atomicAdd(vals + at.ab, s);
    if (at.ba >= 0) atomicAdd(vals + at.ba, s);
  }
}

// pairs of few values (n_light of them, first in the list): a warp each
template <typename V>
__global__ void __launch_bounds__(256) gram_reduce_kernel(const GramPair* __restrict__ pairs, int n_pairs,
                                                          const int64_t* __restrict__ pos, const V* __restrict__ scr,
                                                          double* __restrict__ vals) {
  const int lane = threadIdx.x & 31;
  const int w0 = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, nw = (gridDim.x * blockDim.x) >> 5;
  for (int p = w0; p < n_pairs; p += nw) {
    const GramPair gp = pairs[p];
    const int ne = gp.ma * gp.mb;
    const V* src = scr + gp.base;
    if (ne > 16) {   // one tile at a time, an entry (or two) per lane
      for (int e = lane; e < ne; e += 32) {
        const double s = tile_sum(src + e, ne, 0, 1, gp.cnt);
        const EntryPos at = entry_pos(gp, pos, e);
        gram_write(gp, at, in_range(src + e, ne, 0, gp.cnt, s), vals);
      }
    } else {         // 32 / ne tiles side by side
      const int T = 32 / ne, e = lane % ne, t = lane / ne;
      const double part = t < T ? tile_sum(src + e, ne, t, T, gp.cnt) : 0.0;
      double s = 0.0;
      for (int k = 0; k < T; ++k) s += __shfl_sync(0xffffffffu, part, (k * ne + e) & 31);
      if (lane < ne) {
        const EntryPos at = entry_pos(gp, pos, e);
        gram_write(gp, at, in_range(src + e, ne, 0, gp.cnt, s), vals);
      }
    }
  }
}

// the other pairs: a CTA per run of some GRAM_RUN_VALUES values; the CTA that
// finishes a pair last adds its runs in order
template <typename V>
__global__ void __launch_bounds__(256) gram_reduce_run_kernel(const GramPair* __restrict__ pairs,
                                                              const GramRun* __restrict__ runs,
                                                              const int64_t* __restrict__ pos,
                                                              const V* __restrict__ scr, double* __restrict__ part,
                                                              int* __restrict__ done, double* __restrict__ vals) {
  __shared__ double red[256];
  __shared__ int last;
  const GramRun rn = runs[blockIdx.x];
  const GramPair gp = pairs[rn.pair];
  const int ne = gp.ma * gp.mb, T = 256 / ne;
  const int e = threadIdx.x % ne, t = threadIdx.x / ne;
  if (t < T) red[threadIdx.x] = tile_sum(scr + gp.base + e, ne, rn.k0 + t, T, rn.k1);
  __syncthreads();
  double s = 0.0;
  if ((int)threadIdx.x < ne) {
    for (int k = 0; k < T; ++k) s += red[k * ne + threadIdx.x];
    s = in_range(scr + gp.base + threadIdx.x, ne, rn.k0, rn.k1, s);
    if (rn.n_runs == 1)
      gram_write(gp, entry_pos(gp, pos, threadIdx.x), s, vals);
    else
      part[(int64_t)(rn.first + rn.run) * 64 + threadIdx.x] = s;
  }
  if (rn.n_runs == 1) return;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(&done[rn.first], 1) == rn.n_runs - 1;
  __syncthreads();
  if (!last) return;
  __threadfence();
  if ((int)threadIdx.x < ne) {
    s = 0.0;
    for (int k = 0; k < rn.n_runs; ++k) s += __ldcg(part + (int64_t)(rn.first + k) * 64 + threadIdx.x);
    gram_write(gp, entry_pos(gp, pos, threadIdx.x), s, vals);
  }
  if (threadIdx.x == 0) done[rn.first] = 0;   // ready for the next call
}

// ---------------------------------------------------------------------------
// jobs and launches
// ---------------------------------------------------------------------------
void gram64_blocking(int maxc, int* cb, int* two) {
  const int m = ((maxc < 4 ? 4 : maxc) + 3) & ~3;
  *cb = m < GRAM64_CB ? m : GRAM64_CB;
  *two = m > GRAM64_CB;
}

// The jobs of the tiles' column counts, grouped by kernel form: form g = 1..6
// takes up to 16 g columns (the triangle's accumulators fit the registers up
// to 96); a tile past 96 columns is cut into blocks of 64, a diagonal job each
// and an off-diagonal job (form 7, 64 x 64) for every two.
void gram_plan_jobs(const std::vector<TileWork>& tiles, const std::vector<int64_t>& tab0,
                    const std::vector<int>& tile_ncol, std::vector<GramJob>& jobs, std::vector<GramRange>& ranges) {
  std::vector<GramJob> by[GRAM_FORMS + 1];
  for (int t = 0; t < (int)tile_ncol.size(); ++t) {
    const int C = tile_ncol[t];
    if (C <= 0) continue;
    const int e0 = tiles[t].e0, L = tiles[t].e1 - e0;
    if (C <= 96) {
      by[(C + 15) / 16].push_back(GramJob{tab0[t], e0, L, 0, C, 0, C});
      continue;
    }
    for (int a = 0; a < C; a += 64) {
      const int na = std::min(64, C - a);
      by[(na + 15) / 16].push_back(GramJob{tab0[t], e0, L, a, na, a, na});
      for (int b = a + 64; b < C; b += 64)
        by[GRAM_FORMS].push_back(GramJob{tab0[t], e0, L, a, na, b, std::min(64, C - b)});
    }
  }
  for (int f = GRAM_FORMS; f >= 1; --f) {   // the longest jobs first
    if (by[f].empty()) continue;
    ranges.push_back(GramRange{(int)jobs.size(), (int)(jobs.size() + by[f].size()), f, 0});
    jobs.insert(jobs.end(), by[f].begin(), by[f].end());
  }
}

int configure_gram(bool f64) {
  if (f64) return allow_max_dynamic_smem(gram_f64_kernel) >= (int)gram64_smem(GRAM64_CB, 1);
  int ok = 1;
#define AP_GT_CFG(NM, NN, DIAG) ok &= allow_max_dynamic_smem(gram_tile_kernel<NM, NN, DIAG>) >= gt_smem<NM, NN, DIAG>()
  AP_GT_CFG(1, 2, true);
  AP_GT_CFG(2, 4, true);
  AP_GT_CFG(3, 6, true);
  AP_GT_CFG(4, 8, true);
  AP_GT_CFG(5, 10, true);
  AP_GT_CFG(6, 12, true);
  AP_GT_CFG(4, 8, false);
#undef AP_GT_CFG
  return ok;
}

template <typename T>
void launch_gram(const TileWork* work, const GramRange* ranges, int n_ranges, const int* jt_src,
                 const SourceDev* srcs, const ImageDev* imgs, const T* dbuf, const T* jbuf, const GramPlan& gp,
                 double* vals, int* status, cudaStream_t st, const ForkJoin* fj) {
  // pass 1: the launches write disjoint scratch, so they run side by side on
  // the auxiliary streams (their tails overlap)
  int used = 0;
  const bool fork = fj && n_ranges > 1;
  if (fork) cudaEventRecord(fj->fork, st);
  for (int r = 0; r < n_ranges; ++r) {
    const GramRange& g = ranges[r];
    const int n = g.t1 - g.t0;
    if (n <= 0) continue;
    cudaStream_t s = st;
    if (fork) {
      s = fj->aux[used % N_AUX_STREAMS];
      if (used < N_AUX_STREAMS) cudaStreamWaitEvent(s, fj->fork, 0);
      ++used;
    }
    if constexpr (sizeof(T) == 4) {
      const GramJob* jobs = gp.jobs + g.t0;
      const float* cbuf = reinterpret_cast<const float*>(jbuf);
      switch (g.form) {
        case 1: gt_launch<1, 2, true>(jobs, n, gp, cbuf, status, s); break;
        case 2: gt_launch<2, 4, true>(jobs, n, gp, cbuf, status, s); break;
        case 3: gt_launch<3, 6, true>(jobs, n, gp, cbuf, status, s); break;
        case 4: gt_launch<4, 8, true>(jobs, n, gp, cbuf, status, s); break;
        case 5: gt_launch<5, 10, true>(jobs, n, gp, cbuf, status, s); break;
        case 6: gt_launch<6, 12, true>(jobs, n, gp, cbuf, status, s); break;
        default: gt_launch<4, 8, false>(jobs, n, gp, cbuf, status, s); break;
      }
    } else {
      gram_f64_kernel<<<n, TILE_THREADS, gram64_smem(g.form, g.two), s>>>(
          work, jt_src, srcs, imgs, reinterpret_cast<const double*>(dbuf), reinterpret_cast<const double*>(jbuf), gp.tab0,
          gp.tab, reinterpret_cast<double*>(gp.scr), g.t0, g.form, g.two);
    }
  }
  for (int k = 0; k < used && k < N_AUX_STREAMS; ++k) {
    cudaEventRecord(fj->join[k], fj->aux[k]);
    cudaStreamWaitEvent(st, fj->join[k], 0);
  }
  using V = typename std::conditional<sizeof(T) == 4, float2, double>::type;
  const V* scr = reinterpret_cast<const V*>(gp.scr);
  if (gp.n_light > 0) {
    const int blocks = (int)std::min<int64_t>(((int64_t)gp.n_light * 32 + 255) / 256, 8192);
    gram_reduce_kernel<V><<<blocks, 256, 0, st>>>(gp.pairs, gp.n_light, gp.pos, scr, vals);
  }
  if (gp.n_runs > 0)
    gram_reduce_run_kernel<V><<<gp.n_runs, 256, 0, st>>>(gp.pairs, gp.runs, gp.pos, scr, gp.part, gp.done, vals);
}

template void launch_gram<float>(const TileWork*, const GramRange*, int, const int*, const SourceDev*,
                                 const ImageDev*, const float*, const float*, const GramPlan&, double*, int*,
                                 cudaStream_t, const ForkJoin*);
template void launch_gram<double>(const TileWork*, const GramRange*, int, const int*, const SourceDev*,
                                  const ImageDev*, const double*, const double*, const GramPlan&, double*, int*,
                                  cudaStream_t, const ForkJoin*);

}  // namespace ap
