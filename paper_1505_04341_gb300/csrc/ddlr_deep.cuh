// ddlr_deep.cuh -- triangular solves with deep factor blocks (many dependency
// levels, as natural elimination orders and fill give): one CTA per interior
// block, one thread-block cluster for C_a, the solution in shared memory.
//
// What bounds such a solve is its level chain: C_a of the 64^3 grid in natural
// order has 67,032 rows in 160 levels, 319 dependent steps of about 420 rows; a
// 14^3 interior block has 43 levels.  One launch per level costs a launch and a
// trip through L2 per step (3.2 us each inside a CUDA graph).  Here the block is
// cut into parts, one CTA each, and a step of a part is a handoff between two
// sets of warps, loads of earlier results from the CTA's own shared memory and
// the row's chain of FMAs; nothing else is on the chain:
//  * the two sets of warps take the levels in turn, and while one computes,
//    the other has its next level's entries, addresses and own values in
//    registers (the factor streams into a ring by bulk copies well ahead);
//  * a result that another part needs is pushed into that part's shared memory
//    (st.async, completion counted on an mbarrier of the level that reads it
//    first) by a warp of its own, so parts run as a pipeline and never meet at
//    a cluster barrier (a form with a cluster barrier per level took 0.92 us
//    per step on the same problem, most of it the barrier's release and wait).
// C_a of 64^3 (8 CTAs): 1.03 ms -> 0.20 ms per solve, 0.6 us a step; its 64
// interior blocks: 70 us (copies one level ahead of a barrier per level) -> 50.
// C_a's parts are ranges of the interface nodes' original order, in which a
// natural elimination order only depends on earlier parts.
#pragma once
#include "ddlr_kernels.cuh"

namespace ddlr {

// Warps of one set, and of one for wide levels: C_a, and blocks that have an SM each
// and kDeepWideRows rows a level on average.  Below that line the two are alike (a
// solve, FP64, edges of 11 and 13: 41.6 and 42.2 us, 47.6 and 46.2), above it a level
// takes a warp several slices (15: 60.4 and 52.5, 23: 121 and 96, 28: 219 and 177;
// FP32, 35: 285 and 219; C_a, FP64, 64^3 on 8 CTAs 201 and 199, 48^3 in 27 boxes on 2
// 171 and 131).  Two blocks to an SM fill it with the narrow sets (FP32, 112 x 112 x 96
// in 294 boxes: 82 and 100).
constexpr int kDeepSetWarps = 4, kDeepWideWarps = 8, kDeepWideRows = 80;
__host__ __device__ constexpr int deep_threads(int sw) { return (2 * sw + 1) * 32; }   // two sets and the copy / push warp
constexpr int kDeepMaxCtas = 16;
constexpr int kDeepBars = 32;            // ring mbarriers: stages in flight at most

// One part: a CTA's rows.  A slice is up to 32 rows of one level (one warp),
// contiguous in device order; a stage is one level of one sweep.  Forward
// stages come first.
struct DeepPart {
  int slice0, nslice;      // its slices
  int stage0, nstage, nfwd;// its stages
  int nhalo;               // values received from other parts
};
struct DeepStage {
  int src;                 // packed data (from the L or L^T pack): start,
  unsigned short bytes, pos;// size, place in the ring,
  int lin;                 // running total before it with the gaps at the ring's end; all / 128
  int a;                   // its first slice, counted from the part's first
  int rows, z0;            // its rows, the first one's position in the part's shared memory
  int halo;                // values received whose first use is here
  int push;                // its first entry in the push list; the next stage's starts where it ends
};
static_assert(sizeof(DeepStage) == 32 && sizeof(DeepPart) == 24, "tables are copied as words");

// Geometry of one launch: ctas = CTAs of a cluster (1: independent blocks)
struct DeepGeo {
  int ctas, nparts, sw;    // sw: warps of a set
  int ring_bytes;          // staging ring (multiple of 128)
  int zcap, scap, tcap;    // most rows + received values, slices, stages of a part
  const DeepPart *part;
  const DeepStage *stage;
  const int4 *push;        // {position here, part's rank, position there, stage there}
  const int4 *sl;          // per slice: {L offset / 128, position << 6 | rows, U offset / 128, L width | U width << 16}
  const int2 *srow;        // per slice: {first row, rows}
};

// stored width of a slice: beyond four entries a multiple of four, so that the
// row's chain is straight code (a test per entry costs as much as its FMA)
constexpr int kDeepMaxWidth = 0xffff;
inline int deep_width(int w) { return w <= 4 ? w : (w + 3) & ~3; }
// width of slice entry e for direction dir (1: L^T)
__host__ __device__ inline int deep_w(const int4 &e, int dir) {
  return dir ? int(unsigned(e.w) >> 16) : int(unsigned(e.w) & 0xffffu);
}
template <typename T>
__host__ __device__ inline size_t deep_slice_bytes(int w) {
  return size_t(w) * 32 * (sizeof(T) + 4) + 32 * sizeof(T);
}
template <typename T>
__host__ __device__ inline size_t deep_smem_bytes(const DeepGeo &g) {
  return 16 * kDeepBars + size_t(g.ring_bytes) + al128(size_t(g.zcap + 1) * sizeof(T)) +
         al128(size_t(g.tcap + 1) * sizeof(DeepStage)) + al128(size_t(g.scap) * 16) +
         (g.ctas > 1 ? size_t(g.tcap) * 8 : 0);
}

// Columns of the packed data: position in the part's shared memory, rpos[row]
// for the part's own rows (fix-ups for received values follow).  Padding reads
// the row itself with a value of 0.  One CTA per slice.
template <typename T>
__global__ void k_deep_cols(DeepGeo g, const int2 *l_span, const int2 *u_span, const int *l_col, const int *u_col,
                            const int *rpos, unsigned char *pk_l, unsigned char *pk_u) {
  const int4 e = g.sl[blockIdx.x];
  const int2 sr = g.srow[blockIdx.x];
  for (int dir = 0; dir < 2; dir++) {
    const int w = deep_w(e, dir);
    unsigned char *p = dir ? pk_u + size_t(e.z) * 128 : pk_l + size_t(e.x) * 128;
    int *pc = reinterpret_cast<int *>(p + size_t(w) * 32 * sizeof(T));
    for (int i = threadIdx.x; i < w * 32; i += blockDim.x) {
      const int kk = i >> 5, ln = i & 31, r = sr.x + min(ln, sr.y - 1);
      const int2 sp = (dir ? u_span : l_span)[r];
      const bool live = ln < sr.y && kk < sp.y;
      pc[i] = rpos[live ? (dir ? u_col : l_col)[sp.x + 32 * kk] : r];
    }
  }
}
// fix[i] = {slice, direction, entry of the slice, position of the received value}
template <typename T>
__global__ void k_deep_fix(int cnt, DeepGeo g, const int4 *fix, unsigned char *pk_l, unsigned char *pk_u) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= cnt) return;
  const int4 f = fix[i], e = g.sl[f.x];
  const int w = deep_w(e, f.y);
  unsigned char *p = f.y ? pk_u + size_t(e.z) * 128 : pk_l + size_t(e.x) * 128;
  reinterpret_cast<int *>(p + size_t(w) * 32 * sizeof(T))[f.z] = f.w;
}

// Values and inverse diagonal of the packed data (every numeric setup)
template <typename T>
__global__ void k_deep_pack(DeepGeo g, const int2 *l_span, const int2 *u_span, const T *lval, const T *uval,
                            const T *dinv, unsigned char *pk_l, unsigned char *pk_u) {
  const int4 e = g.sl[blockIdx.x];
  const int2 sr = g.srow[blockIdx.x];
  for (int dir = 0; dir < 2; dir++) {
    const int w = deep_w(e, dir);
    unsigned char *p = dir ? pk_u + size_t(e.z) * 128 : pk_l + size_t(e.x) * 128;
    T *pv = reinterpret_cast<T *>(p);
    T *pd = reinterpret_cast<T *>(p + size_t(w) * 32 * (sizeof(T) + 4));
    for (int i = threadIdx.x; i < w * 32; i += blockDim.x) {
      const int kk = i >> 5, ln = i & 31;
      T v = T(0);
      if (ln < sr.y) {
        const int2 sp = (dir ? u_span : l_span)[sr.x + ln];
        if (kk < sp.y) v = (dir ? uval : lval)[sp.x + 32 * kk];
      }
      pv[i] = v;
    }
    for (int i = threadIdx.x; i < 32; i += blockDim.x) pd[i] = i < sr.y ? dinv[sr.x + i] : T(0);
  }
}

__device__ __forceinline__ unsigned cluster_rank() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// shared address `a` of this CTA in CTA `rank` of the cluster
__device__ __forceinline__ uint32_t cluster_map(uint32_t a, int rank) {
  uint32_t r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
  return r;
}
// store into a peer's shared memory, its bytes counted on the peer's mbarrier
__device__ __forceinline__ void st_async(uint32_t a, double v, uint32_t bar) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b64 [%0], %1, [%2];" ::"r"(a),
               "l"(__double_as_longlong(v)), "r"(bar)
               : "memory");
}
__device__ __forceinline__ void st_async(uint32_t a, float v, uint32_t bar) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];" ::"r"(a),
               "r"(__float_as_int(v)), "r"(bar)
               : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t *bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
// wait acquiring a peer's st.async results
__device__ __forceinline__ bool mbar_try_wait_cluster(uint64_t *bar, unsigned parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
// named barriers 1 and 2: end of a level of set 0 and of set 1 (of SW warps each)
template <int SW>
__device__ __forceinline__ void set_arrive(int set) {
  asm volatile("bar.arrive %0, %1;" ::"r"(1 + set), "n"(2 * SW * 32) : "memory");
}
template <int SW>
__device__ __forceinline__ void set_sync(int set) {
  asm volatile("bar.sync %0, %1;" ::"r"(1 + set), "n"(2 * SW * 32) : "memory");
}

// acc - sum of the first W prefetched entries, the loads before the FMAs
template <typename T, int W>
__device__ __forceinline__ T deep_chain(T acc, const T *zs, const int *ad, const T *av) {
  T zv[W];
#pragma unroll
  for (int u = 0; u < W; u++) zv[u] = zs[ad[u]];
#pragma unroll
  for (int u = 0; u < W; u++) acc -= av[u] * zv[u];
  return acc;
}

// z = (L L^T)^-1 x on the rows of the launch's blocks: forward over the levels
// with L, then backward with L^T.  CTA b takes part b; with g.ctas > 1 the grid
// is one cluster.  Waits are bounded (limit_ns): a thread whose wait runs out
// sets *err and the CTA's late flag; the CTA then runs through its stages
// without waiting or computing (its warps keep to the named barriers) and starts
// no more copies, but its pushes are made all the same, whatever they carry:
// every CTA issues all of its pushes before the last barrier, so that after it a
// CTA that stopped counting them waits until its mbarriers have the bytes of all.
// These last waits, and those for the copies in flight, are for transfers that
// have started; they have a limit of their own (kDeepExitWaitNs).  give_up_at
// (tests; else -1): the last part's copy warp gives up after this stage.
// Four narrow CTAs share an SM: that many fit its registers.
template <typename T, int SW>
__global__ void __launch_bounds__(deep_threads(SW), SW == kDeepSetWarps ? 4 : 2)
k_deep_solve(DeepGeo g, const unsigned char *pk_l, const unsigned char *pk_u, const T *x, T *z, const int *gate,
             int *err, unsigned long long limit_ns, int give_up_at) {
  if (gate && *gate) return;               // the same word for every CTA, not written meanwhile
  extern __shared__ __align__(128) unsigned char smraw[];
  constexpr int NT = deep_threads(SW);
  const int tid = threadIdx.x, wi = tid >> 5, ln = tid & 31;
  const DeepPart P = g.part[blockIdx.x];
  const int nst = P.nstage;
  uint64_t *bar = reinterpret_cast<uint64_t *>(smraw);     // ring stages
  uint64_t *done = bar + kDeepBars;                        // levels finished by their set
  unsigned char *ring = smraw + 16 * kDeepBars;
  T *zs = reinterpret_cast<T *>(ring + g.ring_bytes);
  DeepStage *st = reinterpret_cast<DeepStage *>(reinterpret_cast<unsigned char *>(zs) + al128(size_t(g.zcap + 1) * sizeof(T)));
  int4 *sl = reinterpret_cast<int4 *>(reinterpret_cast<unsigned char *>(st) + al128(size_t(g.tcap + 1) * sizeof(DeepStage)));
  uint64_t *halo = reinterpret_cast<uint64_t *>(reinterpret_cast<unsigned char *>(sl) + al128(size_t(g.scap) * 16));
  __shared__ int s_late;
  {
    const int4 *src = reinterpret_cast<const int4 *>(g.stage + P.stage0);
    int4 *dst = reinterpret_cast<int4 *>(st);
    for (int i = tid; i < 2 * (nst + 1); i += NT) dst[i] = src[i];   // one more: the end of the push list
    for (int i = tid; i < P.nslice; i += NT) sl[i] = g.sl[P.slice0 + i];
  }
  const int2 *srow = g.srow + P.slice0;
  if (tid == 0) {
    for (int q = 0; q < kDeepBars; q++) {
      mbar_init(bar + q, 1);
      mbar_init(done + q, SW);
    }
    s_late = 0;
  }
  if (g.ctas > 1)
    for (int i = tid; i < nst; i += NT) mbar_init(halo + i, 1);
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
#pragma unroll 4
  for (int i = wi; i < P.nslice; i += NT / 32) {           // the right-hand side
    const int2 sr = srow[i];
    const int p = g.sl[P.slice0 + i].y >> 6;
    if (ln < sr.y) zs[p + ln] = x[sr.x + ln];
  }
  __syncthreads();
  if (g.ctas > 1) {
    for (int i = tid; i < nst; i += NT) mbar_expect_tx(halo + i, unsigned(st[i].halo) * unsigned(sizeof(T)));
    __syncwarp();
    cluster_sync_all();
  }
  auto is_late = [&]() { return *(volatile int *)&s_late != 0; };
  auto give_up = [&]() { atomicExch(&s_late, 1); *err = 1; };
  if (wi == 2 * SW) {
    // ---- the copy and push warp
    int jn = 0;            // next stage to bring in
    auto produce = [&](int jc) {                           // stages from jc on are live
      const int lim = jc < nst ? st[jc].lin + g.ring_bytes / 128 : 0x7fffffff;
      while (jn < nst && jn - jc < kDeepBars) {
        const DeepStage s = st[jn];
        if (s.lin + s.bytes > lim) break;
        uint64_t *bj = bar + (jn % kDeepBars);
        mbar_expect_tx(bj, unsigned(s.bytes) * 128u);
        tma_load_1d(ring + size_t(s.pos) * 128, (jn < P.nfwd ? pk_l : pk_u) + size_t(s.src) * 128,
                    unsigned(s.bytes) * 128u, bj);
        jn++;
      }
    };
    if (ln == 0) produce(0);
    const uint32_t zb = smem_u32(zs), hb = smem_u32(halo);
    int4 pe = make_int4(0, 0, 0, 0);                       // this lane's first push of the next stage
    if (nst > 0 && st[0].push + ln < st[1].push) pe = g.push[st[0].push + ln];
    bool late = false;
    // two loops, the second only for give_up_at: a test for it in the loop took 7 % of
    // a solve with narrow levels
    const int jt = give_up_at >= 0 && blockIdx.x == gridDim.x - 1 ? min(nst, give_up_at + 1) : nst;
    for (int j = 0, seg = 0; seg < 2; seg++) {
      if (seg == 1 && j < nst) give_up();
      for (const int je = seg == 0 ? jt : nst; j < je; j++) {
        const int p0 = st[j].push + ln, p1 = st[j + 1].push;
        // the sets run ahead of this warp by fewer than kDeepBars levels: it
        // brings in level j + kDeepBars only after level j
        uint64_t *dj = done + (j % kDeepBars);
        const unsigned par = unsigned(j / kDeepBars) & 1u;
        if (!late && !mbar_try_wait(dj, par)) {
          const unsigned long long t0 = gtimer_ns();
          while (!mbar_try_wait(dj, par)) {
            if (is_late()) break;
            if (gtimer_ns() - t0 > limit_ns) { give_up(); break; }
          }
        }
        late = __any_sync(0xffffffffu, is_late());
        for (int p = p0; p < p1; p += 32) {
          if (p != p0) pe = g.push[p];
          st_async(cluster_map(zb + unsigned(pe.z) * unsigned(sizeof(T)), pe.y), zs[pe.x],
                   cluster_map(hb + unsigned(pe.w) * 8u, pe.y));
        }
        if (j + 1 < nst && p1 + ln < st[j + 2].push) pe = g.push[p1 + ln];
        if (ln == 0 && !late) {
          // the level is done with its place in the ring: order its reads before
          // the copies into it
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
          produce(j + 1);
        }
        __syncwarp();
      }
    }
    if (ln == 0) {
      // every issued copy has arrived before the CTA may leave (on the normal
      // way all have been waited for by the levels that read them)
      const unsigned long long t0 = gtimer_ns();
      for (int q = max(0, jn - kDeepBars); q < jn; q++)
        while (!mbar_try_wait(bar + (q % kDeepBars), unsigned(q / kDeepBars) & 1u))
          if (gtimer_ns() - t0 > kDeepExitWaitNs) break;
    }
    __syncwarp();
  } else {
    // ---- set wi / SW: levels of its parity; this warp's slices a + ws, a + ws + SW, ...
    const int set = wi / SW, ws = wi % SW;
    constexpr int U = 4;
    // nr: rows from this warp's slice on; zp: this lane's place, zi: the same, a spare
    // place past the slice's last row
    int a = 0, nr = 0, w = 0, hl = 0, zp = 0, zi = 0;
    T acc = T(0), dr = T(0), av[U];
    int ad[U];
    const unsigned char *pe = nullptr;
    auto wait_for = [&](uint64_t *mb, unsigned par, bool peer) {
      if (peer ? mbar_try_wait_cluster(mb, par) : mbar_try_wait(mb, par)) return true;
      const unsigned long long t0 = gtimer_ns();
      while (!(peer ? mbar_try_wait_cluster(mb, par) : mbar_try_wait(mb, par))) {
        if (is_late()) return false;
        if (gtimer_ns() - t0 > limit_ns) { give_up(); return false; }
      }
      return true;
    };
    auto entry = [&](int k, T &v) {
      v = reinterpret_cast<const T *>(pe)[k * 32 + ln];
      return reinterpret_cast<const int *>(pe + size_t(w) * 32 * sizeof(T))[k * 32 + ln];
    };
    auto open_slice = [&](const DeepStage &s, bool fwd, int i) {
      const int4 e = sl[i];
      w = deep_w(e, fwd ? 0 : 1);
      zi = ln < nr ? zp : g.zcap;
      pe = ring + size_t(s.pos + (fwd ? e.x : e.z) - s.src) * 128;
      dr = reinterpret_cast<const T *>(pe + size_t(w) * 32 * (sizeof(T) + 4))[ln];
      acc = zs[zi];
#pragma unroll
      for (int u = 0; u < U; u++)
        if (u < w) ad[u] = entry(u, av[u]);
    };
    // all of a level that does not depend on other rows' results.  Once the CTA is
    // late no warp reads the ring again, also one that had no slice at the stage
    // that never came: 32 stages on, the parity it would wait for is that of a phase
    // long over.  (A stage has a warp that waits for it, so every warp sees it late
    // before then.)
    bool ok = true;
    auto prefetch = [&](int j) {
      const DeepStage s = st[j];
      const bool late = is_late();             // (read while the wait is under way)
      a = s.a + ws;
      nr = s.rows - ws * 32;
      zp = s.z0 + ws * 32 + ln;
      hl = s.halo;
      if (nr > 0) {
        ok = ok && wait_for(bar + (j % kDeepBars), unsigned(j / kDeepBars) & 1u, false) && !late;
        if (ok) open_slice(s, j < P.nfwd, a);
      }
    };
    if (set < nst) prefetch(set);
    __syncwarp();
    for (int j = set; j < nst; j += 2) {
      if (j > 0) set_sync<SW>(set ^ 1);                        // level j - 1 is done
      if (hl > 0 && nr > 0) ok = ok && wait_for(halo + j, 0u, true);
      // the turn: the top level's forward results were not there to prefetch
      // (every other backward level is at least three levels after its forward)
      if (j == P.nfwd && nr > 0) acc = zs[zi];
      for (int i = a; ok && nr > 0; i += SW, nr -= SW * 32, zp += SW * 32) {
        if (i != a) open_slice(st[j], j < P.nfwd, i);
        switch (min(w, U + 1)) {
          case 0: break;
          case 1: acc = deep_chain<T, 1>(acc, zs, ad, av); break;
          case 2: acc = deep_chain<T, 2>(acc, zs, ad, av); break;
          case 3: acc = deep_chain<T, 3>(acc, zs, ad, av); break;
          case 4: acc = deep_chain<T, 4>(acc, zs, ad, av); break;
          default:
            acc = deep_chain<T, 4>(acc, zs, ad, av);
            for (int k0 = U; k0 < w; k0 += U) {            // w is a multiple of U
              T zv[U];
#pragma unroll
              for (int u = 0; u < U; u++) ad[u] = entry(k0 + u, av[u]);
#pragma unroll
              for (int u = 0; u < U; u++) zv[u] = zs[ad[u]];
#pragma unroll
              for (int u = 0; u < U; u++) acc -= av[u] * zv[u];
            }
        }
        zs[zi] = acc * dr;
      }
      __syncwarp();
      if (j + 1 < nst) set_arrive<SW>(set);
      if (ln == 0) mbar_arrive(done + (j % kDeepBars));
      if (j + 2 < nst) prefetch(j + 2);
      __syncwarp();
    }
  }
  __syncthreads();
#pragma unroll 4
  for (int i = wi; i < P.nslice; i += NT / 32) {           // the result
    const int2 sr = srow[i];
    if (ln < sr.y) z[sr.x + ln] = zs[(sl[i].y >> 6) + ln];
  }
  __syncwarp();
  if (g.ctas > 1) {
    cluster_sync_all();
    if (is_late()) {
      // its peers' last pushes into this CTA
      const unsigned long long t0 = gtimer_ns();
      for (int i = tid; i < nst; i += NT)
        while (!mbar_try_wait_cluster(halo + i, 0u))
          if (gtimer_ns() - t0 > kDeepExitWaitNs) break;
    }
  }
}

// ------------------------------------------------------------ narrow blocks
// Exact factors in natural order have about one row per level and tens of
// entries per row (a 31 x 31 box: 961 levels of one row, 31 entries): their
// chain is the rows themselves, and a thread per row left it at 31 dependent
// FMAs of 64 cycles per row.  Such a block is taken in panels of 32 consecutive
// rows instead: t = x - (entries left of the panel) z, four threads per row,
// then z = L_JJ^-1 t with the inverse of the panel's own triangle, formed once
// per numeric setup; backward likewise with the entries below the panel and the
// transposed inverse.  A panel is two dot products of about 8 FMAs per thread
// and two barriers.  One CTA per block, its solution in shared memory; the next
// panel's data is loaded while the current one computes.
// 2 x 2 exact blocks of 31 x 31: 3.63 ms per solve -> 0.077 ms (62 panel steps
// of 1.24 us; its C_a of 252 rows, 221 levels: 441 launches -> 0.025 ms).
constexpr int kPanelRows = 32, kPanelLanes = 4, kPanelNT = kPanelRows * kPanelLanes;
constexpr int kPanelInv = kPanelRows / kPanelLanes;   // inverse entries per thread
struct PanelGeo {
  int nblk, rcap;            // blocks, rows of the largest
  const int2 *blk;           // per block: {first panel, panels}
  const int4 *pan;           // per panel: {first entry row / kPanelNT of L, width of L, the same of L^T}
  const int2 *prow;          // per panel: {first row, rows}
  const int *col;            // entries: position of the row in the block
};

// the panels' inverse triangles, row-distributed for both directions:
// inv[((2 J + dir) kPanelInv + q) kPanelNT + 4 r + g] = (L^-1)[r][4 q + g], for
// dir 1 (L^-1)[4 q + g][r].  One warp per panel.
template <typename T>
__global__ void k_panel_inv(const int2 *prow, const int *f_rp, const int *f_ci, const double *fval,
                            T *inv) {
  __shared__ double L[kPanelRows][kPanelRows + 1], X[kPanelRows][kPanelRows + 1];
  const int J = blockIdx.x, ln = threadIdx.x;
  const int2 pr = prow[J];
  for (int r = 0; r < kPanelRows; r++) { L[r][ln] = 0.0; X[r][ln] = 0.0; }
  __syncwarp();
  if (ln < pr.y)
    for (int q = f_rp[pr.x + ln]; q < f_rp[pr.x + ln + 1]; q++)
      if (f_ci[q] >= pr.x) L[ln][f_ci[q] - pr.x] = fval[q];
  __syncwarp();
  // lane c: column c of the inverse
  if (ln < pr.y)
    for (int r = ln; r < pr.y; r++) {
      double v = r == ln ? 1.0 : 0.0;
      for (int c = ln; c < r; c++) v -= L[r][c] * X[c][ln];
      X[r][ln] = v / L[r][r];
    }
  __syncwarp();
  for (int dir = 0; dir < 2; dir++)
    for (int q = 0; q < kPanelInv; q++)
      for (int h = 0; h < kPanelLanes; h++) {
        const int t = h * 32 + ln, r = t / kPanelLanes, c = q * kPanelLanes + t % kPanelLanes;
        inv[((size_t)(2 * J + dir) * kPanelInv + q) * kPanelNT + t] = T(dir ? X[c][r] : X[r][c]);
      }
}

// entry values (every numeric setup): slot src of L or, in the rows of entries
// marked in dir, of L^T
template <typename T>
__global__ void k_panel_vals(long long n, const int *src, const unsigned char *dir, const T *lval, const T *uval,
                             T *ent) {
  const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= n) return;
  const int q = src[e];
  ent[e] = q < 0 ? T(0) : (dir[e / kPanelNT] ? uval : lval)[q];
}

template <typename T>
inline size_t panel_smem_bytes(int rcap) { return (size_t(rcap) + kPanelRows) * sizeof(T); }

// one panel's data in registers
template <typename T, int W>
struct PanelRegs {
  T v[W], iv[kPanelInv];
  int c[W];
};

// z = (L L^T)^-1 x on the blocks' rows.  x and z: device order.
template <typename T>
__global__ void __launch_bounds__(kPanelNT)
k_panel_solve(PanelGeo g, const T *ent, const T *inv, const T *x, T *z, const int *gate) {
  if (gate && *gate) return;
  extern __shared__ __align__(128) unsigned char smraw[];
  T *zs = reinterpret_cast<T *>(smraw), *ts = zs + g.rcap;
  constexpr int W = 8;                          // entries per thread held ahead
  const int tid = threadIdx.x, r = tid / kPanelLanes, gl = tid % kPanelLanes;
  const int2 bp = g.blk[blockIdx.x];
  if (bp.y == 0) return;
  const int row0 = g.prow[bp.x].x, nb = g.prow[bp.x + bp.y - 1].x + g.prow[bp.x + bp.y - 1].y - row0;
  for (int i = tid; i < nb; i += kPanelNT) zs[i] = x[row0 + i];
  const int steps = 2 * bp.y;
  PanelRegs<T, W> N;
  int nw = 0, noff = 0;
  // step t: panel t forward, or panel steps - 1 - t backward
  auto load = [&](int t) {
    const bool fwd = t < bp.y;
    const int J = bp.x + (fwd ? t : steps - 1 - t);
    const int4 pn = g.pan[J];
    noff = fwd ? pn.x : pn.z;
    nw = fwd ? pn.y : pn.w;
#pragma unroll
    for (int u = 0; u < W; u++)
      if (u < nw) {
        const size_t e = size_t(noff + u) * kPanelNT + tid;
        N.v[u] = ent[e];
        N.c[u] = g.col[e];
      } else {
        N.v[u] = T(0);
        N.c[u] = 0;
      }
    const T *ip = inv + ((size_t)(2 * J + (fwd ? 0 : 1)) * kPanelInv) * kPanelNT + tid;
#pragma unroll
    for (int q = 0; q < kPanelInv; q++) N.iv[q] = ip[q * kPanelNT];
  };
  load(0);
  __syncthreads();
  for (int t = 0; t < steps; t++) {
    const bool fwd = t < bp.y;
    const int J = fwd ? t : steps - 1 - t, p0 = J * kPanelRows;
    const PanelRegs<T, W> C = N;
    const int w = nw, off = noff;
    if (t + 1 < steps) load(t + 1);
    // entries outside the panel
    T a = T(0);
    if (w > 0) {                                // fours of entries without a test each (padding: 0 * z_0)
#pragma unroll
      for (int u = 0; u < 4; u++) a += C.v[u] * zs[C.c[u]];
    }
    if (w > 4) {
#pragma unroll
      for (int u = 4; u < W; u++) a += C.v[u] * zs[C.c[u]];
    }
    for (int u = W; u < w; u++) {
      const size_t e = size_t(off + u) * kPanelNT + tid;
      a += ent[e] * zs[g.col[e]];
    }
#pragma unroll
    for (int d = 1; d < kPanelLanes; d <<= 1) a += __shfl_xor_sync(0xffffffffu, a, d);
    if (gl == 0) ts[r] = p0 + r < nb ? zs[p0 + r] - a : T(0);
    __syncthreads();
    // the panel's triangle; rows (columns) past a warp's last have no entries
    // there, so each warp stops at its own
    const int wq = tid >> 5, lo = fwd ? 0 : 2 * wq, hi = fwd ? 2 * wq + 2 : kPanelInv;
    T s = T(0);
#pragma unroll
    for (int q = 0; q < kPanelInv; q += 2)
      if (q >= lo && q < hi) {
        s += C.iv[q] * ts[q * kPanelLanes + gl];
        s += C.iv[q + 1] * ts[(q + 1) * kPanelLanes + gl];
      }
#pragma unroll
    for (int d = 1; d < kPanelLanes; d <<= 1) s += __shfl_xor_sync(0xffffffffu, s, d);
    if (gl == 0 && p0 + r < nb) zs[p0 + r] = s;
    __syncthreads();
  }
  for (int i = tid; i < nb; i += kPanelNT) z[row0 + i] = zs[i];
}

}  // namespace ddlr
