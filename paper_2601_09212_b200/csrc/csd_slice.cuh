// Calls in stream order with few sequences or unaligned rows (sm_100a): a sequence's rows are split over the
// VOCABULARY, one slice of every row per block, and the blocks of a sequence form one thread-block cluster of up to 16.
//
// Such a call is bound by latency, not by bandwidth.  The position split of csd_fused.cuh gives a block two rows
// whatever the vocabulary, at most gamma blocks to a sequence, and fetches the draw's rows again twice.  Split
// over the vocabulary, every block has the same work for any gamma, up to 16 blocks serve one sequence, and where a
// slice of all rows fits the block's shared memory each logit is fetched once:
//   1. every row's slice comes in by one bulk copy per array, as many rows at once as fit (the rest follow as slots
//      free up);
//   2. each warp takes units of 512 logits and leaves (m, s) of its part of each row;
//   3. the parts go into every block of the cluster (distributed shared memory); one cluster barrier later every
//      block knows all rows' normalisers, so every warp runs all accept tests itself and nothing further is exchanged
//      to agree on the first rejection;
//   4. each block sums Eq. opt_G over its slice of the two rows, from shared memory; the slices' totals go into every
//      block; one cluster barrier later the block whose slice holds the crossing C(x) > u Z picks the token and emits.
#pragma once
#include "csd_fused.cuh"

namespace csd {

constexpr int kSliceThreads = 512;      // two blocks per SM
constexpr int kSliceWarps = kSliceThreads / 32;
constexpr int kSliceCluster = 16;       // blocks of a sequence (above 8: a non-portable cluster size)
constexpr int kSliceRows = 128;
constexpr int kSliceUnit = 512;         // logits of a warp's unit of work: 16 per lane
static_assert(kSliceRows <= kBlockRows, "a block's row results live in RowStats");

// How a call is laid out; chosen by the host.
struct SliceGeo {
  int slots, slot_bytes;   // rows whose slices the block holds at once; bytes of one (all arrays)
  int vec_ok;              // rows are whole 16-byte vectors at 16-byte aligned addresses
  int wpr_log2;            // 2^this warps work on a row at once
  int direct;              // the warps' parts of a row go to the other blocks as they are (else merged first)
  int rec_off, stash_off, tile_off, arena_off;   // dynamic shared memory after SliceSmem: offsets in bytes
};
struct SliceArgs {
  FusedArgs f;
  SliceGeo g;
};

struct SliceSmem {
  alignas(8) uint64_t full[kSliceRows];
  int left[kSliceRows];      // warps that have yet to read the slot's row
  int issued[kSliceRows];    // rows announced to the slot's barrier so far
  int cur[kSliceRows];       // the latest of them
  uint32_t xflag[kSliceCluster];        // a bounded wait gave up in that block
  double zs[2][kSliceCluster];          // by parity of the pass: its total over each block's slice
  RowStats rs;
  int abort;
  FinishSmem fin;
  FinishStage fst;
};
constexpr int kSliceHeader = (int)((sizeof(SliceSmem) + 127) / 128 * 128);

__device__ __forceinline__ uint32_t cluster_map(const void* local, uint32_t rank) {
  uint32_t remote;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(smem_addr(local)), "r"(rank));
  return remote;
}
__device__ __forceinline__ void cluster_store_f2(float2* local, uint32_t rank, float2 v) {
  asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(cluster_map(local, rank)), "f"(v.x), "f"(v.y) : "memory");
}

// ---- the block's place -----------------------------------------------------------------------------------------
template <typename T, bool CFG>
struct Slice {
  static constexpr int VEC = Elem<T>::kVec;
  static constexpr int TILE = 32 * VEC;
  static constexpr int ES = (int)sizeof(T);
  static constexpr int ARR = CFG ? 2 : 1;
  const SliceArgs& a;
  SliceSmem& sm;
  unsigned char* base;     // the dynamic shared memory
  BlockShare sh;
  int c, me, b;            // blocks of the sequence, this block's rank, the sequence
  int R;                   // rows
  int my_tiles, x_begin, n, upr;   // the slice: tiles of the draw, first element, elements, units
  int tid, lane, warp;

  __device__ __forceinline__ Slice(const SliceArgs& args, SliceSmem& s, unsigned char* raw) : a(args), sm(s), base(raw) {
    tid = threadIdx.x; lane = tid & 31; warp = tid >> 5;
    const FinishArgs& f = a.f.fin;
    c = a.f.ctas_per_seq;
    b = blockIdx.x / c;
    me = blockIdx.x - b * c;
    const int ntiles = (f.V + TILE - 1) / TILE;   // a slice is a whole number of tiles of the draw
    const int tile0 = (int)((long long)ntiles * me / c);
    my_tiles = (int)((long long)ntiles * (me + 1) / c) - tile0;
    x_begin = tile0 * TILE;
    n = min(f.V, x_begin + my_tiles * TILE) - x_begin;
    upr = (n + kSliceUnit - 1) / kSliceUnit;
    sh.seq_begin = b; sh.seq_end = b + 1;
    sh.pos_begin = 0; sh.pos_end = f.gamma;
    sh.bonus = f.T == f.gamma + 1 ? 1 : 0;
    sh.rows_per_seq = 2 * f.gamma + sh.bonus;
    sh.n_rows = sh.rows_per_seq;
    sh.slot = me;
    R = sh.n_rows;
  }
  __device__ __forceinline__ Row<T, CFG> row(int r) const {
    int bb, which, i;
    local_row(sh, r, a.f.fin.gamma, bb, which, i);
    return row_at<T, CFG>(a.f.fin, bb, which, i);
  }
  __device__ __forceinline__ int slot_of(int r) const {   // r modulo slots (usually r itself)
    while (r >= a.g.slots) r -= a.g.slots;
    return r;
  }
  __device__ __forceinline__ unsigned char* slot(int r) const { return base + a.g.arena_off + slot_of(r) * a.g.slot_bytes; }

  // One thread: announces and starts the copies of row r's slice into its slot.  Unaligned slices are copied from the
  // 16-byte boundary below their first element to the one above their last (a granule that holds an element of the
  // row lies within a page of the row's allocation); their elements then sit a few bytes into the slot.
  __device__ __forceinline__ void issue(const int r, const bool drop = false) const {
    const int s = slot_of(r);
    unsigned char* dst = slot(r);
    const Row<T, CFG> w = row(r);
    *(volatile int*)&sm.cur[s] = r;
    ++sm.issued[s];
    if (a.g.vec_ok) {
      const uint32_t bytes = (uint32_t)(n * ES);
      mbar_expect_tx(&sm.full[s], bytes * ARR);
      if (drop) return;   // (test aid, see FusedArgs)
      bulk_load_row(dst, w.cond, x_begin, bytes, a.f.fin.V, &sm.full[s]);
      if (CFG) bulk_load_row(dst + a.g.slot_bytes / 2, w.uncond, x_begin, bytes, a.f.fin.V, &sm.full[s]);
    } else {
#ifdef CSD_CHECKED
      if (!checked_ok(x_begin, n, a.f.fin.V, 4)) return;
#endif
      uintptr_t from[2], to[2];
      uint32_t total = 0;
#pragma unroll
      for (int k = 0; k < ARR; ++k) {
        from[k] = (uintptr_t)((k == 0 ? w.cond : w.uncond) + x_begin);
        to[k] = (from[k] + (uintptr_t)(n * ES) + 15) & ~(uintptr_t)15;
        from[k] &= ~(uintptr_t)15;
        total += (uint32_t)(to[k] - from[k]);
      }
      mbar_expect_tx(&sm.full[s], total);
      if (drop) return;
#pragma unroll
      for (int k = 0; k < ARR; ++k)
        bulk_load(dst + k * (a.g.slot_bytes / 2), (const void*)from[k], (uint32_t)(to[k] - from[k]), &sm.full[s]);
    }
  }
  // One warp: row r's slice has arrived.  A slot's later rows are announced only when the row before has been read
  // by everybody; a warp that had no part in that row must not take its barrier's phase for this row's.
  __device__ __forceinline__ bool wait_row(const int r) const {
    if (r < a.g.slots) return mbar_wait(&sm.full[r], 0, a.f.wait_limit);
    const int s = slot_of(r);
    if (*(volatile int*)&sm.cur[s] != r) {
      const long long t0 = clock64();
      while (*(volatile int*)&sm.cur[s] != r)
        if (clock64() - t0 > a.f.wait_limit) return false;
    }
    __syncwarp();
    return mbar_wait(&sm.full[s], (uint32_t)(r / a.g.slots) & 1u, a.f.wait_limit);
  }
  // This warp has read its units of row r: the row's last reader hands the slot to the row that follows in it.
  __device__ __forceinline__ void release_row(const int r, const bool ok) const {
    if (a.g.slots >= R) return;
    __syncwarp();
    if (lane == 0) {
      const int s = slot_of(r);
      if (!ok) *(volatile int*)&sm.abort = 1;
      __threadfence_block();
      if (atom_add_shared(&sm.left[s], -1) == 1) {
        sm.left[s] = 1 << a.g.wpr_log2;
        __threadfence_block();
        if (r + a.g.slots < R && *(volatile int*)&sm.abort == 0) {
          fence_before_bulk();
          issue(r + a.g.slots);
        }
      }
    }
  }
  // Whole block: row r's slice is in its slot (a row that had made room for a later one comes back, an L2 hit).
  // False if the wait gave up.
  __device__ __forceinline__ bool need(const int r) const {
    const int s = slot_of(r);
    __syncthreads();   // everybody is done with what the slot holds
    if (sm.cur[s] == r) return true;
    __syncthreads();
    if (tid == 0) { fence_before_bulk(); issue(r); }
    __syncthreads();
    return mbar_wait(&sm.full[s], (uint32_t)(sm.issued[s] - 1) & 1u, a.f.wait_limit);
  }
  // where row r's slice begins in its slot, per array
  __device__ __forceinline__ void slice_at(const int r, const unsigned char*& p, const unsigned char*& pu) const {
    p = slot(r);
    pu = p + a.g.slot_bytes / 2;
    if (!a.g.vec_ok) {
      const Row<T, CFG> w = row(r);
      p += (uintptr_t)(w.cond + x_begin) & 15u;
      if (CFG) pu += (uintptr_t)(w.uncond + x_begin) & 15u;
    }
  }
  // The 16 values of this lane of unit k (value e is element unit_index(e) of the unit); what lies beyond the slice
  // reads -inf.
  __device__ __forceinline__ void unit(const unsigned char* p, const unsigned char* pu, const int k, float (&z)[16]) const {
    const int m = n - k * kSliceUnit;   // elements from here on
    p += k * kSliceUnit * ES;
    pu += k * kSliceUnit * ES;
    const float scale = a.f.fin.cfg_scale;
    if (a.g.vec_ok) {
#pragma unroll
      for (int v = 0; v < 16 / VEC; ++v) {
        const int xo = (v * 32 + lane) * VEC;
        float zc[VEC];
        if (xo < m) {
          unpack_vec<T>(p + xo * ES, zc);
          if (CFG) {
            float zu[VEC];
            unpack_vec<T>(pu + xo * ES, zu);
            cfg_mix_vec<VEC>(zc, zu, scale);
          }
        } else {
#pragma unroll
          for (int e = 0; e < VEC; ++e) zc[e] = CSD_NEG_INF;
        }
#pragma unroll
        for (int e = 0; e < VEC; ++e) z[v * VEC + e] = zc[e];
      }
    } else {   // (consecutive lanes, consecutive elements: no bank conflicts whatever the row's offset)
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        const int xo = i * 32 + lane;
        z[i] = CSD_NEG_INF;
        if (xo < m) {
          z[i] = load_scalar_smem<T>(p + xo * ES);
          if (CFG) z[i] = cfg_mix(z[i], load_scalar_smem<T>(pu + xo * ES), scale);
        }
      }
    }
  }
  __device__ __forceinline__ int unit_index(const int e) const {
    return a.g.vec_ok ? (e / VEC * 32 + lane) * VEC + e % VEC : e * 32 + lane;
  }
  // VEC consecutive values from element xo of the slice on; beyond its end -inf
  __device__ __forceinline__ void vec_at(const unsigned char* p, const unsigned char* pu, const int xo, float (&z)[VEC]) const {
    const float scale = a.f.fin.cfg_scale;
    if (a.g.vec_ok && xo < n) {
      unpack_vec<T>(p + xo * ES, z);
      if (CFG) {
        float zu[VEC];
        unpack_vec<T>(pu + xo * ES, zu);
        cfg_mix_vec<VEC>(z, zu, scale);
      }
    } else {
#pragma unroll
      for (int e = 0; e < VEC; ++e) {
        z[e] = CSD_NEG_INF;
        if (xo + e < n) {
          z[e] = load_scalar_smem<T>(p + (xo + e) * ES);
          if (CFG) z[e] = cfg_mix(z[e], load_scalar_smem<T>(pu + (xo + e) * ES), scale);
        }
      }
    }
  }
  // A pass's total over all slices: `mine` (valid in warp 0) is this block's.  Every thread gets the total Z, and in
  // lane q block q's total zk and the running total incl.
  __device__ __forceinline__ double total(const double mine, const int parity, double& zk, double& incl) const {
    if (warp == 0 && lane < c) cluster_store_f64(&sm.zs[parity][me], (uint32_t)lane, mine);
    if (c > 1) { cluster_arrive(); cluster_wait(); }
    else __syncthreads();
    zk = lane < c ? sm.zs[parity][lane] : 0.0;
    incl = zk;
    for (int off = 1; off < c; off <<= 1) {
      const double t = __shfl_up_sync(0xffffffffu, incl, off);
      if (lane >= off) incl += t;
    }
    return __shfl_sync(0xffffffffu, incl, c - 1);
  }
  // sum of the block's tile sums, the same in every lane of warp 0
  __device__ __forceinline__ double my_total(const double* tile_sums) const {
    double z = 0.0;
    if (warp == 0) {
      for (int t = lane; t < my_tiles; t += 32) z += tile_sums[t];
#pragma unroll 1
      for (int off = my_tiles > 8 ? 16 : 4; off > 0; off >>= 1) z += __shfl_xor_sync(0xffffffffu, z, off);
      z = __shfl_sync(0xffffffffu, z, 0);   // (with up to eight tiles only the lowest lanes hold it)
    }
    return z;
  }
  // the block whose slice holds the crossing C(x) > target; if rounding leaves none, the last with weight
  __device__ __forceinline__ int owner_of(const double target, const double zk, const double incl) const {
    const unsigned crossing = __ballot_sync(0xffffffffu, incl > target && zk > 0.0);
    const unsigned has_mass = __ballot_sync(0xffffffffu, zk > 0.0);
    return crossing ? __ffs(crossing) - 1 : 31 - __clz(has_mass);
  }
};

// Running statistics of a warp over units of one row, relative to a warp-uniform maximum (see verify_plain_kernel).
struct UnitStats {
  float M, s, nML, dlt;
  int cnt;
  __device__ __forceinline__ void begin() { M = CSD_NEG_INF; s = 0.0f; nML = 0.0f; dlt = 0.0f; cnt = 0; }
  __device__ __forceinline__ void add(const float (&z)[16]) {
    float m4[4] = {CSD_NEG_INF, CSD_NEG_INF, CSD_NEG_INF, CSD_NEG_INF};
#pragma unroll
    for (int e = 0; e < 16; ++e) m4[e & 3] = fmaxf(m4[e & 3], z[e]);
    int key = __float_as_int(fmaxf(fmaxf(m4[0], m4[1]), fmaxf(m4[2], m4[3])));
    key ^= (key >> 31) & 0x7fffffff;
    key = __reduce_max_sync(0xffffffffu, key);
    key ^= (key >> 31) & 0x7fffffff;
    const float wm = __int_as_float(key);
    if (wm > M) {   // a new maximum: what was counted as "equal to the maximum" becomes ordinary mass
      const float ML = wm * kLog2e, dlt_new = fmaf(wm, kLog2e, -ML);
      s = (s * ex2f(-dlt) + (float)cnt) * ex2f((M - wm) * kLog2e) * ex2f(dlt_new);
      cnt = 0;
      M = wm;
      nML = -ML;
      dlt = dlt_new;
    }
    const uint64_t l2e2 = pack2(kLog2e, kLog2e), nm2 = pack2(nML, nML);
    float acc[4] = {0.0f, 0.0f, 0.0f, 0.0f};
    if (wm == M) {   // values equal to the reference are counted, not summed
      int c2[2] = {0, 0};
#pragma unroll
      for (int e = 0; e < 16; e += 2) {
        float x0, x1;
        unpack2(fma2(pack2(z[e], z[e + 1]), l2e2, nm2), x0, x1);
        const float e0 = ex2f(x0), e1 = ex2f(x1);
        if (z[e] == M) ++c2[0]; else acc[e & 2] += e0;
        if (z[e + 1] == M) ++c2[1]; else acc[(e & 2) + 1] += e1;
      }
      cnt += c2[0] + c2[1];
    } else {
#pragma unroll
      for (int e = 0; e < 16; e += 2) {
        float x0, x1;
        unpack2(fma2(pack2(z[e], z[e + 1]), l2e2, nm2), x0, x1);
        acc[e & 2] += ex2f(x0);
        acc[(e & 2) + 1] += ex2f(x1);
      }
    }
    s += (acc[0] + acc[1]) + (acc[2] + acc[3]);
  }
  // (m, s) with sum exp(z) = (1 + s) exp(m); valid in every lane
  __device__ __forceinline__ float2 end() {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    cnt = __reduce_add_sync(0xffffffffu, cnt);
    return make_float2(M, s * ex2f(-dlt) + (float)(cnt - 1));
  }
};

// The parts of one row, one per lane of a group of `width` lanes (16 or 32; identity in lanes beyond), merged;
// valid in every lane of the group.
__device__ __forceinline__ float2 merge_parts(const float2 v, const int lane, const int width) {
  float m = v.x;
  for (int off = width >> 1; off > 0; off >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, off));
  // one part that attains the maximum keeps its "1 +" apart
  const unsigned group = width == 32 ? 0xffffffffu : 0xffffu << (lane & 16);
  const unsigned at = __ballot_sync(0xffffffffu, v.x == m) & group;
  float s = v.x == CSD_NEG_INF ? v.y - v.y : (1.0f + v.y) * ex2f((v.x - m) * kLog2e);   // (a NaN sum must survive)
  if (lane == __ffs(at) - 1) s = v.y;
  for (int off = width >> 1; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
  return make_float2(m, s);
}

// ---- phase 1: (m, s) of every row's parts --------------------------------------------------------------------------
// Returns false (in this warp) if a wait gave up.
template <typename T, bool CFG>
__device__ __forceinline__ bool slice_rows_plain(const Slice<T, CFG>& k) {
  float2* const parts = reinterpret_cast<float2*>(k.base + (k.a.g.direct ? k.a.g.rec_off : k.a.g.stash_off));
  const int wl = k.a.g.wpr_log2, part = k.warp & ((1 << wl) - 1), R = k.R;
  bool ok = true, peers = k.c == 1;
  for (int r = k.warp >> wl; r < R; r += kSliceWarps >> wl) {
    if (ok && !k.wait_row(r)) ok = false;
    const unsigned char *p, *pu;
    k.slice_at(r, p, pu);
    UnitStats st;
    st.begin();
    for (int u = part; u < k.upr; u += 1 << wl) {
      float z[16];
      k.unit(p, pu, u, z);
      st.add(z);
    }
    k.release_row(r, ok);
    const float2 v = st.end();
    if (k.a.g.direct) {   // into every block
      if (!peers) { cluster_wait(); peers = true; }   // every peer is running
      if (k.lane < k.c) cluster_store_f2(&parts[((k.me << wl) + part) * R + r], (uint32_t)k.lane, v);
    } else if (k.lane == 0) {
      parts[(r << wl) + part] = v;
    }
  }
  if (!peers) cluster_wait();
  return ok;
}

// Per tile of the slice, the sum of what `weight(xo)` returns for the lane's VEC values from element xo on.
template <typename T, bool CFG, typename W>
__device__ __forceinline__ void slice_tiles(const Slice<T, CFG>& k, double* tile_sums, W weight) {
  for (int t = k.warp; t < k.my_tiles; t += kSliceWarps) {
    const int xo = t * Slice<T, CFG>::TILE + k.lane * Elem<T>::kVec;
    float acc = xo < k.n ? weight(xo) : 0.0f;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
    if (k.lane == 0) tile_sums[t] = (double)acc;
  }
  __syncthreads();
}

// ---- phase 2: accept tests, the draw, the emitted block ---------------------------------------------------------------
template <typename T, bool CFG, bool TOPK>
__device__ __forceinline__ void slice_finish_chain(const Slice<T, CFG>& k, int status_any) {
  constexpr int VEC = Elem<T>::kVec;
  SliceSmem& sm = k.sm;
  const FinishArgs& f = k.a.f.fin;
  const int L = f.gamma, tid = k.tid, lane = k.lane, warp = k.warp, b = k.b;
  double* const tile_sums = reinterpret_cast<double*>(k.base + k.a.g.tile_off);
  // Eq. relax and the accept tests: every warp takes them all, one position per lane
  auto usable = [](const float2 v) { return v.x > CSD_NEG_INF && v.x < CSD_POS_INF && v.y >= 0.0f && v.y < CSD_POS_INF; };
  bool acc = true;
  int flag = 0;
  if (lane < L) {
    const float2 t = sm.rs.ms[2 * lane], d = sm.rs.ms[2 * lane + 1];
    const int tok = sm.fst.tok[lane];
    float fa = 0.0f, p = __int_as_float(0x7fc00000), q = p;
    if (!usable(t) || !usable(d)) flag = 1;
    else if (tok < 0 || tok >= f.V) flag = 2;
    else {
      const float zt = sm.rs.tokz[2 * lane], zd = sm.rs.tokz[2 * lane + 1];
      const float dt = (zt < sm.rs.thr[2 * lane] ? CSD_NEG_INF : zt) - t.x;
      const float dd = (zd < sm.rs.thr[2 * lane + 1] ? CSD_NEG_INF : zd) - d.x;
      p = ex2f(dt * kLog2e) / (1.0f + t.y);
      q = ex2f(dd * kLog2e) / (1.0f + d.y);
      if (dd == CSD_NEG_INF) fa = 1.0f;         // q = 0: p/q = +inf, and 0/0 := 1
      else if (dt == CSD_NEG_INF) fa = 0.0f;    // p = 0 < q
      else fa = fminf(1.0f, sm.fst.omega[lane] * ex2f((dt - dd) * kLog2e) * ((1.0f + d.y) / (1.0f + t.y)));
    }
    acc = sm.fst.uni[lane] <= fa;
    if (warp == 0 && k.me == 0) {
      if (f.dbg_p) f.dbg_p[(int64_t)b * L + lane] = p;
      if (f.dbg_q) f.dbg_q[(int64_t)b * L + lane] = q;
      if (f.dbg_f) f.dbg_f[(int64_t)b * L + lane] = fa;
    }
  }
  const unsigned rej = __ballot_sync(0xffffffffu, !acc);
  const int j = rej ? __ffs(rej) - 1 : L, tau = j;   // the for/break of Algorithm 1
  const bool rejected = j < L;
  int status = 0, token = -1;
  bool draw = false;
  PairCtx ctx;
  ctx.mode = 1;
  if (rejected) {
    status |= __shfl_sync(0xffffffffu, flag, j);
    draw = usable(sm.rs.ms[2 * j]);
    ctx.mode = usable(sm.rs.ms[2 * j + 1]) ? 0 : 1;
  } else if (k.sh.bonus) {
    draw = usable(sm.rs.ms[2 * L]);
    if (!draw) status |= 1;
  }
  double Z = 0.0;
  int owner = 0;   // the block that emits
  if (draw) {
    ctx.Mt = sm.rs.ms[2 * j].x; ctx.St = sm.rs.ms[2 * j].y;
    ctx.Md = j < L ? sm.rs.ms[2 * j + 1].x : 0.0f; ctx.Sd = j < L ? sm.rs.ms[2 * j + 1].y : 0.0f;
    ctx.inv_t = 1.0f / (1.0f + ctx.St);
    ctx.inv_den = ctx.inv_t / (1.0f + ctx.Sd);
    ctx.one_minus_omega = 1.0f - (j < L ? sm.fst.omega[j] : 0.0f);
    Row<T, CFG> ft, fd;   // (their filters)
    ft.thr = sm.rs.thr[2 * j];
    fd.thr = j < L ? sm.rs.thr[2 * j + 1] : CSD_NEG_INF;
    const int rt = 2 * j, rd = rejected ? 2 * j + 1 : 2 * j;   // local rows
    if (k.a.g.slots < k.R) {
      if (!k.need(rt)) status_any |= 8;
      if (rd != rt && !k.need(rd)) status_any |= 8;
    }
    const unsigned char *pt, *ptu, *pd, *pdu;
    k.slice_at(rt, pt, ptu);
    k.slice_at(rd, pd, pdu);
    auto load = [&](const int xo, float (&zt)[VEC], float (&zd)[VEC]) {
      k.vec_at(pt, ptu, xo, zt);
      if (ctx.mode == 0) k.vec_at(pd, pdu, xo, zd);
#pragma unroll
      for (int e = 0; e < VEC; ++e) {
        if (TOPK) zt[e] = ft.filter(zt[e]);
        zd[e] = ctx.mode == 0 ? (TOPK ? fd.filter(zd[e]) : zd[e]) : 0.0f;
      }
    };
    const float u = sm.fst.uni[L];
    for (int attempt = 0; attempt < 2; ++attempt) {
      slice_tiles(k, tile_sums, [&](const int xo) {
        float zt[VEC], zd[VEC], sum = 0.0f;
        load(xo, zt, zd);
#pragma unroll
        for (int e = 0; e < VEC; e += 2) {
          float g0, g1;
          weight_of_pair(zt[e], zt[e + 1], zd[e], zd[e + 1], ctx, g0, g1);
          sum += g0;
          sum += g1;
        }
        return sum;
      });
      double zk, incl;
      Z = k.total(k.my_total(tile_sums), attempt, zk, incl);
      if (!(Z > 0.0) || !(Z < (double)CSD_POS_INF)) {
        Z = 0.0;
        if (attempt == 0 && ctx.mode == 0) {   // empty positive part: fall back to G := P_j
          ctx.mode = 1;
          status |= 4;
          __syncthreads();
          continue;
        }
        break;   // nothing to draw from
      }
      const double target = (double)u * Z;
      owner = k.owner_of(target, zk, incl);
      if (owner == k.me) {
        if (warp == 0) {
          const double target_here = target - __shfl_sync(0xffffffffu, incl - zk, k.me);
          locate_crossing_tile(tile_sums, k.my_tiles, u, lane, sm.fin, &target_here);
          __syncwarp();
          const int t = sm.fin.pick_tile;
          int tok = -1;
          if (t >= 0) {
            const int xo = t * Slice<T, CFG>::TILE + lane * VEC;
            float zt[VEC], zd[VEC], g[VEC];
            load(xo, zt, zd);
#pragma unroll
            for (int e = 0; e < VEC; ++e) g[e] = xo + e < k.n ? weight_of(zt[e], zd[e], ctx) : 0.0f;
            tok = pick_in_tile<VEC>(g, k.x_begin + xo, sm.fin.pick_prefix, target_here, lane);
          }
          if (lane == 0) sm.fin.token = tok;
        }
        __syncthreads();
        token = sm.fin.token;
      }
      break;
    }
    if (f.dbg_G && Z > 0.0) {   // each block writes its slice
      float* G_out = f.dbg_G + (int64_t)b * f.V + k.x_begin;
      const float invZ = (float)(1.0 / Z);
      for (int xo = tid * VEC; xo < k.n; xo += kSliceThreads * VEC) {
        float zt[VEC], zd[VEC];
        load(xo, zt, zd);
#pragma unroll
        for (int e = 0; e < VEC; ++e)
          if (xo + e < k.n) G_out[xo + e] = weight_of(zt[e], zd[e], ctx) * invZ;
      }
    }
  }
  if (f.dbg_G && !(Z > 0.0))
    for (int x = tid; x < k.n; x += kSliceThreads) f.dbg_G[(int64_t)b * f.V + k.x_begin + x] = 0.0f;
  // ---- emit x_{1:tau+1} ----------------------------------------------------------------------------------------
  if (owner != k.me) return;
  if (tid <= L) f.out_tokens[(int64_t)b * (L + 1) + tid] = tid < tau ? sm.fst.tok[tid] : (tid == tau ? token : -1);
  if (tid == 0) {
    if (f.out_accept_len) f.out_accept_len[b] = tau;
    if (f.out_status) f.out_status[b] = status | status_any;
  }
}

template <typename T, bool CFG>
__global__ void __launch_bounds__(kSliceThreads, 2) verify_slice_kernel(const SliceArgs a) {
  extern __shared__ __align__(128) unsigned char fused_smem_raw[];
  SliceSmem& sm = *reinterpret_cast<SliceSmem*>(fused_smem_raw);
  const Slice<T, CFG> k(a, sm, fused_smem_raw);
  const FinishArgs& f = a.f.fin;
  const int tid = k.tid, lane = k.lane, c = k.c, R = k.R, slots = a.g.slots;

  if (tid < slots) { mbar_init(&sm.full[tid], 1); sm.left[tid] = 1 << a.g.wpr_log2; sm.issued[tid] = 0; sm.cur[tid] = -1; }
  if (tid == 0) sm.abort = 0;
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  __syncthreads();
  if (c > 1) cluster_arrive();   // first half; waited for before the first store to a peer
  call_begin(a.f.ordered, a.f.signal != 0);

  if (lane == 0)
    for (int r = k.warp; r < R && r < slots; r += kSliceWarps)
      k.issue(r, r == 0 && a.f.drop_first_copy != 0 && blockIdx.x == 0);
  // The copies are under way: the small inputs and the drafted tokens' logits (two dependent trips to memory) are
  // fetched in their shadow and put into shared memory when the rows have been read.  Thread r takes row r's token.
  const int L = f.gamma;
  int tok = -1;
  float uni = 0.0f, omega = 0.0f, ztok = CSD_POS_INF;
  if (tid <= L) uni = __ldcg(&f.uniforms[(int64_t)k.b * (L + 1) + tid]);
  if (tid < L) omega = __ldcg(&f.schedule[tid]);
  if (tid < 2 * L) {
    tok = __ldcg(&f.tokens[(int64_t)k.b * L + (tid >> 1)]);
    if (tok >= 0 && tok < f.V) ztok = k.row(tid).load_one(tok);
  }
  bool ok = slice_rows_plain<T, CFG>(k);
  if (tid <= L) sm.fst.uni[tid] = uni;
  if (tid < L) sm.fst.omega[tid] = omega >= 0.0f ? omega : 0.0f;
  if (tid < 2 * L && !(tid & 1)) sm.fst.tok[tid >> 1] = tok;
  if (tid < R) sm.rs.tokz[tid] = ztok;
  if (!ok) *(volatile int*)&sm.abort = 1;
  const int wl = a.g.wpr_log2;
  float2* const xs = reinterpret_cast<float2*>(fused_smem_raw + a.g.rec_off);   // [c][parts][R]
  if (!a.g.direct) {   // the warps' parts of a row are merged before they go to the other blocks
    __syncthreads();
    const float2* const stash = reinterpret_cast<const float2*>(fused_smem_raw + a.g.stash_off);
    for (int r0 = 2 * k.warp; r0 < R; r0 += 2 * kSliceWarps) {
      const int r = r0 + (lane >> 4), part = lane & 15;
      const float2 v = merge_parts((part < (1 << wl) && r < R) ? stash[(r << wl) + part] : make_float2(CSD_NEG_INF, -1.0f), lane, 16);
      if (part < c && r < R) cluster_store_f2(&xs[k.me * R + r], (uint32_t)part, v);
    }
  }
  __syncthreads();
  const bool aborted = sm.abort != 0;
  if (aborted && tid == 0) {
    if (a.f.error_flag) atomicExch(a.f.error_flag, 1);
    // copies that may still be in flight must land before the block leaves: each slot's latest, bounded
    for (int s = 0; s < slots; ++s)
      if (sm.issued[s] > 0) (void)mbar_wait(&sm.full[s], (uint32_t)(sm.issued[s] - 1) & 1u, a.f.wait_limit);
  }
  if (tid < c) cluster_store(&sm.xflag[k.me], (uint32_t)tid, aborted ? 1u : 0u);
  if (c > 1) { cluster_arrive(); cluster_wait(); }
  else __syncthreads();

  // ---- every row's statistics over the whole vocabulary ----------------------------------------------------------
  const int np = a.g.direct ? c << wl : c;   // parts of a row, at most 32
  if (np <= 16) {
    for (int r0 = 2 * k.warp; r0 < R; r0 += 2 * kSliceWarps) {
      const int r = r0 + (lane >> 4), q = lane & 15;
      const float2 v = merge_parts((q < np && r < R) ? xs[q * R + r] : make_float2(CSD_NEG_INF, -1.0f), lane, 16);
      if (q == 0 && r < R) { sm.rs.ms[r] = v; sm.rs.thr[r] = CSD_NEG_INF; }
    }
  } else {
    for (int r = k.warp; r < R; r += kSliceWarps) {
      const float2 v = merge_parts(lane < np ? xs[lane * R + r] : make_float2(CSD_NEG_INF, -1.0f), lane, 32);
      if (lane == 0) { sm.rs.ms[r] = v; sm.rs.thr[r] = CSD_NEG_INF; }
    }
  }
  int status_any = 0;
  for (int q = 0; q < c; ++q) status_any |= sm.xflag[q] ? 8 : 0;
  if (a.f.error_flag && __ldcg(a.f.error_flag)) status_any |= 8;
  __syncthreads();
  slice_finish_chain<T, CFG, false>(k, status_any);
}

}  // namespace csd
