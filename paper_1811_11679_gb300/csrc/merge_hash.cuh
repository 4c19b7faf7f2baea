// merge_hash.cuh -- annihilation over a flat hash table (the default path).
//
// The annihilation step (HANDE-QMC paper Sec. 2.4 and App. B: combine the
// spawned particles on each determinant, merge them into the sorted main list,
// apply the initiator rule to new determinants) needs an order only among the
// NEW determinants that survive it.  Populations are integers, so sums need no
// order at all: every spawn is one thread, whatever its key.
//   match   each spawn is searched in the main list: a table of block ends staged
//           in shared memory, then one aligned node of four keys per level (the
//           last keys of blocks of 4^l entries, written by the det pass), so a
//           level costs one 32-byte sector per key word instead of the two that
//           bisection reads.  A listed key: its amount is added to the entry.  A
//           new key: the first spawn to claim a hash slot represents the key,
//           later spawns with that key add into the representative's staged
//           amount and OR their initiator bit.  The slot holds a spawn index and
//           the staged keys are read-only here, so no key is published and any
//           key width works with one 32-bit compare-and-swap.
//   decide  final population of each listed entry (occupation rounding), 64
//           entries' keep bits in one word; each representative: initiator
//           rule, rounding, slot cleared, and if it survives its rank of
//           arrival among the survivors inserted in front of the same 64
//           entries.  The last block scans the group counts.
//   place   survivors copied group by group.
//   write   diagonal elements of the survivors; entries and survivors to their final places in the new list: an
//           entry's place follows from the keep bits and the survivors in front
//           of it, a survivor's rank in its group from counting smaller keys.
//           One thread closes the iteration meanwhile (shift, record).
// What bounds them: match by L1 passes (one 32-byte sector per lane and level) and
// L2 latency, decide and write by HBM and latency, the diagonal elements by the
// FP64 unit (their sums are ordered), which runs beside the copy of the other
// blocks.  Measured in us, the bucket kernels they replace (scatter, warp and
// block merges, scans, compaction, diagonals, record) -> these four: ueg 14e/38 at
// 1e6 walkers 220 -> 72, molecule at 1e7 240 -> 142, hubbard 2d 18 at 2.2e6 310 -> 118.
#pragma once

namespace hande {

constexpr int kMatchThreads = 512;
constexpr int kListThreads = 512;                     // decide and write: 16 groups per block
constexpr int kGroup = 64;                            // main-list entries per keep word
constexpr int kGroups = kListThreads / 32;            // groups per block tile (one warp each)
constexpr int kListTile = kGroup * kGroups;           // 1024 entries
constexpr int kRankChunk = 512;                       // sorted runs of a large group
template <int W>
__host__ __device__ constexpr int match_split() {     // staged search keys per block
  return 4096 / W;                                    // 32 KB
}

// block tiles of a list of n entries (positions 0 .. n, the last one behind the list)
__host__ __device__ __forceinline__ int64_t list_tiles(int64_t n) { return n / kListTile + 1; }

template <int W>
__device__ __forceinline__ uint32_t spawn_hash(const Key<W>& k) {
  uint64_t x = k.w[0];
#pragma unroll
  for (int j = 1; j < W; ++j) x = (x ^ (x >> 29)) * 0xBF58476D1CE4E5B9ull + k.w[j];
  x ^= x >> 32;
  x *= 0x9E3779B97F4A7C15ull;
  return (uint32_t)(x >> 32);
}
// slots used for ns spawns: a power of two of at least 2 ns (at most the table)
__device__ __forceinline__ uint32_t hash_mask(const Params& P, int64_t ns) {
  uint64_t m = 1024;
  while (m < 2 * (uint64_t)ns && m < P.hash_size) m <<= 1;
  return (uint32_t)(m - 1);
}

// The 32-element chunk of warp wid of a block in one round of the grid: in block
// order, or (spread) to all blocks before any block gets a second one.
__device__ __forceinline__ int64_t chunk_of(const VGrid vg, int wid, bool spread) {
  return spread ? (int64_t)wid * vg.n + vg.b : (int64_t)vg.b * (blockDim.x >> 5) + wid;
}

// ------------------------------------------------------------------ match
// One aligned 32-byte sector in one load.  The lanes of a warp read 32 different
// sectors, one L1 pass each: as two 16-byte loads a level took 64 passes, and
// the search of 1.4e6 spawns (43 000 warps) 60 us instead of 56.
__device__ __forceinline__ void load_node(const uint64_t* p, uint64_t (&w)[4]) {
  asm volatile("ld.global.nc.v4.u64 {%0, %1, %2, %3}, [%4];"
               : "=l"(w[0]), "=l"(w[1]), "=l"(w[2]), "=l"(w[3])
               : "l"(p));
}

// How many of the node's keys a[4 b .. 4 b + 3] (those below index `valid`) are
// below k; hit: one of them is k.  Every node is an aligned 32-byte sector per word.
template <int W>
__device__ __forceinline__ uint32_t node_below(const uint64_t* a, int64_t stride, uint32_t first, uint32_t valid,
                                               const Key<W>& k, bool& hit) {
  hit = false;
  if (first >= valid) return 0;   // past the last whole block: nothing to read
  bool lt[4], eq[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    eq[q] = first + q < valid;
    lt[q] = false;
  }
#pragma unroll
  for (int j = W - 1; j >= 0; --j) {
    uint64_t w[4];
    load_node(a + j * stride + first, w);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      lt[q] = lt[q] || (eq[q] && w[q] < k.w[j]);
      eq[q] = eq[q] && w[q] == k.w[j];
    }
  }
  hit = eq[0] || eq[1] || eq[2] || eq[3];
  return (uint32_t)lt[0] + (uint32_t)lt[1] + (uint32_t)lt[2] + (uint32_t)lt[3];
}

template <int W>
__device__ __forceinline__ void d_match(const Params& P, int cur, const VGrid vg) {
  constexpr int S = match_split<W>();
  __shared__ uint64_t ssp[W * S];
  __shared__ uint32_t swarp[kMatchThreads / 32];
  DevState* st = P.st;
  const int64_t ns = st->nspawn < P.scap ? st->nspawn : P.scap;
  const uint32_t n = (uint32_t)st->ndet[cur];
  // every block stages search keys, so spawns spread over all blocks only when
  // each block gets at least eight warps of them (UEG 1e6 walkers: 31 -> 28 us;
  // small replicas of a batch: 17 -> 20 us, hence the limit)
  const bool spread = ns >= (int64_t)vg.n * 256;
  if (__syncthreads_or((int)st->error) || chunk_of(vg, 0, spread) * 32 >= ns) return;
  const uint64_t* key = P.key[cur];
  unsigned long long* pop = (unsigned long long*)P.pop[cur];
  // block ends of level `top` go to shared memory: at most S of them, and no more
  // than an eighth of the spawns (every block stages them)
  const uint32_t most = ns / 8 < S ? (uint32_t)(ns / 8) : (uint32_t)S;
  int top = 1;
  while ((n >> (2 * top)) > most && top < kEndLevels - 1) ++top;
  const int nsp = (int)(n >> (2 * top));
  for (int i = threadIdx.x; i < nsp; i += blockDim.x) {
#pragma unroll
    for (int j = 0; j < W; ++j) ssp[j * S + i] = P.s_end[top][j * end_stride(P.cap, top) + i];
  }
  __syncthreads();
  const uint32_t mask = hash_mask(P, ns);
  const int lane = (int)warp_lane(), wid = (int)(threadIdx.x >> 5);
  const int64_t step = (int64_t)vg.n * blockDim.x;
  for (int64_t s0 = chunk_of(vg, 0, spread) * 32; s0 < ns; s0 += step) {
    const int64_t s = s0 + (spread ? (int64_t)wid * vg.n : wid) * 32 + lane;
    bool rep = false;
    if (s < ns) {
      const Key<W> k = load_key<W>(P.s_key, P.scap, s);
      const int64_t amt = P.s_amt[s];
      uint32_t* meta = reinterpret_cast<uint32_t*>(P.s_meta + s);   // {slot << 1 | initiator, position}
      int lo = 0, hi = nsp;   // block ends below k
      while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (key_lt<W>(load_key<W>(ssp, S, mid), k)) lo = mid + 1;
        else hi = mid;
      }
      uint32_t pos = (uint32_t)lo;   // the block of level l that holds the first entry >= k
      bool hit = false;
      for (int l = top - 1; l >= 0; --l)
        pos = 4 * pos + node_below<W>(l ? P.s_end[l] : key, l ? end_stride(P.cap, l) : P.cap, 4 * pos, n >> (2 * l), k, hit);
      if (hit) {
        atomicAdd(&pop[pos], (unsigned long long)amt);
      } else {
        uint32_t h = spawn_hash<W>(k) & mask;
        for (uint32_t probe = 0; probe <= mask; ++probe) {
          const uint32_t old = atomicCAS(&P.hash_tab[h], 0u, (uint32_t)s + 1u);
          if (old == 0) {
            rep = true;
            meta[1] = pos;
            if (h) atomicOr(&meta[0], h << 1);
            break;
          }
          const int64_t o = (int64_t)old - 1;
          if (key_eq<W>(load_key<W>(P.s_key, P.scap, o), k)) {
            atomicAdd((unsigned long long*)&P.s_amt[o], (unsigned long long)amt);
            if (meta[0] & 1u) atomicOr(reinterpret_cast<uint32_t*>(P.s_meta + o), 1u);
            break;
          }
          h = (h + 1) & mask;
        }
      }
    }
    // representatives listed, one counter update per block
    const unsigned m = __ballot_sync(0xffffffffu, rep);
    if (lane == 0) swarp[wid] = (uint32_t)__popc(m);
    __syncthreads();
    if (wid == 0) {
      const uint32_t v = lane < kMatchThreads / 32 ? swarp[lane] : 0u;
      uint32_t x = v;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
      }
      unsigned long long base = 0;
      if (lane == 31) base = atomicAdd((unsigned long long*)&st->nuniq, (unsigned long long)x);
      base = __shfl_sync(0xffffffffu, base, 31);
      if (lane < kMatchThreads / 32) swarp[lane] = (uint32_t)base + x - v;
    }
    __syncthreads();
    if (rep) P.u_spawn[swarp[wid] + __popc(m & ((1u << lane) - 1u))] = (uint32_t)s;
    __syncthreads();
  }
}
template <int W>
__global__ void __launch_bounds__(kMatchThreads) k_match(Params P, int cur) { d_match<W>(P, cur, VGrid{(int)blockIdx.x, (int)gridDim.x}); }
// the same for a replica of a batch (parameter blocks PP[replica])
template <int W>
__global__ void __launch_bounds__(kMatchThreads) kb_match(const Params* PP, const int* off, int R, int cur) {
  __shared__ Params sP;
  __shared__ VGrid vg;
  if (!batch_block(PP, off, R, sP, vg)) return;
  d_match<W>(sP, cur, vg);
}

// ------------------------------------------------------------------ decide
// survivors in the groups of tile c before group g (g = kGroups: all of them)
__device__ __forceinline__ uint32_t group_new_before(const uint32_t* gnew, int64_t c, int g) {
  uint32_t s = 0;
#pragma unroll
  for (int q = 0; q < kGroups; q += 4) {
    const uint4 v = *reinterpret_cast<const uint4*>(gnew + c * kGroups + q);
    s += (q < g ? v.x : 0u) + (q + 1 < g ? v.y : 0u) + (q + 2 < g ? v.z : 0u) + (q + 3 < g ? v.w : 0u);
  }
  return s;
}

template <int W>
__device__ __forceinline__ void d_decide(const Params& P, int cur, const VGrid vg) {
  __shared__ int64_t sh64[32];
  __shared__ uint32_t scnt[kGroups];
  __shared__ unsigned long long wsum[kGroups];
  __shared__ unsigned long long s_carry;
  __shared__ int s_last;
  DevState* st = P.st;
  const int64_t n = st->ndet[cur], t = st->iter + 1, nu = st->nuniq;
  const int64_t nct = list_tiles(n), want = (nu + 31) / 32;
  const int64_t active = nct > want ? nct : want;   // blocks with work
  if (__syncthreads_or((int)st->error) || vg.b >= active) return;
  const int lane = (int)(threadIdx.x & 31), wid = (int)(threadIdx.x >> 5);
  int64_t* pop = P.pop[cur];
  const uint8_t* fl = P.flags[cur];
  int64_t nws = 0;
  for (int64_t c = vg.b; c < nct; c += vg.n) {
    const int64_t g = c * kGroups + wid;
    unsigned m[2];
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int64_t i = g * kGroup + u * 32 + lane;
      bool keep = false;
      if (i < n) {
        int64_t p = pop[i];
        const bool always = (fl[i] & (F_CORE | F_REF)) != 0;
        if (!always && P.real_amp && p != 0 && iabs64(p) < kOne) {
          // the determinant's occupation draw, stored by the det pass
          const int64_t one = (int64_t)P.occ_draw[i] < iabs64(p) ? kOne : 0;
          p = p < 0 ? -one : one;
          pop[i] = p;
        }
        keep = always || p != 0;
        if (iabs64(p) >= (int64_t(1) << 62)) set_error(st, ERR_OVERFLOW);
        nws += iabs64(p);
      }
      m[u] = __ballot_sync(0xffffffffu, keep);
    }
    if (lane == 0) {
      P.g_keep[g] = (uint64_t)m[0] | ((uint64_t)m[1] << 32);
      scnt[wid] = (uint32_t)(__popc(m[0]) + __popc(m[1]));
    }
    __syncthreads();
    if (threadIdx.x < kGroups) {
      const uint32_t v = scnt[threadIdx.x];
      uint32_t x = v;
#pragma unroll
      for (int o = 1; o < kGroups; o <<= 1) {
        const uint32_t y = __shfl_up_sync((1u << kGroups) - 1u, x, o);
        if ((int)threadIdx.x >= o) x += y;
      }
      P.g_pre[c * kGroups + threadIdx.x] = x - v;
      if (threadIdx.x == kGroups - 1) P.t_keep[c] = x;
    }
    __syncthreads();
  }
  for (int64_t i = (int64_t)vg.b * blockDim.x + threadIdx.x; i < n / kDetTile + 33; i += (int64_t)vg.n * blockDim.x)
    P.det_state[i] = 0ull;   // look-back of the next det pass
  for (int64_t i = chunk_of(vg, wid, true) * 32 + lane; i < nu; i += (int64_t)vg.n * blockDim.x) {
    const int64_t s = P.u_spawn[i];
    const uint64_t meta = P.s_meta[s];
    const uint32_t lo = (uint32_t)meta, pos = (uint32_t)(meta >> 32);
    P.hash_tab[lo >> 1] = 0u;
    int64_t p = P.s_amt[s];
    if ((P.initiator && !(lo & 1u)) || p == 0) p = 0;
    else p = round_small<W>(P, t, load_key<W>(P.s_key, P.scap, s), p);
    uint32_t rank = ~0u;
    if (p != 0) {
      if (iabs64(p) >= (int64_t(1) << 62)) set_error(st, ERR_OVERFLOW);
      nws += iabs64(p);
      P.s_amt[s] = p;
      rank = atomicAdd(&P.g_new[pos / kGroup], 1u);
    }
    P.u_rank[i] = rank;
  }
  const int64_t tot = block_sum<int64_t>(nws, sh64);
  if (threadIdx.x == 0) {
    if (tot) atomicAdd((unsigned long long*)&st->nw_post, (unsigned long long)tot);
  }
  // the last block of the run: exclusive scan of the tiles' entry and survivor
  // counts, new list length
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) {
    s_last = atomicAdd(&st->done_ticket, 1u) == (unsigned)(active < vg.n ? active : vg.n) - 1u;
    s_carry = 0;
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  for (int64_t c0 = 0; c0 < nct; c0 += blockDim.x) {
    const int64_t c = c0 + threadIdx.x;
    unsigned long long v = 0;
    if (c < nct) {
      uint32_t nn = 0;
#pragma unroll
      for (int q = 0; q < kGroups; q += 4) {
        const uint4 x = __ldcg(reinterpret_cast<const uint4*>(P.g_new + c * kGroups + q));
        nn += x.x + x.y + x.z + x.w;
      }
      v = (unsigned long long)__ldcg(&P.t_keep[c]) | ((unsigned long long)nn << 32);
    }
    unsigned long long x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned long long y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    if (lane == 31) wsum[wid] = x;
    __syncthreads();
    const unsigned long long carry = s_carry;
    unsigned long long before = 0;
    for (int w = 0; w < wid; ++w) before += wsum[w];
    if (c < nct) P.t_base[c] = carry + before + x - v;   // {entries kept, survivors} before tile c
    __syncthreads();
    if (threadIdx.x == blockDim.x - 1) s_carry = carry + before + x;
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    const unsigned long long all = s_carry;
    const int64_t nnew = (int64_t)(all >> 32), nd = (int64_t)(all & 0xffffffffull) + nnew;
    st->done_ticket = 0;
    st->nnew = nnew;
    st->ndet[cur ^ 1] = nd;
    if (nd > P.max_det) set_error(st, ERR_STATE_CAPACITY);
  }
}
template <int W>
__global__ void __launch_bounds__(kListThreads, W == 8 ? 2 : 3) k_decide(Params P, int cur) { d_decide<W>(P, cur, VGrid{(int)blockIdx.x, (int)gridDim.x}); }
// the same for a replica of a batch (parameter blocks PP[replica])
template <int W>
__global__ void __launch_bounds__(kListThreads, W == 8 ? 2 : 3) kb_decide(const Params* PP, const int* off, int R, int cur) {
  __shared__ Params sP;
  __shared__ VGrid vg;
  if (!batch_block(PP, off, R, sP, vg)) return;
  d_decide<W>(sP, cur, vg);
}

// ------------------------------------------------------------------ place
// groups with more survivors than this are ranked through sorted runs
__device__ __forceinline__ uint32_t large_group(const Params& P) { return 16u * (uint32_t)P.tile_cap; }

// a key other blocks stored during this kernel
template <int W>
__device__ __forceinline__ Key<W> load_key_l2(const uint64_t* p, int64_t stride, int64_t i) {
  Key<W> k;
#pragma unroll
  for (int j = 0; j < W; ++j) k.w[j] = __ldcg(reinterpret_cast<const unsigned long long*>(p + j * stride + i));
  return k;
}

// The survivors of large groups (a short list whose spawns mostly found new
// keys: the first iterations from one determinant) in runs of kRankChunk, each
// run's order by counting: n_order[run start + rank] = survivor.  One block, which
// reads kRankChunk keys for each survivor of a large group: 5e8 keys for a group
// of 1e6, so a run that starts with very many walkers on one determinant waits
// for it in its first iterations (UEG 30e/66, 2e5 walkers on the reference: 1.3
// ms an iteration over the first four; 3.9 ms with the bucket kernels before).
template <int W>
__device__ void order_large_groups(const Params& P, int64_t nct) {
  const uint32_t lim = large_group(P);
  for (int64_t c = 0; c < nct; ++c) {
    const uint32_t all = group_new_before(P.g_new, c, kGroups);
    if (all <= lim) continue;
    int64_t start = (int64_t)(P.t_base[c] >> 32);
    for (int q = 0; q < kGroups; ++q) {
      const uint32_t kt = P.g_new[c * kGroups + q];
      if (kt > lim) {
        for (int64_t r0 = 0; r0 < kt; r0 += kRankChunk) {
          const int len = (int)(kt - r0 < kRankChunk ? kt - r0 : kRankChunk);
          for (int i = threadIdx.x; i < len; i += blockDim.x) {
            const Key<W> k = load_key_l2<W>(P.b_key, P.scap, start + r0 + i);
            int rank = 0;
            for (int f = 0; f < len; ++f) rank += key_lt<W>(load_key_l2<W>(P.b_key, P.scap, start + r0 + f), k) ? 1 : 0;
            P.n_order[start + r0 + rank] = (uint32_t)(start + r0 + i);
          }
        }
      }
      start += kt;
    }
  }
}

template <int W>
__device__ __forceinline__ void d_place(const Params& P, int cur, const VGrid vg) {
  __shared__ int s_last;
  DevState* st = P.st;
  const int64_t nu = st->nuniq, active = (nu + 31) / 32;
  if (__syncthreads_or((int)st->error) || vg.b >= active) return;
  bool large = false;
  const int lane = (int)warp_lane(), wid = (int)(threadIdx.x >> 5);
  for (int64_t i = chunk_of(vg, wid, true) * 32 + lane; i < nu; i += (int64_t)vg.n * blockDim.x) {
    const uint32_t rank = P.u_rank[i];
    if (rank == ~0u) continue;
    const int64_t s = P.u_spawn[i];
    const uint32_t pos = (uint32_t)(P.s_meta[s] >> 32);
    const int64_t g = pos / kGroup, c = pos / kListTile;
    const int64_t dst = (int64_t)(P.t_base[c] >> 32) + group_new_before(P.g_new, c, (int)(g - c * kGroups)) + rank;
    const Key<W> k = load_key<W>(P.s_key, P.scap, s);
    store_key<W>(P.b_key, P.scap, dst, k);
    P.b_amt[dst] = P.s_amt[s];
    P.n_pos[dst] = pos;
    large = large || rank == large_group(P);   // exactly one survivor of a large group
  }
  if (__syncthreads_or((int)large) && threadIdx.x == 0) atomicAdd(&st->big_ticket, 1u);
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) {
    s_last = atomicAdd(&st->done_ticket, 1u) == (unsigned)(active < vg.n ? active : vg.n) - 1u;
    if (s_last) {
      st->done_ticket = 0;
      s_last = atomicExch(&st->big_ticket, 0u) ? 1 : 0;
    }
  }
  __syncthreads();
  if (!s_last) return;   // also the last block when no group is large
  __threadfence();
  order_large_groups<W>(P, list_tiles(st->ndet[cur]));
}
template <int W>
__global__ void __launch_bounds__(256) k_place(Params P, int cur) { d_place<W>(P, cur, VGrid{(int)blockIdx.x, (int)gridDim.x}); }
// the same for a replica of a batch (parameter blocks PP[replica])
template <int W>
__global__ void __launch_bounds__(256) kb_place(const Params* PP, const int* off, int R, int cur) {
  __shared__ Params sP;
  __shared__ VGrid vg;
  if (!batch_block(PP, off, R, sP, vg)) return;
  d_place<W>(sP, cur, vg);
}

// ------------------------------------------------------------------ write
template <int W, int SYS>
__device__ __forceinline__ void d_write(const Params& P, int cur, const VGrid vg) {
  __shared__ uint32_t hist[kGroups][kGroup];
  __shared__ uint8_t occ[SYS == SYS_HUBBARD ? 1 : kOccMax][kListThreads];
  DevState* st = P.st;
  const int nxt = cur ^ 1;
  const int64_t n = st->ndet[cur], nnew = st->nnew;
  if (__syncthreads_or((int)st->error)) return;
  // the iteration's end: nothing below reads what it changes
  if (vg.b == vg.n - 1 && threadIdx.x == kListThreads - 1) finalize_iteration(P, st->ndet[nxt], st->nw_post);
  const int64_t nct = list_tiles(n);
  const int lane = (int)(threadIdx.x & 31), wid = (int)(threadIdx.x >> 5);
  const uint64_t* key = P.key[cur];
  uint64_t* okey = P.key[nxt];
  // new determinants, one thread each (first: their diagonal elements take longest)
  const uint32_t lim = large_group(P);
  // A warp's FP64 addition takes 64 cycles alone on an SM and 304 among 16: up to
  // one chunk per block, chunks go to all blocks (molecule 1e5 walkers: 24 -> 18
  // us).  Beyond that the first blocks take them while the others copy (molecule
  // 1e7 walkers: 31 us, spread 44).
  const bool spread = nnew <= (int64_t)vg.n * 32;
  for (int64_t i = chunk_of(vg, wid, spread) * 32 + lane; i < nnew; i += (int64_t)vg.n * blockDim.x) {
    const uint32_t pos = P.n_pos[i];
    const Key<W> k = load_key<W>(P.b_key, P.scap, i);
    const int64_t g = pos / kGroup, c = pos / kListTile;
    const uint32_t nb = group_new_before(P.g_new, c, (int)(g - c * kGroups));
    const unsigned long long base = P.t_base[c];
    const int64_t start = (int64_t)(base >> 32) + nb;
    const uint32_t kt = P.g_new[g];
    int64_t rank = 0;
    if (kt <= lim) {
#pragma unroll 4
      for (uint32_t f = 0; f < kt; ++f) rank += key_lt<W>(load_key<W>(P.b_key, P.scap, start + f), k) ? 1 : 0;
    } else {
      for (uint32_t r0 = 0; r0 < kt; r0 += kRankChunk) {
        uint32_t lo = r0, hi = r0 + kRankChunk < kt ? r0 + kRankChunk : kt;
        while (lo < hi) {
          const uint32_t mid = (lo + hi) >> 1;
          if (key_lt<W>(load_key<W>(P.b_key, P.scap, P.n_order[start + mid]), k)) lo = mid + 1;
          else hi = mid;
        }
        rank += lo - r0;
      }
    }
    const int64_t o = (int64_t)(base & 0xffffffffull) + start + P.g_pre[g] +
                      __popcll(P.g_keep[g] & ((1ull << (pos & (kGroup - 1))) - 1ull)) + rank;
    store_key<W>(okey, P.cap, o, k);
    P.pop[nxt][o] = P.b_amt[i];
    P.hdiag[nxt][o] = __dsub_rn(h_diag_listed<W, SYS>(P.sys, k, &occ[0][threadIdx.x], kListThreads), st->e_ref);
    P.flags[nxt][o] = 0;
  }
  // listed entries, one group of 64 per warp
  for (int64_t g = (int64_t)vg.b * kGroups + wid; g < nct * kGroups; g += (int64_t)vg.n * kGroups) {
    const int64_t c = g / kGroups;
    if (g * kGroup >= n) continue;
    const uint64_t keep = P.g_keep[g];
    const uint32_t kt = P.g_new[g];
    const unsigned long long base = P.t_base[c];
    const uint32_t nb = group_new_before(P.g_new, c, (int)(g - c * kGroups));
    int64_t out = (int64_t)(base & 0xffffffffull) + (int64_t)(base >> 32) + nb + P.g_pre[g];
    uint32_t in_front[2] = {0u, 0u};   // survivors at or before the lane's entries
    if (kt) {                          // warp-uniform
      const int64_t start = (int64_t)(base >> 32) + nb;
      hist[wid][lane] = 0u;
      hist[wid][lane + 32] = 0u;
      __syncwarp();
      for (uint32_t f = lane; f < kt; f += 32) atomicAdd(&hist[wid][P.n_pos[start + f] & (kGroup - 1)], 1u);
      __syncwarp();
      uint32_t a = hist[wid][lane], b = hist[wid][lane + 32];
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t x = __shfl_up_sync(0xffffffffu, a, o), y = __shfl_up_sync(0xffffffffu, b, o);
        if (lane >= o) {
          a += x;
          b += y;
        }
      }
      in_front[0] = a;
      in_front[1] = b + __shfl_sync(0xffffffffu, a, 31);
      __syncwarp();
    }
    Key<W> kk[2];
    int64_t pp[2];
    double hh[2];
    uint8_t ff[2];
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int64_t i = g * kGroup + u * 32 + lane;
      if ((keep >> (u * 32 + lane)) & 1ull) {
        kk[u] = load_key<W>(key, P.cap, i);
        pp[u] = P.pop[cur][i];
        hh[u] = P.hdiag[cur][i];
        ff[u] = P.flags[cur][i];
      }
    }
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int b = u * 32 + lane;
      if ((keep >> b) & 1ull) {
        const int64_t o = out + __popcll(keep & ((1ull << b) - 1ull)) + in_front[u];
        store_key<W>(okey, P.cap, o, kk[u]);
        P.pop[nxt][o] = pp[u];
        P.hdiag[nxt][o] = hh[u];
        P.flags[nxt][o] = ff[u] & F_CORE;
        if (ff[u] & F_CORE) P.core_move[g * kGroup + b] = (uint32_t)o;
      }
    }
  }
}
// Eight-word keys take more than 64 registers: held to two blocks per SM the
// kernel spills 72 bytes (an iteration of ueg 14e/97 on 1.6e5 determinants 141
// us, one block 136).
template <int W, int SYS>
__global__ void __launch_bounds__(kListThreads, W == 8 ? 1 : 2) k_write(Params P, int cur) { d_write<W, SYS>(P, cur, VGrid{(int)blockIdx.x, (int)gridDim.x}); }
// the same for a replica of a batch (parameter blocks PP[replica])
template <int W, int SYS>
__global__ void __launch_bounds__(kListThreads, W == 8 ? 1 : 2) kb_write(const Params* PP, const int* off, int R, int cur) {
  __shared__ Params sP;
  __shared__ VGrid vg;
  if (!batch_block(PP, off, R, sP, vg)) return;
  d_write<W, SYS>(sP, cur, vg);
}

}  // namespace hande
