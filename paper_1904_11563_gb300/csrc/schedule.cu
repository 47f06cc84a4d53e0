// a1: symbolic peel.  One CTA turns an erasure mask into the peel plan:
// the surviving cells and, round by round, the sources that a surviving
// cell with exactly one unknown source resolves (Section I-A decoder read as
// parallel rounds).  Resolver = lowest such cell id; depth = the round; the
// recovered sources are then listed in (depth, source) order.
//
// Each cell keeps one word: its count of unknown sources in the low bits,
// the sum of those sources' ids + 1 above (modulo the word).  A round walks
// only the sources recovered in the round before (one warp per source, lanes
// over its cells): each lane takes the source out of the cell's word with one
// atomic subtraction, and the lane that brings a count to one finds the one
// source the cell still lacks in what is left of the sum.  That source may
// have been recovered in the same round and still be on its way out; every
// source recovered in a round already carries its depth when the round's
// subtractions start, so the claim test (depth 0, or depth = next round when
// another cell got there first) is exact, and the claims for round r + 1
// happen inside round r: one barrier per round.
//
// What bounds it is the chain of one round (Construction A at full size: 685
// rounds of ~24 sources).  Where a code's graph is a projection grid -- every
// source in one cell of each column, at an affine function of its grid
// position, checked cell by cell when the code is made -- the cells are
// computed, not loaded.  A small code's graph is copied to shared memory
// first.  The cells' initial words are made with the code, the rounds'
// sources are put in ascending order after the last one, a warp per round,
// and a tall code's peel list is filled by a second launch over all SMs.  The
// ready lists live in a ring in shared memory (and in the plan, which serves
// rounds wider than half the ring).  The plan also carries a flat "peel list"
// (per recovered source: its resolver and the blocks to subtract) for the
// numeric peel.
//
// Whole plans, against one thread per position for the lists, tables for the
// cells and two atomics a cell: Construction A n = 32, b = 683 (685 rounds)
// 1307 -> 544 us, of which the rounds are 450 (1330 cycles each: a source
// list read, one atomic on the cell, a claim's look, swap and list slot, the
// barrier); n = 12, b = 120 153 -> 77; n = 8, b = 300 258 -> 177; n = 16,
// b = 2800 with its state in global memory 7050 -> 4280.  Taking four sources
// a warp at once made the rounds slower (550 -> 760 us: their claims queue),
// and so did swapping without a look first (630).  Codes of few, wide rounds
// (n = 27, b = 12: one of 252 sources) 16.6 -> 14.6, n = 32, b = 24 28.9 ->
// 22.9; with rounds of up to 256 ordered by one warp, an element at a time,
// and a warp copying each position's list, these took 49 and 40.  (Four a lane,
// up to 128 sources, cost every plan of many rounds 1 %: registers.)
#include <algorithm>
#include <climits>
#include <mutex>

#include "device_common.cuh"

namespace bpx {
namespace {

constexpr int kThreads = 1024;
constexpr size_t kSmemMax = 224 * 1024;  // dynamic shared memory of a plan's CTA (state + ready lists)
constexpr size_t kSmemSmall = 16 * 1024;  // the same for the 256-thread CTA of small codes

constexpr int kAffineMax = 64;   // columns of the affine table kept in shared memory
constexpr int kRankMax = 96;     // sources of a round ordered by one warp, three a lane, comparing each with all

// The per-cell word: 32 bits in shared memory (when count and sum fit), 64
// bits in the plan otherwise.
template <bool kSmem>
struct CellWord {
  using T = uint32_t;
};
template <>
struct CellWord<false> {
  using T = unsigned long long;
};

// Ints of dynamic shared memory a plan takes with its whole graph in it, and
// whether it is worth copying there: always for a small one, else only where
// the rounds would read the cells from tables (32 columns of a 24 x 9 grid,
// computed cells, two rounds: the copy of its 27000 words costs 10 us).
__host__ __device__ inline long long sched_local_ints(const DevGraph& g) {
  return 2LL * g.num_cells + 5LL * g.S + 2LL * g.num_edges + 2;
}
__host__ __device__ inline bool sched_local(const DevGraph& g, long long smem_ints) {
  const long long ints = sched_local_ints(g);
  return ints <= smem_ints && (ints <= 8192 || !g.affine);
}

// One position of the peel list: its resolver's sources but s, ascending.
__device__ __forceinline__ void fill_position(const int32_t* support, int degree, int s, int32_t* list, int first,
                                              int step) {
  for (int e = first; e < degree; e += 8 * step) {
    int t[8];  // eight loads in flight (the stores could alias them)
#pragma unroll
    for (int u = 0; u < 8; ++u) t[u] = e + u * step < degree ? support[e + u * step] : s;
#pragma unroll
    for (int u = 0; u < 8; ++u)
      if (t[u] != s) list[e + u * step - (t[u] > s ? 1 : 0)] = t[u];  // ascending: those past s move up by one
  }
}

// kSmem: the per-cell words and per-source depths (the state every round
// reads and updates) live in shared memory, followed by the ready ring (and,
// when the launch's smem_ints allow, the graph, the resolvers and the order);
// otherwise in the plan's global arrays.
// cell_mask: the mask has one byte per cell (a processor whose output is
// missing) instead of one per column (a node).
// part: 0 = the whole plan; 1 = what the products need (surviving cells,
// their count and the depth-1 direct map, from the first round alone);
// 2 = the rest of the plan after a part-1 launch, leaving the arrays part 1
// wrote untouched (so that it may run while the products read them).
// fill: write the peel list here (else fill_list_kernel follows).
template <bool kSmem>
__device__ __forceinline__ void schedule_body(const DevGraph& g, const DevPlan& p,
                                              const uint8_t* __restrict__ mask, int32_t* peel_order,
                                              uint8_t* recovered, int32_t* info_out, bool cell_mask, int part,
                                              int smem_ints, bool fill) {
  using W = typename CellWord<kSmem>::T;
  extern __shared__ int32_t dyn_smem[];
  __shared__ int s_warp[32];
  __shared__ int s_cnt[3];  // sources of a round, round r at r % 3
  __shared__ int s_aff[3 * kAffineMax];
  const int tid = threadIdx.x, nt = blockDim.x;
  const int lane = tid & 31, warp = tid >> 5, nwarps = nt >> 5;
  const int C = g.num_cells, S = g.S;
  // count field: low cbits bits, its top bit set only in an erased cell's word
  const int cbits = kSmem ? sched_count_bits(g.sigma) : 32;
  const W cmask = (W(1) << cbits) - 1, gone = W(1) << (cbits - 1);
  W* word = kSmem ? reinterpret_cast<W*>(dyn_smem) : reinterpret_cast<W*>(p.word);
  int32_t* depth = kSmem ? dyn_smem + C : p.depth;
  const bool local = kSmem && sched_local(g, smem_ints);
  // the recovered sources in the order of their claims: all of them in the
  // plan's scratch, and in a ring (a power of two) the rounds of at most half of it
  int32_t* ring = dyn_smem + C + S;
  // (with the graph in shared memory the whole order fits there)
  int32_t* claimed = local ? ring : p.front0;
  const int ring_len = !kSmem || local ? 0 : max(0, smem_ints - C - S);
  const int half = ring_len >= 4 ? (1 << (31 - __clz(ring_len))) / 2 : 0, rmask = 2 * half - 1;
  const int32_t *cell_ptr = g.cell_ptr, *cell_src = g.cell_src, *src_ptr = g.src_ptr, *src_cell = g.src_cell;
  int32_t *res = p.resolver, *ord = p.order;
  if (local) {
    int32_t* at = ring + S;
    auto bring = [&](const int32_t* src, int n) {
      for (int i = tid; i < n; i += nt) {
        const uint32_t to = static_cast<uint32_t>(__cvta_generic_to_shared(at + i));
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(to), "l"(src + i) : "memory");
      }
      const int32_t* r = at;
      at += n;
      return r;
    };
    cell_ptr = bring(g.cell_ptr, C + 1);
    cell_src = bring(g.cell_src, g.num_edges);
    src_ptr = bring(g.src_ptr, S + 1);
    src_cell = bring(g.src_cell, g.num_edges);
    res = at;
    ord = at + S;
  }
  const bool affine = kSmem && !local && g.affine && g.n <= kAffineMax;
  if (affine)
    for (int i = tid; i < 3 * g.n; i += nt) s_aff[i] = p.affine[i];
  // cell c, with w its one unknown source, claims w for round r, whose
  // sources start at `first` of the claim order
  auto claim = [&](int c, int w, int r, int first) {
    if (kSmem) {
      // a look first: up to a column's worth of cells claim one source, and
      // their swaps would queue on its word
      const int had = *reinterpret_cast<volatile int32_t*>(&depth[w]);
      if (had != 0 && had != r) return;  // recovered in an earlier round
    }
    if (local) atomicMin(&res[w], c);
    else if (kSmem) atomicMin(&p.resolver[w], c);
    const int had = atomicCAS(&depth[w], 0, r);
    if (!kSmem && (had == 0 || had == r)) atomicMin(&p.resolver[w], c);
    if (had == 0) {
      const int i = atomicAdd(&s_cnt[r % 3], 1);
      claimed[first + i] = w;
      if (i < half) ring[(first + i) & rmask] = w;
    }
  };
  // [first, last) of this warp's run of 32-wide steps over n items
  auto run_of = [&](int n, int& first, int& last) {
    const int seg = ((n + 31) / 32 + nwarps - 1) / nwarps * 32;
    first = min(n, warp * seg);
    last = min(n, first + seg);
  };
  // the sum of s_warp below this warp, and of all (after a barrier)
  auto warp_base = [&](int* total) {
    int x = lane < nwarps ? s_warp[lane] : 0;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    *total = __shfl_sync(0xffffffffu, x, nwarps - 1);
    const int below = __shfl_sync(0xffffffffu, x, warp > 0 ? warp - 1 : 0);
    return warp > 0 ? below : 0;
  };

  int c0, c1, alive_here = 0;
  run_of(C, c0, c1);
#pragma unroll 4
  for (int b = c0; b < c1; b += 32) {
    const int c = b + lane;
    bool alive = false;
    if (c < c1) {
      alive = (cell_mask ? mask[c] : mask[g.col_of_cell[c]]) == 0;
      W v;
      if (kSmem) {
        v = static_cast<W>(reinterpret_cast<const uint32_t*>(p.word)[c]);
      } else {
        const int e0 = g.cell_ptr[c], e1 = g.cell_ptr[c + 1];
        W x = 0;
        for (int e = e0; e < e1; ++e) x += static_cast<W>(g.cell_src[e] + 1);
        v = (x << cbits) | static_cast<W>(e1 - e0);
      }
      word[c] = alive ? v : v | gone;
      p.cnt[c] = alive ? static_cast<int>(v & cmask) : -1;  // the sign (erased) is read by the two-dimensional GEMM
      if (part != 2) p.direct[c] = -1;
    }
    alive_here += __popc(__ballot_sync(0xffffffffu, alive));
  }
  for (int s = tid; s < S; s += nt) {
    depth[s] = 0;
    res[s] = INT_MAX;
  }
  if (tid == 0) {
    s_cnt[0] = s_cnt[1] = s_cnt[2] = 0;
    p.wave_ptr[0] = 0;
  }
  if (lane == 0) s_warp[warp] = alive_here;
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();

  // Surviving cells in ascending id; the degree-one ones claim their source
  // for round 1.
  int nsurv;
  int at_cell = warp_base(&nsurv);
  for (int b = c0; b < c1; b += 32) {
    const int c = b + lane;
    const W v = c < c1 ? word[c] : gone;
    const bool alive = (v & gone) == 0;
    const unsigned m = __ballot_sync(0xffffffffu, alive);
    if (alive) {
      if (part != 2) p.surv[at_cell + __popc(m & ((1u << lane) - 1u))] = c;
      const int w = static_cast<int>(v >> cbits) - 1;
      if ((v & cmask) == 1 && static_cast<unsigned>(w) < static_cast<unsigned>(S)) claim(c, w, 1, 0);
    }
    at_cell += __popc(m);
  }
  __syncthreads();

  // lanes that share one source's cells: the power of two at or above a
  // source's mean number of cells
  int lanes = 1;
  while (lanes < 32 && static_cast<long long>(lanes) * S < g.num_edges) lanes <<= 1;
  const int j0 = tid / lanes, jl = tid & (lanes - 1);
  // s / k by one multiplication (exact: S k < 2^32 whenever the state fits shared memory)
  const uint32_t kmul = g.k > 1 ? static_cast<uint32_t>((0x100000000ull + g.k - 1) / g.k) : 0u;
  const int max_rounds = part == 1 ? 1 : INT_MAX;
  int round = 1, nrec = 0;
  int direct1 = 0;  // sources of the first round
  for (;;) {
    const int nr = s_cnt[round % 3];
    if (nr == 0) {
      --round;
      break;
    }
    const int wave0 = nrec;
    nrec += nr;
    if (round == 1) direct1 = nr;
    if (tid == 0) {
      p.wave_ptr[round] = nrec;
      s_cnt[(round + 2) % 3] = 0;  // round - 1's length: every thread read it before the last barrier
    }
    if (round >= max_rounds) break;
    auto source = [&](int j) -> int {
      if (nr <= half) return ring[(wave0 + j) & rmask];
      return claimed[wave0 + j];
    };
    auto check = [&](int c, W left) {  // (an erased cell's count stays above 1)
      const int w = static_cast<int>(left >> cbits) - 1;
      if ((left & cmask) == 1 && static_cast<unsigned>(w) < static_cast<unsigned>(S)) claim(c, w, round + 1, nrec);
    };
    for (int j = j0; j < nr; j += nt / lanes) {
      const int s = source(j);
      const W out = W(0) - ((static_cast<W>(s + 1) << cbits) | 1);
      if (affine) {
        const int z = kmul ? static_cast<int>(__umulhi(s, kmul)) : s, l = s - z * g.k;
        for (int col = jl; col < g.n; col += lanes) {
          const int c = s_aff[col] + s_aff[g.n + col] * z + s_aff[2 * g.n + col] * l;
          check(c, atomicAdd(&word[c], out) + out);
        }
      } else {
        const int e1 = src_ptr[s + 1];
        for (int e = src_ptr[s] + jl; e < e1; e += lanes) {
          const int c = src_cell[e];
          check(c, atomicAdd(&word[c], out) + out);
        }
      }
    }
    if (nr > kRankMax) {  // a wide round: its members in ascending id, by two passes over the depths
      int s0, s1, mine = 0;
      run_of(S, s0, s1);
      const volatile int32_t* dep = depth;
      for (int b = s0; b < s1; b += 32)
        mine += __popc(__ballot_sync(0xffffffffu, b + lane < s1 && dep[min(b + lane, S - 1)] == round));
      if (lane == 0) s_warp[warp] = mine;
      __syncthreads();
      int total;
      int at = wave0 + warp_base(&total);
      for (int b = s0; b < s1; b += 32) {
        const bool in = b + lane < s1 && dep[min(b + lane, S - 1)] == round;
        const unsigned m = __ballot_sync(0xffffffffu, in);
        if (in) ord[at + __popc(m & ((1u << lane) - 1u))] = b + lane;
        at += __popc(m);
      }
    }
    __syncthreads();
    ++round;
  }

  if (part == 1) {
    // what the products need: the depth-1 direct map and the survivor count
    __syncthreads();
    for (int s = tid; s < S; s += nt)
      if (depth[s] == 1) p.direct[res[s]] = s;
    if (tid == 0) {
      p.ctr[CTR_NSURV] = nsurv;
      p.ctr[CTR_PLAN] = 0;  // the rest of the plan follows (part 2)
      p.info[BPX_INFO_DEVICE_ERR] = 0;  // cleared before the products run
    }
    return;
  }

  // Ascending order within the narrow rounds: each warp takes a run of
  // rounds, the next one's sources loaded while one is ordered.
  {
    int d0, d1;
    const int seg = (round + nwarps - 1) / nwarps;
    d0 = min(round, warp * seg);
    d1 = min(round, d0 + seg);
    for (int b = d0; b < d1; b += 31) {  // bounds of up to 31 rounds, one a lane
      const int bound = b + lane <= d1 ? p.wave_ptr[b + lane] : 0;
      const int rounds = min(31, d1 - b);
      int w0 = __shfl_sync(0xffffffffu, bound, 0), w1 = __shfl_sync(0xffffffffu, bound, 1);
      int x = w0 + lane < w1 ? claimed[w0 + lane] : INT_MAX;
      for (int q = 0; q < rounds; ++q) {
        const int w2 = __shfl_sync(0xffffffffu, bound, min(q + 2, 31)), n = w1 - w0;
        const int nx = q + 1 < rounds && w1 + lane < w2 ? claimed[w1 + lane] : INT_MAX;
        if (n <= 32) {
          int below = 0;
          for (int t = 0; t < n; ++t) below += __shfl_sync(0xffffffffu, x, t) < x ? 1 : 0;
          if (lane < n) ord[w0 + below] = x;
        } else if (n <= kRankMax) {
          int v[kRankMax / 32], below[kRankMax / 32];
#pragma unroll
          for (int u = 0; u < kRankMax / 32; ++u) {
            v[u] = 32 * u + lane < n ? claimed[w0 + 32 * u + lane] : INT_MAX;
            below[u] = 0;
          }
#pragma unroll
          for (int j = 0; j < kRankMax / 32; ++j) {
            if (32 * j >= n) break;
#pragma unroll 8
            for (int t = 0; t < 32; ++t) {
              const int y = __shfl_sync(0xffffffffu, v[j], t);
#pragma unroll
              for (int u = 0; u < kRankMax / 32; ++u) below[u] += y < v[u] ? 1 : 0;
            }
          }
#pragma unroll
          for (int u = 0; u < kRankMax / 32; ++u)
            if (32 * u + lane < n) ord[w0 + below[u]] = v[u];
        }
        w0 = w1;
        w1 = w2;
        x = nx;
      }
    }
  }
  for (int s = tid; s < S; s += nt) {
    const int d = depth[s];
    if (d == 1 && part != 2) p.direct[res[s]] = s;
    if (recovered) recovered[s] = d > 0 ? 1 : 0;
  }
  __syncthreads();
  // Peel list: for order position i, the resolver and the other sources of
  // its support (ascending), so the numeric peel reads flat descriptors.
  // Each warp takes a run of positions: their lists' starts within the run,
  // then the runs' totals, then the entries.
  int i0, i1, list_len;
  run_of(nrec, i0, i1);
  if (nrec <= nt && fill) {  // a position a thread: no pass over the plan in between
    const int i = i0 + lane;
    const bool in = i < i1;
    const int s = in ? ord[i] : 0, r = in ? res[s] : 0;
    const int e0 = in ? cell_ptr[r] : 0, deg = in ? cell_ptr[r + 1] - e0 : 1;
    int x = deg - 1;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    if (lane == 31) s_warp[warp] = x;
    __syncthreads();
    const int at = warp_base(&list_len) + x - (deg - 1);
    if (in) {
      p.order[i] = s;
      p.pl_res[i] = r;
      p.pl_ptr[i] = at;
      if (S >= kTallSources) p.pos[s] = i;
      fill_position(cell_src + e0, deg, s, p.pl_list + at, 0, 1);
    }
  } else {
    int run = 0;
    for (int b = i0; b < i1; b += 128) {  // four steps at a time: their loads in flight together
      int s[4], r[4], len[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) s[u] = b + 32 * u + lane < i1 ? ord[b + 32 * u + lane] : -1;
#pragma unroll
      for (int u = 0; u < 4; ++u) r[u] = s[u] >= 0 ? res[s[u]] : 0;
#pragma unroll
      for (int u = 0; u < 4; ++u) len[u] = s[u] >= 0 ? cell_ptr[r[u] + 1] - cell_ptr[r[u]] - 1 : 0;
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int i = b + 32 * u + lane;
        int x = len[u];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const int y = __shfl_up_sync(0xffffffffu, x, o);
          if (lane >= o) x += y;
        }
        if (i < i1) {
          p.pl_res[i] = r[u];
          p.pl_ptr[i] = run + x - len[u];
          if (local) p.order[i] = s[u];
        }
        run += __shfl_sync(0xffffffffu, x, 31);
      }
    }
    if (lane == 0) s_warp[warp] = run;
    __syncthreads();
    const int list0 = warp_base(&list_len);
    for (int i = i0 + lane; i < i1; i += 32) {
      const int at = list0 + p.pl_ptr[i];
      p.pl_ptr[i] = at;
      if (!fill) continue;
      const int r = p.pl_res[i], x = ord[i], e0 = cell_ptr[r];
      if (S >= kTallSources) p.pos[x] = i;
      fill_position(cell_src + e0, cell_ptr[r + 1] - e0, x, p.pl_list + at, 0, 1);
    }
  }
  if (tid == 0) p.pl_ptr[nrec] = list_len;
  if (peel_order) {
    for (int i = tid; i < S; i += nt) {
      const int s = i < nrec ? ord[i] : -1;
      peel_order[3 * i + 0] = s;
      peel_order[3 * i + 1] = s >= 0 ? res[s] : -1;
      peel_order[3 * i + 2] = s >= 0 ? depth[s] : -1;
    }
  }
  if (tid == 0) {
    p.ctr[CTR_NSURV] = nsurv;
    p.ctr[CTR_NWAVES] = round;
    p.ctr[CTR_NREC] = nrec;
    p.ctr[CTR_PLAN] = kPlanReady;
    int32_t inf[BPX_INFO_LEN];
    for (int i = 0; i < BPX_INFO_LEN; ++i) inf[i] = 0;
    // part 2 runs beside the products: keep a self-check error they raised
    const int32_t dev_err = part == 2 ? atomicAdd(&p.info[BPX_INFO_DEVICE_ERR], 0) : 0;
    inf[BPX_INFO_STATUS] = dev_err ? dev_err : ((nrec == S) ? BPX_OK : BPX_ERR_UNDECODABLE);
    inf[BPX_INFO_DEVICE_ERR] = dev_err;
    inf[BPX_INFO_RECOVERED] = nrec;
    inf[BPX_INFO_WAVES] = round;
    inf[BPX_INFO_SURVIVING] = nsurv;
    inf[BPX_INFO_DIRECT] = direct1;
    for (int i = 0; i < BPX_INFO_LEN; ++i) {
      if (i == BPX_INFO_DEVICE_ERR || i == BPX_INFO_STATUS) {
        if (dev_err) continue;  // left as the products' atomic writes set them
      }
      p.info[i] = inf[i];
      if (info_out) info_out[i] = inf[i];
    }
  }
}

// The peel list of a tall plan: a warp per position, all SMs.
__global__ void __launch_bounds__(256) fill_list_kernel(DevGraph g, DevPlan p) {
  chain_wait();
  const int n = p.ctr[CTR_NREC], step = gridDim.x * 8;
  for (int i = blockIdx.x * 8 + (threadIdx.x >> 5); i < n; i += step) {
    const int r = p.pl_res[i], e0 = g.cell_ptr[r];
    const int s = p.order[i];
    if ((threadIdx.x & 31) == 0) p.pos[s] = i;
    fill_position(g.cell_src + e0, g.cell_ptr[r + 1] - e0, s, p.pl_list + p.pl_ptr[i], threadIdx.x & 31, 32);
  }
}

template <bool kSmem>
__global__ void __launch_bounds__(kThreads, 1)
schedule_kernel(DevGraph g, DevPlan p, const uint8_t* __restrict__ mask, int32_t* peel_order,
                uint8_t* recovered, int32_t* info_out, bool cell_mask, int part, int smem_ints, bool fill,
                bool clear_f32) {
  chain_wait();
  if (threadIdx.x == 0) {
    if (clear_f32) {  // the staging let in here may raise these words: they are down before
      for (int i = 0; i < kF32Words; ++i) p.ctr[CTR_F32_SIMT + i] = 0;
      __threadfence();
    }
    chain_release();
  }
  schedule_body<kSmem>(g, p, mask, peel_order, recovered, info_out, cell_mask, part, smem_ints, fill);
}

// Grouped launch: CTA j plans job j; smem_ints: the launch's dynamic shared
// memory in int32 words (each job's ready lists take what its state leaves).
template <bool kSmem>
__global__ void __launch_bounds__(kThreads, 1) schedule_group_kernel(const GJob* __restrict__ jobs, int smem_ints) {
  const GJob& J = jobs[blockIdx.x];
  schedule_body<kSmem>(J.g, J.p, J.mask, nullptr, nullptr, J.info_out, false, 0, smem_ints, true);
}

}  // namespace

cudaError_t launch_schedule_group(const GJob* d_jobs, int njobs, size_t max_state_bytes, size_t max_want_bytes,
                                  bool packable, cudaStream_t st) {
  if (njobs <= 0) return cudaSuccess;
  if (packable && max_state_bytes <= kSmemMax) {
    const size_t smem = std::min(kSmemMax, std::max(max_state_bytes, max_want_bytes));
    cudaError_t e = cudaFuncSetAttribute(schedule_group_kernel<true>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(kSmemMax));
    if (e != cudaSuccess) return e;
    schedule_group_kernel<true><<<njobs, kThreads, smem, st>>>(d_jobs, static_cast<int>(smem / 4));
  } else {
    schedule_group_kernel<false><<<njobs, kThreads, 0, st>>>(d_jobs, 0);
  }
  return cudaGetLastError();
}

cudaError_t launch_schedule(const DevGraph& g, const DevPlan& p, const uint8_t* mask,
                            int32_t* peel_order, uint8_t* recovered, int32_t* info_out,
                            cudaStream_t st, bool cell_mask, int part, bool clear_f32) {
  const long long state = static_cast<long long>(g.num_cells) + g.S;  // int32 words
  // Small codes take a 256-thread block with at most 16 KB of shared memory:
  // it fits beside a resident GEMM CTA, so the schedule of one
  // multiplication can run while the GEMM of another still holds every SM.
  const bool small = state <= 4096;
  const int threads = small ? 256 : kThreads;
  const long long room = static_cast<long long>((small ? kSmemSmall : kSmemMax) / 4);
  const bool fill_later = g.S >= kTallSources && part != 1;
  cudaError_t e;
  if (sched_packable32(g.S, g.sigma) && state <= room) {
    const long long ints = sched_local(g, room) ? sched_local_ints(g) : std::min(room, state + 2LL * g.S);
    if ((e = cudaFuncSetAttribute(schedule_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  static_cast<int>(kSmemMax))) != cudaSuccess)
      return e;
    e = launch(schedule_kernel<true>, dim3(1), threads, static_cast<size_t>(ints) * 4, st, g, p, mask, peel_order,
               recovered, info_out, cell_mask, part, static_cast<int>(ints), !fill_later, clear_f32);
  } else {
    e = launch(schedule_kernel<false>, dim3(1), threads, 0, st, g, p, mask, peel_order, recovered, info_out, cell_mask,
               part, 0, !fill_later, clear_f32);
  }
  if (e != cudaSuccess || !fill_later) return e;
  return launch(fill_list_kernel, dim3(std::min((g.S + 7) / 8, 4 * num_sms())), 256, 0, st, g, p);
}

}  // namespace bpx

// ---------------------------------------------------------------------------
// Allocation-free entry point.
//
// Some callers cannot allocate device memory themselves: code that runs inside
// a host runtime which owns the whole device pool (a raw cudaMalloc would
// bypass its accounting or fail against its cap), or latency-critical callers
// that cannot afford the device-wide synchronisation cudaMalloc / cudaFree
// imply.  For them bpx_schedule_noalloc runs the same schedule kernel with its
// scratch (graph copy + peel plan) in the fixed array below instead of a
// caller workspace.  Every GPU that loads this library keeps the array until
// the process exits.
namespace bpx {
namespace {

constexpr size_t kNoAllocBytes = size_t(8) << 20;  // 8 MiB
static __device__ __align__(256) int32_t g_noalloc_scratch[kNoAllocBytes / sizeof(int32_t)];

constexpr int kMaxDevices = 64;
std::mutex g_noalloc_mu;
void* g_noalloc_ptr[kMaxDevices] = {};

}  // namespace

}  // namespace bpx

extern "C" int bpx_schedule_noalloc(const bpx_code* c, const uint8_t* d_mask, int32_t* d_peel_order,
                                    uint8_t* d_recovered, int32_t* d_info, bpx_stream stream) {
  using bpx::fail;
  bpx::clear_error();
  if (!c) return fail(BPX_ERR_INVAL, "bpx_schedule_noalloc: code is NULL");
  if (!d_mask) return fail(BPX_ERR_INVAL, "bpx_schedule_noalloc: erasure mask is NULL");
  const bpx::WsLayout L = bpx::ws_layout(c, 0, 0, 0, 1, BPX_FP32);
  if (L.total > bpx::kNoAllocBytes)
    return fail(BPX_ERR_INVAL,
                "bpx_schedule_noalloc: this code needs %zu bytes of scratch, more than the fixed "
                "%zu-byte array; use bpx_schedule with a workspace",
                L.total, bpx::kNoAllocBytes);
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return fail(BPX_ERR_CUDA, "bpx_schedule_noalloc: %s", cudaGetErrorString(e));
  if (dev < 0 || dev >= bpx::kMaxDevices) return fail(BPX_ERR_UNSUPPORTED, "device id %d too large", dev);
  void* base = nullptr;
  {
    // First call on a device: look up the array's device address with that
    // device current (the array's name is only a host-side stand-in).
    std::lock_guard<std::mutex> lk(bpx::g_noalloc_mu);
    if (!bpx::g_noalloc_ptr[dev]) {
      void* p = nullptr;
      e = cudaGetSymbolAddress(&p, bpx::g_noalloc_scratch);
      if (e != cudaSuccess)
        return fail(BPX_ERR_CUDA, "bpx_schedule_noalloc: cudaGetSymbolAddress: %s", cudaGetErrorString(e));
      bpx::g_noalloc_ptr[dev] = p;
    }
    base = bpx::g_noalloc_ptr[dev];
  }
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  char* b = static_cast<char*>(base);
  struct Part {
    size_t off;
    const void* src;
    size_t bytes;
  } parts[] = {
      {L.g_col_of_cell, c->col_of_cell.data(), c->col_of_cell.size() * 4},
      {L.g_cell_ptr, c->cell_ptr.data(), c->cell_ptr.size() * 4},
      {L.g_cell_src, c->cell_src.data(), c->cell_src.size() * 4},
      {L.g_src_ptr, c->src_ptr.data(), c->src_ptr.size() * 4},
      {L.g_src_cell, c->src_cell.data(), c->src_cell.size() * 4},
      {L.p_word, c->word0.data(), c->word0.size() * 4},
      {L.p_cursor, c->affine.data(), c->affine.size() * 4},
  };
  // The graph of this call's code replaces whatever the previous call left;
  // the kernel initialises every plan array it reads.
  for (const Part& pt : parts) {
    if (pt.bytes == 0) continue;
    e = cudaMemcpyAsync(b + pt.off, pt.src, pt.bytes, cudaMemcpyHostToDevice, st);
    if (e != cudaSuccess) return fail(BPX_ERR_CUDA, "bpx_schedule_noalloc: copy: %s", cudaGetErrorString(e));
  }
  const bpx::DevGraph g = bpx::make_graph(c, base, L);
  const bpx::DevPlan p = bpx::make_plan(base, L);
  e = bpx::launch_schedule(g, p, d_mask, d_peel_order, d_recovered, d_info, st);
  if (e != cudaSuccess) return fail(BPX_ERR_CUDA, "bpx_schedule_noalloc: launch: %s", cudaGetErrorString(e));
  return BPX_OK;
}

