// The whole Chebyshev recursion (Eq. E-2-6 / E-2-7) of small sectors in one launch.
//
// The random vectors are independent, so a block keeps one vector of one
// sector in shared memory as 64-bit fixed point (kpm_fixed.cuh) and makes all
// K/2 products by itself: no launches, queues or grid-wide sums between the steps, one
// block barrier per step.  Thread t owns states t, t + blockDim, ...; v_{n+1}
// overwrites v_{n-1}, which only its owner reads.  What a step reads from global memory is
// the structure of H': per state the bond counts, the diagonal and the indices
// of the flipped states (entry-major, so that a warp reads consecutive words; they
// come from L1 and L2, shared by all blocks of the sector).
//
// The whole 2^N space is the direct sum of its S^z sectors: its vector has the
// signs of the sectors' vectors, so its moments are the sectors' sums, weighted
// by M and M^2 for the weighted ones, and its sectors are what the blocks work on.
#include <algorithm>
#include <cmath>
#include <vector>

#include "kpm_device.cuh"
#include "kpm_fixed.cuh"
#include "kpm_run.h"

namespace kpm {

namespace {

// Per state: `head` (anti-aligned bonds of each group, 8 bits each; their number
// when every bond has its own coefficient), `diag`, and the entries: pairs of
// 16-bit indices, group by group, padded with the index of a zero (grouped), or
// index and bond number.  Entry k of state u of the sector at row0 is
// ent[row0 * n_ent + k * dim + u].
struct SmallLists {
  uint32_t *head;
  FxCoef *diag;
  uint32_t *ent;
  uint64_t *code;  // bitstrings
  int n_ent;
};

struct SmallArgs {
  TablesDev tb;
  SmallLists l;
  const FxCoef *coef;   // [n_sectors][n_coef]: 2/a J_g/2 per group, or per bond
  int n_coef;
  const int *block_sector, *block_column;  // largest sectors first
  i128 *part;           // [sector][R][S][2], in units of 2^kFxSumShift
  int S, R, n_groups;
  int64_t unit;
  uint64_t seed, r0;
  unsigned lim_hi;
  int *flag;
};

struct SmallListArgs {
  TablesDev tb;
  SmallLists l;
  const int64_t *coef;  // [n_sectors][n_coef] J/a, and
  const int64_t *c0;    // [n_sectors] the diagonal without anti-aligned bonds, in units of 2^-59
  int n_coef;
  int *flag;
};

template <bool GROUPED>
__global__ void __launch_bounds__(kThreads)
    small_lists_kernel(const __grid_constant__ SmallListArgs a, const __grid_constant__ BondsDev bd) {
  bool out_of_range = false;
  for (int t = blockIdx.x; t < a.tb.n_tiles; t += gridDim.x) {
    const Tile tile = a.tb.tiles[t];
    const SectorDev sd = a.tb.sectors[tile.sector];
    const int64_t *coef = a.coef + (size_t)tile.sector * a.n_coef;
    const int64_t c0 = a.c0[tile.sector];
    uint32_t hb = tile.b_first;
    for (uint32_t i = threadIdx.x; i < tile.count; i += kThreads) {
      const int64_t row = tile.row0 + i;
      const uint32_t u = (uint32_t)(row - sd.row0);
      const uint64_t s = sd.n_up < 0 ? (uint64_t)u
                                     : sector_unrank(tile.rank0 + i, sd.n_up, tile.b_last, hb, a.tb);
      uint32_t *E = a.l.ent + (size_t)sd.row0 * a.l.n_ent + u;
      int64_t d = c0, sum = 0;
      uint32_t head = 0, pair = 0;
      size_t e = 0;
      const int ng = GROUPED ? bd.n_groups : 1;
      for (int g = 0; g < ng; ++g) {
        const int k0 = GROUPED ? bd.gstart[g] : 0, k1 = GROUPED ? bd.gstart[g + 1] : bd.n_bonds;
        uint32_t cnt = 0;
        for (int k = k0; k < k1; ++k) {
          const int b = GROUPED ? bd.order[k] : k;
          const uint64_t m = bd.mask[b];
          const uint64_t tt = s & m;
          if (tt == 0 || tt == m) continue;
          const uint64_t f = s ^ m;
          const uint32_t rk = sd.n_up < 0 ? (uint32_t)f : sector_rank(f, a.tb);
          const int64_t c = __ldg(coef + (GROUPED ? g : k));
          d -= c;
          sum += llabs(c) >> 8;
          if (!GROUPED) {
            E[(e++) * sd.dim] = rk | ((uint32_t)b << 16);
          } else if (cnt & 1) {
            E[(e++) * sd.dim] = pair | (rk << 16);
          } else {
            pair = rk;
          }
          ++cnt;
        }
        if (GROUPED && (cnt & 1)) E[(e++) * sd.dim] = pair | ((uint32_t)sd.dim << 16);
        head |= cnt << (8 * g);
      }
      // (where the sum is in range, d cannot have overflowed)
      out_of_range |= sum + (llabs(d) >> 8) > kFxRowUnits || llabs(d) > kFxCoefUnits;
      a.l.head[row] = head;
      a.l.code[row] = s;
      a.l.diag[row] = fx_limbs_of(d);
    }
  }
  if (out_of_range) atomicOr(a.flag, kFlagRange);
}

// Sums of NV values over the warp: lane l ends with the sum of value
// (l >> (5 - log2 NV)), halving the values that a lane carries with the distance.
template <int NV>
__device__ __forceinline__ i128 warp_sums(i128 (&v)[NV]) {
  const int lane = threadIdx.x & 31;
  auto exchange = [](i128 x, int o) {
    const unsigned long long lo = __shfl_xor_sync(0xffffffffu, (unsigned long long)x, o);
    const long long hi = __shfl_xor_sync(0xffffffffu, (long long)(x >> 64), o);
    return ((i128)hi << 64) + (i128)lo;
  };
  int o = 16;
#pragma unroll
  for (int h = NV / 2; h > 0; h /= 2, o /= 2) {
    const bool up = (lane & o) != 0;
#pragma unroll
    for (int i = 0; i < h; ++i) {
      const i128 send = up ? v[i] : v[i + h], keep = up ? v[i + h] : v[i];
      v[i] = keep + exchange(send, o);
    }
  }
  for (; o > 0; o /= 2) v[0] += exchange(v[0], o);
  return v[0];
}

// 64-bit element `index` of the array at a shared-memory address.
__device__ __forceinline__ unsigned smem_address(const void *p) {
  return (unsigned)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ long long load_shared(unsigned base, unsigned index) {
  long long v;
  asm volatile("ld.shared.s64 %0, [%1];" : "=l"(v) : "r"(base + 8 * index) : "memory");
  return v;
}
__device__ __forceinline__ void store_shared(unsigned base, unsigned index, long long v) {
  asm volatile("st.shared.s64 [%0], %1;" ::"r"(base + 8 * index), "l"(v) : "memory");
}

constexpr int kSmallThreads = 1024;

// What bounds it: the gathers from shared memory (8-byte words of random banks, 3
// to 6 passes each) and the latency of a step when a sector has few states.  Two
// states per thread at a time, 256 threads, or a launch per size of sector were slower
// (ladder N = 14, M >= 0, R = 25: 0.87, 2.0 and 1.18 ms for 100 products, this form
// 0.73 ms, the list kernels 1.02 ms).  Ring N = 10, whole space, R = 20: 1.0 us per
// product (list kernel 9.9 us, in FP64 25 us); ladder N = 16, R = 100: 57 us per product
// with every vector's sums (list kernel and column sums 100 us).
// Shared memory of a block: two vectors with a zero at the end, and two sets of
// the warps' sums.
constexpr size_t small_smem(int64_t dim) {
  return (size_t)(dim + 1) * 2 * sizeof(long long) + 2 * 2 * 32 * sizeof(i128) + 16;
}

template <bool GROUPED>
__global__ void __launch_bounds__(kSmallThreads, 1) small_run_kernel(const __grid_constant__ SmallArgs a) {
  extern __shared__ __align__(16) unsigned char s_raw[];
  __shared__ FxCoef s_coef[kMaxBonds];
  const int T = blockDim.x, nw = T / 32, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  i128 *slots = reinterpret_cast<i128 *>(s_raw);  // [2][2][32]
  long long *x = reinterpret_cast<long long *>(s_raw + (size_t)2 * 2 * 32 * sizeof(i128));
  const int sec = a.block_sector[blockIdx.x], col = a.block_column[blockIdx.x];
  const SectorDev sd = a.tb.sectors[sec];
  const int D = (int)sd.dim;
  long long *z = x + D + 1;
  for (int i = threadIdx.x; i < a.n_coef; i += T) s_coef[i] = a.coef[(size_t)sec * a.n_coef + i];
  for (int i = threadIdx.x; i < 2 * 2 * 32; i += T) slots[i] = 0;
  const uint32_t *head = a.l.head + sd.row0;
  const FxCoef *diag = a.l.diag + sd.row0;
  const uint32_t *ent = a.l.ent + (size_t)sd.row0 * a.l.n_ent;
  {
    // v_0 = +-U
    const uint64_t h = splitmix64(splitmix64(a.seed) ^ (a.r0 + (uint64_t)col));
    for (int u = threadIdx.x; u < D; u += T) {
      x[u] = (splitmix64(h ^ a.l.code[sd.row0 + u]) >> 63) ? -a.unit : a.unit;
      z[u] = 0;
    }
    if (threadIdx.x == 0) x[D] = z[D] = 0;
  }
  __syncthreads();
  unsigned top = 0;
  const int flag = threadIdx.x == 0 ? __ldcg(a.flag) & kFlagRange : 0;
  i128 *out = a.part + ((size_t)sec * a.R + col) * a.S * 2;
  for (int n = 0; n < a.S; ++n) {
    FxDot xx, yx;
    const unsigned xs = smem_address(x), zs = smem_address(z);
    for (int u = threadIdx.x; u < D; u += T) {
      int hd = (int)__ldg(head + u);
      const FxCoef dc = diag[u];
      const uint32_t *E = ent + u;
      FxSum s;
      if (GROUPED) {
        for (int g = 0; g < a.n_groups; ++g, hd >>= 8) {
          long long gs = 0;
          int left = hd & 255;
          for (; left > 2; left -= 4, E += 2 * D) {
            const uint32_t p = __ldg(E), q = __ldg(E + D);
            gs += (load_shared(xs, p & 0xffffu) + load_shared(xs, p >> 16)) +
                  (load_shared(xs, q & 0xffffu) + load_shared(xs, q >> 16));
          }
          if (left > 0) {
            const uint32_t p = __ldg(E);
            E += D;
            gs += load_shared(xs, p & 0xffffu) + load_shared(xs, p >> 16);
          }
          s.add(s_coef[g], fx_split(gs));
        }
      } else {
        for (; hd > 0; hd -= 4) {
          uint32_t p[4];
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            p[q] = q < hd ? __ldg(E) : (uint32_t)D;
            E += q < hd ? D : 0;
          }
#pragma unroll
          for (int q = 0; q < 4; ++q) s.add(s_coef[p[q] >> 16], fx_split(load_shared(xs, p[q] & 0xffffu)));
          // the low limbs' sum holds 8 products: carry
          s.mid += s.ll >> kFxBits;
          s.ll &= (1ll << kFxBits) - 1;
        }
      }
      const FxLimbs xl = fx_split(load_shared(xs, u));
      s.add(dc, xl);
      const long long y = n == 0 ? s.half_value() : s.value() - load_shared(zs, u);
      top = max(top, (unsigned)((unsigned long long)y >> 32) + a.lim_hi);
      store_shared(zs, u, y);
      xx.square(xl);
      yx.product(xl, fx_split(y));
    }
    i128 *slot = slots + (n & 1) * 2 * 32;
    if (warp * 32 < D) {  // the slots of warps without states stay zero
      i128 acc[2] = {xx.square_value(), yx.product_value()};
      const i128 v = warp_sums<2>(acc);
      if ((lane & 15) == 0) slot[(lane >> 4) * 32 + warp] = v;
    }
    // a vector that left the range ends (the run's results are not used): looked at every 16
    // steps, and after the first one whether the coefficients had left it
    if ((n & 15) == 0) {
      if (__syncthreads_or(top >= 2 * a.lim_hi || (n == 0 && flag != 0))) break;
    } else {
      __syncthreads();
    }
    // one warp (another at every step) adds the warps' sums while the others go on;
    // this slot is written again only after the next barrier
    if (warp == n % nw) {
      i128 w[2] = {slot[lane], slot[32 + lane]};
      const i128 r = warp_sums<2>(w);
      if ((lane & 15) == 0) out[(size_t)n * 2 + (lane >> 4)] = fx_sum_units(r);
    }
    long long *swap = x;
    x = z;
    z = swap;
  }
  if (__any_sync(0xffffffffu, top >= 2 * a.lim_hi) && lane == 0) atomicOr(a.flag, kFlagRange);
}

// sums[step][sector][q] over the vectors (and, for the whole space, over its
// sectors), and (sums_r) every vector's: of step 0 the dot products, of step n > 0
// already the moments' 2 <v_n|v_n> - <v_0|v_0> and 2 <v_{n+1}|v_n> - <v_1|v_0>, which FP64
// would round to 2^-54 of terms near 1 where the difference is some 1/sqrt(D).  Sector i
// of the run is made of the blocks' sectors first[i] .. first[i + 1] - 1.  The sums are exact
// integers, rounded once: a vector's is below 2^16 states times 2^108 (U <= 2^54, norm 1) in
// units of 2^20, and doubled, with 512 vectors and (2M)^2 <= 2^8, below 2^123.
// A warp takes one step of one sector, its lanes the vectors.
constexpr int kSumsThreads = 128;
template <int NQ>
__global__ void __launch_bounds__(kSumsThreads)
    small_sums_kernel(const i128 *part, const int *first, const SectorDev *sub, int n_sites, double *sums,
                      double *sums_r, int S, int ns, int R) {
  const int lane = threadIdx.x & 31;
  for (int i = (blockIdx.x * kSumsThreads + threadIdx.x) / 32; i < S * ns; i += gridDim.x * kSumsThreads / 32) {
    const int n = i % S, sec = i / S;
    const int k0 = first[sec], k1 = first[sec + 1];
    const double scale = sub[k0].fx_scale * (1 << kFxSumShift);
    i128 acc[NQ];
#pragma unroll
    for (int q = 0; q < NQ; ++q) acc[q] = 0;
    for (int r = lane; r < R; r += 32) {
      i128 v[2] = {0, 0};
      for (int k = k0; k < k1; ++k) {
        const i128 *mine = part + ((size_t)k * R + r) * S * 2;
        const int m = NQ == 6 ? 2 * sub[k].n_up - n_sites : 0;
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          const i128 p = n == 0 ? mine[q] : 2 * mine[2 * n + q] - mine[q];
          v[q] += p;
          if (NQ == 6) {
            acc[(2 + q) % NQ] += p * m;
            acc[(4 + q) % NQ] += p * (m * m);
          }
        }
      }
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        acc[q] += v[q];
        if (sums_r != nullptr)
          sums_r[(((size_t)n * ns + sec) * R + r) * 2 + q] = i128_to_double(v[q]) * scale;
      }
    }
    double *o = sums + ((size_t)n * ns + sec) * NQ;
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
      const i128 w = warp_sum_i128(acc[q]);
      if (lane == 0) o[q] = i128_to_double(w) * scale * (q < 2 ? 1.0 : q < 4 ? 0.5 : 0.25);
    }
  }
}

int small_entries(const BondsDev &b) {
  if (b.n_groups == 0) return b.n_bonds;
  int n = 0;
  for (int g = 0; g < b.n_groups; ++g) n += (b.gstart[g + 1] - b.gstart[g] + 1) / 2;
  return std::max(1, n);
}

// n_up of the blocks' sectors: the run's, with N + 1 for the whole space.
std::vector<int32_t> sub_sectors(const Plan &p, std::vector<int> *first) {
  std::vector<int32_t> out;
  for (int i = 0; i < p.n_sectors; ++i) {
    if (first) first->push_back((int)out.size());
    if (p.n_up[i] >= 0)
      out.push_back(p.n_up[i]);
    else
      for (int k = 0; k <= p.N; ++k) out.push_back(k);
  }
  if (first) first->push_back((int)out.size());
  return out;
}

}  // namespace

bool small_applies(const kpm_model *m, int n_sectors, const int32_t *n_up) {
  if (m->n_bonds == 0 || m->n_bonds > 255) return false;  // bond counts of 8 bits
  for (int i = 0; i < n_sectors; ++i) {
    const int64_t d = n_up[i] < 0 ? binom(m->n_sites, m->n_sites / 2) : binom(m->n_sites, n_up[i]);
    if (d > kSmallMaxDim) return false;
  }
  return true;
}

// Whether one launch is the faster form of a prepared run.  A product of one vector takes a
// block 0.14 ns (bonds with their own couplings: 0.21 ns) per state and for each of its
// neighbours + 3, and one block has it to itself: the largest sector sets the step, or
// all of them when they fill the chip.  The kernels that spread a step over the chip take 10 us
// at least (whole space, with its weighted sums: 22 us; FP64 vectors: 14 us with lists, 20 us
// without), and 1.1e-6 us
// (1.3e-6; FP64 vectors 3e-5) per state, neighbour + 3 and vector.  Measured for K = 200,
// S^z = 0 sector, one launch against the others in ms: 3432 states (ladder, R = 1 / 24 / 100) 0.83
// against 1.6 / 1.0 / 1.3; 6435 states (J1-J2 chain, R = 1 / 4 / 8 / 100) 1.8 against 2.0 / 1.4 /
// 1.0 / 1.9; 12870 states (J1-J2 chain, R = 1 / 8 / 64 / 100) 3.4 against 2.0 / 1.2 / 1.8 / 3.1,
// (random couplings, R = 8) 5.5 against 1.4; whole space of 16 sites (ring, R = 8 / 100) 2.1 / 7.0
// against 2.6 / 9.2.  Over 195 such runs the choice is 0.4% slower than the better one in
// the mean, 12% at most.
bool small_pays(const kpm_model *m, const MomentsRun &r) {
  double largest = 0.0, total = 0.0;
  for (int32_t k : sub_sectors(r.plan, nullptr)) {
    const double N = m->n_sites, flips = N > 1 ? m->n_bonds * 2.0 * k * (N - k) / (N * (N - 1)) : 0.0;
    const double work = (double)binom(m->n_sites, k) * (flips + 3.0);
    largest = std::max(largest, work);
    total += work;
  }
  const int R = r.lay.R;
  const double one = (r.bonds.n_groups > 0 ? 1.4e-4 : 2.1e-4) * std::max(largest, total * R / kSms);
  const bool full = r.plan.any_full;
  double stepped = r.fixed || r.weighted ? std::max(full ? 22.0 : 10.0, (full ? 1.3e-6 : 1.1e-6) * total * R)
                                         : std::max(r.list_stride > 0 ? 14.0 : 20.0, 3e-5 * total * r.lay.Rp);
  // every vector's moments: another pass over the vectors, which one launch does not need
  if (r.per_vector) stepped *= 1.6;
  return one <= stepped;
}

int prepare_small(const kpm_model *m, MomentsRun *r) {
  if (!r->plan.any_full) return KPM_OK;  // the run's own sectors
  const std::vector<int32_t> sub = sub_sectors(r->plan, nullptr);
  // tiles only deal out the states when the lists are built
  return build_plan(m, (int)sub.size(), sub.data(), kThreads, &r->small_run.plan);
}

namespace {
const Plan &blocks_plan(const MomentsRun &r) { return r.plan.any_full ? r.small_run.plan : r.plan; }
}  // namespace

size_t small_bytes(const MomentsRun &r) {
  const Plan &p = blocks_plan(r);
  const size_t ns = p.n_sectors, rows = p.total_rows, R = r.lay.R;
  return tables_bytes(r.plan) + (r.plan.any_full ? tables_bytes(p) : 0) + align256((size_t)r.S * r.plan.n_sectors * r.NQ * 8) +
         align256((size_t)2 * r.S * 4) + 256 +
         (r.per_vector ? align256((size_t)r.S * r.plan.n_sectors * R * 16) : 0) + align256(rows * 4) +
         align256(rows * sizeof(FxCoef)) + align256(rows * 8) + align256(rows * small_entries(r.bonds) * 4) +
         2 * align256(ns * std::max(kMaxGroups, r.bonds.n_bonds) * sizeof(FxCoef)) + align256(ns * 8) +
         align256((r.plan.n_sectors + 1) * 4) + 2 * align256(ns * R * 4) + align256(ns * R * r.S * 2 * sizeof(i128));
}

int setup_small(MomentsRun &r, const std::vector<SectorDev> &sec, Arena &arena, cudaStream_t s) {
  SmallRun &m = r.small_run;
  const Plan &p = blocks_plan(r);
  const size_t ns = p.n_sectors, rows = p.total_rows, R = r.lay.R;
  const BondsDev &bd = r.bonds;
  std::vector<int> first;
  sub_sectors(r.plan, &first);
  std::vector<SectorDev> sub(ns);
  for (int i = 0; i < r.plan.n_sectors; ++i)
    for (int k = first[i]; k < first[i + 1]; ++k) {
      sub[k] = sec[i];  // a, b and the norm of the run's sector
      sub[k].row0 = p.row0[k];
      sub[k].dim = p.dim[k];
      sub[k].n_up = p.n_up[k];
      sub[k].hb_begin = p.hb_begin[k];
      sub[k].Mval = p.n_up[k] - 0.5 * p.N;
    }
  if (r.plan.any_full)
    KPM_TRY(upload_tables(p, sub, arena, s, &m.tb));
  else
    m.tb = r.tb;
  m.n_ent = small_entries(bd);
  m.n_coef = bd.n_groups > 0 ? bd.n_groups : bd.n_bonds;
  m.head = arena.take<uint32_t>(rows);
  m.diag = arena.take<FxCoef>(rows);
  m.ent = arena.take<uint32_t>(rows * m.n_ent);
  m.code = arena.take<uint64_t>(rows);
  m.part = arena.take<i128>(ns * R * r.S * 2);
  if (r.per_vector) r.sums_r = arena.take<double>((size_t)r.S * r.plan.n_sectors * R * 2);
  KPM_REQUIRE(m.head && m.diag && m.ent && m.code && m.part &&
                  (!r.per_vector || r.sums_r), KPM_ENOMEM, "workspace too small for the small-sector run");
  // couplings of 2H/a, those of the run's sector
  std::vector<FxCoef> c(ns * m.n_coef);
  std::vector<int64_t> units(ns * m.n_coef), c0(ns);
  for (int i = 0; i < r.plan.n_sectors; ++i)
    for (int j = first[i]; j < first[i + 1]; ++j) {
      c0[j] = r.fx_c0[i];
      for (int k = 0; k < m.n_coef; ++k) {
        const int64_t v = r.fx_couplings[(size_t)i * m.n_coef + k];
        units[(size_t)j * m.n_coef + k] = v;
        c[(size_t)j * m.n_coef + k] = fx_limbs_of(v);
      }
    }
  // largest sectors first
  std::vector<int> order(ns), hb, hc;
  for (size_t i = 0; i < ns; ++i) order[i] = (int)i;
  std::stable_sort(order.begin(), order.end(), [&](int q, int w) { return p.dim[q] > p.dim[w]; });
  m.block_dim.clear();
  for (int i : order)
    for (size_t k = 0; k < R; ++k) {
      hb.push_back(i);
      hc.push_back((int)k);
      m.block_dim.push_back((int)p.dim[i]);
    }
  PackedUpload up(arena, s);
  SmallListArgs la;
  KPM_TRY(up.add(c, &m.coef));
  KPM_TRY(up.add(units, &la.coef));
  KPM_TRY(up.add(c0, &la.c0));
  KPM_TRY(up.add(hb, &m.block_sector));
  KPM_TRY(up.add(hc, &m.block_column));
  KPM_TRY(up.add(first, &m.first));
  KPM_TRY(up.send());
  la.tb = m.tb;
  la.n_coef = m.n_coef;
  la.l = SmallLists{m.head, m.diag, m.ent, m.code, m.n_ent};
  la.flag = r.flag;
  const int grid = (int)std::min<int64_t>((int64_t)p.tiles.size(), (int64_t)8 * sm_count());
  if (bd.n_groups > 0)
    small_lists_kernel<true><<<grid, kThreads, 0, s>>>(la, bd);
  else
    small_lists_kernel<false><<<grid, kThreads, 0, s>>>(la, bd);
  KPM_CUDA(cudaGetLastError());
  count_launches(1);
  return KPM_OK;
}

int launch_small(const MomentsRun &r, uint64_t seed, uint64_t r0, cudaStream_t s) {
  const SmallRun &m = r.small_run;
  SmallArgs a;
  a.tb = m.tb;
  a.l = SmallLists{m.head, m.diag, m.ent, m.code, m.n_ent};
  a.coef = m.coef;
  a.n_coef = m.n_coef;
  a.part = m.part;
  a.S = r.S;
  a.R = r.lay.R;
  a.n_groups = r.bonds.n_groups;
  a.unit = r.fx_unit;
  a.seed = seed;
  a.r0 = r0;
  a.lim_hi = (unsigned)((kFxRange * r.fx_unit) >> 32);
  a.flag = r.flag;
  void *fn = r.bonds.n_groups > 0 ? reinterpret_cast<void *>(&small_run_kernel<true>)
                                  : reinterpret_cast<void *>(&small_run_kernel<false>);
  KPM_CUDA(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)small_smem(kSmallMaxDim)));
  // The registers of an SM hold 1024 of these threads: all for one block when its
  // vectors leave no room for another, or when every large block has an SM to
  // itself; otherwise 512, and two blocks share.
  const int n_blocks = (int)m.block_dim.size(), D = m.block_dim[0];
  int large = 0;
  while (large < n_blocks && m.block_dim[large] > kSmallThreads / 2) ++large;
  const bool alone = small_smem(D) > ((size_t)113 << 10) || large <= sm_count();
  const int most = alone ? kSmallThreads : kSmallThreads / 2;
  const int threads = std::min(most, (D + 31) / 32 * 32);
  a.block_sector = m.block_sector;
  a.block_column = m.block_column;
  void *args[] = {(void *)&a};
  const bool prof = r.profile && profiling();
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  if (prof) {
    KPM_CUDA(cudaEventCreate(&e0));
    KPM_CUDA(cudaEventCreate(&e1));
    KPM_CUDA(cudaEventRecord(e0, s));
  }
  KPM_CUDA(cudaLaunchKernel(fn, dim3(n_blocks), dim3(threads), args, small_smem(D), s));
  if (prof) {
    KPM_CUDA(cudaEventRecord(e1, s));
    profile_push(e0, e1);
  }
  count_launches(1);
  const int ns = r.plan.n_sectors, per_block = kSumsThreads / 32;
  const int grid = std::min(4096, (r.S * ns + per_block - 1) / per_block);
  double *sums_r = r.per_vector ? r.sums_r : nullptr;
  if (r.NQ == 6)
    small_sums_kernel<6><<<grid, kSumsThreads, 0, s>>>(m.part, m.first, m.tb.sectors, r.plan.N, r.sums,
                                                       sums_r, r.S, ns, r.lay.R);
  else
    small_sums_kernel<2><<<grid, kSumsThreads, 0, s>>>(m.part, m.first, m.tb.sectors, r.plan.N, r.sums,
                                                       sums_r, r.S, ns, r.lay.R);
  KPM_CUDA(cudaGetLastError());
  count_launches(1);
  return KPM_OK;
}

}  // namespace kpm
