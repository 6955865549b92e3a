// Pauli sum -> CSR and XOR-ELL of a full-space Hamiltonian (Sec. III-E step
// 3), from value tables.
//
// The value of X-mask group g at column c is the group's signed term sum,
// and it depends on c only through the parities of c over the span of the
// group's Z-masks.  The host (plan_build) picks a basis of that span, so the
// value is one entry of a table of 2^rank sums, indexed by a GF(2)-linear
// map of c.  A group of a double excitation has rank 2 to 4; its table has
// at most 64 entries, and which of them are kept (|v| above the drop
// tolerance) is one 64-bit mask, so counting needs no floating point at
// all.  A group of a single excitation has rank N - 1: its terms are cut
// into runs of rank at most 10, one table each, and the value is the sum of
// the runs' entries ("wide" groups, one in 17 at 16 qubits).
//
// What bounds it: integer issue (about 10 instructions per group, row and
// pass) and the writes.  Summing every group's terms per row and pass, as
// the sector builder does, is bound by the float64 pipe (a warp addition
// holds it for 64 cycles): count and fill of the CSR and of the XOR-ELL
// took 5.6 ms each at 16 qubits (complex64), 22.6 ms together; here one
// count of both takes 0.11 ms and the fill of both 0.60 ms.
//
// One warp per block of 8 rows (an XOR-ELL block), lanes over groups: the
// table index of row 8R + i is the index of 8R ^ x xor a three-bit
// combination of the group's low columns, so a lane gets a group's 8 rows
// from one parity evaluation.  Columns of a block fall in aligned column
// blocks R ^ (x >> 3) of 8; their ascending order for block R is the walk of
// the binary trie of the masks x >> 3 with the children swapped at every
// level where R has a 1, so a mask's position is a sum of sibling-subtree
// sizes (a static table) over the set bits of R ^ (x >> 3).  The CSR fill
// places a row's entries by a warp scan over the column blocks in that
// order: no sort.
#include "build_full.h"
#include "dev.cuh"

#include <algorithm>
#include <climits>
#include <cmath>

namespace tq {

// ------------------------------------------------------------------ host plan

namespace {

// Cuts terms [t0, t1) into runs whose Z-masks span at most `cap` dimensions.
// Appends one BuildRun per run and the terms' coordinates in the run's basis.
void cut_runs(const std::vector<uint32_t>& tz, int t0, int t1, int cap, BuildPlan& p) {
    int t = t0;
    while (t < t1) {
        BuildRun r{};
        r.g = -1;
        r.t0 = t;
        uint32_t red[BUILD_MAX_RANK], coord[BUILD_MAX_RANK];   // reduced vectors and their coordinates
        int m = 0;
        for (; t < t1; ++t) {
            uint32_t v = tz[t], c = 0;
            for (int i = 0; i < m; ++i)
                if ((v ^ red[i]) < v) {
                    v ^= red[i];
                    c ^= coord[i];
                }
            if (v) {
                if (m == cap) break;
                r.b[m] = tz[t];
                red[m] = v;
                coord[m] = c | (1u << m);
                c = 1u << m;
                // keep the reduced vectors descending, so one pass reduces
                for (int i = m; i > 0 && red[i] > red[i - 1]; --i) {
                    std::swap(red[i], red[i - 1]);
                    std::swap(coord[i], coord[i - 1]);
                }
                ++m;
            }
            p.comb.push_back(c);
        }
        r.t1 = t;
        r.m = m;
        r.tab = p.n_entries;
        p.n_entries += 1 << m;
        for (int j = 0; j < 3; ++j)
            for (int i = 0; i < m; ++i) r.low[j] |= ((r.b[i] >> j) & 1u) << i;
        p.runs.push_back(r);
    }
}

int rank_of(const std::vector<uint32_t>& tz, int t0, int t1) {
    uint32_t red[32];
    int m = 0;
    for (int t = t0; t < t1; ++t) {
        uint32_t v = tz[t];
        for (int i = 0; i < m; ++i) v = std::min(v, v ^ red[i]);
        if (v) red[m++] = v;
    }
    return m;
}

}  // namespace

BuildPlan plan_build(int nq, const std::vector<uint32_t>& gx, const std::vector<int>& goff,
                     const std::vector<uint32_t>& tz, const std::vector<uint32_t>& dz) {
    BuildPlan p;
    const int G = (int)gx.size();
    p.comb.reserve(tz.size());
    // runs in group order (so term t's coordinates are comb[t])
    for (int g = 0; g < G; ++g) {
        const bool wide = rank_of(tz, goff[g], goff[g + 1]) > BUILD_SMALL_RANK;
        const int first = (int)p.runs.size();
        cut_runs(tz, goff[g], goff[g + 1], wide ? BUILD_MAX_RANK : BUILD_SMALL_RANK, p);
        BuildGroup rec{};
        if (wide) {
            rec.low = BUILD_WIDE;
            rec.b[0] = (uint32_t)p.wx.size();
            p.wx.push_back(gx[g]);
            p.woff.push_back(first);
            p.wend.push_back((int)p.runs.size());
        } else {
            BuildRun& r = p.runs[first];             // rank <= BUILD_SMALL_RANK: one run
            r.g = g;
            for (int i = 0; i < r.m; ++i) rec.b[i] = r.b[i];
            rec.low = r.low[0] | (r.low[1] << 8) | (r.low[2] << 16);
            rec.tab = (uint32_t)r.tab;
        }
        p.rec.push_back(rec);
    }
    // column blocks: runs of groups with equal x >> 3 (gx ascends)
    for (int g = 0; g < G; ++g)
        if (g == 0 || (gx[g] >> 3) != (gx[g - 1] >> 3)) {
            p.hx.push_back(gx[g] >> 3);
            p.hoff.push_back(g);
        }
    p.hoff.push_back(G);
    const int H = (int)p.hx.size();
    p.levels = std::max(0, nq - 3);
    p.sib.assign((size_t)p.levels * H, 0);
    for (int b = 0; b < p.levels; ++b)
        for (int i = 0; i < H;) {
            // masks that agree above bit b form a run; its two halves are siblings
            int j = i, half = i;
            while (j < H && (p.hx[j] >> (b + 1)) == (p.hx[i] >> (b + 1))) {
                if (!((p.hx[j] >> b) & 1)) half = j + 1;
                ++j;
            }
            for (int k = i; k < j; ++k) p.sib[(size_t)b * H + k] = (uint32_t)(k < half ? j - half : half - i);
            i = j;
        }
    // diagonal terms by their low 8 Z bits (the bins of one transform tile)
    std::vector<int> order(dz.size());
    for (size_t i = 0; i < order.size(); ++i) order[i] = (int)i;
    std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return (dz[a] & 255u) < (dz[b] & 255u); });
    p.dorder = order;
    p.dbin.assign(257, 0);
    for (uint32_t z : dz) ++p.dbin[(z & 255u) + 1];
    for (int i = 0; i < 256; ++i) p.dbin[i + 1] += p.dbin[i];
    return p;
}

// -------------------------------------------------------------------- kernels

namespace {

constexpr int BW = 8;                    // warps per CTA of the counting pass
constexpr int BLOCKS_PER_WARP = 1;       // row blocks per warp there (8: too few warps, 279 us at 16 qubits)
constexpr int SEG_BLOCKS = BW * BLOCKS_PER_WARP;
constexpr int FILL_BW = 4;               // warps per CTA of the fills

// One thread per (run, entry): the entry's term sum in term order.  A small
// run is at most 64 entries, so its kept and ambiguous entries are two
// 64-bit masks.
__global__ void k_build_tables(const BuildRun* __restrict__ runs, int n_runs, const uint32_t* __restrict__ comb,
                               const double* __restrict__ tc, double* __restrict__ T, float* __restrict__ Tf,
                               unsigned long long tol, unsigned long long amb, uint2* keep, uint2* amb_mask) {
    const int r = blockIdx.x;
    if (r >= n_runs) return;
    const BuildRun run = runs[r];
    for (int e = threadIdx.x; e < (1 << run.m); e += blockDim.x) {
        double v = 0.0;
        for (int t = run.t0; t < run.t1; ++t) {
            const double c = tc[t];
            v += parity32((uint32_t)e & comb[t]) ? -c : c;
        }
        const unsigned long long a = (unsigned long long)__double_as_longlong(v) & 0x7fffffffffffffffull;
        T[run.tab + e] = v;
        Tf[run.tab + e] = (float)v;
        if (run.g >= 0 && a > tol) {
            atomicOr(e < 32 ? &keep[run.g].x : &keep[run.g].y, 1u << (e & 31));
            if (a <= amb) atomicOr(e < 32 ? &amb_mask[run.g].x : &amb_mask[run.g].y, 1u << (e & 31));
        }
    }
}

// Diagonal: a CTA's 256 consecutive rows share the high bits, so the signed
// terms are binned by their low 8 Z bits (bin order is term order) and one
// 256-point Walsh-Hadamard transform in shared memory gives all 256 sums: 8
// float64 additions per row and the bins, where the term sum takes one
// addition per row and term (137 at 16 qubits; 52 -> 9 us).
__global__ void __launch_bounds__(256)
k_build_diag(long long D, const int* __restrict__ dbin, const uint32_t* __restrict__ dz, const double* __restrict__ dc,
             double* __restrict__ diag) {
    __shared__ double s[256];
    const int t = threadIdx.x;
    for (long long r0 = (long long)blockIdx.x * 256; r0 < D; r0 += (long long)gridDim.x * 256) {
        const uint32_t hi = (uint32_t)r0;      // low 8 bits clear
        double v = 0.0;
        for (int i = dbin[t]; i < dbin[t + 1]; ++i) {
            const double c = dc[i];
            v += parity32(hi & dz[i]) ? -c : c;
        }
        s[t] = v;
        __syncthreads();
#pragma unroll
        for (int o = 1; o < 256; o <<= 1) {
            const double a = s[t & ~o], b = s[t | o];
            __syncthreads();
            s[t] = (t & o) ? a - b : a + b;
            __syncthreads();
        }
        if (r0 + t < D) diag[r0 + t] = s[t];
        __syncthreads();
    }
}

__device__ __forceinline__ uint32_t small_index(const BuildGroup& g, uint32_t c) {
    uint32_t e = 0;
#pragma unroll
    for (int i = 0; i < BUILD_SMALL_RANK; ++i) e |= (uint32_t)(__popc(c & g.b[i]) & 1) << i;
    return e;
}

// The 8 rows' kept bits of a small group: bit i is keep bit e ^ low(i).
__device__ __forceinline__ uint32_t kept_rows(uint2 keep, uint32_t low, uint32_t e) {
    const uint32_t l0 = low & 63u, l1 = (low >> 8) & 63u, l2 = (low >> 16) & 63u;
    uint32_t k = 0;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const uint32_t ei = e ^ ((i & 1) ? l0 : 0u) ^ ((i & 2) ? l1 : 0u) ^ ((i & 4) ? l2 : 0u);
        k |= (((ei < 32 ? keep.x : keep.y) >> (ei & 31)) & 1u) << i;
    }
    return k;
}
__device__ __forceinline__ uint32_t small_entry(uint32_t low, uint32_t e, int i) {
    return e ^ ((i & 1) ? (low & 63u) : 0u) ^ ((i & 2) ? ((low >> 8) & 63u) : 0u) ^
           ((i & 4) ? ((low >> 16) & 63u) : 0u);
}

__device__ __forceinline__ BuildGroup load_group(const BuildGroup* __restrict__ rec, int g) {
    const uint4* q = reinterpret_cast<const uint4*>(rec + g);
    const uint4 a = __ldg(q), b = __ldg(q + 1);
    BuildGroup r;
    r.b[0] = a.x;
    r.b[1] = a.y;
    r.b[2] = a.z;
    r.b[3] = a.w;
    r.b[4] = b.x;
    r.b[5] = b.y;
    r.low = b.z;
    r.tab = b.w;
    return r;
}

// The 8 values of wide group w in row block R, run sums added in run order.
__device__ __forceinline__ void wide_values(const BuildView& v, int w, uint32_t R, double (&a)[8]) {
    const uint32_t c = (R << 3) ^ v.wx[w];
#pragma unroll
    for (int i = 0; i < 8; ++i) a[i] = 0.0;
    for (int r = v.woff[w]; r < v.wend[w]; ++r) {
        const BuildRun* run = v.runs + r;
        const int m = run->m;
        uint32_t e = 0;
        for (int i = 0; i < m; ++i) e |= (uint32_t)(__popc(c & run->b[i]) & 1) << i;
        const uint32_t l0 = run->low[0], l1 = run->low[1], l2 = run->low[2];
        const double* T = v.T + run->tab;
        double x[8];
#pragma unroll
        for (int i = 0; i < 8; ++i)
            x[i] = T[e ^ ((i & 1) ? l0 : 0u) ^ ((i & 2) ? l1 : 0u) ^ ((i & 4) ? l2 : 0u)];
        if (r == v.woff[w]) {
#pragma unroll
            for (int i = 0; i < 8; ++i) a[i] = x[i];
        } else {
#pragma unroll
            for (int i = 0; i < 8; ++i) a[i] += x[i];
        }
    }
}

// |v| as ordered bits (float64 compares hold the float64 pipe; these do not).
__device__ __forceinline__ unsigned long long abs_bits(double v) {
    return (unsigned long long)__double_as_longlong(v) & 0x7fffffffffffffffull;
}

__device__ __forceinline__ uint32_t valid_rows(long long D, long long R) {
    const long long left = D - R * 8;
    return left >= 8 ? 0xffu : (1u << left) - 1u;
}

// Bit i of k into the 16-bit halves of four words (rows 2q, 2q + 1 in word q).
__device__ __forceinline__ void add_rows(uint32_t (&w)[4], uint32_t k) {
    w[0] += (k & 1u) | ((k & 2u) << 15);
    w[1] += ((k >> 2) & 1u) | ((k & 8u) << 13);
    w[2] += ((k >> 4) & 1u) | ((k & 32u) << 11);
    w[3] += ((k >> 6) & 1u) | ((k & 128u) << 9);
}

// Entries per row and pairs per row block, with their sums per segment of
// SEG_BLOCKS row blocks (one CTA).  Row counts stay below 2^16: a row has
// at most G entries, and G is below 2^14 for 26 qubits.
__global__ void __launch_bounds__(BW * 32)
k_build_count(BuildView v, long long D, long long B, unsigned long long tol, unsigned long long amb, int* rowcnt,
              int* blkcnt, uint2* hcls, int* halfcnt, BuildSeg* seg, unsigned long long* n_amb) {
    extern __shared__ unsigned char sk_raw[];
    __shared__ int s_rows[BW], s_pairs[BW], s_half[BW], s_max[BW];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    unsigned char* wkeep = sk_raw + (size_t)wid * 2 * v.W;      // kept and ambiguous rows of the wide groups
    unsigned char* wamb = wkeep + v.W;
    int rows = 0, pairs = 0, half = 0, mx = 0, namb = 0;
    for (int j = 0; j < BLOCKS_PER_WARP; ++j) {
        const long long R = ((long long)blockIdx.x * BW + wid) * BLOCKS_PER_WARP + j;
        if (R >= B) break;                                       // warp-uniform
        const uint32_t vm = valid_rows(D, R);
        for (int w = lane; w < v.W; w += 32) {
            double a[8];
            wide_values(v, w, (uint32_t)R, a);
            uint32_t k = 0, q = 0;
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const unsigned long long ab = abs_bits(a[i]);
                k |= (ab > tol ? 1u : 0u) << i;
                q |= (ab > tol && ab <= amb ? 1u : 0u) << i;
            }
            wkeep[w] = (unsigned char)k;
            wamb[w] = (unsigned char)q;
        }
        __syncwarp();
        uint32_t cnt[4] = {0u, 0u, 0u, 0u};
        uint32_t any[3] = {0u, 0u, 0u};        // pairs, by class of the mask's top bit (two 16-bit counts a word)
        for (int g = lane; g < v.G; g += 32) {
            const BuildGroup r = load_group(v.rec, g);
            uint32_t k, q = 0;
            if (r.low == BUILD_WIDE) {
                k = wkeep[r.b[0]];
                q = wamb[r.b[0]];
            } else {
                const uint32_t e = small_index(r, ((uint32_t)R << 3) ^ v.gx[g]);
                k = kept_rows(v.keep[g], r.low, e);
                const uint2 am = v.amb[g];
                if (am.x | am.y) q = kept_rows(am, r.low, e);
            }
            k &= vm;
            namb += __popc(q & vm);
            if (k) {
                int c = 0;
                if (v.half_bit)
#pragma unroll
                    for (int j = 0; j < HALF_CLASSES; ++j) c += g >= v.cls[j];
                const uint32_t one = 1u << (16 * (c & 1));
                any[0] += c < 2 ? one : 0u;
                any[1] += (c >> 1) == 1 ? one : 0u;
                any[2] += c > 3 ? one : 0u;
            }
            add_rows(cnt, k);
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) cnt[q] = __reduce_add_sync(0xffffffffu, cnt[q]);
#pragma unroll
        for (int q = 0; q < 3; ++q) any[q] = __reduce_add_sync(0xffffffffu, any[q]);
        if (lane < 8 && (vm >> lane) & 1u) {
            const uint32_t word = lane < 2 ? cnt[0] : lane < 4 ? cnt[1] : lane < 6 ? cnt[2] : cnt[3];
            const int n = (int)((word >> (16 * (lane & 1))) & 0xffffu);
            rowcnt[R * 8 + lane] = n;
            mx = max(mx, n);
            rows += n;
        }
        if (lane == 0) {
            static_assert(HALF_CLASSES == 4, "four 16-bit offsets per block");
            const uint32_t o1 = any[0] & 0xffffu, o2 = o1 + (any[0] >> 16), o3 = o2 + (any[1] & 0xffffu),
                           o4 = o3 + (any[1] >> 16), o5 = o4 + any[2];
            blkcnt[R] = (int)o5;
            pairs += (int)o5;
            if (v.half_bit) {
                // the half pass takes a class where the row's bit is 0
                const uint32_t top = (uint32_t)(R >> (v.half_bit - 3));
                const int n = (int)(o1 + ((top & 1u) ? 0u : o2 - o1) + ((top & 2u) ? 0u : o3 - o2) +
                                    ((top & 4u) ? 0u : o4 - o3) + ((top & 8u) ? 0u : o5 - o4));
                hcls[R] = make_uint2(o1 | (o2 << 16), o3 | (o4 << 16));
                // the split's measure: a block's own work is that of about 48 pairs
                halfcnt[R] = n + 48;
                half += n + 48;
            }
        }
        __syncwarp();
    }
    rows = __reduce_add_sync(0xffffffffu, rows);
    mx = __reduce_max_sync(0xffffffffu, mx);
    namb = __reduce_add_sync(0xffffffffu, namb);
    if (lane == 0) {
        s_rows[wid] = rows;
        s_pairs[wid] = pairs;
        s_half[wid] = half;
        s_max[wid] = mx;
        if (namb) atomicAdd(n_amb, (unsigned long long)namb);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        BuildSeg o{0, 0, 0, 0};
        for (int i = 0; i < BW; ++i) {
            o.rows += s_rows[i];
            o.pairs += s_pairs[i];
            o.half += s_half[i];
            o.max_row = max(o.max_row, s_max[i]);
        }
        seg[blockIdx.x] = o;
    }
}

// Exclusive offsets of the segments (one CTA, coalesced rounds of 1024).
__global__ void __launch_bounds__(1024) k_build_scan(const BuildSeg* __restrict__ seg, int n, BuildOffsets* off,
                                                     BuildTotals* out) {
    __shared__ long long sw[3][32];
    __shared__ int sm[32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    long long base[3] = {0, 0, 0};
    int mx = 0;
    for (int i0 = 0; i0 < n; i0 += 1024) {
        const int i = i0 + threadIdx.x;
        const BuildSeg s = i < n ? seg[i] : BuildSeg{0, 0, 0, 0};
        const long long own[3] = {s.rows, s.pairs, s.half};
        long long inc[3] = {own[0], own[1], own[2]};
        mx = max(mx, s.max_row);
#pragma unroll
        for (int o = 1; o < 32; o <<= 1)
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                const long long a = __shfl_up_sync(0xffffffffu, inc[q], o);
                if (lane >= o) inc[q] += a;
            }
        if (lane == 31)
#pragma unroll
            for (int q = 0; q < 3; ++q) sw[q][wid] = inc[q];
        __syncthreads();
        long long at[3];
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            at[q] = base[q] + inc[q] - own[q];
            for (int w = 0; w < 32; ++w) {
                if (w < wid) at[q] += sw[q][w];
                base[q] += sw[q][w];
            }
        }
        if (i < n) off[i] = {at[0], at[1], at[2]};
        __syncthreads();
    }
    mx = __reduce_max_sync(0xffffffffu, mx);
    if (lane == 0) sm[wid] = mx;
    __syncthreads();
    if (threadIdx.x == 0) {
        int m = 0;
        for (int w = 0; w < 32; ++w) m = max(m, sm[w]);
        out->rows = base[0];
        out->pairs = base[1];
        out->half = base[2];
        out->max_row = m;
    }
}

// rowptr and xptr of one segment per CTA from its offsets (nothing when a
// total does not fit int32: the host refuses the build then).
__global__ void __launch_bounds__(SEG_BLOCKS * 8)
k_build_offsets(const int* __restrict__ rowcnt, const int* __restrict__ blkcnt, const int* __restrict__ halfcnt,
                const BuildOffsets* __restrict__ off, const BuildTotals* __restrict__ tot, long long D, long long B,
                int* rowptr, int* xptr, int* hptr) {
    constexpr int NW = SEG_BLOCKS * 8 / 32;
    static_assert(SEG_BLOCKS <= 32, "the pair counts of a segment are scanned by one warp");
    __shared__ int sr[NW];
    if (tot->rows >= INT_MAX || tot->pairs >= INT_MAX) return;
    const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
    const long long r = (long long)blockIdx.x * SEG_BLOCKS * 8 + t, b = (long long)blockIdx.x * SEG_BLOCKS + t;
    const BuildOffsets o = off[blockIdx.x];
    const int c = r < D ? rowcnt[r] : 0;
    const int x = t < SEG_BLOCKS && b < B ? blkcnt[b] : 0;
    const int y = hptr && t < SEG_BLOCKS && b < B ? halfcnt[b] : 0;
    int ci = c, xi = x, yi = y;
#pragma unroll
    for (int k = 1; k < 32; k <<= 1) {
        const int a0 = __shfl_up_sync(0xffffffffu, ci, k), a1 = __shfl_up_sync(0xffffffffu, xi, k),
                  a2 = __shfl_up_sync(0xffffffffu, yi, k);
        if (lane >= k) {
            ci += a0;
            xi += a1;
            yi += a2;
        }
    }
    if (lane == 31) sr[wid] = ci;
    __syncthreads();
    int before = 0;
    for (int w = 0; w < wid; ++w) before += sr[w];
    if (r < D) rowptr[r] = (int)o.rows + before + ci - c;
    if (t < SEG_BLOCKS && b < B) {
        xptr[b] = (int)o.pairs + xi - x;
        if (hptr) hptr[b] = (int)min(o.half + yi - y, 0x7fffffffll);   // balance only: may saturate
    }
    if (blockIdx.x == 0 && t == 0) {
        rowptr[D] = (int)tot->rows;
        xptr[B] = (int)tot->pairs;
        if (hptr) hptr[B] = (int)min(tot->half, 0x7fffffffll);
    }
}

// Wide values of one row block into shared memory, rounded to VT, with their
// kept rows; a dropped value is zero.
template <typename VT>
__device__ __forceinline__ void stage_wide(const BuildView& v, uint32_t R, uint32_t vm, unsigned long long tol,
                                           int lane, VT* wval, unsigned char* wkeep) {
    for (int w = lane; w < v.W; w += 32) {
        double a[8];
        wide_values(v, w, R, a);
        uint32_t k = 0;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const bool keep = abs_bits(a[i]) > tol && ((vm >> i) & 1u);
            k |= (keep ? 1u : 0u) << i;
            wval[8 * w + i] = keep ? (VT)a[i] : VT(0);
        }
        wkeep[w] = (unsigned char)k;
    }
}

template <typename VT> __device__ __forceinline__ const VT* table(const BuildView& v);
template <> __device__ __forceinline__ const double* table<double>(const BuildView& v) { return v.T; }
template <> __device__ __forceinline__ const float* table<float>(const BuildView& v) { return v.Tf; }

template <typename VT> __device__ __forceinline__ void store8(VT* dst, const VT (&a)[8]);
template <> __device__ __forceinline__ void store8<float>(float* dst, const float (&a)[8]) {
    reinterpret_cast<float4*>(dst)[0] = make_float4(a[0], a[1], a[2], a[3]);
    reinterpret_cast<float4*>(dst)[1] = make_float4(a[4], a[5], a[6], a[7]);
}
template <> __device__ __forceinline__ void store8<double>(double* dst, const double (&a)[8]) {
#pragma unroll
    for (int i = 0; i < 4; ++i) reinterpret_cast<double2*>(dst)[i] = make_double2(a[2 * i], a[2 * i + 1]);
}

// XOR-ELL pairs of a block in ascending mask order, compacted by ballot.
template <typename VT>
__global__ void __launch_bounds__(FILL_BW * 32)
k_build_xell(BuildView v, long long D, long long B, unsigned long long tol, const int* __restrict__ xptr,
             uint32_t* __restrict__ xmask, VT* __restrict__ xval) {
    extern __shared__ __align__(16) unsigned char sk_raw[];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    VT* wval = reinterpret_cast<VT*>(sk_raw) + (size_t)wid * 8 * v.W;
    unsigned char* wkeep = sk_raw + (size_t)FILL_BW * 8 * v.W * sizeof(VT) + (size_t)wid * v.W;
    const VT* __restrict__ T = table<VT>(v);
    for (long long R = (long long)blockIdx.x * FILL_BW + wid; R < B; R += (long long)gridDim.x * FILL_BW) {
        const uint32_t vm = valid_rows(D, R);
        stage_wide<VT>(v, (uint32_t)R, vm, tol, lane, wval, wkeep);
        __syncwarp();
        long long base = xptr[R];
        for (int g0 = 0; g0 < v.G; g0 += 32) {
            const int g = g0 + lane;
            uint32_t k = 0, e = 0;
            BuildGroup r{};
            if (g < v.G) {
                r = load_group(v.rec, g);
                if (r.low == BUILD_WIDE) {
                    k = wkeep[r.b[0]];
                } else {
                    e = small_index(r, ((uint32_t)R << 3) ^ v.gx[g]);
                    k = kept_rows(v.keep[g], r.low, e) & vm;
                }
            }
            const unsigned ball = __ballot_sync(0xffffffffu, k != 0);
            if (k) {
                const long long pos = base + __popc(ball & ((1u << lane) - 1u));
                VT a[8];
                if (r.low == BUILD_WIDE) {
#pragma unroll
                    for (int i = 0; i < 8; ++i) a[i] = wval[8 * r.b[0] + i];
                } else {
#pragma unroll
                    for (int i = 0; i < 8; ++i)
                        a[i] = (k >> i) & 1u ? __ldg(T + r.tab + small_entry(r.low, e, i)) : VT(0);
                }
                xmask[pos] = v.gx[g];
                store8<VT>(xval + pos * 8, a);
            }
            base += __popc(ball);
        }
        __syncwarp();
    }
}

// Spreads the 8 bits of k to the 8 nibbles of a word.
__device__ __forceinline__ uint32_t spread8(uint32_t k) {
    uint32_t x = k & 0xffu;
    x = (x | (x << 12)) & 0x000f000fu;
    x = (x | (x << 6)) & 0x03030303u;
    return (x | (x << 3)) & 0x11111111u;
}

// CSR entries of a block, columns ascending per row (see the file comment).
template <typename VT>
__global__ void __launch_bounds__(FILL_BW * 32)
k_build_csr(BuildView v, long long D, long long B, long long nnz, unsigned long long tol,
            const int* __restrict__ rowptr, int* __restrict__ col, VT* __restrict__ val) {
    extern __shared__ __align__(16) unsigned char sk_raw[];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    VT* wval = reinterpret_cast<VT*>(sk_raw) + (size_t)wid * 8 * v.W;
    unsigned short* perm = reinterpret_cast<unsigned short*>(sk_raw + (size_t)FILL_BW * 8 * v.W * sizeof(VT)) +
                           (size_t)wid * v.H;
    unsigned char* wkeep = sk_raw + (size_t)FILL_BW * (8 * v.W * sizeof(VT) + 2 * v.H) + (size_t)wid * v.W;
    const VT* __restrict__ T = table<VT>(v);
    for (long long R = (long long)blockIdx.x * FILL_BW + wid; R < B; R += (long long)gridDim.x * FILL_BW) {
        const uint32_t vm = valid_rows(D, R);
        stage_wide<VT>(v, (uint32_t)R, vm, tol, lane, wval, wkeep);
        // the column blocks in ascending order of R ^ hx
        for (int h = lane; h < v.H; h += 32) {
            const uint32_t c = (uint32_t)R ^ v.hx[h];
            uint32_t pos = 0;
            for (int b = 0; b < v.levels; ++b)
                if ((c >> b) & 1u) pos += v.sib[(size_t)b * v.H + h];
            perm[pos] = (unsigned short)h;
        }
        __syncwarp();
        int base[8];                                 // next position of each row
#pragma unroll
        for (int i = 0; i < 8; ++i) base[i] = (vm >> i) & 1u ? rowptr[R * 8 + i] : 0;
        for (int h0 = 0; h0 < v.H; h0 += 32) {
            int g0 = 0, ng = 0;
            uint32_t cblk = 0;
            if (h0 + lane < v.H) {
                const int h = perm[h0 + lane];
                g0 = v.hoff[h];
                ng = v.hoff[h + 1] - g0;
                cblk = ((uint32_t)R ^ v.hx[h]) << 3;
            }
            // kept rows (a byte), low mask bits and table index per group
            unsigned long long K = 0, E = 0;
            uint32_t xl = 0, own[4] = {0u, 0u, 0u, 0u};
            for (int t = 0; t < ng; ++t) {
                const BuildGroup r = load_group(v.rec, g0 + t);
                const uint32_t x = v.gx[g0 + t];
                uint32_t k;
                if (r.low == BUILD_WIDE) {
                    k = wkeep[r.b[0]];
                } else {
                    const uint32_t e = small_index(r, ((uint32_t)R << 3) ^ x);
                    k = kept_rows(v.keep[g0 + t], r.low, e) & vm;
                    E |= (unsigned long long)e << (6 * t);
                }
                K |= (unsigned long long)k << (8 * t);
                xl |= (x & 7u) << (3 * t);
                add_rows(own, k);
            }
            uint32_t inc[4] = {own[0], own[1], own[2], own[3]};
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const uint32_t a = __shfl_up_sync(0xffffffffu, inc[q], o);
                    if (lane >= o) inc[q] += a;
                }
            }
            for (int t = 0; t < ng; ++t) {
                const uint32_t k = (uint32_t)(K >> (8 * t)) & 0xffu;
                if (!k) continue;
                const uint32_t x3 = (xl >> (3 * t)) & 7u;
                // entries of the other groups of this column block that come
                // first, per row: those whose column i ^ x' is below i ^ x,
                // i.e. the rows where i ^ x has the highest bit of x ^ x'
                uint32_t rank = 0;
                for (int u = 0; u < ng; ++u) {
                    if (u == t) continue;
                    const uint32_t d = x3 ^ ((xl >> (3 * u)) & 7u);
                    const int hb = d & 4u ? 2 : d & 2u ? 1 : 0;
                    uint32_t first = hb == 2 ? 0xf0u : hb == 1 ? 0xccu : 0xaau;
                    if ((x3 >> hb) & 1u) first ^= 0xffu;
                    rank += spread8((uint32_t)(K >> (8 * u)) & first);
                }
                const BuildGroup r = load_group(v.rec, g0 + t);
                const uint32_t e = (uint32_t)(E >> (6 * t)) & 63u;
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    if (!((k >> i) & 1u)) continue;
                    const uint32_t before = ((inc[i >> 1] - own[i >> 1]) >> (16 * (i & 1))) & 0xffffu;
                    const long long pos = (long long)base[i] + before + ((rank >> (4 * i)) & 15u);
                    if (pos >= nnz) continue;
                    col[pos] = (int)(cblk | ((uint32_t)i ^ x3));
                    val[pos] = r.low == BUILD_WIDE ? wval[8 * r.b[0] + i] : __ldg(T + r.tab + small_entry(r.low, e, i));
                }
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const uint32_t tot = __shfl_sync(0xffffffffu, inc[q], 31);
                base[2 * q] += (int)(tot & 0xffffu);
                base[2 * q + 1] += (int)(tot >> 16);
            }
        }
        __syncwarp();
    }
}

int fill_grid(long long B, int sms) {
    const long long g = (B + FILL_BW - 1) / FILL_BW, cap = (long long)sms * 16;
    return (int)(g < cap ? g : cap);
}

}  // namespace

int build_segments(long long B) { return (int)((B + SEG_BLOCKS - 1) / SEG_BLOCKS); }

int launch_build_tables(const BuildView& v, int n_runs, const uint32_t* comb, const double* tc, double* T, float* Tf,
                        unsigned long long tol, unsigned long long amb, uint2* keep, uint2* amb_mask, cudaStream_t s) {
    k_build_tables<<<n_runs, 64, 0, s>>>(v.runs, n_runs, comb, tc, T, Tf, tol, amb, keep, amb_mask);
    return 1;
}

int launch_build_diag(long long D, const int* dbin, const uint32_t* dz, const double* dc, double* diag, int sms,
                      cudaStream_t s) {
    const long long g = (D + 255) / 256, cap = (long long)sms * 8;
    k_build_diag<<<(int)(g < cap ? g : cap), 256, 0, s>>>(D, dbin, dz, dc, diag);
    return 1;
}

int launch_build_count(const BuildView& v, long long D, long long B, unsigned long long tol, unsigned long long amb,
                       int* rowcnt, int* blkcnt, int* halfcnt, BuildSeg* seg, BuildOffsets* off, BuildTotals* tot,
                       int* rowptr, int* xptr, uint2* hcls, int* hptr, cudaStream_t s) {
    const int n = build_segments(B);
    k_build_count<<<n, BW * 32, (size_t)BW * 2 * v.W, s>>>(v, D, B, tol, amb, rowcnt, blkcnt, hcls, halfcnt, seg,
                                                           &tot->amb);
    k_build_scan<<<1, 1024, 0, s>>>(seg, n, off, tot);
    k_build_offsets<<<n, SEG_BLOCKS * 8, 0, s>>>(rowcnt, blkcnt, halfcnt, off, tot, D, B, rowptr, xptr, hptr);
    return 3;
}

int launch_build_fill(const BuildView& v, long long D, long long B, long long nnz, unsigned long long tol, int prec,
                      const int* rowptr, int* col, void* val, const int* xptr, uint32_t* xmask, void* xval, int sms,
                      cudaStream_t s) {
    const int grid = fill_grid(B, sms);
    const size_t vb = prec == TQ_C128 ? 8 : 4;
    const size_t sx = (size_t)FILL_BW * v.W * (8 * vb + 1);
    const size_t sc = (size_t)FILL_BW * (v.W * (8 * vb + 1) + 2 * (size_t)v.H);
    if (prec == TQ_C128) {
        allow_smem(k_build_xell<double>);
        allow_smem(k_build_csr<double>);
        k_build_xell<double><<<grid, FILL_BW * 32, sx, s>>>(v, D, B, tol, xptr, xmask, static_cast<double*>(xval));
        k_build_csr<double><<<grid, FILL_BW * 32, sc, s>>>(v, D, B, nnz, tol, rowptr, col, static_cast<double*>(val));
    } else {
        allow_smem(k_build_xell<float>);
        allow_smem(k_build_csr<float>);
        k_build_xell<float><<<grid, FILL_BW * 32, sx, s>>>(v, D, B, tol, xptr, xmask, static_cast<float*>(xval));
        k_build_csr<float><<<grid, FILL_BW * 32, sc, s>>>(v, D, B, nnz, tol, rowptr, col, static_cast<float*>(val));
    }
    return 2;
}

}  // namespace tq
