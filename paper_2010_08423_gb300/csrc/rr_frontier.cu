// rr_frontier.cu -- the frontier engine: a query's sums over the rows that
// matter to it, without sieve points.
//
// Rows that matter. P_l[e] can be non-zero only when a walk of l edges from the
// source ends with e, and it reaches an output only when a walk goes on from e
// to the query's last layer. Both sets are found first, per layer, as bitmaps
// over the row lists: forward, a row is active at layer l when its window holds
// a row active at l - 1 (x_plan); backward, an active row is needed when a
// needed row of the next layer has it in its window. The layers then run over
// the needed rows alone, stored densely in list order (x_wedge).
//
// Wedge form. Summed over all sieve points L, a walk contributes the permanent
// of its vertices' z rows, which in characteristic 2 is their determinant.
//  * Columns are eliminated with the source's row: with pivot label p
//    (z_{s,p} != 0) and rho_j = z_{s,j} / z_{s,p}, z'_{u,j} = z_{u,j} + z_{u,p}
//    rho_j leaves the determinant unchanged and makes z'_s zero outside p, so it
//    is z_{s,p} times the determinant of the other vertices' z' over the
//    K = k - 1 other labels.
//  * That determinant is the wedge product of the z' rows, so layer l keeps per
//    row the values on the (l-1)-subsets of the K labels instead of one per
//    sieve point: R_l[e]_T = y_{e,l} sum_{j in T} z'_{u,j} W_{T\j}, u the tail
//    of e, W = the sum of R_{l-1} over e's window (layer 1: y_{e,1} z_{s,p});
//    the last layer ends with witness[w] += sum_j z'_{w,j} (sum of R_{k-1})_{[K]\j}.
// Each value is the same element of GF(2^64) as the sum over the sieve points.
//
// Why. On a Chung-Lu graph with n = 1e6, m = 1e7 the sieve-point engine
// multiplies 1,024 points for each of 330,000 rows at each layer of a k = 10
// query; walks from the source that reach the last layer pass 1,400 to 62,000
// of them per layer, with at most 126 values each. Measured against that engine
// on three graphs of each kind (how many rows matter differs several times over):
//   motif, k = 10, n = 1e6, m = 1e7                 23.1-26.8 -> 0.36-1.07 ms a query
//   from a hub, k = 12, n = 2e5, m = 2e6            24.7-41.4 -> 0.61-1.31 ms
//   contacts, k = 12, n = 2,000, m = 30,011         4.4-4.7 -> 0.19 ms
//   uniform, k = 8, n = 1e5, m = 1e6                52-60 -> 25 us (a handful of rows)
//   n = 1,000, m = 10,000, k = 5                    26-27 -> 19 us
// What bounds it now: with many rows the products (issue slots of the integer
// multiplies and XORs: 257 cycles per warp product and scheduler, the loop alone),
// with few the chain of layers, some 45 grid barriers of 1.6 us at k = 12, and in
// one block's shared memory about 2 us a layer.
#include <algorithm>
#include <cstring>
#include <iterator>
#include <type_traits>

#include "rr_frontier.cuh"

namespace rr {

namespace {

constexpr int kThreads = 512;
constexpr int kWarps = kThreads / 32;
constexpr uint32_t kTeams = 5;        // team sizes of a wedge block: 1, 2, 4, 8 warps, all of them
__host__ __device__ constexpr uint32_t team_threads(uint32_t t) { return t + 1 < kTeams ? 32u << t : (uint32_t)kThreads; }
__host__ __device__ constexpr uint32_t team_count(uint32_t t) { return (uint32_t)kThreads / team_threads(t); }
// A team's share of the block's shared memory.
__host__ __device__ constexpr uint32_t team_smem(uint32_t smem, uint32_t t) { return smem / team_count(t) / 16u * 16u; }
constexpr uint32_t kMaxRows = 32;     // rows of one item: the lanes of the team's first warp
constexpr uint32_t kSplit = 28;       // words of a split multiplier: 9 pieces of 3 classes, padded to whole 16-byte loads
constexpr uint32_t kSup1 = 16, kSup2 = 256, kSup3 = 4096;  // blocks per partial sum
constexpr uint32_t kScanBlocks = 48, kScanSpan = 6, kScanLong = 4096;  // when a level's prefix sums are completed (x_scans)
// Bitmap words per scan tile (a block takes four per thread at a time), and the
// longest bitmap whose tiles count what lies before them themselves: 16 reads of
// 16 bytes per thread at most, against a pass of its own and its barrier.
constexpr uint32_t kTileWords = 2048, kDirectWords = 32768;
__host__ __device__ constexpr uint32_t x_tile_words(uint32_t words)
{
    return words <= kDirectWords ? kTileWords : ((words + 255u) / 256u + kTileWords - 1u) / kTileWords * kTileWords;
}

__host__ __device__ constexpr uint32_t x_binom(uint32_t n, uint32_t d)
{
    uint64_t r = 1;
    if (d > n) return 0;
    for (uint32_t i = 1; i <= d; ++i) r = r * (n - d + i) / i;
    return (uint32_t)r;
}

// the same at run time (n, d <= kXMaxLabels + 1)
struct XBinomials {
    uint16_t v[kXMaxLabels + 2][kXMaxLabels + 2];
    constexpr XBinomials() : v()
    {
        for (uint32_t i = 0; i < kXMaxLabels + 2; ++i)
            for (uint32_t d = 0; d < kXMaxLabels + 2; ++d) v[i][d] = (uint16_t)x_binom(i, d);
    }
};
__constant__ XBinomials c_binom;
__device__ __forceinline__ uint32_t x_binom_dev(uint32_t n, uint32_t d) { return c_binom.v[n][d]; }

// Subset tables: for every subset size d and d-subset T of [kXMaxLabels] in
// colexicographic order, element i of T and the rank of T without it, packed
// j | rank << 8, stored [i][T]. Colex order lists the subsets of the first K
// labels first, so one table serves every K.
__host__ __device__ constexpr uint32_t x_tab_off(uint32_t d)
{
    uint32_t o = 0;
    for (uint32_t i = 1; i < d; ++i) o += i * x_binom(kXMaxLabels, i);
    return o;
}

struct XTabOffsets {
    uint32_t v[kXMaxLabels + 2];
    constexpr XTabOffsets() : v()
    {
        for (uint32_t d = 1; d < kXMaxLabels + 2; ++d) v[d] = x_tab_off(d);
    }
};
__constant__ XTabOffsets c_tab_off;
__device__ __forceinline__ uint32_t x_tab_off_dev(uint32_t d) { return c_tab_off.v[d]; }

// For K <= kPackedLabels the tables of [K] once more, packed ([d][i][T], K 2^(K-1)
// words), so that a block copies them in one go.
constexpr uint32_t kPackedLabels = 11;
__host__ __device__ constexpr uint32_t x_packed_off(uint32_t K)  // sum of i 2^(i-1), i < K
{
    return (K - 2u) * (1u << (K - 1u)) + 1u;
}

__global__ void __launch_bounds__(128) k_packed_table(const uint32_t *__restrict__ tab, uint32_t *__restrict__ packed)
{
    const uint32_t K = blockIdx.y + 1;
    uint32_t *o = packed + x_packed_off(K);
    for (uint32_t d = 1; d <= K; ++d) {
        const uint32_t c = x_binom_dev(K, d), cm = x_binom_dev(kXMaxLabels, d), *src = tab + x_tab_off_dev(d);
        for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < d * c; i += gridDim.x * blockDim.x) o[i] = src[i / c * cm + i % c];
        o += d * c;
    }
}

__global__ void __launch_bounds__(128) k_subset_table(uint32_t *__restrict__ tab)
{
    constexpr uint32_t W = kXMaxLabels + 1;
    __shared__ uint32_t bin[W][W];
    for (uint32_t i = threadIdx.x; i < W * W; i += blockDim.x) bin[i / W][i % W] = x_binom(i / W, i % W);
    __syncthreads();
    const uint32_t d = blockIdx.y + 1, cm = bin[kXMaxLabels][d];
    const uint32_t T = blockIdx.x * blockDim.x + threadIdx.x;
    if (T >= cm) return;
    uint32_t set = 0, t = T, c = kXMaxLabels;
    for (uint32_t i = d; i >= 1; --i) {  // the largest c with C(c, i) <= t
        do --c;
        while (bin[c][i] > t);
        set |= 1u << c;
        t -= bin[c][i];
    }
    // rank without element i: the elements above it move down one place
    uint32_t below = 0, above = 0, pos = 0;
    for (uint32_t m = set; m; m &= m - 1) {
        const uint32_t e = (uint32_t)__ffs((int)m) - 1u;
        if (pos) above += bin[e][pos];  // places 1.. with the lowest element gone
        ++pos;
    }
    pos = 0;
    uint32_t *o = tab + x_tab_off(d) + T;
    for (uint32_t m = set; m; m &= m - 1) {
        const uint32_t e = (uint32_t)__ffs((int)m) - 1u;
        o[pos * cm] = e | ((below + above) << 8);
        const uint32_t rest = m & (m - 1);
        below += bin[e][pos + 1];
        if (rest) above -= bin[__ffs((int)rest) - 1][pos + 1];
        ++pos;
    }
}

__device__ __forceinline__ uint64_t now_ns()
{
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// The blocks that work together: the whole grid (cooperative launch, a barrier
// on a counter in device memory), or one block with a query of its own. The
// counter wait is bounded by time and by iterations; when it gives up it sets
// the error flag, and the blocks return.
//
// Two counters take turns, so that a block that is late to look at one barrier
// does not see what others said at the next (nobody reaches the one after that
// without it). A counter holds the arrivals there, plus 2^20 for each block that
// came with something to tell, modulo 2^32: once all have arrived, what is above
// the arrivals known to be there is what was told, also after the thousands of
// barriers of a batch whose queries run one after another.
constexpr uint32_t kTellOne = 1u << 20;  // above the blocks of a launch
struct Meetings {
    uint32_t count;    // so far
    uint32_t told[2];  // at each counter
    uint32_t result;   // of the last: 1 all came, 2 some told
};
struct View {
    uint32_t b, n;  // this block among n
    uint32_t *ctr, *err;  // ctr: two, 128 bytes apart
    Meetings *meet;       // shared memory, kept by thread 0
    uint64_t limit;       // of a wait (ns)
    bool some = false;    // some block came to the last barrier with something to tell
    // worker w of n, the items before `base` dealt out: its first item from there on
    __device__ static uint32_t first_item(uint32_t base, uint32_t w, uint32_t n)
    {
        if (!base) return w;
        const uint32_t r = base % n;
        return w >= r ? w - r : w + n - r;
    }
    // In two halves, for what may go on until the other blocks' part is needed:
    // arrive() publishes the block's writes, wait() returns once every block has
    // arrived.
    __device__ void arrive(bool tell = false)
    {
        __syncthreads();
        arrived(tell);
    }
    __device__ void arrived(bool tell)
    {
        if (threadIdx.x == 0) {
            const uint32_t turn = meet->count++ & 1u;
            asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(ctr + turn * 32u), "r"(tell ? kTellOne + 1u : 1u) : "memory");
        }
    }
    __device__ bool wait()
    {
        if (threadIdx.x == 0) {
            const uint32_t s = meet->count - 1u, turn = s & 1u;
            const uint32_t target = (s / 2u + 1u) * n;
            uint32_t v = 0, good = 0;
            uint64_t t0 = 0;
            for (uint32_t it = 0; it < 200000000u; ++it) {
                asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(ctr + turn * 32u) : "memory");
                v -= target;
                if (!(v & (kTellOne - 1u))) {
                    good = 1;
                    break;
                }
                if ((it & 1023u) != 1023u) continue;
                if (!t0) t0 = now_ns();
                if (*(volatile uint32_t *)err || now_ns() - t0 > limit) break;
            }
            if (!good) *(volatile uint32_t *)err = 1u;
            v /= kTellOne;
            meet->result = good | (v != meet->told[turn] ? 2u : 0u);
            meet->told[turn] = v;
        }
        __syncthreads();
        const uint32_t r = meet->result;
        some = (r & 2u) != 0;
        return (r & 1u) != 0;
    }
    __device__ bool sync()
    {
        if (n == 1) {
            __syncthreads();
            return true;
        }
        arrive();
        return wait();
    }
    // sync(), and whether any thread of any block came with `mine` (told by the
    // counter itself: no flag to read after the barrier)
    __device__ bool sync_or(bool mine, bool &any)
    {
        any = __syncthreads_or(mine);
        if (n == 1) return true;
        arrived(any);
        const bool good = wait();
        any = some;
        return good;
    }
};

// Some bit in the words [w, w1) of a bitmap, four at a time (bitmaps start on
// 256-byte boundaries).
__device__ __forceinline__ bool any_words(const uint32_t *A, uint32_t w, uint32_t w1)
{
    for (; w < w1 && (w & 3u); ++w)
        if (A[w]) return true;
    for (; w + 4u <= w1; w += 4u) {
        const uint4 x = *reinterpret_cast<const uint4 *>(A + w);
        if (x.x | x.y | x.z | x.w) return true;
    }
    for (; w < w1; ++w)
        if (A[w]) return true;
    return false;
}

// Long windows. A pass that reads every word of every window takes (rows that
// leave a vertex) x (rows that enter it) / 32 words a layer: k = 5 through two
// vertices with 20,000, 100,000 and 400,000 edges each way and waits as long as the
// time range took 0.44, 4.0 and 48.9 ms (0.36, 0.34 and 1.26 ms with summaries), and
// larger ones would outlast a barrier's wait. So a bitmap that windows of more than
// kWideWords words read has three summaries, each a bit per word of the level below
// it (at most 2^26 words, 2,048 in the last): S, the words of A that hold a row, and
// F, the words of N that some window covers whole. A window of more than kLongWords
// words then takes at most 2 kLongWords words of each level: the passes are linear in
// the rows, with a barrier more a layer. That barrier is why shorter windows are read
// directly. Graphs without such windows have kernels without the tests for summaries
// (x_plan<false>; one form for both: k = 12 on n = 2,000, m = 30,011 +1.4 %, both
// forms in one kernel: k = 8 arrival and bounded queries on n = 2e5, m = 2e6 +1 %). The
// summaries' functions are inlined: x_plan makes no call where the lanes of a warp
// have parted.
constexpr uint32_t kWideWords = 512;
constexpr uint32_t kLongWords = 128;
// Words of the first summary of `words` words, and of all three.
__host__ __device__ __forceinline__ uint32_t x_sum_level(uint32_t words) { return ((words + 31u) / 32u + 3u) / 4u * 4u; }
__host__ __device__ __forceinline__ uint32_t x_sum_words(uint32_t words)
{
    const uint32_t a = x_sum_level(words), b = x_sum_level(a);
    return a + b + x_sum_level(b);
}
// Where a level's summaries lie (X.sums: in 256-byte groups, from 1): S, then F.
struct XSums {
    uint32_t *S, *F;
};
__device__ __forceinline__ XSums x_sums(const XTmpl &t, const XLL &X)
{
    uint32_t *const S = reinterpret_cast<uint32_t *>(t.clear) + (size_t)(X.sums - 1u) * 64u;
    return XSums{S, S + x_sum_words(X.words)};
}
// The summaries of a level's A (the upper two were cleared): a warp a word of the first.
__device__ __forceinline__ void sum_level(const XLL &X, uint32_t *S, uint32_t gw, uint32_t nw)
{
    const uint32_t lane = threadIdx.x & 31u, n1 = (X.words + 31u) / 32u, l1 = x_sum_level(X.words);
    uint32_t *const S2 = S + l1, *const S3 = S2 + x_sum_level(l1);
    for (uint32_t i = gw; i < n1; i += nw) {
        const uint32_t w = i * 32u + lane;
        const uint32_t on = __ballot_sync(0xffffffffu, w < X.words && X.A[w] != 0);
        if (lane == 0) {
            S[i] = on;
            if (on) {
                const uint32_t b2 = 1u << (i & 31u), b3 = 1u << ((i >> 5) & 31u);
                if (!(__ldcg(S2 + (i >> 5)) & b2)) atomicOr(S2 + (i >> 5), b2);
                if (!(__ldcg(S3 + (i >> 10)) & b3)) atomicOr(S3 + (i >> 10), b3);
            }
        }
    }
}
// any_words over [a, b), by the summaries.
__device__ __forceinline__ bool any_long(const uint32_t *A, const uint32_t *S, uint32_t words, uint32_t a, uint32_t b)
{
    for (int level = 0;; ++level) {
        if (level == 3 || b - a <= kLongWords) return any_words(A, a, b);
        const uint32_t a1 = (a + 31u) & ~31u, b1 = b & ~31u;
        if (any_words(A, a, a1) || any_words(A, b1, b)) return true;
        a = a1 >> 5;
        b = b1 >> 5;
        A = level ? A + words : S;
        words = x_sum_level(words);
    }
}
// The words [a, b) are needed whole.
__device__ __forceinline__ void mark_long(uint32_t *F, uint32_t words, uint32_t a, uint32_t b)
{
    auto set = [&](uint32_t w, uint32_t mask) {
        if (mask & ~__ldcg(F + w)) atomicOr(F + w, mask);
    };
    for (int level = 0;; ++level) {  // the bits [a, b) of this summary
        const uint32_t w0 = a >> 5, w1 = (b - 1u) >> 5;
        const uint32_t first = 0xffffffffu << (a & 31u), last = 0xffffffffu >> (31u - ((b - 1u) & 31u));
        if (w0 == w1) {
            set(w0, first & last);
            return;
        }
        if (level == 2 || w1 - w0 <= 8u) {
            set(w0, first);
            for (uint32_t w = w0 + 1u; w < w1; ++w) set(w, 0xffffffffu);
            set(w1, last);
            return;
        }
        set(w0, first);
        set(w1, last);
        a = w0 + 1u;  // the words between, whole: bits of the next summary
        b = w1;
        words = x_sum_level(words);
        F += words;
    }
}
// Whether word w is marked.
__device__ __forceinline__ bool covered(const uint32_t *F, uint32_t words, uint32_t w)
{
    bool on = false;
    for (int level = 0; level < 3; ++level) {
        on |= (F[w >> 5] >> (w & 31u)) & 1u;
        w >>= 5;
        words = x_sum_level(words);
        F += words;
    }
    return on;
}

// Rows of partial sums over nb blocks: of 16, 256 and 4,096 blocks.
__host__ __device__ __forceinline__ uint32_t x_sup_rows(uint64_t nb)
{
    return (uint32_t)(nb / kSup1 + nb / kSup2 + nb / kSup3 + 3u);
}

// Needed rows of a level at positions below x (rank: the bitmap's word and the
// rows before it).
__device__ __forceinline__ uint32_t rank_below(const uint2 *rank, uint32_t x)
{
    const uint2 r = rank[x >> 5];
    return r.y + __popc(r.x & ((1u << (x & 31u)) - 1u));
}

// One wedge item: `rows` consecutive needed rows of a level, taken by a team of
// 1 << team warps. Few rows get large teams (all warps of a block on one row:
// the layer's latency counts), many rows one warp each (no block-wide waits; the
// warps cover each other's loads). Of the team sizes and rows per item (at most
// kMaxRows) that a team's share of shared memory holds, the pair is taken whose
// busiest team has the least to do, counted in product steps of a warp (about
// 1,000 cycles with four warps on a scheduler) with the measured cost of an
// item's other parts. Chosen once per level list, by the warp that counts its
// rows; the next level reads the rows' prefix sums by it. With powers of two and
// rows added until every team had an item, layers of 2,500 to 4,000 rows left
// the warps idle for a third of the time. Store items of up to 32 rows instead of
// 16 fill the last wave better where many short rows meet large teams (k = 12 from
// a hub of n = 2e5 1.35 -> 1.31 ms on one graph, at-most-k 3.58 -> 3.49 ms on one).
struct XShape {
    uint32_t team, rows, scan;  // team: log2
};
__host__ __device__ __forceinline__ XShape x_shape_of(uint32_t s) { return XShape{s & 0xffu, (s >> 8) & 0xffu, s >> 16}; }
__host__ __device__ __forceinline__ uint32_t x_item_bytes(uint32_t rows, uint32_t K, const XLL &X)
{
    return X.out ? rows * (K * 8u + 8u + 64u) : rows * (K * (4u * kSplit) + (X.cin + X.cout + X.uout) * 8u + 64u);
}
// Quarter steps of one item.
__device__ __forceinline__ uint32_t x_item_cost(uint32_t rows, uint32_t t, uint32_t K, const XLL &X)
{
    const uint32_t T = team_threads(t), W = T / 32u;
    auto rounds = [&](uint32_t n) { return (n + T - 1u) / T; };
    if (X.out) return 12u + 10u * rounds(rows * X.cout);
    const uint32_t per_warp = (rows + W - 1u) / W;
    uint32_t c = 16u + per_warp * (4u + X.cin / 64u) + rounds(rows * K) * 20u + rounds(rows * X.cout) * X.d * 4u +
                 rows * rounds(X.cout + X.uout);
    if (X.uout) c += rounds(rows * X.uout) * (X.d + 5u) * 4u;
    return c;
}
// By one warp; every lane returns the choice.
__device__ __noinline__ uint32_t x_choose_shape(uint32_t smem, uint32_t blocks, uint32_t cnt, uint32_t K, const XLL &X)
{
    const uint32_t lane = threadIdx.x & 31u;
    uint32_t best = 0xffffffffu, pick = 0;
    for (uint32_t i = lane; i < kTeams * kMaxRows; i += 32u) {
        const uint32_t t = i / kMaxRows, rows = i % kMaxRows + 1u;
        if ((rows > 1u || t + 1u < kTeams) && x_item_bytes(rows, K, X) > team_smem(smem, t)) continue;
        const uint32_t items = (cnt + rows - 1u) / rows, teams = blocks * team_count(t);
        const uint32_t cost = (items + teams - 1u) / teams * x_item_cost(rows, t, K, X);
        if (cost < best) {
            best = cost;
            pick = t | rows << 8;
        }
    }
    const uint32_t least = __reduce_min_sync(0xffffffffu, best);
    const uint32_t who = __ffs((int)__ballot_sync(0xffffffffu, best == least)) - 1u;
    pick = __shfl_sync(0xffffffffu, pick, (int)who);
    // room for the sums of all blocks (taken where the windows span many of them)
    const uint32_t rows = pick >> 8, nb = (cnt + rows - 1u) / rows;
    if (!X.out && nb >= kScanBlocks && (rows == 1u || nb <= X.ipcap)) pick |= 1u << 16;
    return pick;
}

// Carry-less inner products. gf64_mul splits both operands into 9 16-bit pieces
// (two Karatsuba levels) of 3 bit classes; everything after the 81 integer
// products of classes is linear, so a sum of products XORs them class by class
// and is put together and reduced once. The multipliers of a row serve all its
// subsets: their 27 words are formed once and read from shared memory in seven
// 16-byte loads (nine, a piece each, kept the shared-memory pipe as busy as the
// ALU: at-most-k, k = 10, on n = 1e6, m = 1e7 4.82 -> 4.62 ms).
// Per product this leaves 81 IMAD, about 41 three-input XORs and the 31
// instructions that split the other operand, against 240 of gf64_mul. An IMAD
// takes two issue cycles of its scheduler and the others one each, together 257
// cycles a product and warp with the loads and the end of a sum. Forms with fewer
// IMADs cost more: 48 64-bit multiplies of 32-bit pieces in four classes 350.
__device__ __forceinline__ uint64_t finish27(const uint32_t (&z)[27])
{
    uint64_t r[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        uint32_t c[3];
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            const uint32_t *q = z + 9 * i + 3 * j;
            c[j] = (q[0] & 0x49249249u) | (q[1] & 0x92492492u) | (q[2] & 0x24924924u);
        }
        const uint32_t m = c[2] ^ c[0] ^ c[1];
        r[i] = ((uint64_t)(c[1] ^ (m >> 16)) << 32) | (uint32_t)(c[0] ^ (m << 16));
    }
    const uint64_t m = r[2] ^ r[0] ^ r[1];
    return gf64_reduce(r[1] ^ (m >> 32), r[0] ^ (m << 32));
}

// One out-of-line multiply for the small queries' path: it runs each of its
// products once or twice, and fetching 4 KB of instructions again for every
// inlined copy took longer than the product (see x_tiny).
__device__ __noinline__ uint64_t mul_call(uint64_t a, uint64_t b) { return gf64_mul(a, b); }

// z'_{u,j}: the source's column eliminated (see the top of the file); a set of
// sources keeps all k labels as they are.
template <bool CALL = false>
__device__ __forceinline__ uint64_t zprime(const XQuery &Q, const uint64_t *omega, const uint8_t *color, uint32_t u, uint32_t j)
{
    auto mul = [](uint64_t x, uint64_t y) { return CALL ? mul_call(x, y) : gf64_mul(x, y); };
    if (!Q.colored) {
        const uint64_t zj = sm_draw(Q.key_z, (uint64_t)u * 32u + (j < Q.pivot ? j : j + 1u));
        return Q.multi ? zj : zj ^ mul(sm_draw(Q.key_z, (uint64_t)u * 32u + Q.pivot), Q.rho[j]);
    }
    const uint32_t c = color[u], d0 = Q.first[c], mu = Q.mu[c];
    uint64_t r = 0;
    for (uint32_t d = d0; d < d0 + mu; ++d) r ^= mul(sm_draw(Q.key_g, (uint64_t)u * 32u + d), omega[d * Q.K + j]);
    return r;
}
// omega'_{d,j} at i = d K + j: the shade factor with the source's column eliminated
template <bool CALL = false>
__device__ __forceinline__ uint64_t shade_factor(const XQuery &Q, uint32_t i)
{
    auto mul = [](uint64_t x, uint64_t y) { return CALL ? mul_call(x, y) : gf64_mul(x, y); };
    const uint32_t d = i / Q.K, j = i - d * Q.K;
    const uint64_t oj = sm_draw(Q.key_o, (uint64_t)d * 32u + (j < Q.pivot ? j : j + 1u));
    return Q.multi ? oj : oj ^ mul(sm_draw(Q.key_o, (uint64_t)d * 32u + Q.pivot), Q.rho[j]);
}
// A vertex walks may pass: it has a colour of M and is not deleted.
__device__ __forceinline__ bool allowed(const XQuery &Q, const uint8_t *color, uint32_t v)
{
    if (Q.colored && !Q.mu[color[v]]) return false;
    return !(Q.vmask && Q.vmask[v]);
}

// Forward and backward passes, ranks and row records of one query. Each pass is
// short (10 MB of row windows and bitmaps on n = 1e6, m = 1e7), so the dependent
// reads between two barriers bound it: a level's first windows are read before
// the barrier they wait at, whether a level is alive comes with the barrier, the
// warps take the steps of all level lists in one sequence. WIDE: with summaries.
template <bool WIDE>
__device__ __noinline__ bool x_plan(const XArgs &a, const XOne &o, View &v)
{
    const XQuery &Q = o.q;
    const XTmpl &t = o.t;
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    const uint32_t gw = v.b * kWarps + warp, nw = v.n * kWarps;
    const uint32_t gt = v.b * kThreads + threadIdx.x, nt = v.n * kThreads;
    constexpr uint32_t U = 2;  // bitmap words per warp and step

    // cleared first: needed-row bitmaps, summaries, counts
    for (uint32_t i = gt; i < t.clear4; i += nt) t.clear[i] = make_uint4(0, 0, 0, 0);
    if (v.b == 0)
        for (uint32_t i = threadIdx.x; i < t.nll; i += kThreads) {
            t.cnt[i] = 0;
            t.span[i] = 0;
        }
    if (Q.colored && v.b == v.n - 1)
        // shade factors with the source's column eliminated
        for (uint32_t i = threadIdx.x; i < Q.k * Q.K; i += kThreads) t.omega[i] = shade_factor(Q, i);
    const bool check = Q.colored || Q.vmask;
    uint32_t lmax = t.maxlev;
    uint32_t nlo[U] = {}, nhi[U] = {};  // the next level's first windows
    for (uint32_t l = 1; l <= t.maxlev; ++l) {
        bool live = false;
        uint32_t base = 0;
        for (uint32_t li = t.runs[l].first; li < t.runs[l].first + t.runs[l].count; ++li) {
            const XLL &X = t.ll[li];
            const XList &L = a.lists[X.list];
            const uint32_t steps = (L.words + U - 1) / U, i0 = View::first_item(base, gw, nw);
            const XLL &P = t.ll[X.prev];
            const uint32_t *const Ap = P.A;
            const bool none = Q.dead || (X.out && Q.pivot > l && !Q.multi);  // z_s is zero over the labels of k' = l + 1
            if (l == 1) {
                // a stream of tails: eight words a step keep enough reads in flight
                constexpr uint32_t U1 = 8;
                const uint32_t steps1 = (L.words + U1 - 1) / U1;
                for (uint32_t i = View::first_item(base, gw, nw); i < steps1; i += nw) {
                    uint32_t u[U1];
#pragma unroll
                    for (uint32_t x = 0; x < U1; ++x) {
                        const uint32_t r = (i * U1 + x) * 32u + lane;
                        u[x] = r < L.count ? L.src[r] : 0xffffffffu;
                    }
#pragma unroll
                    for (uint32_t x = 0; x < U1; ++x) {
                        bool on = u[x] != 0xffffffffu && !none && (Q.multi ? Q.smask[u[x]] != 0 : u[x] == Q.source);
                        if (on && check) on = !(Q.vmask && Q.vmask[u[x]]) && allowed(Q, a.color, L.head[(i * U1 + x) * 32u + lane]);
                        const uint32_t word = __ballot_sync(0xffffffffu, on);
                        if (lane == x && i * U1 + x < L.words) X.A[i * U1 + x] = word;
                        live |= word != 0;
                    }
                }
                base += steps1;
                continue;
            }
            // first the rows' windows, then both end words of each, then what lies
            // between
            for (uint32_t i = i0; i < steps; i += nw) {
                const bool ready = base == 0 && i == gw;
                const uint32_t w0 = i * U;
                uint32_t lo[U], hi[U], fw[U], lw[U];
                bool act[U];
#pragma unroll
                for (uint32_t x = 0; x < U; ++x) {
                    const uint32_t r = (w0 + x) * 32u + lane;
                    lo[x] = ready ? nlo[x] : r < L.count ? L.lo[r] : 0u;
                    hi[x] = ready ? nhi[x] : r < L.count ? L.hi[r] : 0u;
                }
#pragma unroll
                for (uint32_t x = 0; x < U; ++x) {
                    fw[x] = hi[x] > lo[x] ? Ap[lo[x] >> 5] : 0u;
                    lw[x] = hi[x] > lo[x] ? Ap[(hi[x] - 1u) >> 5] : 0u;
                }
#pragma unroll
                for (uint32_t x = 0; x < U; ++x) {
                    const uint32_t m0 = 0xffffffffu << (lo[x] & 31u), m1 = 0xffffffffu >> (31u - ((hi[x] - 1u) & 31u));
                    const uint32_t first = lo[x] >> 5, last = (hi[x] - 1u) >> 5;
                    if (hi[x] <= lo[x]) act[x] = false;
                    else if (first == last) act[x] = (fw[x] & m0 & m1) != 0;
                    else if ((fw[x] & m0) || (lw[x] & m1)) act[x] = true;
                    else if (WIDE && P.sums && last - first > kLongWords) act[x] = any_long(Ap, x_sums(t, P).S, P.words, first + 1u, last);
                    else act[x] = any_words(Ap, first + 1u, last);
                }
                if (check) {
                    uint32_t h[U];
#pragma unroll
                    for (uint32_t x = 0; x < U; ++x) h[x] = act[x] ? L.head[(w0 + x) * 32u + lane] : 0u;
#pragma unroll
                    for (uint32_t x = 0; x < U; ++x)
                        // walks through vertices without a colour of M, or deleted ones, are zero
                        if (act[x] && !allowed(Q, a.color, h[x])) act[x] = false;
                }
#pragma unroll
                for (uint32_t x = 0; x < U; ++x) {
                    const uint32_t word = __ballot_sync(0xffffffffu, act[x] && !none);
                    if (lane == x && w0 + x < L.words) X.A[w0 + x] = word;
                    live |= word != 0;
                }
            }
            base += steps;
        }
        if (l < t.maxlev) {
            const XList &L = a.lists[t.ll[t.runs[l + 1].first].list];
#pragma unroll
            for (uint32_t x = 0; x < U; ++x) {
                const uint32_t r = (gw * U + x) * 32u + lane;
                nlo[x] = r < L.count ? L.lo[r] : 0u;
                nhi[x] = r < L.count ? L.hi[r] : 0u;
            }
        }
        bool some;
        if (!v.sync_or(live, some)) return false;
        if (!some) {
            lmax = l - 1;
            break;
        }
        if (const XLL &X = t.ll[t.runs[l].first]; WIDE && l < t.maxlev && X.sums) {  // (the store level comes first)
            sum_level(X, x_sums(t, X).S, gw, nw);
            if (!v.sync()) return false;
        }
    }
    // no walk as long as an output needs: every count stays zero
    if (lmax == 0 || (!t.every && lmax < t.maxlev)) return v.sync();

    // backward: the rows of layer l - 1 in the window of a needed row of layer l
    // (at-most-k: every layer has outputs, every active row is needed)
    // Word w of level X's N, with what the long windows need whole.
    auto needed = [&t](const XLL &X, uint32_t w) {
        uint32_t m = X.N[w];
        if (WIDE && X.sums && covered(x_sums(t, X).F, X.words, w)) X.N[w] = m = X.A[w];
        return m;
    };
    if (!t.every)
        for (uint32_t l = lmax; l >= 2; --l) {
            const XLL &X = t.ll[t.runs[l].first];  // (one list a level)
            const XList &L = a.lists[X.list];
            const uint32_t steps = (L.words + U - 1) / U;
            const XLL &P = t.ll[X.prev];
            const uint32_t *const Ap = P.A;
            uint32_t *const Np = P.N;
            for (uint32_t i = gw; i < steps; i += nw) {
                const uint32_t w0 = i * U;
                const uint32_t mine = lane < U && w0 + lane < L.words ? needed(X, w0 + lane) : 0u;
                if (!__any_sync(0xffffffffu, mine != 0)) continue;
                uint32_t lo[U], hi[U];
#pragma unroll
                for (uint32_t x = 0; x < U; ++x) {
                    const bool on = (__shfl_sync(0xffffffffu, mine, (int)x) >> lane) & 1u;
                    const uint32_t r = (w0 + x) * 32u + lane;
                    lo[x] = on ? L.lo[r] : 0u;
                    hi[x] = on ? L.hi[r] : 0u;
                }
                uint32_t m[U], have[U];  // the window's first words
#pragma unroll
                for (uint32_t x = 0; x < U; ++x) {
                    m[x] = have[x] = 0;
                    if (hi[x] > lo[x]) {
                        m[x] = Ap[lo[x] >> 5] & (0xffffffffu << (lo[x] & 31u));
                        have[x] = Np[lo[x] >> 5];
                    }
                }
#pragma unroll
                for (uint32_t x = 0; x < U; ++x) {
                    if (hi[x] <= lo[x]) continue;
                    const uint32_t b0 = lo[x] >> 5, b1 = (hi[x] - 1) >> 5;
                    const uint32_t last = 0xffffffffu >> (31u - ((hi[x] - 1) & 31u));
                    if (b1 == b0) m[x] &= last;
                    if (m[x] & ~have[x]) atomicOr(Np + b0, m[x]);
                    uint32_t w = b0 + 1;
                    if (WIDE && P.sums && b1 - b0 > kLongWords) {
                        mark_long(x_sums(t, P).F, P.words, w, b1);
                        w = b1;
                    }
                    for (; w <= b1; ++w) {
                        const uint32_t mw = Ap[w] & (w == b1 ? last : 0xffffffffu);
                        if (mw & ~Np[w]) atomicOr(Np + w, mw);
                    }
                }
            }
            if (!v.sync()) return false;
        }
    if (const XLL &X = t.ll[t.runs[1].first]; WIDE && !t.every && X.sums) {  // (the other levels' words were completed on the way)
        for (uint32_t w = gt; w < X.words; w += nt) needed(X, w);
        if (!v.sync()) return false;
    }

    // ranks: per bitmap word the rows before it, and the levels' row counts. A
    // block takes a tile of kTileWords words; what lies before it, it counts
    // itself in lists of at most kDirectWords words, else the tiles' sums come
    // first.
    __shared__ uint32_t part[32];
    if (threadIdx.x < 32) part[threadIdx.x] = 0;
    __syncthreads();
    const uint32_t nll = t.runs[lmax].first + t.runs[lmax].count;  // level lists up to lmax
    bool tiled = false;
    for (uint32_t li = 0; li < nll; ++li) tiled |= t.ll[li].words > kDirectWords;
    for (uint32_t pass = tiled ? 0u : 1u; pass < 2; ++pass) {
        uint32_t base = 0;
        for (uint32_t li = 0; li < nll; ++li) {
            const XLL &X = t.ll[li];
            const uint32_t words = X.words, tw = x_tile_words(words), tiles = (words + tw - 1) / tw;
            const bool direct = words <= kDirectWords;
            if (pass == 0 && direct) continue;
            for (uint32_t i = View::first_item(base, v.b, v.n); i < tiles; i += v.n) {
                const uint32_t end = min(words, (i + 1) * tw);
                uint32_t sum = 0;
                if (pass == 0) {
                    for (uint32_t w = i * tw + threadIdx.x; w < end; w += kThreads) sum += __popc(X.N[w]);
                } else if (direct) {  // rows before the tile (tiles are whole 16-byte groups)
                    const uint4 *const N4 = reinterpret_cast<const uint4 *>(X.N);
                    for (uint32_t w = threadIdx.x; w < i * tw / 4u; w += kThreads) {
                        const uint4 y = N4[w];
                        sum += __popc(y.x) + __popc(y.y) + __popc(y.z) + __popc(y.w);
                    }
                } else if (threadIdx.x < i) {
                    sum = X.tsum[threadIdx.x];
                }
                uint32_t run_base = 0;
                if (i || pass == 0) {
                    sum = __reduce_add_sync(0xffffffffu, sum);
                    __syncthreads();
                    if (lane == 0) part[warp] = sum;
                    __syncthreads();
                    run_base = __reduce_add_sync(0xffffffffu, part[lane]);
                }
                if (pass == 0) {
                    if (threadIdx.x == 0) X.tsum[i] = run_base;
                    continue;
                }
                for (uint32_t w0 = i * tw; w0 < end; w0 += 4u * kThreads) {
                    // four words per thread
                    const uint32_t w = w0 + 4u * threadIdx.x;
                    uint32_t c[4], mysum = 0;
#pragma unroll
                    for (uint32_t x = 0; x < 4; ++x) {
                        c[x] = w + x < end ? X.N[w + x] : 0u;
                        mysum += __popc(c[x]);
                    }
                    uint32_t inc = mysum;
#pragma unroll
                    for (int d = 1; d < 32; d <<= 1) {
                        const uint32_t y = __shfl_up_sync(0xffffffffu, inc, d);
                        if (lane >= (uint32_t)d) inc += y;
                    }
                    __syncthreads();
                    if (lane == 31) part[warp] = inc;
                    __syncthreads();
                    const uint32_t other = part[lane];
                    const uint32_t before = __reduce_add_sync(0xffffffffu, lane < warp ? other : 0u);
                    uint32_t at = run_base + before + inc - mysum;
#pragma unroll
                    for (uint32_t x = 0; x < 4; ++x) {
                        if (w + x < end) X.rank[w + x] = make_uint2(c[x], at);
                        at += __popc(c[x]);
                    }
                    run_base += __reduce_add_sync(0xffffffffu, other);
                }
                if (end == words && warp == 0) {
                    const uint32_t shape = x_choose_shape(a.smem, v.n, run_base, Q.K, X);
                    if (lane == 0) {
                        t.cnt[li] = run_base;
                        t.shape[li] = shape;
                    }
                }
            }
            base += tiles;
        }
        if (!v.sync()) return false;
    }

    // the needed rows' windows, edges and tails, in list order, and how many rows
    // of the level below the windows hold together
    uint32_t base = 0;
    for (uint32_t li = 0; li < nll; ++li) {
        const XLL &X = t.ll[li];
        const XList &L = a.lists[X.list];
        const uint2 *const rank = X.rank, *const below = t.ll[X.prev].rank;
        if (X.level == 1) {
            // layer 1: few rows in long lists, a word per lane
            const uint32_t steps1 = (L.words + 31u) / 32u;
            for (uint32_t i = View::first_item(base, gw, nw); i < steps1; i += nw) {
                const uint32_t w = i * 32u + lane;
                const uint2 mine = w < L.words ? rank[w] : make_uint2(0, 0);
                uint32_t at = mine.y;
                for (uint32_t m = mine.x; m; m &= m - 1u, ++at) {
                    const uint32_t r = w * 32u + (uint32_t)__ffs((int)m) - 1u;
                    X.meta[at] = make_uint4(0, 0, L.eid[r], L.src[r]);
                    if (X.mhead) X.mhead[at] = L.head[r];
                    if (X.mtime) X.mtime[at] = L.time[r];
                }
            }
            base += steps1;
            continue;
        }
        const uint32_t steps = (L.words + U - 1) / U;
        uint64_t span = 0;
        for (uint32_t i = View::first_item(base, gw, nw); i < steps; i += nw) {
            const uint32_t w0 = i * U;
            const uint2 mine = lane < U && w0 + lane < L.words ? rank[w0 + lane] : make_uint2(0, 0);
            if (!__any_sync(0xffffffffu, mine.x != 0)) continue;
            uint32_t lo[U], hi[U], at[U], hd[U];
            uint4 m[U];
#pragma unroll
            for (uint32_t x = 0; x < U; ++x) {
                const uint32_t word = __shfl_sync(0xffffffffu, mine.x, (int)x);
                at[x] = __shfl_sync(0xffffffffu, mine.y, (int)x) + __popc(word & ((1u << lane) - 1u));
                const uint32_t r = (w0 + x) * 32u + lane;
                lo[x] = hi[x] = 0;
                if (!((word >> lane) & 1u)) {
                    at[x] = 0xffffffffu;
                } else {
                    lo[x] = L.lo[r];
                    hi[x] = L.hi[r];
                    m[x].z = L.eid[r];
                    m[x].w = L.src[r];
                    if (X.mhead) hd[x] = L.head[r];
                }
            }
#pragma unroll
            for (uint32_t x = 0; x < U; ++x) {
                m[x].x = m[x].y = 0;
                if (at[x] != 0xffffffffu) {
                    m[x].x = rank_below(below, lo[x]);
                    m[x].y = rank_below(below, hi[x]);
                    span += m[x].y - m[x].x;
                }
            }
#pragma unroll
            for (uint32_t x = 0; x < U; ++x)
                if (at[x] != 0xffffffffu) {
                    X.meta[at[x]] = m[x];
                    if (X.mhead) X.mhead[at[x]] = hd[x];
                    if (X.mtime) X.mtime[at[x]] = L.time[(w0 + x) * 32u + lane];
                }
        }
        base += steps;
        if (__any_sync(0xffffffffu, span != 0)) {
#pragma unroll
            for (int f = 16; f > 0; f >>= 1) span += __shfl_xor_sync(0xffffffffu, (unsigned long long)span, f);
            if (lane == 0) atomicAdd(t.span + X.prev, (unsigned long long)span);
        }
    }
    // the partial sums of layer 1's blocks
    for (uint32_t li = t.runs[1].first; li < t.runs[1].first + t.runs[1].count; ++li) {
        const XLL &X = t.ll[li];
        const uint32_t c = t.cnt[li];
        if (X.out || !c) continue;
        const uint32_t words = x_sup_rows(c) * (X.cout + X.uout);
        for (uint32_t w = gt; w < words; w += nt) X.sup[w] = 0;
    }
    return v.sync();
}

__device__ __forceinline__ void store_split(uint32_t *o, uint64_t v)
{
    const uint32_t w[3] = {(uint32_t)v, (uint32_t)(v >> 32), (uint32_t)v ^ (uint32_t)(v >> 32)};
    uint32_t p[28];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const uint32_t x[3] = {w[i], w[i] >> 16, w[i] ^ (w[i] >> 16)};
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            p[9 * i + 3 * j] = x[j] & 0x9249u;
            p[9 * i + 3 * j + 1] = x[j] & 0x2492u;
            p[9 * i + 3 * j + 2] = x[j] & 0x4924u;
        }
    }
    p[27] = 0;
    uint4 *q = reinterpret_cast<uint4 *>(o);
#pragma unroll
    for (int i = 0; i < 7; ++i) q[i] = make_uint4(p[4 * i], p[4 * i + 1], p[4 * i + 2], p[4 * i + 3]);
}

// z += x y for one piece of the two operands: their three classes each
struct Piece {
    uint32_t c0, c1, c2;
};
__device__ __forceinline__ Piece piece_of(uint32_t v)
{
    return Piece{v & 0x9249u, v & 0x2492u, v & 0x4924u};
}

__device__ __forceinline__ void load_split(const uint32_t *m, uint32_t (&y)[28])
{
    const uint4 *const q = reinterpret_cast<const uint4 *>(m);
#pragma unroll
    for (int i = 0; i < 7; ++i) {
        const uint4 t = q[i];
        y[4 * i] = t.x;
        y[4 * i + 1] = t.y;
        y[4 * i + 2] = t.z;
        y[4 * i + 3] = t.w;
    }
}

// sum over the d elements j of subset T of m_j w_{T \ j} (m: split multipliers).
// Two products a round: their six class products and the accumulator meet in
// three three-input XORs, 27 fewer a round than one product at a time (the ALU
// pipe bounds the loop: 94 of its operations a product measured, 82 so; k = 12
// from a hub of n = 2e5, m = 2e6 774 -> 733 us).
__device__ __forceinline__ uint64_t wedge_at(const uint32_t *__restrict__ tb, uint32_t cm, uint32_t T, uint32_t d,
                                             const uint32_t *m, const uint64_t *w)
{
    uint32_t z[27];
#pragma unroll
    for (int i = 0; i < 27; ++i) z[i] = 0;
    uint32_t e = __ldg(tb + T), i = 1;
#pragma unroll 1
    for (; i < d; i += 2) {
        const uint32_t f = __ldg(tb + i * cm + T), next = i + 1 < d ? __ldg(tb + (i + 1) * cm + T) : 0u;
        const uint64_t v = w[e >> 8], u = w[f >> 8];
        uint32_t y[28], g[28];
        load_split(m + (e & 255u) * kSplit, y);
        load_split(m + (f & 255u) * kSplit, g);
#pragma unroll
        for (int h = 0; h < 3; ++h) {
            const uint32_t x = h == 0 ? (uint32_t)v : h == 1 ? (uint32_t)(v >> 32) : (uint32_t)v ^ (uint32_t)(v >> 32);
            const uint32_t t = h == 0 ? (uint32_t)u : h == 1 ? (uint32_t)(u >> 32) : (uint32_t)u ^ (uint32_t)(u >> 32);
            const uint32_t xh = x >> 16, th = t >> 16;
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                const Piece a = piece_of(j == 0 ? x : j == 1 ? xh : x ^ xh), b = piece_of(j == 0 ? t : j == 1 ? th : t ^ th);
                const uint32_t y0 = y[9 * h + 3 * j], y1 = y[9 * h + 3 * j + 1], y2 = y[9 * h + 3 * j + 2];
                const uint32_t g0 = g[9 * h + 3 * j], g1 = g[9 * h + 3 * j + 1], g2 = g[9 * h + 3 * j + 2];
                uint32_t *const q = z + 9 * h + 3 * j;
                q[0] = ((q[0] ^ (a.c0 * y0) ^ (a.c1 * y2)) ^ (a.c2 * y1) ^ (b.c0 * g0)) ^ (b.c1 * g2) ^ (b.c2 * g1);
                q[1] = ((q[1] ^ (a.c0 * y1) ^ (a.c1 * y0)) ^ (a.c2 * y2) ^ (b.c0 * g1)) ^ (b.c1 * g0) ^ (b.c2 * g2);
                q[2] = ((q[2] ^ (a.c0 * y2) ^ (a.c1 * y1)) ^ (a.c2 * y0) ^ (b.c0 * g2)) ^ (b.c1 * g1) ^ (b.c2 * g0);
            }
        }
        e = next;
    }
    if (i == d) {  // the last of an odd number
        const uint64_t v = w[e >> 8];
        uint32_t y[28];
        load_split(m + (e & 255u) * kSplit, y);
#pragma unroll
        for (int h = 0; h < 3; ++h) {
            const uint32_t x = h == 0 ? (uint32_t)v : h == 1 ? (uint32_t)(v >> 32) : (uint32_t)v ^ (uint32_t)(v >> 32);
            const uint32_t xh = x >> 16;
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                const Piece a = piece_of(j == 0 ? x : j == 1 ? xh : x ^ xh);
                const uint32_t y0 = y[9 * h + 3 * j], y1 = y[9 * h + 3 * j + 1], y2 = y[9 * h + 3 * j + 2];
                uint32_t *const q = z + 9 * h + 3 * j;
                q[0] ^= (a.c0 * y0) ^ (a.c1 * y2) ^ (a.c2 * y1);
                q[1] ^= (a.c0 * y1) ^ (a.c1 * y0) ^ (a.c2 * y2);
                q[2] ^= (a.c0 * y2) ^ (a.c1 * y1) ^ (a.c2 * y0);
            }
        }
    }
    return finish27(z);
}

__device__ __forceinline__ void xor_shared(uint64_t *p, uint64_t v)
{
    uint32_t *w = reinterpret_cast<uint32_t *>(p);
    if ((uint32_t)v) atomicXor(w, (uint32_t)v);
    if ((uint32_t)(v >> 32)) atomicXor(w + 1, (uint32_t)(v >> 32));
}

// Level list li's prefix sums are completed (x_scan_blocks): when the windows
// that read it span more than kScanSpan blocks on average, and for long levels,
// where a few windows of thousands of rows hold their teams up. Otherwise the
// pass and its barrier (4 us) cost more than the extra reads: levels from 256,
// 1,024, 4,096, 16,384 blocks on: arrival, k = 8, 269, 258, 248, 248 us; bounded,
// k = 8, 368, 368, 353, 353 us; at-most-k, k = 10, on n = 1e6, m = 1e7 4.15, 4.15,
// 4.14, 4.15 ms, and 4.45 ms by the average alone.
__host__ __device__ __forceinline__ bool x_scans(const XTmpl &t, uint32_t li)
{
    const XShape sh = x_shape_of(t.shape[li]);
    if (!sh.scan || t.ll[li].level >= t.maxlev) return false;
    if (t.cnt[li] >= kScanLong * sh.rows) return true;
    uint64_t readers = 0;
    for (uint32_t i = t.runs[t.ll[li].level + 1].first, e = i + t.runs[t.ll[li].level + 1].count; i < e; ++i) readers += t.cnt[i];
    return t.span[li] > readers * sh.rows * kScanSpan;
}

// What a level reads of the level below: per needed row `stride` values, prefix
// sums within blocks of `rows` rows.
struct XBelow {
    const uint64_t *R, *IP;    // the rows; scanned levels: the sums of all blocks up to each
    const uint64_t *s1, *s2, *s3;
    uint32_t stride, rows, scan;
};
__device__ __forceinline__ XBelow x_below(const XTmpl &t, uint32_t prev, bool U)
{
    const XLL &P = t.ll[prev];
    const XShape sh = x_shape_of(t.shape[prev]);
    const uint32_t cnt = t.cnt[prev], nb = (cnt + sh.rows - 1u) / sh.rows;
    XBelow b;
    b.stride = U ? P.uout : P.cout;
    b.rows = sh.rows;
    b.scan = x_scans(t, prev) ? 1u : 0u;
    b.R = U ? P.U : P.R;
    // (P.IP: the cout columns of ipcap blocks, then the uout ones)
    b.IP = sh.rows == 1u ? b.R : P.IP + (U ? (size_t)P.ipcap * P.cout : 0);
    b.s1 = P.sup + (U ? (size_t)x_sup_rows(nb) * P.cout : 0);
    b.s2 = b.s1 + (size_t)(nb / kSup1 + 1u) * b.stride;
    b.s3 = b.s2 + (size_t)(nb / kSup2 + 1u) * b.stride;
    return b;
}
// A window's two ends in its block structure.
struct XEnds {
    uint32_t b0, b1;        // first and end block: whole blocks [b0, b1) lie between
    const uint64_t *p0, *p1;  // the row before each end inside its block, or null
};
__device__ __forceinline__ XEnds x_ends(const XBelow &B, uint32_t ra, uint32_t rb)
{
    XEnds e;
    e.b0 = ra / B.rows;
    e.b1 = rb / B.rows;
    e.p0 = ra - e.b0 * B.rows ? B.R + (size_t)(ra - 1u) * B.stride : nullptr;
    e.p1 = rb - e.b1 * B.rows ? B.R + (size_t)(rb - 1u) * B.stride : nullptr;
    if (B.scan && e.b0 == e.b1) e.b0 = e.b1 = 0;
    return e;
}
// The blocks [i, e) in as few pieces as the partial sums allow: the next one.
__device__ __forceinline__ const uint64_t *x_piece(const XBelow &B, uint32_t &i, uint32_t e)
{
    const uint64_t *p;
    if (!(i % kSup3) && i + kSup3 <= e) {
        p = B.s3 + (size_t)(i / kSup3) * B.stride;
        i += kSup3;
    } else if (!(i % kSup2) && i + kSup2 <= e) {
        p = B.s2 + (size_t)(i / kSup2) * B.stride;
        i += kSup2;
    } else if (!(i % kSup1) && i + kSup1 <= e) {
        p = B.s1 + (size_t)(i / kSup1) * B.stride;
        i += kSup1;
    } else {
        p = B.R + ((size_t)(i + 1u) * B.rows - 1u) * B.stride;
        ++i;
    }
    return p;
}
// XOR of the rows [ra, rb)'s values first, first + step, .. into dst; one warp.
// N values a lane and three rows of them are read before the first is used: one
// load and store after another, each store held back the loads behind it, and
// the teams of an SM wait here together (at-most-k, k = 10, on n = 1e6, m = 1e7
// 4.62 -> 4.27 ms, k = 12 from a hub of n = 2e5 685 -> 635 us).
template <uint32_t N>
__device__ __forceinline__ void window_values(const XBelow &B, const XEnds &e, uint32_t count, uint32_t first, uint32_t step,
                                              uint64_t *dst)
{
    for (uint32_t s0 = first; s0 < count; s0 += N * step) {
        uint64_t t[3][N];
        auto load = [&](uint64_t (&o)[N], const uint64_t *p) {
#pragma unroll
            for (uint32_t x = 0; x < N; ++x) o[x] = p && s0 + x * step < count ? __ldcg(p + s0 + x * step) : 0ull;
        };
        auto add = [&](uint64_t (&o)[N]) {
#pragma unroll
            for (uint32_t x = 0; x < N; ++x) t[0][x] ^= o[x];
        };
        load(t[0], e.p0);
        load(t[1], e.p1);
        if (B.scan) {  // (all of this is warp-uniform)
            if (e.b0 != e.b1) {
                load(t[2], e.b0 ? B.IP + (size_t)(e.b0 - 1u) * B.stride : nullptr);
                add(t[1]);
                load(t[1], B.IP + (size_t)(e.b1 - 1u) * B.stride);
                add(t[2]);
            }
            add(t[1]);
        } else {
            uint32_t i = e.b0;
            if (i < e.b1) {
                load(t[2], x_piece(B, i, e.b1));
                add(t[2]);
            }
            add(t[1]);
            while (i < e.b1) {
                load(t[1], x_piece(B, i, e.b1));
                load(t[2], i < e.b1 ? x_piece(B, i, e.b1) : nullptr);
                add(t[1]);
                add(t[2]);
            }
        }
#pragma unroll
        for (uint32_t x = 0; x < N; ++x)
            if (s0 + x * step < count) dst[s0 + x * step] = t[0][x];
    }
}
__device__ __forceinline__ void window_sum(const XBelow &B, uint32_t ra, uint32_t rb, uint32_t count, uint32_t first,
                                           uint32_t step, uint64_t *dst)
{
    const XEnds e = x_ends(B, ra, rb);
    if (count > 2u * step) window_values<4>(B, e, count, first, step, dst);
    else window_values<2>(B, e, count, first, step, dst);
}

// Completes a level's prefix sums: IP[b] = the XOR of the blocks up to b (rows of
// one: in place). A warp takes 16 blocks and 32 columns, the sums before them
// from the partial sums. A window then takes four reads instead of one per
// piece: of a layer of 136,000 rows of 126 values the windows were a quarter of
// the time with up to 30 pieces one after another.
__device__ __forceinline__ void x_scan_blocks(const XTmpl &t, uint32_t li, const View &v)
{
    const XLL &X = t.ll[li];
    const uint32_t lane = threadIdx.x & 31u, gw = v.b * kWarps + (threadIdx.x >> 5), nw = v.n * kWarps;
    const uint32_t cnt = t.cnt[li], rows = x_shape_of(t.shape[li]).rows, nb = (cnt + rows - 1u) / rows;
    const uint32_t groups = (nb + kSup1 - 1u) / kSup1;
    const uint32_t cr = X.R ? (X.cout + 31u) / 32u : 0u, cu = (X.uout + 31u) / 32u, cols = cr + cu;
    for (uint32_t i = gw; i < groups * cols; i += nw) {
        const uint32_t g = i / cols, c = i - g * cols;
        const bool U = c >= cr;
        const XBelow B = x_below(t, li, U);
        const uint32_t s = (U ? c - cr : c) * 32u + lane;
        if (s >= B.stride) continue;
        uint64_t *const R = (U ? X.U : X.R) + s;
        uint64_t *const IP = rows == 1u ? R : X.IP + (U ? (size_t)X.ipcap * X.cout : 0) + s;
        uint64_t acc = 0;
        const uint32_t first = g * kSup1;
        for (uint32_t b = 0; b < first / kSup3; ++b) acc ^= B.s3[(size_t)b * B.stride + s];
#pragma unroll 4
        for (uint32_t b = first / kSup3 * (kSup3 / kSup2); b < first / kSup2; ++b) acc ^= B.s2[(size_t)b * B.stride + s];
#pragma unroll 4
        for (uint32_t b = first / kSup2 * (kSup2 / kSup1); b < g; ++b) acc ^= B.s1[(size_t)b * B.stride + s];
        uint64_t tot[kSup1];
#pragma unroll
        for (uint32_t b = 0; b < kSup1; ++b)
            tot[b] = first + b < nb ? R[(size_t)(min(cnt, (first + b + 1u) * rows) - 1u) * B.stride] : 0ull;
#pragma unroll
        for (uint32_t b = 0; b < kSup1; ++b) {
            acc ^= tot[b];
            if (first + b < nb) IP[(size_t)(first + b) * B.stride] = acc;
        }
    }
}

// Layers lbeg..lend of a query over its needed rows. One item = a
// block of consecutive needed rows of one level, taken by one team of warps:
// their window sums of the level below, the multipliers y z'_j (split), one
// thread per (row, subset) for the wedge, the running XOR over the block's rows.
// The store level below an out level keeps U = z'_v ^ (its value), v the row's
// head, on the label sets the output needs: the window of an out row lies in one
// vertex's rows, so the wedge with that vertex is taken once per stored row, not
// per out row, and an out row needs y sum_j z'_{w,j} U_j only, one product per
// label and one per row.
__device__ __noinline__ bool x_wedge(const XArgs &a, const XOne &o, View &v, uint32_t lbeg, uint32_t lend, bool last_sync)
{
    extern __shared__ __align__(16) uint64_t sm_all[];
    const XQuery &Q = o.q;
    const XTmpl &t_ = o.t;
    const uint32_t lane = threadIdx.x & 31u;
    const uint32_t gt = v.b * kThreads + threadIdx.x, nt = v.n * kThreads;
    for (uint32_t l = lbeg; l <= lend; ++l) {
        bool any = false;
        uint32_t base_item = 0;
        for (uint32_t li = t_.runs[l].first; li < t_.runs[l].first + t_.runs[l].count; ++li) {
            const uint32_t cnt = t_.cnt[li];
            if (!cnt) continue;
            any = true;
            const XLL &X = t_.ll[li];
            const uint32_t cin = X.cin, cout = X.cout, uout = X.uout, d = X.d;
            const uint32_t K = X.out ? cout : Q.K;  // labels in use
            const XShape sh = x_shape_of(t_.shape[li]);
            const uint32_t rows = sh.rows, nb = (cnt + rows - 1) / rows;
            // the thread's team, its number in the grid and its shared memory
            const uint32_t tsize = team_threads(sh.team), team = threadIdx.x / tsize, tid = threadIdx.x % tsize;
            const uint32_t nteam = v.n * team_count(sh.team), gteam = team * v.n + v.b, twarps = tsize / 32u;
            const uint32_t tsmem = team_smem(a.smem, sh.team);
            uint64_t *const sm = sm_all + (size_t)team * (tsmem / 8);
            uint32_t *const msp = reinterpret_cast<uint32_t *>(sm);  // rows x K split multipliers
            uint64_t *const dr = sm + (size_t)rows * K * (kSplit / 2), *const G = dr + rows * cin, *const Us = G + rows * cout;
            uint4 *const smeta = reinterpret_cast<uint4 *>(sm + (tsmem / 8 - rows * 8u));
            uint32_t *const shead = reinterpret_cast<uint32_t *>(smeta + rows), *const srun = shead + rows;
            uint32_t *const sfirst = srun + rows;  // (rows + 1)
            auto sync = [&] {
                if (sh.team == 0) __syncwarp();
                else if (sh.team + 1u == kTeams) __syncthreads();
                else asm volatile("bar.sync %0, %1;" ::"r"(team + 1u), "r"(tsize) : "memory");
            };
            XBelow B{};
            if (l > 1) B = x_below(t_, X.prev, X.out != 0);
            uint64_t *const E = X.out ? Q.E : nullptr, *const S = Q.S + (size_t)X.row * a.n;
            for (uint32_t it = View::first_item(base_item, gteam, nteam); it < nb; it += nteam) {
                const uint32_t row0 = it * rows, nr = min(rows, cnt - row0);
                sync();
                // (at most 32 rows: the team's first warp)
                if (tid < 32u) {
                    uint32_t h = 0xffffffffu;
                    if (tid < nr) {
                        uint4 mt = X.meta[row0 + tid];
                        if (X.mhead) shead[tid] = h = X.mhead[row0 + tid];
                        smeta[tid] = mt;
                    }
                    // runs of equal heads: their first rows, and each row's run
                    const uint32_t up = __shfl_up_sync(0xffffffffu, h, 1);
                    const uint32_t starts = __ballot_sync(0xffffffffu, tid < nr && (tid == 0 || h != up));
                    const uint32_t run = __popc(starts & (0xffffffffu >> (31u - tid))) - 1u;
                    if (tid < nr) {
                        srun[tid] = run;
                        if ((starts >> tid) & 1u) sfirst[run] = tid;
                        if (tid == 0) sfirst[nr] = __popc(starts);
                    }
                }
                sync();
                if (!X.out) {
                    if (l > 1) {
                        // a warp takes whole rows, or with fewer rows than warps a share of
                        // one row's columns
                        const uint32_t w = tid >> 5, share = twarps / nr;
                        if (share <= 1u) {
                            for (uint32_t q = w; q < nr; q += twarps)
                                window_sum(B, smeta[q].x, smeta[q].y, cin, lane, 32u, dr + q * cin);
                        } else if (w < share * nr) {
                            const uint32_t q = w / share;
                            window_sum(B, smeta[q].x, smeta[q].y, cin, (w - q * share) * 32u + lane, 32u * share, dr + q * cin);
                        }
                    }
                    if (l == 1) {
                        // y_{e,1} z_{s,p}; a set of sources: y_{e,1} z_{s,j}
                        for (uint32_t t = tid; t < nr * cout; t += tsize) {
                            const uint32_t q = t / cout;
                            G[t] = gf64_mul(sm_draw(Q.key_y, (uint64_t)smeta[q].z * 32u),
                                            Q.multi ? zprime(Q, t_.omega, a.color, smeta[q].w, t - q * cout) : Q.d0);
                        }
                    } else {
                        for (uint32_t t = tid; t < nr * K; t += tsize) {
                            const uint32_t q = t / K, j = t - q * K;
                            const uint64_t y = sm_draw(Q.key_y, (uint64_t)smeta[q].z * 32u + (l - 1u));
                            store_split(msp + (size_t)t * kSplit, gf64_mul(y, zprime(Q, t_.omega, a.color, smeta[q].w, j)));
                        }
                        sync();
                        const uint32_t *const tb = a.tab + x_tab_off_dev(d);
                        const uint32_t cm = x_binom_dev(kXMaxLabels, d);
                        for (uint32_t t = tid; t < nr * cout; t += tsize) {
                            const uint32_t q = t / cout, T = t - q * cout;
                            G[t] = wedge_at(tb, cm, T, d, msp + (size_t)q * K * kSplit, dr + q * cin);
                        }
                    }
                    sync();
                    if (uout) {  // U on the d+1-subsets of the first d + 2 labels; z' once per run of heads
                        for (uint32_t t = tid, n = sfirst[nr] * uout; t < n; t += tsize) {
                            const uint32_t r = t / uout, j = t - r * uout;
                            store_split(msp + (size_t)t * kSplit, zprime(Q, t_.omega, a.color, shead[sfirst[r]], j));
                        }
                        sync();
                        const uint32_t *const tb = a.tab + x_tab_off_dev(d + 1u);
                        const uint32_t cm = x_binom_dev(kXMaxLabels, d + 1u);
                        for (uint32_t t = tid; t < nr * uout; t += tsize) {
                            const uint32_t q = t / uout, T = t - q * uout;
                            Us[t] = wedge_at(tb, cm, T, d + 1u, msp + (size_t)srun[q] * uout * kSplit, G + q * cout);
                        }
                        sync();
                    }
                    const bool whole = nb >= kSup1 && nr == rows;
                    for (uint32_t s = X.R ? tid : cout + tid; s < cout + uout; s += tsize) {
                        const bool isU = s >= cout;
                        const uint32_t st = isU ? uout : cout, c = isU ? s - cout : s;
                        const uint64_t *const g = (isU ? Us : G) + c;
                        uint64_t *const out = (isU ? X.U : X.R) + c;
                        uint64_t acc = 0;
                        for (uint32_t q = 0; q < nr; ++q) {
                            acc ^= g[q * st];
                            out[(size_t)(row0 + q) * st] = acc;
                        }
                        if (whole) {
                            auto add = [&](uint64_t *p) { atomicXor(reinterpret_cast<unsigned long long *>(p), (unsigned long long)acc); };
                            uint64_t *const s1 = X.sup + (isU ? (size_t)x_sup_rows(nb) * cout : 0) + c;
                            uint64_t *const s2 = s1 + (size_t)(nb / kSup1 + 1u) * st, *const s3 = s2 + (size_t)(nb / kSup2 + 1u) * st;
                            add(s1 + (size_t)(it / kSup1) * st);
                            if (nb >= kSup2) add(s2 + (size_t)(it / kSup2) * st);
                            if (nb >= kSup3) add(s3 + (size_t)(it / kSup3) * st);
                        }
                    }
                } else {
                    // z'_w of the runs' heads, and the sums of the rows
                    uint64_t *const zw = sm, *const sum = sm + rows * K;
                    for (uint32_t t = tid, n = sfirst[nr] * K; t < n; t += tsize) {
                        const uint32_t r = t / K;
                        zw[t] = zprime(Q, t_.omega, a.color, shead[sfirst[r]], t - r * K);
                    }
                    for (uint32_t q = tid; q < nr; q += tsize) sum[q] = 0;
                    struct Raw {
                        uint64_t a, b, c, d;
                    };
                    const uint32_t n = nr * K;
                    auto read = [&](uint32_t t) -> Raw {  // U of (row, subset) t, in pieces
                        Raw r{0, 0, 0, 0};
                        if (t >= n) return r;
                        const uint32_t q = t / K, T = t - q * K;
                        if (l == 1) {  // the source's z row itself
                            r.a = Q.multi ? zprime(Q, t_.omega, a.color, smeta[q].w, T) : Q.d0;
                            return r;
                        }
                        const XEnds e = x_ends(B, smeta[q].x, smeta[q].y);
                        uint32_t i = e.b0;
                        const uint64_t *pc = nullptr, *pd = nullptr;
                        if (B.scan) {
                            if (e.b0) pc = B.IP + (size_t)(e.b0 - 1u) * B.stride;
                            if (e.b1) pd = B.IP + (size_t)(e.b1 - 1u) * B.stride;
                            i = e.b1;
                        } else {
                            if (i < e.b1) pc = x_piece(B, i, e.b1);
                            if (i < e.b1) pd = x_piece(B, i, e.b1);
                        }
                        if (e.p0) r.a = e.p0[T];
                        if (e.p1) r.b = e.p1[T];
                        if (pc) r.c = pc[T];
                        if (pd) r.d = pd[T];
                        while (i < e.b1) r.a ^= x_piece(B, i, e.b1)[T];
                        return r;
                    };
                    auto use = [&](uint32_t t, uint64_t u) {  // T misses one label, whose z' it meets
                        const uint32_t q = t / K, T = t - q * K;
                        xor_shared(sum + q, gf64_mul(u, zw[srun[q] * K + (K - 1u - T)]));
                    };
                    // the next value is read while this one is multiplied; its pieces'
                    // XOR waits until it is used (taken at once, it held up the product:
                    // at-most-k, k = 10, on n = 1e6, m = 1e7 4.21 -> 4.15 ms)
                    Raw r = read(tid);
                    sync();
                    for (uint32_t t = tid; t < n; t += tsize) {
                        const uint64_t u = r.a ^ r.b ^ r.c ^ r.d;
                        r = read(t + tsize);
                        use(t, u);
                    }
                    sync();
                    if (tid < 32u) {
                        uint64_t x = 0;
                        if (tid < nr) {
                            const uint32_t e = smeta[tid].z;
                            x = gf64_mul(sum[tid], sm_draw(Q.key_y, (uint64_t)e * 32u + (l - 1u)));
                            if (E) E[e] = x;
                            if (X.Ec) X.Ec[row0 + tid] = x;
                        }
                        // runs of equal heads: one atomic, by the run's last row
                        const uint32_t first = tid < nr ? sfirst[srun[tid]] : tid;
#pragma unroll
                        for (int f = 1; f < 32; f <<= 1) {
                            const uint64_t y = __shfl_up_sync(0xffffffffu, (unsigned long long)x, f);
                            if (tid >= first + f) x ^= y;
                        }
                        if (tid < nr && x && (tid + 1u == nr || srun[tid + 1u] != srun[tid]))
                            atomicXor(reinterpret_cast<unsigned long long *>(S + shead[tid]), (unsigned long long)x);
                    }
                }
            }
            base_item += nb;
            __syncthreads();  // the next level list may form other teams
        }
        if (l < t_.maxlev)  // clear the next level's partial sums
            for (uint32_t li = t_.runs[l + 1].first; li < t_.runs[l + 1].first + t_.runs[l + 1].count; ++li) {
                const uint32_t cnt = t_.cnt[li];
                const XLL &X = t_.ll[li];
                if (X.out || !cnt) continue;
                const uint32_t rows = x_shape_of(t_.shape[li]).rows, nb = (cnt + rows - 1u) / rows;
                if (nb < kSup1) continue;
                const uint32_t w = x_sup_rows(nb) * (X.cout + X.uout);
                for (uint32_t i = gt; i < w; i += nt) X.sup[i] = 0;
            }
        const uint32_t st = t_.runs[l].first;  // the store level list, if the level has one
        const bool scan = l < t_.maxlev && t_.cnt[st] && x_scans(t_, st);
        if (any && (l < lend || last_sync || scan))
            if (!v.sync()) return false;
        if (scan) {
            x_scan_blocks(t_, st, v);
            if (!v.sync()) return false;
        }
    }
    return true;
}

// Minimum arrival times and bitmaps, after the last layer.
__device__ __noinline__ void x_outputs(const XArgs &a, const XOne &o, const View &v)
{
    const XQuery &Q = o.q;
    const uint32_t gt = v.b * kThreads + threadIdx.x, nt = v.n * kThreads;
    uint32_t base = 0;  // the threads take the rows of all levels in one sequence
    for (uint32_t li = 0; li < o.t.nll; ++li) {
        const XLL &X = o.t.ll[li];
        if (!X.Ec) continue;
        uint32_t *const R = Q.R + (size_t)X.row * a.n;
        // runs of equal head and time among the out rows (consecutive: the
        // rows keep the list's order)
        const uint32_t cnt = o.t.cnt[li];
        const uint32_t i0 = View::first_item(base, gt, nt);
        base += cnt;
        for (uint32_t i = i0; i < cnt; i += nt) {
            const uint32_t h = X.mhead[i], t = X.mtime[i];
            if (i && X.mhead[i - 1] == h && X.mtime[i - 1] == t) continue;
            uint64_t e = X.Ec[i];
            for (uint32_t x = i + 1; x < cnt && X.mhead[x] == h && X.mtime[x] == t; ++x) e ^= X.Ec[x];
            if (e) atomicMin(R + h, t);
        }
    }
    if (!Q.bitmap) return;
    // a warp takes 32 vertices: whole lines of the witness rows
    const uint32_t rows = o.t.every ? Q.k - 1 : 1u, lane = threadIdx.x & 31u;
    for (uint32_t w = gt >> 5; w < (a.n + 31u) / 32u; w += nt >> 5) {
        const uint32_t x = w * 32u + lane;
        uint64_t any = 0;
        if (x < a.n)
            for (uint32_t r = 0; r < rows; ++r) any |= Q.S[(size_t)r * a.n + x];
        const uint32_t word = __ballot_sync(0xffffffffu, any != 0);
        if (lane < 4u && w * 4u + lane < (a.n + 7u) / 8u) Q.bitmap[w * 4u + lane] = (uint8_t)(word >> (8u * lane));
    }
}

// ---------------------------------------------------------------------------
// Queries whose walks are few: one block, everything in shared memory, no
// bitmaps. What bounds such a query is its chain of dependent steps, so each
// layer is one load forward and one product after that:
//  * forward, the frontier is pushed along the edges sorted by (tail, time);
//    every edge's record names the edges that may follow it, so a layer reads
//    its rows with one dependent load. A level holds at most kTinyRows rows, each
//    with the set of the level below's rows in its window as a bit mask, and the
//    backward pass (one warp) and the window sums read no memory at all;
//  * the multipliers y z'_j of all levels are formed at once, before the layers,
//    and the subset tables are copied to shared memory beside layer 1;
//  * a layer's products (row, subset, element) are spread over the threads and
//    meet in shared memory, its window sums taken on the way: one block barrier
//    a layer.
//  * code that runs once is fetched once: one out-of-line multiply, no unrolled
//    loops (inlined copies made the step with the multipliers 2.5 us, 1.1 so).
// Uniform n = 1e5, m = 1e6, k = 8: 33.5 us with two loads, a window-sum step and
// global tables a layer, 25.5 us so; 16 sources, k = 6, n = 20,011: 91 us over
// the bitmaps (128 rows a level), 33 us here. A frontier that has kTinyGrow rows
// and grows is given up with layers to go (it would not fit, and the bitmap
// passes start that much later). Returns kTinyNoFit, with nothing written,
// when the query does not fit. Witnesses are written only after every block has
// cleared its part (clear: the barrier they arrived at).
// ---------------------------------------------------------------------------
constexpr uint32_t kTinyRows = 256, kTinyWords = kTinyRows / 32, kTinyTotal = 1024, kTinyPairs = 1024, kTinyHash = 512;
constexpr uint32_t kTinyGrow = 64;       // rows from which a growing frontier is given up early
constexpr uint32_t kTinyRange = 1024;    // followers of one edge, at most
enum { kTinyDone = 0, kTinyNoFit = 1, kTinyFailed = 2 };

struct TinyMem {
    uint4 row[kTinyTotal];                  // tail, head, time, edge
    uint2 next[kTinyTotal];                 // the edges that may follow: first record, count
    uint32_t mask[kTinyTotal][kTinyWords];  // rows of the level below in the window
    uint32_t need[kXMaxLevels + 1][kTinyWords];
    uint32_t base[kXMaxLevels + 2];         // first row of each level
    uint32_t cn[kXMaxLevels + 2];           // needed rows before each level
    uint32_t hkey[2][kTinyHash], hval[kTinyHash];
    uint32_t pair[kTinyPairs];
    uint32_t npair[2], count[2], over, need_g, need_d, toff[kXMaxLabels + 2], bin[kXMaxLabels + 2];
    uint64_t warm;
    uint16_t list[kTinyTotal];              // needed rows
    uint8_t lev[kTinyTotal];                // and their levels
    uint64_t acc[kTinyTotal];               // their sums
    uint64_t omega[(kXMaxLabels + 1) * (kXMaxLabels + 1)];
};

// XOR of the level below's values s of the rows in `mk`, by their places among
// its needed rows `nd`.
__device__ __forceinline__ uint64_t tiny_window(const uint32_t *mk, const uint32_t *nd, uint32_t words, const uint64_t *Gp,
                                                uint32_t cin, uint32_t s)
{
    uint64_t v = 0;
    uint32_t before = 0;
#pragma unroll 1
    for (uint32_t x = 0; x < words; ++x) {
        const uint32_t need = nd[x];
        for (uint32_t m = mk[x] & need; m; m &= m - 1)
            v ^= Gp[(before + __popc(need & ((m & (0u - m)) - 1u))) * cin + s];
        before += __popc(need);
    }
    return v;
}

__device__ __noinline__ int x_tiny(const XArgs &a, const XQuery &Q, bool every, View &clear, bool &cleared)
{
    extern __shared__ __align__(16) uint64_t sm_all[];
    TinyMem &M = *reinterpret_cast<TinyMem *>(sm_all);
    constexpr uint32_t kHead = (uint32_t)((sizeof(TinyMem) + 15) / 16 * 2);
    uint64_t *pool = sm_all + kHead;
    uint32_t pool_n = a.smem / 8 - kHead;
    const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5;
    const uint32_t k = Q.k, K = Q.K, sh = Q.multi ? 1u : 0u, last = k - 1;
    // subset tables of the first K labels, where they are small
    const bool tables = K <= kPackedLabels;
    uint32_t *const tab = reinterpret_cast<uint32_t *>(pool);
    if (tables) {
        const uint32_t w = K * (1u << (K - 1u));
        pool += (w + 1u) / 2u;
        pool_n -= (w + 1u) / 2u;
    }

    if (tid == 0) {
        M.count[0] = M.count[1] = M.npair[0] = M.npair[1] = M.over = 0;
        M.base[1] = 0;
    }
    for (uint32_t i = tid; i < 2u * kTinyHash; i += kThreads) M.hkey[0][i] = 0;
    __syncthreads();
    // layer 1: the edges leaving the source(s); beside it (the upper warps) the
    // subset tables and the shade factors
    bool wide = false;  // a source with more edges than kTinyRange
    if (warp >= kWarps / 2) {
        const uint32_t t = tid - kThreads / 2;
        if (t == 0) M.warm = mul_call(Q.key_y, Q.d0);  // fetches the multiply's code
        if (tables) {
            const uint32_t *const src = a.packed + x_packed_off(K);
#pragma unroll 4
            for (uint32_t i = t; i < K << (K - 1u); i += kThreads / 2) tab[i] = __ldg(src + i);
        }
        if (t <= K) {  // C(K, t), and where the packed table of t-subsets starts
            M.bin[t] = x_binom_dev(K, t);
            uint32_t off = 0;
            for (uint32_t d = 1; d < t; ++d) off += d * x_binom_dev(K, d);
            M.toff[t] = off;
        }
        if (Q.colored)
            for (uint32_t i = t; i < Q.k * K; i += kThreads / 2) M.omega[i] = shade_factor<true>(Q, i);
    } else if (!Q.dead) {
        const uint32_t ns = Q.multi ? Q.nslist : 1u;
        for (uint32_t i = warp; i < ns; i += kWarps / 2) {
            const uint32_t s = Q.multi ? Q.slist[i] : Q.source;
            if (Q.vmask && Q.vmask[s]) continue;
            const uint32_t o0 = a.ooff[s], o1 = a.ooff[s + 1];
            if (o1 - o0 > kTinyRange) {
                wide = true;
                continue;
            }
#pragma unroll 1
            for (uint32_t o = o0 + lane; o < o1; o += 32u) {
                const uint4 r = a.orec[o];  // head, time, edge, first follower
                const uint32_t fl = a.olen[o];
                if (!allowed(Q, a.color, r.x) || (!Q.multi && r.x == s)) continue;
                const uint32_t at = atomicAdd(&M.count[1], 1u);
                if (at < kTinyRows) {
                    M.row[at] = make_uint4(s, r.x, r.y, r.z);
                    M.next[at] = make_uint2(r.w, fl);
                }
            }
        }
    }
    // (the barrier's own answer, not M.over: the first warps past it may set that
    // for layer 2 before the last ones have looked)
    const bool over1 = __syncthreads_or(wide);
    uint32_t n = M.count[1], lmax = 1;
    const uint32_t n1 = n;
    uint32_t prev = n;
    if (over1 || n > kTinyRows) return kTinyNoFit;
    if (tid == 0) M.base[2] = n;
    // forward; the hash table, counters and pairs of a level are cleared while
    // the one before it uses the other
    for (uint32_t l = 2; l <= last && n; ++l) {
        const uint32_t b1 = M.base[l - 1] + n, b0 = b1 - n, par = l & 1u;  // (base[l] is written by now or below)
#pragma unroll 1
        for (uint32_t f = warp; f < n; f += kWarps) {
            const uint32_t v = M.row[b0 + f].y;
            const uint2 nx = M.next[b0 + f];
            if (nx.y > kTinyRange) {
                if (lane == 0) M.over = 1;
                continue;
            }
#pragma unroll 1
            for (uint32_t i = lane; i < nx.y; i += 32u) {
                const uint32_t p = nx.x + i;
                const uint4 r = a.orec[p];
                const uint32_t fl = l < last ? a.olen[p] : 0u;
                if (!allowed(Q, a.color, r.x) || (!Q.multi && r.x == Q.source)) continue;
                // the row's place in the level (one per edge)
                uint32_t h = (p * 2654435761u) >> 23;  // 9 bits: kTinyHash
                bool placed = false;
                for (uint32_t tries = 0; tries < kTinyHash && !placed; ++tries) {
                    const uint32_t key = atomicCAS(&M.hkey[par][h], 0u, p + 1u);
                    if (key == 0u) {
                        const uint32_t at = atomicAdd(&M.count[par], 1u);
                        M.hval[h] = at;
                        if (at < kTinyRows && b1 + at < kTinyTotal) {
                            M.row[b1 + at] = make_uint4(v, r.x, r.y, r.z);
                            M.next[b1 + at] = make_uint2(r.w, fl);
#pragma unroll
                            for (uint32_t x = 0; x < kTinyWords; ++x) M.mask[b1 + at][x] = 0;
                        }
                    }
                    placed = key == 0u || key == p + 1u;
                    if (!placed) h = (h + 1u) % kTinyHash;
                }
                const uint32_t pp = atomicAdd(&M.npair[par], 1u);
                if (!placed || pp >= kTinyPairs) M.over = 1;
                else M.pair[pp] = f << 16 | h;
                if (M.over) break;
            }
        }
        __syncthreads();
        n = M.count[par];
        if (M.over || n > kTinyRows || b1 + n > kTinyTotal || (n > kTinyGrow && n > prev + prev / 8u && l + 2u < last)) return kTinyNoFit;
        prev = n;
#pragma unroll 1
        for (uint32_t i = tid; i < M.npair[par]; i += kThreads) {
            const uint32_t f = M.pair[i] >> 16, e = M.hval[M.pair[i] & 0xffffu];
            atomicOr(&M.mask[b1 + e][f >> 5], 1u << (f & 31u));
        }
        for (uint32_t i = tid; i < kTinyHash; i += kThreads) M.hkey[par ^ 1u][i] = 0;
        if (tid == 0) {
            M.base[l] = b1;
            M.base[l + 1] = b1 + n;
            M.count[par ^ 1u] = M.npair[par ^ 1u] = 0;
        }
        if (n) lmax = l;
        __syncthreads();
    }
    if (n == 0 && !every) return kTinyDone;  // no walk of k vertices: every sum is zero
    if (n1 == 0) return kTinyDone;
    const uint32_t top = every ? lmax : last;

    // backward, the row counts and the space the layers take: one warp
    if (warp == 0) {
        __syncwarp();  // base[2] is lane 0's (k = 2: no layer's barriers came between)
#pragma unroll 1
        for (uint32_t i = lane; i < (top + 1u) * kTinyWords; i += 32u) {
            const uint32_t l = i / kTinyWords;
            uint32_t all = 0;
            if (l >= 1 && (every || l == top)) {
                const uint32_t c = M.base[l + 1] - M.base[l], b = (i % kTinyWords) * 32u;
                all = c >= b + 32u ? 0xffffffffu : c > b ? (1u << (c - b)) - 1u : 0u;
            }
            M.need[l][i % kTinyWords] = all;
        }
        __syncwarp();
#pragma unroll 1
        for (uint32_t l = top; l >= 2 && !every; --l) {
            const uint32_t b = M.base[l], c = M.base[l + 1] - b, words = (b - M.base[l - 1] + 31u) / 32u;
#pragma unroll 1
            for (uint32_t x = 0; x < words; ++x) {
                uint32_t m = 0;
#pragma unroll 1
                for (uint32_t e = lane; e < c; e += 32u)
                    if ((M.need[l][e >> 5] >> (e & 31u)) & 1u) m |= M.mask[b + e][x];
                m = __reduce_or_sync(0xffffffffu, m);
                if (lane == 0) M.need[l - 1][x] = m;
            }
            __syncwarp();
        }
        uint32_t c = 0;  // lane l: the needed rows of level l
        if (lane >= 1 && lane <= top)
#pragma unroll
            for (uint32_t x = 0; x < kTinyWords; ++x) c += __popc(M.need[lane][x]);
        uint32_t inc = c;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t o = __shfl_up_sync(0xffffffffu, inc, d);
            if (lane >= (uint32_t)d) inc += o;
        }
        if (lane >= 1 && lane <= top + 1u) M.cn[lane] = inc - c;
        const uint32_t d = lane - 1u + sh;
        const bool on = lane >= 1 && lane <= top;
        const uint32_t g = __reduce_max_sync(0xffffffffu, on ? c * M.bin[d] : 0u);
        const uint32_t w = __reduce_max_sync(0xffffffffu, on && lane > 1 ? c * M.bin[d - 1u] : 0u);
        if (lane == 0) {
            M.need_g = g;
            M.need_d = w;
        }
    }
    __syncthreads();
    const uint32_t total = M.cn[top + 1], need_g = M.need_g, need_d = M.need_d;
    if (2u * total * K + need_d + 3u * need_g > pool_n) return kTinyNoFit;
    uint64_t *const mul = pool, *const zw = mul + total * K, *const dr = zw + total * K;
    uint64_t *G[3] = {dr + need_d, dr + need_d + need_g, dr + need_d + 2u * need_g};  // level l's values in G[l % 3]
    // the needed rows by level
    for (uint32_t i = tid, rows = M.base[top + 1]; i < rows; i += kThreads) {
        uint32_t l = 1;
#pragma unroll 1
        while (i >= M.base[l + 1]) ++l;
        const uint32_t e = i - M.base[l];
        if (!((M.need[l][e >> 5] >> (e & 31u)) & 1u)) continue;
        uint32_t at = M.cn[l] + __popc(M.need[l][e >> 5] & ((1u << (e & 31u)) - 1u));
#pragma unroll 1
        for (uint32_t x = 0; x < (e >> 5); ++x) at += __popc(M.need[l][x]);
        M.list[at] = (uint16_t)i;
        M.lev[at] = (uint8_t)l;
        M.acc[at] = 0;
    }
    for (uint32_t i = tid; i < need_g; i += kThreads) G[2][i] = 0;
    __syncthreads();
#pragma unroll 1
    for (uint32_t i = tid; i < 2u * total * K; i += kThreads) {
        const bool second = i >= total * K;
        const uint32_t x = second ? i - total * K : i, at = x / K, j = x - at * K, l = M.lev[at];
        const uint4 r = M.row[M.list[at]];
        if (second) {
            if (every || l == top) zw[x] = zprime<true>(Q, M.omega, a.color, r.y, j);
        } else if (l > 1 || Q.multi) {
            const uint64_t y = sm_draw(Q.key_y, (uint64_t)r.w * 32u + (l - 1u));
            mul[x] = mul_call(y, zprime<true>(Q, M.omega, a.color, r.x, j));
            if (l == 1) G[1][at * K + j] = mul[x];
        } else if (j == 0) {
            G[1][at] = mul_call(sm_draw(Q.key_y, (uint64_t)r.w * 32u), Q.d0);
        }
    }
    __syncthreads();
    // the layers: step l forms level l's values and the witness terms of level l - 1
    for (uint32_t l = 2; l <= top + 1u; ++l) {
        uint64_t *const Gc = G[l % 3u], *const Gp = G[(l + 2u) % 3u], *const Gn = G[(l + 1u) % 3u];
        if (l <= top) {
            const uint32_t c0 = M.cn[l], c = M.cn[l + 1] - c0, d = l - 1 + sh, cout = M.bin[d], cin = M.bin[d - 1];
            const uint64_t *const ml = mul + c0 * K;
            const uint32_t *const tb = tables ? tab + M.toff[d] : a.tab + x_tab_off_dev(d);
            const uint32_t cm = tables ? cout : x_binom_dev(kXMaxLabels, d);
            const uint32_t *const nd = M.need[l - 1];
            const uint32_t words = (M.base[l] - M.base[l - 1] + 31u) / 32u;  // of the level below's masks
            if (c * cout * d <= 4u * kThreads) {
#pragma unroll 1
                for (uint32_t i = tid; i < c * cout * d; i += kThreads) {
                    const uint32_t q = i / (cout * d), r = i - q * cout * d, x = r / cout, T = r - x * cout;
                    const uint32_t e = tb[x * cm + T];
                    const uint64_t w = tiny_window(M.mask[M.list[c0 + q]], nd, words, Gp, cin, e >> 8);
                    xor_shared(&Gc[q * cout + T], mul_call(ml[q * K + (e & 255u)], w));
                }
            } else {
#pragma unroll 1
                for (uint32_t i = tid; i < c * cin; i += kThreads) {
                    const uint32_t q = i / cin;
                    dr[i] = tiny_window(M.mask[M.list[c0 + q]], nd, words, Gp, cin, i - q * cin);
                }
                __syncthreads();
#pragma unroll 1
                for (uint32_t i = tid; i < c * cout; i += kThreads) {
                    const uint32_t q = i / cout, T = i - q * cout;
                    uint64_t v = 0;
                    for (uint32_t x = 0; x < d; ++x) {
                        const uint32_t e = tb[x * cm + T];
                        v ^= mul_call(ml[q * K + (e & 255u)], dr[q * cin + (e >> 8)]);
                    }
                    Gc[i] = v;
                }
            }
            if (l < top) {  // the next level's products add up from zero (it was read two steps ago)
                const uint32_t w = (M.cn[l + 2] - M.cn[l + 1]) * M.bin[d + 1u];
                for (uint32_t i = tid; i < w; i += kThreads) Gn[i] = 0;
            }
        }
        if (every ? !(Q.pivot > l - 1u && !Q.multi) : l == top + 1u) {
            // times z'_w over the first labels of k' = l
            const uint32_t c0 = M.cn[l - 1], c = M.cn[l] - c0, K2 = l - 1u + sh, st = M.bin[l - 2u + sh];
#pragma unroll 1
            for (uint32_t i = tid; i < c * K2; i += kThreads) {
                const uint32_t q = i / K2, T = i - q * K2;
                xor_shared(&M.acc[c0 + q], mul_call(Gp[q * st + T], zw[(c0 + q) * K + (K2 - 1u - T)]));
            }
        }
        __syncthreads();
    }
    // the witnesses: rows of one level and head together
    if (!cleared) {
        if (!clear.wait()) return kTinyFailed;
        cleared = true;
    }
    const uint32_t first = every ? 0u : M.cn[top];
    for (uint32_t at = first + tid; at < total; at += kThreads) {
        const uint32_t l = M.lev[at], c0 = M.cn[l], c1 = M.cn[l + 1];
        const uint4 r = M.row[M.list[at]];
        const size_t off = (size_t)(every ? l - 1u : 0u) * a.n + r.y;
        uint64_t sum = 0, same = 0;
        bool lead = true;
#pragma unroll 1
        for (uint32_t x = c0; x < c1; ++x) {
            const uint4 o = M.row[M.list[x]];
            if (o.y != r.y) continue;
            if (x < at) lead = false;
            sum ^= M.acc[x];
            if (o.z == r.z) same ^= M.acc[x];
        }
        if (lead && sum) {
            Q.S[off] = sum;
            if (Q.bitmap && !every) {
                // the head's byte: every vertex of it with a non-zero sum
                uint32_t bits = 0;
                for (uint32_t x = c0; x < c1; ++x) {
                    const uint32_t h = M.row[M.list[x]].y;
                    if (h >> 3 != r.y >> 3 || (bits >> (h & 7u)) & 1u) continue;
                    uint64_t hs = 0;
                    for (uint32_t z = x; z < c1; ++z)
                        if (M.row[M.list[z]].y == h) hs ^= M.acc[z];
                    if (hs) bits |= 1u << (h & 7u);
                }
                Q.bitmap[r.y >> 3] = (uint8_t)bits;
            }
        }
        if (Q.E) Q.E[r.w] = M.acc[at];
        if (Q.R && same) atomicMin(Q.R + off, r.z);  // the XOR over the head's rows of the same time
    }
    if (Q.bitmap && every) {  // the bytes of the rows' heads over all witness rows
        __threadfence();
        __syncthreads();
        for (uint32_t at = tid; at < total; at += kThreads) {
            const uint32_t b = M.row[M.list[at]].y >> 3;
            uint32_t bits = 0;
            for (uint32_t w = 0; w < k - 1; ++w)
                for (uint32_t i = 0; i < 8; ++i) {
                    const uint32_t x = b * 8 + i;
                    if (x < a.n && __ldcg(Q.S + (size_t)w * a.n + x) != 0) bits |= 1u << i;
                }
            Q.bitmap[b] = (uint8_t)bits;
        }
    }
    return kTinyDone;
}

// Inverse (x != 0) by the extended Euclidean algorithm on binary polynomials.
__host__ __device__ static uint64_t gf64_inverse(uint64_t x)
{
    unsigned __int128 u = x, v = ((unsigned __int128)1 << 64) | 0x1B, g1 = 1, g2 = 0;
    auto deg = [](unsigned __int128 w) {
        const uint64_t hi = (uint64_t)(w >> 64), lo = (uint64_t)w;
#ifdef __CUDA_ARCH__
        return hi ? 127 - __clzll((long long)hi) : (lo ? 63 - __clzll((long long)lo) : -1);
#else
        return hi ? 127 - __builtin_clzll(hi) : (lo ? 63 - __builtin_clzll(lo) : -1);
#endif
    };
    while (u != 1) {
        int j = deg(u) - deg(v);
        if (j < 0) {
            const unsigned __int128 tu = u, tg = g1;
            u = v;
            v = tu;
            g1 = g2;
            g2 = tg;
            j = -j;
        }
        u ^= v << j;
        g1 ^= g2 << j;
    }
    return (uint64_t)g1;
}

// A batch's queries come without what depends on the source's z row (x_query
// forms it on the host for a single query: 0.7 us each, 180 us of a batch of 256
// with the blocks waiting); a warp forms it beside the clearing.
__device__ __noinline__ void x_constants(XQuery &Q, const uint8_t *color)
{
    const uint32_t lane = threadIdx.x & 31u, s = Q.source, k = Q.k;
    uint64_t z = 0;
    if (lane < k) {
        if (!Q.colored) {
            z = sm_draw(Q.key_z, (uint64_t)s * 32u + lane);
        } else {
            const uint32_t c = color[s];
            for (uint32_t d = Q.first[c]; d < (uint32_t)Q.first[c] + Q.mu[c]; ++d)
                z ^= gf64_mul(sm_draw(Q.key_g, (uint64_t)s * 32u + d), sm_draw(Q.key_o, (uint64_t)d * 32u + lane));
        }
    }
    const uint32_t set = __ballot_sync(0xffffffffu, z != 0);
    if (!set) {  // x_s is zero at every point
        if (lane == 0) Q.dead = 1;
        return;
    }
    const uint32_t p = (uint32_t)__ffs((int)set) - 1u;
    const uint64_t d0 = __shfl_sync(0xffffffffu, (unsigned long long)z, (int)p);
    const uint64_t rho = gf64_mul(z, gf64_inverse(d0));
    if (lane < k && lane != p) Q.rho[lane - (lane > p ? 1u : 0u)] = rho;
    if (lane == 0) {
        Q.pivot = p;
        Q.d0 = d0;
    }
}

// The scratch pointers of a template, from offsets + 1 to addresses.
__device__ __forceinline__ void relocate(XTmpl &t, uint8_t *base)
{
    const uint64_t b = reinterpret_cast<uint64_t>(base) - 1u;
    auto fix = [b](auto &p) {
        if (p) p = reinterpret_cast<std::remove_reference_t<decltype(p)>>(reinterpret_cast<uint64_t>(p) + b);
    };
    for (uint32_t i = threadIdx.x; i < t.nll; i += blockDim.x) {
        XLL &x = t.ll[i];
        fix(x.A);
        fix(x.N);
        fix(x.rank);
        fix(x.tsum);
        fix(x.meta);
        fix(x.mhead);
        fix(x.mtime);
        fix(x.R);
        fix(x.U);
        fix(x.sup);
        fix(x.IP);
        fix(x.Ec);
    }
    if (threadIdx.x == 0) {
        fix(t.clear);
        fix(t.cnt);
        fix(t.shape);
        fix(t.span);
        fix(t.omega);
    }
}

__device__ __forceinline__ void copy_words(void *dst, const void *src, uint32_t bytes)
{
    for (uint32_t i = threadIdx.x; i < bytes / 4; i += blockDim.x)
        static_cast<uint32_t *>(dst)[i] = static_cast<const uint32_t *>(src)[i];
}
// From the parameter bank: it serves one address per warp at a time, so a warp
// reads 32 words with the same index on all lanes and every lane keeps its own.
__device__ __forceinline__ void copy_params(void *dst, const void *src, uint32_t bytes)
{
    const uint32_t lane = threadIdx.x & 31u;
    for (uint32_t w = threadIdx.x & ~31u; w < bytes / 4; w += blockDim.x) {
        uint32_t mine = 0;
#pragma unroll
        for (uint32_t i = 0; i < 32; ++i) {
            const uint32_t x = w + i < bytes / 4 ? static_cast<const uint32_t *>(src)[w + i] : 0u;
            if (lane == i) mine = x;
        }
        if (w + lane < bytes / 4) static_cast<uint32_t *>(dst)[w + lane] = mine;
    }
}

// The description of one query, in shared memory (it is read all the time at
// run-time indexes; indexed reads of the parameter bank took a microsecond a
// phase).
template <bool BATCH>
__device__ __forceinline__ void load_query(XOne &o, const XArgs &a, const XOne &one, uint32_t q, uint32_t lane)
{
    __syncthreads();
    if (BATCH) copy_words(&o.q, a.xq + q, sizeof(XQuery));
    else copy_params(&o.q, &one.q, sizeof(XQuery));
    __syncthreads();
    if (BATCH) copy_words(&o.t, a.xt + o.q.k, sizeof(XTmpl));
    else copy_params(&o.t, &one.t, sizeof(XTmpl));
    __syncthreads();
    relocate(o.t, a.scratch + lane * a.stride);
    __syncthreads();
}

// First: every query in one block's shared memory (x_tiny). Those that do not
// fit are left to the bitmap passes: one query at a time by the whole grid, or,
// when there are many, one per block.
// WIDE: the passes with summaries (x_plan).
template <bool BATCH, bool WIDE>
__global__ void __launch_bounds__(kThreads, 1)
k_frontier(const __grid_constant__ XArgs a_, const __grid_constant__ XOne one_, uint32_t plan, uint32_t lbeg, uint32_t lend,
           uint32_t fin)
{
    __shared__ __align__(16) XArgs a;
    __shared__ __align__(16) XOne o;
    __shared__ uint32_t next;
    __shared__ Meetings meet;
    copy_params(&a, &a_, sizeof(XArgs));
    __syncthreads();
    if (threadIdx.x == 0) meet = Meetings{};
    View grid{blockIdx.x, gridDim.x, a.ctl, a.err, &meet, a.limit};
    auto absent = [&](uint32_t at) { return a.absent == at && blockIdx.x == gridDim.x - 1u; };
    bool ok = !absent(1);
    // cleared first: witnesses and bitmaps (a single query's first block goes on
    // with the query)
    const uint32_t skip = !BATCH && a.tiny && gridDim.x > 1 ? 1u : 0u;
    if (BATCH)
        for (uint32_t q = blockIdx.x + (threadIdx.x >> 5) * gridDim.x; q < a.nq; q += kWarps * gridDim.x) x_constants(a.xq[q], a.color);
    if (plan && blockIdx.x >= skip) {
        const uint32_t gt = (blockIdx.x - skip) * blockDim.x + threadIdx.x, nt = (gridDim.x - skip) * blockDim.x;
        if ((reinterpret_cast<uint64_t>(a.szero) & 15u) == 0) {
            ulonglong2 *z = reinterpret_cast<ulonglong2 *>(a.szero);
            for (uint64_t i = gt; i < a.szero_n / 2; i += nt) z[i] = make_ulonglong2(0, 0);
            if (gt == 0 && (a.szero_n & 1)) a.szero[a.szero_n - 1] = 0;
        } else {
            for (uint64_t i = gt; i < a.szero_n; i += nt) a.szero[i] = 0;
        }
        for (uint64_t i = gt; i < a.bzero_n; i += nt) a.bzero[i] = 0;
    }
    uint32_t left = BATCH ? 0u : 1u;
    if (plan && a.tiny && ok) {
        grid.arrive();
        bool cleared = false;
        if (BATCH) {
            ok = cleared = grid.wait();  // the queries' constants are any block's
            while (ok) {
                __syncthreads();
                if (threadIdx.x == 0) next = atomicAdd(a.ctl + 2, 1u);
                __syncthreads();
                const uint32_t q = next;
                if (q >= a.nq) break;
                copy_words(&o.q, a.xq + q, sizeof(XQuery));
                __syncthreads();
                const int r = x_tiny(a, o.q, false, grid, cleared);
                ok = r != kTinyFailed;
                if (threadIdx.x == 0) {
                    if (r == kTinyNoFit) a.left[atomicAdd(a.ctl + 3, 1u)] = q;
                    else if (r == kTinyDone) a.xq[q].done = 1;
                }
            }
            ok = ok && !absent(2) && grid.sync();
            if (ok) left = *(volatile uint32_t *)(a.ctl + 3);
        } else if (blockIdx.x == 0) {
            copy_params(&o.q, &one_.q, sizeof(XQuery));
            __syncthreads();
            if (a.skip) {  // called off: no walks (an exit at the kernel's start cost every query 0.5 %)
                if (threadIdx.x == 0 && *a.skip) o.q.dead = 1;
                __syncthreads();
            }
            const int r = x_tiny(a, o.q, one_.t.every, grid, cleared);
            ok = r != kTinyFailed;
            left = r == kTinyNoFit ? 1u : 0u;
            grid.arrive(left != 0);  // done: the others leave, and so does this block
            if (left) ok = grid.wait();
        } else {
            grid.arrive();
            ok = grid.wait();
            left = grid.some ? 1u : 0u;
        }
    }
    if (!BATCH && ok && left) load_query<BATCH>(o, a, one_, 0, 0);
    if (ok && left) {
        if (BATCH && a.lanes > 1 && left >= gridDim.x / 4) {
            View solo{0u, 1u, a.ctl, a.err, &meet, a.limit};
            while (blockIdx.x < a.lanes) {
                __syncthreads();
                if (threadIdx.x == 0) next = atomicAdd(a.ctl + 4, 1u);
                __syncthreads();
                if (next >= left) break;
                load_query<BATCH>(o, a, one_, a.left[next], blockIdx.x);
                x_plan<WIDE>(a, o, solo);
                x_wedge(a, o, solo, 1u, o.t.maxlev, true);
                x_outputs(a, o, solo);
                if (threadIdx.x == 0) a.xq[a.left[next]].done = 1;
            }
        } else {
            for (uint32_t i = 0; i < left && ok; ++i) {
                if (BATCH) load_query<BATCH>(o, a, one_, a.left[i], 0);
                if (plan) ok = x_plan<WIDE>(a, o, grid);
                const uint32_t l1 = BATCH ? o.t.maxlev : lend;
                if (ok && l1) ok = x_wedge(a, o, grid, BATCH ? 1u : lbeg, l1, fin != 0);
                if (ok && fin) x_outputs(a, o, grid);
                if (BATCH && ok) ok = grid.sync();  // the scratch is the next query's
                if (BATCH && ok && blockIdx.x == 0 && threadIdx.x == 0) a.xq[a.left[i]].done = 1;
            }
        }
    }
    // the last block to leave marks a failed batch's unfinished queries, and clears
    // the counters for the next launch
    __syncthreads();
    if (threadIdx.x == 0) {
        if (!ok) __threadfence();  // (wait() has set err)
        if (atomicAdd(a.ctl + 1, 1u) == gridDim.x - 1) {
            if (BATCH && a.status) {
                if (*(volatile uint32_t *)a.err) {
                    __threadfence();
                    for (uint32_t q = 0; q < a.nq; ++q)
                        if (!*(volatile uint32_t *)&a.xq[q].done) a.status[a.xq[q].index] = (int32_t)RR_ETIMEDOUT;
                }
                a.ctl[5] = 0;
            }
            for (int i = 0; i < 5; ++i) a.ctl[i] = 0;
            a.ctl[32] = 0;
        }
    }
}

// The record of every edge in (tail, time) order: head, time, input index, and
// the range of edges that may follow it (they leave the head no earlier and at
// most its waiting time later).
__global__ void k_out_records(uint32_t m, const uint32_t *__restrict__ off, const uint32_t *__restrict__ time,
                              const uint32_t *__restrict__ dst, const uint32_t *__restrict__ eid,
                              const uint32_t *__restrict__ delta, uint4 *__restrict__ rec, uint32_t *__restrict__ len)
{
    for (uint32_t o = blockIdx.x * blockDim.x + threadIdx.x; o < m; o += gridDim.x * blockDim.x) {
        const uint32_t v = dst[o], t = time[o];
        const uint64_t until = (uint64_t)t + delta[v];
        uint32_t lo = off[v];
        const uint32_t end = off[v + 1];
        for (uint32_t hi = end; lo < hi;) {
            const uint32_t mid = lo + (hi - lo) / 2;
            if (time[mid] < t) lo = mid + 1;
            else hi = mid;
        }
        uint32_t e = lo;
        for (uint32_t hi = end; e < hi;) {
            const uint32_t mid = e + (hi - e) / 2;
            if (time[mid] <= until) e = mid + 1;
            else hi = mid;
        }
        rec[o] = make_uint4(v, t, eid[o], lo);
        len[o] = e - lo;
    }
}

// start[i] = first position of entry i's window in the list before (0-based):
// its index b when set, else the first row of the tail's segment there (the
// rows with smaller heads come before it); and the longest window. A row of
// blocks per list.
struct WindowList {
    uint32_t count, prev_count;
    const uint32_t *a, *b, *src, *prev_head;
    uint32_t *start;
};
struct WindowLists {
    WindowList l[6];
    uint32_t *longest;  // per list
};
__global__ void k_window_start(const __grid_constant__ WindowLists lists)
{
    const WindowList &L = lists.l[blockIdx.y];
    uint32_t most = 0;
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < L.count; i += gridDim.x * blockDim.x) {
        uint32_t s = L.b[i];
        if (!s && L.a[i]) {
            const uint32_t u = L.src[i];
            uint32_t lo = 0, hi = L.prev_count;
            while (lo < hi) {
                const uint32_t mid = lo + (hi - lo) / 2;
                if (L.prev_head[mid] < u) lo = mid + 1;
                else hi = mid;
            }
            s = lo;
        }
        L.start[i] = s;
        if (L.a[i] > s) most = max(most, L.a[i] - s);
    }
    most = __reduce_max_sync(0xffffffffu, most);
    if ((threadIdx.x & 31u) == 0 && most) atomicMax(lists.longest + blockIdx.y, most);
}

}  // namespace

rr_status frontier_out_reserve(Graph &g)
{
    // (with the packed subset tables behind them; both buffers of a small graph
    // stay below 1 MiB, where an allocation needs no mapping of its own: 120 us)
    const uint64_t m = std::max<uint64_t>(1, g.m);
    RR_CUDA(g.o_buf.reserve(m * (sizeof(uint4) + 4) + ((uint64_t)g.n + 1 + x_packed_off(kPackedLabels + 1)) * 4));
    RR_CUDA(g.x_tab.reserve((size_t)x_tab_off(kXMaxLabels + 1) * 4));
    g.o_rec = g.o_buf.as<uint4>();
    g.o_len = reinterpret_cast<uint32_t *>(g.o_rec + m);
    g.o_off = g.o_len + m;
    g.x_packed = g.o_off + g.n + 1;
    return RR_OK;
}

rr_status frontier_out_records(Graph &g, const uint32_t *d_time, const uint32_t *d_dst, const uint32_t *d_eid,
                               const uint32_t *d_delta, cudaStream_t st)
{
    const unsigned grid = (unsigned)std::min<uint64_t>(152ull * 64, (g.m + 255) / 256);
    k_out_records<<<grid, 256, 0, st>>>((uint32_t)g.m, g.o_off, d_time, d_dst, d_eid, d_delta, g.o_rec, g.o_len);
    RR_LAUNCHED();
    return RR_OK;
}

// ---- host side ------------------------------------------------------------------

rr_status frontier_load(Graph &g, cudaStream_t st)
{
    RR_CUDA(cudaDeviceGetAttribute(&g.x_sms, cudaDevAttrMultiProcessorCount, g.dev));
    int smem = 0;
    RR_CUDA(cudaDeviceGetAttribute(&smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, g.dev));
    g.x_smem_max = (uint32_t)smem;
    const void *const kernels[] = {(const void *)k_frontier<false, false>, (const void *)k_frontier<true, false>,
                                   (const void *)k_frontier<false, true>, (const void *)k_frontier<true, true>};
    for (const void *f : kernels) {
        cudaFuncAttributes at{};
        RR_CUDA(cudaFuncGetAttributes(&at, f));
        g.x_smem_max = std::min<uint32_t>(g.x_smem_max, (uint32_t)(smem - (int)at.sharedSizeBytes));
    }
    g.x_smem_max = g.x_smem_max / 64 * 64;
    for (const void *f : kernels) RR_CUDA(cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)g.x_smem_max));
    // blocks that wait on one another need a cooperative launch with a block on
    // every SM; where that is not to be had, queries run over sieve points
    int coop = 0;
    RR_CUDA(cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, g.dev));
    for (const void *f : kernels) {
        int per = 0;
        RR_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, f, kThreads, g.x_smem_max));
        if (!coop || per < 1) g.x_sms = 0;
    }
    if (!g.x_sms) return RR_OK;
    k_subset_table<<<dim3((x_binom(kXMaxLabels, kXMaxLabels / 2) + 127) / 128, kXMaxLabels), 128, 0, st>>>(g.x_tab.as<uint32_t>());
    RR_LAUNCHED();
    k_packed_table<<<dim3(8, kPackedLabels), 128, 0, st>>>(g.x_tab.as<uint32_t>(), g.x_packed);
    RR_LAUNCHED();
    struct {
        RowList *L, *prev;
        DevBuf *a, *b;
        uint32_t **start;
    } w[] = {{&g.state_list, &g.prod_list, &g.state_list.a0, &g.state_list.b0, &g.state_list.w0},
             {&g.win_list, &g.prod_list, &g.win_list.a0, &g.win_list.b0, &g.win_list.w0},
             {&g.deep_list, &g.state_list, &g.deep_list.a1, &g.deep_list.b1, &g.deep_list.w1},
             {&g.tail_list, &g.state_list, &g.tail_list.a1, &g.tail_list.b1, &g.tail_list.w1},
             {&g.deep_list, &g.deep_list, &g.deep_list.a3, &g.deep_list.b3, &g.deep_list.w3},
             {&g.tail3_list, &g.deep_list, &g.tail3_list.a3, &g.tail3_list.b3, &g.tail3_list.w3}};
    uint64_t total = 0, most = 0;
    for (auto &x : w) {
        total += (x.L->count + 63u) / 64u * 64u;  // each on a 256-byte boundary
        most = std::max<uint64_t>(most, x.L->count);
    }
    if (!most) return RR_OK;
    RR_CUDA(g.x_win.reserve((total + std::size(w)) * 4));
    uint32_t *at = g.x_win.as<uint32_t>();
    WindowLists lists{};
    lists.longest = at + total;
    RR_CUDA(cudaMemsetAsync(lists.longest, 0, sizeof g.x_longest, st));
    for (size_t i = 0; i < std::size(w); ++i) {
        auto &x = w[i];
        *x.start = at;
        at += (x.L->count + 63u) / 64u * 64u;
        lists.l[i] = WindowList{(uint32_t)x.L->count, (uint32_t)x.prev->count, x.a->as<uint32_t>(), x.b->as<uint32_t>(),
                                x.L->src.as<uint32_t>(), x.prev->head.as<uint32_t>(), *x.start};
    }
    k_window_start<<<dim3((unsigned)std::min<uint64_t>(152ull * 32, (most + 255) / 256), (unsigned)std::size(w)), 256, 0, st>>>(lists);
    RR_LAUNCHED();
    // (the load waits for the stream at its end)
    RR_CUDA(cudaMemcpyAsync(g.x_longest, lists.longest, sizeof g.x_longest, cudaMemcpyDeviceToHost, st));
    return RR_OK;
}

static void x_lists(const Graph &g, XList *out)
{
    auto set = [&](uint32_t id, const RowList &L, const uint32_t *lo, const DevBuf &hi) {
        out[id] = XList{L.head.as<uint32_t>(), L.eid.as<uint32_t>(), L.src.as<uint32_t>(), lo,
                        hi.as<uint32_t>(), L.time.as<uint32_t>(), (uint32_t)L.count, (uint32_t)(L.count / 32 + 1)};
    };
    set(kXProd, g.prod_list, g.prod_list.w0, g.prod_list.a0);
    set(kXState, g.state_list, g.state_list.w0, g.state_list.a0);
    set(kXDeep1, g.deep_list, g.deep_list.w1, g.deep_list.a1);
    set(kXDeep3, g.deep_list, g.deep_list.w3, g.deep_list.a3);
    set(kXWin, g.win_list, g.win_list.w0, g.win_list.a0);
    set(kXTail, g.tail_list, g.tail_list.w1, g.tail_list.a1);
    set(kXTail3, g.tail3_list, g.tail3_list.w3, g.tail3_list.a3);
    out[kXAll] = XList{g.row_head.as<uint32_t>(), g.row_eid.as<uint32_t>(), g.row_src.as<uint32_t>(), nullptr, nullptr,
                       g.row_t.as<uint32_t>(), (uint32_t)g.m, (uint32_t)(g.m / 32 + 1)};
}

// Bump allocation of the scratch: offsets + 1 in place of addresses.
struct XBump {
    uint64_t used = 0;
    template <class T>
    T *take(uint64_t count)
    {
        T *p = reinterpret_cast<T *>(used + 1);
        used += (count * sizeof(T) + 255) / 256 * 256;
        return p;
    }
};

static uint32_t x_store_list(uint32_t l)
{
    return l == 1 ? kXProd : l == 2 ? kXState : l == 3 ? kXDeep1 : kXDeep3;
}
static uint32_t x_out_list(uint32_t l)
{
    return l == 1 ? kXAll : l == 2 ? kXWin : l == 3 ? kXTail : kXTail3;
}

// The levels of a k-vertex query, the store level first: store levels 1..k-2, an
// out level k-1 (every = false) or out levels 1..k-1 (every = true: at-most-k),
// and their scratch. multi: a set of sources, all k labels, subsets larger by
// one. Returns the scratch's bytes.
static uint64_t x_template(const Graph &g, const XList *lists, uint32_t k, bool every, bool multi, bool arrivals, XTmpl &t)
{
    std::memset(&t, 0, sizeof t);
    // (by list: x_longest is in the order of frontier_load's windows)
    const uint32_t *const w = g.x_longest, longest[kXLists] = {0, w[0], w[2], w[4], w[1], w[3], w[5], 0};
    const uint32_t sh = multi ? 1u : 0u, K = k - 1 + sh;
    t.maxlev = k - 1;
    t.every = every ? 1u : 0u;
    uint32_t store[kXMaxLevels + 1] = {0};
    for (uint32_t l = 1; l <= k - 1; ++l) {
        t.runs[l].first = t.nll;
        for (int out = 0; out < 2; ++out) {
            if (out ? !(every || l == k - 1) : l > k - 2) continue;
            XLL &x = t.ll[t.nll];
            x.level = l;
            x.out = (uint32_t)out;
            x.list = out ? x_out_list(l) : x_store_list(l);
            x.words = lists[x.list].words;
            x.d = l - 1 + sh;
            x.prev = l > 1 ? store[l - 1] : t.nll;
            if (out) {
                x.cout = l + sh;  // labels of k' = l + 1
                x.row = every ? l - 1 : 0u;
            } else {
                x.cin = l >= 2 ? x_binom(K, x.d - 1) : 0u;
                x.cout = x_binom(K, x.d);
                x.uout = every || l == k - 2 ? x.d + 2 : 0u;  // the out level above uses d + 2 labels
                store[l] = t.nll;
            }
            ++t.nll;
        }
        t.runs[l].count = t.nll - t.runs[l].first;
    }
    XBump b;
    t.clear = b.take<uint4>(0);
    if (!every)
        for (uint32_t i = 0; i < t.nll; ++i)
            if (!t.ll[i].out) t.ll[i].N = b.take<uint32_t>(t.ll[i].words);
    for (uint32_t i = 0; i < t.nll; ++i) {  // levels read by long windows
        const XLL &x = t.ll[i];
        XLL &p = t.ll[x.prev];
        if (x.level < 2 || longest[x.list] <= kWideWords * 32u || p.sums) continue;
        p.sums = (uint32_t)(b.used / 256 + 1);
        b.take<uint32_t>((uint64_t)x_sum_words(p.words) * (every ? 1 : 2));
    }
    t.clear4 = (uint32_t)(b.used / 16);
    uint64_t ping[2] = {0, 0}, ipw[2] = {0, 0}, supw = 0;
    for (uint32_t i = 0; i < t.nll; ++i) {
        const XLL &x = t.ll[i];
        if (x.out) continue;
        const uint64_t c = lists[x.list].count, w = x.cout + x.uout;
        if (x.level >= 3) {
            ping[x.level & 1u] = std::max<uint64_t>(ping[x.level & 1u], c * w);
            ipw[x.level & 1u] = std::max<uint64_t>(ipw[x.level & 1u], (c / 4 + 1) * w);
        }
        supw = std::max<uint64_t>(supw, (uint64_t)x_sup_rows(c) * w);
    }
    uint64_t *pp[2] = {b.take<uint64_t>(ping[0]), b.take<uint64_t>(ping[1])};
    uint64_t *ip[2] = {b.take<uint64_t>(ipw[0]), b.take<uint64_t>(ipw[1])};
    uint64_t *sup[3] = {b.take<uint64_t>(supw), b.take<uint64_t>(supw), b.take<uint64_t>(supw)};
    for (uint32_t i = 0; i < t.nll; ++i) {
        XLL &x = t.ll[i];
        const uint64_t c = lists[x.list].count;
        x.A = b.take<uint32_t>(x.words);
        if (x.out || every) x.N = x.A;
        x.rank = b.take<uint2>(x.words);
        x.tsum = b.take<uint32_t>(256);
        x.meta = b.take<uint4>(c);
        if (x.out || x.uout) x.mhead = b.take<uint32_t>(c);
        if (x.out && arrivals) {
            x.mtime = b.take<uint32_t>(c);
            x.Ec = b.take<uint64_t>(c);
        }
        if (!x.out) {
            const bool up = x.level + 1 <= k - 2;  // a store level above reads R
            x.R = x.level >= 3 ? pp[x.level & 1u] : b.take<uint64_t>(c * (x.cout + x.uout));
            if (x.uout) x.U = x.R + c * x.cout;
            if (!up) x.R = nullptr;
            x.ipcap = (uint32_t)(c / 4 + 1);  // blocks IP holds (four rows or more a block)
            x.IP = x.level >= 3 ? ip[x.level & 1u] : b.take<uint64_t>((uint64_t)x.ipcap * (x.cout + x.uout));
            x.sup = sup[x.level % 3];
        }
    }
    t.omega = b.take<uint64_t>((uint64_t)k * k);
    t.cnt = b.take<uint32_t>(t.nll);
    t.shape = b.take<uint32_t>(t.nll);
    t.span = b.take<unsigned long long>(t.nll);
    return b.used;
}

// Whether some level has summaries.
static bool x_wide(const XTmpl &t)
{
    return std::any_of(t.ll, t.ll + t.nll, [](const XLL &x) { return x.sums != 0; });
}

static void x_args(const Graph &g, XArgs &a)
{
    x_lists(g, a.lists);
    a.n = g.n;
    a.color = g.color.as<uint8_t>();
    a.tab = g.x_tab.as<uint32_t>();
    a.packed = g.x_packed;
    a.ooff = g.o_off;
    a.orec = g.o_rec;
    a.olen = g.o_len;
    a.smem = g.x_smem_max / 16u * 16u;
}

// Products with one factor: its 16 multiples by polynomials of degree < 4, and
// the other factor four bits at a time.
struct GfTimes {
    uint64_t t[16];
    explicit GfTimes(uint64_t a)
    {
        t[0] = 0;
        t[1] = a;
        for (int i = 2; i < 16; ++i) t[i] = i & 1 ? t[i - 1] ^ a : shl(t[i / 2], 1);
    }
    static uint64_t shl(uint64_t v, int n)  // v x^n, n <= 4
    {
        return gf64_reduce(v >> (64 - n), v << n);
    }
    uint64_t operator()(uint64_t b) const
    {
        uint64_t r = t[b >> 60];
        for (int s = 56; s >= 0; s -= 4) r = shl(r, 4) ^ t[(b >> s) & 15u];
        return r;
    }
};

// constants: with what depends on the source's z row.
static void x_query(const Graph &g, const rr_query &q, bool multi, bool constants, XQuery &X)
{
    std::memset(&X, 0, sizeof X);
    const QueryKeys keys = make_keys(q.seed);
    const uint32_t k = q.k, s = q.source;
    X.source = s;
    X.k = k;
    X.K = k - 1;
    X.colored = q.motif ? 1u : 0u;
    X.key_y = keys.key_y;
    X.key_z = keys.key_z;
    X.key_g = keys.key_gamma;
    X.key_o = keys.key_omega;
    uint64_t zs[kXMaxLabels + 1];
    constants = constants && !multi;
    if (multi) {
        X.multi = 1;
        X.K = X.pivot = k;
    }
    if (q.motif) {
        ShadeTable sh;
        make_shades(q.motif, k, &sh);
        for (int c = 0; c < 256; ++c) {
            X.first[c] = (uint8_t)sh.first[c];
            X.mu[c] = (uint8_t)sh.mu[c];
        }
        if (!constants) return;
        const uint32_t c = g.h_color[s];
        for (uint32_t j = 0; j < k; ++j) {
            zs[j] = 0;
            for (uint32_t d = sh.first[c]; d < sh.first[c] + sh.mu[c]; ++d)
                zs[j] ^= gf64_mul(sm_draw(X.key_g, (uint64_t)s * 32u + d), sm_draw(X.key_o, (uint64_t)d * 32u + j));
        }
    } else {
        if (!constants) return;
        for (uint32_t j = 0; j < k; ++j) zs[j] = sm_draw(X.key_z, (uint64_t)s * 32u + j);
    }
    uint32_t p = 0;
    while (p < k && !zs[p]) ++p;
    if (p == k) {  // x_s is zero at every point
        X.dead = 1;
        return;
    }
    X.pivot = p;
    X.d0 = zs[p];
    const GfTimes by_inverse(gf64_inverse(zs[p]));
    for (uint32_t j = 0, t = 0; j < k; ++j)
        if (j != p) X.rho[t++] = by_inverse(zs[j]);
}

bool uses_frontier(const Graph &g, uint32_t k)
{
    return g.x_sms && g.compact && !g.point_flags && k >= 2 && k - 1 <= kXMaxLabels && !g.tune_forced[k];
}

uint64_t frontier_bytes(const Graph &g, uint32_t k, bool every, bool multi, bool arrivals)
{
    XList lists[kXLists];
    x_lists(g, lists);
    XTmpl t;
    return x_template(g, lists, k, every, multi, arrivals, t);
}

bool frontier_fits(const Graph &g, Workspace &ws, uint32_t k, uint64_t budget, bool every, bool multi, bool arrivals,
                   rr_status *st)
{
    *st = RR_OK;
    // a set of sources keeps all k labels, at-most-k answers every smaller k too
    if (!uses_frontier(g, k) || (multi && k > kXMaxLabels)) return false;
    for (uint32_t kk = 2; every && kk < k; ++kk)
        if (!uses_frontier(g, kk)) return false;
    const uint64_t need = frontier_bytes(g, k, every, multi, arrivals);
    if (need > g.x_scratch_max) return false;
    if (need > ws.state.bytes && budget == 0) {
        size_t free_b = 0, total_b = 0;
        if (cudaMemGetInfo(&free_b, &total_b) != cudaSuccess) return false;
        budget = (uint64_t)(0.6 * (double)(free_b + ws.state.bytes));
    }
    if (need > ws.state.bytes && need > budget) return false;
    const cudaError_t e = ws.state.reserve(need);
    if (e == cudaErrorMemoryAllocation) {  // (not in one piece, or taken meanwhile: the sieve points need less)
        (void)cudaGetLastError();
        return false;
    }
    if (e != cudaSuccess) *st = cuda_fail(e, "cudaMalloc (query scratch)", __FILE__, __LINE__);
    return true;
}

template <bool BATCH, bool WIDE>
static rr_status x_launch(const Graph &g, const XArgs &a, const XOne &one, cudaStream_t st)
{
    cudaLaunchAttribute at[1];
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)g.x_sms);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = a.smem;
    cfg.stream = st;
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    if (BATCH || a.tiny) {
        const int ts = timing_begin(st);
        RR_CUDA(cudaLaunchKernelEx(&cfg, k_frontier<BATCH, WIDE>, a, one, 1u, 1u, one.t.maxlev, 1u));
        timing_end(ts, kTimeBatch, st);
        RR_LAUNCHED();
        return RR_OK;
    }
    // kernel timing: one launch for the passes over the bitmaps and one per
    // layer, each timed
    for (uint32_t l = 0; l <= one.t.maxlev; ++l) {
        const int ts = timing_begin(st);
        RR_CUDA(cudaLaunchKernelEx(&cfg, k_frontier<BATCH, WIDE>, a, one, l ? 0u : 1u, l, l, l == one.t.maxlev ? 1u : 0u));
        timing_end(ts, l == one.t.maxlev ? kTimeLast : l <= 1 ? kTimeFirst : l == 2 ? kTimeSecond : l == 3 ? kTimeThird : kTimeMid, st);
        RR_LAUNCHED();
    }
    return RR_OK;
}

rr_status frontier_reserve(Workspace &ws, cudaStream_t st)
{
    if (!ws.x_bar.p) {
        RR_CUDA(ws.x_bar.reserve(256));
        RR_CUDA(cudaMemsetAsync(ws.x_bar.p, 0, 256, st));
    }
    if (!ws.x_err) {
        RR_CUDA(cudaHostAlloc(&ws.x_err, 64, cudaHostAllocMapped));
        *ws.x_err = 0;
    }
    return RR_OK;
}

rr_status frontier_error(Workspace &ws)
{
    if (!ws.x_err || !*(volatile uint32_t *)ws.x_err) return RR_OK;
    *ws.x_err = 0;
    return fail(RR_ETIMEDOUT, "a bounded wait of the query's kernel expired");
}

rr_status frontier_error(const Graph &g)
{
    rr_status s = frontier_error(g.ws);
    for (const auto &w : g.fan.ws)  // (every flag, so that a call is reported once)
        if (const rr_status f = frontier_error(*w); f != RR_OK) s = f;
    return s;
}

// report: an earlier call's expired wait is this call's to report.
static rr_status x_control(const Graph &g, Workspace &ws, cudaStream_t st, bool report, XArgs &a)
{
    a.limit = g.x_wait_ns;
    a.absent = g.x_absent;
    rr_status s = frontier_reserve(ws, st);
    if (s == RR_OK && report) s = &ws == &g.ws ? frontier_error(g) : frontier_error(ws);
    if (s != RR_OK) return s;
    a.ctl = ws.x_bar.as<uint32_t>();
    uint32_t *d = nullptr;
    RR_CUDA(cudaHostGetDevicePointer(&d, ws.x_err, 0));
    a.err = d;
    return RR_OK;
}

// Results to pinned host buffers: witness words and bitmap bytes in one launch
// where the copy engine takes two transfers, each started after the one before
// (rr_reach_sync, k = 6, n = 24,000: 71 -> 64 us; n = 1e6, 8 MB: 112 -> 106 us, the
// largest tried: longer ones stay with the copy engine).
constexpr uint64_t kCopyOutMax = 8ull << 20;
__global__ void __launch_bounds__(256) k_copy_out(const uint64_t *__restrict__ w, uint64_t *__restrict__ hw, uint64_t n,
                                                  const uint8_t *__restrict__ b, uint8_t *__restrict__ hb, uint64_t nb)
{
    const uint64_t t = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x, step = (uint64_t)gridDim.x * blockDim.x;
    if (hw) {
        if ((reinterpret_cast<uint64_t>(hw) & 15u) == 0) {
            const ulonglong2 *const s2 = reinterpret_cast<const ulonglong2 *>(w);
            ulonglong2 *const d2 = reinterpret_cast<ulonglong2 *>(hw);
            for (uint64_t i = t; i < n / 2; i += step) d2[i] = s2[i];
            if (t == 0 && (n & 1)) hw[n - 1] = w[n - 1];
        } else {
            for (uint64_t i = t; i < n; i += step) hw[i] = w[i];
        }
    }
    if (hb) {
        if ((reinterpret_cast<uint64_t>(hb) & 15u) == 0) {
            const uint4 *const s4 = reinterpret_cast<const uint4 *>(b);
            uint4 *const d4 = reinterpret_cast<uint4 *>(hb);
            for (uint64_t i = t; i < nb / 16; i += step) d4[i] = s4[i];
            for (uint64_t i = nb / 16 * 16 + t; i < nb; i += step) hb[i] = b[i];
        } else {
            for (uint64_t i = t; i < nb; i += step) hb[i] = b[i];
        }
    }
}

// The device address of `count` values in pinned host memory, or null: also where
// their last byte is not pinned with the first (a registered range that ends inside
// the caller's buffer) or they are not aligned as the kernel stores them. Those are
// for the copy engine, whose checks are the runtime's.
template <class T>
static T *pinned(T *p, uint64_t count)
{
    if (!p || !count || reinterpret_cast<uintptr_t>(p) % sizeof(T)) return nullptr;
    const void *const ends[2] = {p, reinterpret_cast<const uint8_t *>(p + count) - 1};
    void *dev[2] = {nullptr, nullptr};
    for (int i = 0; i < 2; ++i) {
        cudaPointerAttributes at{};
        if (cudaPointerGetAttributes(&at, ends[i]) != cudaSuccess) {
            cudaGetLastError();
            return nullptr;
        }
        if (at.type != cudaMemoryTypeHost || !at.devicePointer) return nullptr;
        dev[i] = at.devicePointer;
    }
    if (static_cast<uint8_t *>(dev[1]) - static_cast<uint8_t *>(dev[0]) != (ptrdiff_t)(count * sizeof(T) - 1)) return nullptr;
    return static_cast<T *>(dev[0]);
}

rr_status copy_out(const uint64_t *d_w, uint64_t *h_w, uint64_t n, const uint8_t *d_b, uint8_t *h_b, uint64_t nb, cudaStream_t st)
{
    uint64_t *const pw = pinned(h_w, n);
    uint8_t *const pb = pinned(h_b, nb);
    if ((h_w && !pw) || (h_b && !pb) || n * 8 > kCopyOutMax) {
        if (h_w) RR_CUDA(cudaMemcpyAsync(h_w, d_w, n * 8, cudaMemcpyDeviceToHost, st));
        if (h_b) RR_CUDA(cudaMemcpyAsync(h_b, d_b, nb, cudaMemcpyDeviceToHost, st));
        return RR_OK;
    }
    if (!pw && !pb) return RR_OK;
    k_copy_out<<<(unsigned)std::min<uint64_t>(304, (n / 2 + 255) / 256 + 1), 256, 0, st>>>(d_w, pw, n, d_b, pb, nb);
    RR_LAUNCHED();
    return RR_OK;
}

// One query on st. every: witness rows of k' = 2..k (plain queries); d_R: the
// minimum arrival times (n per witness row, set to UINT32_MAX by the caller).
// src: a set of sources. d_skip: a device word that calls the query off when set.
rr_status frontier_query(const Graph &g, Workspace &ws, const rr_query *q, bool every, uint8_t *d_bitmap,
                         uint64_t *d_witness, cudaStream_t st, uint64_t *d_E, const uint8_t *d_vmask, uint32_t *d_R,
                         const SourceSet *src, const uint32_t *d_skip)
{
    XArgs a{};
    x_args(g, a);
    rr_status s = x_control(g, ws, st, true, a);
    if (s != RR_OK) return s;
    XOne one;
    x_template(g, a.lists, q->k, every, src != nullptr, d_R != nullptr, one.t);
    x_query(g, *q, src != nullptr, true, one.q);
    XQuery &Q = one.q;
    Q.S = d_witness;
    Q.E = d_E;
    Q.R = d_R;
    Q.bitmap = d_bitmap;
    Q.vmask = d_vmask;
    if (src) {
        Q.smask = src->mask;
        Q.slist = src->list;
        Q.nslist = src->count;
    }
    a.nq = 1;
    a.skip = d_skip;
    a.scratch = ws.state.as<uint8_t>();
    a.lanes = 1;
    a.szero = d_witness;
    a.szero_n = (uint64_t)g.n * (every ? q->k - 1 : 1);
    a.bzero = d_bitmap;
    a.bzero_n = d_bitmap ? (g.n + 7) / 8 : 0;
    a.tiny = g_timing.load(std::memory_order_relaxed) ? 0u : 1u;
    return x_wide(one.t) ? x_launch<false, true>(g, a, one, st) : x_launch<false, false>(g, a, one, st);
}

// The level lists of the last single query of k vertices that took the passes on
// the graph's workspace: level, whether an out level, needed rows, rows per block,
// whether its prefix sums were completed. Synchronous.
rr_status frontier_levels(const Graph &g, uint32_t k, bool every, uint32_t *out, uint32_t *count)
{
    XList lists[kXLists];
    x_lists(g, lists);
    XTmpl t;
    if (x_template(g, lists, k, every, false, false, t) > g.ws.state.bytes) return fail(RR_EINVAL, "rr_debug_levels: no such query");
    RR_CUDA(cudaDeviceSynchronize());
    uint32_t cnt[kXMaxLL], shape[kXMaxLL];
    unsigned long long span[kXMaxLL];
    auto host = [&](auto &p, auto *h) {
        const cudaError_t e = cudaMemcpy(h, g.ws.state.as<uint8_t>() + (reinterpret_cast<uint64_t>(p) - 1u), t.nll * sizeof *h, cudaMemcpyDeviceToHost);
        p = h;
        return e;
    };
    RR_CUDA(host(t.cnt, cnt));
    RR_CUDA(host(t.shape, shape));
    RR_CUDA(host(t.span, span));
    for (uint32_t li = 0; li < t.nll; ++li, out += 5) {
        out[0] = t.ll[li].level;
        out[1] = t.ll[li].out;
        out[2] = cnt[li];
        out[3] = cnt[li] ? x_shape_of(shape[li]).rows : 0u;
        out[4] = cnt[li] && !t.ll[li].out && x_scans(t, li) ? 1u : 0u;
    }
    *count = t.nll;
    return RR_OK;
}

// A batch in one launch: the queries' descriptions go to the device with one
// copy, blocks take queries from a counter (x_tiny), and the queries that do not
// fit follow, one per block when there are many and their regions of scratch are
// small, or one at a time by the whole grid. idx: the queries of qs to run
// (the witnesses of all nq are cleared), those whose scratch does not fit `budget`
// taken out; false when none is left.
bool frontier_batch(const Graph &g, const rr_query *qs, uint32_t nq, std::vector<uint32_t> &idx, uint64_t budget,
                    uint8_t *d_bitmaps, uint64_t *d_witness, int32_t *d_status, cudaStream_t st, rr_status *ret)
{
    *ret = RR_OK;
    Workspace &ws = g.ws;
    BatchBuffers &B = g.batch;
    XArgs a{};
    x_args(g, a);
    bool used[kXMaxLabels + 2] = {false};
    for (uint32_t i : idx) used[qs[i].k] = true;
    budget = std::min(budget, g.x_scratch_max);
    auto run = [&]() -> rr_status {
        uint64_t stride = 0;
        bool wide = false, fits = true;
        std::vector<XTmpl> tm(kXMaxLabels + 2);
        for (uint32_t k = 2; k <= kXMaxLabels + 1; ++k)
            if (used[k]) {
                const uint64_t need = x_template(g, a.lists, k, false, false, false, tm[k]);  // (whole 256-byte groups)
                if (need > budget) {
                    used[k] = fits = false;
                    continue;
                }
                stride = std::max(stride, need);
                wide |= x_wide(tm[k]);
            }
        if (!fits) idx.erase(std::remove_if(idx.begin(), idx.end(), [&](uint32_t i) { return !used[qs[i].k]; }), idx.end());
        if (idx.empty()) return RR_EAGAIN;
        const uint32_t count = (uint32_t)idx.size();
        const size_t tbytes = sizeof(XTmpl) * (kXMaxLabels + 2), qbytes = sizeof(XQuery) * (size_t)count;
        // Queries one per block only where kBatchScratch holds a region for every
        // block of the grid. Larger regions belong to graphs whose queries are long
        // on one SM, and fewer of them leave SMs idle: 64 queries on n = 1e6, m = 1e7,
        // k = 6..12, took 1,322 ms from hubs on six blocks, 64 ms one after another
        // over the grid (k = 5..8, 53 blocks: 59 and 21 ms; 256 of k = 6..12 from any
        // vertex: 576 and 48 ms). On n = 2e5, m = 2e6 regions of 87 MB, k = 5..8, take
        // 5.4 ms one per block and 7.7 ms over the grid, of 226 MB 9.5 and 9.6 ms, of
        // 726 MB (35 blocks) 26.7 and 11.8 ms.
        constexpr uint64_t kBatchScratch = 24ull << 30;
        const uint64_t room = std::min<uint64_t>(budget, kBatchScratch);
        a.lanes = room / stride >= (uint64_t)g.x_sms ? std::min<uint32_t>((uint32_t)g.x_sms, count) : 1u;
        cudaError_t e = ws.state.reserve(a.lanes * stride);
        if (e == cudaErrorMemoryAllocation && a.lanes > 1) {
            (void)cudaGetLastError();
            a.lanes = 1;
            e = ws.state.reserve(stride);
        }
        if (e == cudaErrorMemoryAllocation) {
            (void)cudaGetLastError();
            return RR_EAGAIN;
        }
        RR_CUDA(e);
        // (with statuses a batch tells of itself alone: a server's tickets do not fail
        // for another call's wait)
        rr_status s = x_control(g, ws, st, !d_status, a);
        if (s != RR_OK) return s;
        RR_CUDA(B.xq.reserve(tbytes + qbytes));
        RR_CUDA(B.left.reserve((size_t)count * 4));
        s = B.stage_wait(tbytes + qbytes);
        if (s != RR_OK) return s;
        std::memcpy(B.h_stage, tm.data(), tbytes);
        XQuery *hq = reinterpret_cast<XQuery *>(B.h_stage + tbytes);
        const size_t nb = (g.n + 7) / 8;
        for (uint32_t j = 0; j < count; ++j) {
            const uint32_t i = idx[j];
            x_query(g, qs[i], false, false, hq[j]);
            hq[j].index = i;
            hq[j].S = d_witness + (size_t)i * g.n;
            hq[j].bitmap = d_bitmaps ? d_bitmaps + (size_t)i * nb : nullptr;
        }
        RR_CUDA(cudaMemcpyAsync(B.xq.p, B.h_stage, tbytes + qbytes, cudaMemcpyHostToDevice, st));
        s = B.stage_done(st);
        if (s != RR_OK) return s;
        a.xt = B.xq.as<XTmpl>();
        a.xq = reinterpret_cast<XQuery *>(B.xq.as<uint8_t>() + tbytes);
        a.left = B.left.as<uint32_t>();
        a.nq = count;
        a.scratch = ws.state.as<uint8_t>();
        a.stride = stride;
        a.szero = d_witness;
        a.szero_n = (uint64_t)g.n * nq;
        a.bzero = d_bitmaps;
        a.bzero_n = d_bitmaps ? (uint64_t)nb * nq : 0;
        a.status = d_status;
        if (d_status) a.err = a.ctl + 5;  // the caller looks at the statuses: nothing left for the next call to report
        a.tiny = 1;
        static const XOne none{};
        return wide ? x_launch<true, true>(g, a, none, st) : x_launch<true, false>(g, a, none, st);
    };
    *ret = run();
    if (*ret != RR_EAGAIN) return true;
    *ret = RR_OK;
    return false;
}

}  // namespace rr
