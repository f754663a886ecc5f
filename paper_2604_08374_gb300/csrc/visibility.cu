// visibility.cu -- visibility graph of an obstacle grid, built on the device
// (Sec. 3.1).  Two free cells see each other iff the closed segment between
// their centres meets no obstacle cell's closed square.  Nodes are the cells of
// the largest 4-connected free component, numbered in raster order (Sec. 3.2),
// so neighbour lists come out sorted and delta-encode into mostly one-byte
// LEB128 varints.
//
// Method: the angular sweep of Sec. 3.1 ("SparkSieve angular sweep": per
// source, eight octants expand outwards while a list of open gaps in
// tan-space [0, 1] loses the ranges obstacles cover), with the gaps' ends kept
// as exact integer fractions so that the result equals the pairwise rule above
// for every pair.  Pipeline: (host) main component and numbering, obstacle
// bitmaps; (device) per source, the four octants that see the cells after it in
// raster order swept into its row of a bit matrix, and the matrix joined with
// its transpose (visibility is symmetric); the bytes of every row's LEB128 list
// counted, with the degrees and range lookups; (host) prefix sum into offsets;
// (device) the lists written.  Graphs whose matrix would be too large
// (kMatrixBytes) or too empty (kMatrixView) have all eight octants of a source swept into one CTA's node
// bitmap and its list written to a stage in the order the sources finish, from
// where it is brought to its place; the ordinary load path then validates the
// stream and derives degrees.
#include <algorithm>
#include <utility>
#include <vector>

#include "runs.cuh"

namespace vga {
namespace {

constexpr int kMaxSide = 16384;

// Mean length of the row and column of free main-component cells that a node's
// cell lies in, over 256 nodes.
double mean_view(int W, int H, const std::vector<uint32_t> &cells, const std::vector<int32_t> &node_of_cell) {
    const size_t n = cells.size(), step = std::max<size_t>(n / 256, 1);
    double sum = 0.0;
    size_t count = 0;
    for (size_t v = step / 2; v < n; v += step, count++) {
        const size_t c = cells[v];
        const int x = (int)(c % (size_t)W), y = (int)(c / (size_t)W);
        int seen = 2;
        for (int k = 1; k <= x && node_of_cell[c - k] >= 0; k++) seen++;
        for (int k = 1; x + k < W && node_of_cell[c + k] >= 0; k++) seen++;
        for (int k = 1; k <= y && node_of_cell[c - (size_t)k * W] >= 0; k++) seen++;
        for (int k = 1; y + k < H && node_of_cell[c + (size_t)k * W] >= 0; k++) seen++;
        sum += 0.5 * seen;
    }
    return count ? sum / (double)count : 0.0;
}

// Largest 4-connected free component (ties: lowest raster index), numbered in
// raster order.  Returns the raster cell of every node.
std::vector<uint32_t> main_component_cells(int W, int H, const uint8_t *obst) {
    const size_t C = (size_t)W * H;
    std::vector<int32_t> label(C, -1);
    std::vector<uint32_t> queue;
    queue.reserve(C);
    int32_t best = -1, next = 0;
    size_t best_size = 0;
    for (size_t c = 0; c < C; c++) {
        if (obst[c] || label[c] >= 0) continue;
        const int32_t L = next++;
        queue.clear();
        queue.push_back((uint32_t)c);
        label[c] = L;
        for (size_t head = 0; head < queue.size(); head++) {
            const uint32_t cur = queue[head];
            const int x = (int)(cur % (uint32_t)W), y = (int)(cur / (uint32_t)W);
            const int nb[4][2] = {{x - 1, y}, {x + 1, y}, {x, y - 1}, {x, y + 1}};
            for (auto &q : nb) {
                if (q[0] < 0 || q[1] < 0 || q[0] >= W || q[1] >= H) continue;
                const size_t nc = (size_t)q[1] * W + q[0];
                if (obst[nc] || label[nc] >= 0) continue;
                label[nc] = L;
                queue.push_back((uint32_t)nc);
            }
        }
        if (queue.size() > best_size) {
            best_size = queue.size();
            best = L;
        }
    }
    std::vector<uint32_t> cells;
    cells.reserve(best_size);
    for (size_t c = 0; c < C; c++)
        if (best >= 0 && label[c] == best) cells.push_back((uint32_t)c);
    return cells;
}

// Hilbert-curve position of (x, y) in a 2^k x 2^k square (Sec. 3.2, optional
// Hilbert reordering): walk the levels from the coarsest; each level adds its
// quadrant's rank in curve order (0, 1, 2, 3 for lower-left, upper-left,
// upper-right, lower-right in the current frame) times the quadrant size, then
// maps the point into that quadrant's own frame (the lower quadrants are
// transposed, the lower-right one also mirrored).
uint64_t hilbert_position(int k, uint32_t x, uint32_t y) {
    uint64_t d = 0;
    for (int lvl = k - 1; lvl >= 0; lvl--) {
        const uint32_t half = 1u << lvl;
        const uint32_t qx = (x >> lvl) & 1u, qy = (y >> lvl) & 1u;
        const uint32_t rank = qx ? (qy ? 2u : 3u) : (qy ? 1u : 0u);
        d += (uint64_t)rank << (2 * lvl);
        x &= half - 1u;
        y &= half - 1u;
        if (!qy) {
            if (qx) {
                x = half - 1u - x;
                y = half - 1u - y;
            }
            const uint32_t t = x;
            x = y;
            y = t;
        }
    }
    return d;
}

// ---------------------------------------------------------------------------
// The sweep.  From a source s, each of the 8 octants is swept column by column
// outwards.  In octant coordinates a cell is (k, r): k >= 0 steps along the
// major axis, 0 <= r <= k + 1 along the minor one.  The closed square of an
// obstacle at (k, r) is seen from s's centre under the closed range of slopes
// (minor / major) [(2r - 1) / (2k + 1), (2r + 1) / (2k - 1)] (k >= 1), so the
// slopes in [0, 1] that no obstacle of columns 0 .. k - 1 blocks form a list of
// disjoint intervals, each end open or closed.  A target (k, r) is visible iff
// r / k lies in one of them, except that the target on the diagonal (r = k)
// is also blocked by the obstacle (k, k - 1), which its segment touches at a
// corner inside column k.  After column k's targets, each interval loses the
// slope ranges of the column's obstacles in rows a - 1 .. b + 1 (a .. b being
// the interval's target rows; no other row's range meets it); the remaining
// pieces carry on to column k + 1.  Every blocking range is at least 1/k wide,
// so at most k + 1 intervals are alive at column k + 1.
// ---------------------------------------------------------------------------

constexpr int kSweepWarps = 8;                     // one warp per octant
constexpr int kSweepThreads = kSweepWarps * 32;
constexpr int kSweepCap = 48;                      // intervals per list in shared memory
constexpr int kPad = 64;                           // margin bits (obstacles) on both sides of a line
constexpr uint32_t kNoSource = 0xffffffffu;
// Largest bit matrix of the graph (N^2 / 8 bytes: up to 370,000 nodes).  A bound on
// scratch, not where the ways cross: 365,000 cells of city take 0.22 s with it and
// 0.64 without, 501,000 would take 0.33 and 1.13.
constexpr uint64_t kMatrixBytes = 16ull << 30;
// From kMatrixNodes nodes on, the matrix is used where the nodes' mean view along
// a row or column is at least N / kMatrixView cells.  Its passes take time with
// N^2, and what it saves of the sweep grows with how far the nodes see.  Build
// with the matrix against without, ms: N = 236,000: views of 4 cells (a maze) 27.1
// and 12.5, 12 (rooms) 26.5 and 18.5, 30 30.4 and 32.9, 60 39.2 and 62.0; N = 100,000: 4
// 7.8 and 5.5, 9 8.1 and 7.8, 12 7.5 and 7.8, 30 10.5 and 15.0; N = 46,000: 5 3.3 and 3.4,
// 9 3.4 and 3.9; N = 360,000: 12 55 and 34, 30 61 and 67, 60 76 and 127.
constexpr uint32_t kMatrixNodes = 32768, kMatrixView = 10000;

// Test hooks: a smaller shared-memory list capacity sends more sources down
// the global-list retry (and makes the stage of the lists' bytes so small that
// some are swept again); a node limit selects the builder with a bitmap per CTA and, above
// it, moves the bitmap to global memory.
int g_sweep_smem_cap = kSweepCap;
uint32_t g_sweep_smem_bitmap_nodes = 0;   // 0: as many as shared memory allows

// A slope n / d (d > 0) with its end open or closed.
struct Slope {
    int n, d;
    bool open;
};

__device__ __forceinline__ int slope_cmp(const Slope &a, const Slope &b) {
    const int l = a.n * b.d, r = b.n * a.d;   // |numerators|, denominators < 2^15
    return l < r ? -1 : (l > r ? 1 : 0);
}

__device__ __forceinline__ bool interval_nonempty(const Slope &lo, const Slope &hi) {
    const int c = slope_cmp(lo, hi);
    return c < 0 || (c == 0 && !lo.open && !hi.open);
}

// Stored slopes lie in [0, 1] with denominators below 2^15 (sides <= 16384).
__device__ __forceinline__ uint32_t slope_pack(const Slope &s) {
    return (uint32_t)s.n | ((uint32_t)s.d << 15) | (s.open ? 1u << 30 : 0u);
}
__device__ __forceinline__ Slope slope_unpack(uint32_t w) {
    return Slope{(int)(w & 0x7fffu), (int)((w >> 15) & 0x7fffu), ((w >> 30) & 1u) != 0};
}

struct SweepArgs {
    const uint32_t *rowbits;   // H lines of words_r words: bit x + kPad of line y = obstacle (x, y)
    const uint32_t *colbits;   // W lines of words_c words: bit y + kPad of line x = obstacle (x, y)
    int W, H, words_r, words_c;
    const int32_t *node_of_cell;   // W * H: node id, or -1 off the main component
    const int32_t *node_of_cell_t; // the same by columns (rows kernel)
    uint32_t *matrix;              // rows kernel: a row of `pitch` words per node
    uint32_t pitch;
    const uint32_t *cells;         // n: raster cell of each node
    uint32_t n;
    const uint32_t *sources;       // the sources to sweep (nullptr: nodes 0 .. count - 1)
    uint32_t count;
    uint32_t *next;                // work counter, zero at launch
    uint64_t *row_bytes;           // kSweepCount, kSweepStage: bytes of each source's list
    const uint64_t *offsets;       // kSweepWrite: each list's first byte
    uint8_t *out;                  // the lists (kSweepWrite) or the stage (kSweepStage)
    unsigned long long *stage_used;    // kSweepStage: bytes of the stage given out, zero at launch
    uint64_t stage_cap;
    uint64_t *stage_at;            // kSweepStage: each list's first byte in the stage, or kNotStaged
    uint32_t *retry, *retry_count; // sources whose interval lists outgrew shared memory
    uint2 *glists;                 // global interval lists (cap glist_cap each, 2 per warp)
    int glist_cap;
    uint32_t *gbitmap;             // global node bitmaps, words_n per CTA (large graphs)
    uint32_t words_n;              // ceil(n / 32)
    int mask_words;                // row-mask (and staged obstacle) words per warp
    int smem_cap;                  // interval-list capacity in shared memory (<= kSweepCap)
    int *err;                      // nonzero: a visible cell off the component, or a list overflow
};

// 32 obstacle bits of a line starting at bit pos (pos >= 0, within the margins).
// Positions past a line's ends read as obstacles, like its margins.
__device__ __forceinline__ uint32_t line_bits32(const uint32_t *__restrict__ line, int lw, int pos) {
    if (pos < 0 || (pos >> 5) + 1 >= lw) return 0xffffffffu;
    const int w = pos >> 5, s = pos & 31;
    return __funnelshift_r(__ldg(line + w), __ldg(line + w + 1), s);
}

// Obstacle bits of rows r0 .. r0 + 31 of one octant column (bit j = row r0 + j).
__device__ __forceinline__ uint32_t column_bits(const uint32_t *__restrict__ line, int lw, int c0, bool neg, int r0) {
    return neg ? __brev(line_bits32(line, lw, c0 - r0 - 31)) : line_bits32(line, lw, c0 + r0);
}

__device__ __forceinline__ bool column_obst(const uint32_t *__restrict__ line, int lw, int c0, bool neg, int r) {
    const int pos = neg ? c0 - r : c0 + r;
    if (pos < 0 || (pos >> 5) >= lw) return true;
    return (__ldg(line + (pos >> 5)) >> (pos & 31)) & 1u;
}

// Rows a .. b of column k whose slopes r / k lie in [lo, hi] (b < a: none).
// Numerators are at most 2k + 3 and k < 2^14, so the products fit 32 bits.
__device__ __forceinline__ void interval_rows(const Slope &lo, const Slope &hi, int k, int &a, int &b) {
    const uint32_t nl = (uint32_t)lo.n * (uint32_t)k, nh = (uint32_t)hi.n * (uint32_t)k;
    uint32_t qa = (nl + (uint32_t)lo.d - 1u) / (uint32_t)lo.d;
    if (lo.open && qa * (uint32_t)lo.d == nl) qa++;
    const uint32_t qb = nh / (uint32_t)hi.d;
    a = (int)qa;
    b = (int)qb - ((hi.open && qb * (uint32_t)hi.d == nh) ? 1 : 0);
}

// Obstacle bits of rows y .. y + 31 of the current column from its words
// staged in shared memory (obw[w] holds rows 32w .. 32w + 31).
__device__ __forceinline__ uint32_t staged_bits(const uint32_t *obw, int y) {
    return __funnelshift_r(obw[y >> 5], obw[(y >> 5) + 1], y & 31);
}

// Appends to out (through the warp's counter) the pieces of interval
// [lo, hi] left after the obstacles of column k in rows r0 .. r1 (read from
// the column's staged words); pieces past cap are counted but not stored.
__device__ void interval_pieces(Slope lo, const Slope &hi, int k, int r0, int r1, const uint32_t *obw, uint2 *out,
                                int *count, int cap) {
    int y = r0;
    while (y <= r1) {
        const int lim = min(32, r1 - y + 1);
        const uint32_t valid = lim == 32 ? 0xffffffffu : ((1u << lim) - 1u);
        const uint32_t ob = staged_bits(obw, y) & valid;
        if (!ob) {
            y += lim;
            continue;
        }
        const int s = y + __ffs(ob) - 1;
        // the run's last obstacle row: the row before the next free one
        int e = r1;
        for (int z = s; z <= r1;) {
            const int lim2 = min(32, r1 - z + 1);
            const uint32_t valid2 = lim2 == 32 ? 0xffffffffu : ((1u << lim2) - 1u);
            const uint32_t fr = ~staged_bits(obw, z) & valid2;
            if (fr) {
                e = z + __ffs(fr) - 2;
                break;
            }
            z += lim2;
        }
        const Slope mn{2 * s - 1, 2 * k + 1, true}, mx{2 * e + 1, 2 * k - 1, true};
        const Slope phi = slope_cmp(hi, mn) < 0 ? hi : mn;
        if (interval_nonempty(lo, phi)) {
            const int at = atomicAdd(count, 1);
            if (at < cap) out[at] = make_uint2(slope_pack(lo), slope_pack(phi));
        }
        const int c2 = slope_cmp(mx, lo);
        if (c2 > 0) lo = mx;
        else if (c2 == 0) lo.open = true;
        y = e + 1;
    }
    if (interval_nonempty(lo, hi)) {
        const int at = atomicAdd(count, 1);
        if (at < cap) out[at] = make_uint2(slope_pack(lo), slope_pack(hi));
    }
}

__device__ __forceinline__ uint32_t varint_len(uint32_t x) {
    return x < (1u << 7) ? 1u : x < (1u << 14) ? 2u : x < (1u << 21) ? 3u : x < (1u << 28) ? 4u : 5u;
}

// One warp sweeps octant `oct` of source (sx, sy), setting the bits of the
// visible nodes in bm (ROWS: a row of the matrix in global memory; else the
// CTA's bitmap, with the range of ids kept in id_lo and id_hi).  Returns false
// when the interval list outgrew cap.
template <bool ROWS>
__device__ bool sweep_octant(const SweepArgs &A, int oct, int sx, int sy, uint32_t *bm, uint2 *la, uint2 *lb,
                             int cap, uint32_t *mask, uint32_t *obw, int *count, int &id_lo, int &id_hi) {
    const int lane = threadIdx.x & 31;
    const bool xmajor = (oct >> 2) == 0;
    const int smaj = (oct & 1) ? -1 : 1;
    const bool neg = (oct & 2) != 0;
    const int smin = neg ? -1 : 1;
    const int maj0 = xmajor ? sx : sy, min0 = xmajor ? sy : sx;
    const int maj_n = xmajor ? A.W : A.H;
    const uint32_t *base = xmajor ? A.colbits : A.rowbits;
    const int lw = xmajor ? A.words_c : A.words_r;
    const int c0 = min0 + kPad;
    // column 0: the obstacle (0, 1) blocks slope 1 and beyond
    if (lane == 0) {
        const bool o01 = column_obst(base + (size_t)maj0 * lw, lw, c0, neg, 1);
        la[0] = make_uint2(slope_pack(Slope{0, 1, false}), slope_pack(Slope{1, 1, o01}));
    }
    __syncwarp();
    int na = 1;
    for (int k = 1; na > 0; k++) {
        const int maj = maj0 + smaj * k;
        if (maj < 0 || maj >= maj_n) break;
        const uint32_t *line = base + (size_t)maj * lw;
        // 1. the target rows of every interval into the row mask
        int amin = 0x7fffffff, bmax = -1, rmax = 0;
        int a0 = 0, b0 = -1;   // rows of this lane's first interval, kept for step 3
        for (int i = lane; i < na; i += 32) {
            const uint2 iv = la[i];
            const Slope lo = slope_unpack(iv.x), hi = slope_unpack(iv.y);
            int a, b;
            interval_rows(lo, hi, k, a, b);
            if (i == lane) {
                a0 = a;
                b0 = b;
            }
            if (b >= A.mask_words * 32 - 33) {   // b <= k < the major extent: never taken
                atomicOr(A.err, 4);
                b = A.mask_words * 32 - 34;
            }
            rmax = max(rmax, b + 1);
            if (a <= b) {
                amin = min(amin, a);
                bmax = max(bmax, b);
                for (int w = a >> 5; w <= (b >> 5); w++) {
                    const int lo_b = max(a - w * 32, 0), hi_b = min(b - w * 32, 31);
                    const uint32_t bits = (hi_b == 31 ? 0xffffffffu : ((1u << (hi_b + 1)) - 1u)) & ~((1u << lo_b) - 1u);
                    atomicOr(mask + w, bits);
                }
            }
        }
        amin = __reduce_min_sync(0xffffffffu, amin);
        bmax = __reduce_max_sync(0xffffffffu, bmax);
        rmax = __reduce_max_sync(0xffffffffu, rmax);
        // the column's obstacle words for rows 0 .. rmax + 32, staged once for
        // steps 2 and 3
        for (int w = lane; w <= (rmax >> 5) + 1; w += 32) obw[w] = column_bits(line, lw, c0, neg, w * 32);
        __syncwarp();
        // 2. visible targets: masked rows that are free; the diagonal target
        //    also needs (k, k - 1) free
        if (bmax >= 0) {
            const bool diag_blocked = column_obst(line, lw, c0, neg, k - 1);
            for (int w = amin >> 5; w <= (bmax >> 5); w++) {
                const uint32_t m = mask[w];
                uint32_t vis = m & ~obw[w];
                if (diag_blocked && k >= w * 32 && k < w * 32 + 32) vis &= ~(1u << (k - w * 32));
                if (ROWS) {
                    const int r = w * 32 + lane;
                    const bool sees = (vis >> lane) & 1u;
                    int id = -1;
                    if (sees) {
                        const int minor = min0 + smin * r;
                        id = xmajor ? __ldg(A.node_of_cell_t + (size_t)maj * A.H + minor)
                                    : __ldg(A.node_of_cell + (size_t)maj * A.W + minor);
                        if (id < 0) atomicOr(A.err, 1);
                    }
                    // cells of a row have consecutive ids in raster order: the
                    // lanes of up to two words join theirs into one atomic
                    uint32_t left = __ballot_sync(0xffffffffu, id >= 0);
                    if (!xmajor) {
#pragma unroll
                        for (int join = 0; join < 2; join++) {
                            if (!left) break;
                            const int lead = __ffs(left) - 1;
                            const int word = __shfl_sync(0xffffffffu, id >> 5, lead);
                            const bool same = ((left >> lane) & 1u) && (id >> 5) == word;
                            const uint32_t bits = __reduce_or_sync(0xffffffffu, same ? 1u << (id & 31) : 0u);
                            if (lane == lead) atomicOr(bm + word, bits);
                            left &= ~__ballot_sync(0xffffffffu, same);
                        }
                    }
                    if ((left >> lane) & 1u) atomicOr(bm + (id >> 5), 1u << (id & 31));
                } else if ((vis >> lane) & 1u) {
                    const int r = w * 32 + lane;
                    const int x = xmajor ? maj : sx + smin * r;
                    const int y = xmajor ? sy + smin * r : maj;
                    const int id = __ldg(A.node_of_cell + (size_t)y * A.W + x);
                    if (id >= 0) {
                        atomicOr(bm + (id >> 5), 1u << (id & 31));
                        id_lo = min(id_lo, id);
                        id_hi = max(id_hi, id);
                    } else {
                        atomicOr(A.err, 1);
                    }
                }
                __syncwarp();
                if (lane == 0) mask[w] = 0u;
            }
        }
        __syncwarp();
        // 3. the pieces each interval leaves for column k + 1, appended to
        //    the other list in any order
        if (lane == 0) *count = 0;
        __syncwarp();
        for (int i = lane; i < na; i += 32) {
            const uint2 iv = la[i];
            const Slope lo = slope_unpack(iv.x), hi = slope_unpack(iv.y);
            int a = a0, b = b0;
            if (i != lane) interval_rows(lo, hi, k, a, b);
            interval_pieces(lo, hi, k, max(a - 1, 0), b + 1, obw, lb, count, cap);
        }
        __syncwarp();
        const int total = *count;
        if (total > cap) return false;
        uint2 *t = la;
        la = lb;
        lb = t;
        na = total;
    }
    return true;
}

// What becomes of a source's list: its bytes are counted; or written at its
// place in the CSR (which the counts of all lists before it fix); or counted
// and written to the next free bytes of a stage, in the order the sources
// finish, from where stage_gather_kernel brings every list to its place.
enum SweepMode { kSweepCount, kSweepWrite, kSweepStage };
constexpr uint64_t kNotStaged = ~0ull;

// Persistent CTAs of 8 warps take sources from a counter; each warp sweeps
// one octant into the CTA's node bitmap, then the warps encode the bitmap's
// set bits as the source's LEB128 delta list (MODE).  GLOBAL_LISTS: interval lists in global memory with room for the
// proven maximum (retried sources); otherwise kSweepCap entries in shared
// memory, and a source whose list outgrows them is queued for the retry.
template <SweepMode MODE, bool GLOBAL_LISTS, bool SMEM_BITMAP>
__global__ void __launch_bounds__(kSweepThreads, 6) visibility_sweep_kernel(SweepArgs A) {
    extern __shared__ __align__(16) uint8_t smem[];
    __shared__ uint32_t s_src;
    __shared__ int s_overflow, s_lo[kSweepWarps], s_hi[kSweepWarps];
    __shared__ int s_first[kSweepWarps], s_last[kSweepWarps];
    __shared__ uint32_t s_bytes[kSweepWarps];
    __shared__ int s_count[kSweepWarps];
    __shared__ uint64_t s_at;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint8_t *p = smem;
    uint32_t *bm;
    if (SMEM_BITMAP) {
        bm = reinterpret_cast<uint32_t *>(p);
        p += (size_t)((A.words_n + 3) & ~3u) * 4;
    } else {
        bm = A.gbitmap + (size_t)blockIdx.x * A.words_n;
    }
    uint2 *la, *lb;
    int cap;
    if (GLOBAL_LISTS) {
        la = A.glists + ((size_t)blockIdx.x * kSweepWarps + warp) * 2 * A.glist_cap;
        lb = la + A.glist_cap;
        cap = A.glist_cap;
    } else {
        la = reinterpret_cast<uint2 *>(p) + (size_t)warp * 2 * kSweepCap;
        lb = la + kSweepCap;
        cap = A.smem_cap;
        p += (size_t)kSweepWarps * 2 * kSweepCap * sizeof(uint2);
    }
    uint32_t *mask = reinterpret_cast<uint32_t *>(p) + (size_t)warp * A.mask_words;
    uint32_t *obw = reinterpret_cast<uint32_t *>(p) + (size_t)(kSweepWarps + warp) * A.mask_words;
    for (uint32_t w = threadIdx.x; w < A.words_n; w += blockDim.x) bm[w] = 0u;
    for (int w = lane; w < A.mask_words; w += 32) mask[w] = 0u;
    for (;;) {
        if (threadIdx.x == 0) {
            const uint32_t i = atomicAdd(A.next, 1u);
            s_src = i < A.count ? (A.sources ? A.sources[i] : i) : kNoSource;
            s_overflow = 0;
        }
        __syncthreads();
        const uint32_t u = s_src;
        if (u == kNoSource) break;
        const uint32_t cell = A.cells[u];
        const int sx = (int)(cell % (uint32_t)A.W), sy = (int)(cell / (uint32_t)A.W);
        int id_lo = 0x7fffffff, id_hi = -1;
        if (!sweep_octant<false>(A, warp, sx, sy, bm, la, lb, cap, mask, obw, &s_count[warp], id_lo, id_hi)) {
            if (lane == 0) s_overflow = 1;
            for (int w = lane; w < A.mask_words; w += 32) mask[w] = 0u;
        }
        id_lo = __reduce_min_sync(0xffffffffu, id_lo);
        id_hi = __reduce_max_sync(0xffffffffu, id_hi);
        if (lane == 0) {
            s_lo[warp] = id_lo;
            s_hi[warp] = id_hi;
        }
        __syncthreads();
        int lo = 0x7fffffff, hi = -1;
#pragma unroll
        for (int w = 0; w < kSweepWarps; w++) {
            lo = min(lo, s_lo[w]);
            hi = max(hi, s_hi[w]);
        }
        const bool overflow = s_overflow != 0;
        if (hi >= 0 && !overflow) {
            // encode: warp w takes an equal share of the bitmap words lo/32 .. hi/32
            const uint32_t w0 = (uint32_t)lo >> 5, w1 = ((uint32_t)hi >> 5) + 1;
            const uint32_t per = (w1 - w0 + kSweepWarps - 1) / kSweepWarps;
            const uint32_t mb = min(w0 + warp * per, w1), me = min(mb + per, w1);
            // phase A: first and last id of the share, and its bytes without
            // the leading varint of its first id
            int first = -1, last = -1;
            uint32_t bytes = 0;
            for (uint32_t c = mb; c < me; c += 32) {
                const uint32_t wi = c + lane;
                const uint32_t word = wi < me ? (SMEM_BITMAP ? bm[wi] : __ldcg(bm + wi)) : 0u;
                const int wl = word ? (int)(wi * 32 + 31 - __clz(word)) : -1;
                const int wf = word ? (int)(wi * 32 + __ffs(word) - 1) : 0x7fffffff;
                int incl = wl;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int t = __shfl_up_sync(0xffffffffu, incl, o);
                    if (lane >= o && t > incl) incl = t;
                }
                int excl = __shfl_up_sync(0xffffffffu, incl, 1);
                if (lane == 0) excl = -1;
                if (last > excl) excl = last;
                uint32_t nb = 0;
                if (word) {
                    nb = (uint32_t)__popc(word) - 1u;
                    if (excl >= 0) nb += varint_len((uint32_t)(wf - excl));
                }
                bytes += __reduce_add_sync(0xffffffffu, nb);
                const int cf = __reduce_min_sync(0xffffffffu, wf);
                if (first < 0 && cf != 0x7fffffff) first = cf;
                const int cl = __shfl_sync(0xffffffffu, incl, 31);
                if (cl > last) last = cl;
            }
            if (lane == 0) {
                s_first[warp] = first;
                s_last[warp] = last;
                s_bytes[warp] = bytes;
            }
            __syncthreads();
            // each share's leading varint follows the last id of the shares before it
            int prev = -1, run = -1;
            uint64_t start = 0, total = 0;
            for (int w = 0; w < kSweepWarps; w++) {
                if (w == warp) prev = run;
                uint32_t bw = s_bytes[w];
                if (s_first[w] >= 0) bw += varint_len(run < 0 ? (uint32_t)s_first[w] : (uint32_t)(s_first[w] - run));
                if (w < warp) start += bw;
                total += bw;
                if (s_last[w] > run) run = s_last[w];
            }
            if (MODE != kSweepWrite && threadIdx.x == 0) A.row_bytes[u] = total;
            uint64_t list_at = 0, end = 0;
            bool write = false;
            if (MODE == kSweepWrite) {
                list_at = A.offsets[u];
                end = A.offsets[u + 1];
                write = true;
            } else if (MODE == kSweepStage) {
                if (threadIdx.x == 0) {
                    s_at = atomicAdd(A.stage_used, (unsigned long long)((total + 15) & ~15ull));
                    if (s_at + total > A.stage_cap) s_at = kNotStaged;
                    A.stage_at[u] = s_at;
                }
                __syncthreads();
                list_at = s_at;
                write = list_at != kNotStaged;
                end = list_at + total;
            }
            if (write) {
                // phase B: write the share's varints from its first byte on
                uint64_t pos = list_at + start;
                int run_prev = prev;
                for (uint32_t c = mb; c < me; c += 32) {
                    const uint32_t wi = c + lane;
                    const uint32_t word = wi < me ? (SMEM_BITMAP ? bm[wi] : __ldcg(bm + wi)) : 0u;
                    const int wl = word ? (int)(wi * 32 + 31 - __clz(word)) : -1;
                    int incl = wl;
#pragma unroll
                    for (int o = 1; o < 32; o <<= 1) {
                        const int t = __shfl_up_sync(0xffffffffu, incl, o);
                        if (lane >= o && t > incl) incl = t;
                    }
                    int excl = __shfl_up_sync(0xffffffffu, incl, 1);
                    if (lane == 0) excl = -1;
                    if (run_prev > excl) excl = run_prev;
                    uint32_t nb = 0;
                    if (word) {
                        const uint32_t wf = wi * 32 + (__ffs(word) - 1);
                        nb = (uint32_t)__popc(word) - 1u + varint_len(excl < 0 ? wf : wf - (uint32_t)excl);
                    }
                    uint32_t sc = nb;
#pragma unroll
                    for (int o = 1; o < 32; o <<= 1) {
                        const uint32_t t = __shfl_up_sync(0xffffffffu, sc, o);
                        if (lane >= o) sc += t;
                    }
                    if (word) {
                        uint64_t q = pos + (sc - nb);
                        uint32_t left = word;
                        int last_id = excl;
                        while (left) {
                            const uint32_t id = wi * 32 + (__ffs(left) - 1);
                            left &= left - 1u;
                            uint32_t x = last_id < 0 ? id : id - (uint32_t)last_id;
                            do {
                                uint8_t byte = (uint8_t)(x & 0x7fu);
                                x >>= 7;
                                if (x) byte |= 0x80u;
                                if (q < end) A.out[q] = byte;   // the count pass sized the list
                                else atomicOr(A.err, 8);
                                q++;
                            } while (x);
                            last_id = (int)id;
                        }
                    }
                    pos += __shfl_sync(0xffffffffu, sc, 31);
                    const int cl = __shfl_sync(0xffffffffu, incl, 31);
                    if (cl > run_prev) run_prev = cl;
                }
            }
        } else if (MODE != kSweepWrite && threadIdx.x == 0) {
            A.row_bytes[u] = 0;
            if (MODE == kSweepStage) A.stage_at[u] = 0;
        }
        if (overflow && threadIdx.x == 0) {
            if (GLOBAL_LISTS) {
                atomicOr(A.err, 2);
            } else {
                A.retry[atomicAdd(A.retry_count, 1u)] = u;
            }
        }
        // every warp has read its share: clear the words this source set (a
        // global bitmap is set by atomics in the L2, so it is read and
        // cleared there, past the L1)
        __syncthreads();
        if (hi >= 0)
            for (uint32_t w = ((uint32_t)lo >> 5) + threadIdx.x; w <= ((uint32_t)hi >> 5); w += blockDim.x) {
                if (SMEM_BITMAP) bm[w] = 0u;
                else __stcg(bm + w, 0u);
            }
        __syncthreads();
    }
}

// The rows kernel: a warp takes (source, octant) pairs from a counter and sweeps
// the octant into the source's row of the matrix.  Only the four octants that
// hold the cells after the source in raster order (and the rest of its own row)
// are swept; rows_join_kernel adds the other half.  No bitmap in shared memory
// and no octant that waits for another's, so 48 warps an SM stay busy: bound by
// the chain of steps from column to column.  City grid: 75 ms, with the joining 5,
// the counting 7 and the encoding 10, where a CTA of eight octants with a bitmap in
// shared memory took 229.
constexpr int kRowsOctants = 4;
template <bool GLOBAL_LISTS>
__global__ void __launch_bounds__(kSweepThreads, 6) visibility_rows_kernel(SweepArgs A) {
    extern __shared__ __align__(16) uint8_t smem[];
    __shared__ int s_count[kSweepWarps];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint8_t *p = smem;
    uint2 *la, *lb;
    int cap;
    if (GLOBAL_LISTS) {
        la = A.glists + ((size_t)blockIdx.x * kSweepWarps + warp) * 2 * A.glist_cap;
        lb = la + A.glist_cap;
        cap = A.glist_cap;
    } else {
        la = reinterpret_cast<uint2 *>(p) + (size_t)warp * 2 * kSweepCap;
        lb = la + kSweepCap;
        cap = A.smem_cap;
        p += (size_t)kSweepWarps * 2 * kSweepCap * sizeof(uint2);
    }
    uint32_t *mask = reinterpret_cast<uint32_t *>(p) + (size_t)warp * A.mask_words;
    uint32_t *obw = reinterpret_cast<uint32_t *>(p) + (size_t)(kSweepWarps + warp) * A.mask_words;
    for (int w = lane; w < A.mask_words; w += 32) mask[w] = 0u;
    __syncwarp();
    for (;;) {
        uint32_t i = 0;
        if (lane == 0) i = atomicAdd(A.next, 1u);
        i = __shfl_sync(0xffffffffu, i, 0);
        if (i >= A.count) break;
        const uint32_t item = A.sources ? A.sources[i] : i;
        const uint32_t u = item / kRowsOctants, o = item % kRowsOctants;
        const int oct = o < 2u ? (int)o : (int)(2u * o);  // 0, 1 (|dx| >= dy), 4, 6 (dy >= |dx|)
        const uint32_t cell = A.cells[u];
        int id_lo = 0, id_hi = 0;
        if (!sweep_octant<true>(A, oct, (int)(cell % (uint32_t)A.W), (int)(cell / (uint32_t)A.W),
                                A.matrix + (size_t)u * A.pitch, la, lb, cap, mask, obw, &s_count[warp], id_lo, id_hi)) {
            if (lane == 0) {
                if (GLOBAL_LISTS) atomicOr(A.err, 2);
                else A.retry[atomicAdd(A.retry_count, 1u)] = item;
            }
            for (int w = lane; w < A.mask_words; w += 32) mask[w] = 0u;
        }
        __syncwarp();
    }
}

// out[x * H + y] = in[y * W + x], one 32 x 32 tile a CTA of 32 x 8 threads.  (On
// the host the transposition took 1.5 s of a 16,384 x 16,384 grid's build, which
// takes 0.45 s with it here.)
__global__ void __launch_bounds__(256) cells_transpose_kernel(const int32_t *__restrict__ in, int W, int H,
                                                             int32_t *__restrict__ out) {
    __shared__ int32_t tile[32][33];
    const int x0 = blockIdx.x * 32, y0 = blockIdx.y * 32, tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    for (int j = ty; j < 32; j += 8)
        if (x0 + tx < W && y0 + j < H) tile[j][tx] = in[(size_t)(y0 + j) * W + x0 + tx];
    __syncthreads();
    for (int j = ty; j < 32; j += 8)
        if (x0 + j < W && y0 + tx < H) out[(size_t)(x0 + j) * H + y0 + tx] = tile[tx][j];
}

// Transpose of the warp's 32 x 32 bits (lane = row, bit = column).
__device__ __forceinline__ uint32_t transpose32(uint32_t x, int lane) {
    const uint32_t keep[5] = {0x0000ffffu, 0x00ff00ffu, 0x0f0f0f0fu, 0x33333333u, 0x55555555u};
#pragma unroll
    for (int s = 0; s < 5; s++) {
        const int d = 16 >> s;
        const uint32_t y = __shfl_xor_sync(0xffffffffu, x, d);
        x = (lane & d) ? (x & ~keep[s]) | ((y >> d) & keep[s]) : (x & keep[s]) | ((y << d) & ~keep[s]);
    }
    return x;
}

// matrix |= transpose(matrix), one CTA per pair of mirrored tiles of kTile x
// kTile bits (blockIdx.x <= blockIdx.y), both in shared memory.  The matrix's
// sides are multiples of kTile.  Bound: its bytes read and written once (14 GB
// for the city).
constexpr int kTile = 512, kTileWords = kTile / 32, kTilePitch = kTileWords + 1;
constexpr size_t kJoinSmem = 2ull * kTile * kTilePitch * 4;
__global__ void __launch_bounds__(256) rows_join_kernel(uint32_t *__restrict__ matrix, uint32_t pitch) {
    extern __shared__ __align__(16) uint32_t s_bits[];
    const uint32_t ti = blockIdx.x, tj = blockIdx.y;
    if (ti > tj) return;
    const bool diagonal = ti == tj;
    uint32_t *a = s_bits, *b = diagonal ? s_bits : s_bits + kTile * kTilePitch;
    auto tile = [&](uint32_t rt, uint32_t ct, int x) {  // 16 bytes x of tile (rt, ct)
        return reinterpret_cast<uint4 *>(matrix + (size_t)(rt * kTile + x / (kTileWords / 4)) * pitch + ct * kTileWords) +
               x % (kTileWords / 4);
    };
    constexpr int kChunks = kTile * kTileWords / 4;
    for (int x = threadIdx.x; x < kChunks; x += blockDim.x) {
        uint32_t *d = a + (x / (kTileWords / 4)) * kTilePitch + 4 * (x % (kTileWords / 4));
        const uint4 v = *tile(ti, tj, x);
        d[0] = v.x, d[1] = v.y, d[2] = v.z, d[3] = v.w;
        if (!diagonal) {
            uint32_t *e = d + (b - a);
            const uint4 w = *tile(tj, ti, x);
            e[0] = w.x, e[1] = w.y, e[2] = w.z, e[3] = w.w;
        }
    }
    __syncthreads();
    const int lane = threadIdx.x & 31;
    for (int q = threadIdx.x >> 5; q < kTileWords * kTileWords; q += blockDim.x >> 5) {
        const int bi = q / kTileWords, bj = q % kTileWords;
        if (diagonal && bi > bj) continue;
        uint32_t &x = a[(bi * 32 + lane) * kTilePitch + bj], &y = b[(bj * 32 + lane) * kTilePitch + bi];
        const uint32_t xv = x, yv = y;
        const uint32_t xt = transpose32(xv, lane), yt = transpose32(yv, lane);
        __syncwarp();
        x = xv | yt;
        if (!diagonal || bi != bj) y = yv | xt;
    }
    __syncthreads();
    for (int x = threadIdx.x; x < kChunks; x += blockDim.x) {
        const uint32_t *d = a + (x / (kTileWords / 4)) * kTilePitch + 4 * (x % (kTileWords / 4));
        *tile(ti, tj, x) = make_uint4(d[0], d[1], d[2], d[3]);
        if (!diagonal) {
            const uint32_t *e = d + (b - a);
            *tile(tj, ti, x) = make_uint4(e[0], e[1], e[2], e[3]);
        }
    }
}

// What the graph object keeps of a row of the matrix: the node's degree, its
// list's bytes and its range lookups (a run of L ids takes run_lookup_count(L)
// of them), one warp per row, 32 words a step.  A run is counted where it ends;
// its start follows from the last clear bit before it.
constexpr int kEncodeWarps = 8;
__global__ void __launch_bounds__(kEncodeWarps * 32) rows_count_kernel(const uint32_t *__restrict__ matrix,
                                                                      uint32_t pitch, uint32_t words, uint32_t n,
                                                                      int scheme, uint64_t *__restrict__ row_bytes,
                                                                      uint32_t *__restrict__ degree,
                                                                      uint32_t *__restrict__ lookups) {
    const int lane = threadIdx.x & 31;
    const uint64_t u = (uint64_t)blockIdx.x * kEncodeWarps + (threadIdx.x >> 5);
    if (u >= n) return;
    const uint32_t *row = matrix + u * pitch;
    int run = -1, clear = -1;  // last set and last clear id so far
    uint32_t ids = 0, more = 0, lks = 0;
    uint32_t next = lane < (int)words ? __ldcs(row + lane) : 0u;
    for (uint32_t c = 0; c < words; c += 32) {
        const uint32_t wi = c + lane;
        const uint32_t word = next;
        next = wi + 32 < words ? __ldcs(row + wi + 32) : 0u;
        const int last_id = (int)(c * 32 + 1023);
        if (!__any_sync(0xffffffffu, word != 0u)) {
            clear = last_id;
            continue;
        }
        int set = word ? (int)(wi * 32 + 31 - __clz(word)) : -1;
        int zero = ~word ? (int)(wi * 32 + 31 - __clz(~word)) : -1;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int x = __shfl_up_sync(0xffffffffu, set, o), y = __shfl_up_sync(0xffffffffu, zero, o);
            if (lane >= o) {
                set = max(set, x);
                zero = max(zero, y);
            }
        }
        int set_before = __shfl_up_sync(0xffffffffu, set, 1), zero_before = __shfl_up_sync(0xffffffffu, zero, 1);
        if (lane == 0) set_before = zero_before = -1;
        set_before = max(set_before, run);
        zero_before = max(zero_before, clear);
        run = max(run, __shfl_sync(0xffffffffu, set, 31));
        clear = max(clear, __shfl_sync(0xffffffffu, zero, 31));
        uint32_t after = __shfl_down_sync(0xffffffffu, word, 1);
        const uint32_t over = __shfl_sync(0xffffffffu, next, 0);
        if (lane == 31) after = over;
        if (word) {
            const uint32_t wf = wi * 32 + (__ffs(word) - 1);
            ids += __popc(word);
            more += varint_len(set_before < 0 ? wf : wf - (uint32_t)set_before) - 1u;
            for (uint32_t ends = word & ~(word >> 1 | after << 31); ends; ends &= ends - 1u) {
                const int k = __ffs(ends) - 1;
                const uint32_t z = ~word & ((1u << k) - 1u);
                const int start = z ? (int)(wi * 32 + 32 - __clz(z)) : zero_before + 1;
                lks += run_lookup_count(wi * 32 + k + 1u - (uint32_t)start, scheme);
            }
        }
    }
    ids = __reduce_add_sync(0xffffffffu, ids);
    more = __reduce_add_sync(0xffffffffu, more);
    lks = __reduce_add_sync(0xffffffffu, lks);
    if (lane == 0) {
        row_bytes[u] = (uint64_t)ids + more;
        degree[u] = ids;
        lookups[u] = lks;
    }
}

// LEB128 delta lists of the matrix's rows, one warp per row, 32 words a step.
// Within a word every delta is below 128, so only a word's first id can take
// more than one byte.  Most bytes are the 1 of a consecutive id: a step's bytes
// (at most 32 x 36) are filled with ones in shared memory, the lanes put in the
// deltas where runs start, and the step is stored 16 bytes at a time.
__global__ void __launch_bounds__(kEncodeWarps * 32) rows_encode_kernel(const uint32_t *__restrict__ matrix,
                                                                       uint32_t pitch, uint32_t words, uint32_t n,
                                                                       const uint64_t *__restrict__ offsets,
                                                                       uint8_t *__restrict__ out, int *err) {
    constexpr uint32_t kBuf = 32 * 36 + 32;
    __shared__ __align__(16) uint8_t s_buf[kEncodeWarps][kBuf];
    const int lane = threadIdx.x & 31;
    const uint64_t u = (uint64_t)blockIdx.x * kEncodeWarps + (threadIdx.x >> 5);
    if (u >= n) return;
    uint8_t *buf = s_buf[threadIdx.x >> 5];
    const uint32_t *row = matrix + u * pitch;
    int run = -1;  // last id so far
    uint64_t pos = offsets[u];
    const uint64_t end = offsets[u + 1];
    uint32_t next = lane < (int)words ? __ldcs(row + lane) : 0u;
    for (uint32_t c = 0; c < words; c += 32) {
        const uint32_t wi = c + lane;
        const uint32_t word = next;
        next = wi + 32 < words ? __ldcs(row + wi + 32) : 0u;
        if (!__any_sync(0xffffffffu, word != 0u)) continue;
        int incl = word ? (int)(wi * 32 + 31 - __clz(word)) : -1;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o && t > incl) incl = t;
        }
        int excl = __shfl_up_sync(0xffffffffu, incl, 1);
        if (lane == 0) excl = -1;
        if (run > excl) excl = run;
        const uint32_t wf = wi * 32 + (uint32_t)(word ? __ffs(word) - 1 : 0);
        const uint32_t first = word ? varint_len(excl < 0 ? wf : wf - (uint32_t)excl) : 0u;  // bytes of the first id
        const uint32_t nb = word ? (uint32_t)__popc(word) - 1u + first : 0u;
        run = max(run, __shfl_sync(0xffffffffu, incl, 31));
        uint32_t sc = nb;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t t = __shfl_up_sync(0xffffffffu, sc, o);
            if (lane >= o) sc += t;
        }
        const uint32_t total = __shfl_sync(0xffffffffu, sc, 31);
        const uint32_t head = (uint32_t)(pos & 15u);  // the buffer holds the bytes from pos - head on
        const uint32_t e = head + total;
        if (pos + total > end) {  // the count pass sized the list
            if (lane == 0) atomicOr(err, 8);
            break;
        }
        for (uint32_t x = 16u * lane; x < e; x += 512u)
            *reinterpret_cast<uint4 *>(buf + x) = make_uint4(0x01010101u, 0x01010101u, 0x01010101u, 0x01010101u);
        __syncwarp();
        if (word) {
            const uint32_t q = head + sc - nb;
            const bool goes_on = excl >= 0 && (uint32_t)excl + 1u == wi * 32;  // the id before the word is set
            uint32_t starts = word & ~(word << 1 | (goes_on ? 1u : 0u));
            if (starts & (word & (0u - word))) {  // the first id starts a run
                uint32_t x = excl < 0 ? wf : wf - (uint32_t)excl, at = q;
                starts &= starts - 1u;
                while (x > 0x7fu) {
                    buf[at++] = (uint8_t)(x | 0x80u);
                    x >>= 7;
                }
                buf[at] = (uint8_t)x;
            }
            for (; starts; starts &= starts - 1u) {
                const int k = __ffs(starts) - 1;
                const uint32_t below = word & ((1u << k) - 1u);
                buf[q + first - 1u + __popc(below)] = (uint8_t)(k - (31 - __clz(below)));
            }
        }
        __syncwarp();
        uint8_t *dst = out + (pos - head);
        const uint32_t b0 = head ? 16u : 0u, b1 = e & ~15u;
        if (head && lane >= (int)head && lane < 16 && lane < (int)e) dst[lane] = buf[lane];
        for (uint32_t x = b0 + 16u * lane; x < b1; x += 512u)
            *reinterpret_cast<uint4 *>(dst + x) = *reinterpret_cast<const uint4 *>(buf + x);
        const uint32_t t0 = max(b1, b0) + lane;
        if (t0 < e) dst[t0] = buf[t0];
        pos += total;
        __syncwarp();
    }
}

// Brings the staged lists to their places in the CSR, one warp per list: the
// stage's lists start on 16-byte boundaries, the CSR's anywhere, so each lane
// builds aligned 16-byte words of the destination from five words of the
// source (the stage is readable 16 bytes past its end).
__global__ void __launch_bounds__(256) stage_gather_kernel(const uint8_t *__restrict__ stage,
                                                           const uint64_t *__restrict__ stage_at,
                                                           const uint64_t *__restrict__ offsets, uint32_t n,
                                                           uint8_t *__restrict__ out) {
    const int lane = threadIdx.x & 31;
    const uint64_t v = (uint64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (v >= n || stage_at[v] == kNotStaged) return;
    const uint64_t o0 = offsets[v], o1 = offsets[v + 1];
    const uint8_t *src = stage + stage_at[v];
    const uint64_t up = (o0 + 15) & ~15ull, down = o1 & ~15ull;
    const uint64_t b0 = up < o1 ? up : o1, b1 = down > b0 ? down : b0;
    if (o0 + lane < b0) out[o0 + lane] = src[lane];
    if (b1 + lane < o1) out[b1 + lane] = src[b1 - o0 + lane];
    const uint32_t *w = reinterpret_cast<const uint32_t *>(src + ((b0 - o0) & ~3ull));
    const uint32_t shift = 8u * (uint32_t)((b0 - o0) & 3u);
    for (uint64_t q = lane; q < (b1 - b0) / 16; q += 32) {
        uint32_t x[5];
#pragma unroll
        for (int i = 0; i < 5; i++) x[i] = __ldcs(w + 4 * q + i);
        uint4 y;
        y.x = __funnelshift_r(x[0], x[1], shift);
        y.y = __funnelshift_r(x[1], x[2], shift);
        y.z = __funnelshift_r(x[2], x[3], shift);
        y.w = __funnelshift_r(x[3], x[4], shift);
        *reinterpret_cast<uint4 *>(out + b0 + 16 * q) = y;
    }
}

}  // namespace
}  // namespace vga

using namespace vga;

extern "C" {

int vga_visibility_count(int W, int H, const uint8_t *obst, uint32_t *n_nodes) {
    clear_error();
    if (!obst || !n_nodes || W < 1 || H < 1 || W > kMaxSide || H > kMaxSide) {
        set_error("vga_visibility_count: bad arguments (W=%d, H=%d)", W, H);
        return VGA_EINVAL;
    }
    *n_nodes = (uint32_t)main_component_cells(W, H, obst).size();
    return VGA_OK;
}

int vga_visibility_build_ordered(int W, int H, const uint8_t *obst, int order, uint64_t *cell_of_node,
                                 vga_graph **out) {
    clear_error();
    if (!obst || !out || W < 1 || H < 1 || W > kMaxSide || H > kMaxSide || (order != 0 && order != 1)) {
        set_error("vga_visibility_build: bad arguments (W=%d, H=%d, order=%d, limit %d)", W, H, order, kMaxSide);
        return VGA_EINVAL;
    }
    std::vector<uint32_t> cells = main_component_cells(W, H, obst);
    if (order == 1) {
        int k = 1;
        while ((1 << k) < std::max(W, H)) k++;
        std::vector<std::pair<uint64_t, uint32_t>> keyed(cells.size());
        for (size_t i = 0; i < cells.size(); i++)
            keyed[i] = {hilbert_position(k, cells[i] % (uint32_t)W, cells[i] / (uint32_t)W), cells[i]};
        std::sort(keyed.begin(), keyed.end());
        for (size_t i = 0; i < cells.size(); i++) cells[i] = keyed[i].second;
    }
    const uint32_t n = (uint32_t)cells.size();
    if (cell_of_node)
        for (uint32_t v = 0; v < n; v++) cell_of_node[v] = cells[v];
    // obstacle bitmaps with kPad margin bits of obstacles on both ends of
    // every line: row-major lines for the octants that step along y, and
    // column-major ones for those that step along x
    const int words_r = (W + 2 * kPad + 31) / 32, words_c = (H + 2 * kPad + 31) / 32;
    std::vector<uint32_t> rowbits((size_t)H * words_r, 0xffffffffu), colbits((size_t)W * words_c, 0xffffffffu);
    for (int y = 0; y < H; y++)
        for (int x = 0; x < W; x++)
            if (!obst[(size_t)y * W + x]) {
                const int pr = x + kPad, pc = y + kPad;
                rowbits[(size_t)y * words_r + (pr >> 5)] &= ~(1u << (pr & 31));
                colbits[(size_t)x * words_c + (pc >> 5)] &= ~(1u << (pc & 31));
            }
    std::vector<int32_t> node_of_cell((size_t)W * H, -1);
    for (uint32_t v = 0; v < n; v++) node_of_cell[cells[v]] = (int32_t)v;
    const int maxdim = std::max(W, H);
    const uint32_t words_n = (n + 31) / 32;
    const int mask_words = maxdim / 32 + 2;
    int dev = 0, sms = 0, smem_optin = 0;
    VGA_CHECK_CUDA(cudaGetDevice(&dev));
    VGA_CHECK_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    VGA_CHECK_CUDA(cudaDeviceGetAttribute(&smem_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
    const size_t list_smem = (size_t)kSweepWarps * 2 * kSweepCap * sizeof(uint2);
    const size_t mask_smem = (size_t)2 * kSweepWarps * mask_words * 4;   // row masks and staged obstacle words
    const size_t bitmap_smem = (size_t)((words_n + 3) & ~3u) * 4;
    // the node bitmap stays in shared memory while two CTAs fit an SM
    const uint32_t pitch = (words_n + kTileWords - 1) / kTileWords * kTileWords;
    const uint64_t matrix_bytes = 32ull * pitch * pitch * 4;
    bool by_rows = n && g_sweep_smem_bitmap_nodes == 0 && matrix_bytes <= kMatrixBytes &&
                   (n < kMatrixNodes || mean_view(W, H, cells, node_of_cell) * kMatrixView >= (double)n);
    const bool smem_bitmap = bitmap_smem + list_smem + mask_smem + 1024 <= (size_t)smem_optin / 2 &&
                             (g_sweep_smem_bitmap_nodes == 0 || n <= g_sweep_smem_bitmap_nodes);
    const int glist_cap = maxdim + 2;   // at most k + 1 intervals are alive at column k + 1

    DeviceBuffer d_rowbits, d_colbits, d_noc, d_cells, d_rowbytes, d_counter, d_retry, d_err, d_off, d_gbitmap, d_glists;
    VGA_TRY(d_rowbits.alloc(rowbits.size() * 4));
    VGA_TRY(d_colbits.alloc(colbits.size() * 4));
    VGA_TRY(d_noc.alloc(node_of_cell.size() * 4));
    VGA_TRY(d_cells.alloc((size_t)std::max<uint32_t>(n, 1) * 4));
    VGA_TRY(d_rowbytes.alloc((size_t)std::max<uint32_t>(n, 1) * 8));
    VGA_TRY(d_counter.alloc(6 * sizeof(uint32_t)));
    if (by_rows && d_retry.alloc((size_t)n * 4 * kRowsOctants) != VGA_OK) {
        cudaGetLastError();
        clear_error();
        by_rows = false;
    }
    if (!by_rows) VGA_TRY(d_retry.alloc((size_t)std::max<uint32_t>(n, 1) * 4));
    VGA_TRY(d_err.alloc(sizeof(int)));
    VGA_TRY(d_off.alloc(((size_t)n + 1) * 8));
    cudaStream_t stream = 0;
    VGA_CHECK_CUDA(cudaMemcpyAsync(d_rowbits.ptr, rowbits.data(), rowbits.size() * 4, cudaMemcpyHostToDevice, stream));
    VGA_CHECK_CUDA(cudaMemcpyAsync(d_colbits.ptr, colbits.data(), colbits.size() * 4, cudaMemcpyHostToDevice, stream));
    VGA_CHECK_CUDA(cudaMemcpyAsync(d_noc.ptr, node_of_cell.data(), node_of_cell.size() * 4, cudaMemcpyHostToDevice,
                                   stream));
    if (n) VGA_CHECK_CUDA(cudaMemcpyAsync(d_cells.ptr, cells.data(), (size_t)n * 4, cudaMemcpyHostToDevice, stream));
    VGA_CHECK_CUDA(cudaMemsetAsync(d_counter.ptr, 0, 6 * sizeof(uint32_t), stream));
    VGA_CHECK_CUDA(cudaMemsetAsync(d_err.ptr, 0, sizeof(int), stream));

    SweepArgs sa{};
    sa.rowbits = d_rowbits.as<uint32_t>();
    sa.colbits = d_colbits.as<uint32_t>();
    sa.W = W;
    sa.H = H;
    sa.words_r = words_r;
    sa.words_c = words_c;
    sa.node_of_cell = d_noc.as<int32_t>();
    sa.cells = d_cells.as<uint32_t>();
    sa.n = n;
    sa.row_bytes = d_rowbytes.as<uint64_t>();
    sa.retry = d_retry.as<uint32_t>();
    sa.retry_count = d_counter.as<uint32_t>() + 2;
    sa.glist_cap = glist_cap;
    sa.words_n = words_n;
    sa.mask_words = mask_words;
    sa.smem_cap = g_sweep_smem_cap;
    sa.err = d_err.as<int>();

    // one launch of the sweep over `count` sources (sources == nullptr: all
    // nodes), interval lists in shared memory or (retries) in global memory
    auto launch = [&](SweepMode mode, bool global_lists, const uint32_t *sources, uint32_t count,
                      uint32_t *counter) -> int {
        if (!count) return VGA_OK;
        const size_t smem = (smem_bitmap ? bitmap_smem : 0) + (global_lists ? 0 : list_smem) + mask_smem;
        void (*fn)(SweepArgs);
#define VGA_SW(M)                                                                                   \
    if (global_lists)                                                                               \
        fn = smem_bitmap ? visibility_sweep_kernel<M, true, true> : visibility_sweep_kernel<M, true, false>;   \
    else                                                                                            \
        fn = smem_bitmap ? visibility_sweep_kernel<M, false, true> : visibility_sweep_kernel<M, false, false>
        if (mode == kSweepWrite) VGA_SW(kSweepWrite);
        else if (mode == kSweepStage) VGA_SW(kSweepStage);
        else VGA_SW(kSweepCount);
#undef VGA_SW
        VGA_CHECK_CUDA(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        int per_sm = 0;
        VGA_CHECK_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, kSweepThreads, smem));
        if (per_sm < 1) {
            set_error("visibility sweep: %zu bytes of shared memory do not fit an SM", smem);
            return VGA_EINVAL;
        }
        const uint32_t grid = (uint32_t)std::min<uint64_t>((uint64_t)sms * per_sm, count);
        if (!smem_bitmap) {
            const size_t need = (size_t)grid * words_n * 4;
            if (d_gbitmap.bytes < need) VGA_TRY(d_gbitmap.alloc(need));
            VGA_CHECK_CUDA(cudaMemsetAsync(d_gbitmap.ptr, 0, need, stream));
        }
        if (global_lists) {
            const size_t need = (size_t)grid * kSweepWarps * 2 * glist_cap * sizeof(uint2);
            if (d_glists.bytes < need) VGA_TRY(d_glists.alloc(need));
        }
        SweepArgs a = sa;
        a.sources = sources;
        a.count = count;
        a.next = counter;
        a.gbitmap = d_gbitmap.as<uint32_t>();
        a.glists = d_glists.as<uint2>();
        fn<<<grid, kSweepThreads, smem, stream>>>(a);
        count_launch();
        VGA_CHECK_CUDA(cudaGetLastError());
        return VGA_OK;
    };

    // Without the matrix the lists are swept once, into a stage of the size they are expected to
    // take: the bound of n - 1 varints a list (one more byte for every 128 ids
    // that a delta skips) while that is small, else what every kSampleStep-th
    // source's list takes, and a twentieth on top.  What a full stage leaves
    // out, and everything when the stage cannot be had, is swept again straight
    // to its place in the CSR.
    std::vector<uint64_t> offsets((size_t)n + 1, 0);
    std::vector<uint32_t> again;   // sources to be swept again
    bool all_again = false;        // every source
    uint32_t n_retry = 0;
    DeviceBuffer d_stage, d_stage_at;
    uint32_t *retry_list = d_retry.as<uint32_t>();
    auto read_row_bytes = [&](std::vector<uint64_t> &rb) -> int {
        rb.resize(n);
        int err = 0;
        VGA_CHECK_CUDA(cudaMemcpyAsync(rb.data(), d_rowbytes.ptr, (size_t)n * 8, cudaMemcpyDeviceToHost, stream));
        VGA_CHECK_CUDA(cudaMemcpyAsync(&err, d_err.ptr, sizeof(int), cudaMemcpyDeviceToHost, stream));
        VGA_CHECK_CUDA(cudaStreamSynchronize(stream));
        if (err) {
            set_error("visibility sweep failed its own checks (code %d)", err);
            return VGA_ECORRUPT;
        }
        return VGA_OK;
    };
    // counters: [0], [1] sources taken, [2] retries, [4..5] stage bytes given out
    auto sweep = [&](SweepMode mode, const uint32_t *sources, uint32_t count) -> int {
        VGA_CHECK_CUDA(cudaMemsetAsync(d_counter.ptr, 0, 3 * sizeof(uint32_t), stream));
        VGA_TRY(launch(mode, false, sources, count, d_counter.as<uint32_t>()));
        VGA_CHECK_CUDA(cudaMemcpyAsync(&n_retry, sa.retry_count, 4, cudaMemcpyDeviceToHost, stream));
        VGA_CHECK_CUDA(cudaStreamSynchronize(stream));
        return launch(mode, true, retry_list, n_retry, d_counter.as<uint32_t>() + 1);
    };
    BuiltGraph built;  // what the matrix tells of the graph (without it, the load path derives it)
    DeviceBuffer d_matrix;
    // The bit matrix and what it tells.  VGA_ENOMEM: no room for it and what goes with it.
    auto build_rows = [&]() -> int {
        DeviceBuffer d_noc_t, d_lookups;
        VGA_TRY(d_noc_t.alloc((size_t)W * H * 4));
        VGA_TRY(d_lookups.alloc((size_t)n * 4));
        VGA_TRY(built.degree.alloc((size_t)n * 4));
        VGA_TRY(d_matrix.alloc(matrix_bytes));
        cells_transpose_kernel<<<dim3((W + 31) / 32, (H + 31) / 32), 256, 0, stream>>>(sa.node_of_cell, W, H,
                                                                                      d_noc_t.as<int32_t>());
        count_launch();
        VGA_CHECK_CUDA(cudaGetLastError());
        VGA_CHECK_CUDA(cudaMemsetAsync(d_matrix.ptr, 0, matrix_bytes, stream));
        sa.node_of_cell_t = d_noc_t.as<int32_t>();
        sa.matrix = d_matrix.as<uint32_t>();
        sa.pitch = pitch;
        auto sweep_rows = [&](bool global_lists, const uint32_t *sources, uint32_t count, uint32_t *counter) -> int {
            if (!count) return VGA_OK;
            auto fn = global_lists ? visibility_rows_kernel<true> : visibility_rows_kernel<false>;
            const size_t smem = (global_lists ? 0 : list_smem) + mask_smem;
            VGA_CHECK_CUDA(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
            int per_sm = 0;
            VGA_CHECK_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, kSweepThreads, smem));
            if (per_sm < 1) {
                set_error("visibility sweep: %zu bytes of shared memory do not fit an SM", smem);
                return VGA_EINVAL;
            }
            const uint32_t grid = (uint32_t)std::min<uint64_t>((uint64_t)sms * per_sm, (count + kSweepWarps - 1) / kSweepWarps);
            if (global_lists) VGA_TRY(d_glists.alloc((size_t)grid * kSweepWarps * 2 * glist_cap * sizeof(uint2)));
            SweepArgs a = sa;
            a.sources = sources;
            a.count = count;
            a.next = counter;
            a.glists = d_glists.as<uint2>();
            fn<<<grid, kSweepThreads, smem, stream>>>(a);
            count_launch();
            VGA_CHECK_CUDA(cudaGetLastError());
            return VGA_OK;
        };
        VGA_TRY(sweep_rows(false, nullptr, n * kRowsOctants, d_counter.as<uint32_t>()));
        VGA_CHECK_CUDA(cudaMemcpyAsync(&n_retry, sa.retry_count, 4, cudaMemcpyDeviceToHost, stream));
        VGA_CHECK_CUDA(cudaStreamSynchronize(stream));
        VGA_TRY(sweep_rows(true, retry_list, n_retry, d_counter.as<uint32_t>() + 1));
        VGA_CHECK_CUDA(cudaFuncSetAttribute(rows_join_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kJoinSmem));
        const unsigned tiles = pitch / kTileWords;
        rows_join_kernel<<<dim3(tiles, tiles), 256, kJoinSmem, stream>>>(sa.matrix, pitch);
        count_launch();
        built.scheme = table_scheme_auto(n, dev);
        rows_count_kernel<<<(n + kEncodeWarps - 1) / kEncodeWarps, kEncodeWarps * 32, 0, stream>>>(
            sa.matrix, pitch, words_n, n, built.scheme, sa.row_bytes, built.degree.as<uint32_t>(),
            d_lookups.as<uint32_t>());
        count_launch();
        VGA_CHECK_CUDA(cudaGetLastError());
        std::vector<uint32_t> deg(n);
        built.lookups.resize(n);
        VGA_CHECK_CUDA(cudaMemcpyAsync(deg.data(), built.degree.ptr, (size_t)n * 4, cudaMemcpyDeviceToHost, stream));
        VGA_CHECK_CUDA(cudaMemcpyAsync(built.lookups.data(), d_lookups.ptr, (size_t)n * 4, cudaMemcpyDeviceToHost,
                                       stream));
        std::vector<uint64_t> rb;
        VGA_TRY(read_row_bytes(rb));
        for (uint32_t v = 0; v < n; v++) {
            offsets[v + 1] = offsets[v] + rb[v];
            built.edges += deg[v];
            built.max_degree = std::max(built.max_degree, deg[v]);
        }
        return VGA_OK;
    };
    // after a way that had no room: what it left behind, and its error
    auto start_over = [&]() -> int {
        cudaGetLastError();
        clear_error();
        d_matrix.reset();
        built.degree.reset();
        d_stage.reset();
        d_stage_at.reset();
        d_gbitmap.reset();
        d_glists.reset();
        std::fill(offsets.begin(), offsets.end(), 0);
        VGA_CHECK_CUDA(cudaMemsetAsync(d_counter.ptr, 0, 6 * sizeof(uint32_t), stream));
        VGA_CHECK_CUDA(cudaMemsetAsync(d_err.ptr, 0, sizeof(int), stream));
        return VGA_OK;
    };
    // all octants of every source into CTAs' bitmaps, the lists counted and (kSweepStage) staged
    auto build_sources = [&](SweepMode mode) -> int {
        constexpr uint64_t kStageSmall = 256ull << 20;
        constexpr uint32_t kSampleStep = 128;
        std::vector<uint64_t> rb;
        uint64_t cap = (uint64_t)n * ((uint64_t)n + n / 64 + 32);
        if (mode == kSweepStage && cap > kStageSmall) {
            std::vector<uint32_t> sample;
            for (uint32_t v = kSampleStep / 2; v < n; v += kSampleStep) sample.push_back(v);
            DeviceBuffer d_sample;
            VGA_TRY(d_sample.alloc(sample.size() * 4));
            VGA_CHECK_CUDA(cudaMemcpyAsync(d_sample.ptr, sample.data(), sample.size() * 4, cudaMemcpyHostToDevice,
                                           stream));
            VGA_TRY(sweep(kSweepCount, d_sample.as<uint32_t>(), (uint32_t)sample.size()));
            VGA_TRY(read_row_bytes(rb));
            uint64_t sum = 0;
            for (uint32_t v : sample) sum += rb[v];
            cap = std::min<uint64_t>(cap, (uint64_t)((double)sum / sample.size() * n * 1.05) + 32ull * n);
        }
        if (sa.smem_cap < kSweepCap) cap = std::min<uint64_t>(cap, 64ull * n);   // the test hook fills the stage, too
        if (mode == kSweepStage) {
            VGA_TRY(d_stage_at.alloc((size_t)n * 8));
            VGA_TRY(d_stage.alloc(cap + 16));
        }
        sa.out = d_stage.as<uint8_t>();
        sa.stage_used = reinterpret_cast<unsigned long long *>(d_counter.as<uint32_t>() + 4);
        sa.stage_cap = cap;
        sa.stage_at = d_stage_at.as<uint64_t>();
        VGA_TRY(sweep(mode, nullptr, n));
        unsigned long long used = ~0ull;
        if (mode == kSweepStage)
            VGA_CHECK_CUDA(cudaMemcpyAsync(&used, sa.stage_used, 8, cudaMemcpyDeviceToHost, stream));
        VGA_TRY(read_row_bytes(rb));
        for (uint32_t v = 0; v < n; v++) offsets[v + 1] = offsets[v] + rb[v];
        if (mode == kSweepCount) {
            all_again = true;
        } else if (used > cap) {
            std::vector<uint64_t> at(n);
            VGA_CHECK_CUDA(cudaMemcpy(at.data(), d_stage_at.ptr, (size_t)n * 8, cudaMemcpyDeviceToHost));
            for (uint32_t v = 0; v < n; v++)
                if (at[v] == kNotStaged) again.push_back(v);
        }
        return VGA_OK;
    };
    // each way needs less memory than the one before it
    int rc = VGA_OK;
    if (by_rows) {
        rc = build_rows();
        if (rc == VGA_ENOMEM) {
            by_rows = false;
            VGA_TRY(start_over());
        }
    }
    if (n && !by_rows) {
        rc = build_sources(kSweepStage);
        if (rc == VGA_ENOMEM) {
            VGA_TRY(start_over());
            rc = build_sources(kSweepCount);
        }
    }
    VGA_TRY(rc);
    const uint64_t n_bytes = offsets[n];
    DeviceBuffer d_bytes;
    if (d_bytes.alloc(n_bytes + kBytePad) != VGA_OK) {
        if (!d_stage.ptr && !d_matrix.ptr) return VGA_ENOMEM;
        // no room beside the stage or the matrix: every list is swept again
        cudaGetLastError();
        clear_error();
        d_stage.reset();
        d_stage_at.reset();
        d_matrix.reset();
        all_again = true;
        VGA_TRY(d_bytes.alloc(n_bytes + kBytePad));
    }
    VGA_CHECK_CUDA(cudaMemcpyAsync(d_off.ptr, offsets.data(), ((size_t)n + 1) * 8, cudaMemcpyHostToDevice, stream));
    VGA_CHECK_CUDA(cudaMemsetAsync(d_bytes.as<uint8_t>() + n_bytes, 0, kBytePad, stream));
    if (d_matrix.ptr) {
        rows_encode_kernel<<<(n + kEncodeWarps - 1) / kEncodeWarps, kEncodeWarps * 32, 0, stream>>>(
            sa.matrix, pitch, words_n, n, d_off.as<uint64_t>(), d_bytes.as<uint8_t>(), sa.err);
        count_launch();
        VGA_CHECK_CUDA(cudaGetLastError());
    }
    if (n && d_stage.ptr) {
        stage_gather_kernel<<<(n + 7) / 8, 256, 0, stream>>>(d_stage.as<uint8_t>(), d_stage_at.as<uint64_t>(),
                                                            d_off.as<uint64_t>(), n, d_bytes.as<uint8_t>());
        count_launch();
        VGA_CHECK_CUDA(cudaGetLastError());
    }
    d_stage.reset();
    if (all_again || !again.empty()) {
        DeviceBuffer d_again;
        if (!all_again) {
            VGA_TRY(d_again.alloc(again.size() * 4));
            VGA_CHECK_CUDA(cudaMemcpyAsync(d_again.ptr, again.data(), again.size() * 4, cudaMemcpyHostToDevice,
                                           stream));
        }
        sa.offsets = d_off.as<uint64_t>();
        sa.out = d_bytes.as<uint8_t>();
        VGA_TRY(sweep(kSweepWrite, d_again.as<uint32_t>(), all_again ? n : (uint32_t)again.size()));
    }
    int err = 0;
    VGA_CHECK_CUDA(cudaMemcpyAsync(&err, d_err.ptr, sizeof(int), cudaMemcpyDeviceToHost, stream));
    VGA_CHECK_CUDA(cudaStreamSynchronize(stream));
    if (err) {
        set_error("visibility sweep failed its own checks (code %d)", err);
        return VGA_ECORRUPT;
    }
    d_matrix.reset();
    uint64_t *po = d_off.as<uint64_t>();
    uint8_t *pb = d_bytes.as<uint8_t>();
    d_off.release();
    d_bytes.release();
    if (by_rows) VGA_TRY(make_built_graph(n, n_bytes, po, pb, built, out));
    else VGA_TRY(finish_graph_load(n, n_bytes, po, pb, nullptr, stream, out));
    // the builder knows every node's cell: the grouped union groups 2 x 2 blocks
    (*out)->cells.swap(cells);
    (*out)->cells_W = W;
    (*out)->cells_H = H;
    return VGA_OK;
}

int vga_set_visibility_sweep_limits(int smem_list_cap, uint32_t smem_bitmap_nodes) {
    clear_error();
    if (smem_list_cap < 0 || smem_list_cap > kSweepCap) {
        set_error("vga_set_visibility_sweep_limits: list capacity %d outside 0..%d", smem_list_cap, kSweepCap);
        return VGA_EINVAL;
    }
    g_sweep_smem_cap = smem_list_cap ? smem_list_cap : kSweepCap;
    g_sweep_smem_bitmap_nodes = smem_bitmap_nodes;
    return VGA_OK;
}

int vga_visibility_build(int W, int H, const uint8_t *obst, uint64_t *cell_of_node, vga_graph **out) {
    return vga_visibility_build_ordered(W, H, obst, 0, cell_of_node, out);
}

}  // extern "C"
