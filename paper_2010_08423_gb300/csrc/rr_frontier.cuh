// rr_frontier.cuh -- structures of the frontier engine (rr_frontier.cu): one
// query evaluated over the rows that matter to it, in wedge form.
#pragma once
#include <cstdint>

#include "rr_device.cuh"
#include "rr_internal.h"

namespace rr {

// Largest number of reduced labels (k - 1) the engine takes: its subset tables
// hold every subset of [kXMaxLabels], and a row of C(15, 7) = 6,435 values is
// what a block's shared memory holds twice.
constexpr uint32_t kXMaxLabels = 15;
constexpr uint32_t kXMaxLevels = kXMaxLabels + 1;  // levels 1..k-1
constexpr uint32_t kXMaxLL = 2 * kXMaxLevels;      // level lists of one query

// A row list as the engine reads it: rows in head order, windows as the
// half-open range [lo, hi) of 0-based positions in the list of the level before.
struct XList {
    const uint32_t *head, *eid, *src, *lo, *hi, *time;
    uint32_t count;
    uint32_t words;  // bitmap words: count / 32 + 1
};
enum XListId : uint32_t {
    kXProd = 0, kXState = 1, kXDeep1 = 2, kXDeep3 = 3, kXWin = 4, kXTail = 5, kXTail3 = 6, kXAll = 7, kXLists = 8
};

// One query. Scratch pointers are the template's (XTmpl), the rest its own.
struct XQuery {
    uint32_t source, k, K, pivot;         // K: labels of the wedge
    uint32_t colored, dead, multi, nslist; // multi: a set of sources (slist, nslist vertices; smask, n flags)
    uint64_t key_y, key_z, key_g, key_o;
    uint64_t d0;                          // z_{s,pivot}
    uint64_t rho[kXMaxLabels + 1];        // z_{s,j'} / z_{s,pivot} for reduced label j
    uint64_t *S;                          // witness rows (n values each)
    uint64_t *E;                          // per-edge sums (by input edge) or null
    uint32_t *R;                          // minimum arrival times (n per witness row) or null
    uint8_t *bitmap;
    const uint8_t *vmask;                 // deleted vertices or null
    const uint32_t *slist;
    const uint8_t *smask;
    uint32_t index, done;                 // batch form: place in the call's list; its results are written
    uint8_t first[256], mu[256];          // coloured: first shade and multiplicity per colour
};

// One level of one query over one row list. Store levels keep their rows'
// values for the next level; out levels add to a witness. The pointers are
// offsets + 1 into the scratch until the kernel adds its base (0: none).
struct XLL {
    uint32_t list, level, prev, out;  // prev: the store level below (itself at level 1)
    uint32_t d, cin, cout, uout;      // d: subset size of the values; cin / cout: values read / kept per row;
                                      // uout: store levels below an out level: values kept for it per row
    uint32_t words, row, ipcap, sums; // row: out levels' witness row; sums: summaries, in the template's `clear` (x_sums)
    uint32_t *A, *N;                  // active rows, needed rows (bitmaps)
    uint2 *rank;                      // per word of N: the word and the needed rows before it
    uint32_t *tsum;                   // rows per scan tile (256)
    uint4 *meta;                      // per needed row: window [x, y) in needed rows of prev, edge, tail
    uint32_t *mhead, *mtime;          // heads; out levels with arrivals: times
    uint64_t *R, *U;                  // store levels: prefix sums of the cout values and of the uout ones
    uint64_t *sup;                    // sums of 16, 256 and 4,096 blocks (R's, then U's)
    uint64_t *IP;                     // sums of all blocks up to each, of ipcap blocks at most (R's, then U's)
    uint64_t *Ec;                     // out levels with arrivals: per-row sums
};

struct XRun {
    uint32_t first, count;  // level lists [first, first + count) of one level
};

// The levels of a k-vertex query and their scratch.
struct XTmpl {
    uint32_t nll, maxlev, clear4, every;
    uint4 *clear;          // needed-row bitmaps and summaries to clear
    uint32_t *cnt;         // per level list: needed rows
    uint32_t *shape;       // per level list: log2 warps per team | rows per item << 8 | scanned << 16
    unsigned long long *span;  // per store level: rows of it in the windows of the level above, together
    uint64_t *omega;       // coloured: shade factors omega'_{d,j}, k x K
    XRun runs[kXMaxLevels + 1];
    XLL ll[kXMaxLL];
};

struct XArgs {
    XList lists[kXLists];
    uint32_t n, nq;
    XQuery *xq;            // batch form (device); null: the launch's own parameter block
    const XTmpl *xt;       // batch form: by k
    uint8_t *scratch;      // `lanes` regions of `stride` bytes
    uint64_t stride;
    uint32_t lanes;
    uint64_t *szero;       // witnesses and bitmaps to clear
    uint64_t szero_n;
    uint8_t *bzero;
    uint64_t bzero_n;
    uint32_t *ctl;         // [0], [32] barriers, [1] blocks done, [2] next query, [3] queries left, [4] next of them,
                           // [5] batch form with status: its err
    uint32_t *left;        // batch form: the queries left to the bitmap passes
    int32_t *status;       // batch form: by index, RR_ETIMEDOUT for queries unfinished when a wait gave up, or null
    uint32_t *err;         // set when a bounded wait gave up: the host's flag, with status ctl[5]
    uint64_t limit;        // of such a wait (ns)
    uint32_t absent;       // (tests) the last block leaves before this meeting: 1 the first, 2 a batch's second
    const uint8_t *color;
    const uint32_t *tab, *packed;  // subset tables
    const uint32_t *ooff;  // edges by (tail, time): offsets (n + 1),
    const uint4 *orec;     // head, time, input index, first edge that may follow
    const uint32_t *olen;  // and how many
    const uint32_t *skip;  // set: the query is not wanted any more (or null)
    uint32_t smem;         // dynamic shared memory of a block
    uint32_t tiny;         // try every query in one block's shared memory first
};

struct XOne {
    XQuery q;
    XTmpl t;
};

}  // namespace rr
