// State of the coarse-grained decomposition (Algorithm 3) shared by its two
// drivers: the per-round kernels of cd.cu and the one-launch form of
// cd_persist.cu.
#pragma once

#include "engine.cuh"
#include "internal.cuh"

namespace receipt {

constexpr int NBUCKET = LOG_BUCKETS;
constexpr int NTIER = 5;  // warp, hybrid, global, sliced, dense window
constexpr double DGM_FRAC = 0.125;  // stale share of live entries that triggers a compaction

struct CdDev {
    unsigned long long hi;
    int32_t nF, nNext, nLw, nLc, nLg, nLo, nLs, nLb, nLd;
    int32_t par;      // device-driven rounds: which of two buffers holds the activeSet
    int32_t burst_k;  // device-driven rounds: rounds run by the current graph launch
    int32_t pad2;
    int32_t work[6];
    unsigned long long work64;  // item counter of the sliced tier
    unsigned long long peeled_edges;  // adjacency entries of assigned vertices (for DGM)
    int32_t n_remaining;
    int32_t range;  // 0-based index of the range being peeled
    unsigned long long wrem_prev;
    double tgt_prev;
    unsigned long long wedges;
    // per tier: wedges, mids, anchors, nonzero pairs (support atomics)
    unsigned long long tier_w[NTIER], tier_m[NTIER], tier_a[NTIER], tier_p[NTIER];
    unsigned long long front_w;  // sum of wfull over a full-scan activeSet (C_peel)
    unsigned long long hist_w[NBUCKET];
    uint32_t hist_c[NBUCKET];
};

// ---------------------------------------------------------------------
// One-launch form (cd_persist.cu)
// ---------------------------------------------------------------------
// A peeled vertex with updates to make: its edges [q0, q0 + deg) and the key
// window [kb, kb + w) of this item. Every remaining vertex it can share a
// butterfly with lies in its items' windows: one item, or, past DENSE_KEYS
// keys, several (`part` numbers them, -1 for the only one).
struct alignas(16) PersistAnchor {
    int64_t q0;
    int32_t x, deg, kb, w, part;
    uint32_t wedges;  // of group anchors
};
constexpr int PERSIST_SLICES = 4;        // items of one anchor, at most
constexpr int PERSIST_WIDE_SLICES = 16;  // with groups for the short walks

// One round of the one-launch form, counters cumulative over the call
// (warp-table anchors, dense-window anchors).
struct PersistRound {
    int32_t range, frontier;
    unsigned long long hi, anchors[2], wedges[2];
};

// How anchors are counted: dense windows, groups of warps too, or by lists made
// beforehand.
enum { PERSIST_WINDOWS = 0, PERSIST_GROUPS = 1, PERSIST_LISTS = 2 };
enum { PERSIST_RANGE = 0, PERSIST_PEEL = 1, PERSIST_SCAN = 2 };          // where to go on
enum { PERSIST_DONE = 0, PERSIST_RECOUNT = 1, PERSIST_RECORDS_FULL = 2 };  // why it stopped

struct PersistDev {
    unsigned int bar;  // grid barrier: arrivals since the launch
    int32_t err;       // a barrier wait ran out
    int32_t mode, stop, range, nrec, dgm_passes;
    int32_t hk, sk;  // histograms, scans made so far
    int32_t pad;
    unsigned long long hi, peeled, peeled_at_dgm, wrem_prev;
    double tgt_prev;
    // an activeSet: its size, its anchors per tier, work counters, wedges
    // (C_peel), adjacency entries, wedges of the anchors with updates. Three
    // sets in turn: the current scan's, the next one's (cleared), the last
    // one's (perhaps still being read by a CTA that has yet to go on)
    struct Set {
        int32_t nF, nLw, nLd, workW, workD, nG[3];
        unsigned long long front_w, front_e, upd_w;
    } set[3];
};

struct PersistArgs {
    int32_t n, n_o;
    int64_t m;
    const int64_t *off_s;
    const int32_t *adj_s;
    const int64_t *off_o;
    int32_t *len_o;  // working copy of the other side's lists: lengths, keys
    int32_t *adj_o;
    unsigned long long *sup, *init;
    const unsigned long long *wfull;
    int32_t *sub;
    CdDev *st;
    PersistDev *pd;
    unsigned long long *hist_w;  // 3 x NBUCKET: the current histogram, the next one
    uint32_t *hist_c;            // (cleared), the last one (perhaps still being read)
    const int32_t *part_of;      // packed graph of every vertex (null: one graph)
    const int32_t *pfirst;       // first vertex of every packed graph
    int32_t *plast;              // 3 x nparts, beside the histograms: last remaining vertex
    int32_t nparts;
    int32_t *F;
    PersistAnchor *Lw, *Ld;
    PersistAnchor *Lg;  // 3 x n: anchors for groups of 1, up to 4, up to 16 warps
    PersistRound *rec;
    int32_t rec_cap;
    int32_t P, range_cap, warp_max_w, dgm;
    double dgm_frac;
    int32_t huc;  // the recount rule is on
    double huc_factor;
    const unsigned long long *crcnt;
    const uint32_t *pool;            // update lists (PERSIST_LISTS)
    const unsigned long long *list;  // where each vertex's lies
    int32_t group;                   // dense-window anchors per fetch, at most
};

// Whether a decomposition can run in the one-launch form.
bool cd_persist_fits(const Decomp &D);
// ... and whether lists of every vertex's updates should be made for it.
bool cd_persist_by_lists(const Decomp &D);
// ... with the short walks counted by groups of warps (`wide` below).
bool cd_persist_wide(const Decomp &D);
// CTAs of the one-launch form for m edges.
int cd_persist_grid(int64_t m, int form);
// Dense-window anchors that a CTA may fetch at once.
int cd_persist_group(const Decomp &D);
// Enqueues one launch (state in a.pd).
void cd_persist_launch(const PersistArgs &a, int grid, int form, cudaStream_t s);

// ---------------------------------------------------------------------
// Updates of a large activeSet through the other side's hubs (cd_hub.cu)
// ---------------------------------------------------------------------
struct HubDev {
    int32_t nA, nE;          // anchors, their edges past the hubs
    int32_t nQs, nQ;         // rows of the quadratic form: sparse, the others
    int32_t nR, nMid, nBig;  // pulling vertices; those of warp and of CTA size
    int32_t nTouch, cursor, work, work_mid;
    uint32_t flags[16];      // tiles of the second digit that are not zero
};

struct HubArgs {
    int32_t n;
    const int64_t *off_s;
    const int32_t *adj_s;
    unsigned long long *sup;
    const int32_t *sub;
    CdDev *st;
    const int32_t *A;        // anchors (st->nLb of them)
    const uint32_t *mask;    // hub masks of side s, 8 words each
    const int32_t *plen;     // hubs among every vertex's neighbours
    const uint32_t *heavy;   // masks of the other side over the heavy vertices
    int2 *cb;                // per other-side vertex: adjacent anchors, start of their list
    int32_t *touch;          // other-side vertices with an adjacent anchor
    int32_t *Qs, *Q, *R, *mid, *big;
    int32_t *aoff;           // per anchor: first of its edges past the hubs
    uint32_t *amask, *cols;  // anchors' hub masks and their transpose
    int32_t colw;
    uint32_t *gram;          // G as B fragments, two digits
    uint32_t *gtri;          // G's strictly lower triangle, row by row
    int32_t *ey;             // per edge past the hubs: its middle vertex,
    int2 *ek;                // its anchor and its place in the middle vertex's list
    int32_t *alist;
    HubDev *hd;
};

class HubPath {
  public:
    static constexpr int HUBS = 256;
    static constexpr int32_t MAX_ANCHORS = DENSE_KEYS;  // one dense window
    // Whether a decomposition can and should use it: half of the wedges pass
    // through hubs, and a vertex that is not heavy has a degree below 65,535
    // (16-bit counters). Synchronises s.
    static bool suits(const Decomp &D, cudaStream_t s);
    HubPath() = default;
    ~HubPath();
    HubPath(const HubPath &) = delete;
    HubPath &operator=(const HubPath &) = delete;
    // Masks and work space of one decomposition, `bytes` of them at most. False
    // (and nothing kept) when there is no memory for them.
    bool init(const Decomp &D, cudaStream_t s);
    static size_t bytes(int64_t m, int64_t n, int64_t n_o);
    // Enqueues the updates of the anchors A (st->nLb of them, at most nF,
    // assigned to their subset already) to every remaining vertex's support.
    void round(const Decomp &D, CdDev *st, const int32_t *A, int32_t nF, cudaStream_t s);

  private:
    DevBuf<uint32_t> mask_, heavy_, amask_, cols_, gram_, gtri_;
    DevBuf<int32_t> plen_, touch_, Qs_, Q_, R_, mid_, big_, aoff_, ey_, alist_;
    DevBuf<int2> cb_, ek_;
    DevBuf<HubDev> hd_;
    cudaEvent_t ev_[5] = {};
};

}  // namespace receipt
