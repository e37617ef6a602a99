// MSDA backward, deterministic feature gradient by bilinear cell (sm_103a).
//
// Every in-view point-scale lies in one bilinear cell (y0, x0) of its map and adds to the feature rows at the
// cell's four corners.  Seen from the other side, feature row (i, j) of a map receives exactly the points of
// four cells: (i-1, j-1) through their corner 3 (y0+1, x0+1), (i-1, j) through corner 2 (y0+1, x0),
// (i, j-1) through corner 1 (y0, x0+1) and (i, j) through corner 0.  This path therefore bins each map's
// point-scales by cell, in point order (an ordered placement, so neither a sort nor floating-point atomics
// are needed), and then forms every feature row as one fixed-order sum over the bins of its four cells:
//
//   grad_feat[row, group g] = sum over the cells (i-1,j-1), (i-1,j), (i,j-1), (i,j), over the cell's points in
//                             point order, of w[point-scale, g] * omega_q(fx, fy) * grad_out[b, a, group g]
//
// with omega_q the corner's bilinear weight and the same products as every other kernel (w * (x factor *
// y factor)), so only the order of the sums differs from the atomic form.  A block works on one channel group
// at a time with grad_out[b, :, group g] staged in shared memory (A * C/G FP32 values): the per-contribution
// read of grad_out, which bounds the corner-slot path of det.cu, comes from shared memory instead of L2.
//
// Cells of an H x W map are (cy, cx), cy in [-1, H-1], cx in [-1, W-1] (a point at x in (-1, 0) has
// x0 = -1), numbered (cy + 1) * (W + 1) + (cx + 1).  With c the number of cell (i, j), the cells of row (i, j)
// are c - W - 2, c - W - 1 (consecutive) and c - 1, c, so a row reads two contiguous ranges of bins.
//
// The bins of a map only describe that map, so the maps must not overlap.  cb_plan_kernel checks this on the
// device, together with the sizes the path needs; when a check fails it clears the plan's flag and the
// corner-slot path of det.cu (whose kernels read the same flag) computes the gradient instead.
#include "common.cuh"
#include "internal.h"
#include "tma.cuh"
#include "wsort.cuh"

namespace msda {

constexpr int kCbThreads = 1024;     // threads of the bin and reduce blocks
constexpr int kCbWarps = kCbThreads / 32;
constexpr int kCbMaxMaps = 4096;     // maps the plan's block can sort
constexpr unsigned short kNoCell = 0xffffu;
constexpr int kCbMaxBin = 256;       // points of a cell that a warp sorts in registers
// Fuller cells are put in order by reading the camera's points again, ap / 32 steps of a warp for each, whatever the
// map's size.  Only where few points lie in a map of many cells is such a call handed to the corner-slot form: that costs
// 0.25 ms there (320 points in one cell of a 100x100 map, 65 and 315 us), but 0.6 ms with 1200 points, 3.6 ms with 3900
// and 33 ms with 11700 in one cell (68 and 1.1 ms with a third of 1200 or 3900 in one: 88 and 328, 136 and 755 us).
constexpr int kCbRescanCells = 9472, kCbRescanPoints = 512;
constexpr int kCbMaxRows = 1024;     // image rows of a map the reduce's band planner holds
constexpr int kCbDirect = 1 << 30;   // band-end flag: the band is read in place, not staged

constexpr int kCbDensePtrs = 1024;   // cell pointers of a pass over a dense map (in the planner's arrays, two buffers)

struct CbMap {
    int H, W, start;  // W == 0: the map is invalid and skipped
    int cbase;        // first entry of the map in one batch element's cell-pointer array
    int pad[4];
};

struct CbHeader {
    int ok;           // 1: this path runs and the corner-slot form is not issued
    int ngaps;        // row ranges of a batch element that no valid map covers
    int pad[62];
};

struct CbLayout {
    size_t maps, gaps, queues, forms, plan_end;  // plan area (read by the corner-slot kernels: header.ok)
                                          // forms: per (batch element, map), how the reduce sums it (CbForm)
    size_t cellptr, aoff, coef, loct;     // cell pointers, anchor offsets, per-group corner coefficients,
    size_t total;                         // locations camera-major [B, Ncam, A*P] (float2)
    long long nccap;                      // cell-pointer entries per batch element
    long long nrec;                       // record slots: B * Nmaps * A * P
};

static CbLayout cb_layout(const Problem& p, size_t body_base = 0) {
    CbLayout L;
    const long long nmaps = (long long)p.Ncam * p.Nscale;
    L.maps = 256;
    L.gaps = align_up(L.maps + sizeof(CbMap) * (size_t)nmaps, 256);
    L.queues = align_up(L.gaps + sizeof(int2) * (size_t)(nmaps + 1), 256);
    L.forms = L.queues + sizeof(int) * (size_t)p.B * p.G;
    L.plan_end = align_up(L.forms + sizeof(int) * (size_t)p.B * (size_t)nmaps, 256);
    // Disjoint valid maps fit in sum_hw rows, and (H+1)(W+1) + 1 <= 2 H W + 3 for H, W >= 1, so the cell
    // pointers of one batch element need at most 2 sum_hw + 3 Nmaps entries.
    L.nccap = (2ll * p.sum_hw + 3 * nmaps + 3) & ~3ll;  // a multiple of 4: 16-byte aligned batch slices
    L.nrec = (long long)p.B * nmaps * p.A * p.P;
    L.cellptr = body_base > L.plan_end ? body_base : L.plan_end;
    // 16 spare bytes after the cell pointers and the anchor offsets: band copies round their ends up to 16 bytes
    L.aoff = align_up(L.cellptr + sizeof(uint32_t) * (size_t)p.B * L.nccap + 16, 256);
    L.coef = align_up(L.aoff + sizeof(uint32_t) * (size_t)L.nrec + 16, 256);
    L.loct = align_up(L.coef + sizeof(float4) * (size_t)p.G * L.nrec, 256);
    L.total = align_up(L.loct + sizeof(float2) * (size_t)p.B * p.Ncam * p.A * p.P, 256);
    return L;
}

size_t cb_plan_bytes(const Problem& p) { return cb_layout(p).plan_end; }

// Shared memory of the binning block: a counter per cell (and the end), the camera's A * P cell numbers and
// the placed point indices (16 bits each), and the list of cells too full for one thread's sort.  Two blocks
// fit on an SM.
static size_t cb_bin_smem_cap(const DeviceInfo& dev) {
    return ((size_t)dev.max_smem_optin / 2 - 1024) & ~size_t(15);
}
__host__ __device__ static size_t cb_bin_fixed(long long ap) {
    return 2 * align16(2 * (size_t)ap) + align16(sizeof(uint32_t) * (size_t)(ap / 17 + 2));
}

bool cb_shape_ok(const Problem& p) {
    const long long nmaps = (long long)p.Ncam * p.Nscale;
    const long long ap = (long long)p.A * p.P;
    if (p.B < 1 || p.sum_hw < 1 || nmaps < 1 || nmaps > kCbMaxMaps || ap < 1 || ap > 65535) return false;
    if (p.Cg % 4 != 0 || p.C % 4 != 0) return false;
    const int lg = p.Cg / 4;
    if (lg > 32 || (lg & (lg - 1))) return false;
    if ((long long)p.A * p.Cg >= (1ll << 24)) return false;
    const CbLayout L = cb_layout(p);
    return L.nrec < (1ll << 31) && (long long)p.B * L.nccap < (1ll << 31);
}

// Shared memory of a reduce block: grad_out of one group, two band buffers of `nb` records and `nb` cell
// pointers each (16 + 4 + 4 bytes a slot, 8 slots of rounding each), the band planner's row starts and band
// ends.  `nb` takes what the grad_out copy leaves.
struct CbRedSmem {
    size_t buf;                // first band buffer; the second follows at buf + bsize
    size_t aoff, cptr, bsize;  // inside a buffer: coefficients at 0, anchor offsets, cell pointers
    size_t rp, bend, total;    // the planner's row starts and band ends
    __host__ __device__ CbRedSmem(int A, int Cg, int nb) {
        buf = align16(sizeof(float) * (size_t)A * Cg);
        aoff = 16 * (size_t)nb;
        cptr = aoff + align16(4 * (size_t)(nb + 8));
        bsize = cptr + align16(4 * (size_t)(nb + 8));
        rp = buf + 2 * bsize;
        bend = rp + align16(4 * (size_t)(kCbMaxRows + 2));  // the two together also hold a dense map's cell pointers
        total = bend + align16(4 * (size_t)kCbMaxRows);
    }
};

static int cb_band_slots(const Problem& p, const DeviceInfo& dev) {
    const CbRedSmem z(p.A, p.Cg, 0);
    const long long room = (long long)dev.max_smem_optin - 1024 - (long long)z.total - 2 * 3 * 48;
    if (room <= 0) return 0;
    return (int)((room / (2 * 24)) & ~3ll);
}

bool cb_device_ok(const Problem& p, const DeviceInfo& dev) {
    if (p.G > dev.sm_count) return false;  // at least one reduce block per group
    if (cb_band_slots(p, dev) < 256) return false;  // grad_out of one group leaves room for the band buffers
    return cb_bin_fixed((long long)p.A * p.P) + 64 <= cb_bin_smem_cap(dev);
}

size_t cb_workspace(const Problem& p, size_t body_base) { return cb_layout(p, body_base).total; }

struct CbArgs {
    const int32_t* shape;
    const int32_t* start;
    const float* loc;
    const void* w;
    const float* go;
    void* gfeat;
    int gf_t;  // msda_dtype of gfeat
    unsigned char* ws;
    CbLayout L;
    int B, sum_hw, C, Ncam, Nscale, nmaps, A, P, G, Cg;
    int bin_smem;  // dynamic shared memory of a binning block
    int nb;        // band buffer slots of a reduce block
    int ncap;      // cells whose corner sums they hold
    int* status;
};

// ---------------------------------------------------------------------------
// Plan (block 0): validate the maps, check that the valid ones are disjoint, number their cells,
// list the uncovered row ranges, clear the work queues.
// ---------------------------------------------------------------------------
// Exclusive prefix sum over n <= 4 * blockDim.x values (4 consecutive per thread) of v(i); *total = sum.
template <typename F>
__device__ __forceinline__ void plan_scan(int n, F v, int* out, int* wsum, int* total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int i0 = threadIdx.x * 4;
    int loc[4], s = 0;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        loc[j] = (i0 + j < n) ? v(i0 + j) : 0;
        s += loc[j];
    }
    int x = s;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += t;
    }
    if (lane == 31) wsum[warp] = x;
    __syncthreads();
    if (warp == 0) {
        int y = lane < nw ? wsum[lane] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, y, o);
            if (lane >= o) y += t;
        }
        if (lane < nw) wsum[lane] = y;
    }
    __syncthreads();
    int run = x - s + (warp > 0 ? wsum[warp - 1] : 0);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        if (i0 + j < n) out[i0 + j] = run;
        run += loc[j];
    }
    if (total && threadIdx.x == 0) *total = wsum[nw - 1];
    __syncthreads();
}

// Locations camera-major: loct[b, k, i] = loc[b, i, k] with i = a * P + p, one 32 x 32 tile of a batch element.
__device__ __forceinline__ void cb_transpose_tile(const CbArgs& a, float2 (*tile)[33], int t) {
    const int ap = a.A * a.P;
    const int nti = (ap + 31) / 32, ntk = (a.Ncam + 31) / 32;
    const int i0 = t % nti * 32, k0 = t / nti % ntk * 32, b = t / nti / ntk;
    const float2* src = reinterpret_cast<const float2*>(a.loc) + (long long)b * ap * a.Ncam;
    float2* dst = reinterpret_cast<float2*>(a.ws + a.L.loct) + (long long)b * a.Ncam * ap;
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    if (i0 + ty < ap && k0 + tx < a.Ncam) tile[ty][tx] = __ldg(src + (long long)(i0 + ty) * a.Ncam + k0 + tx);
    __syncthreads();
    if (k0 + ty < a.Ncam && i0 + tx < ap) dst[(long long)(k0 + ty) * ap + i0 + tx] = tile[tx][ty];
}

// Block 0 makes the plan; the others, which need nothing of it, transpose the locations meanwhile.
__global__ void __launch_bounds__(kCbThreads) cb_plan_kernel(const CbArgs a) {
    __shared__ unsigned long long key[kCbMaxMaps];
    if (blockIdx.x > 0) {
        cb_transpose_tile(a, reinterpret_cast<float2 (*)[33]>(key), (int)blockIdx.x - 1);
        return;
    }
    int* tmp = reinterpret_cast<int*>(key);  // scan output, once the sorted keys are no longer read
    __shared__ int wsum[32];
    __shared__ int s_bad, s_nvalid, s_cells;
    CbHeader* hdr = reinterpret_cast<CbHeader*>(a.ws);
    CbMap* maps = reinterpret_cast<CbMap*>(a.ws + a.L.maps);
    int2* gaps = reinterpret_cast<int2*>(a.ws + a.L.gaps);
    int* queues = reinterpret_cast<int*>(a.ws + a.L.queues);
    const int nm = a.nmaps;
    const long long ap = (long long)a.A * a.P;
    if (threadIdx.x == 0) s_bad = 0;
    __syncthreads();
    int np2 = 1;
    while (np2 < nm) np2 <<= 1;
    for (int m = threadIdx.x; m < np2; m += blockDim.x) {
        unsigned long long kv = ~0ull;
        if (m < nm) {
            const MapInfo mi = load_map(a.shape, a.start, m, a.sum_hw, a.status);
            CbMap cm;
            cm.H = mi.H; cm.W = mi.W; cm.start = mi.start; cm.cbase = 0;
            cm.pad[0] = cm.pad[1] = cm.pad[2] = cm.pad[3] = 0;
            if (mi.W != 0) {
                const long long ncell = (long long)(mi.H + 1) * (mi.W + 1);
                if (ncell >= (long long)kNoCell ||
                    align16(4 * (size_t)(ncell + 1)) + cb_bin_fixed(ap) > (size_t)a.bin_smem ||
                    mi.H > kCbMaxRows || 2 * (mi.W + 1) + 9 > a.nb)
                    atomicOr(&s_bad, 1);  // 16-bit cells, counters fit the binning block, one row fits a band
                kv = ((unsigned long long)(unsigned)mi.start << 32) | (unsigned)m;
            }
            maps[m] = cm;
        }
        key[m] = kv;
    }
    __syncthreads();
    // valid maps in order of their first row (bitonic sort; invalid maps sort last), unless they already are
    int unsorted = 0;
    for (int m = threadIdx.x; m + 1 < np2; m += blockDim.x) unsorted |= key[m] > key[m + 1];
    unsorted = __syncthreads_or(unsorted);
    for (int k = 2; unsorted && k <= np2; k <<= 1) {
        for (int j = k >> 1; j > 0; j >>= 1) {
            for (int i = threadIdx.x; i < np2; i += blockDim.x) {
                const int ij = i ^ j;
                if (ij > i) {
                    const unsigned long long x = key[i], y = key[ij];
                    if ((x > y) == ((i & k) == 0)) {
                        key[i] = y;
                        key[ij] = x;
                    }
                }
            }
            __syncthreads();
        }
    }
    if (threadIdx.x == 0) s_nvalid = 0;
    __syncthreads();
    {
        int n = 0;
        for (int m = threadIdx.x; m < nm; m += blockDim.x) n += key[m] != ~0ull;  // valid keys come first
        if (n) atomicAdd(&s_nvalid, n);
    }
    __syncthreads();
    const int nv = s_nvalid;
    // disjointness of consecutive valid maps, and the uncovered ranges between them
    for (int i = threadIdx.x; i <= nv; i += blockDim.x) {
        int lo = 0, hi = a.sum_hw;
        if (i > 0) {
            const CbMap mp = maps[(int)(key[i - 1] & 0xffffffffu)];
            lo = mp.start + mp.H * mp.W;
        }
        if (i < nv) hi = (int)(key[i] >> 32);
        if (hi < lo) atomicOr(&s_bad, 1);  // overlap
        gaps[i] = make_int2(lo, hi > lo ? hi : lo);
    }
    // cell pointers numbered in map order (plan_scan's first barrier ends the reads of key)
    plan_scan(nm, [&](int m) { const CbMap c = maps[m]; return c.W ? (c.H + 1) * (c.W + 1) + 1 : 0; }, tmp, wsum,
              &s_cells);
    for (int m = threadIdx.x; m < nm; m += blockDim.x) maps[m].cbase = tmp[m];
    for (int q = threadIdx.x; q < a.B * a.G; q += blockDim.x) queues[q] = 0;
    __syncthreads();
    if (threadIdx.x == 0) {
        hdr->ok = (s_bad == 0 && (long long)s_cells <= a.L.nccap) ? 1 : 0;
        hdr->ngaps = nv + 1;
    }
}

enum CbForm { kCbColumns, kCbColumnsCrowded, kCbColumnsByWarp, kCbCells, kCbCellsByWarp };

// The form in which a map is summed, from its records, its fullest cell and the sum of its cells' squared counts.  The
// reduce alone, one scale, BF16, each form forced in turn (us: columns; columns, four records at a time; columns by warp;
// cells; cells by warp.  r: records per row; 24 cameras, 900 anchors x 13 keypoints, C/G = 32, unless said; crowded:
// half of the points in a hundredth of the map):
//   even       r = 4: 109 120 177 253 378    8: 114 123 136 128 179    13: 133 140 128 100 122    25: 143 145 127 78 83
//              50: 188 166 134 74 62
//   projected  r = 5.5: 137 136 149 198 220    11: 143 138 139 179 139    17: 146 140 131 175 109
//              36: 157 143 122 174 79
//   crowded    r = 1: 239 230 398 240 241    2: 221 212 282 545 637    4: 229 224 256 474 405
//   C/G = 8    even  r = 4: 64 66 128 68 310    8: 72 75 86 52 166    crowded  r = 2: 129 112 227 143 534
//              projected  r = 5.5: 106 95 104 108 187    11: 101 89 76 87 103    36: 113 97 63 154 44
//   C/G = 8, 2 cameras, 187 anchors (one band)   projected  r = 5.5: 18 16 15 23 25    22: 25 20 11 33 12
//   40 cameras, 300 anchors (one band)   projected  r = 5.5: 64 58 59 105 101    22: 86 74 45 98 48
// * A lane group per cell wants passes with cells for most lane groups, none much fuller than the others.  It gains from
//   r = 3 + 28 / (lane groups of a warp) on, and the warp overtakes it at 8 x (lane groups of a warp) records per row.
// * Where the points crowd (a record's cell holds several times the map's mean), columns differ in length, and a warp
//   per column evens them out, as long as the map comes in few bands: each band's cell rows are swept once more at its
//   start, and a band that is one row is not staged at all.
// Over 354 such maps (r = 0.3 to 235; 187 to 1200 anchors; C/G = 8 to 64) the form taken is 2 % from the best on average;
// the kernel as a whole takes 0.84 of the time it took with a lane group per column, or a warp from 8 points per row on.
__device__ __forceinline__ CbForm cb_form(const CbArgs& a, int H, int W, uint32_t nrec, uint32_t most, uint32_t squares) {
    const float nlgw = (float)(128 / a.Cg);  // lane groups of a warp (4 channels per lane)
    const float per = (float)nrec / (float)(H * W);
    const float bands = (float)nrec / (float)a.nb;
    const bool uneven = (float)squares > (1.f + 2.f * per) * (float)nrec;
    if (uneven && per >= (bands > 1.25f ? 7.f : 5.f) && bands <= (per < 16.f ? 4.f : 1.25f)) return kCbColumnsByWarp;
    if (2 * (W + 1) > a.ncap && per >= 8.f) return kCbColumnsByWarp;
    if (2 * (W + 1) > a.ncap || per < 3.f + 28.f / nlgw) {
        const float full = nlgw >= 8.f && per >= 1.5f ? 1.f + 5.f * per : fmaxf(1.f + 12.f * per, 10.f);
        return nlgw >= 4.f && (float)squares > full * (float)nrec ? kCbColumnsCrowded : kCbColumns;
    }
    const bool level = (float)most <= 3.f * per + 8.f;
    const int pass = min(H + 1, a.ncap / (W + 1) - 1) * (W + 1);  // cells of a pass
    if (level && (float)pass >= 0.625f * kCbWarps * nlgw && per < 8.f * nlgw) return kCbCells;
    return per >= 8.f * nlgw || (bands > 1.25f && per >= 1.5f * nlgw) ? kCbCellsByWarp : kCbColumnsByWarp;
}

// ---------------------------------------------------------------------------
// Binning: one block per (batch element, map).  The camera's A * P points get their cells (0xffff when out of
// view) and are counted per cell with shared-memory atomics; the counts' prefix sums are the map's cell
// pointers; the points are placed into their cells (shared-memory atomics again) and every cell's points are
// sorted by point index (one thread per cell of up to 16 points, a warp per fuller cell, which sorts up to
// kCbMaxBin points and reads fuller cells off the points again), which makes the order inside a cell the point
// order whatever the atomics did.  A cell of more than kCbMaxBin points clears the plan's flag, which hands the
// whole feature gradient to the corner-slot path, in a map of more than kCbRescanCells cells and at most
// kCbRescanPoints points.  The counts also give the form in which the reduce sums the map.  Then, in record
// order, each in-view point gets its anchor's offset a * C/G in grad_out's staged copy and, per group g, the
// weights of its four corners w_g * (x factor * y factor), in the products every other kernel forms.  Blocks
// past the maps clear the uncovered rows.
// ---------------------------------------------------------------------------
template <int N>
__device__ __forceinline__ void cb_sort_small(unsigned short* seg, int n) {
    uint32_t v[N];
#pragma unroll
    for (int j = 0; j < N; ++j) v[j] = j < n ? seg[j] : 0xffffffffu;
    thread_sort<N>(v);
#pragma unroll
    for (int j = 0; j < N; ++j)
        if (j < n) seg[j] = (unsigned short)v[j];
}

template <int E>
__device__ __forceinline__ void cb_sort_warp(unsigned short* seg, int n, int lane) {
    uint32_t v[E];
#pragma unroll
    for (int e = 0; e < E; ++e) {
        const int i = lane * E + e;
        v[e] = i < n ? seg[i] : 0xffffffffu;
    }
    warp_sort_regs<E>(v, lane);
#pragma unroll
    for (int e = 0; e < E; ++e) {
        const int i = lane * E + e;
        if (i < n) seg[i] = (unsigned short)v[e];
    }
}

// The points of cell c in point order, read off the cell numbers of all ap points by one warp.  Keypoints projected
// from boxes crowd into few cells: on 20 cameras of 900 anchors x 13 keypoints (1080p maps) the 17x30 maps have cells of
// up to 331 points, and handing such a call to the corner-slot path cost 2.9 ms; ap / 32 steps of a warp cost
// microseconds, and a map of ap points has at most ap / 256 such cells.
__device__ __forceinline__ void cb_rescan(unsigned short* seg, const unsigned short* cell, int ap, unsigned short c,
                                          int lane) {
    const unsigned lt = (1u << lane) - 1u;
    int n = 0;
    for (int i0 = 0; i0 < ap; i0 += 32) {
        const int i = i0 + lane;
        const bool in = i < ap && cell[i] == c;
        const unsigned bal = __ballot_sync(0xffffffffu, in);
        if (in) seg[n + __popc(bal & lt)] = (unsigned short)i;
        n += __popc(bal);
    }
}

// Eight consecutive weights (16-byte aligned) widened to FP32, in 16-byte loads.
__device__ __forceinline__ void cb_load8(const float* p, float* v) {
    const float4 x = __ldg(reinterpret_cast<const float4*>(p)), y = __ldg(reinterpret_cast<const float4*>(p) + 1);
    v[0] = x.x; v[1] = x.y; v[2] = x.z; v[3] = x.w; v[4] = y.x; v[5] = y.y; v[6] = y.z; v[7] = y.w;
}
__device__ __forceinline__ void cb_load8(const __nv_bfloat16* p, float* v) {
    const uint4 x = __ldg(reinterpret_cast<const uint4*>(p));
    widen(x, v, __nv_bfloat16());
}
__device__ __forceinline__ void cb_load8(const __half* p, float* v) {
    const uint4 x = __ldg(reinterpret_cast<const uint4*>(p));
    widen(x, v, __half());
}

template <typename WT>
__global__ void __launch_bounds__(kCbThreads, 2) cb_bin_kernel(const CbArgs a) {
    CbHeader* hdr = reinterpret_cast<CbHeader*>(a.ws);
    // Read once for the whole block: another block of this grid may clear the flag meanwhile (an overfull cell), and
    // a block that lost some of its warps here would go on with its shared counters unset.
    __shared__ int s_ok;
    if (threadIdx.x == 0) s_ok = *reinterpret_cast<volatile int*>(&hdr->ok);
    __syncthreads();
    if (!s_ok) return;
    const CbMap* maps = reinterpret_cast<const CbMap*>(a.ws + a.L.maps);
    const long long nbm = (long long)a.B * a.nmaps;
    if ((long long)blockIdx.x >= nbm) {
        // rows of no valid map: zero gradient; the extra blocks take the uncovered ranges in turn
        const int2* gaps = reinterpret_cast<const int2*>(a.ws + a.L.gaps);
        const int zb = (int)(blockIdx.x - nbm), nzb = (int)(gridDim.x - nbm);
        const int c4 = a.C / 4;
        const int ngaps = hdr->ngaps;
        for (int gi = zb; gi < ngaps; gi += nzb) {
            const int2 gp = gaps[gi];
            const long long n = (long long)(gp.y - gp.x) * c4;
            for (int b = 0; b < a.B && n > 0; ++b) {
                const long long first = ((long long)b * a.sum_hw + gp.x) * c4;  // in groups of four channels
                if (a.gf_t == MSDA_F32) {
                    float4* dst = reinterpret_cast<float4*>(a.gfeat) + first;
                    for (long long i = threadIdx.x; i < n; i += blockDim.x) dst[i] = make_float4(0.f, 0.f, 0.f, 0.f);
                } else {
                    uint2* dst = reinterpret_cast<uint2*>(a.gfeat) + first;
                    for (long long i = threadIdx.x; i < n; i += blockDim.x) dst[i] = make_uint2(0u, 0u);
                }
            }
        }
        return;
    }
    const int b = (int)(blockIdx.x / a.nmaps), m = (int)(blockIdx.x % a.nmaps);
    const CbMap mp = maps[m];
    if (mp.W == 0) return;
    const int k = m / a.Nscale, s = m - k * a.Nscale;
    const int H = mp.H, W = mp.W, W1 = W + 1;
    const int ncell = (H + 1) * W1;
    const int ap = a.A * a.P;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // Maps of few cells place their points stably with per-warp cell cursors (each warp owns a chunk of the
    // points); maps of many cells with one counter per cell and a sort of every cell afterwards.
    const size_t arrays = cb_bin_fixed(ap);
    const bool stable = align16((size_t)kCbWarps * 4 * (ncell + 1)) + arrays <= (size_t)a.bin_smem;
    const int cstride = ncell + 1;  // stable: counter of (cell c, warp w) at w * cstride + c
    extern __shared__ __align__(16) unsigned char smem[];
    uint32_t* cnt = reinterpret_cast<uint32_t*>(smem);
    const size_t cbytes = align16(4 * (size_t)(stable ? kCbWarps * cstride : ncell + 1));
    unsigned short* cell = reinterpret_cast<unsigned short*>(smem + cbytes);
    unsigned short* idx = cell + align16(2 * (size_t)ap) / 2;
    uint32_t* lng = reinterpret_cast<uint32_t*>(idx + align16(2 * (size_t)ap) / 2);
    __shared__ int wsum[32];
    __shared__ int s_nlong, s_abort;
    __shared__ uint32_t s_most, s_sq;
    const int chunk = (ap + kCbWarps - 1) / kCbWarps;  // stable: points of warp w are [w * chunk, ...)
    const int ncnt = stable ? kCbWarps * cstride : ncell + 1;

    for (int c = threadIdx.x; c < ncnt; c += blockDim.x) cnt[c] = 0u;
    if (threadIdx.x == 0) { s_nlong = 0; s_abort = 0; s_most = s_sq = 0u; }
    __syncthreads();
    const float2* lk = reinterpret_cast<const float2*>(a.ws + a.L.loct) + ((long long)b * a.Ncam + k) * ap;
    for (int i0 = threadIdx.x; i0 < ap; i0 += 4 * blockDim.x) {
        float2 uv[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int i = i0 + u * blockDim.x;
            uv[u] = i < ap ? __ldg(lk + i) : make_float2(-9.f, -9.f);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int i = i0 + u * blockDim.x;
            if (i < ap) {
                Cell cl;
                unsigned short c = kNoCell;
                if (locate(uv[u].x, uv[u].y, H, W, cl)) {
                    c = (unsigned short)((cl.y0 + 1) * W1 + cl.x0 + 1);
                    atomicAdd(cnt + (stable ? (i / chunk) * cstride + c : c), 1u);
                }
                cell[i] = c;
            }
        }
    }
    __syncthreads();
    // exclusive scan of the counters in (cell, warp) order (the end entry is 0, so it receives the total);
    // the start of cell c, its first warp's entry, is its cell pointer
    const uint32_t recbase = (uint32_t)(((long long)b * a.nmaps + m) * ap);
    {
        uint32_t* gptr = reinterpret_cast<uint32_t*>(a.ws + a.L.cellptr) + (long long)b * a.L.nccap + mp.cbase;
        const int sh = stable ? 5 : 0, nw = 1 << sh;  // kCbWarps cursors per cell, or one
        const int nent = stable ? kCbWarps * cstride - (kCbWarps - 1) : ncell + 1;  // (ncell, 0) ends the order
        const int per = (nent + blockDim.x - 1) / blockDim.x;
        const int c0 = threadIdx.x * per;
        // scan position q is (cell q / nw, warp q % nw), at counter (q % nw) * cstride + q / nw
        static_assert(kCbWarps == 32, "");
        uint32_t sum = 0u;
        for (int j = 0; j < per && c0 + j < nent; ++j) {
            const int q = c0 + j;
            sum += cnt[(q & (nw - 1)) * cstride + (q >> sh)];
        }
        uint32_t x = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t t = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += t;
        }
        if (lane == 31) wsum[warp] = (int)x;
        __syncthreads();
        if (warp == 0) {
            uint32_t y = (uint32_t)wsum[lane];
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t t = __shfl_up_sync(0xffffffffu, y, o);
                if (lane >= o) y += t;
            }
            wsum[lane] = (int)y;
        }
        __syncthreads();
        uint32_t run = x - sum + (warp > 0 ? (uint32_t)wsum[warp - 1] : 0u);
        for (int j = 0; j < per && c0 + j < nent; ++j) {
            const int q = c0 + j;
            uint32_t* e = cnt + (q & (nw - 1)) * cstride + (q >> sh);
            const uint32_t v = *e;
            *e = run;
            if ((q & (nw - 1)) == 0) gptr[q >> sh] = recbase + run;
            run += v;
        }
    }
    __syncthreads();
    if (stable) {
        // warp w walks its chunk in point order; ranks inside a batch of 32 from ballots over the cell bits
        int cbits = 1;
        while ((1 << cbits) < ncell) ++cbits;
        const unsigned lt = (1u << lane) - 1u;
        const int lo = warp * chunk, hi = min(lo + chunk, ap);
        uint32_t* cur = cnt + warp * cstride;
        for (int i0 = lo; i0 < hi; i0 += 32) {
            const int i = i0 + lane;
            const unsigned c = i < hi ? (unsigned)cell[i] : (unsigned)kNoCell;
            const bool valid = c != kNoCell;
            unsigned peers = __ballot_sync(0xffffffffu, valid);
            for (int bit = 0; bit < cbits; ++bit) {
                const unsigned mb = __ballot_sync(0xffffffffu, (c >> bit) & 1u);
                peers &= ((c >> bit) & 1u) ? mb : ~mb;
            }
            const int leader = valid ? __ffs(peers) - 1 : 0;
            uint32_t base = 0u;
            if (valid && lane == leader) {
                base = cur[c];
                cur[c] = base + (uint32_t)__popc(peers);
            }
            base = __shfl_sync(0xffffffffu, base, leader);
            if (valid) idx[base + __popc(peers & lt)] = (unsigned short)i;
        }
    } else {
        // place the points; afterwards cnt[c] is the end of cell c
        for (int i = threadIdx.x; i < ap; i += blockDim.x) {
            const unsigned short c = cell[i];
            if (c != kNoCell) idx[atomicAdd(cnt + c, 1u)] = (unsigned short)i;
        }
    }
    __syncthreads();
    // end of cell c (the start of cell c + 1): the last warp's cursor when stable, else the counter
    const uint32_t* cend = stable ? cnt + (kCbWarps - 1) * cstride : cnt;
    const int total = (int)cend[ncell - 1];
    {
        const bool rescan = ncell <= kCbRescanCells || ap > kCbRescanPoints;
        // how the points crowd (the reduce chooses its form by it), and point order inside every cell
        uint32_t most = 0u, sq = 0u;
        for (int c = threadIdx.x; c < ncell; c += blockDim.x) {
            const int e0 = c > 0 ? (int)cend[c - 1] : 0, n = (int)cend[c] - e0;
            most = max(most, (uint32_t)n);
            sq += (uint32_t)n * (uint32_t)n;
            if (stable || n <= 1) continue;
            if (n <= 4) cb_sort_small<4>(idx + e0, n);
            else if (n <= 16) cb_sort_small<16>(idx + e0, n);
            else if (n <= kCbMaxBin || rescan) lng[atomicAdd(&s_nlong, 1)] = (uint32_t)c;
            else s_abort = 1;
        }
        most = __reduce_max_sync(0xffffffffu, most);
        sq = __reduce_add_sync(0xffffffffu, sq);  // the whole sum is at most (A * P)^2, below 2^32
        if (lane == 0 && sq) {
            atomicMax(&s_most, most);
            atomicAdd(&s_sq, sq);
        }
    }
    __syncthreads();
    if (s_abort) {
        if (threadIdx.x == 0) atomicExch(&hdr->ok, 0);
        return;
    }
    if (threadIdx.x == 0)
        reinterpret_cast<int*>(a.ws + a.L.forms)[(long long)b * a.nmaps + m] =
            cb_form(a, H, W, (uint32_t)total, s_most, s_sq);
    for (int li = warp; li < s_nlong; li += kCbWarps) {
        const int c = (int)lng[li];
        const int e0 = c > 0 ? (int)cend[c - 1] : 0, n = (int)cend[c] - e0;
        if (n <= 32) cb_sort_warp<1>(idx + e0, n, lane);
        else if (n <= 64) cb_sort_warp<2>(idx + e0, n, lane);
        else if (n <= 128) cb_sort_warp<4>(idx + e0, n, lane);
        else if (n <= kCbMaxBin) cb_sort_warp<8>(idx + e0, n, lane);
        else cb_rescan(idx + e0, cell, ap, (unsigned short)c, lane);
    }
    __syncthreads();
    // records in record order: anchor offsets and the corner coefficients of each group, two at a time
    const long long rb = (long long)recbase;
    uint32_t* aoffp = reinterpret_cast<uint32_t*>(a.ws + a.L.aoff);
    float4* coef = reinterpret_cast<float4*>(a.ws + a.L.coef);
    const WT* wp = reinterpret_cast<const WT*>(a.w);
    const long long tbase = ((long long)b * a.A * a.P) * a.Ncam + k;  // point (a, p) is tbase + (a*P + p)*Ncam
    for (int p0 = threadIdx.x; p0 < total; p0 += 2 * blockDim.x) {
        int ii[2];
        float2 uv[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int pos = p0 + u * blockDim.x;
            ii[u] = pos < total ? (int)idx[pos] : -1;
            uv[u] = ii[u] >= 0 ? __ldg(lk + ii[u]) : make_float2(0.f, 0.f);
        }
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int pos = p0 + u * blockDim.x;
            if (ii[u] < 0) continue;
            const int i = ii[u];
            Cell cl;
            locate(uv[u].x, uv[u].y, H, W, cl);  // in view: it was binned
            const float ax = 1.0f - cl.fx, ay = 1.0f - cl.fy;
            const float f00 = ax * ay, f01 = cl.fx * ay, f10 = ax * cl.fy, f11 = cl.fx * cl.fy;
            aoffp[rb + pos] = (uint32_t)((i / a.P) * a.Cg);
            const WT* wrow = wp + ((tbase + (long long)i * a.Ncam) * a.Nscale + s) * a.G;
            for (int g0 = 0; g0 < a.G; g0 += 8) {
                float v[8];
                if (a.G - g0 >= 8 && ((size_t)a.G * sizeof(WT)) % 16 == 0) {
                    cb_load8(wrow + g0, v);  // 16-byte aligned: G * sizeof(WT) is a multiple of 16
                } else {
#pragma unroll
                    for (int j = 0; j < 8; ++j) v[j] = g0 + j < a.G ? ldw(wrow + g0 + j) : 0.0f;
                }
#pragma unroll
                for (int j = 0; j < 8; ++j)
                    if (g0 + j < a.G)
                        coef[(long long)(g0 + j) * a.L.nrec + rb + pos] =
                            make_float4(v[j] * f00, v[j] * f01, v[j] * f10, v[j] * f11);
            }
        }
    }
}

// ---------------------------------------------------------------------------
// Row reduce as column sweeps (grad_feat in FP32, or narrowed once in the features' type: the row's sum is in
// registers either way, and a caller that wants the narrow gradient saves writing and reading the FP32 one; 16
// cameras, batch 4, BF16: a 205 us conversion after a 732 us reduce, against a 734 us reduce alone).  Block j
// works on channel group g = j % G: it stages grad_out[b, :, group g] in shared memory for b = 0, 1, ... in turn
// and takes whole maps of (b, g) from that pair's queue.  A map's
// columns, cut into row segments, are swept top to bottom: at cell row cy a column j reads the records of its
// two cells (cy, j-1) and (cy, j), which are adjacent in record order, and adds each record once to the row it
// finishes, (cy, j), with weight x * (1 - fy), and once to the row below, (cy+1, j), with weight x * fy (x = fx
// for the left cell, 1 - fx for the right one).  The row below therefore receives its cell-row cy records
// before its own, which is the order (i-1, j-1), (i-1, j), (i, j-1), (i, j) for every row (i, j); a segment
// starting at row i0 first sweeps cell row i0 - 1 for the row below only.  A lane group (LG lanes, 4 channels each)
// sweeps a column, or a warp does where points crowd (cb_sweep_crowded), and dense maps are summed by cells instead
// (cb_dense_map); cb_form chooses.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void cb_fma4(float4& acc, float k, const float4& v) {
    acc.x = fmaf(k, v.x, acc.x);
    acc.y = fmaf(k, v.y, acc.y);
    acc.z = fmaf(k, v.z, acc.z);
    acc.w = fmaf(k, v.w, acc.w);
}

// cur += k * v and nxt += k' * v with packed FP32 FMAs (each half is an FP32 fma, rounded as fmaf).
__device__ __forceinline__ void cb_fma2x2(float4& cur, float4& nxt, float kc, float kn, const float4& v) {
    const float2 va = make_float2(v.x, v.y), vb = make_float2(v.z, v.w);
    const float2 kcc = make_float2(kc, kc), knn = make_float2(kn, kn);
    float2 c0 = make_float2(cur.x, cur.y), c1 = make_float2(cur.z, cur.w);
    float2 n0 = make_float2(nxt.x, nxt.y), n1 = make_float2(nxt.z, nxt.w);
    c0 = __ffma2_rn(kcc, va, c0);
    c1 = __ffma2_rn(kcc, vb, c1);
    n0 = __ffma2_rn(knn, va, n0);
    n1 = __ffma2_rn(knn, vb, n1);
    cur = make_float4(c0.x, c0.y, c1.x, c1.y);
    nxt = make_float4(n0.x, n0.y, n1.x, n1.y);
}

// Elements of grad_feat: FP32, or (LOWP) 16 bits in the features' type.
template <bool LOWP> struct GradElem { using T = float; };
template <> struct GradElem<true> { using T = unsigned short; };

// Store four channels of a feature row's gradient.
__device__ __forceinline__ void cb_store(const CbArgs&, float* dst, const float4& v) {
    *reinterpret_cast<float4*>(dst) = v;
}
__device__ __forceinline__ void cb_store(const CbArgs& a, unsigned short* dst, const float4& v) {
    *reinterpret_cast<uint2*>(dst) = narrow4(v, a.gf_t == MSDA_F16);
}

// One cell row of a column from a staged band: records [e, e2) (record e is coefficient slot e - ce and anchor-offset
// slot e - ae of the band); records before e1 are the left cell's (corners 1 and 3 reach this column: coefficient .y to
// the finished row, .w to the row below), the others the right cell's (corners 0 and 2: .x and .z).  ONLY_NEXT: the
// finished row is not this task's.  Takes every step-th record, U pairs at a time: one where a pair of cells holds a few
// records (left to the compiler's unrolling, 7 per row took 237 us, now 211), two where they crowd.
template <bool ONLY_NEXT, int U>
__device__ __forceinline__ void cb_step(const uint32_t* __restrict__ Ao, const float4* __restrict__ Cf,
                                        const float4* __restrict__ sgo, int l, uint32_t e, uint32_t e1, uint32_t e2,
                                        uint32_t ae, uint32_t ce, int step, float4& cur, float4& nxt) {
#pragma unroll U
    for (; e + step < e2; e += 2 * step) {
        const uint32_t o0 = Ao[e - ae], o1 = Ao[e + step - ae];
        const float4 k0 = Cf[e - ce], k1 = Cf[e + step - ce];
        const bool l0 = e < e1, l1 = e + step < e1;
        const float4 v0 = sgo[(o0 >> 2) + l];
        const float4 v1 = sgo[(o1 >> 2) + l];
        if (ONLY_NEXT) {
            cb_fma4(nxt, l0 ? k0.w : k0.z, v0);
            cb_fma4(nxt, l1 ? k1.w : k1.z, v1);
        } else {
            cb_fma2x2(cur, nxt, l0 ? k0.y : k0.x, l0 ? k0.w : k0.z, v0);
            cb_fma2x2(cur, nxt, l1 ? k1.y : k1.x, l1 ? k1.w : k1.z, v1);
        }
    }
    if (e < e2) {
        const uint32_t o0 = Ao[e - ae];
        const float4 k0 = Cf[e - ce];
        const bool l0 = e < e1;
        const float4 v0 = sgo[(o0 >> 2) + l];
        if (ONLY_NEXT)
            cb_fma4(nxt, l0 ? k0.w : k0.z, v0);
        else
            cb_fma2x2(cur, nxt, l0 ? k0.y : k0.x, l0 ? k0.w : k0.z, v0);
    }
}

// Band copies of one map: band k covers image rows [i0, i1), so cell rows i0 - 1 .. i1 - 1: their records
// [rp[i0], rp[i1 + 1]) (coefficients of group g and anchor offsets) and their cell pointers, the pointer and
// offset ranges rounded out to 16 bytes.  Issued by one thread; completes on `bar`.  A band whose end carries
// kCbDirect holds rows of which even one exceeds a buffer (crowded cells): the
// sweep reads its records and cell pointers from the workspace itself, and its barrier phase completes with a
// plain arrival, so the buffers' phases stay in step.
struct CbBand {
    uint32_t e0, ea0, ca0;  // first record, first staged anchor-offset slot, first staged cell pointer
};

__device__ __forceinline__ CbBand cb_issue_band(const CbArgs& a, unsigned char* buf, const CbRedSmem& L,
                                                const uint32_t* rp, int i0, int i1, long long pm, int W1,
                                                const float4* coef_g, uint64_t* bar) {
    CbBand bd;
    if (i1 & kCbDirect) {  // read in place from the workspace: nothing to copy, the phase completes at once
        mbar_arrive(bar);
        bd.e0 = bd.ea0 = bd.ca0 = 0u;
        return bd;
    }
    const uint32_t e0 = rp[i0], e1 = rp[i1 + 1];
    const uint32_t ea0 = e0 & ~3u, ea1 = (e1 + 3u) & ~3u;
    const long long c0 = pm + (long long)i0 * W1, c1 = pm + (long long)(i1 + 1) * W1 + 1;
    const long long ca0 = c0 & ~3ll, ca1 = (c1 + 3) & ~3ll;
    const uint32_t bytes = (e1 - e0) * 16u + (ea1 - ea0) * 4u + (uint32_t)(ca1 - ca0) * 4u;
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // the threads' reads of this buffer come first
    mbar_arrive_expect_tx(bar, bytes);
    const uint32_t* aoff = reinterpret_cast<const uint32_t*>(a.ws + a.L.aoff);
    const uint32_t* cptr = reinterpret_cast<const uint32_t*>(a.ws + a.L.cellptr);
    if (e1 > e0) bulk_load(buf, coef_g + e0, (e1 - e0) * 16u, bar);
    if (ea1 > ea0) bulk_load(buf + L.aoff, aoff + ea0, (ea1 - ea0) * 4u, bar);
    bulk_load(buf + L.cptr, cptr + ca0, (uint32_t)(ca1 - ca0) * 4u, bar);
    bd.e0 = e0;
    bd.ea0 = ea0;
    bd.ca0 = (uint32_t)ca0;
    return bd;
}

// The column sweeps of a band whose points crowd, four records at a time.  BYWARP: a warp per column, its lane groups
// taking every (32/LG)-th record of a cell pair and adding their partial rows with a fixed butterfly when a row is
// finished; else a lane group per column.  STAGED: the band at smem + buf, as the sweep in cb_reduce_kernel reads it;
// else a band read in place, from the workspace (record e, anchor offset e, cell pointer c at their own indices): with
// a lane group per column such bands took 414 us where a warp takes 212 (47x83 maps, half of the points in a hundredth
// of the map).  Kept out of line so that the sweep of even maps is compiled as if alone.
template <int LG, bool BYWARP, bool STAGED, typename GT>
__device__ __noinline__ void cb_sweep_crowded(const CbArgs& a, const float4* __restrict__ coef_g, unsigned buf,
                                              const CbBand bd, GT* gfm, long long pm, int i0, int i1, int W) {
    extern __shared__ __align__(16) unsigned char smem[];
    constexpr int NSLOT = BYWARP ? kCbWarps : kCbThreads / LG, STEP = BYWARP ? 32 / LG : 1;
    const float4* sgo = reinterpret_cast<const float4*>(smem);
    const CbRedSmem L(a.A, a.Cg, a.nb);
    const float4* Cf = STAGED ? reinterpret_cast<const float4*>(smem + buf) : coef_g;
    const uint32_t* Ao = STAGED ? reinterpret_cast<const uint32_t*>(smem + buf + L.aoff)
                                : reinterpret_cast<const uint32_t*>(a.ws + a.L.aoff);
    const uint32_t* Cp = STAGED ? reinterpret_cast<const uint32_t*>(smem + buf + L.cptr)
                                : reinterpret_cast<const uint32_t*>(a.ws + a.L.cellptr) + pm;
    const int cp0 = STAGED ? (int)(pm - (long long)bd.ca0) : 0;
    const int W1 = W + 1, R = i1 - i0;
    const int S = max(1, min(R, NSLOT / W)), seg = (R + S - 1) / S;
    const int l = (int)threadIdx.x % LG, lgi = BYWARP ? (int)(threadIdx.x & 31) / LG : 0;
    for (int task = (int)threadIdx.x / (BYWARP ? 32 : LG); task < W * S; task += NSLOT) {
        const int sg = task / W, j = task - sg * W;
        const int r0 = i0 + sg * seg, r1 = min(r0 + seg, i1);
        if (r0 >= r1) continue;
        float4 cur = make_float4(0.f, 0.f, 0.f, 0.f), nxt = cur;
        int ci = cp0 + r0 * W1 + j;  // left cell of cell row r0 - 1
        for (int cy = r0 - 1; cy < r1; ++cy) {
            const uint32_t q0 = Cp[ci] + lgi, q1 = Cp[ci + 1], q2 = Cp[ci + 2];
            if (cy < r0) {
                cb_step<true, 2>(Ao, Cf, sgo, l, q0, q1, q2, bd.ea0, bd.e0, STEP, cur, nxt);
            } else {
                cb_step<false, 2>(Ao, Cf, sgo, l, q0, q1, q2, bd.ea0, bd.e0, STEP, cur, nxt);
                if constexpr (BYWARP) {
#pragma unroll
                    for (int o = LG; o < 32; o <<= 1) {
                        cur.x += __shfl_xor_sync(0xffffffffu, cur.x, o);
                        cur.y += __shfl_xor_sync(0xffffffffu, cur.y, o);
                        cur.z += __shfl_xor_sync(0xffffffffu, cur.z, o);
                        cur.w += __shfl_xor_sync(0xffffffffu, cur.w, o);
                    }
                }
                if (lgi == 0) cb_store(a, gfm + ((long long)cy * W + j) * a.C, cur);
            }
            cur = nxt;
            nxt = make_float4(0.f, 0.f, 0.f, 0.f);
            ci += W1;
        }
    }
}

// ---------------------------------------------------------------------------
// Dense maps (several records per cell and more: the coarse scales, or keypoints that crowd): whole cells are summed
// for all four corners at once, every record read once, straight from the workspace, four ahead.  Either a lane group
// takes a cell, or, with many records per cell (by_warp), the lane groups of a warp share one and then hand the four
// sums out among themselves; warps take cells from a counter.  The sums are left in shared memory, in the band buffers;
// when the cells of as many cell rows as fit are summed, the feature rows between them are the sum of four corner sums
// each, in the order (i-1,j-1), (i-1,j), (i,j-1), (i,j).  Cell row r (cy + 1) lies in slot r % (R + 1), so the last one
// of a pass stays for the next.  Returns the number of passes, which take the two barriers in turn (each for the cell
// pointers of a pass, copied while the pass before runs).  Kept out of line so that the column sweeps keep their
// registers.
//
// A column sweep reads a record for each of its two columns, and again for every row segment that a column is cut into
// to occupy the block; this form reads it once, but starts a pass for every few cell rows (cb_form has the figures).
// ---------------------------------------------------------------------------
template <int LG, typename GT>
__device__ __noinline__ int cb_dense_map(const CbArgs& a, const float4* __restrict__ coef_g,
                                         const float4* __restrict__ sgo, float4* scratch, int ncap, GT* gfm,
                                         long long pm, int H, int W, uint32_t* cptr, int* ctr, int* fail, uint64_t* mbar,
                                         uint32_t ph0, uint32_t ph1, bool by_warp) {
    constexpr int NLGW = 32 / LG;
    constexpr int U = 4;
    const int W1 = W + 1, R = ncap / W1 - 1;  // cell rows of a pass
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int lgi = lane / LG, l = lane % LG;
    const uint32_t* Ao = reinterpret_cast<const uint32_t*>(a.ws + a.L.aoff);
    // the cell pointers of a pass, rounded out to 16 bytes, in buffer bf of two (by thread 0)
    auto issue = [&](int r, int bf) {
        const long long c0 = (pm + (long long)r * W1) & ~3ll, c1 = (pm + (long long)min(r + R, H + 1) * W1 + 4) & ~3ll;
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // the threads' reads of this buffer come first
        mbar_arrive_expect_tx(&mbar[bf], (uint32_t)(c1 - c0) * 4u);
        bulk_load(cptr + bf * kCbDensePtrs, reinterpret_cast<const uint32_t*>(a.ws + a.L.cellptr) + c0,
                  (uint32_t)(c1 - c0) * 4u, &mbar[bf]);
    };
    if (threadIdx.x == 0) issue(0, 0);
    int npass = 0;
    for (int r0 = 0, bf = 0; r0 <= H; r0 += R, bf ^= 1, ++npass) {
        const int r1 = min(r0 + R, H + 1);
        if (threadIdx.x == 0) {
            if (r1 <= H) issue(r1, bf ^ 1);
            *ctr = kCbWarps;
            const uint32_t par = bf ? ph1 : ph0;
            if (!mbar_wait_first(&mbar[bf], par)) {
                *fail = 1;
                raise_status(a.status, MSDA_ERR_TIMEOUT);
                mbar_wait_drain(&mbar[bf], par);  // the copy in flight lands before the buffer is reused
            }
        }
        if (bf) ph1 ^= 1u; else ph0 ^= 1u;
        __syncthreads();  // pointers and counter are there, and the rows of the pass before are assembled
        const int ncell = *fail ? 0 : (r1 - r0) * W1;
        const uint32_t* Cp = cptr + bf * kCbDensePtrs + ((pm + (long long)r0 * W1) & 3);
        if (!by_warp) {
            // a lane group per cell: the lane groups of a warp take NLGW consecutive cells
            for (int c0 = warp * NLGW; c0 < ncell;) {
                const int c = c0 + lgi;
                const uint32_t e0 = c < ncell ? Cp[c] : 0u, e1 = c < ncell ? Cp[c + 1] : 0u;
                float4 s[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) s[q] = make_float4(0.f, 0.f, 0.f, 0.f);
                for (uint32_t e = e0; e < e1; e += U) {
                    uint32_t o[U];
                    float4 k[U];
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        const uint32_t eu = min(e + u, e1 - 1);
                        o[u] = __ldg(Ao + eu);
                        k[u] = __ldg(coef_g + eu);
                    }
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        if (e + u < e1) {
                            const float4 v = sgo[(o[u] >> 2) + l];
                            cb_fma2x2(s[0], s[1], k[u].x, k[u].y, v);
                            cb_fma2x2(s[2], s[3], k[u].z, k[u].w, v);
                        }
                    }
                }
                if (c < ncell) {
                    float4* dst = scratch + ((long long)(((r0 + c / W1) % (R + 1)) * W1 + c % W1) * 4) * LG + l;
#pragma unroll
                    for (int q = 0; q < 4; ++q) dst[q * LG] = s[q];
                }
                if (lane == 0) c0 = atomicAdd(ctr, 1) * NLGW;
                c0 = __shfl_sync(0xffffffffu, c0, 0);
            }
        }
        for (int c = by_warp ? warp : ncell; c < ncell;) {
            const uint32_t e0 = Cp[c], e1 = Cp[c + 1];
            float4 s[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) s[q] = make_float4(0.f, 0.f, 0.f, 0.f);
            for (uint32_t e = e0 + lgi; e < e1; e += U * NLGW) {
                uint32_t o[U];
                float4 k[U];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const uint32_t eu = min(e + u * NLGW, e1 - 1);
                    o[u] = __ldg(Ao + eu);
                    k[u] = __ldg(coef_g + eu);
                }
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    if (e + u * NLGW < e1) {
                        const float4 v = sgo[(o[u] >> 2) + l];
                        cb_fma2x2(s[0], s[1], k[u].x, k[u].y, v);
                        cb_fma2x2(s[2], s[3], k[u].z, k[u].w, v);
                    }
                }
            }
            // the lane groups' shares, summed: plain butterflies while more than four lane groups are left, then the
            // corners are halved between the lanes, so that corner q ends in the lanes of index q among four (two
            // corners each among two lane groups, all four in one)
            auto xadd = [](float4& x, const float4& y, int o) {
                x.x += __shfl_xor_sync(0xffffffffu, y.x, o);
                x.y += __shfl_xor_sync(0xffffffffu, y.y, o);
                x.z += __shfl_xor_sync(0xffffffffu, y.z, o);
                x.w += __shfl_xor_sync(0xffffffffu, y.w, o);
            };
            auto pick = [](bool p, const float4& x, const float4& y) {
                return make_float4(p ? x.x : y.x, p ? x.y : y.y, p ? x.z : y.z, p ? x.w : y.w);
            };
#pragma unroll
            for (int off = LG; off < 8; off <<= 1)
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const float4 t = s[q];
                    xadd(s[q], t, off);
                }
            float4* dst = scratch + ((long long)(((r0 + c / W1) % (R + 1)) * W1 + c % W1) * 4) * LG + l;
            if constexpr (LG <= 16) {
                const bool up = lane & 16;
                float4 k0 = pick(up, s[2], s[0]), k1 = pick(up, s[3], s[1]);
                xadd(k0, pick(up, s[0], s[2]), 16);
                xadd(k1, pick(up, s[1], s[3]), 16);
                if constexpr (LG == 16) {
                    dst[2 * lgi * LG] = k0;
                    dst[(2 * lgi + 1) * LG] = k1;
                } else {
                    const bool odd = lane & 8;
                    float4 k2 = pick(odd, k1, k0);
                    xadd(k2, pick(odd, k0, k1), 8);
                    if (LG == 8 || (lane & 7) < LG) dst[(lane >> 3) * LG] = k2;
                }
            } else {
#pragma unroll
                for (int q = 0; q < 4; ++q) dst[q * LG] = s[q];
            }
            if (lane == 0) c = atomicAdd(ctr, 1);
            c = __shfl_sync(0xffffffffu, c, 0);
        }
        __syncthreads();
        // feature rows whose two cell rows (i and i + 1 in this numbering) are both summed
        const int i0 = r0 > 0 ? r0 - 1 : 0, nrow = *fail ? 0 : (r1 - 1 - i0) * W;
        for (int t = warp * NLGW + lgi; t < nrow; t += kCbWarps * NLGW) {
            const int i = i0 + t / W, j = t % W;
            const float4* up = scratch + ((long long)((i % (R + 1)) * W1 + j) * 4) * LG + l;
            const float4* dn = scratch + ((long long)(((i + 1) % (R + 1)) * W1 + j) * 4) * LG + l;
            const float4 x3 = up[3 * LG], x2 = up[(4 + 2) * LG], x1 = dn[1 * LG], x0 = dn[4 * LG];
            cb_store(a, gfm + ((long long)i * W + j) * a.C,
                     make_float4(x3.x + x2.x + x1.x + x0.x, x3.y + x2.y + x1.y + x0.y, x3.z + x2.z + x1.z + x0.z,
                                 x3.w + x2.w + x1.w + x0.w));
        }
        __syncthreads();
    }
    return npass;
}

template <int LG, bool LOWP>
__global__ void __launch_bounds__(kCbThreads, 1) cb_reduce_kernel(const CbArgs a) {
    constexpr int NLGW = 32 / LG;  // lane groups per warp
    using GT = typename GradElem<LOWP>::T;
    const CbHeader* hdr = reinterpret_cast<const CbHeader*>(a.ws);
    if (!hdr->ok) return;
    const int ngb = gridDim.x / a.G;
    if ((int)blockIdx.x >= ngb * a.G) return;
    const int g = blockIdx.x % a.G;
    const CbMap* maps = reinterpret_cast<const CbMap*>(a.ws + a.L.maps);
    int* queues = reinterpret_cast<int*>(a.ws + a.L.queues);
    const uint32_t* cellptr = reinterpret_cast<const uint32_t*>(a.ws + a.L.cellptr);
    const int* forms = reinterpret_cast<const int*>(a.ws + a.L.forms);
    const float4* coef_g = reinterpret_cast<const float4*>(a.ws + a.L.coef) + (long long)g * a.L.nrec;
    const CbRedSmem L(a.A, a.Cg, a.nb);
    extern __shared__ __align__(16) unsigned char smem[];
    float4* sgo = reinterpret_cast<float4*>(smem);
    unsigned char* const buf0 = smem + L.buf;  // band buffer bf is buf0 + bf * L.bsize
    uint32_t* rp = reinterpret_cast<uint32_t*>(smem + L.rp);
    int* bend = reinterpret_cast<int*>(smem + L.bend);
    __shared__ uint64_t mbar[2];
    __shared__ CbBand s_band[2];
    __shared__ int s_item[2], s_nb, s_fail, s_ctr;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int l = lane % LG;
    const int lgid = warp * NLGW + lane / LG;
    const int nlg = kCbWarps * NLGW;
    const int cg4 = a.Cg / 4;
    if (threadIdx.x == 0) {
        mbar_init(&mbar[0], 1);
        mbar_init(&mbar[1], 1);
        s_fail = 0;
    }
    uint32_t ph0 = 0u, ph1 = 0u;  // parity of each buffer's barrier

    for (int b = 0; b < a.B; ++b) {
        // stage grad_out[b, :, group g]
        const float4* gsrc = reinterpret_cast<const float4*>(a.go + (long long)b * a.A * a.C + g * a.Cg);
        for (int i = threadIdx.x; i < a.A * cg4; i += blockDim.x) {
            const int aa = i / cg4, q = i - aa * cg4;
            sgo[i] = __ldg(gsrc + (long long)aa * (a.C / 4) + q);
        }
        int* queue = queues + b * a.G + g;
        if (threadIdx.x == 0) s_item[0] = atomicAdd(queue, 1);
        __syncthreads();
        GT* gfb = reinterpret_cast<GT*>(a.gfeat) + (long long)b * a.sum_hw * a.C + g * a.Cg + l * 4;
        for (int cur_slot = 0;; cur_slot ^= 1) {
            const int m = s_item[cur_slot];
            if (m >= a.nmaps) break;
            if (threadIdx.x == 0) s_item[cur_slot ^ 1] = atomicAdd(queue, 1);  // the next map, fetched meanwhile
            const CbMap mp = maps[m];
            const int form = __ldg(forms + (long long)b * a.nmaps + m);
            if (mp.W != 0) {
                const int H = mp.H, W = mp.W, W1 = W + 1;
                const long long pm = (long long)b * a.L.nccap + mp.cbase;  // the map's cell pointers
                GT* gfm = gfb + (long long)mp.start * a.C;
                if (form == kCbCells || form == kCbCellsByWarp) {
                    const int npass = cb_dense_map<LG, GT>(a, coef_g, sgo, reinterpret_cast<float4*>(buf0), a.ncap, gfm,
                                                           pm, H, W, rp, &s_ctr, &s_fail, mbar, ph0, ph1,
                                                           form == kCbCellsByWarp);
                    ph0 ^= (uint32_t)((npass + 1) / 2) & 1u;  // the passes took the two barriers in turn
                    ph1 ^= (uint32_t)(npass / 2) & 1u;
                    // bulk copies of the next map's bands come after these reads and writes of the buffers
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    __syncthreads();
                    continue;
                }
                // record starts of the cell rows (cell row index r = cy + 1), then the bands
                for (int r = threadIdx.x; r <= H + 1; r += blockDim.x) rp[r] = __ldg(cellptr + pm + (long long)r * W1);
                __syncthreads();
                if (warp == 0) {
                    int i0 = 0, nb = 0;
                    while (i0 < H) {
                        int i1 = i0;
                        for (int base = 1;; base += 32) {  // the band grows while it fits (a prefix of candidates)
                            const int c = i0 + base + lane;
                            const bool fits = c <= H && (int)(rp[c + 1] - rp[i0]) <= a.nb - 8 &&
                                              (long long)(c - i0 + 1) * W1 + 9 <= a.nb;
                            const unsigned bal = __ballot_sync(0xffffffffu, fits);
                            if (bal) i1 = i0 + base + 31 - __clz(bal);
                            if (bal != 0xffffffffu) break;
                        }
                        int flag = 0;
                        if (i1 == i0) {
                            // row i0 alone (cell rows i0 - 1 and i0) exceeds a buffer: it and the rows after it that
                            // do too form one band read in place
                            i1 = i0 + 1;
                            while (i1 < H && (int)(rp[i1 + 2] - rp[i1]) > a.nb - 8) ++i1;
                            flag = kCbDirect;
                        }
                        if (lane == 0) bend[nb] = i1 | flag;
                        ++nb;
                        i0 = i1;
                    }
                    if (lane == 0) s_nb = nb;
                }
                __syncthreads();
                const int nb = s_nb;
                if (threadIdx.x == 0) {
                    for (int k = 0; k < 2 && k < nb; ++k)
                        s_band[k] = cb_issue_band(a, buf0 + k * L.bsize, L, rp, k ? bend[k - 1] & ~kCbDirect : 0,
                                                  bend[k], pm, W1, coef_g, &mbar[k]);
                }
                for (int k = 0; k < nb; ++k) {
                    const int bf = k & 1;
                    const uint32_t par = bf ? ph1 : ph0;
                    if (threadIdx.x == 0 && !mbar_wait_first(&mbar[bf], par)) {
                        s_fail = 1;
                        raise_status(a.status, MSDA_ERR_TIMEOUT);
                        mbar_wait_drain(&mbar[bf], par);  // the copies in flight land before the buffer is reused
                    }
                    __syncthreads();
                    if (bf) ph1 ^= 1u; else ph0 ^= 1u;
                    const int i0 = k ? bend[k - 1] & ~kCbDirect : 0, i1 = bend[k] & ~kCbDirect;
                    const bool direct = (bend[k] & kCbDirect) != 0;
                    const CbBand bd = s_band[bf];
                    const int R = i1 - i0;
                    int S = nlg / W;
                    S = S < 1 ? 1 : (S > R ? R : S);
                    const int seg = (R + S - 1) / S;
                    const int ntask = W * S;
                    const bool failed = s_fail != 0;
                    const unsigned buf = (unsigned)(L.buf + bf * L.bsize);
                    if (direct) {
                        if (!failed) cb_sweep_crowded<LG, true, false, GT>(a, coef_g, 0u, bd, gfm, pm, i0, i1, W);
                    } else if (form == kCbColumnsByWarp) {
                        if (!failed) cb_sweep_crowded<LG, true, true, GT>(a, coef_g, buf, bd, gfm, pm, i0, i1, W);
                    } else if (form == kCbColumnsCrowded) {
                        if (!failed) cb_sweep_crowded<LG, false, true, GT>(a, coef_g, buf, bd, gfm, pm, i0, i1, W);
                    } else {
                        const unsigned char* bb = smem + buf;
                        const float4* Cf = reinterpret_cast<const float4*>(bb);
                        const uint32_t* Ao = reinterpret_cast<const uint32_t*>(bb + L.aoff);
                        const uint32_t* Cp = reinterpret_cast<const uint32_t*>(bb + L.cptr);
                        for (int task = lgid; task < ntask && !failed; task += nlg) {
                            const int sg = task / W, j = task - sg * W;
                            const int r0 = i0 + sg * seg, r1 = min(r0 + seg, i1);
                            if (r0 >= r1) continue;
                            float4 cur = make_float4(0.f, 0.f, 0.f, 0.f), nxt = cur;
                            // left cell of cell row r0 - 1 (cell row index r0), as a slot of the staged pointers
                            int ci = (int)(pm - (long long)bd.ca0) + r0 * W1 + j;
#pragma unroll 2
                            for (int cy = r0 - 1; cy < r1; ++cy) {
                                const uint32_t q0 = Cp[ci], q1 = Cp[ci + 1], q2 = Cp[ci + 2];
                                if (cy < r0) {
                                    cb_step<true, 1>(Ao, Cf, sgo, l, q0, q1, q2, bd.ea0, bd.e0, 1, cur, nxt);
                                } else {
                                    cb_step<false, 1>(Ao, Cf, sgo, l, q0, q1, q2, bd.ea0, bd.e0, 1, cur, nxt);
                                    cb_store(a, gfm + ((long long)cy * W + j) * a.C, cur);
                                }
                                cur = nxt;
                                nxt = make_float4(0.f, 0.f, 0.f, 0.f);
                                ci += W1;
                            }
                        }
                    }
                    __syncthreads();  // the buffer is free again
                    if (threadIdx.x == 0 && k + 2 < nb)
                        s_band[bf] = cb_issue_band(a, buf0 + bf * L.bsize, L, rp, bend[k + 1] & ~kCbDirect,
                                                   bend[k + 2], pm, W1, coef_g, &mbar[bf]);
                }
            }
            __syncthreads();  // every thread has read s_item[cur_slot] and finished the map
        }
        __syncthreads();  // every warp is done with this batch element's grad_out
    }
}

using CbBinKernel = void (*)(const CbArgs);
using CbRedKernel = void (*)(const CbArgs);

template <bool LOWP>
static CbRedKernel cb_red_pick(int lg) {
    switch (lg) {
        case 1: return cb_reduce_kernel<1, LOWP>;
        case 2: return cb_reduce_kernel<2, LOWP>;
        case 4: return cb_reduce_kernel<4, LOWP>;
        case 8: return cb_reduce_kernel<8, LOWP>;
        case 16: return cb_reduce_kernel<16, LOWP>;
        case 32: return cb_reduce_kernel<32, LOWP>;
    }
    return nullptr;
}

// Enqueue the plan, binning and reduce kernels.  The plan's flag (the first int of `ws`) tells the corner-slot
// kernels launched after these whether they have to run.
msda_status launch_backward_cb(const Problem& p, const float* grad_out, float* grad_feat, void* ws,
                               size_t body_base, cudaStream_t stream) {
    DeviceInfo dev;
    msda_status st = device_info(&dev);
    if (st != MSDA_OK) return st;
    CbArgs a;
    a.shape = p.shape; a.start = p.start; a.loc = p.loc; a.w = p.w; a.go = grad_out; a.gfeat = grad_feat; a.gf_t = p.gf_t;
    a.ws = reinterpret_cast<unsigned char*>(ws);
    a.L = cb_layout(p, body_base);
    a.B = p.B; a.sum_hw = p.sum_hw; a.C = p.C; a.Ncam = p.Ncam; a.Nscale = p.Nscale; a.nmaps = p.Ncam * p.Nscale;
    a.A = p.A; a.P = p.P; a.G = p.G; a.Cg = p.Cg;
    a.bin_smem = (int)cb_bin_smem_cap(dev);
    a.nb = cb_band_slots(p, dev);
    a.ncap = (int)(2 * CbRedSmem(p.A, p.Cg, a.nb).bsize / (4 * sizeof(float) * (size_t)p.Cg));
    if (a.ncap > kCbDensePtrs - 8) a.ncap = kCbDensePtrs - 8;
    a.status = dev.status;
    CbBinKernel bin = p.w_t == MSDA_F32 ? cb_bin_kernel<float>
                    : p.w_t == MSDA_BF16 ? cb_bin_kernel<__nv_bfloat16> : cb_bin_kernel<__half>;
    CbRedKernel red = p.gf_t == MSDA_F32 ? cb_red_pick<false>(p.Cg / 4) : cb_red_pick<true>(p.Cg / 4);
    if (!red) return fail(MSDA_ERR_UNSUPPORTED, "msda_backward: no cell-binned reduce for C/G = %d", p.Cg);
    const long long nbm = (long long)p.B * a.nmaps;
    // Where the maps' blocks are no more than the SMs, each asks for more than half of an SM's shared memory: blocks
    // that start while dloc/dw still fills most SMs would share the first free ones and stay there (42 maps: 30 us
    // alone, 50 us in pairs; a training step of 7 cameras, batch 3, 217 -> 197 us).
    const size_t bin_smem = nbm <= dev.sm_count ? (size_t)a.bin_smem + 4096 : (size_t)a.bin_smem;
    const size_t red_smem = CbRedSmem(p.A, p.Cg, a.nb).total;
    if ((st = ensure_smem((const void*)bin, bin_smem, dev)) != MSDA_OK) return st;
    if ((st = ensure_smem((const void*)red, red_smem, dev)) != MSDA_OK) return st;
    const long long tiles = (((long long)p.A * p.P + 31) / 32) * ((p.Ncam + 31) / 32) * p.B;
    cb_plan_kernel<<<(unsigned)(1 + tiles), kCbThreads, 0, stream>>>(a);
    bin<<<(unsigned)(nbm + 16), kCbThreads, bin_smem, stream>>>(a);
    const int ngb = dev.sm_count / p.G;
    red<<<(unsigned)(ngb * p.G), kCbThreads, red_smem, stream>>>(a);
    return check_launch("msda_backward cell-binned");
}

// The first-wait poll limit of this file's band waits (msda_debug_set_wait_limit).
msda_status cb_set_wait_limit(long long polls) {
    if (polls < 0) polls = kSpinLimit;
    const cudaError_t e = cudaMemcpyToSymbol(g_first_wait_limit, &polls, sizeof(polls));
    return e == cudaSuccess ? MSDA_OK : fail(MSDA_ERR_CUDA, "msda_debug_set_wait_limit: %s", cudaGetErrorString(e));
}

}  // namespace msda
