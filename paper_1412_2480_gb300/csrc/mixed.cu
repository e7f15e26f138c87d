// mixed.cu -- the MIXED32 particle half of the step.
//
// Particles: int32 cell (i | j << 16) + FP32 in-cell offsets (ox, oy) in [0,1) + FP32
// momenta: 24 bytes per particle, structure-of-arrays, binned by (tile, species); a tile
// is tx x ty cells. Each bin has a stayer segment (capacity cap) and eight outboxes
// (capacity capo each), one per neighbouring tile. Bins are double-buffered: a step reads
// buffer `parity` and writes buffer `parity ^ 1`.
//
// A handle may hold many simulations of different sizes and shape orders (the batched
// parameter scan). Their tiles form one global list; each simulation's bins and count
// slots sit at its own offsets.
//
// Per step (inside the captured step graph):
//   0. k_mixed_begin clears the current and the next buffer's counts; k_push_overflow:
//      particles parked in the overflow list (no room in a bin; normally none) are pushed
//      straight from global memory;
//   1. k_push_tile<P>, one persistent launch per shape order P present: each CTA takes
//      the next tile of that order, or part of a tile (tile_plan.h), from a device work
//      counter (tiles listed largest first, so uneven simulations balance across the
//      SMs), stages the FP32 field window (tile + 2 cells below, 3 above, in x and y)
//      into shared memory and zeroes a fixed-point current window of the same size. Its
//      particles are its own stayer segment plus the eight neighbours' outboxes addressed
//      to it. Warps run independently (no block barrier in the particle loop): each
//      gathers E^n, B^n, pushes (Boris), moves and deposits J^{n+1/2} (Esirkepov) with
//      native integer shared-memory atomics, then writes each particle to the next
//      buffer's stayer segment or to the outbox of the neighbour it moved into, taking
//      slots from warp-aggregated counters. The current window is added to the global
//      fixed-point current at the end;
//   2. k_mixed_end, after the field update: the buffers swap.
// No migration kernel runs, and in steady state global atomics only add the windows and,
// where a tile is split, take slots (one per warp and destination). A particle found
// outside its tile is pushed with the same arithmetic and the same current rounding on
// global memory, so results never depend on bin capacity; a particle that finds no room
// goes to the overflow list and the host re-sorts with larger bins after the pic_step
// call. Count slots record every particle sent to a segment, parked ones included;
// readers clamp them to the segment's capacity.
#include <algorithm>
#include <cmath>
#include <mutex>
#include <vector>

#include "density_fixed.h"
#include "esirkepov.cuh"
#include "inject.cuh"
#include "mixed.h"
#include "tile_plan.h"

namespace pic {

constexpr int kTileThreads = 256;
static_assert(kTileThreads == kPartUnit, "parts of whole rounds of a CTA");
constexpr double kBinSlack = 1.25;  // stayer capacity over the expected particles of a tile
constexpr int kNbr = 8;          // outboxes per bin, one per neighbouring tile
constexpr int kSegs = 1 + kNbr;  // count slots per bin: [0] stayers, [1 + o] outbox o

struct PartArrays {  // staging: one plain array per attribute
    int* cij;
    float *ox, *oy, *ux, *uy, *uz;
    int* gs;
};

// Bins and overflow lists: AoSoA of 32-particle chunks, each chunk holding its 32 cells,
// then 32 x-offsets, y-offsets, ux, uy, uz (6 x 128 bytes): a warp touches whole lines
// and one base pointer addresses every attribute.
constexpr int kFields = 6;
struct Slots {
    unsigned* p;
    int* gs;  // species of each slot (overflow lists only)
};

__host__ __device__ __forceinline__ size_t aos(long long k, int f) {
    return (size_t)(k >> 5) * (32 * kFields) + (size_t)f * 32 + (size_t)(k & 31);
}

struct MixedArgs {
    const GridDev* grids;
    const int* tile_grid;  // simulation of each global tile
    const int2* items;     // work of this launch's shape order: (tile, part), largest tiles first
    int nitems;
    int* work;             // next item to take (zeroed every step)
    long long ntot;
    const float* F32;
    long long* Jfix;
    unsigned* buf[2];
    int* cnt[2];     // [nbins * kSegs] per parity: particles sent to each segment
    int* ovf_in[2];  // [ntiles_total] per parity: particles the overflow kernel moved in
    Slots ovf[2];
    long long ovf_cap;
    CgState* cg;
    DevStatus* st;
};

struct MixedState {
    int ngrids = 0;
    GridDev* G = nullptr;  // host descriptors [ngrids], owned by the caller
    const GridDev* dgrids = nullptr;
    long long ntot = 0;
    float* F32 = nullptr;
    long long* Jfix = nullptr;
    CgState* cg = nullptr;
    DevStatus* st = nullptr;
    unsigned* buf[2] = {nullptr, nullptr};
    Slots ovf[2]{};
    int* cnt[2] = {nullptr, nullptr};  // [ntiles_total * 2 * kSegs] per parity, then ovf_in
    int* ovf_in[2] = {nullptr, nullptr};  // [ntiles_total] per parity (inside cnt's block)
    long long nslots = 0, ovf_cap = 0;
    int ntiles_total = 0;
    int* tile_grid = nullptr;     // device [ntiles_total]
    std::vector<int> host_tile_grid;
    std::vector<int> tlist;       // tiles grouped by shape order, largest first
    int order_first[4] = {0, 0, 0, 0}, order_n[4] = {0, 0, 0, 0};
    int2* items = nullptr;        // device: (tile, part) of each order's launch, in tlist's order
    int item_first[4] = {0, 0, 0, 0}, item_n[4] = {0, 0, 0, 0};
    int* work = nullptr;          // device [4]: work counter of each order's launch
    size_t smem[4] = {0, 0, 0, 0};  // dynamic shared memory of each order's launch
    int resident[4] = {0, 0, 0, 0}; // CTAs of each order's launch the device holds at once
    int nsm = 0;                  // SMs of the device
    int pblocks[4] = {0, 0, 0, 0};  // persistent CTAs of each order's launch
    std::vector<long long> n;     // live particles [2 g + species]
    std::vector<double> expect;   // particles of a tile of simulation g, both species, on average
    unsigned long long* injected = nullptr;  // device [2 ngrids]: pairs added by the injector
    int inject_grids = 0;         // simulations with an injector
    long long inject_threads = 0; // rows x most pairs per row, over those simulations
    int* inj_grid = nullptr;      // device [inject_grids]: their indices
    long long* inj_first = nullptr;  // device [inject_grids + 1]: first thread of each
    long long rebins = 0;
    long long gen = 0;  // allocation generation of the bin buffers
    bool lost = true;   // no bins, or none that the descriptors and counts fit: nothing may run on them
};

namespace {

__host__ __device__ __forceinline__ long long bin_stride(const GridDev& G) {
    return G.cap + kNbr * G.capo;
}

// Outbox index of a move by (dx, dy) tiles, (dx, dy) != (0, 0).
__host__ __device__ __forceinline__ int outbox_of(int dx, int dy) {
    const int d = (dy + 1) * 3 + (dx + 1);
    return d < 4 ? d : d - 1;
}

__host__ __device__ __forceinline__ void dir_of(int o, int& dx, int& dy) {
    const int d = o < 4 ? o : o + 1;
    dx = d % 3 - 1;
    dy = d / 3 - 1;
}

// The tile (within its simulation) whose bin holds segment k of the particles tile
// (txi, tyi) pushes: its own stayers (k = 0), or the outbox k - 1 of the neighbour on the
// opposite side, which is addressed to it.
__device__ __forceinline__ int segment_source(const GridDev& G, int txi, int tyi, int k) {
    if (k == 0) return tyi * G.ntx + txi;
    int dx, dy;
    dir_of(k - 1, dx, dy);
    const int sx = (txi - dx + G.ntx) % G.ntx, sy = (tyi - dy + G.nty) % G.nty;
    return sy * G.ntx + sx;
}

// Particles of species s sent to segment k of bin `src` in the last step (count slots of
// the current buffer). The count includes those that found no room and were parked in
// the overflow list; the segment itself holds at most its capacity of them.
__device__ __forceinline__ int segment_sent(const GridDev& G, const int* ccur, int src, int s, int k) {
    return ccur[((long long)G.tile_first * 2 + (long long)src * 2 + s) * kSegs + k];
}

// Particles whose cell lies in tile lt at the start of the step, both species, wherever
// they are stored: those sent to its segments (parked ones included) and those the
// overflow kernel moved into it. This count does not depend on which particles found
// room in the bins, so neither does the rounding it sets.
__device__ __forceinline__ int tile_population(const GridDev& G, const int* ccur, const int* oin, int lt) {
    const int tyi = lt / G.ntx, txi = lt - tyi * G.ntx;
    int n = oin[G.tile_first + lt];
    for (int s = 0; s < 2; s++)
        for (int k = 0; k < kSegs; k++) n += segment_sent(G, ccur, segment_source(G, txi, tyi, k), s, k);
    return n;
}

// Tile (within its simulation) of cell (i, j).
__device__ __forceinline__ int tile_of(const GridDev& G, int i, int j) { return (j / G.ty) * G.ntx + i / G.tx; }

// ---------------------------------------------------------------------------------
// Memory views used by the shared push arithmetic.
// ---------------------------------------------------------------------------------
// The tile's current window accumulates fixed point in two 32-bit words per node: 32-bit
// integer shared atomics are single native instructions, while float and 64-bit ones
// loop on compare-and-swap. Every single-particle contribution to a node is bounded by
// u/2 (GridDev::jscale = 2^40/u). A contribution v becomes x = v 2^k/u, split into its
// nearest integer hi and the rest r = x - hi in [-1/2, 1/2], and lo = round(r 2^lb);
// integers come from one FMA with 1.5 * 2^23 (exact below 2^22 in magnitude). Each tile
// picks k, lb <= 30 - log2(n + 1) from its population n, the particles whose cell lies in
// it (no word can wrap, whatever the distribution), with k <= 22 and lb <= 16, i.e. a
// resolution of 2^-(k+lb) u. The flush adds hi 2^(40-k) + lo 2^(40-k-lb) exactly into
// the 64-bit global current.
// A particle pushed on global memory (outside its tile's window, or parked in the
// overflow list) rounds the same way, with the k and lb of the tile its cell lies in, so
// a particle's current does not depend on the path it takes and a run is bit-for-bit
// reproducible whichever particles find room in the bins.
constexpr float kMagic = 12582912.0f;  // 1.5 * 2^23
constexpr int kMagicBits = 0x4B400000;

struct FixedScale {
    int k, lb;
    float js;   // window scale 2^k / u
    float jlb;  // 2^lb
};

__device__ __forceinline__ FixedScale fixed_scale(const GridDev& G, int n_tile) {
    const int room = 30 - (32 - __clz(n_tile));  // n_tile < 2^(30 - room)
    FixedScale f;
    f.k = min(22, room);
    f.lb = min(16, room);
    f.js = G.js40 * __int_as_float((127 + f.k) << 23);  // js40 2^k: exact, = jscale 2^(k-40) rounded
    f.jlb = (float)(1 << f.lb);
    return f;
}

// x (window units) -> the two words (hi, lo)
__device__ __forceinline__ void fixed_split(float x, float jlb, int& hi, int& lo) {
    const float xr = xadd(x, kMagic);
    hi = __float_as_int(xr) - kMagicBits;
    const float r = xsub(x, xsub(xr, kMagic));  // exact: |r| <= 1/2
    lo = __float_as_int(xfma(r, jlb, kMagic)) - kMagicBits;
}

// Two contributions at once (the same four roundings each): two FP32 operations per issue
// slot. At order 3 (48 to 65 contributions per particle, 16 warps per SM) instructions and
// their latency bound the tile kernel (issue 61% active, shared-memory data path 68%): half
// full 8192 x 512 with 16 per cell and species 4837 -> 4530 us per step, a twelve-run scan of
// all orders 1190 -> 1150. At order 2 issue (70%) and the data path (73% in a cold beam, 78%
// in a hot plasma, most of it bank conflicts of the atomics) bound it together and 2048 x 512
// stays at 2.69 ms.
__device__ __forceinline__ void fixed_split2(float x0, float x1, F2 jlb2, int hi[2], int lo[2]) {
    const F2 m = f2_dup(kMagic), x = f2(x0, x1);
    const F2 xr = add2(x, m);
    const F2 r = sub2(x, add2(xr, f2_dup(-kMagic)));
    const float2 h = f2_get(xr), l = f2_get(fma2(r, jlb2, m));
    hi[0] = __float_as_int(h.x) - kMagicBits;
    hi[1] = __float_as_int(h.y) - kMagicBits;
    lo[0] = __float_as_int(l.x) - kMagicBits;
    lo[1] = __float_as_int(l.y) - kMagicBits;
}

// (hi, lo) summed in a window -> global fixed-point units
__device__ __forceinline__ long long fixed_value(long long hi, long long lo, const FixedScale& f) {
    return hi * (1ll << (40 - f.k)) + lo * (1ll << (40 - f.k - f.lb));
}

// The tile's field window pairs the components that share a lattice -- (Ex, By) at
// (i+1/2, j) and (Ey, Bx) at (i, j+1/2) -- as float2, so one 64-bit load serves two
// components; Ez and Bz follow as plain arrays: [(Ex,By) x NW][(Ey,Bx) x NW][Ez][Bz].
struct WinMem {  // tile window in shared memory; indices are window-local
    const float* fw;
    int* jhi;
    int* jlo;
    int wx, nw;
    float js;   // window scale 2^k / u
    float jlb;  // 2^lb
    __device__ __forceinline__ float2 ld_exby(int ix, int iy) const {
        return reinterpret_cast<const float2*>(fw)[iy * wx + ix];
    }
    __device__ __forceinline__ float2 ld_eybx(int ix, int iy) const {
        return reinterpret_cast<const float2*>(fw + 2 * nw)[iy * wx + ix];
    }
    __device__ __forceinline__ float ld_ez(int ix, int iy) const { return fw[4 * nw + iy * wx + ix]; }
    __device__ __forceinline__ float ld_bz(int ix, int iy) const { return fw[5 * nw + iy * wx + ix]; }
    // x: the contribution already in window units (the push folds js into its deposit
    // constants). A lane whose high word is zero leaves it alone for Jy and Jz (c, a
    // constant once the deposit is unrolled): below half a window unit, as the transverse
    // currents of a relativistic beam are, a contribution lives in the low word only, and
    // an atomic with fewer active lanes takes fewer shared-memory wavefronts (its bank
    // conflicts are among the active lanes). Jx, large along the beam, skips the test.
    // Adding zero changes nothing, so the current is the same to the bit.
    __device__ __forceinline__ void add_words(int c, int k, int hi, int lo) const {
        if (c == 0 || hi != 0) atomicAdd(&jhi[k], hi);
        atomicAdd(&jlo[k], lo);
    }
    // Contributions go in pairs, each held until its partner comes (the deposit is unrolled,
    // so which is which is known when it is compiled).
    struct Adder {
        const WinMem& M;
        bool have;
        int c0, k0;
        float x0;
        bool on0;
        __device__ __forceinline__ void operator()(int c, int ix, int iy, float x, bool on) {
            const int k = c * M.nw + iy * M.wx + ix;
            if (!have) {
                have = true;
                c0 = c;
                k0 = k;
                x0 = x;
                on0 = on;
                return;
            }
            have = false;
            int hi[2], lo[2];
            fixed_split2(x0, x, f2_dup(M.jlb), hi, lo);
            if (on0) M.add_words(c0, k0, hi[0], lo[0]);
            if (on) M.add_words(c, k, hi[1], lo[1]);
        }
        __device__ __forceinline__ void last() {  // the one without a partner
            if (!have) return;
            have = false;
            int hi, lo;
            fixed_split(x0, M.jlb, hi, lo);
            if (on0) M.add_words(c0, k0, hi, lo);
        }
    };
    __device__ __forceinline__ Adder adder() const { return Adder{*this, false, 0, 0, 0.f, false}; }
};

struct GlobalMem {  // global grid arrays of one simulation; indices are global
    const float* F;
    unsigned long long* J;
    long long ntot;
    int nx, ny;
    FixedScale f;  // the rounding of the tile the particle's cell lies in
    float js;      // = f.js: contributions arrive in that tile's window units
    int walls;
    __device__ __forceinline__ long long at(int ix, int iy) const {
        return (long long)wrapi(iy, ny) * nx + wrapi(ix, nx);
    }
    __device__ __forceinline__ float ld(int c, int ix, int iy) const {
        if (!walls) return __ldg(F + c * ntot + at(ix, iy));
        const bool half = c == 0 || c == 4 || c == 5;  // Ex, By, Bz at half-integer x
        int s;
        const int cx = wall_col(ix, nx, half, !half, s);
        return s == 0 ? 0.f : (float)s * __ldg(F + c * ntot + (long long)wrapi(iy, ny) * nx + cx);
    }
    // x: the contribution in window units (times js), rounded as the window rounds it
    struct Adder {
        const GlobalMem& M;
        __device__ __forceinline__ void operator()(int c, int ix, int iy, float x, bool on) {
            if (on) M.add(c, ix, iy, x);
        }
        __device__ __forceinline__ void last() {}
    };
    __device__ __forceinline__ Adder adder() const { return Adder{*this}; }
    __device__ __forceinline__ void add(int c, int ix, int iy, float x) const {
        int hi, lo;
        fixed_split(x, f.jlb, hi, lo);
        const long long v = fixed_value(hi, lo, f);
        if (!walls) {
            atomicAdd(J + c * ntot + at(ix, iy), (unsigned long long)v);
            return;
        }
        int s;
        const int cx = wall_col(ix, nx, c == 0, c == 0, s);  // mirror image: Jx odd
        if (s != 0) atomicAdd(J + c * ntot + (long long)wrapi(iy, ny) * nx + cx, (unsigned long long)(s * v));
    }
};

template <int P, typename Mem>
__device__ __forceinline__ float gather(const Mem& M, int c, int bx, const float wx[P + 1], int by,
                                        const float wy[P + 1]) {
    float acc = 0.f;
#pragma unroll
    for (int b = 0; b <= P; b++) {
        float ra = 0.f;
#pragma unroll
        for (int a = 0; a <= P; a++) ra = fmaf(wx[a], M.ld(c, bx + a, by + b), ra);
        acc = fmaf(wy[b], ra, acc);
    }
    return acc;
}

// All six components at a particle: E, B. (bxe, wxe, bye, wye): the x and y shape of the
// half-integer-x lattice components (Ex, By, Bz in x; Ey, Bx, Bz in y use (bxh..)); in
// the node-averaged reading every component uses the node shape.
template <int P>
__device__ __forceinline__ void gather_fields(const GlobalMem& M, int bx0, const float wx0[P + 1], int bxh,
                                              const float wxh[P + 1], int by0, const float wy0[P + 1], int byh,
                                              const float wyh[P + 1], float E[3], float B[3]) {
    E[0] = gather<P>(M, 0, bxh, wxh, by0, wy0);
    E[1] = gather<P>(M, 1, bx0, wx0, byh, wyh);
    E[2] = gather<P>(M, 2, bx0, wx0, by0, wy0);
    B[0] = gather<P>(M, 3, bx0, wx0, byh, wyh);
    B[1] = gather<P>(M, 4, bxh, wxh, by0, wy0);
    B[2] = gather<P>(M, 5, bxh, wxh, byh, wyh);
}

template <int P>
__device__ __forceinline__ void gather_fields(const WinMem& M, int bx0, const float wx0[P + 1], int bxh,
                                              const float wxh[P + 1], int by0, const float wy0[P + 1], int byh,
                                              const float wyh[P + 1], float E[3], float B[3]) {
    float2 a = make_float2(0.f, 0.f), b = make_float2(0.f, 0.f);
    float ez = 0.f, bz = 0.f;
#pragma unroll
    for (int r = 0; r <= P; r++) {
        float2 ra = make_float2(0.f, 0.f), rb = make_float2(0.f, 0.f);
        float rz = 0.f, rbz = 0.f;
#pragma unroll
        for (int t = 0; t <= P; t++) {
            const float2 va = M.ld_exby(bxh + t, by0 + r);
            const float2 vb = M.ld_eybx(bx0 + t, byh + r);
            ra.x = fmaf(wxh[t], va.x, ra.x);
            ra.y = fmaf(wxh[t], va.y, ra.y);
            rb.x = fmaf(wx0[t], vb.x, rb.x);
            rb.y = fmaf(wx0[t], vb.y, rb.y);
            rz = fmaf(wx0[t], M.ld_ez(bx0 + t, by0 + r), rz);
            rbz = fmaf(wxh[t], M.ld_bz(bxh + t, byh + r), rbz);
        }
        a.x = fmaf(wy0[r], ra.x, a.x);
        a.y = fmaf(wy0[r], ra.y, a.y);
        b.x = fmaf(wyh[r], rb.x, b.x);
        b.y = fmaf(wyh[r], rb.y, b.y);
        ez = fmaf(wy0[r], rz, ez);
        bz = fmaf(wyh[r], rbz, bz);
    }
    E[0] = a.x;
    B[1] = a.y;
    E[1] = b.x;
    B[0] = b.y;
    E[2] = ez;
    B[2] = bz;
}

struct PushConst {
    float h;        // (q/m) dt / 2
    float dt_idx;   // dt / dx
    float dt_idy;   // dt / dy
    float fx, fy;   // q dx / (dt dx dy), q dy / (dt dx dy)
    float fz;       // q / (dx dy)   (times vz)
    int deposit;
    int nodal;      // the fields hold node averages: every component on the node lattice
};

// Gather, Boris push, move with carry into the neighbouring cell, and deposit, for one
// particle at cell (i, j) of M's index space with offsets (ox, oy). On return ox, oy, u
// hold the new state and di, dj the cell carry (-1, 0, +1). Returns false (and leaves
// the position unchanged) if the move is not below one cell or is not finite.
template <int P, typename Mem>
__device__ __forceinline__ bool push_one(const Mem& M, const PushConst& K, int i, int j, float& ox,
                                         float& oy, float u[3], int& di, int& dj, float& ek) {
    int bx0, by0;
    float wx0[P + 1], wy0[P + 1];
    shape_nodes<P, float>(i, ox, bx0, wx0);
    shape_nodes<P, float>(j, oy, by0, wy0);
    float E[3], B[3];
    if (K.nodal) {  // node-averaged fields: the deposit's weights for every component
        gather_fields<P>(M, bx0, wx0, bx0, wx0, by0, wy0, by0, wy0, E, B);
    } else {
        // Ex (i+1/2, j), Ey (i, j+1/2), Ez (i, j), Bx (i, j+1/2), By (i+1/2, j), Bz (i+1/2, j+1/2)
        int bxh, byh;
        float wxh[P + 1], wyh[P + 1];
        shape_nodes_half<P, float>(i, ox, bxh, wxh);
        shape_nodes_half<P, float>(j, oy, byh, wyh);
        gather_fields<P>(M, bx0, wx0, bxh, wxh, by0, wy0, byh, wyh, E, B);
    }
    // (the rounding of the update is explicit: xmul, xfma, ... in pic_internal.cuh)
    const float g2_old = xfma(u[2], u[2], xfma(u[1], u[1], xfma(u[0], u[0], 1.f)));
    boris<float>(K.h, E, B, u);
    const float ig = rsqrtf(xfma(u[2], u[2], xfma(u[1], u[1], xfma(u[0], u[0], 1.f))));
    const float dX = xmul(xmul(K.dt_idx, u[0]), ig), dY = xmul(xmul(K.dt_idy, u[1]), ig);
    di = 0;
    dj = 0;
    if (!(fabsf(dX) < 1.f && fabsf(dY) < 1.f)) return false;
    ek += xmul(g2_old, rsqrtf(g2_old)) + rcp_push(ig) - 2.f;  // gamma before + gamma after - 2
    float x1 = xadd(ox, dX), y1 = xadd(oy, dY);
    if (x1 >= 1.f) { x1 = xsub(x1, 1.f); di = 1; }
    else if (x1 < 0.f) { x1 = xadd(x1, 1.f); di = -1; if (x1 >= 1.f) { x1 = 0.f; di = 0; } }
    if (y1 >= 1.f) { y1 = xsub(y1, 1.f); dj = 1; }
    else if (y1 < 0.f) { y1 = xadd(y1, 1.f); dj = -1; if (y1 >= 1.f) { y1 = 0.f; dj = 0; } }
    if (K.deposit) {
        auto add = M.adder();
        esirkepov<P, float>(i, ox, j, oy, i + di, x1, j + dj, y1, xmul(K.fx, M.js), xmul(K.fy, M.js),
                            xmul(xmul(K.fz, xmul(u[2], ig)), M.js), add);
    }
    ox = x1;
    oy = y1;
    return true;
}

__device__ __forceinline__ PushConst push_const(const GridDev& G, int s) {
    PushConst K;
    K.h = G.pk_h[s];
    K.dt_idx = G.pk_dtx;
    K.dt_idy = G.pk_dty;
    K.fx = G.pk_fx[s];
    K.fy = G.pk_fy[s];
    K.fz = G.pk_fz[s];
    K.deposit = G.deposit;
    K.nodal = G.nodal;
    return K;
}

__device__ __forceinline__ void flag_bad(DevStatus* st, const float u[3]) {
    if (isfinite(u[0] + u[1] + u[2])) atomicAdd(&st->cfl_viol, 1ull);
    else atomicAdd(&st->nan_count, 1ull);
    st->stop_next = 1u;
}

__device__ __forceinline__ void put(unsigned* P, long long k, int c, float ox, float oy,
                                    const float u[3]) {
    __stcs(P + aos(k, 0), (unsigned)c);
    __stcs(reinterpret_cast<float*>(P) + aos(k, 1), ox);
    __stcs(reinterpret_cast<float*>(P) + aos(k, 2), oy);
    __stcs(reinterpret_cast<float*>(P) + aos(k, 3), u[0]);
    __stcs(reinterpret_cast<float*>(P) + aos(k, 4), u[1]);
    __stcs(reinterpret_cast<float*>(P) + aos(k, 5), u[2]);
}

__device__ __forceinline__ void get(const unsigned* P, long long k, int& c, float& ox, float& oy,
                                    float u[3]) {
    const float* F = reinterpret_cast<const float*>(P);
    c = (int)__ldcs(P + aos(k, 0));
    ox = __ldcs(F + aos(k, 1));
    oy = __ldcs(F + aos(k, 2));
    u[0] = __ldcs(F + aos(k, 3));
    u[1] = __ldcs(F + aos(k, 4));
    u[2] = __ldcs(F + aos(k, 5));
}

// Append to the overflow list of the next buffer; a full list is a fatal error. An
// entry records its simulation and species as gs = species | (simulation << 1).
__device__ __forceinline__ void to_overflow(unsigned* op, int* ogs, long long ovf_cap, DevStatus* st,
                                         int nxt, int c, float ox, float oy, float u0, float u1,
                                         float u2, int gs) {
    const unsigned long long o = atomicAdd(&st->ovf_count[nxt], 1ull);
    atomicAdd(&st->overflow, 1ull);
    if ((long long)o < ovf_cap) {
        const float u[3] = {u0, u1, u2};
        put(op, (long long)o, c, ox, oy, u);
        ogs[o] = gs;
    } else {
        atomicAdd(&st->lost, 1ull);  // storage exhausted: the step fails with PIC_ENOMEM
        st->stop_next = 1u;
    }
}

// ---------------------------------------------------------------------------------
// 1. Tile kernel
// ---------------------------------------------------------------------------------
// Cell of a window node on a periodic axis of n cells: k lies in [-2, n + window), so one
// wrap does unless the grid is smaller than the window's margins.
__device__ __forceinline__ int wrap_window(int k, int n) {
    if (k < 0) k += n;
    while (k >= n) k -= n;
    return k;
}

// Resident CTAs per SM the order-2 tile kernel is compiled for (register budget).
#ifndef PIC_TILE_MIN_BLOCKS_P2
#define PIC_TILE_MIN_BLOCKS_P2 3
#endif

template <int P>
__global__ void __launch_bounds__(kTileThreads, P == 1 ? 3 : (P == 2 ? PIC_TILE_MIN_BLOCKS_P2 : 2))
k_push_tile(const MixedArgs a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int s_start[2][kSegs + 1];     // virtual start of each segment, per species
    __shared__ long long s_base[2][kSegs];     // physical first slot of each segment
    __shared__ int s_out[2][kSegs];            // next-buffer counts (stayers, outboxes)
    __shared__ int s_sent[2][kSegs + 1];       // particles sent to each segment; [0][kSegs]: moved
                                               // in by the overflow kernel
    __shared__ double s_red[32];
    __shared__ int s_item, s_pop;
    DevStatus* st = a.st;
    if (st->stop) return;
    const int par = (int)st->parity, nxp = par ^ 1;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
    for (;;) {
        // every thread reads s_item between these two barriers; thread 0 writes it again
        // only after the barriers inside the tile body
        if (threadIdx.x == 0) s_item = atomicAdd(a.work, 1);
        __syncthreads();
        const int item = s_item;
        if (item >= a.nitems) break;
        const int2 tp = __ldg(a.items + item);
        const int t = tp.x, part = tp.y;      // global tile, part of its particles
        const int g = __ldg(a.tile_grid + t);
        const GridDev& G = a.grids[g];
        const int lt = t - G.tile_first;      // tile within its simulation
        const int tyi = lt / G.ntx, txi = lt - tyi * G.ntx;
        const int X0 = txi * G.tx, Y0 = tyi * G.ty;
        const int X1 = min(X0 + G.tx, G.nx), Y1 = min(Y0 + G.ty, G.ny);
        const int nx = G.nx, ny = G.ny;
        const int WX = G.wx, NW = G.wx * G.wy;
        const long long cap = G.cap, capo = G.capo, stride = bin_stride(G);
        const int parts = G.parts;
        int* jw = reinterpret_cast<int*>(smem_raw);  // [0, 3 NW) hi words, [3 NW, 6 NW) lo words
        float* fw = reinterpret_cast<float*>(smem_raw + (size_t)6 * NW * sizeof(int));
        if (threadIdx.x < 2 * kSegs) {
            const int s = threadIdx.x / kSegs, k = threadIdx.x - (threadIdx.x / kSegs) * kSegs;
            const int src = segment_source(G, txi, tyi, k);
            const long long off = k == 0 ? 0 : cap + (long long)(k - 1) * capo;
            const long long b = (long long)src * 2 + s;
            const int sent = segment_sent(G, par ? a.cnt[1] : a.cnt[0], src, s, k);
            s_sent[s][k] = sent;
            s_start[s][k + 1] = (int)min((long long)sent, k == 0 ? cap : capo);  // prefix-summed below
            s_base[s][k] = G.bin_off + b * stride + off;
            if (threadIdx.x == 0) s_sent[0][kSegs] = (par ? a.ovf_in[1] : a.ovf_in[0])[t];
            s_out[s][k] = 0;
        }
        __syncthreads();
        if (threadIdx.x < 2) {
            const int s = threadIdx.x;
            s_start[s][0] = 0;
            for (int k = 1; k <= kSegs; k++) s_start[s][k] += s_start[s][k - 1];
        } else if (threadIdx.x == 2) {  // the sum tile_population() forms
            int n = s_sent[0][kSegs];
            for (int s = 0; s < 2; s++)
                for (int k = 0; k < kSegs; k++) n += s_sent[s][k];
            s_pop = n;
        }
        __syncthreads();
        // this item's range [lo, hi) of the tile's particles: species 0, padded to whole
        // chunks, then species 1; parts of the planned size, or equal ones where the tile
        // holds more than was planned for
        const int v1 = (s_start[0][kSegs] + 31) & ~31;
        const int vend = v1 + s_start[1][kSegs];
        const int share = ((vend + parts - 1) / parts + kPartUnit - 1) / kPartUnit * kPartUnit;
        const int chunk = max(G.pchunk, share);
        const int lo = (int)min((long long)vend, (long long)part * chunk);
        const int hi = part == parts - 1 ? vend : min(vend, lo + chunk);
        if (lo >= hi) continue;  // (uniform over the CTA) nothing to push, no current to add
        // The window, one node per thread and round: its wrapped (or mirrored) cell once for
        // all six components, whose loads are all in flight together.
        const float* Fg = a.F32 + G.cell_off;
        for (int w = threadIdx.x; w < NW; w += blockDim.x) {
            const int wy = w / WX, wx = w - wy * WX;
            const float* R = Fg + (long long)wrap_window(Y0 - 2 + wy, ny) * nx;
            float ex, ey, ez, bx, by, bz;
            if (!G.walls) {
                R += wrap_window(X0 - 2 + wx, nx);
                ex = R[0];
                ey = R[a.ntot];
                ez = R[2 * a.ntot];
                bx = R[3 * a.ntot];
                by = R[4 * a.ntot];
                bz = R[5 * a.ntot];
            } else {  // conductor images: Ex, By, Bz even, Ey, Ez, Bx odd
                int sh, si;
                const float* Rh = R + wall_col(X0 - 2 + wx, nx, true, false, sh);
                const float* Ri = R + wall_col(X0 - 2 + wx, nx, false, true, si);
                const float fh = (float)sh, fi = (float)si;
                ex = fh * Rh[0];
                by = fh * Rh[4 * a.ntot];
                bz = fh * Rh[5 * a.ntot];
                ey = si == 0 ? 0.f : fi * Ri[a.ntot];
                ez = si == 0 ? 0.f : fi * Ri[2 * a.ntot];
                bx = si == 0 ? 0.f : fi * Ri[3 * a.ntot];
            }
            reinterpret_cast<float2*>(fw)[w] = make_float2(ex, by);
            reinterpret_cast<float2*>(fw + 2 * NW)[w] = make_float2(ey, bx);
            fw[4 * NW + w] = ez;
            fw[5 * NW + w] = bz;
#pragma unroll
            for (int c = 0; c < 6; c++) jw[c * NW + w] = 0;
        }
        __syncthreads();
        const FixedScale fs = fixed_scale(G, s_pop);
        const WinMem W{fw, jw, jw + 3 * NW, WX, NW, fs.js, fs.jlb};
        const GlobalMem M{a.F32 + G.cell_off, reinterpret_cast<unsigned long long*>(a.Jfix + G.cell_off),
                          a.ntot, nx, ny, fs, fs.js, G.walls};
        const unsigned* cur = par ? a.buf[1] : a.buf[0];
        unsigned* nxt = par ? a.buf[0] : a.buf[1];
        int* cnxt = (nxp ? a.cnt[1] : a.cnt[0]) + (long long)t * 2 * kSegs;
        float ek = 0.f;
        for (int s = 0; s < 2; s++) {
            const PushConst K = push_const(G, s);
            const int first = max(lo - (s ? v1 : 0), 0), total = min(hi - (s ? v1 : 0), s_start[s][kSegs]);
            const long long own = G.bin_off + ((long long)lt * 2 + s) * stride;
            const int st1 = s_start[s][1];  // end of the stayer segment
            for (int c0 = first + warp * 32; c0 < total; c0 += nwarp * 32) {
                const int v = c0 + lane;
                const bool valid = v < total;
                int dest = -1, cnew = 0;
                float ox = 0.f, oy = 0.f, u[3] = {0.f, 0.f, 0.f};
                if (valid) {
                    // segment of slot v: the stayers, else one of the outboxes addressed here
                    int seg = 0;
                    if (v >= st1) {
                        seg = 1;
#pragma unroll
                        for (int k = 2; k < kSegs; k++) seg += (v >= s_start[s][k]) ? 1 : 0;
                    }
                    const long long e = s_base[s][seg] + (v - s_start[s][seg]);
                    int c;
                    get(cur, e, c, ox, oy, u);
                    const int ci = c & 0xffff, cj = c >> 16;
                    int di, dj;
                    bool ok;
                    if (ci >= X0 && ci < X1 && cj >= Y0 && cj < Y1)
                        ok = push_one<P>(W, K, ci - X0 + 2, cj - Y0 + 2, ox, oy, u, di, dj, ek);
                    else
                        ok = push_one<P>(M, K, ci, cj, ox, oy, u, di, dj, ek);
                    if (!ok) flag_bad(st, u);
                    const int ni = G.walls ? reflect_x(ci + di, nx, ox, u[0]) : wrapi(ci + di, nx);
                    const int nj = wrapi(cj + dj, ny);
                    cnew = ni | (nj << 16);
                    if (ni >= X0 && ni < X1 && nj >= Y0 && nj < Y1) {
                        dest = 0;
                    } else {
                        int dtx = ni / G.tx - txi, dty = nj / G.ty - tyi;
                        if (dtx > 1) dtx -= G.ntx;
                        if (dtx < -1) dtx += G.ntx;
                        if (dty > 1) dty -= G.nty;
                        if (dty < -1) dty += G.nty;
                        dest = (abs(dtx) <= 1 && abs(dty) <= 1 && (dtx | dty)) ? 1 + outbox_of(dtx, dty) : -1;
                    }
                }
                const unsigned act = __ballot_sync(0xffffffffu, valid);
                const unsigned stay = __ballot_sync(0xffffffffu, valid && dest == 0);
                if (valid) {
                    // lanes bound for the same bin (usually the whole warp stays in its tile)
                    const unsigned grp = stay == act ? act : __match_any_sync(act, dest);
                    const int leader = __ffs(grp) - 1;
                    const int rank = __popc(grp & ((1u << lane) - 1u));
                    int b0 = 0;
                    // slots of the next buffer: the tile's counters, in shared memory while
                    // one CTA pushes the whole tile
                    if (lane == leader && dest >= 0)
                        b0 = atomicAdd(parts == 1 ? &s_out[s][dest] : cnxt + s * kSegs + dest, __popc(grp));
                    b0 = __shfl_sync(grp, b0, leader) + rank;
                    long long slot = -1;
                    if (dest == 0 && b0 < cap) slot = own + b0;
                    else if (dest > 0 && b0 < capo) slot = own + cap + (long long)(dest - 1) * capo + b0;
                    if (slot >= 0) {
                        put(nxt, slot, cnew, ox, oy, u);
                    } else {
                        to_overflow(nxp ? a.ovf[1].p : a.ovf[0].p, nxp ? a.ovf[1].gs : a.ovf[0].gs,
                                    a.ovf_cap, st, nxp, cnew, ox, oy, u[0], u[1], u[2], s | (g << 1));
                        if (dest < 0)  // sent to no bin: count it in its tile's population
                            atomicAdd((nxp ? a.ovf_in[1] : a.ovf_in[0]) + G.tile_first +
                                          tile_of(G, cnew & 0xffff, cnew >> 16), 1);
                    }
                }
            }
        }
        __syncthreads();
        if (parts == 1 && threadIdx.x < 2 * kSegs)
            cnxt[threadIdx.x] = (&s_out[0][0])[threadIdx.x];  // sent, parked ones included
        // add the current window into the global fixed-point current
        unsigned long long* Jg = reinterpret_cast<unsigned long long*>(a.Jfix + G.cell_off);
        for (int w = threadIdx.x; w < NW; w += blockDim.x) {
            const int wy = w / WX, wx = w - wy * WX;
            unsigned long long* R = Jg + (long long)wrap_window(Y0 - 2 + wy, ny) * nx;
            const int gx = G.walls ? 0 : wrap_window(X0 - 2 + wx, nx);
#pragma unroll
            for (int c = 0; c < 3; c++) {
                const int hi = jw[c * NW + w], lw = jw[(3 + c) * NW + w];
                if ((hi | lw) == 0) continue;
                const unsigned long long v = (unsigned long long)fixed_value(hi, lw, fs);
                int col = gx, sg = 1;
                if (G.walls) col = wall_col(X0 - 2 + wx, nx, c == 0, c == 0, sg);  // mirror: Jx odd
                if (sg != 0) atomicAdd(R + c * a.ntot + col, sg > 0 ? v : 0ull - v);
            }
        }
        const double sum = block_sum((double)ek, s_red);  // begins with a block barrier
        if (threadIdx.x == 0 && sum != 0.0) atomicAdd(&a.cg[g].uk, 0.5 * G.w * sum);
        __syncthreads();
    }
}

// ---------------------------------------------------------------------------------
// 0. Overflow particles: global-memory push; they stay in the overflow list until the
// host re-sorts after the pic_step call.
// ---------------------------------------------------------------------------------
// Start of a step, over the whole device: the deferred stop flag and step counter, the
// kinetic-energy accumulators and the work counters (block 0); J = 0; the next buffer's
// count slots and overflow count (a stopped step reads none of them again). One launch in
// place of four small ones: on small grids a step is made of launches.
__global__ void __launch_bounds__(256)
k_mixed_begin(const MixedArgs a, int ngrids, long long nj2, int ncnt, int* work) {
    DevStatus* st = a.st;
    const int nxp = (int)(st->parity ^ 1u);
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x, nt = (long long)gridDim.x * blockDim.x;
    longlong2* J = reinterpret_cast<longlong2*>(a.Jfix);  // (allocated with room for whole pairs)
    for (long long k = t; k < nj2; k += nt) J[k] = make_longlong2(0, 0);
    int* c = nxp ? a.cnt[1] : a.cnt[0];
    for (int k = (int)t; k < ncnt; k += (int)nt) c[k] = 0;
    if (blockIdx.x != 0) return;
    if (threadIdx.x < 4) work[threadIdx.x] = 0;
    if (threadIdx.x == 0) {
        if (st->stop_next) st->stop = 1u;
        if (!st->stop) st->steps_done += 1ull;
        st->ovf_count[nxp] = 0ull;
    }
    for (int g = threadIdx.x; g < ngrids; g += blockDim.x) a.cg[g].uk = 0.0;
}

template <int P>
__device__ __forceinline__ bool push_global(const GridDev& G, const GlobalMem& M, int s, int ci, int cj,
                                            float& ox, float& oy, float u[3], int& di, int& dj,
                                            float& ek) {
    return push_one<P>(M, push_const(G, s), ci, cj, ox, oy, u, di, dj, ek);
}

__global__ void __launch_bounds__(kTileThreads)
k_push_overflow(const MixedArgs a) {
    DevStatus* st = a.st;
    if (st->stop) return;
    const int par = (int)st->parity;
    const long long n = min((long long)st->ovf_count[par], a.ovf_cap);
    const Slots O = par ? a.ovf[1] : a.ovf[0];
    for (long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x; k < n;
         k += (long long)gridDim.x * blockDim.x) {
        int c;
        float ox, oy, u[3];
        get(O.p, k, c, ox, oy, u);
        const int gs = O.gs[k];
        const int s = gs & 1, g = gs >> 1;
        const GridDev& G = a.grids[g];
        const int ci = c & 0xffff, cj = c >> 16;
        // round the current as the tile the particle's cell lies in rounds its window
        const FixedScale fs = fixed_scale(G, tile_population(G, par ? a.cnt[1] : a.cnt[0],
                                                             par ? a.ovf_in[1] : a.ovf_in[0], tile_of(G, ci, cj)));
        const GlobalMem M{a.F32 + G.cell_off, reinterpret_cast<unsigned long long*>(a.Jfix + G.cell_off),
                          a.ntot, G.nx, G.ny, fs, fs.js, G.walls};
        int di, dj;
        float ek = 0.f;
        bool ok;
        switch (G.order) {
        case 1: ok = push_global<1>(G, M, s, ci, cj, ox, oy, u, di, dj, ek); break;
        case 2: ok = push_global<2>(G, M, s, ci, cj, ox, oy, u, di, dj, ek); break;
        default: ok = push_global<3>(G, M, s, ci, cj, ox, oy, u, di, dj, ek); break;
        }
        if (!ok) flag_bad(st, u);
        if (ek != 0.f) atomicAdd(&a.cg[g].uk, 0.5 * G.w * (double)ek);
        const int ni = G.walls ? reflect_x(ci + di, G.nx, ox, u[0]) : wrapi(ci + di, G.nx);
        const int nj = wrapi(cj + dj, G.ny);
        const int cnew = ni | (nj << 16);
        to_overflow(par ? a.ovf[0].p : a.ovf[1].p, par ? a.ovf[0].gs : a.ovf[1].gs, a.ovf_cap, st,
                    par ^ 1, cnew, ox, oy, u[0], u[1], u[2], gs);
        atomicAdd((par ? a.ovf_in[0] : a.ovf_in[1]) + G.tile_first + tile_of(G, ni, nj), 1);
    }
}

// The injector's pairs of this step, straight into the next buffer: the stayer segment
// of the tile holding their cell (the tile kernels have finished with it), or the
// overflow list when it is full. One thread per (simulation, row, pair).
__global__ void k_inject_mixed(const MixedArgs a, const int* inj_grid, const long long* inj_first, int ngr,
                               unsigned long long* injected) {
    DevStatus* st = a.st;
    if (st->stop) return;
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    int q = 0;
    while (q + 1 < ngr && t >= inj_first[q + 1]) q++;
    if (t >= inj_first[ngr]) return;
    const int g = inj_grid[q];
    const GridDev& G = a.grids[g];
    const long long local = t - inj_first[q];
    const long long kmax = (long long)ceil(G.ppc * inj_width(G)) + 1;
    const int j = (int)(local / kmax);
    const long long k = local - (long long)j * kmax;
    const long long n = (long long)st->steps_done - 1;
    if (j >= G.ny || k >= inj_count(G, n)) return;
    double x, y;
    inj_position(G, n, j, k, x, y);
    int ci = (int)floor(x);
    float ox = (float)(x - ci);
    if (ox >= 1.f) {
        ox = 0.f;
        ci += 1;
    }
    if (ci < 0 || ci >= G.nx) return;  // (the plane starts at least two cells from the wall)
    const int cj = j;
    const float oy = (float)(y - cj);
    const int nxp = (int)st->parity ^ 1;
    unsigned* nxt = nxp ? a.buf[1] : a.buf[0];
    int* cnxt = nxp ? a.cnt[1] : a.cnt[0];
    const int lt = (cj / G.ty) * G.ntx + ci / G.tx;
    const long long stride = bin_stride(G);
    for (int s = 0; s < 2; s++) {
        double u[3];
        inj_momentum(G, n, j, k, s, u);
        const float uf[3] = {(float)u[0], (float)u[1], (float)u[2]};
        const int cell = ci | (cj << 16);
        const int slot = atomicAdd(&cnxt[((long long)(G.tile_first + lt) * 2 + s) * kSegs], 1);
        if (slot < G.cap)
            put(nxt, G.bin_off + ((long long)lt * 2 + s) * stride + slot, cell, ox, oy, uf);
        else
            to_overflow(nxp ? a.ovf[1].p : a.ovf[0].p, nxp ? a.ovf[1].gs : a.ovf[0].gs, a.ovf_cap, st, nxp,
                        cell, ox, oy, uf[0], uf[1], uf[2], s | (g << 1));
        atomicAdd(&injected[2 * g + s], 1ull);
    }
}

// End of a step: the buffers swap; PCG statistics.
__global__ void k_mixed_end(DevStatus* st, int ngrids, CgState* cg) {
    if (st->stop) return;
    if (threadIdx.x == 0) st->parity ^= 1u;
    for (int g = threadIdx.x; g < ngrids; g += blockDim.x) {
        CgState& s = cg[g];
        s.last_iters = s.iters;
        s.max_iters = s.iters > s.max_iters ? s.iters : s.max_iters;
        s.total_iters += s.iters;
    }
}

// ---------------------------------------------------------------------------------
// Loading and re-sorting (one simulation at a time; tile indices are local to it)
// ---------------------------------------------------------------------------------
// Cell and FP32 offset of a position x on an axis of n cells (length L, 1/d = id). A position
// in [0, L) is not folded: x / L rounds below one, so the fold would give x back. The FP64
// pipe bounds the kernel (two lanes per cycle and SM), and the fold's division was half of
// its instructions; nor does a position in range need the remainder, x / d rounding to n at
// most.
__device__ __forceinline__ int stage_axis(double x, double L, double id, int n, float& f) {
    const bool in = x >= 0.0 && x < L;
    if (!in) x = x - floor(x / L) * L;
    x *= id;
    const double c = floor(x);
    int i = (int)c;
    f = (float)(in ? x - c : x - i);
    if (f >= 1.f) { f = 0.f; i += 1; }
    if (in) return i >= n ? i - n : i;
    return ((i % n) + n) % n;
}
__device__ __forceinline__ bool finite64(double v) { return (__double2hiint(v) & 0x7ff00000) != 0x7ff00000; }

// FP64 physical particles -> staging (cell + FP32 offsets, FP32 momenta). 1.05e6
// particles: 91 -> 53 us.
__global__ void k_stage_fp64(long long n, const double* x, const double* y, const double* ux,
                             const double* uy, const double* uz, GridDev G, PartArrays S,
                             unsigned long long* nbad) {
    const long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    double X = x[k], Y = y[k];
    const double a = ux[k], b = uy[k], c = uz[k];
    const double Lx = G.nx * G.dx, Ly = G.ny * G.dy;
    if (!finite64(X) || !finite64(Y) || !finite64(a) || !finite64(b) || !finite64(c) ||
        (G.walls && !(X >= 0.0 && X < Lx))) {
        atomicAdd(nbad, 1ull);
        X = 0.0;
        Y = 0.0;
    }
    float fx, fy;
    const int i = stage_axis(X, Lx, G.idx, G.nx, fx), j = stage_axis(Y, Ly, G.idy, G.ny, fy);
    S.cij[k] = i | (j << 16);
    S.ox[k] = fx;
    S.oy[k] = fy;
    S.ux[k] = (float)a;
    S.uy[k] = (float)b;
    S.uz[k] = (float)c;
}

// ---- the load / re-sort into tile bins (a counting sort, no library) ------------------
// A bin lists one particle of every cell of its tile, then a second of every cell, and
// so on, so that the 32 lanes of a warp work on 32 different cells: the particle of rank
// r in its cell (0, 1, ...) at cell cin of the tile goes to the slot that the key
// r * cells_per_tile + cin has among the tile's occupied keys. Keys are unique within a
// tile, so the slot is a prefix count over an occupancy bitmap of the tile's key range:
//   k_rank      rank within the cell (counter per cell), the tile and the key; tile
//               counts; the largest rank;
//   k_setbits   one bit per particle in its tile's bitmap;
//   k_scanbits  per tile, the exclusive prefix of the bitmap words' bit counts;
//   k_scatter   slot = prefix of the key's word + bits below the key within the word.
__global__ void k_rank(long long n, GridDev G, const int* cij, unsigned int* cellcnt, int* bincnt,
                       unsigned int* maxrank, unsigned int* key, int* tile) {
    const long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const bool valid = k < n;
    const int c = valid ? cij[k] : 0;
    const int i = c & 0xffff, j = c >> 16;
    const long long cell = (long long)j * G.nx + i;
    // warp-aggregated rank within the cell (neighbouring particles often share a cell)
    const unsigned act = __ballot_sync(0xffffffffu, valid);
    if (!valid) return;
    const unsigned grp = __match_any_sync(act, cell);
    const int lane = threadIdx.x & 31;
    const int leader = __ffs(grp) - 1;
    unsigned base = 0;
    if (lane == leader) base = atomicAdd(&cellcnt[cell], (unsigned)__popc(grp));
    const unsigned rank = __shfl_sync(grp, base, leader) + __popc(grp & ((1u << lane) - 1u));
    const int t = (j / G.ty) * G.ntx + i / G.tx;
    const unsigned grpt = __match_any_sync(act, t);
    if (lane == __ffs(grpt) - 1) atomicAdd(&bincnt[t], __popc(grpt));
    const unsigned rmax = __reduce_max_sync(act, rank);
    if (lane == __ffs(act) - 1) atomicMax(maxrank, rmax);
    const unsigned cin = (unsigned)((j - (j / G.ty) * G.ty) * G.tx + (i - (i / G.tx) * G.tx));
    key[k] = rank * (unsigned)(G.tx * G.ty) + cin;
    tile[k] = t;
}

// words: bitmap words per tile; the bitmap holds tiles t0 .. t0 + ntg - 1
__global__ void k_setbits(long long n, const unsigned int* key, const int* tile, int t0, int ntg, long long words,
                          unsigned int* bits) {
    const long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    const int t = tile[k] - t0;
    if (t < 0 || t >= ntg) return;
    const unsigned q = key[k];
    atomicOr(bits + (long long)t * words + (q >> 5), 1u << (q & 31));
}

// One block per tile: pref[w] = bits set in words 0 .. w-1 of the tile's bitmap.
__global__ void __launch_bounds__(256) k_scanbits(long long words, const unsigned int* bits, unsigned int* pref) {
    __shared__ unsigned int s_warp[8];
    __shared__ unsigned int s_carry;
    const unsigned int* b = bits + (long long)blockIdx.x * words;
    unsigned int* o = pref + (long long)blockIdx.x * words;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (threadIdx.x == 0) s_carry = 0;
    __syncthreads();
    for (long long w0 = 0; w0 < words; w0 += blockDim.x) {
        const long long w = w0 + threadIdx.x;
        const unsigned v = w < words ? (unsigned)__popc(b[w]) : 0u;
        unsigned x = v;  // inclusive scan within the warp
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const unsigned y = __shfl_up_sync(0xffffffffu, x, d);
            if (lane >= d) x += y;
        }
        if (lane == 31) s_warp[warp] = x;
        __syncthreads();
        unsigned before = s_carry;
        for (int q = 0; q < warp; q++) before += s_warp[q];
        if (w < words) o[w] = before + x - v;
        __syncthreads();
        if (threadIdx.x == blockDim.x - 1) s_carry = before + x;
        __syncthreads();
    }
}

__global__ void k_scatter(long long n, GridDev G, int s, const unsigned int* key, const int* tile, int t0,
                          int ntg, long long words, const unsigned int* bits, const unsigned int* pref,
                          PartArrays S, unsigned* B) {
    const long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= n) return;
    const int t = tile[p];
    if (t < t0 || t >= t0 + ntg) return;
    const unsigned q = key[p];
    const long long wq = (long long)(t - t0) * words + (q >> 5);
    const long long r = (long long)pref[wq] + __popc(bits[wq] & ((1u << (q & 31)) - 1u));
    const long long dst = G.bin_off + ((long long)t * 2 + s) * bin_stride(G) + r;
    const float u[3] = {S.ux[p], S.uy[p], S.uz[p]};
    put(B, dst, S.cij[p], S.ox[p], S.oy[p], u);
}

// cnt points at the simulation's first count slot.
__global__ void k_set_counts(int ntiles, int s, const int* bincnt, int* cnt) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= ntiles) return;
    int* c = cnt + ((long long)t * 2 + s) * kSegs;
    c[0] = bincnt[t];
    for (int k = 1; k < kSegs; k++) c[k] = 0;
}

// Copy every segment of species s's bins (offsets from a host prefix sum, one entry per
// (tile, segment)) into staging form.
__device__ __forceinline__ void to_staging(const unsigned* P, long long k, PartArrays S, long long d) {
    int c;
    float ox, oy, u[3];
    get(P, k, c, ox, oy, u);
    S.cij[d] = c;
    S.ox[d] = ox;
    S.oy[d] = oy;
    S.ux[d] = u[0];
    S.uy[d] = u[1];
    S.uz[d] = u[2];
}

__global__ void k_gather_bins(GridDev G, int s, const int* cnt, const long long* off, const unsigned* B,
                              PartArrays S) {
    const int t = blockIdx.x / kSegs, k = blockIdx.x - (blockIdx.x / kSegs) * kSegs;
    const long long b = (long long)t * 2 + s;
    const long long lim = k == 0 ? G.cap : G.capo;
    const int n = (int)min((long long)cnt[b * kSegs + k], lim);
    const long long src0 = G.bin_off + b * bin_stride(G) + (k == 0 ? 0 : G.cap + (long long)(k - 1) * G.capo);
    const long long dst0 = off[blockIdx.x];
    for (int q = threadIdx.x; q < n; q += blockDim.x) to_staging(B, src0 + q, S, dst0 + q);
}

// Overflow-list entries with code gs (species | simulation << 1) appended after `base`.
__global__ void k_gather_overflow(long long n_over, int gs, Slots O, long long base,
                                  unsigned long long* cursor, PartArrays S) {
    const long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n_over || O.gs[k] != gs) return;
    const long long d = base + (long long)atomicAdd(cursor, 1ull);
    to_staging(O.p, k, S, d);
}

// Node density (q[s] per particle, 0: species left out) and w times the total momentum
// straight from the bins: a block takes part `blockIdx.y` of the particles of one (tile,
// species), all nine segments (one block row more: the overflow list). rho, mom: null where
// not asked for.
//
// In FP64 throughout the kernel was bound by that pipe (two lanes per cycle and SM, 28
// operations per particle at order 2: 376 us for 8.4e6 particles). Here contributions are whole
// numbers that keep their relative accuracy (density_fixed.h), and so are the sums in the
// tile's window in shared memory: 96 bits, which hold a contribution of 2^-34 to 53 places and
// a sum of 256 full weights (what wraps goes to the output at once). FP64 is left to the
// window's nodes when the block is done and to the particles that density_contributions
// refuses (1% at order 2, 3.5% at order 3 of random ones), which wait until then: one of them
// would cost its whole warp the FP64 path. So every node's density, also one that only the far
// edges of shapes reach, is as accurate as a sum in FP64 or better (order 2, 16 per cell: 9e-17
// against 3.2e-16, relative to the density's norm; 200 particles on 64 x 48 cells: 2e-16 of
// each node at most, both).
// 1024 x 256 with 16 per cell (8.4e6 particles, 101 MB), order 2: 118 us, bound by instruction
// issue (64% active; 360 instructions per 32 particles) and by the three atomics per node (3.0
// wavefronts each); order 3 216 us. With 64-bit sums, exact to 2^-56 of a full weight, they
// were 106 and 199 us, but the sparse plasma's nodes were off by up to 1e-10 of themselves.
struct DensityArgs {
    double q[2], w;
    double *rho, *mom;
};

template <int P>
__device__ __noinline__ void density_global(const GridDev& G, int c, float fx, float fy, double q, double* rho) {
    deposit_rho<P>(G, c & 0xffff, (double)fx, c >> 16, (double)fy, q, rho);
}

// rho += v at the node (ix, iy), which may lie beyond the grid's edges by a window's margin
__device__ __forceinline__ void density_node(const GridDev& G, int ix, int iy, double v, double* rho) {
    int sign = 1, col;
    if (G.walls) col = wall_col(ix, G.nx, false, false, sign);
    else col = wrap_window(ix, G.nx);
    if (sign) atomicAdd(rho + (long long)wrap_window(iy, G.ny) * G.nx + col, v);
}

struct DensityWin {
    unsigned* w;         // words of the sums: wx per row, then the next word's plane of nw
    int wx, nw, X0, Y0;  // the window's row length, size and first node
    double unit;
    double* rho;
};

// the sums of window nodes k0 + (bit / 4) wx + bit % 4 passed 2^96 units
__device__ __noinline__ void density_wrapped(const GridDev& G, int k0, unsigned bits, int X0, int Y0, double unit,
                                             double* rho) {
    for (; bits; bits &= bits - 1) {
        const int n = __ffs(bits) - 1, k = k0 + (n >> 2) * G.wx + (n & 3);
        density_node(G, X0 + k % G.wx, Y0 + k / G.wx, unit * 79228162514264337593543950336.0, rho);
    }
}

// v (of one or two words) and the carry of l + u
__device__ __forceinline__ void carry_into(unsigned l, unsigned u, unsigned& v0, unsigned& v1) {
    asm("{\n .reg .u32 t;\n add.cc.u32 t, %2, %3;\n addc.cc.u32 %0, %0, 0;\n addc.u32 %1, %1, 0;\n}\n"
        : "+r"(v0), "+r"(v1)
        : "r"(l), "r"(u));
}
__device__ __forceinline__ void carry_into(unsigned l, unsigned u, unsigned& v) {
    asm("{\n .reg .u32 t;\n add.cc.u32 t, %1, %2;\n addc.u32 %0, %0, 0;\n}\n" : "+r"(v) : "r"(l), "r"(u));
}

// 96-bit sums of a row's nodes, each from three 32-bit atomics: the one that sees a word wrap
// carries. All lowest words, then all middle and all highest ones: one wait for each, not for
// each node. At order 1 the highest word gets carries only. Returns which sums wrapped: none
// while the high words found are below 2^32 - 2^24 - 1, as a contribution's is at most 2^24 and
// a carry, and only then is each looked at (at order 1 it would take 2^34 particles).
template <int P>
__device__ __forceinline__ unsigned density_add(const DensityWin& W, int k, const Words (&v)[P + 1]) {
    unsigned l[P + 1], mid[P + 1], hi[P + 1], most = 0, wrapped = 0;
    unsigned* w = W.w + k;
#pragma unroll
    for (int a = 0; a <= P; a++) l[a] = atomicAdd(w + a, v[a].w[0]);
    w += W.nw;
#pragma unroll
    for (int a = 0; a <= P; a++) {
        mid[a] = v[a].w[1];
        hi[a] = v[a].w[2];
        if (P == 1) carry_into(l[a], v[a].w[0], mid[a]);  // (its contributions' middle word is below 2^31)
        else carry_into(l[a], v[a].w[0], mid[a], hi[a]);
        l[a] = atomicAdd(w + a, mid[a]);
    }
    w += W.nw;
#pragma unroll
    for (int a = 0; a <= P; a++) {
        carry_into(l[a], mid[a], hi[a]);
        if (P == 1) {
            if (hi[a]) atomicAdd(w + a, hi[a]);
        } else {
            l[a] = atomicAdd(w + a, hi[a]);
            most = max(most, l[a]);
        }
    }
    if (P > 1 && most >= 0xfeffffffu) {
#pragma unroll
        for (int a = 0; a <= P; a++) wrapped |= l[a] + hi[a] < l[a] ? 1u << a : 0u;
    }
    return wrapped;
}

template <int P>
__device__ __forceinline__ bool density_window(const GridDev& G, const DensityWin& W, int i, unsigned Fx, int j,
                                               unsigned Fy) {
    unsigned wrapped = 0;
    int k0 = 0;
    const bool ok = density_contributions<P>(i, Fx, j, Fy, [&](int bx, int by, int r, const Words (&v)[P + 1]) {
        k0 = by * W.wx + bx;
        wrapped |= density_add<P>(W, k0 + r * W.wx, v) << 4 * r;
    });
    if (wrapped) density_wrapped(G, k0, wrapped, W.X0, W.Y0, W.unit, W.rho);
    return ok;
}

constexpr int kDensityRare = 256;  // particles of a block kept for the end

// MOM: with the momentum. (Not a test in the loop: its FP64 instructions then went through the
// pipe without effect, 6 per 32 particles: 138 instead of 118 us.)
template <int P, bool MOM>
__global__ void __launch_bounds__(256) k_density(const MixedArgs a, int g, int nbins, const DensityArgs d) {
    extern __shared__ unsigned dens_win[];  // [3][wx * wy]: words of the sums
    __shared__ long long s_rare[kDensityRare];
    __shared__ int s_nrare;
    const GridDev& G = a.grids[g];
    const DevStatus* st = a.st;
    const int par = (int)st->parity;
    const int tid = threadIdx.x;
    double m[3] = {0.0, 0.0, 0.0};
    const auto momentum = [&](const float* F, long long k) {
#pragma unroll
        for (int c = 0; c < 3; c++) m[c] += (double)__ldcs(F + aos(k, 3 + c));
    };
    if ((int)blockIdx.x < nbins) {
        // (species by halves of the grid: with alternating ones a species left out would
        // idle every other SM)
        const int s = (int)blockIdx.x >= G.ntiles ? 1 : 0, t = (int)blockIdx.x - s * G.ntiles;
        const long long bin = 2ll * t + s;
        const double q = s ? d.q[1] : d.q[0];
        double* rho = q != 0.0 ? d.rho : nullptr;
        if (!(MOM || rho)) return;
        const unsigned* B = par ? a.buf[1] : a.buf[0];
        const float* F = reinterpret_cast<const float*>(B);
        const int* cnt = (par ? a.cnt[1] : a.cnt[0]) + ((long long)G.tile_first * 2 + bin) * kSegs;
        const int X0 = t % G.ntx * G.tx, Y0 = t / G.ntx * G.ty, NW = G.wx * G.wy;
        const int nx = G.nx, ny = G.ny, tx = G.tx, ty = G.ty;
        // a unit of the words (density_fixed.h)
        const double unit = P == 1 ? q / 4611686018427387904.0
                                   : q * ((P == 3 ? 4.0 / 9.0 : 1.0) / 309485009821345068724781056.0);
        const DensityWin W{dens_win, G.wx, NW, X0 - 2, Y0 - 2, unit, rho};
        if (rho)
            for (int k = tid; k < 3 * NW; k += 256) dens_win[k] = 0u;
        if (tid == 0) s_nrare = 0;
        __syncthreads();
        long long base = G.bin_off + bin * bin_stride(G);
        for (int k = 0; k < kSegs; k++) {
            const int lim = (int)(k == 0 ? G.cap : G.capo), n = min(cnt[k], lim);
            for (int v = (int)blockIdx.y * 256 + tid; v < n; v += (int)gridDim.y * 256) {
                if (rho) {
                    const int c = (int)__ldcs(B + aos(base + v, 0));
                    const float fx = __ldcs(F + aos(base + v, 1)), fy = __ldcs(F + aos(base + v, 2));
                    // cell within the window (its origin is X0 - 2, Y0 - 2): the tile's own
                    // and, in the outboxes, the next ones around it, across the periodic edge
                    int i = (c & 0xffff) - X0 + 2, j = (c >> 16) - Y0 + 2;
                    if (i < 1) i += nx;
                    else if (i > tx + 2) i -= nx;
                    if (j < 1) j += ny;
                    else if (j > ty + 2) j -= ny;
                    unsigned Fx, Fy;
                    const bool fine = fixed_offset(__float_as_uint(fx), Fx) & fixed_offset(__float_as_uint(fy), Fy);
                    if (!(fine && i >= 1 && i <= tx + 2 && j >= 1 && j <= ty + 2 && density_window<P>(G, W, i, Fx, j, Fy))) {
                        const int e = atomicAdd(&s_nrare, 1);
                        if (e < kDensityRare) s_rare[e] = base + v;
                        else density_global<P>(G, c, fx, fy, q, rho);
                    }
                }
                if (MOM) momentum(F, base + v);
            }
            base += lim;
        }
        if (rho) {
            __syncthreads();
            // (kept for now: a warp of them costs what one of them would have cost its warp)
            for (int e = tid; e < min(s_nrare, kDensityRare); e += 256) {
                const long long k = s_rare[e];
                density_global<P>(G, (int)B[aos(k, 0)], F[aos(k, 1)], F[aos(k, 2)], q, rho);
            }
            for (int k = tid; k < NW; k += 256) {
                // the sum's leading 64 bits: one conversion and one product in FP64, the power
                // of two into the exponent
                const unsigned w0 = W.w[k], w1 = W.w[NW + k], w2 = W.w[2 * NW + k];
                const int lead = clz32(w2), e = 32 - lead;  // (e = 0: w2 = 0)
                const u64 v = e ? (u64)__funnelshift_l(w1, w2, lead) << 32 | __funnelshift_l(w0, w1, lead) : (u64)w1 << 32 | w0;
                if (v) {
                    const double x = W.unit * (double)v;
                    density_node(G, W.X0 + k % G.wx, W.Y0 + k / G.wx,
                                 __hiloint2double(__double2hiint(x) + (e << 20), __double2loint(x)), rho);
                }
            }
        }
    } else {
        const Slots O = par ? a.ovf[1] : a.ovf[0];
        const float* F = reinterpret_cast<const float*>(O.p);
        const long long n = min((long long)st->ovf_count[par], a.ovf_cap);
        for (long long k = (long long)blockIdx.y * 256 + tid; k < n; k += (long long)gridDim.y * 256) {
            const int gs = O.gs[k];
            if (gs >> 1 != g) continue;
            const double q = gs & 1 ? d.q[1] : d.q[0];
            if (d.rho && q != 0.0)
                density_global<P>(G, (int)O.p[aos(k, 0)], F[aos(k, 1)], F[aos(k, 2)], q, d.rho);
            if (MOM) momentum(F, k);
        }
    }
    if constexpr (MOM) {
        __shared__ double s_m[3][256];
#pragma unroll
        for (int c = 0; c < 3; c++) s_m[c][tid] = m[c];
        __syncthreads();
        if (tid >= 96) return;
        const double t = warp_of_block_sum(s_m[tid >> 5]);
        if ((tid & 31) == 0 && t != 0.0) atomicAdd(d.mom + (tid >> 5), d.w * t);
    }
}

using DensityKernel = void (*)(const MixedArgs, int, int, const DensityArgs);
constexpr DensityKernel kDensityKernels[3][2] = {  // [order - 1][with momentum]
    {k_density<1, false>, k_density<1, true>}, {k_density<2, false>, k_density<2, true>}, {k_density<3, false>, k_density<3, true>}};

__global__ void k_unstage(long long n, GridDev G, PartArrays S, double* out) {
    const long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    const int c = S.cij[k];
    out[k] = ((double)(c & 0xffff) + (double)S.ox[k]) * G.dx;
    out[n + k] = ((double)(c >> 16) + (double)S.oy[k]) * G.dy;
    out[2 * n + k] = S.ux[k];
    out[3 * n + k] = S.uy[k];
    out[4 * n + k] = S.uz[k];
}

// ---- host helpers -------------------------------------------------------------------

template <typename T>
cudaError_t dalloc(T** p, size_t n) {
    *p = nullptr;
    return cudaMalloc((void**)p, (n ? n : 1) * sizeof(T));
}

// Temporaries of loads, re-sorts and diagnostics (staging arrays, sort keys, bitmaps)
// come from a library-owned stream-ordered memory pool that keeps its memory for the
// next call (release threshold: never), so that a load or a re-sort does not map and
// unmap gigabytes of device memory each time (cudaMalloc / cudaFree of that size cost
// from tens to hundreds of ms, depending on the device's history).
cudaMemPool_t temp_pool(cudaError_t* e) {
    static std::mutex mu;
    static cudaMemPool_t pools[64] = {};
    int dev = 0;
    *e = cudaGetDevice(&dev);
    if (*e != cudaSuccess) return nullptr;
    if (dev < 0 || dev >= 64) {
        *e = cudaErrorInvalidDevice;
        return nullptr;
    }
    std::lock_guard<std::mutex> lk(mu);
    if (!pools[dev]) {
        cudaMemPoolProps pp{};
        pp.allocType = cudaMemAllocationTypePinned;
        pp.location.type = cudaMemLocationTypeDevice;
        pp.location.id = dev;
        *e = cudaMemPoolCreate(&pools[dev], &pp);
        if (*e != cudaSuccess) {
            pools[dev] = nullptr;
            return nullptr;
        }
        unsigned long long keep = ~0ull;  // the attribute is a 64-bit unsigned
        *e = cudaMemPoolSetAttribute(pools[dev], cudaMemPoolAttrReleaseThreshold, &keep);
        if (*e != cudaSuccess) return nullptr;
    }
    return pools[dev];
}

template <typename T>
cudaError_t talloc(T** p, size_t n, cudaStream_t st) {
    return temp_alloc(reinterpret_cast<void**>(p), (n ? n : 1) * sizeof(T), st);
}

void tfree(void* p, cudaStream_t st) { temp_free(p, st); }

void free_parts(PartArrays& A, cudaStream_t st) {
    void* ps[] = {A.cij, A.ox, A.oy, A.ux, A.uy, A.uz, A.gs};
    for (void* p : ps) tfree(p, st);
    A = PartArrays{};
}

cudaError_t alloc_parts(PartArrays& A, size_t n, bool with_gs, cudaStream_t st) {
    A = PartArrays{};
    cudaError_t e = talloc(&A.cij, n, st);
    if (e == cudaSuccess) e = talloc(&A.ox, n, st);
    if (e == cudaSuccess) e = talloc(&A.oy, n, st);
    if (e == cudaSuccess) e = talloc(&A.ux, n, st);
    if (e == cudaSuccess) e = talloc(&A.uy, n, st);
    if (e == cudaSuccess) e = talloc(&A.uz, n, st);
    if (e == cudaSuccess && with_gs) e = talloc(&A.gs, n, st);
    if (e != cudaSuccess) free_parts(A, st);
    return e;
}

// Staged particles of every (simulation, species), index 2 g + s.
struct Staged {
    std::vector<PartArrays> S;
    std::vector<long long> n;
    cudaStream_t st;
    Staged(int ngrids, cudaStream_t stream) : S(2 * ngrids), n(2 * ngrids, 0), st(stream) {}
    ~Staged() {
        for (PartArrays& a : S) free_parts(a, st);
    }
};

MixedArgs make_args(MixedState* m, int order) {
    MixedArgs a{};
    a.grids = m->dgrids;
    a.tile_grid = m->tile_grid;
    a.items = m->items + m->item_first[order];
    a.nitems = m->item_n[order];
    a.work = m->work + order;
    a.ntot = m->ntot;
    a.F32 = m->F32;
    a.Jfix = m->Jfix;
    for (int p = 0; p < 2; p++) {
        a.buf[p] = m->buf[p];
        a.cnt[p] = m->cnt[p];
        a.ovf_in[p] = m->ovf_in[p];
        a.ovf[p] = m->ovf[p];
    }
    a.ovf_cap = m->ovf_cap;
    a.cg = m->cg;
    a.st = m->st;
    return a;
}

unsigned grid1(long long n, int b = 256) { return (unsigned)std::max<long long>(1, (n + b - 1) / b); }

#define MCK(call)                                                                     \
    do {                                                                              \
        cudaError_t e_ = (call);                                                      \
        if (e_ != cudaSuccess) {                                                      \
            err = std::string(#call) + " failed: " + cudaGetErrorString(e_);          \
            return PIC_ECUDA;                                                         \
        }                                                                             \
    } while (0)

int read_status(MixedState* m, DevStatus& hs, cudaStream_t st, std::string& err) {
    MCK(cudaMemcpyAsync(&hs, m->st, sizeof hs, cudaMemcpyDeviceToHost, st));
    MCK(cudaStreamSynchronize(st));
    return PIC_OK;
}

long long round32(double c) { return ((long long)std::ceil(c) + 31) / 32 * 32; }

int* cnt_of(MixedState* m, int par, int g) {
    return m->cnt[par] + (long long)m->G[g].tile_first * 2 * kSegs;
}

// Sort n staged particles of species s of simulation g into the stayer segments of
// buffer `par`. Returns PIC_ENOMEM (nothing written) when a bin would overflow, with
// the fullest bin's count in *need.
int sort_into_bins(MixedState* m, int g, int par, int s, PartArrays S, long long n, cudaStream_t st,
                   long long* need, std::string& err) {
    const GridDev& G = m->G[g];
    const int ntiles = G.ntiles;
    unsigned int* cellcnt = nullptr;
    int* bincnt = nullptr;
    unsigned int* maxrank = nullptr;
    unsigned int *key = nullptr, *bits = nullptr, *pref = nullptr;
    int* tile = nullptr;
    int rc = PIC_OK;
    cudaError_t e = cudaSuccess;
    auto A = [&](cudaError_t r) {
        if (e == cudaSuccess) e = r;
    };
    A(talloc(&cellcnt, (size_t)G.ncell, st));
    A(talloc(&bincnt, (size_t)ntiles, st));
    A(talloc(&maxrank, 1, st));
    A(talloc(&key, (size_t)n, st));
    A(talloc(&tile, (size_t)n, st));
    if (e == cudaSuccess) {
        A(cudaMemsetAsync(cellcnt, 0, G.ncell * sizeof(unsigned), st));
        A(cudaMemsetAsync(bincnt, 0, ntiles * sizeof(int), st));
        A(cudaMemsetAsync(maxrank, 0, sizeof(unsigned), st));
        if (n) k_rank<<<grid1(n), 256, 0, st>>>(n, G, S.cij, cellcnt, bincnt, maxrank, key, tile);
        A(cudaGetLastError());
    }
    std::vector<int> hcnt(ntiles);
    unsigned int hmax = 0;
    if (e == cudaSuccess) {
        A(cudaMemcpyAsync(hcnt.data(), bincnt, ntiles * sizeof(int), cudaMemcpyDeviceToHost, st));
        A(cudaMemcpyAsync(&hmax, maxrank, sizeof hmax, cudaMemcpyDeviceToHost, st));
        A(cudaStreamSynchronize(st));
    }
    if (e == cudaSuccess) {
        long long mx = 0;
        for (int t = 0; t < ntiles; t++) mx = std::max<long long>(mx, hcnt[t]);
        if (need) *need = mx;
        const long long cpt = (long long)G.tx * G.ty;
        if (mx > G.cap) {
            rc = PIC_ENOMEM;  // caller grows the bins and retries
        } else if ((long long)hmax + 1 > (long long)(0xffffffffu / cpt)) {
            err = "a cell holds too many particles of one species for the bin keys";
            rc = PIC_EINVAL;  // (not PIC_ENOMEM: larger bins would not help)
        } else {
            // a tile's keys are rank * cells + cell: ranks 0 .. hmax. Tiles go in groups
            // whose bitmaps fit a fixed budget (one group unless cells are very uneven).
            const long long words = ((long long)(hmax + 1) * cpt + 31) / 32;
            const long long budget = 64ll << 20;  // bitmap words per group (256 MB)
            const int group = (int)std::max(1ll, std::min<long long>(ntiles, budget / words));
            A(talloc(&bits, (size_t)group * words, st));
            A(talloc(&pref, (size_t)group * words, st));
            for (int t0 = 0; t0 < ntiles && e == cudaSuccess; t0 += group) {
                const int ntg = std::min(group, ntiles - t0);
                A(cudaMemsetAsync(bits, 0, (size_t)ntg * words * sizeof(unsigned), st));
                if (n) k_setbits<<<grid1(n), 256, 0, st>>>(n, key, tile, t0, ntg, words, bits);
                k_scanbits<<<(unsigned)ntg, 256, 0, st>>>(words, bits, pref);
                if (n)
                    k_scatter<<<grid1(n), 256, 0, st>>>(n, G, s, key, tile, t0, ntg, words, bits, pref, S,
                                                        m->buf[par]);
                A(cudaGetLastError());
            }
            if (e == cudaSuccess) {
                k_set_counts<<<grid1(ntiles), 256, 0, st>>>(ntiles, s, bincnt, cnt_of(m, par, g));
                A(cudaGetLastError());
                A(cudaStreamSynchronize(st));
            }
        }
    }
    void* ps[] = {cellcnt, bincnt, maxrank, key, tile, bits, pref};
    for (void* p : ps) tfree(p, st);
    if (e != cudaSuccess) {
        err = std::string("bin sort failed: ") + cudaGetErrorString(e);
        return PIC_ECUDA;
    }
    return rc;
}

// Refuses work on bins that could not be allocated anew: their particles are gone.
int check_bins(const MixedState* m, std::string& err) {
    if (!m->lost) return PIC_OK;
    err = "the particles were lost when their bins could not be allocated; free the handle";
    return PIC_ESTATE;
}

// All live particles of species s of simulation g (every bin segment of buffer `par` +
// its overflow-list entries) into a new staging set.
int gather_species(MixedState* m, int g, int par, int s, PartArrays& S, long long& n, cudaStream_t st,
                   std::string& err) {
    if (int rc = check_bins(m, err)) return rc;
    const GridDev& G = m->G[g];
    const long long nb_seg = (long long)G.ntiles * kSegs;
    std::vector<int> cnt(2 * nb_seg);
    MCK(cudaMemcpyAsync(cnt.data(), cnt_of(m, par, g), cnt.size() * sizeof(int), cudaMemcpyDeviceToHost, st));
    DevStatus hs{};
    MCK(cudaMemcpyAsync(&hs, m->st, sizeof hs, cudaMemcpyDeviceToHost, st));
    MCK(cudaStreamSynchronize(st));
    std::vector<long long> off(nb_seg + 1, 0);
    for (int t = 0; t < G.ntiles; t++)
        for (int k = 0; k < kSegs; k++) {
            const long long lim = k == 0 ? G.cap : G.capo;
            const long long q = (long long)t * kSegs + k;
            off[q + 1] = off[q] + std::min<long long>(cnt[((long long)t * 2 + s) * kSegs + k], lim);
        }
    const long long nb = off[nb_seg];
    const long long no = std::min<long long>((long long)hs.ovf_count[par], m->ovf_cap);
    MCK(alloc_parts(S, (size_t)(nb + no), false, st));
    long long* doff = nullptr;
    unsigned long long* cursor = nullptr;
    MCK(talloc(&doff, off.size(), st));
    MCK(talloc(&cursor, 1, st));
    MCK(cudaMemcpyAsync(doff, off.data(), off.size() * sizeof(long long), cudaMemcpyHostToDevice, st));
    MCK(cudaMemsetAsync(cursor, 0, sizeof(unsigned long long), st));
    k_gather_bins<<<(unsigned)nb_seg, 256, 0, st>>>(G, s, cnt_of(m, par, g), doff, m->buf[par], S);
    if (no) k_gather_overflow<<<grid1(no), 256, 0, st>>>(no, s | (g << 1), m->ovf[par], nb, cursor, S);
    unsigned long long hcur = 0;
    MCK(cudaMemcpyAsync(&hcur, cursor, sizeof hcur, cudaMemcpyDeviceToHost, st));
    MCK(cudaStreamSynchronize(st));
    tfree(doff, st);
    tfree(cursor, st);
    n = nb + (long long)hcur;
    return PIC_OK;
}

// The tile kernels' work items (tile_plan.h): the wanted size from the particles there are, the
// parts of a tile from those its bins have room for.
int plan_items(MixedState* m, std::string& err) {
    std::vector<int2> items;
    for (int P = 1; P <= 3; P++) {
        m->item_first[P] = (int)items.size();
        double mean = 0.0;
        for (int g = 0; g < m->ngrids; g++)
            if (m->G[g].order == P) mean += m->expect[g] * m->G[g].ntiles / m->order_n[P];
        const double size = split_size(m->order_n[P], std::max(m->resident[P], 1), mean);
        for (int g = 0; g < m->ngrids; g++) {
            GridDev& G = m->G[g];
            if (G.order != P) continue;
            const TileSplit t = split_tile(G.cap * (2.0 / kBinSlack), m->expect[g], size);
            G.parts = t.parts;
            G.pchunk = t.pchunk;
        }
        for (int q = m->order_first[P]; q < m->order_first[P] + m->order_n[P]; q++)
            for (int part = 0; part < m->G[m->host_tile_grid[m->tlist[q]]].parts; part++)
                items.push_back(make_int2(m->tlist[q], part));
        m->item_n[P] = (int)items.size() - m->item_first[P];
        m->pblocks[P] = std::min(m->item_n[P], m->resident[P]);
    }
    if (m->items) cudaFree(m->items);
    m->items = nullptr;
    if (dalloc(&m->items, items.size()) != cudaSuccess) {
        cudaGetLastError();
        err = "work item allocation failed (" + std::to_string(items.size()) + " items)";
        return PIC_ENOMEM;
    }
    MCK(cudaMemcpy(m->items, items.data(), items.size() * sizeof(int2), cudaMemcpyHostToDevice));
    return PIC_OK;
}

// (Re)allocate both bin buffers with per-simulation stayer capacity cap[g] and outbox
// capacity capo[g] (contents are not preserved; all counts are zeroed).
int alloc_bins(MixedState* m, const std::vector<long long>& cap, const std::vector<long long>& capo,
               cudaStream_t st, std::string& err) {
    m->lost = true;  // until the caller has filled them
    for (int p = 0; p < 2; p++) {
        if (m->buf[p]) cudaFree(m->buf[p]);
        m->buf[p] = nullptr;
    }
    m->gen++;
    long long off = 0;
    for (int g = 0; g < m->ngrids; g++) {
        GridDev& G = m->G[g];
        G.cap = cap[g];
        G.capo = capo[g];
        G.bin_off = off;
        off += (long long)G.ntiles * 2 * bin_stride(G);
    }
    m->nslots = off;
    if (int rc = plan_items(m, err)) return rc;
    for (int p = 0; p < 2; p++) {
        cudaError_t e = dalloc(&m->buf[p], (size_t)m->nslots * kFields);
        if (e != cudaSuccess) {
            cudaGetLastError();
            err = "bin allocation failed (" + std::to_string(m->nslots) + " slots per buffer)";
            return PIC_ENOMEM;
        }
        MCK(cudaMemsetAsync(m->cnt[p], 0, (size_t)m->ntiles_total * (2 * kSegs + 1) * sizeof(int), st));
    }
    return PIC_OK;
}

// Gather every simulation's particles of buffer `par` into staging.
int gather_all(MixedState* m, int par, Staged& A, cudaStream_t st, std::string& err) {
    for (int g = 0; g < m->ngrids; g++)
        for (int s = 0; s < 2; s++)
            if (int rc = gather_species(m, g, par, s, A.S[2 * g + s], A.n[2 * g + s], st, err)) return rc;
    return PIC_OK;
}

// Allocate bins of at least the given capacities and sort everything staged in A into
// buffer `par`, growing a simulation's stayer capacity whenever one of its bins would
// overflow. Uploads the descriptors and clears the overflow lists.
int place_all(MixedState* m, int par, Staged& A, std::vector<long long> cap, std::vector<long long> capo,
              cudaStream_t st, std::string& err) {
    int rc = PIC_OK;
    for (int g = 0; g < m->ngrids; g++)  // (a species that is still to be loaded is like the other)
        if (const long long n = std::max(A.n[2 * g], A.n[2 * g + 1])) m->expect[g] = 2.0 * n / m->G[g].ntiles;
    for (int attempt = 0; attempt < 8; attempt++) {
        rc = alloc_bins(m, cap, capo, st, err);
        if (rc) return rc;
        bool grown = false;
        for (int g = 0; g < m->ngrids && rc == PIC_OK; g++)
            for (int s = 0; s < 2 && rc == PIC_OK; s++) {
                long long need = 0;
                rc = sort_into_bins(m, g, par, s, A.S[2 * g + s], A.n[2 * g + s], st, &need, err);
                if (rc == PIC_ENOMEM) {
                    cap[g] = std::max(cap[g] * 3 / 2 + 32, round32(1.25 * (double)need + 32.0));
                    grown = true;
                }
            }
        if (!grown) break;
        rc = PIC_ENOMEM;
    }
    if (rc) return rc;
    MCK(cudaMemcpyAsync((void*)m->dgrids, m->G, m->ngrids * sizeof(GridDev), cudaMemcpyHostToDevice, st));
    MCK(cudaMemsetAsync(&m->st->ovf_count, 0, sizeof(DevStatus::ovf_count), st));
    // the counts now come from the bins themselves, injected pairs included
    MCK(cudaMemsetAsync(m->injected, 0, 2 * m->ngrids * sizeof(unsigned long long), st));
    MCK(cudaStreamSynchronize(st));
    for (int q = 0; q < 2 * m->ngrids; q++) m->n[q] = A.n[q];
    m->lost = false;
    return PIC_OK;
}

// Re-sort every simulation into fresh bins with capacities at least (cap_min, capo_min).
int rebuild(MixedState* m, std::vector<long long> cap_min, std::vector<long long> capo_min,
            cudaStream_t st, std::string& err) {
    DevStatus hs{};
    if (int rc = read_status(m, hs, st, err)) return rc;
    const int par = (int)hs.parity;
    Staged A(m->ngrids, st);
    if (int rc = gather_all(m, par, A, st, err)) return rc;
    for (int g = 0; g < m->ngrids; g++) {
        cap_min[g] = std::max(cap_min[g], m->G[g].cap);
        capo_min[g] = std::max(capo_min[g], m->G[g].capo);
    }
    if (int rc = place_all(m, par, A, cap_min, capo_min, st, err)) return rc;
    m->rebins++;
    return PIC_OK;
}

std::vector<long long> current_caps(MixedState* m, bool outboxes) {
    std::vector<long long> v(m->ngrids);
    for (int g = 0; g < m->ngrids; g++) v[g] = outboxes ? m->G[g].capo : m->G[g].cap;
    return v;
}

}  // namespace

// =====================================================================================

cudaError_t temp_alloc(void** p, size_t bytes, cudaStream_t st) {
    *p = nullptr;
    cudaError_t e = cudaSuccess;
    cudaMemPool_t pool = temp_pool(&e);
    if (!pool) return e == cudaSuccess ? cudaErrorMemoryAllocation : e;
    return cudaMallocFromPoolAsync(p, bytes ? bytes : 1, pool, st);
}

cudaError_t scratch_alloc(void** p, size_t bytes, cudaStream_t st) {
    if (bytes <= kScratchKept) return temp_alloc(p, bytes, st);
    *p = nullptr;
    return cudaMallocAsync(p, bytes, st);
}

void temp_free(void* p, cudaStream_t st) {
    if (p) cudaFreeAsync(p, st);
}

int mixed_create(MixedState** out, const pic_params* p, int ngrids, GridDev* G,
                 const GridDev* dgrids, long long ntot, float* F32, long long* Jfix, CgState* cg,
                 DevStatus* st, std::string& err) {
    *out = nullptr;
    MixedState* m = new MixedState();
    m->ngrids = ngrids;
    m->G = G;
    m->dgrids = dgrids;
    m->ntot = ntot;
    m->F32 = F32;
    m->Jfix = Jfix;
    m->cg = cg;
    m->st = st;
    m->n.assign(2 * ngrids, 0);
    // tiles of every simulation, one global numbering
    int ntiles = 0;
    long long expect = 0;
    std::vector<long long> cap(ngrids), capo(ngrids);
    for (int g = 0; g < ngrids; g++) {
        const pic_params& q = p[g];
        GridDev& D = G[g];
        int tx = q.tile_x, ty = q.tile_y;
        if (tx <= 0) tx = std::min(32, q.nx);
        if (ty <= 0) ty = std::min(16, q.ny);
        D.tx = std::min(tx, q.nx);
        D.ty = std::min(ty, q.ny);
        D.ntx = (q.nx + D.tx - 1) / D.tx;
        D.nty = (q.ny + D.ty - 1) / D.ty;
        D.ntiles = D.ntx * D.nty;
        D.tile_first = ntiles;
        ntiles += D.ntiles;
        D.wx = D.tx + 5;
        D.wy = D.ty + 5;
        const size_t sm = (size_t)6 * D.wx * D.wy * sizeof(int) + (size_t)6 * D.wx * D.wy * sizeof(float);
        m->smem[D.order] = std::max(m->smem[D.order], sm);
        const double slack = q.bin_slack > 0 ? q.bin_slack : kBinSlack;
        cap[g] = round32((double)q.ppc * D.tx * D.ty * slack + 64.0);
        m->expect.push_back(round32((double)q.ppc * D.tx * D.ty * kBinSlack + 64.0) * (2.0 / kBinSlack));
        capo[g] = round32((double)q.ppc * std::max(D.tx, D.ty) * 1.5 + 32.0);
        expect += 2ll * q.ppc * (long long)q.nx * q.ny;
    }
    m->ntiles_total = ntiles;
    // per-order tile lists, largest expected work first
    std::vector<int> tg(ntiles);
    std::vector<int>& tl = m->tlist;
    std::vector<std::pair<long long, int>> order_tiles[4];
    for (int g = 0; g < ngrids; g++) {
        const GridDev& D = G[g];
        for (int t = 0; t < D.ntiles; t++) {
            tg[D.tile_first + t] = g;
            const int tyi = t / D.ntx, txi = t - tyi * D.ntx;
            const long long cells = (long long)(std::min(D.tx, D.nx - txi * D.tx)) *
                                    std::min(D.ty, D.ny - tyi * D.ty);
            order_tiles[D.order].push_back({cells * p[g].ppc, D.tile_first + t});
        }
    }
    for (int P = 1; P <= 3; P++) {
        std::stable_sort(order_tiles[P].begin(), order_tiles[P].end(),
                         [](const std::pair<long long, int>& x, const std::pair<long long, int>& y) {
                             return x.first > y.first;
                         });
        m->order_first[P] = (int)tl.size();
        m->order_n[P] = (int)order_tiles[P].size();
        for (auto& e : order_tiles[P]) tl.push_back(e.second);
    }
    m->host_tile_grid = tg;
    m->ovf_cap = std::max<long long>(65536, expect / 8);
    m->ovf_cap = (m->ovf_cap + 31) / 32 * 32;
    cudaError_t e = cudaSuccess;
    for (int q = 0; q < 2 && e == cudaSuccess; q++) {
        e = dalloc(&m->cnt[q], (size_t)ntiles * (2 * kSegs + 1));
        if (e == cudaSuccess) m->ovf_in[q] = m->cnt[q] + (size_t)ntiles * 2 * kSegs;
        if (e == cudaSuccess) e = dalloc(&m->ovf[q].p, (size_t)m->ovf_cap * kFields);
        if (e == cudaSuccess) e = dalloc(&m->ovf[q].gs, (size_t)m->ovf_cap);
    }
    // injector tables
    {
        std::vector<int> ig;
        std::vector<long long> first(1, 0);
        for (int g = 0; g < ngrids; g++) {
            if (!G[g].inject) continue;
            const double w = (1.0 + std::sqrt(1.0 - 1.0 / (G[g].gamma0 * G[g].gamma0))) * G[g].cfl;
            const long long kmax = (long long)std::ceil(G[g].ppc * w) + 1;
            ig.push_back(g);
            first.push_back(first.back() + (long long)G[g].ny * kmax);
        }
        m->inject_grids = (int)ig.size();
        m->inject_threads = first.back();
        if (e == cudaSuccess) e = dalloc(&m->injected, (size_t)2 * ngrids);
        if (e == cudaSuccess) e = cudaMemset(m->injected, 0, 2 * ngrids * sizeof(unsigned long long));
        if (e == cudaSuccess && !ig.empty()) {
            e = dalloc(&m->inj_grid, ig.size());
            if (e == cudaSuccess) e = dalloc(&m->inj_first, first.size());
            if (e == cudaSuccess) e = cudaMemcpy(m->inj_grid, ig.data(), ig.size() * sizeof(int), cudaMemcpyHostToDevice);
            if (e == cudaSuccess)
                e = cudaMemcpy(m->inj_first, first.data(), first.size() * sizeof(long long), cudaMemcpyHostToDevice);
        }
    }
    if (e == cudaSuccess) e = dalloc(&m->tile_grid, (size_t)ntiles);
    if (e == cudaSuccess) e = dalloc(&m->work, 4);
    if (e == cudaSuccess) e = cudaMemcpy(m->tile_grid, tg.data(), ntiles * sizeof(int), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemset(m->work, 0, 4 * sizeof(int));
    int rc = PIC_OK;
    // Shared-memory opt-in: only ever raised, since the attribute belongs to the kernel
    // and other handles in the process may need more than this one.
    int dev = 0;
    if (e == cudaSuccess) e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&m->nsm, cudaDevAttrMultiProcessorCount, dev);
    auto setup = [&](auto kern, int P) {
        if (m->order_n[P] == 0) return cudaSuccess;
        cudaFuncAttributes fa{};
        cudaError_t r = cudaFuncGetAttributes(&fa, kern);
        if (r == cudaSuccess && (size_t)fa.maxDynamicSharedSizeBytes < m->smem[P])
            r = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)m->smem[P]);
        int nb = 0;
        if (r == cudaSuccess)
            r = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kern, kTileThreads, m->smem[P]);
        if (r == cudaSuccess && nb < 1) r = cudaErrorInvalidConfiguration;
        m->resident[P] = nb * m->nsm;
        return r;
    };
    if (rc == PIC_OK && e == cudaSuccess) e = setup(k_push_tile<1>, 1);
    if (rc == PIC_OK && e == cudaSuccess) e = setup(k_push_tile<2>, 2);
    if (rc == PIC_OK && e == cudaSuccess) e = setup(k_push_tile<3>, 3);
    // (the densities' window at its largest: the same value from every handle)
    const int dens = 3 * kMaxWinCells * (int)sizeof(unsigned);
    for (const auto& k : kDensityKernels)
        for (int mom = 0; mom < 2; mom++)
            if (e == cudaSuccess) e = cudaFuncSetAttribute(k[mom], cudaFuncAttributeMaxDynamicSharedMemorySize, dens);
    if (rc == PIC_OK && e == cudaSuccess) {
        rc = alloc_bins(m, cap, capo, 0, err);
        if (rc == PIC_OK) e = cudaDeviceSynchronize();
    }
    if (rc == PIC_OK && e == cudaSuccess) {
        e = cudaMemcpy((void*)dgrids, G, ngrids * sizeof(GridDev), cudaMemcpyHostToDevice);
    }
    if (rc == PIC_OK && e != cudaSuccess) {
        err = std::string("MIXED32 setup failed: ") + cudaGetErrorString(e);
        cudaGetLastError();
        rc = PIC_ENOMEM;
    }
    if (rc != PIC_OK) {
        mixed_destroy(m);
        return rc;
    }
    m->lost = false;
    *out = m;
    return PIC_OK;
}

void mixed_destroy(MixedState* m) {
    if (!m) return;
    for (int p = 0; p < 2; p++) {
        void* ps[] = {m->buf[p], m->ovf[p].p, m->ovf[p].gs, m->cnt[p]};
        for (void* q : ps)
            if (q) cudaFree(q);
    }
    void* ps[] = {m->tile_grid, m->items, m->work, m->injected, m->inj_grid, m->inj_first};
    for (void* q : ps)
        if (q) cudaFree(q);
    delete m;
}

int mixed_load(MixedState* m, int g, int s, const double* x, const double* y, const double* ux,
               const double* uy, const double* uz, long long n, cudaStream_t st, std::string& err) {
    if (int rc = check_bins(m, err)) return rc;
    DevStatus hs{};
    if (int rc = read_status(m, hs, st, err)) return rc;
    // fold any overflow-list particles back into bins first so the list holds none of s
    if (hs.ovf_count[hs.parity]) {
        int rc = rebuild(m, current_caps(m, false), current_caps(m, true), st, err);
        if (rc) return rc;
    }
    const int par = (int)hs.parity;
    double* in = nullptr;
    PartArrays S{};
    unsigned long long* nbad = nullptr;
    MCK(talloc(&in, 5 * (size_t)std::max<long long>(n, 1), st));
    const double* src[5] = {x, y, ux, uy, uz};
    for (int a = 0; a < 5 && n; a++)
        MCK(cudaMemcpyAsync(in + a * n, src[a], n * sizeof(double), cudaMemcpyDefault, st));
    MCK(alloc_parts(S, (size_t)n, false, st));
    MCK(talloc(&nbad, 1, st));
    MCK(cudaMemsetAsync(nbad, 0, sizeof(unsigned long long), st));
    if (n)
        k_stage_fp64<<<grid1(n), 256, 0, st>>>(n, in, in + n, in + 2 * n, in + 3 * n, in + 4 * n, m->G[g],
                                               S, nbad);
    unsigned long long hbad = 0;
    MCK(cudaMemcpyAsync(&hbad, nbad, sizeof hbad, cudaMemcpyDeviceToHost, st));
    MCK(cudaStreamSynchronize(st));
    tfree(in, st);
    tfree(nbad, st);
    if (hbad) {
        free_parts(S, st);
        err = "non-finite particle position or momentum, or a position outside the walls";
        return PIC_EINVAL;
    }
    long long need = 0;
    int rc = sort_into_bins(m, g, par, s, S, n, st, &need, err);  // also zeroes s's outbox counts
    if (rc == PIC_ENOMEM) {
        // a bin would overflow: re-sort everything with larger bins for this simulation
        Staged A(m->ngrids, st);
        rc = gather_all(m, par, A, st, err);
        if (rc == PIC_OK) {
            free_parts(A.S[2 * g + s], st);
            A.S[2 * g + s] = S;
            A.n[2 * g + s] = n;
            S = PartArrays{};
            std::vector<long long> cap = current_caps(m, false);
            cap[g] = std::max(cap[g], round32(1.25 * (double)need + 32.0));
            rc = place_all(m, par, A, cap, current_caps(m, true), st, err);
            m->rebins++;
        }
    } else if (rc == PIC_OK) {
        MCK(cudaMemcpyAsync((void*)(m->dgrids + g), m->G + g, sizeof(GridDev), cudaMemcpyHostToDevice, st));
        MCK(cudaStreamSynchronize(st));
        m->n[2 * g + s] = n;
    }
    free_parts(S, st);
    return rc;
}

void mixed_enqueue(MixedState* m, cudaStream_t st, int part) {
    if (part == 0) {
        const long long nj2 = (3 * m->ntot + 1) / 2;
        const int ncnt = m->ntiles_total * (2 * kSegs + 1);
        const unsigned nb = (unsigned)std::min<long long>(8 * m->nsm, std::max<long long>(1, (nj2 + 255) / 256));
        k_mixed_begin<<<nb, 256, 0, st>>>(make_args(m, 0), m->ngrids, nj2, ncnt, m->work);
        k_push_overflow<<<m->nsm, kTileThreads, 0, st>>>(make_args(m, 0));
    } else if (part == 1) {
        for (int P = 1; P <= 3; P++) {
            if (m->order_n[P] == 0) continue;
            const MixedArgs a = make_args(m, P);
            const unsigned nb = (unsigned)m->pblocks[P];
            switch (P) {
            case 1: k_push_tile<1><<<nb, kTileThreads, m->smem[1], st>>>(a); break;
            case 2: k_push_tile<2><<<nb, kTileThreads, m->smem[2], st>>>(a); break;
            default: k_push_tile<3><<<nb, kTileThreads, m->smem[3], st>>>(a); break;
            }
        }
    } else if (part == 2) {
        if (m->inject_grids)
            k_inject_mixed<<<(unsigned)((m->inject_threads + 255) / 256), 256, 0, st>>>(
                make_args(m, 0), m->inj_grid, m->inj_first, m->inject_grids, m->injected);
    } else {
        k_mixed_end<<<1, 128, 0, st>>>(m->st, m->ngrids, m->cg);
    }
}

int mixed_before_steps(MixedState* m, cudaStream_t, std::string& err) { return check_bins(m, err); }

int mixed_step_kernels(const MixedState* m) {
    int k = 3;  // k_mixed_begin, k_push_overflow, k_mixed_end
    for (int P = 1; P <= 3; P++) k += m->order_n[P] > 0 ? 1 : 0;
    return k + (m->inject_grids ? 1 : 0);
}

int mixed_after_steps(MixedState* m, const DevStatus& hs, cudaStream_t st, std::string& err) {
    if (m->inject_grids) {  // the injector's pairs join the live counts
        std::vector<unsigned long long> add((size_t)2 * m->ngrids);
        MCK(cudaMemcpyAsync(add.data(), m->injected, add.size() * sizeof(unsigned long long), cudaMemcpyDeviceToHost, st));
        MCK(cudaMemsetAsync(m->injected, 0, add.size() * sizeof(unsigned long long), st));
        MCK(cudaStreamSynchronize(st));
        for (size_t q = 0; q < add.size(); q++) m->n[q] += (long long)add[q];
    }
    const int par = (int)hs.parity;
    if (hs.ovf_count[par] == 0) return PIC_OK;
    // particles are parked in the overflow list: re-sort with room to spare. Grow each
    // simulation's stayer capacity to 1.25x its fullest tile and double its outboxes if
    // any is full.
    std::vector<int> cnt((size_t)m->ntiles_total * 2 * kSegs);
    MCK(cudaMemcpyAsync(cnt.data(), m->cnt[par], cnt.size() * sizeof(int), cudaMemcpyDeviceToHost, st));
    MCK(cudaStreamSynchronize(st));
    std::vector<long long> cap(m->ngrids), capo(m->ngrids);
    const long long excess = (long long)hs.ovf_count[par];  // upper bound on any tile's excess
    for (int g = 0; g < m->ngrids; g++) {
        const GridDev& G = m->G[g];
        long long mx = 0;
        bool outbox_full = false;
        for (long long b = (long long)G.tile_first * 2; b < (long long)(G.tile_first + G.ntiles) * 2; b++) {
            long long tot = 0;
            for (int k = 0; k < kSegs; k++) {
                tot += cnt[b * kSegs + k];
                if (k > 0 && cnt[b * kSegs + k] >= G.capo) outbox_full = true;
            }
            mx = std::max(mx, tot);
        }
        cap[g] = std::max(round32(1.25 * (double)std::min(mx + excess, 2 * mx + 64)), G.cap);
        capo[g] = outbox_full ? 2 * G.capo : G.capo;
    }
    return rebuild(m, cap, capo, st, err);
}

long long mixed_count(MixedState* m, int g, int s) { return m->n[2 * g + s]; }

int mixed_rho_momentum(MixedState* m, int g, const double q_s[2], double* rho, double* mom, cudaStream_t st,
                       std::string& err) {
    if (int rc = check_bins(m, err)) return rc;
    const GridDev& G = m->G[g];
    const DensityArgs d{{q_s[0], q_s[1]}, G.w, rho, mom};
    const int nbins = 2 * G.ntiles;
    // Parts of a bin: 4096 particles each (5120 of its capacity) keep the window's cost, its
    // zeroing and its nodes' FP64, below a tenth of the block's time; half as many where that
    // leaves fewer than the eight blocks that an SM holds (512 x 256, 8 per cell: 30 -> 22 us;
    // 1024 x 256, 16 per cell: 92 us against 98 with the short parts).
    const long long chunk = nbins * std::max(1ll, G.cap / 5120) < 8 * m->nsm ? 2560 : 5120;
    const dim3 nb((unsigned)nbins + 1, (unsigned)std::max(1ll, std::min(64ll, G.cap / chunk)));
    const size_t sm = d.rho ? (size_t)3 * G.wx * G.wy * sizeof(unsigned) : 0;
    const MixedArgs a = make_args(m, 0);
    const DensityKernel kern = kDensityKernels[G.order - 1][mom ? 1 : 0];
    kern<<<nb, 256, sm, st>>>(a, g, nbins, d);
    MCK(cudaGetLastError());
    return PIC_OK;
}
long long mixed_rebins(MixedState* m) { return m->rebins; }
long long mixed_generation(MixedState* m) { return m->gen; }

int mixed_particles(MixedState* m, int g, int s, double* out, long long n, cudaStream_t st,
                    std::string& err) {
    DevStatus hs{};
    if (int rc = read_status(m, hs, st, err)) return rc;
    PartArrays S{};
    long long got = 0;
    int rc = gather_species(m, g, (int)hs.parity, s, S, got, st, err);
    if (rc) return rc;
    if (got != n) {
        free_parts(S, st);
        err = "particle count mismatch (" + std::to_string(got) + " live, " + std::to_string(n) + " requested)";
        return PIC_ESTATE;
    }
    double* t = nullptr;
    MCK(talloc(&t, 5 * (size_t)std::max<long long>(n, 1), st));
    if (n) k_unstage<<<grid1(n), 256, 0, st>>>(n, m->G[g], S, t);
    MCK(cudaMemcpyAsync(out, t, 5 * n * sizeof(double), cudaMemcpyDefault, st));
    MCK(cudaStreamSynchronize(st));
    tfree(t, st);
    free_parts(S, st);
    return PIC_OK;
}

}  // namespace pic
