// Lattices kept on the chip for a whole launch: the steps of Eq. 1 for a
// two-buffer lattice that fits the GPU's shared memory.
//
// The lattice is cut into tiles of at most W columns by TH rows, one CTA
// each, all resident at once (a cooperative launch).  A CTA holds its tile's
// post-collision populations, decoded to the arithmetic type, in shared
// memory with a ring of two cells around them, and updates them in place:
//   phase 1  every warp pulls its rows into registers (13 loads a node) and
//            writes the moments of Eq. 2 to shared memory; the ring's
//            nearest rows and columns give the moments beside the tile;
//   phase 2  after a barrier, every warp collides its rows with the
//            neighbours' moments and writes the populations back, each
//            rounded through the storage type exactly as by the step kernel.
// The last two steps of a launch also write the lattice's buffers: the
// state, and the one before it for the residual.  Every value has the bits
// that the step kernel gives it.
//
// What bounds it.  The step kernel's time on a small lattice is the latency
// of one tile through L2: staged rows, moments, one collision, stores, the
// release and the neighbours' acquire.  Here a step is two barriers, one
// collision's latency per row a warp holds, and the exchange of the ring.
// us per step, the step kernel against this one (one jet, 200 steps a launch):
// 64 x 32 FP32 6.7 -> 3.0 (the pipe 5.2 -> 2.9), 200 x 96 FP32 8.7 -> 3.0 and FP64 19.5 -> 16.1,
// 900 x 140 FP32 11.5 -> 4.3, 640 x 160 FP16 moment-split 15.4 -> 4.4,
// 1024 x 256 16.4 -> 7.3 and FP32 12.6 -> 6.0.  With the exchange's waits taken out the last
// takes 4.6: the rest is the way of a value through L2 and the slowest tile
// of each neighbourhood, one at a lattice edge, whose ghosts come after its
// collisions.
//
// Exchange.  A tile sends the values that the rings of the eight tiles
// around it hold straight to their inboxes in device memory, each in one
// 8-byte word with the number of its step: a reader polls the values
// themselves, so a step costs one store and one load across L2 and no fence,
// flag or extra round trip.  (With the ring kept in the lattice's buffers
// and flags released after the stores, 1024 x 256 FP32 took 5 us a step
// longer.)  An
// inbox has two halves, for even and odd steps: a tile sends step k + 2 only
// after it has read every neighbour's step k + 1, which was sent after the
// neighbour had read step k.
//
// Deadlock freedom.  All CTAs are resident, and a tile of step k waits only
// for tiles of step k - 1.  The waits are bounded all the same: a wait that
// runs out raises LBM_STATUS_TIMEOUT, and every CTA leaves.
#pragma once

#include "lbm_kernels.cuh"

namespace lbm {

struct ResCtl {
    unsigned long long *box;  // inboxes: [step parity][tile][RES_WORDS]
    unsigned base;            // number of the launch's first step
    int nsteps;
    int ns, nb;               // tiles across and up
    int spin_limit;
    int first;                // first step of the launch (0; the self-test starts at 1, whose waits are never met)
};

// one of nt near-equal parts of n: its first element and its length
__device__ __forceinline__ void res_part(int n, int nt, int t, int &lo, int &len)
{
    lo = (int)((int64_t)n * t / nt);
    len = (int)((int64_t)n * (t + 1) / nt) - lo;
}

struct ResTile {
    int ts, tb;  // tile column and row
    int x0, w;   // its columns x0 .. x0 + w - 1
    int j0, h;   // its rows
    __device__ __forceinline__ ResTile(int nx, int nr, int ns, int nb, int t)
    {
        ts = t % ns;
        tb = t / ns;
        res_part(nx, ns, ts, x0, w);
        res_part(nr, nb, tb, j0, h);
    }
};

// tile shapes: the most rows of a tile, the rows a warp holds and the nodes a lane holds of a
// row (at most `widest`: 2, in FP64 1; FP64 has shapes 0 and 2)
__host__ __device__ constexpr int res_rows(int shape) { return shape == 0 || shape == 3 ? 8 : 16; }
__host__ __device__ constexpr int res_nv(int shape, int widest) { return shape == 3 ? 1 : widest; }
__host__ __device__ constexpr int res_rpw(int shape) { return shape == 1 ? 2 : 1; }

constexpr int RES_CORNERS = 32;     // corner entries of an inbox (res_corner; two unused)
constexpr int RES_EDGES = 6;        // tasks of filling ghosts: left, right, bottom and top in halves of 32 columns
constexpr int RES_SEND_MAX = 96;    // corner entries a tile sends

// a tile's shared memory: 13 planes of populations with a ring of two cells,
// three planes of moments (rho u_x, rho u_r, T - T0) with a ring of one, the
// property table, and the corner entries the tile receives and sends
template <class C, int NV, int TH>
struct ResMem {
    static constexpr int W = 32 * NV;
    static constexpr int PW = W + 4, PL = (TH + 4) * PW;
    static constexpr int MW = W + 2, ML = (TH + 2) * MW;
    static constexpr int VALUES = (13 * PL + 3 * ML) * (int)sizeof(C);
    static constexpr int TAB = std::is_same<C, float>::value ? SMEM_TAB * (int)sizeof(float2) : 0;
    // words of an inbox: 24 plane rows, 16 plane columns, corners
    static constexpr int WPV = (int)sizeof(C) / 4;
    static constexpr int COLS = 24 * W, CORNERS = COLS + 16 * TH, ENTRIES = CORNERS + RES_CORNERS;
    static constexpr int WORDS = ENTRIES * WPV;
    static constexpr int BYTES = VALUES + TAB + RES_SEND_MAX * 8 + 8 + ENTRIES * 2;
    C *pop, *mom;  // population 0 and rho u_x of the tile's first node
    unsigned char *raw;
    // (from the declaration of the dynamic shared memory, so that every access is one to shared memory)
    __device__ __forceinline__ ResMem()
    {
        extern __shared__ __align__(16) unsigned char smem_raw[];
        raw = smem_raw;
        pop = reinterpret_cast<C *>(raw) + 2 * PW + 2;
        mom = reinterpret_cast<C *>(raw) + 13 * PL + MW + 1;
    }
    __device__ __forceinline__ C &P(int q, int r, int c) const { return pop[q * PL + r * PW + c]; }
    __device__ __forceinline__ C &M(int m, int r, int c) const { return mom[m * ML + r * MW + c]; }
    __device__ __forceinline__ float2 *tab() const { return reinterpret_cast<float2 *>(raw + VALUES); }
    // corner entries to send: (offset in pop, who sends it) and the destination word; their number
    __device__ __forceinline__ int2 *send() const { return reinterpret_cast<int2 *>(raw + VALUES + TAB); }
    __device__ __forceinline__ int &nsend() const { return *reinterpret_cast<int *>(send() + RES_SEND_MAX); }
    // entries of the inbox that a warp has taken charge of in this step
    __device__ __forceinline__ int &taken() const { return (&nsend())[1]; }
    // where each entry received goes (an offset from the first value), or RES_NONE
    __device__ __forceinline__ unsigned short *recv() const
    {
        return reinterpret_cast<unsigned short *>(send() + RES_SEND_MAX) + 4;
    }
};
constexpr int RES_NONE = 0xffff;

// 8-byte words of a tile's inbox
__host__ __device__ constexpr int64_t res_box_words(int value_bytes, int shape)
{
    return (int64_t)(24 * 32 * res_nv(shape, value_bytes == 8 ? 1 : 2) + 16 * res_rows(shape) + RES_CORNERS) *
           (value_bytes / 4);
}

// a value and the number of its step, one 8-byte word per 4 bytes of value
template <class C>
__device__ __forceinline__ void box_put(unsigned long long *b, C v, unsigned seq)
{
    if constexpr (sizeof(C) == 4) {
        const unsigned long long w = (unsigned long long)seq << 32 | __float_as_uint(v);
        asm volatile("st.relaxed.gpu.global.b64 [%0], %1;\n" ::"l"(b), "l"(w) : "memory");
    } else {
        const unsigned long long u = (unsigned long long)__double_as_longlong(v), s = (unsigned long long)seq << 32;
        asm volatile("st.relaxed.gpu.global.b64 [%0], %1;\n" ::"l"(b), "l"(s | (u & 0xffffffffull)) : "memory");
        asm volatile("st.relaxed.gpu.global.b64 [%0], %1;\n" ::"l"(b + 1), "l"(s | (u >> 32)) : "memory");
    }
}

__device__ __forceinline__ unsigned long long box_word(const unsigned long long *b)
{
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.b64 %0, [%1];\n" : "=l"(v) : "l"(b) : "memory");
    return v;
}

// the value of an entry; clears ok if it is not that of step seq yet
template <class C>
__device__ __forceinline__ C box_get(const unsigned long long *b, unsigned seq, bool &ok)
{
    const unsigned long long w = box_word(b);
    ok = ok && (unsigned)(w >> 32) == seq;
    if constexpr (sizeof(C) == 4) {
        return __uint_as_float((unsigned)w);
    } else {
        const unsigned long long x = box_word(b + 1);
        ok = ok && (unsigned)(x >> 32) == seq;
        return __longlong_as_double((long long)((w & 0xffffffffull) | (x << 32)));
    }
}

// ---- which ring cells a tile takes from others ---------------------------------------
// Ring rows and columns beside a tile lie in the tiles beside it; each plane
// of them that a pull reads is sent: of rows -1 and h the planes without
// radial velocity and those that move into the tile, of rows -2 and h + 1
// (for the moments of the ring's rows) the latter, of columns -1 and w those
// that move into the tile and f2, f4 (for rho u_r there), of -2 and w + 1
// f5, f8 and f6, f7.  The corners, and the boundary values that a
// neighbour's edge node writes, are single entries:
// entry e of a tile: population q of cell (r, c), in tile coordinates; false if unused
struct ResEntry {
    int q, r, c;
};
__device__ __forceinline__ bool res_corner(const ResTile &a, int nx, int nr, int e, ResEntry &x)
{
    const bool below = a.j0 > 0, above = a.j0 + a.h < nr, left = a.x0 > 0, right = a.x0 + a.w < nx;
    if (e < 24) {
        const int m = e % 6;
        const bool east = (e / 6) & 1, north = e >= 12;
        const bool side = east ? right : left, end = north ? above : below;
        x.r = north ? a.h + (m == 5) : -1 - (m == 5);
        x.c = east ? a.w + (m == 4) : -1 - (m == 4);
        x.q = north ? (east ? 7 : 8) : (east ? 6 : 5);  // pulled by the corner node and the ring's nodes beside it
        if (m == 1)
            x.q = north ? 4 : 2;
        if (m == 2)
            x.q = east ? 3 : 1;
        if (m == 3)
            x.q = east ? 11 : 9;
        return m == 0 ? side || end : (m == 1 || m == 4 ? side : end);
    }
    // a wall's bounced-back value for the node beside the tile, beyond the tile's own edge node
    const int m = e - 24;
    if (m >= 6)
        return false;
    x.q = m == 0 || m == 5 ? 6 : (m == 1 ? 5 : (m == 3 ? 8 : 7));
    x.c = m < 4 ? (m & 1 ? a.w - 1 : 0) : a.w;
    x.r = m < 4 ? (m < 2 ? -1 : a.h) : (m == 4 ? 0 : a.h - 1);
    return m < 4 ? (m & 1 ? right : left) && !(m < 2 ? below : above) : !right && (m == 4 ? below : above);
}

// the node whose collision or boundary rule writes population q of cell (i, j)
template <class C>
__device__ __forceinline__ void res_writer(const StepParams<C> &p, int q, int i, int j, int &wi, int &wj)
{
    wi = i;
    wj = j;
    if (j < 0 && p.bc_bottom == BOTTOM_WALL)
        wi += q == 5 ? 1 : (q == 6 ? -1 : 0);
    if (j >= p.nr && p.bc_top == TOP_WALL)
        wi += q == 7 ? -1 : (q == 8 ? 1 : 0);
    if (i >= p.nx && p.bc_out == OUT_WALL)
        wj += q == 6 ? 1 : (q == 7 ? -1 : 0);
    wi = min(max(wi, 0), p.nx - 1);
    wj = min(max(wj, 0), p.nr - 1);
}

// Lists where the entries the tile receives go, and the corner entries it
// sends.  An entry sent is tagged with its sender: the warp that holds the
// node's row, or 64 + the edge task (RES_EDGES) whose ghost it is.
template <class C, int NV, int TH, int RPW>
__device__ __noinline__ void res_lists(const StepParams<C> &p, const int ns, const int nb, const ResTile a)
{
    using Mem = ResMem<C, NV, TH>;
    const Mem t;
    const bool below = a.j0 > 0, above = a.j0 + a.h < p.nr, left = a.x0 > 0, right = a.x0 + a.w < p.nx;
    for (int e = threadIdx.x; e < Mem::ENTRIES; e += blockDim.x) {
        ResEntry x;
        bool used;
        if (e < Mem::COLS) {  // plane n of the rows: FLAT, UP of -1; UP of -2; FLAT, DOWN of h; DOWN of h + 1
            const int n = e / Mem::W, u = n >> 2;
            constexpr unsigned flat = 1u | 3u << 4 | 9u << 8 | 11u << 12, up = 2u | 5u << 4 | 6u << 8 | 10u << 12,
                               down = 4u | 7u << 4 | 8u << 8 | 12u << 12;
            x.q = (int)((u == 0 || u == 3 ? flat : (u < 3 ? up : down)) >> (4 * (n & 3)) & 15u);
            x.r = u < 3 ? (u == 2 ? -2 : -1) : (u == 5 ? a.h + 1 : a.h);
            x.c = e % Mem::W;
            used = (u < 3 ? below : above) && x.c < a.w;
        } else if (e < Mem::CORNERS) {  // plane n of the columns -1, -2; w, w + 1
            const int n = (e - Mem::COLS) / TH, m = n & 7;
            constexpr unsigned west = 5u | 8u << 4 | 1u << 8 | 9u << 12 | 2u << 16 | 4u << 20 | 5u << 24 | 8u << 28,
                               east = 6u | 7u << 4 | 3u << 8 | 11u << 12 | 2u << 16 | 4u << 20 | 6u << 24 | 7u << 28;
            x.q = (int)((n < 8 ? west : east) >> (4 * m) & 15u);
            x.r = (e - Mem::COLS) % TH;
            x.c = n < 8 ? (m < 6 ? -1 : -2) : (m < 6 ? a.w : a.w + 1);
            used = (n < 8 ? left : right) && x.r < a.h;
        } else {
            used = res_corner(a, p.nx, p.nr, e - Mem::CORNERS, x);
            if (used) {
                int wi, wj;
                res_writer<C>(p, x.q, a.x0 + x.c, a.j0 + x.r, wi, wj);
                used = wi < a.x0 || wi >= a.x0 + a.w || wj < a.j0 || wj >= a.j0 + a.h;
            }
        }
        t.recv()[e] = used ? x.q * Mem::PL + (x.r + 2) * Mem::PW + x.c + 2 : RES_NONE;
    }
    for (int n = threadIdx.x; n < 9 * RES_CORNERS; n += blockDim.x) {
        const int d = n / RES_CORNERS, e = n % RES_CORNERS;
        const int s = a.ts + d % 3 - 1, b = a.tb + d / 3 - 1;
        if (d == 4 || s < 0 || s >= ns || b < 0 || b >= nb)
            continue;
        const ResTile o(p.nx, p.nr, ns, nb, b * ns + s);
        ResEntry x;
        if (!res_corner(o, p.nx, p.nr, e, x))
            continue;
        const int i = o.x0 + x.c, j = o.j0 + x.r;
        int wi, wj;
        res_writer<C>(p, x.q, i, j, wi, wj);
        if (wi < a.x0 || wi >= a.x0 + a.w || wj < a.j0 || wj >= a.j0 + a.h)
            continue;
        int who = (j - a.j0) / RPW;
        if (i < 0 || i >= p.nx)
            who = 64 + (i < 0 ? 0 : 1);
        else if (j < 0 || j >= p.nr)
            who = 64 + (j < 0 ? 2 : 4) + (wi - a.x0 >= 32);
        const int m = atomicAdd(&t.nsend(), 1);
        if (m < RES_SEND_MAX)
            t.send()[m] = make_int2((x.q * Mem::PL + (j - a.j0) * Mem::PW + (i - a.x0) + 1024) | who << 20,
                                    ((b * ns + s) * Mem::ENTRIES + Mem::CORNERS + e) * Mem::WPV);
    }
}

// ---- receiving ---------------------------------------------------------------------------
// one more poll of a wait?  Sleeps between polls; false, in the whole warp, when the wait runs out or
// another's did.  (A vote; with lane 0's reading handed round, as in wait_given_up, a step took 1%
// longer here.)
template <class C>
__device__ __forceinline__ bool res_poll_again(const StepParams<C> &p, int spin_limit, int it)
{
    if (it >= spin_limit ||
        (it > 64 && __any_sync(0xffffffffu, *static_cast<const volatile int *>(p.status) & STATUS_TIMEOUT)))
        return false;
    if (it > 32)
        __nanosleep(it < 256 ? 32 : 1024);
    return true;
}

// Receives the ring of state number seq: warps take pieces of the inbox until
// none is left (one that fills ghosts comes late and finds less to do), and
// every thread polls its entries of a piece and puts each value where the
// tile's table says.  (One unrolled loop per kind of ring row and column
// instead of the table cost the kernel 80 registers; pieces of 8 entries a
// thread took 7.8 us a step on the 1024 x 256 FP32 jet, of 4 7.4, of 2 7.6.)
template <class C, int NV, int TH>
__device__ __noinline__ bool res_receive(const StepParams<C> &p, const int spin_limit, const unsigned long long *box,
                                         unsigned seq)
{
    using Mem = ResMem<C, NV, TH>;
    constexpr int B = 4;
    const Mem t;
    const int lane = threadIdx.x & 31;
    C *cells = reinterpret_cast<C *>(t.raw);
    for (;;) {
        int e0 = 0;
        if (lane == 0)
            e0 = atomicAdd(&t.taken(), 32 * B);
        e0 = __shfl_sync(0xffffffffu, e0, 0);
        if (e0 >= Mem::ENTRIES)
            return true;
        e0 += lane;
        int off[B];
        C v[B];
#pragma unroll
        for (int n = 0; n < B; ++n) {
            const int e = e0 + 32 * n;
            off[n] = e < Mem::ENTRIES ? t.recv()[e] : RES_NONE;
        }
        // (only what has not come yet is read again: polls compete with the values on their way)
        bool got[B];
#pragma unroll
        for (int n = 0; n < B; ++n)
            got[n] = off[n] == RES_NONE;
#pragma unroll 1
        for (int it = 0;; ++it) {
            bool all = true;
#pragma unroll
            for (int n = 0; n < B; ++n) {
                if (!got[n]) {
                    got[n] = true;
                    v[n] = box_get<C>(box + (e0 + 32 * n) * Mem::WPV, seq, got[n]);
                }
            }
#pragma unroll
            for (int n = 0; n < B; ++n)
                all = all && got[n];
            if (__all_sync(0xffffffffu, all))
                break;
            if (!res_poll_again<C>(p, spin_limit, it))
                return false;
        }
#pragma unroll
        for (int n = 0; n < B; ++n)
            if (off[n] != RES_NONE)
                cells[off[n]] = v[n];
    }
}

// sends the corner entries tagged `who`
template <class C, int NV, int TH>
__device__ __forceinline__ void res_send_corners(unsigned long long *half, const ResMem<C, NV, TH> &t, int who, unsigned seq)
{
    __syncwarp();  // the values were written by this warp's lanes
    const int n = min(t.nsend(), RES_SEND_MAX);
    for (int e = threadIdx.x & 31; e < n; e += 32) {
        const int2 x = t.send()[e];
        if (x.x >> 20 == who)
            box_put<C>(half + x.y, t.pop[(x.x & 0xfffff) - 1024], seq);
    }
}

// Sends what the rings of the tiles beside this one hold of the warp's rows,
// r0 .. r0 + RPW - 1.  Columns: a lane per row, side and plane; rows: the
// planes of a row at the tile's lower or upper edge, a lane per column.
template <class C, int NV, int TH, int RPW>
__device__ __noinline__ void res_send(unsigned long long *half, const ResTile a, int own, int ns, int r0, bool below,
                                      bool above, bool left, bool right, unsigned seq)
{
    using Mem = ResMem<C, NV, TH>;
    const Mem t;
    const int lane = threadIdx.x & 31;
    // entry e of tile n's inbox
    auto box = [&](int n, int e) { return half + ((int64_t)n * Mem::WORDS + e * Mem::WPV); };
    __syncwarp();  // the values were written by this warp's lanes
    {
        const int n = lane & 7, east = (lane >> 3) & 1, r = r0 + (lane >> 4);
        if (lane < 16 * RPW && r < a.h && (east ? right : left)) {
            // of column 0: f6, f7, f3, g2, f2, f4; of 1: f6, f7; of w - 1: f5, f8, f1, g0, f2, f4; of w - 2: f5, f8
            constexpr unsigned qw = 6u | 7u << 4 | 3u << 8 | 11u << 12 | 2u << 16 | 4u << 20 | 6u << 24 | 7u << 28,
                               qe = 5u | 8u << 4 | 1u << 8 | 9u << 12 | 2u << 16 | 4u << 20 | 5u << 24 | 8u << 28;
            const int q = (int)((east ? qe : qw) >> (4 * n) & 15u);
            const int c = east ? a.w - 1 - (n >= 6) : (n >= 6);
            box_put<C>(box(own + (east ? 1 : -1), Mem::COLS + ((east ? 0 : 8) + n) * TH + r), t.P(q, r, c), seq);
        }
    }
#pragma unroll 1
    for (int r = r0; r < min(r0 + RPW, a.h); ++r) {
        const bool down = below && r <= 1, up = above && r >= a.h - 2;
        const bool flat_down = below && r == 0, flat_up = above && r == a.h - 1;
        if (!down && !up)
            continue;
#pragma unroll
        for (int c = 0; c < NV; ++c) {
            const int col = lane + 32 * c;
            if (col >= a.w)
                continue;
            const C *o = &t.P(0, r, col);
            auto put = [&](unsigned long long *b, int e, int q) { box_put<C>(b + e * Mem::WPV, o[q * Mem::PL], seq); };
            if (flat_down || flat_up) {
                unsigned long long *b = box(flat_down ? own - ns : own + ns, (flat_down ? 12 * Mem::W : 0) + col);
                put(b, 0, 1), put(b, Mem::W, 3), put(b, 2 * Mem::W, 9), put(b, 3 * Mem::W, 11);
            }
            if (down) {
                unsigned long long *b = box(own - ns, (r == 0 ? 16 : 20) * Mem::W + col);
                put(b, 0, 4), put(b, Mem::W, 7), put(b, 2 * Mem::W, 8), put(b, 3 * Mem::W, 12);
            }
            if (up) {
                unsigned long long *b = box(own + ns, (r == a.h - 1 ? 4 : 8) * Mem::W + col);
                put(b, 0, 2), put(b, Mem::W, 5), put(b, 2 * Mem::W, 6), put(b, 3 * Mem::W, 10);
            }
        }
    }
    res_send_corners<C, NV, TH>(half, t, r0 / RPW, seq);
}

// ---- the tile's steps -----------------------------------------------------------------------
// cell (r, c) of the tile from a stored state
template <class S, class C, int NV, int TH>
__device__ __forceinline__ void res_load_cell(const StepParams<C> &p, const S *src, const ResMem<C, NV, TH> &t, int i,
                                              int j, int r, int c)
{
    const int64_t o = cell(p, 0, i, j);
    float2 jj = make_float2(0.f, 0.f);
    float T = 0.f;
    if constexpr (IsSplit<S>::value) {
        const float *M = split_m(src, p.plane);
        jj = __ldcg(reinterpret_cast<const float2 *>(M) + o);
        T = __ldcg(M + 2 * p.plane + o);
    }
    C v[13];
#pragma unroll
    for (int q = 0; q < 13; ++q)
        v[q] = load_as<S, C>(src + o + q * p.plane);
#pragma unroll
    for (int q = 0; q < 13; ++q) {
        if constexpr (IsSplit<S>::value)
            v[q] = split_add<C>(p, q, jj.x, jj.y, T, v[q]);
        t.P(q, r, c) = v[q];
    }
}

// stores population q of a node with moments (jx, jr, dT): returns the value as a pull decodes it
template <class S, class C>
__device__ __forceinline__ C res_round(const StepParams<C> &p, int q, C v, C jx, C jr, C dT, S &s)
{
    if constexpr (IsSplit<S>::value) {
        s = store_as<S, C>(split_sub<C>(p, q, jx, jr, dT, v));
        return split_add<C>(p, q, jx, jr, dT, load_as_shared<S, C>(&s));
    } else {
        s = store_as<S, C>(v);
        return load_as_shared<S, C>(&s);
    }
}

// Moment-split storage: the thermal populations of a lattice-edge node as
// write_ghosts forms them (edge_add), whose rounding is not quite a pull's:
// kept beside the tile for res_ghosts.
template <class C, int NV, int TH>
__device__ __forceinline__ C *res_edge_g(const ResMem<C, NV, TH> &t, const StepParams<C> &p, int i, int j, int r, int c)
{
    constexpr int W = 32 * NV;
    const int n = i == 0 ? r : (i == p.nx - 1 ? TH + r : (j == 0 ? 2 * TH + c : 2 * TH + W + c));
    return reinterpret_cast<C *>(t.raw + ResMem<C, NV, TH>::BYTES) + 4 * n;
}

template <class S, class C, int NV, int TH>
__host__ __device__ constexpr int res_smem()
{
    return ResMem<C, NV, TH>::BYTES + (IsSplit<S>::value ? 4 * (2 * TH + 64 * NV) * (int)sizeof(C) : 0);
}

// Ghost cells of lattice-edge node (r, c) of the tile beyond one edge (SIDE: 0
// first column, 1 last column, 2 bottom row, 3 top row), from its populations
// in shared memory: into the tile's ring and, with OUT, into the state dst;
// the row's inlet velocity with noise, without, and temperature.  These are
// the longest chain of a step of a tile at a lattice edge, for which its
// neighbours wait: one edge and no stored state at a time leaves the least of
// it (filling all of a node's ghosts in one call cost 777 x 301 FP16
// moment-split 1.6 of 10.2 us a step, 640 x 160 2.1 of 6.4).
template <class S, class C, int NV, int TH, int SIDE, bool OUT>
__device__ __noinline__ void res_ghosts(const StepParams<C> &p, S *dst, const int x0, const int j0, int r, int c, C uin,
                                        C u0, C Tin)
{
    using Mem = ResMem<C, NV, TH>;
    const Mem t;
    const C *own = &t.P(0, r, c);
    C fo[9], go[4];
#pragma unroll
    for (int k = 0; k < 9; ++k)
        fo[k] = own[k * Mem::PL];
#pragma unroll
    for (int k = 0; k < 4; ++k)
        go[k] = own[(9 + k) * Mem::PL];
    // moment-split storage: the moments the ghost cells carry (ghost_moments), if any
    C gx = C(0), gr = C(0), gT = C(0);
    bool carried = false;
    if constexpr (IsSplit<S>::value) {
        const C *eg = res_edge_g<C, NV, TH>(t, p, x0 + c, j0 + r, r, c);
#pragma unroll
        for (int k = 0; k < 4; ++k)
            go[k] = eg[k];
        if (SIDE == 0) {
            gx = p.rho0 * u0;
            gT = Tin - p.T0;
            carried = true;
        } else {
            gx = t.M(0, r, c);
            gr = SIDE == 2 ? -t.M(1, r, c) : t.M(1, r, c);
            gT = t.M(2, r, c);
            carried = SIDE == 1 ? p.bc_out != OUT_WALL
                                : (SIDE == 2 ? p.bc_bottom == BOTTOM_AXIS : p.bc_top == TOP_OPEN);
        }
    }
    const int pl = (int)p.plane;
    auto W = [&](int q, int ci, int cj, C v) {
        S s;
        const int o = (cj + 1) * p.pitch + ci + PAD_COLS;
        // the lattice's corner cells and those beyond walls: no moments, the population whole
        if (IsSplit<S>::value && carried && (SIDE > 1 || (cj >= 0 && cj < p.nr))) {
            if constexpr (IsSplit<S>::value) {
                if constexpr (OUT) {
                    const MomRef M{split_m(dst, p.plane), p.plane};
                    M.j(o) = make_float2(gx, gr);
                    M.T(o) = gT;
                }
                // (write_ghosts' rounding: beyond the axis as in a collision's store)
                s = store_as<S, C>(SIDE == 2 ? split_sub<C>(p, q, gx, gr, gT, v) : edge_sub<C>(p, q, gx, gr, gT, v));
                v = split_add<C>(p, q, gx, gr, gT, load_as_shared<S, C>(&s));
            }
        } else {
            s = store_as<S, C>(v);
            v = load_as_shared<S, C>(&s);
        }
        t.P(q, cj - j0, ci - x0) = v;
        if constexpr (OUT)
            dst[o + q * pl] = s;
    };
    ghost_rules<C, 1 << SIDE>(p, fo, go, x0 + c, j0 + r, [&]() -> C { return uin; }, [&]() -> C { return Tin; }, W);
}

__device__ __forceinline__ void named_barrier(int id, bool wait)
{
    if (wait)
        asm volatile("bar.sync %0, %1;\n" ::"r"(id), "r"((int)blockDim.x) : "memory");
    else
        asm volatile("bar.arrive %0, %1;\n" ::"r"(id), "r"((int)blockDim.x) : "memory");
}

// edge task n of a tile: one lane per node
template <class S, class C, int NV, int TH, bool OUT>
__device__ __forceinline__ void res_edge_task(const StepParams<C> &p, S *dst, const ResTile &a, int n, C uin, C u0,
                                              C Tin)
{
    const int lane = threadIdx.x & 31, c = lane + 32 * (n & 1);
    if (n == 0) {
        if (lane < a.h)
            res_ghosts<S, C, NV, TH, 0, OUT>(p, dst, a.x0, a.j0, lane, 0, uin, u0, Tin);
    } else if (n == 1) {
        if (lane < a.h)
            res_ghosts<S, C, NV, TH, 1, OUT>(p, dst, a.x0, a.j0, lane, a.w - 1, C(0), C(0), C(0));
    } else if (c < a.w) {
        if (n < 4)
            res_ghosts<S, C, NV, TH, 2, OUT>(p, dst, a.x0, a.j0, 0, c, C(0), C(0), C(0));
        else
            res_ghosts<S, C, NV, TH, 3, OUT>(p, dst, a.x0, a.j0, a.h - 1, c, C(0), C(0), C(0));
    }
}

// All steps of one tile.  RPW: rows per warp.  Returns false when a wait ran out.
template <class S, class C, int NV, int TH, int RPW>
__device__ __forceinline__ bool res_tile(const StepParams<C> &p, const ResCtl &ctl, const ResTile &a)
{
    // (one FP32 node a lane by the instructions of two, so that every tile shape gives the same bits)
    using V = Vec<C, NV == 1 && std::is_same<C, float>::value ? -1 : NV>;
    using Mem = ResMem<C, NV, TH>;
    const Mem t;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
    const bool below = a.j0 > 0, above = a.j0 + a.h < p.nr, left = a.x0 > 0, right = a.x0 + a.w < p.nx;
    const bool alone = ctl.ns * ctl.nb == 1;
    const float2 *stab = nullptr;
    if (threadIdx.x == 0)
        t.nsend() = t.taken() = 0;
    if constexpr (std::is_same<C, float>::value) {
        if (p.ntab > 1 && p.ntab <= SMEM_TAB) {
            load_smem_table(p, t.tab());
            stab = t.tab();
        }
    }
    __syncthreads();
    if (!alone)
        res_lists<C, NV, TH, RPW>(p, ctl.ns, ctl.nb, a);
    {  // the tile and its ring, whole
        const S *src = static_cast<const S *>(p.src);
        for (int e = threadIdx.x; e < (a.h + 4) * Mem::PW; e += blockDim.x) {
            const int r = e / Mem::PW - 2, c = e % Mem::PW - 2;
            const int i = a.x0 + c, j = a.j0 + r;
            if (c < a.w + 2 && i >= -1 && i <= p.nx && j >= -1 && j <= p.nr)
                res_load_cell<S, C, NV, TH>(p, src, t, i, j, r, c);
        }
    }
    // inboxes: this tile's, and those of the tiles beside it
    const int64_t words = (int64_t)Mem::WORDS, half_words = words * ctl.ns * ctl.nb;
    const int own = a.tb * ctl.ns + a.ts;
    // the inlet's values for lane = row (warp 0)
    C u0 = C(0), Tin = C(0);
    if (warp == 0 && !left && lane < a.h) {
        u0 = p.u_in[a.j0 + lane];
        Tin = p.T_in[a.j0 + lane];
    }

    for (int k = ctl.first; k < ctl.nsteps; ++k) {
        const bool last = k + 2 >= ctl.nsteps;  // this state goes to memory
        S *dst = static_cast<S *>((k & 1) ? const_cast<void *>(p.src) : p.dst);
        const unsigned seq = ctl.base + (unsigned)k;  // of the state this step pulls; it sends seq + 1
        C uin = C(0);
        if (warp == 0 && !left)
            uin = noisy_velocity<C>(p, u0, a.j0 + lane, p.step + k + 1);
        bool ok = true;
        if (k > 0 && !alone)
            ok = res_receive<C, NV, TH>(p, ctl.spin_limit, ctl.box + (seq & 1u) * half_words + own * words, seq);
        if (__syncthreads_or(!ok))
            return false;
        if (threadIdx.x == 0)
            t.taken() = 0;  // (read again only after the next barrier)

        // phase 1: pull, moments
        V f[RPW][9], g[RPW][4];
        Mom<V> m[RPW];
        auto pull_row = [&](int r, V (&pf)[9], V (&pg)[4]) {
            const C *o = &t.P(0, r, lane);
#pragma unroll
            for (int c = 0; c < NV; ++c) {
#pragma unroll
                for (int q = 0; q < 9; ++q)
                    pf[q].set(c, o[q * Mem::PL - ey9(q) * Mem::PW - ex9(q) + 32 * c]);
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    pg[q].set(c, o[(9 + q) * Mem::PL - ey4(q) * Mem::PW - ex4(q) + 32 * c]);
            }
        };
        auto put_moments = [&](int r, const Mom<V> &mm) {
#pragma unroll
            for (int c = 0; c < NV; ++c)
                if (lane + 32 * c < a.w) {
                    t.M(0, r, lane + 32 * c) = mm.jx[c];
                    t.M(1, r, lane + 32 * c) = mm.jr[c];
                    t.M(2, r, lane + 32 * c) = mm.dT[c];
                }
        };
#pragma unroll
        for (int u = 0; u < RPW; ++u) {
            const int r = warp * RPW + u;
            if (r < a.h) {
                pull_row(r, f[u], g[u]);
                m[u] = moments<V>(f[u], g[u]);
                put_moments(r, m[u]);
            }
        }
        // the ring: its rows and (rho u_r) columns beside the tile
        for (int n = warp; n < 3; n += warps) {
            if (n < 2) {
                if (n ? above : below) {
                    V rf[9], rg[4];
                    const int r = n ? a.h : -1;
                    pull_row(r, rf, rg);
                    put_moments(r, moments<V>(rf, rg));
                }
            } else {
                for (int e = lane; e < 2 * a.h; e += 32) {
                    const int r = e >> 1, c = e & 1 ? a.w : -1;
                    if (e & 1 ? right : left)  // as in moments()
                        t.M(1, r, c) = (t.P(2, r - 1, c) - t.P(4, r + 1, c)) +
                                       (t.P(5, r - 1, c - 1) - t.P(8, r + 1, c - 1)) +
                                       (t.P(6, r - 1, c + 1) - t.P(7, r + 1, c + 1));
                }
            }
        }
        __syncthreads();

        // phase 2: collide, write back, send
        unsigned long long *half = ctl.box + ((seq + 1) & 1u) * half_words;
        const bool send = !alone && k + 1 < ctl.nsteps;
#pragma unroll 1
        for (int u = 0; u < RPW; ++u) {
            const int r = warp * RPW + u, j = a.j0 + r;
            if (r >= a.h)
                break;
            auto get_moments = [&](int rr) {
                Mom<V> mm;
                mm.drho = V(C(0));
#pragma unroll
                for (int c = 0; c < NV; ++c) {
                    mm.jx.set(c, t.M(0, rr, lane + 32 * c));
                    mm.jr.set(c, t.M(1, rr, lane + 32 * c));
                    mm.dT.set(c, t.M(2, rr, lane + 32 * c));
                }
                return mm;
            };
            const Mom<V> &mc = m[0];
            const Mom<V> mp = j == 0 ? ghost_bottom<C, V>(p, mc) : get_moments(r - 1);
            const Mom<V> mn = j == p.nr - 1 ? ghost_top<C, V>(p, mc) : get_moments(r + 1);
            V jl, jrr;
#pragma unroll
            for (int c = 0; c < NV; ++c) {
                const int col = lane + 32 * c;
                C l = t.M(1, r, col - 1), rr = t.M(1, r, col + 1);
                if (a.x0 + col == 0)
                    l = C(0);  // the imposed inflow has no radial component
                if (a.x0 + col == p.nx - 1)
                    rr = p.bc_out == OUT_OUTFLOW ? mc.jr[c] : -mc.jr[c];
                jl.set(c, l);
                jrr.set(c, rr);
            }
            V fo[9], go[4];
            const C inv_r = C(1) / (p.r0 + C(j) + C(0.5));
            collide<C, V>(p, f[0], g[0], mc, inv_r, C(0.5) * (mn.jx - mp.jx), C(0.5) * (mn.jr - mp.jr),
                          C(0.5) * (jrr - jl), C(0.5) * (mn.dT - mp.dT), fo, go, stab);
            const unsigned pl = (unsigned)p.plane;
#pragma unroll
            for (int c = 0; c < NV; ++c) {
                const int col = lane + 32 * c;
                const C jx = mc.jx[c], jr = mc.jr[c], dT = mc.dT[c];
                S s[13];
                C v[13];
#pragma unroll
                for (int q = 0; q < 13; ++q)
                    v[q] = res_round<S, C>(p, q, q < 9 ? fo[q < 9 ? q : 0][c] : go[q < 9 ? 0 : q - 9][c], jx, jr, dT,
                                           s[q]);
                if (col >= a.w)
                    continue;
#pragma unroll
                for (int q = 0; q < 13; ++q)
                    t.P(q, r, col) = v[q];
                if constexpr (IsSplit<S>::value) {
                    const int i = a.x0 + col;
                    if ((c == 0 && !left && col == 0) || (!right && col == a.w - 1) || j == 0 || j == p.nr - 1) {
                        C *eg = res_edge_g<C, NV, TH>(t, p, i, j, r, col);
#pragma unroll
                        for (int q = 0; q < 4; ++q)
                            eg[q] = edge_add<C>(p, 9 + q, jx, jr, dT, load_as_shared<S, C>(&s[9 + q]));
                    }
                }
                if (last) {
                    const unsigned o = (unsigned)((j + 1) * p.pitch + a.x0 + col + PAD_COLS);
                    if constexpr (IsSplit<S>::value) {
                        const MomRef M{split_m(dst, p.plane), p.plane};
                        M.j(o) = make_float2(jx, jr);
                        M.T(o) = dT;
                    }
#pragma unroll
                    for (int q = 0; q < 13; ++q)
                        dst[o + q * pl] = s[q];
                }
            }
            if constexpr (RPW == 2) {  // the next row, in the same registers
                if (u == 0) {
#pragma unroll
                    for (int q = 0; q < 9; ++q)
                        f[0][q] = f[1][q];
#pragma unroll
                    for (int q = 0; q < 4; ++q)
                        g[0][q] = g[1][q];
                    m[0] = m[1];
                }
            }
        }
        if (send)
            res_send<C, NV, TH, RPW>(half, a, own, ctl.ns, warp * RPW, below, above, left, right, seq + 1);
        if (!left || !right || !below || !above) {
            // the lattice's edge nodes fill the ghosts, a warp per task; the others do not wait
            auto task = [&](int n) {
                return n == 0 ? !left : (n == 1 ? !right : (n < 4 ? !below : !above) && 32 * (n & 1) < a.w);
            };
            bool mine = false;
            for (int n = warp; n < RES_EDGES; n += warps)
                mine = mine || task(n);
            named_barrier(1, mine);
            for (int n = warp; n < RES_EDGES; n += warps) {
                if (!task(n))
                    continue;
                if (last)
                    res_edge_task<S, C, NV, TH, true>(p, dst, a, n, uin, u0, Tin);
                else
                    res_edge_task<S, C, NV, TH, false>(p, dst, a, n, uin, u0, Tin);
                if (send)
                    res_send_corners<C, NV, TH>(half, t, 64 + n, seq + 1);
            }
        }
    }
    return true;
}

template <class S, class C, int NV, int TH, int RPW>
__global__ void __launch_bounds__(32 * TH / RPW, RPW == 2 ? 2 : 1)
    res_run_kernel(const __grid_constant__ StepParams<C> p, const ResCtl ctl)
{
    const ResTile a(p.nx, p.nr, ctl.ns, ctl.nb, (int)blockIdx.x);
    if (!res_tile<S, C, NV, TH, RPW>(p, ctl, a) && threadIdx.x == 0)
        atomicOr(p.status, STATUS_TIMEOUT);
}

}  // namespace lbm
