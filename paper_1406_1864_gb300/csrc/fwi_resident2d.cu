// fwi_resident2d.cu -- the 2-D time loops with the wavefields resident on the
// chip (sm_103a).
//
// The streaming steps (fwi_step2d.cu) read and write every wavefield once per
// time level: at 300 x 1000 cells and 96 shots they run at 0.8 to 0.97 of the
// HBM copy rate, and a small model (4 shots of 100 x 200) spends its level on
// launch, descriptor and copy latencies. Neither is needed: a level of one
// shot is 1.4 MB, the chip's 152 SMs hold 33 MB of shared memory, and a level
// depends on its neighbours through a 4-cell halo only. Here one cooperative
// launch runs a whole time loop. A shot's padded grid is cut into tiles, one
// CTA each; the CTA keeps its tile (and halo) of S shots in shared memory for
// all levels and goes on to the next S shots (the next round) when they are done.
// Per level and shot only the tile's outer 4 rows and columns are exchanged, as
// packets through L2, and the sponge checkpoint, the traces and the adjoint
// source touch HBM.
//
// Exchange. After a level's compute warps have arrived on the shot's `done`
// barrier, the export warp sends the tile's outer 4 rows and columns to global
// memory as 8-byte packets {value, level}; the import warps of the neighbouring
// tiles read those packets until they carry the level they wait for, store the
// halo in shared memory and arrive on the shot's `full` barrier, which the
// compute warps wait on. A packet is one access, so neither side needs a fence
// or a flag: a first version with flags (fence, flag, poll, fence, copy) took
// about 4 us per exchange. While one shot's halo travels, the compute warps
// advance the other S - 1 shots.
//
// Packets alternate between two buffers. A tile makes its exchanges in one
// order, k = 1, 2, ... over all rounds, and sends the k-th once it has the
// (k - 1)-th of its neighbours: within a round because level v is computed from
// their level v - 1, after a round's end because the round ended with their
// last one. The neighbours in turn sent their (k - 1)-th after they had read this
// tile's (k - 2)-th. So the buffer of exchange k - 2 is free, and k & 1 picks the
// buffer. The level's own parity would not do: a round has nt - 2 exchanges,
// and with nt odd the next round's level 1, which a tile computes from no packet
// at all, would land on the last level's packets while a neighbour held up
// elsewhere may still have to read them.
//
// Phases. full[s] of a level completes when the halo has arrived (32 lanes of
// an import warp), the data warp has the level's amplitudes and adjoint source
// in place and has read the last level's traces (32 lanes), and the export warp
// has seen the level's cells complete and has read the last level's (32). done[s]
// completes when every compute warp has written the next level. So full(v)
// implies done(v - 1), and neither barrier can get a phase ahead of a warp
// that tests it. Every warp takes the shots in the same order.
//
// Arithmetic. The updates are the streaming steps' own (lap4, lane pairs), so
// wavefields, checkpoints and traces are bitwise the same; only the order in
// which shots and levels are summed differs (illumination and imaging sums
// stay in registers over the S shots and up to RES_SUM levels). Cells of a tile outside
// the padded grid have c2 = 0 and stay zero.
//
// Bound and measured. Per 128 points of a row the forward update is 112 cycles of
// a scheduler's FP32 pipe and, with R rows per thread, (R + 8) / R + 4 16-byte
// shared-memory accesses per thread (4 cycles each). Small shots are bound by the
// way of the halo (about 2 us: packets out through L2 and in), large ones by the
// latency of a warp's rows at 10 to 12 warps per SM, and passes with a checkpoint
// also by the data warp that writes it. us per level, streaming steps (default
// tiles) / resident, of plain forward passes, forward passes with checkpoint and
// illumination, and backward passes; * where the resident loop is not taken
// (choose_resident decides per problem and pass):
//   37 x 83, 3 shots       5.8 / 2.4    6.1 / 2.4    7.7 / 3.3
//   100 x 200, 4 shots     6.1 / 2.4    6.4 / 2.6    8.8 / 3.5
//   100 x 200, 64 shots   13.5 / 6.3   14.5 / 8.7   22.2 / 18.1
//   150 x 460, 24 shots   12.7 / 5.9   14.0 / 10.0  23.9 / 24.1 *
//   150 x 460, 80 shots   27.8 / 20.0  32.8 / 31.0  49.6 / 80.2 *
//   300 x 1000, 1 shot     4.4 / 3.6    4.7 / 3.8    4.8 / 6.0 *
//   300 x 1000, 12 shots  17.4 / 12.1  18.9 / 15.9  27.5 / 44.4 *
//   300 x 1000, 48 shots  51.1 / 50.5  58.6 / 70.1 * 83 / 176 *
//   400 x 1200, 32 shots  49.9 / 56.4 * 55.5 / 80.7 * 81 / 145 *
// Every wait is bounded (2 s of %globaltimer), after which the CTA sets ST_TIMEOUT
// and leaves.
#include "fwi_device.cuh"
#include "fwi_resident.h"

#include <algorithm>
#include <array>
#include <cmath>
#include <mutex>
#include <set>

namespace fwi {
namespace {

// A field tile in shared memory: rows of RES_P floats (up to RES_W float4
// columns and the halo on each side); the damping factors: rows of RES_KP. Fixed
// pitches make every stencil access an immediate offset from one address.
constexpr int RES_W = 32, RES_P = 4 * RES_W + 2 * RADIUS, RES_KP = 4 * RES_W;

__device__ __forceinline__ void mbar_arrive(uint32_t bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

// bounded wait that also ends when another thread of the CTA has given up
__device__ __forceinline__ bool res_wait(uint32_t bar, uint32_t parity, volatile int *s_abort)
{
    if (mbar_try_wait(bar, parity)) return true;
    const uint64_t t0 = globaltimer_ns();
    for (uint32_t it = 0; it < (1u << 30); ++it) {
        if (mbar_try_wait(bar, parity)) return true;
        if ((it & 63u) == 63u && (*s_abort != 0 || globaltimer_ns() - t0 > WAIT_NS)) break;
    }
    *s_abort = 1;
    return false;
}

__device__ __forceinline__ void copy4(float *dst, const float *src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}

__device__ __forceinline__ void copy16(float *dst, const float *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}

__device__ __forceinline__ void copies_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }

// all committed copies of this thread but those of the last n groups (at
// least: n above 3 is taken as 3)
__device__ __forceinline__ void copies_wait_but(int n)
{
    if (n <= 0)
        asm volatile("cp.async.wait_group 0;" ::: "memory");
    else if (n == 1)
        asm volatile("cp.async.wait_group 1;" ::: "memory");
    else if (n == 2)
        asm volatile("cp.async.wait_group 2;" ::: "memory");
    else
        asm volatile("cp.async.wait_group 3;" ::: "memory");
}

__device__ __forceinline__ void copies_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// limit of a polling loop: true when the CTA has given up, or this loop has
// spun for WAIT_NS (which makes the CTA give up)
struct Patience {
    uint64_t t0 = 0;
    uint32_t it = 0;
    __device__ bool over(volatile int *abort)
    {
        if ((++it & 255u) != 0) return false;
        if (*abort != 0) return true;
        const uint64_t now = globaltimer_ns();
        if (t0 == 0) t0 = now;
        if (now - t0 <= WAIT_NS) return false;
        *abort = 1;
        return true;
    }
};

// two packets {value, level} of the exchange, each one 8-byte access
__device__ __forceinline__ void ld_packets(const uint2 *p, uint64_t &a, uint64_t &b)
{
    asm volatile("ld.relaxed.gpu.global.v2.b64 {%0, %1}, [%2];" : "=l"(a), "=l"(b) : "l"(p) : "memory");
}

__device__ __forceinline__ void st_packets(uint2 *p, float a, float b, uint32_t tag)
{
    const uint64_t x = (uint64_t)tag << 32 | __float_as_uint(a), y = (uint64_t)tag << 32 | __float_as_uint(b);
    asm volatile("st.relaxed.gpu.global.v2.b64 [%0], {%1, %2};" ::"l"(p), "l"(x), "l"(y) : "memory");
}

// The thread's points and where they sit: rows i0 .. i0 + R - 1, columns
// j0 .. j0 + 3 of the padded grid.
template <int R>
struct Own {
    bool on;           // the thread has points of the tile
    int i0, j0;        // first row and column
    int so;            // offset of the first point in a shared-memory field tile
    int ko;            // and in a tile without halo
    unsigned in;       // rows with points in the padded grid
    unsigned bmask;    // sponge points: 4 bits per row
};

// this CTA's tile
struct Cta {
    int set, tile, bz, bx, r0, c0;
};

__device__ __forceinline__ Cta cta_of(const ResTile &t)
{
    Cta c;
    const int nt = t.ntx * t.ntz;
    c.set = blockIdx.x / nt;
    c.tile = blockIdx.x - c.set * nt;
    c.bz = c.tile / t.ntx;
    c.bx = c.tile - c.bz * t.ntx;
    c.r0 = c.bz * t.th;
    c.c0 = c.bx * t.w4;
    return c;
}

template <int R>
__device__ __forceinline__ void own_init(Own<R> &o, const Lay2D &L, const ResTile &t, const Cta &c, int thread)
{
    const int col = thread % t.w4, grp = thread / t.w4;
    o.on = grp < t.g;
    o.i0 = c.r0 + grp * R;
    o.j0 = 4 * (c.c0 + col);
    o.so = (grp * R + RADIUS) * RES_P + RADIUS + 4 * col;
    o.ko = grp * R * RES_KP + 4 * col;
    o.in = o.bmask = 0;
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int i = o.i0 + r;
        const bool in = o.on && i < L.nzp && o.j0 < L.nxp;
        if (in) o.in |= 1u << r;
        unsigned mask = 0;
        if (in) {
#pragma unroll
            for (int p = 0; p < 4; ++p)
                if (o.j0 + p < L.nxp && band_index(L, i, o.j0 + p) >= 0) mask |= 1u << p;
        }
        o.bmask |= mask << (4 * r);
    }
}

// Exchange tables of a tile, one entry per float4 of its edge strips in the
// order top (4 rows of w4), bottom, left (th rows), right: where the float4
// is in a shared-memory field tile, and where the halo it mirrors comes from:
// element `src` of the neighbours' packets (4 each) goes to `dst`; src < 0
// where there is no neighbour.
struct Xch {
    int own, src, dst;
};

__device__ __forceinline__ void xch_init(Xch *x, const ResTile &t, const Cta &c)
{
    const int ne = t.ne, w4 = t.w4, th = t.th, p = RES_P;
    for (int e = threadIdx.x; e < ne; e += blockDim.x) {
        Xch v;
        if (e < 8 * w4) { // rows: the tile above mirrors at its bottom strip and conversely
            const bool top = e < 4 * w4;
            const int k = (top ? e : e - 4 * w4) / w4, cc = e - (top ? 0 : 4 * w4) - k * w4, row = top ? k : th - RADIUS + k;
            v.own = (row + RADIUS) * p + RADIUS + 4 * cc;
            v.dst = ((top ? k - RADIUS : th + k) + RADIUS) * p + RADIUS + 4 * cc;
            const int nb = top ? (c.bz > 0 ? c.tile - t.ntx : -1) : (c.bz < t.ntz - 1 ? c.tile + t.ntx : -1);
            v.src = nb < 0 ? -1 : nb * ne + (top ? 4 * w4 : 0) + k * w4 + cc;
        } else {
            const int q = e - 8 * w4;
            const bool left = q < th;
            const int rr = left ? q : q - th;
            v.own = (rr + RADIUS) * p + RADIUS + (left ? 0 : 4 * (w4 - 1));
            v.dst = (rr + RADIUS) * p + (left ? 0 : RADIUS + 4 * w4);
            const int nb = left ? (c.bx > 0 ? c.tile - 1 : -1) : (c.bx < t.ntx - 1 ? c.tile + 1 : -1);
            v.src = nb < 0 ? -1 : nb * ne + 8 * w4 + (left ? th : 0) + rr;
        }
        x[e] = v;
    }
}

// The tile's sponge cells, one entry per float4 of a field tile that holds any:
// x: offset in the tile, a bit per sponge cell (<< 24) and whether all four are
// 16 aligned bytes of the checkpoint (bit 28); y: checkpoint index of the
// float4's first column.
__device__ __forceinline__ void band_init(int2 *list, int *count, const Lay2D &L, const ResTile &t, const Cta &c)
{
    for (int e = threadIdx.x; e < t.th * t.w4; e += blockDim.x) {
        const int rr = e / t.w4, cc = e - rr * t.w4, i = c.r0 + rr, j = 4 * (c.c0 + cc);
        unsigned mask = 0;
        int base = 0;
        for (int p = 3; p >= 0; --p)
            if (i < L.nzp && j + p < L.nxp && band_index(L, i, j + p) >= 0) {
                mask |= 1u << p;
                base = band_index(L, i, j + p) - p;
            }
        if (mask == 0) continue;
        const unsigned vec = mask == 15u && (base & 3) == 0;
        list[atomicAdd(count, 1)] = make_int2((int)(((rr + RADIUS) * RES_P + RADIUS + 4 * cc) | mask << 24 | vec << 28), base);
    }
}
constexpr int BAND_OFF = 0xffffff;

// What row r of the thread's points reads besides the column window: the 4
// values left and right of it, and its point in the buffer that the new level
// replaces. Rows are loaded one ahead: a load that follows the previous row's
// store in program order would wait for it (the two buffers never overlap, but
// the compiler cannot know).
struct RowIn {
    float4 a0, a2, prev;
    __device__ __forceinline__ void load(const float *f, const float *g)
    {
        a0 = lds4(f - 4);
        a2 = lds4(f + 4);
        prev = lds4(g);
    }
};

// q = Lhat of row r from its RowIn and the column window zc of rows r - 4 ..
// r + 4; ctr: the row's own values
template <int NZ>
__device__ __forceinline__ void row_lap(float2 (&q)[2], float2 (&ctr)[2], const RowIn &x, const float4 (&zc)[NZ], int r)
{
    const float4 a1 = zc[r + RADIUS];
    const float w[12] = {x.a0.x, x.a0.y, x.a0.z, x.a0.w, a1.x, a1.y, a1.z, a1.w, x.a2.x, x.a2.y, x.a2.z, x.a2.w};
    lap4<4, NZ, true>(q, w, zc, r);
    ctr[0] = lo2(a1);
    ctr[1] = hi2(a1);
}

// One point, with the operations and roundings of the lane pairs: Lhat at f in
// a field tile.
__device__ __forceinline__ float point_lap(const float *f)
{
    const float c = f[0];
    float q = 0.f;
    const float w[4] = {W1, W2, W3, W4};
#pragma unroll
    for (int k = 4; k >= 1; --k) {
        const float d = __fadd_rn(__fmaf_rn(c, -2.f, __fadd_rn(f[-k], f[k])),
                                  __fmaf_rn(c, -2.f, __fadd_rn(f[-k * RES_P], f[k * RES_P])));
        q = k == 4 ? __fmul_rn(w[3], d) : __fmaf_rn(w[k - 1], d, q);
    }
    return q;
}

// element (row, col) of a register array of the thread's points
template <int R>
__device__ __forceinline__ float pick(const float4 (&v)[R], int row, int col)
{
    float x = 0.f;
#pragma unroll
    for (int r = 0; r < R; ++r)
        if (row == r) x = comp(v[r], col);
    return x;
}

// v[row][col] = x
template <int R>
__device__ __forceinline__ void put(float2 (&v)[R][2], int row, int col, float x)
{
#pragma unroll
    for (int r = 0; r < R; ++r) {
        if (row != r) continue;
        if (col == 0) v[r][0].x = x;
        if (col == 1) v[r][0].y = x;
        if (col == 2) v[r][1].x = x;
        if (col == 3) v[r][1].y = x;
    }
}

template <int R>
__device__ __forceinline__ float get(const float2 (&v)[R][2], int row, int col)
{
    float x = 0.f;
#pragma unroll
    for (int r = 0; r < R; ++r)
        if (row == r) x = col == 0 ? v[r][0].x : (col == 1 ? v[r][0].y : (col == 2 ? v[r][1].x : v[r][1].y));
    return x;
}

// The update's coefficients of the thread's points: ca = c2 / (1 + eta dt) in
// registers (c2 itself where eta = 0, zero outside the padded grid), and the
// factor (1 - eta dt) / (1 + eta dt) of the tile in shared memory, which only
// threads with sponge points read. Both are products the streaming steps form
// at every level, so the updates' bits do not change.
template <int R>
__device__ __forceinline__ void coefficients(float4 (&ca)[R], float *kb, const Own<R> &o, const ResArgs &a)
{
#pragma unroll
    for (int r = 0; r < R; ++r) {
        ca[r] = make_float4(0.f, 0.f, 0.f, 0.f);
        float4 k = make_float4(1.f, 1.f, 1.f, 1.f);
        if (o.in >> r & 1) {
            const long long g = fidx(a.L, o.i0 + r, o.j0);
            const float4 c2 = __ldg(reinterpret_cast<const float4 *>(a.c2 + g));
            const float4 ia = __ldg(reinterpret_cast<const float4 *>(a.damp + g));
            const float2 lo = mul2(lo2(c2), lo2(ia)), hi = mul2(hi2(c2), hi2(ia));
            ca[r] = make_float4(lo.x, lo.y, hi.x, hi.y);
            const float2 two = make_float2(2.f, 2.f), m1 = make_float2(-1.f, -1.f);
            const float2 kl = fma2(lo2(ia), two, m1), kh = fma2(hi2(ia), two, m1);
            k = make_float4(kl.x, kl.y, kh.x, kh.y);
        }
        if (o.on) *reinterpret_cast<float4 *>(kb + r * RES_KP) = k;
    }
}

// one damped leapfrog step of a row: u + fma(ca, q, kb (u - u_prev))
template <bool SPONGE>
__device__ __forceinline__ void row_update(float2 (&out)[2], const float2 (&u)[2], const float4 &prev, const float2 (&q)[2],
                                           const float4 &ca, const float *kb)
{
    float2 t[2] = {sub2(u[0], lo2(prev)), sub2(u[1], hi2(prev))};
    if (SPONGE) {
        const float4 k = lds4(kb);
        t[0] = mul2(lo2(k), t[0]);
        t[1] = mul2(hi2(k), t[1]);
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) out[h] = add2(u[h], fma2(half2of(ca, h), q[h], t[h]));
}

__device__ __forceinline__ bool finite4(const float4 &v)
{
    return isfinite(v.x) && isfinite(v.y) && isfinite(v.z) && isfinite(v.w);
}

struct ResBars {
    uint64_t full[RES_SMAX], done[RES_SMAX];
};
constexpr int RES_IMPORT = RES_SVC - 2;   // import warps (shots in turn); one export, one data warp
constexpr int RES_FULL = 3 * 32;          // arrivals of a full phase

// static shared state of a CTA: the shots in flight
struct ResShared {
    ResBars bars;
    float amp[2][RES_SMAX]; // source amplitude, by parity of the step
    int2 src[RES_SMAX];     // source cell
    int2 rng[RES_SMAX];     // receiver-table range of (tile, shot)
    int rrow[RES_SMAX];     // backward: padded row of the receivers of (tile, shot)
    int nband;              // entries of the tile's sponge list
    int abort;
};

__device__ __forceinline__ void res_init(ResShared &sh, int nw)
{
    if (threadIdx.x == 0) {
        for (int s = 0; s < RES_SMAX; ++s) {
            mbar_init(smem_u32(&sh.bars.full[s]), RES_FULL);
            mbar_init(smem_u32(&sh.bars.done[s]), nw);
        }
        fence_mbar_init();
        sh.abort = 0;
        sh.nband = 0;
    }
}

// The service loops below are functions of their own: inlined, their hoisted
// addresses would take the compute warps' registers. Levels are counted v =
// 0 .. nlev - 1 (forward: the time level, nlev = nt; backward: v = nt - 1 - m,
// nlev = nt - 1); the first nstep of them are followed by a step. pf, pd:
// phases of full and done before this round. xb: packets of the CTA's slots,
// [slot][buffer][field][tile][ne][4]; slot0: buffer of level 0 (res_slot).

// parity of the buffer that holds level v = 0's current fields: u^0 forward,
// u^{m-1} with m = nt - 1 backward
__device__ __forceinline__ int first_parity(int nf, int nt) { return nf == 2 ? (nt & 1) : 0; }

// Export warp: the tile's edge strips of every level the neighbours need. In the
// backward pass it also copies the checkpointed sponge cells of the level being
// computed into the buffer that receives it, a level ahead: the compute warps
// neither use nor write those cells.
template <int NF>
__device__ __noinline__ void service_export(const ResArgs &a, float *sm, const Xch *xt, const int2 *bl, uint2 *xb,
                                            ResShared *sh, int tile, int b0, int shot0, int nsh, int nlev, int nstep,
                                            uint32_t pd, uint32_t tag0, int slot0)
{
    const int lane = threadIdx.x & 31, ne = a.t.ne, ntiles = a.t.ntx * a.t.ntz, fs = a.t.fs, nt = a.nt;
    const long long blk = (long long)ntiles * ne * 4;
    const int nband = sh->nband;
    // step v writes u^{m-2}, m = nt - 1 - v, to the buffer of m's parity
    auto band = [&](int v, int s) {
        const int m = nt - 1 - v;
        if (NF == 2 && m >= 2) {
            float *u = sm + (4 * s + (m & 1)) * fs;
            const float *bb = a.band + ((long long)(shot0 + s) * nt + (m - 2)) * a.L.nbandp;
#pragma unroll 2
            for (int e = lane; e < nband; e += 32) {
                const int2 x = bl[e];
                float *d = u + (x.x & BAND_OFF);
                if (m == 2) { // u^0 = 0
                    for (int p = 0; p < 4; ++p)
                        if (x.x >> (24 + p) & 1) d[p] = 0.f;
                } else if (x.x >> 28 & 1) {
                    copy16(d, bb + x.y);
                } else {
                    for (int p = 0; p < 4; ++p)
                        if (x.x >> (24 + p) & 1) copy4(d + p, bb + x.y + p);
                }
            }
        }
        copies_commit();
    };
    for (int s = 0; s < nsh; ++s) mbar_arrive(smem_u32(&sh->bars.full[s])); // level 0
    if (NF == 2)
        for (int s = 0; s < nsh; ++s) band(0, s);
    for (int v = 1; v < nlev; ++v)
        for (int s = 0; s < nsh; ++s) {
            const bool ok = res_wait(smem_u32(&sh->bars.done[s]), (pd + v - 1) & 1u, &sh->abort);
            if (NF == 2) copies_wait_but(nsh - 1);
            if (!__all_sync(0xffffffffu, ok)) {
                copies_wait();
                return;
            }
            mbar_arrive(smem_u32(&sh->bars.full[s]));
            __syncwarp(); // the other lanes' copies
            if (v < nstep && ntiles > 1) {
                const int b = (v + b0) & 1;
                const uint32_t tag = tag0 + v;
#pragma unroll
                for (int f = 0; f < NF; ++f) {
                    const float *fl = sm + (2 * NF * s + 2 * f + b) * fs;
                    uint2 *out = xb + ((s * 2 + ((slot0 + v) & 1)) * NF + f) * blk + (long long)tile * ne * 4;
#pragma unroll 2
                    for (int e = lane; e < ne; e += 32) {
                        if (xt[e].src < 0) continue;
                        const float4 x = lds4(fl + xt[e].own);
                        st_packets(out + 4 * e, x.x, x.y, tag);
                        st_packets(out + 4 * e + 2, x.z, x.w, tag);
                    }
                }
            }
            if (NF == 2) band(v, s);
        }
    copies_wait();
}

// Import warp h: the halos of shots h, h + RES_IMPORT, ...
template <int NF>
__device__ __noinline__ void service_import(float *sm, const Xch *xt, const uint2 *xb, ResShared *sh, int ne, int ntiles,
                                            int fs, int b0, int nsh, int nlev, int nstep, uint32_t pf, uint32_t tag0,
                                            int slot0, int h)
{
    const int lane = threadIdx.x & 31;
    for (int s = h; s < nsh; s += RES_IMPORT) mbar_arrive(smem_u32(&sh->bars.full[s])); // level 0: in place
    const long long blk = (long long)ntiles * ne * 4;
    for (int v = 1; v < nlev; ++v)
        for (int s = h; s < nsh; s += RES_IMPORT) {
            bool ok = res_wait(smem_u32(&sh->bars.full[s]), (pf + v - 1) & 1u, &sh->abort);
            if (!__all_sync(0xffffffffu, ok)) return;
            if (v < nstep && ntiles > 1) {
                const int b = (v + b0) & 1;
                const uint32_t tag = tag0 + v;
                Patience pt;
#pragma unroll
                for (int f = 0; f < NF; ++f) {
                    float *fl = sm + (2 * NF * s + 2 * f + b) * fs;
                    const uint2 *in = xb + ((s * 2 + ((slot0 + v) & 1)) * NF + f) * blk;
                    constexpr int B = 4; // float4s in flight per lane
                    for (int e0 = lane; e0 < ne; e0 += 32 * B) {
                        uint64_t q[B][4];
                        int src[B];
                        bool missing = false;
#pragma unroll
                        for (int k = 0; k < B; ++k) {
                            src[k] = e0 + 32 * k < ne ? xt[e0 + 32 * k].src : -1;
                            if (src[k] >= 0) {
                                ld_packets(in + 4LL * src[k], q[k][0], q[k][1]);
                                ld_packets(in + 4LL * src[k] + 2, q[k][2], q[k][3]);
                            }
                        }
                        do {
                            missing = false;
#pragma unroll
                            for (int k = 0; k < B; ++k) {
                                if (src[k] < 0) continue;
                                const bool here = (uint32_t)(q[k][0] >> 32) == tag && (uint32_t)(q[k][1] >> 32) == tag &&
                                                  (uint32_t)(q[k][2] >> 32) == tag && (uint32_t)(q[k][3] >> 32) == tag;
                                if (!here) {
                                    missing = true;
                                    ld_packets(in + 4LL * src[k], q[k][0], q[k][1]);
                                    ld_packets(in + 4LL * src[k] + 2, q[k][2], q[k][3]);
                                }
                            }
                            if (missing && pt.over(&sh->abort)) {
                                ok = false;
                                break;
                            }
                        } while (missing);
#pragma unroll
                        for (int k = 0; k < B; ++k)
                            if (src[k] >= 0)
                                *reinterpret_cast<float4 *>(fl + xt[e0 + 32 * k].dst) =
                                    make_float4(__uint_as_float((uint32_t)q[k][0]), __uint_as_float((uint32_t)q[k][1]),
                                                __uint_as_float((uint32_t)q[k][2]), __uint_as_float((uint32_t)q[k][3]));
                    }
                }
                if (!__all_sync(0xffffffffu, ok)) return;
            }
            mbar_arrive(smem_u32(&sh->bars.full[s]));
        }
}

// Data warp of the forward loop: source amplitudes a step ahead; traces and
// sponge checkpoint of the level whose cells are complete.
__device__ __noinline__ void service_traces(const ResArgs &a, const float *sm, const int2 *list, const int2 *bl,
                                            ResShared *sh, int shot0, int nsh, uint32_t pd)
{
    const int lane = threadIdx.x & 31, nt = a.nt, fs = a.t.fs, nrec = a.nrec;
    const float *wav = a.wav + (long long)shot0 * nt;
    const int nband = sh->nband;
    float *seis = a.seis == nullptr ? nullptr : a.seis + (long long)shot0 * nt * nrec;
    for (int s = 0; s < nsh; ++s)
        if (lane == 0) copy4(&sh->amp[0][s], wav + s * nt);
    copies_wait();
    for (int v = 0; v < nt; ++v) {
        for (int s = 0; s < nsh; ++s) {
            bool ok = v == 0 || res_wait(smem_u32(&sh->bars.done[s]), (pd + v - 1) & 1u, &sh->abort);
            copies_wait_but(nsh - 1);
            if (!__all_sync(0xffffffffu, ok)) {
                copies_wait();
                return;
            }
            mbar_arrive(smem_u32(&sh->bars.full[s]));
            if (lane == 0 && v + 1 < nt - 1) copy4(&sh->amp[(v + 1) & 1][s], wav + s * nt + v + 1);
            copies_commit();
            const float *cur = sm + (2 * s + (v & 1)) * fs;
            if (a.band != nullptr && v > 0) {
                float *bb = a.band + ((long long)(shot0 + s) * nt + v) * a.L.nbandp;
                constexpr int B = 4; // float4s in flight per lane
                for (int e0 = lane; e0 < nband; e0 += 32 * B) {
                    int2 x[B];
                    float4 u[B];
#pragma unroll
                    for (int k = 0; k < B; ++k) x[k] = e0 + 32 * k < nband ? bl[e0 + 32 * k] : make_int2(0, 0);
#pragma unroll
                    for (int k = 0; k < B; ++k) u[k] = lds4(cur + (x[k].x & BAND_OFF));
#pragma unroll
                    for (int k = 0; k < B; ++k) {
                        float *b = bb + x[k].y;
                        if (x[k].x >> 28 & 1) {
                            __stcs(reinterpret_cast<float4 *>(b), u[k]);
                        } else {
                            if (x[k].x >> 24 & 1) b[0] = u[k].x;
                            if (x[k].x >> 25 & 1) b[1] = u[k].y;
                            if (x[k].x >> 26 & 1) b[2] = u[k].z;
                            if (x[k].x >> 27 & 1) b[3] = u[k].w;
                        }
                    }
                }
            }
            if (seis == nullptr) continue;
            const int2 *ls = list + s * RES_MAXE;
            float *out = seis + ((long long)s * nt + v) * nrec;
            const int n = sh->rng[s].y - sh->rng[s].x;
#pragma unroll 4
            for (int e = lane; e < n; e += 32) {
                const int2 en = ls[e];
                out[en.y] = cur[en.x];
            }
        }
    }
    copies_wait();
}

// One step of a shot at the thread's points: f: u^n, g: u^{n-1}, replaced by
// u^{n+1}. MODE 0: the warp has no sponge points, 1: it may. ACC 1: acc +=
// (u^n)^2, 2: += the squared second difference. (The source is added to its one
// point outside the row loop, see fwd_loop: tests in every row would cost all
// warps that ever hold a source.)
template <int R, int MODE, int ACC>
__device__ __forceinline__ void fwd_rows(const float *f, float *g, const float4 (&ca)[R], const float *kb,
                                         float2 (&acc)[R][2])
{
    float4 zc[R + 2 * RADIUS];
#pragma unroll
    for (int k = 0; k <= 2 * RADIUS; ++k) zc[k] = lds4(f + (k - RADIUS) * RES_P);
    RowIn now, nextr;
    now.load(f, g);
#pragma unroll
    for (int r = 0; r < R; ++r) {
        if (r + 1 < R) {
            zc[r + 1 + 2 * RADIUS] = lds4(f + (r + 1 + RADIUS) * RES_P);
            nextr.load(f + (r + 1) * RES_P, g + (r + 1) * RES_P);
        }
        float2 q[2], u0[2], out[2];
        row_lap(q, u0, now, zc, r);
        row_update<MODE != 0>(out, u0, now.prev, q, ca[r], kb + r * RES_KP);
        *reinterpret_cast<float4 *>(g + r * RES_P) = make_float4(out[0].x, out[0].y, out[1].x, out[1].y);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            if (ACC == 1) acc[r][h] = fma2(u0[h], u0[h], acc[r][h]);
            if (ACC == 2) {
                const float2 d2 = add2(fma2(u0[h], make_float2(-2.f, -2.f), out[h]), half2of(now.prev, h));
                acc[r][h] = fma2(d2, d2, acc[r][h]);
            }
        }
        now = nextr;
    }
}

// Sums of u^2 and of the imaging factor are taken in registers over RES_SUM
// levels of the shots in flight and then added to memory: sums over a whole
// pass (2000 terms at 2 shots and nt 1000) rounded to 1.5e-6, streaming 1e-6.
constexpr int RES_SUM = 32;

template <int R>
__device__ __forceinline__ void flush_illum(const ResArgs &a, const Own<R> &o, float2 (&acc)[R][2], int group)
{
    const Lay2D &L = a.L;
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int iz = o.i0 + r - L.P, ix0 = o.j0 - L.P;
        if (o.on && iz >= 0 && iz < L.nz) {
            float *p = a.acc_illum + ((long long)group * L.nz + iz) * L.nx + ix0;
            if (((L.P | L.nx) & 3) == 0) { // (planes of nz nx floats keep the alignment)
                if (ix0 >= 0 && ix0 + 3 < L.nx) red_add4(p, acc[r][0].x, acc[r][0].y, acc[r][1].x, acc[r][1].y);
            } else {
                if (ix0 >= 0 && ix0 < L.nx) atomicAdd(p, acc[r][0].x);
                if (ix0 + 1 >= 0 && ix0 + 1 < L.nx) atomicAdd(p + 1, acc[r][0].y);
                if (ix0 + 2 >= 0 && ix0 + 2 < L.nx) atomicAdd(p + 2, acc[r][1].x);
                if (ix0 + 3 >= 0 && ix0 + 3 < L.nx) atomicAdd(p + 3, acc[r][1].y);
            }
        }
        acc[r][0] = acc[r][1] = make_float2(0.f, 0.f);
    }
}

template <int R>
__device__ __forceinline__ void flush_grad(const ResArgs &a, const Own<R> &o, float2 (&acc)[R][2])
{
    const Lay2D &L = a.L;
#pragma unroll
    for (int r = 0; r < R; ++r) {
        if (o.in >> r & 1) {
            float *p = a.acc_grad + (long long)(o.i0 + r) * L.nxp + o.j0;
            if ((L.nxp & 3) == 0) {
                red_add4(p, acc[r][0].x, acc[r][0].y, acc[r][1].x, acc[r][1].y);
            } else {
                atomicAdd(p, acc[r][0].x);
                if (o.j0 + 1 < L.nxp) atomicAdd(p + 1, acc[r][0].y);
                if (o.j0 + 2 < L.nxp) atomicAdd(p + 2, acc[r][1].x);
                if (o.j0 + 3 < L.nxp) atomicAdd(p + 3, acc[r][1].y);
            }
        }
        acc[r][0] = acc[r][1] = make_float2(0.f, 0.f);
    }
}

// The compute warps' time loop over one round of shots: shots g, g + G, ... of
// the warp's group g.
template <int R, int G, int MODE, int ACC>
__device__ __forceinline__ bool fwd_loop(const ResArgs &a, const Own<R> &o, float *sm, const float4 (&ca)[R], const float *kb,
                                         float2 (&acc)[R][2], ResShared &sh, int group, int accg, int shot0, int nsh, unsigned srcs,
                                         uint32_t pf)
{
    const int nt = a.nt, fs = a.t.fs, lane = threadIdx.x & 31;
    for (int n = 0; n < nt; ++n) {
        const uint32_t par = (pf + n) & 1u;
        if (ACC && n > 0 && n % RES_SUM == 0) flush_illum<R>(a, o, acc, accg);
        for (int s = group; s < nsh; s += G) {
            if (!res_wait(smem_u32(&sh.bars.full[s]), par, &sh.abort)) return false;
            const float *f = sm + (2 * s + (n & 1)) * fs + o.so;
            float *g = sm + (2 * s + ((n + 1) & 1)) * fs + o.so;
            if (n == nt - 1) {
                if (ACC == 1 && o.on) {
#pragma unroll
                    for (int r = 0; r < R; ++r) {
                        const float4 u = lds4(f + r * RES_P);
                        acc[r][0] = fma2(lo2(u), lo2(u), acc[r][0]);
                        acc[r][1] = fma2(hi2(u), hi2(u), acc[r][1]);
                    }
                }
                continue;
            }
            if (a.snaps != nullptr && o.on && n % a.snap_k == 0) { // the state before the step
                float *sp = a.snaps + ((long long)(n / a.snap_k) * 2 * a.ns + shot0 + s) * a.L.fstride + fidx(a.L, o.i0, o.j0);
                float *sq = sp + (long long)a.ns * a.L.fstride;
#pragma unroll
                for (int r = 0; r < R; ++r)
                    if (o.in >> r & 1) {
                        *reinterpret_cast<float4 *>(sp + r * a.L.pitch) = lds4(f + r * RES_P);
                        *reinterpret_cast<float4 *>(sq + r * a.L.pitch) = lds4(g + r * RES_P);
                    }
            }
            if (o.on) {
                // the source's point, if this thread holds it: its u^{n-1} and sum
                // before the row loop replaces them, its update after it
                int srow = -1, scol = 0;
                float prev = 0.f, sum = 0.f;
                if (srcs >> s & 1) {
                    scol = sh.src[s].y - o.j0;
                    srow = (unsigned)scol < 4u ? sh.src[s].x - o.i0 : -1;
                    if ((unsigned)srow < (unsigned)R) {
                        prev = g[srow * RES_P + scol];
                        if (ACC == 2) sum = get<R>(acc, srow, scol);
                    }
                }
                fwd_rows<R, MODE, ACC>(f, g, ca, kb, acc);
                if ((srcs >> s & 1) && (unsigned)srow < (unsigned)R) {
                    const int d = srow * RES_P + scol;
                    const float u0 = f[d], q = __fadd_rn(point_lap(f + d), sh.amp[n & 1][s] * a.src_scale);
                    const float t = __fmul_rn(kb[srow * RES_KP + scol], __fmaf_rn(prev, -1.f, u0));
                    const float un = __fadd_rn(u0, __fmaf_rn(pick<R>(ca, srow, scol), q, t));
                    g[d] = un;
                    if (ACC == 2) {
                        const float d2 = __fadd_rn(__fmaf_rn(u0, -2.f, un), prev);
                        put<R>(acc, srow, scol, __fmaf_rn(d2, d2, sum));
                    }
                }
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&sh.bars.done[s]));
            // the level for the offset-Hessian sums, after the others may go on
            // (this thread's own points: only its next step on this buffer, two
            // levels on, overwrites them)
            if (a.hist != nullptr && o.on) {
                float *hp = a.hist + ((long long)n * a.ns + shot0 + s) * a.L.fstride + fidx(a.L, o.i0, o.j0);
#pragma unroll
                for (int r = 0; r < R; ++r)
                    if (o.in >> r & 1) *reinterpret_cast<float4 *>(hp + r * a.L.pitch) = lds4(g + r * RES_P);
            }
        }
    }
    return true;
}

template <int R, int NW, int G, int ACC>
__global__ void __launch_bounds__(32 * (NW + RES_SVC), 1) k_fwd_resident(const __grid_constant__ ResArgs a)
{
    extern __shared__ unsigned char smem_raw[];
    __shared__ ResShared sh;
    // the damping factors of the tile, then per shot u of even and odd levels
    // and the receiver list
    float *kbs = reinterpret_cast<float *>(align_smem(smem_raw));
    const Lay2D &L = a.L;
    const ResTile &t = a.t;
    float *sm = kbs + RES_KP * t.th;
    const Cta c = cta_of(t);
    const int wid = threadIdx.x >> 5;
    const int fs = t.fs, nt = a.nt;
    int2 *list = reinterpret_cast<int2 *>(sm + 2 * t.s * fs);
    Xch *xt = reinterpret_cast<Xch *>(list + t.s * RES_MAXE);
    int2 *bl = reinterpret_cast<int2 *>(xt + ((t.ne + 1) & ~1));
    xch_init(xt, t, c);
    res_init(sh, NW / G);
    __syncthreads();
    band_init(bl, &sh.nband, L, t, c);
    const int first = c.set * t.per, count = max(0, min(t.per, a.ns - first));

    for (int base = 0, round = 0; base < count; base += t.s, ++round) {
        const int nsh = min(t.s, count - base);
        for (int e = threadIdx.x; e < 2 * nsh * (fs / 4); e += blockDim.x)
            reinterpret_cast<float4 *>(sm)[e] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (threadIdx.x < nsh) {
            const int shot = first + base + threadIdx.x;
            sh.src[threadIdx.x] = a.src_ij[shot];
            sh.rng[threadIdx.x] = a.seis != nullptr
                ? make_int2(a.rptr[c.tile * a.ns + shot], a.rptr[c.tile * a.ns + shot + 1]) : make_int2(0, 0);
        }
        __syncthreads();
        for (int s = 0; s < nsh; ++s)
            for (int e = sh.rng[s].x + threadIdx.x; e < sh.rng[s].y; e += blockDim.x) {
                const int2 en = a.rent[e];
                const int row = en.x / (4 * t.w4), col = en.x - row * (4 * t.w4);
                list[s * RES_MAXE + e - sh.rng[s].x] = make_int2((row + RADIUS) * RES_P + RADIUS + col, en.y);
            }
        __syncthreads();
        if (wid < NW) {
            // ------------------------------------------------ compute warps
            Own<R> o;
            const int group = wid / (NW / G), thread = threadIdx.x - group * (32 * NW / G);
            own_init<R>(o, L, t, c, thread);
            float4 ca[R];
            float2 acc[R][2];
            coefficients<R>(ca, kbs + o.ko, o, a);
            if (ACC) {
#pragma unroll
                for (int r = 0; r < R; ++r) acc[r][0] = acc[r][1] = make_float2(0.f, 0.f);
            }
            unsigned srcs = 0; // shots whose source the warp holds
            for (int s = group; s < nsh; s += G)
                if (__any_sync(0xffffffffu, o.on && (unsigned)(sh.src[s].x - o.i0) < (unsigned)R &&
                                                (unsigned)(sh.src[s].y - o.j0) < 4u))
                    srcs |= 1u << s;
            const uint32_t pf = (uint32_t)(round * nt);
            const bool ok = __any_sync(0xffffffffu, o.bmask != 0)
                ? fwd_loop<R, G, 1, ACC>(a, o, sm, ca, kbs + o.ko, acc, sh, group, c.set * G + group, first + base, nsh, srcs, pf)
                : fwd_loop<R, G, 0, ACC>(a, o, sm, ca, kbs + o.ko, acc, sh, group, c.set * G + group, first + base, nsh, srcs, pf);
            if (ACC && ok) flush_illum<R>(a, o, acc, c.set * G + group);
            // the last two levels: checked, and kept for an adjoint pass
            if (ok && o.on) {
                bool fin = true;
                for (int s = group; s < nsh; s += G)
#pragma unroll
                    for (int b = 0; b < 2; ++b) {
                        float *ug = a.u[b] + (long long)(first + base + s) * L.fstride;
#pragma unroll
                        for (int r = 0; r < R; ++r)
                            if (o.in >> r & 1) {
                                const float4 v = lds4(sm + (2 * s + b) * fs + o.so + r * RES_P);
                                fin = fin && finite4(v);
                                if (a.save) *reinterpret_cast<float4 *>(ug + fidx(L, o.i0 + r, o.j0)) = v;
                            }
                    }
                if (!fin) atomicOr(a.status, ST_NONFINITE);
            }
        } else {
            const uint32_t pf = (uint32_t)(round * nt), pd = (uint32_t)(round * (nt - 1));
            const int ntiles = t.ntx * t.ntz, slot0 = res_slot(round, nt, 0);
            uint2 *xb = a.xch + (long long)c.set * t.s * 2 * ntiles * t.ne * 4;
            if (wid == NW)
                service_export<1>(a, sm, xt, bl, xb, &sh, c.tile, 0, first + base, nsh, nt, nt - 1, pd, pf, slot0);
            else if (wid <= NW + RES_IMPORT)
                service_import<1>(sm, xt, xb, &sh, t.ne, ntiles, fs, 0, nsh, nt, nt - 1, pf, pf, slot0, wid - NW - 1);
            else
                service_traces(a, sm, list, bl, &sh, first + base, nsh, pd);
        }
        __syncthreads();
        if (sh.abort) {
            if (threadIdx.x == 0) atomicOr(a.status, ST_TIMEOUT);
            return;
        }
    }
}

// ----------------------------------------------------------- backward loop
// Per shot in flight: the receivers of the tile, all in one row of it, the
// values fetched for a step, and the row of the adjoint source they make, by
// parity of the step.
struct ResInj {
    float val[2][RES_MAXE];
    float row[2][RES_KP];
    unsigned short col[RES_MAXE];
};

// Data warp of the backward loop: amplitudes and adjoint source of the tile's
// receivers, a step ahead.
__device__ __noinline__ void service_adjoint(const ResArgs &a, ResInj *inj, ResShared *sh, int shot0, int nsh, uint32_t pd)
{
    const int lane = threadIdx.x & 31, nt = a.nt;
    auto fetch = [&](int s, int m) {
        const int b = (nt - 1 - m) & 1;
        if (lane == 0) copy4(&sh->amp[b][s], &a.wav[(long long)(shot0 + s) * nt + m - 1]);
        const int rb = sh->rng[s].x, n = sh->rng[s].y - rb;
        for (int e = lane; e < n; e += 32) copy4(&inj[s].val[b][e], &a.adj[(long long)m * a.nent + rb + e]);
    };
    // the fetched values as a row of the tile (receivers on one cell add up)
    auto assemble = [&](int s, int m) {
        const int b = (nt - 1 - m) & 1, n = sh->rng[s].y - sh->rng[s].x;
        if (n == 0) return;
        float *row = inj[s].row[b];
        *reinterpret_cast<float4 *>(row + 4 * lane) = make_float4(0.f, 0.f, 0.f, 0.f);
        __syncwarp();
        for (int e = lane; e < n; e += 32) atomicAdd(&row[inj[s].col[e]], inj[s].val[b][e] * a.adj_scale);
    };
    for (int s = 0; s < nsh; ++s) fetch(s, nt - 1);
    copies_wait();
    for (int m = nt - 1; m >= 1; --m) {
        const int v = nt - 1 - m;
        for (int s = 0; s < nsh; ++s) {
            bool ok = v == 0 || res_wait(smem_u32(&sh->bars.done[s]), (pd + v - 1) & 1u, &sh->abort);
            copies_wait_but(nsh - 1); // this step's values, fetched nsh groups ago
            if (!__all_sync(0xffffffffu, ok)) {
                copies_wait();
                return;
            }
            assemble(s, m);
            mbar_arrive(smem_u32(&sh->bars.full[s]));
            if (m > 1) fetch(s, m - 1);
            copies_commit();
        }
    }
    copies_wait();
}

// The wavefield half of a backward step at the thread's points: f: u^{m-1}, g:
// u^m, replaced by u^{m-2} in the model (the reverse step; the sponge cells come
// from the checkpoint, see service_export) where store is set; qu = Lhat
// u^{m-1}. MODE as in fwd_rows.
template <int R, int MODE>
__device__ __forceinline__ void bwd_rows_u(float2 (&qu)[R][2], const float *f, float *g, const float4 (&ca)[R],
                                           bool store, unsigned bmask)
{
    float4 zc[R + 2 * RADIUS];
#pragma unroll
    for (int k = 0; k <= 2 * RADIUS; ++k) zc[k] = lds4(f + (k - RADIUS) * RES_P);
    RowIn now, nextr;
    now.load(f, g);
#pragma unroll
    for (int r = 0; r < R; ++r) {
        if (r + 1 < R) {
            zc[r + 1 + 2 * RADIUS] = lds4(f + (r + 1 + RADIUS) * RES_P);
            nextr.load(f + (r + 1) * RES_P, g + (r + 1) * RES_P);
        }
        float2 u1[2], un[2];
        row_lap(qu[r], u1, now, zc, r);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const float2 c = half2of(ca[r], h); // c2 in the model
            un[h] = sub2(u1[h], fma2(make_float2(-c.x, -c.y), qu[r][h], sub2(half2of(now.prev, h), u1[h])));
        }
        const float4 u4 = make_float4(un[0].x, un[0].y, un[1].x, un[1].y);
        const unsigned mk = MODE == 0 ? 0u : bmask >> (4 * r) & 15u;
        if (store && mk == 0) {
            *reinterpret_cast<float4 *>(g + r * RES_P) = u4;
        } else if (MODE != 0 && store && mk != 15u) {
#pragma unroll
            for (int p = 0; p < 4; ++p)
                if (!(mk >> p & 1)) g[r * RES_P + p] = comp(u4, p);
        }
        now = nextr;
    }
}

// The adjoint half: f: psi^{m+1}, g: psi^{m+2}, replaced by psi^m; acc += psi^m
// qu. MODE 2: the receivers of the shot lie in row irow of the thread (any
// other value: none), their adjoint source in `in`.
template <int R, int MODE>
__device__ __forceinline__ void bwd_rows_psi(float2 (&acc)[R][2], const float2 (&qu)[R][2], const float *f, float *g,
                                             const float4 (&ca)[R], const float *kb, int irow, const float *in)
{
    float4 zc[R + 2 * RADIUS];
#pragma unroll
    for (int k = 0; k <= 2 * RADIUS; ++k) zc[k] = lds4(f + (k - RADIUS) * RES_P);
    RowIn now, nextr;
    now.load(f, g);
#pragma unroll
    for (int r = 0; r < R; ++r) {
        if (r + 1 < R) {
            zc[r + 1 + 2 * RADIUS] = lds4(f + (r + 1 + RADIUS) * RES_P);
            nextr.load(f + (r + 1) * RES_P, g + (r + 1) * RES_P);
        }
        float2 q[2], p1[2], pn[2];
        row_lap(q, p1, now, zc, r);
        if (MODE == 2 && irow == r) {
            const float4 v = lds4(in);
            q[0] = add2(q[0], lo2(v));
            q[1] = add2(q[1], hi2(v));
        }
        row_update<MODE != 0>(pn, p1, now.prev, q, ca[r], kb + r * RES_KP);
        *reinterpret_cast<float4 *>(g + r * RES_P) = make_float4(pn[0].x, pn[0].y, pn[1].x, pn[1].y);
        acc[r][0] = fma2(pn[0], qu[r][0], acc[r][0]);
        acc[r][1] = fma2(pn[1], qu[r][1], acc[r][1]);
        now = nextr;
    }
}

// The compute warps' backward time loop over one round of shots.
template <int R, int G, int MODE>
__device__ __forceinline__ bool bwd_loop(const ResArgs &a, const Own<R> &o, float *sm, const float4 (&ca)[R], const float *kb,
                                         float2 (&acc)[R][2], ResShared &sh, const ResInj *inj, int group, int nsh, unsigned srcs,
                                         uint32_t pf)
{
    const int nt = a.nt, fs = a.t.fs, lane = threadIdx.x & 31;
    for (int m = nt - 1; m >= 1; --m) {
        const int step = nt - 1 - m, pc = (m - 1) & 1, pn = m & 1, par = step & 1;
        if (step > 0 && step % RES_SUM == 0) flush_grad<R>(a, o, acc);
        for (int s = group; s < nsh; s += G) {
            if (!res_wait(smem_u32(&sh.bars.full[s]), (pf + step) & 1u, &sh.abort)) return false;
            if (o.on) {
                float *b4 = sm + 4 * s * fs + o.so;
                const float *uc = b4 + pc * fs, *p1 = b4 + (2 + pc) * fs; // u^{m-1}, psi^{m+1}
                float *ua = b4 + pn * fs, *p2 = b4 + (2 + pn) * fs;       // u^m, psi^{m+2}
                int srow = -1, scol = 0;
                float prev = 0.f;
                if (srcs >> s & 1) { // (as in fwd_loop)
                    scol = sh.src[s].y - o.j0;
                    srow = (unsigned)scol < 4u ? sh.src[s].x - o.i0 : -1;
                    if ((unsigned)srow < (unsigned)R) prev = ua[srow * RES_P + scol];
                }
                float2 qu[R][2];
                bwd_rows_u<R, MODE>(qu, uc, ua, ca, m >= 2, o.bmask);
                if ((srcs >> s & 1) && (unsigned)srow < (unsigned)R) { // (a source lies in the model)
                    const int d = srow * RES_P + scol;
                    const float u1 = uc[d], q = __fadd_rn(point_lap(uc + d), sh.amp[par][s] * a.src_scale);
                    put<R>(qu, srow, scol, q);
                    const float t = __fmaf_rn(-pick<R>(ca, srow, scol), q, __fmaf_rn(u1, -1.f, prev));
                    if (m >= 2) ua[d] = __fmaf_rn(t, -1.f, u1);
                }
                const int irow = MODE == 2 ? sh.rrow[s] - o.i0 : -1;
                bwd_rows_psi<R, MODE>(acc, qu, p1, p2, ca, kb, irow, inj[s].row[par] + (o.ko & (RES_KP - 1)));
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&sh.bars.done[s]));
        }
    }
    return true;
}

template <int R, int NW, int G>
__global__ void __launch_bounds__(32 * (NW + RES_SVC), 1) k_bwd_resident(const __grid_constant__ ResArgs a)
{
    extern __shared__ unsigned char smem_raw[];
    __shared__ ResShared sh;
    const Lay2D &L = a.L;
    const ResTile &t = a.t;
    const Cta c = cta_of(t);
    const int wid = threadIdx.x >> 5;
    const int fs = t.fs, nt = a.nt;
    // the damping factors of the tile, per shot u of even / odd levels and psi of
    // even / odd m, then the receiver lists
    float *kbs = reinterpret_cast<float *>(align_smem(smem_raw));
    float *sm = kbs + RES_KP * t.th;
    ResInj *inj = reinterpret_cast<ResInj *>(sm + 4 * t.s * fs);
    Xch *xt = reinterpret_cast<Xch *>(inj + t.s);
    int2 *bl = reinterpret_cast<int2 *>(xt + ((t.ne + 1) & ~1));
    xch_init(xt, t, c);
    res_init(sh, NW / G);
    __syncthreads();
    band_init(bl, &sh.nband, L, t, c);
    const int first = c.set * t.per, count = max(0, min(t.per, a.ns - first));

    for (int base = 0, round = 0; base < count; base += t.s, ++round) {
        const int nsh = min(t.s, count - base);
        // u^{nt-2} and u^{nt-1} with their halo from the forward pass, psi = 0
        const int cols = t.w4 + 2, rows = t.th + 2 * RADIUS;
        for (int e = threadIdx.x; e < 4 * nsh * (fs / 4); e += blockDim.x)
            reinterpret_cast<float4 *>(sm)[e] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (threadIdx.x < nsh) {
            const int shot = first + base + threadIdx.x;
            sh.src[threadIdx.x] = a.src_ij[shot];
            sh.rng[threadIdx.x] = a.adj != nullptr
                ? make_int2(a.rptr[c.tile * a.ns + shot], a.rptr[c.tile * a.ns + shot + 1]) : make_int2(0, 0);
            sh.rrow[threadIdx.x] = sh.rng[threadIdx.x].x < sh.rng[threadIdx.x].y
                ? c.r0 + a.rent[sh.rng[threadIdx.x].x].x / (4 * t.w4) : -RES_KP;
        }
        __syncthreads();
        for (int e = threadIdx.x; e < 2 * nsh * rows * cols; e += blockDim.x) {
            const int f = e / (rows * cols), w = e - f * (rows * cols);
            const int rr = w / cols, cc = w - rr * cols;
            const int i = c.r0 - RADIUS + rr, j = 4 * (c.c0 + cc - 1);
            if (i >= 0 && i < L.nzp && j >= 0 && j < L.nxp) {
                const float *ug = a.u[f & 1] + (long long)(first + base + (f >> 1)) * L.fstride;
                *reinterpret_cast<float4 *>(sm + (4 * (f >> 1) + (f & 1)) * fs + rr * RES_P + 4 * cc) =
                    __ldcg(reinterpret_cast<const float4 *>(ug + fidx(L, i, j)));
            }
        }
        for (int s = 0; s < nsh; ++s)
            for (int e = sh.rng[s].x + threadIdx.x; e < sh.rng[s].y; e += blockDim.x) {
                inj[s].col[e - sh.rng[s].x] = (unsigned short)(a.rent[e].x % (4 * t.w4));
            }
        __syncthreads();
        if (wid < NW) {
            // ------------------------------------------------ compute warps
            Own<R> o;
            const int group = wid / (NW / G), thread = threadIdx.x - group * (32 * NW / G);
            own_init<R>(o, L, t, c, thread);
            float4 ca[R];
            float2 acc[R][2];
            coefficients<R>(ca, kbs + o.ko, o, a);
#pragma unroll
            for (int r = 0; r < R; ++r) acc[r][0] = acc[r][1] = make_float2(0.f, 0.f);
            unsigned srcs = 0; // shots whose source the warp holds
            bool recs = false; // receivers of a shot in the warp's rows
            for (int s = group; s < nsh; s += G) {
                if (__any_sync(0xffffffffu, o.on && (unsigned)(sh.src[s].x - o.i0) < (unsigned)R &&
                                                (unsigned)(sh.src[s].y - o.j0) < 4u))
                    srcs |= 1u << s;
                recs |= (unsigned)(sh.rrow[s] - o.i0) < (unsigned)R;
            }
            const uint32_t pf = (uint32_t)(round * (nt - 1));
            bool ok;
            if (__any_sync(0xffffffffu, recs))
                ok = bwd_loop<R, G, 2>(a, o, sm, ca, kbs + o.ko, acc, sh, inj, group, nsh, srcs, pf);
            else if (__any_sync(0xffffffffu, o.bmask != 0))
                ok = bwd_loop<R, G, 1>(a, o, sm, ca, kbs + o.ko, acc, sh, inj, group, nsh, srcs, pf);
            else
                ok = bwd_loop<R, G, 0>(a, o, sm, ca, kbs + o.ko, acc, sh, inj, group, nsh, srcs, pf);
            if (ok) flush_grad<R>(a, o, acc);
            if (ok && o.on) {
                bool fin = true;
                for (int s = group; s < nsh; s += G)
#pragma unroll
                    for (int r = 0; r < R; ++r)
                        if (o.in >> r & 1) fin = fin && finite4(lds4(sm + (4 * s + 2) * fs + o.so + r * RES_P));
                if (!fin) atomicOr(a.status, ST_NONFINITE);
            }
        } else {
            const uint32_t p0 = (uint32_t)(round * (nt - 1));
            const int ntiles = t.ntx * t.ntz, b0 = first_parity(2, nt), slot0 = res_slot(round, nt, 0);
            uint2 *xb = a.xch + (long long)c.set * t.s * 4 * ntiles * t.ne * 4;
            if (wid == NW)
                service_export<2>(a, sm, xt, bl, xb, &sh, c.tile, b0, first + base, nsh, nt - 1, nt - 1, p0, p0, slot0);
            else if (wid <= NW + RES_IMPORT)
                service_import<2>(sm, xt, xb, &sh, t.ne, ntiles, fs, b0, nsh, nt - 1, nt - 1, p0, p0, slot0, wid - NW - 1);
            else
                service_adjoint(a, inj, &sh, first + base, nsh, p0);
        }
        __syncthreads();
        if (sh.abort) {
            if (threadIdx.x == 0) atomicOr(a.status, ST_TIMEOUT);
            return;
        }
    }
}

// ----------------------------------------- offset Hessian of kept levels
// The offset-Hessian sums of a resident forward pass: its registers hold no 11
// or 13 sums per point, so the pass keeps its levels (small problems only) and
// this kernel sums the products of all of them at once: a CTA takes a 64 x 8 tile
// of the physical points and a run of images, whose rows with 12 columns on each
// side go through two shared-memory stages of OI images; each thread holds the
// sums of its 4 points over the run. Bound by latency (100 x 200, 1596 images: 69
// us, 2.1 TB/s of the images' rows with their columns; issue active 55%, DRAM 31% of
// peak, fixed-latency dependencies and the stages' barriers first among the stalls).
constexpr int OI = 4, OI_W = TX + 2 * HMAX_LIMIT;

template <int NHC>
__global__ void __launch_bounds__(TPB, 4) k_offh_images(const float *__restrict__ u, const __grid_constant__ Lay2D L,
                                                        long long n, int run, int hmax, float *acc_offh)
{
    constexpr int WL = HMAX_LIMIT, NW4 = (2 * WL + 4) / 4;
    __shared__ __align__(16) float sm[2][OI][8 * OI_W];
    const int ntx = (L.nx + TX - 1) / TX, ntz = (L.nz + 7) / 8;
    const int c = blockIdx.x / (ntx * ntz), tile = blockIdx.x - c * (ntx * ntz), bz = tile / ntx, bx = tile - bz * ntx;
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4, iz0 = 8 * bz, ixb = TX * bx;
    const long long k0 = (long long)c * run, k1 = min(n, k0 + run);
    const bool al = (L.P & 3) == 0;
    // images k .. k + OI - 1 into stage b; cells below the model or past the
    // last column's offsets belong to points that are not stored
    auto stage = [&](long long k, int b) {
#pragma unroll 1
        for (int q = 0; q < OI && k + q < k1; ++q) {
            const float *src = u + (k + q) * L.fstride;
            float *dst = sm[b][q];
            if (al) {
                for (int e = threadIdx.x; e < 8 * (OI_W / 4); e += TPB) {
                    const int r = e / (OI_W / 4), c4 = 4 * (e - r * (OI_W / 4)), col = ixb - WL + c4;
                    if (iz0 + r < L.nz && col < L.nx + WL) copy16(dst + r * OI_W + c4, src + fidx(L, iz0 + r + L.P, col + L.P));
                }
            } else {
                for (int e = threadIdx.x; e < 8 * OI_W; e += TPB) {
                    const int r = e / OI_W, cc = e - r * OI_W, col = ixb - WL + cc;
                    if (iz0 + r < L.nz && col < L.nx + WL) copy4(dst + r * OI_W + cc, src + fidx(L, iz0 + r + L.P, col + L.P));
                }
            }
        }
        copies_commit();
    };
    float2 acc[NHC][2];
#pragma unroll
    for (int h = 0; h < NHC; ++h) acc[h][0] = acc[h][1] = make_float2(0.f, 0.f);
    stage(k0, 0);
    int b = 0;
    for (long long k = k0; k < k1; k += OI, b ^= 1) {
        if (k + OI < k1) stage(k + OI, b ^ 1);
        else copies_commit();
        copies_wait_but(1);
        __syncthreads();
        const int nq = (int)min((long long)OI, k1 - k);
#pragma unroll 1
        for (int q = 0; q < nq; ++q) {
            const float *row = &sm[b][q][ty * OI_W + 4 * tx];
            float w[4 * NW4];
#pragma unroll
            for (int e = 0; e < NW4; ++e) {
                const float4 t = lds4(row + 4 * e);
                w[4 * e] = t.x; w[4 * e + 1] = t.y; w[4 * e + 2] = t.z; w[4 * e + 3] = t.w;
            }
            // even h: points (0, 1), (2, 3) on lane pairs; odd h: (1, 2) paired, 0 and 3 scalar
#pragma unroll
            for (int h = 0; h < NHC; ++h) {
                if ((h & 1) == 0) {
#pragma unroll
                    for (int y = 0; y < 2; ++y)
                        acc[h][y] = fma2(f2(w[WL + 2 * y + h], w[WL + 2 * y + 1 + h]),
                                         f2(w[WL + 2 * y - h], w[WL + 2 * y + 1 - h]), acc[h][y]);
                } else {
                    acc[h][0] = fma2(f2(w[WL + 1 + h], w[WL + 2 + h]), f2(w[WL + 1 - h], w[WL + 2 - h]), acc[h][0]);
                    acc[h][1].x = fmaf(w[WL + h], w[WL - h], acc[h][1].x);
                    acc[h][1].y = fmaf(w[WL + 3 + h], w[WL + 3 - h], acc[h][1].y);
                }
            }
        }
        __syncthreads(); // stage b is free
    }
    copies_wait();
    const int iz = iz0 + ty, ix0 = ixb + 4 * tx;
    if (iz >= L.nz || ix0 >= L.nx) return;
    const long long nphys = (long long)L.nz * L.nx, at = (long long)iz * L.nx + ix0;
#pragma unroll
    for (int h = 0; h < NHC; ++h) {
        if (h > hmax) continue;
        const float v[4] = {(h & 1) ? acc[h][1].x : acc[h][0].x, (h & 1) ? acc[h][0].x : acc[h][0].y,
                            (h & 1) ? acc[h][0].y : acc[h][1].x, acc[h][1].y};
#pragma unroll
        for (int p = 0; p < 4; ++p)
            if (ix0 + p < L.nx) atomicAdd(acc_offh + h * nphys + at + p, v[p]);
    }
}

// ------------------------------------------------------------------ host
struct ResVariant {
    int r, nw, g; // rows per thread, compute warps, groups of them
    const void *fn;
};
#define RES_F(R, NW, G, ACC) {R, NW, G, (const void *)k_fwd_resident<R, NW, G, ACC>}
#define RES_FS(ACC) {RES_F(1, 16, 1, ACC), RES_F(2, 12, 1, ACC), RES_F(3, 12, 1, ACC), RES_F(4, 12, 1, ACC), RES_F(3, 12, 2, ACC), RES_F(4, 12, 2, ACC)}
#define RES_B(R, NW, G) {R, NW, G, (const void *)k_bwd_resident<R, NW, G>}
constexpr int RES_NVAR = 6;
const ResVariant g_res[4][RES_NVAR] = {RES_FS(0), RES_FS(1), RES_FS(2),
                                       {RES_B(1, 12, 1), RES_B(2, 12, 1), RES_B(3, 12, 1), RES_B(4, 8, 1), RES_B(3, 12, 2), RES_B(2, 12, 2)}};

const ResVariant *res_variants(ResKind kind, int &n)
{
    n = RES_NVAR;
    return g_res[kind];
}

constexpr int RES_SMEM = 225 * 1024; // dynamic shared memory of a CTA (static parts and alignment beside it)

std::once_flag g_res_once;
int g_res_sms = 152;

void res_prepare()
{
    std::call_once(g_res_once, [] {
        int dev = 0, v = 0;
        if (cudaGetDevice(&dev) == cudaSuccess) {
            if (cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess && v > 0) g_res_sms = v;
            for (int k = 0; k < 4; ++k) {
                int n = 0;
                const ResVariant *vs = res_variants((ResKind)k, n);
                for (int i = 0; i < n; ++i)
                    cudaFuncSetAttribute(vs[i].fn, cudaFuncAttributeMaxDynamicSharedMemorySize, RES_SMEM);
            }
        }
        cudaGetLastError();
    });
}

} // namespace

ResTile res_plan(const Lay2D &L, int ns, ResKind kind)
{
    ResTile best{};
    double best_us = 1e30, best_level = 0.0;
    if (ns < 1) return best;
    res_prepare();
    const bool bwd = kind == RES_BWD;
    int nv = 0;
    const ResVariant *vs = res_variants(kind, nv);
    const int nx4 = (L.nxp + 3) / 4, fields = bwd ? 4 : 2;
    // costs by which the tilings are compared (us): a step of one shot per 128 points
    // of the tile and the service warps per float4 exchanged, which overlap over the
    // shots in flight; the way of a halo to the neighbours
    const double us128 = bwd ? 0.075 : 0.035, us_svc = 0.003, us_way = 0.0055;
    const int mt = ((L.nxp + TX - 1) / TX) * ((L.nzp + 7) / 8); // receiver tables are sized for this many tiles
    for (int vi = 0; vi < nv; ++vi) {
        const int R = vs[vi].r, G = vs[vi].g, NT = 32 * vs[vi].nw / G;
        for (int ntx = 1; ntx <= 64 && ntx <= nx4; ++ntx) {
            const int w4 = (nx4 + ntx - 1) / ntx;
            if ((nx4 + w4 - 1) / w4 != ntx || w4 > RES_W) continue;
            const int gmax = NT / w4;
            for (int ntz = 1; ntz <= g_res_sms; ++ntz) {
                int th = (L.nzp + ntz - 1) / ntz;
                th = (th + R - 1) / R * R;
                if (th < RADIUS) th = (RADIUS + R - 1) / R * R;
                if (th / R > gmax) continue;
                if ((L.nzp + th - 1) / th != ntz) continue;
                const int tiles = ntx * ntz;
                if (tiles > g_res_sms || tiles > mt) break;
                const int fs = (th + 2 * RADIUS) * RES_P;
                const long long per_shot =
                    (long long)fields * fs * 4 + (bwd ? (long long)sizeof(ResInj) : 8LL * RES_MAXE);
                const int ne = 8 * w4 + 2 * th;
                // alignment, damping factors, exchange table, sponge list
                const int fixed = 128 + 4 * RES_KP * th + (int)sizeof(Xch) * (ne + 1) + 8 * th * w4;
                int smax = (int)std::min<long long>(RES_SMAX, (RES_SMEM - fixed) / per_shot);
                if (smax < 1) continue;
                const int sets = std::min(ns, g_res_sms / tiles);
                const int per = (ns + sets - 1) / sets;
                const int rounds0 = (per + smax - 1) / smax;
                const int s = (per + rounds0 - 1) / rounds0;
                const int rounds = (per + s - 1) / s;
                const int nx = tiles > 1 ? ne * fields / 2 : 0;
                const double comp = 0.15 + us128 * ((w4 * (th / R) + 31) / 32) * R, svc = 0.3 + us_svc * nx;
                const double us = rounds * std::max(s * std::max(comp, svc), comp + (tiles > 1 ? 1.1 : 0.4) + us_way * nx);
                if (us > best_us) continue;
                ResTile t{};
                t.ok = 1;
                t.variant = vi;
                t.w4 = w4;
                t.th = th;
                t.g = th / R;
                t.ntx = ntx;
                t.ntz = ntz;
                t.sets = sets;
                t.accs = sets * G;
                t.s = s;
                t.per = per;
                t.fs = fs;
                t.ne = ne;
                t.xch = (long long)sets * s * tiles * ne * fields * 32;
                t.smem = (int)(fixed + s * per_shot);
                // Equal costs are common (they count whole warps and rounds). Then the expected
                // level decides, which knows the variants' rows apart (us per level: forward 45 x
                // 126, 70 shots, one / two rows per thread 5.1 / 4.1; with illumination 367 x 470,
                // 17 shots, four / three rows 14.6 / 11.4; backward 115 x 1153, 16 shots, four /
                // two rows 46 / 33), and between one and two groups of warps the shots in flight:
                // two from 3 on (one / two groups: forward with illumination 100 x 200, 16 shots
                // 4.46 / 4.23, 60 x 120, 32 shots 4.93 / 4.30; backward 37 x 100, 64 shots 15.6 /
                // 14.9; with fewer shots a group idles: backward 100 x 200, 4 shots 3.84 / 4.44,
                // 167 x 716, 1 shot 4.8 / 6.4); else tiles whose rows a warp covers whole, with fewer
                // bank conflicts (forward 153 x 219, 8 shots, 8 / 9 float4s wide 2.9 / 3.4, 72 x
                // 1137, 2 shots, 8 / 6 wide 2.8 / 3.2)
                double level = 0.0; // (not known)
                if (us == best_us) {
                    if (best_level == 0.0) best_level = res_level_us(L, best, kind, false);
                    level = res_level_us(L, t, kind, false);
                }
                if (us == best_us && level >= best_level) {
                    const bool same = best.w4 == w4 && best.th == th && vs[best.variant].r == R;
                    if (level > best_level || !(same ? G > 1 && s >= 3 : 32 % w4 == 0 && 32 % best.w4 != 0)) continue;
                }
                best = t;
                best_us = us;
                best_level = level;
            }
        }
    }
    if (best.ok) best.us = (float)best_us;
    return best;
}

// A round's level: per shot the longest of the compute warps (by rows per thread and
// 128 points), the exchange (by float4s) and the data warp (by float4s of the
// checkpoint, whole ones and those with other cells among them, which go cell by
// cell), over the shots in flight; at least one shot's compute and the way of its
// halo. The maxima are rounded off (8-norm), where two of them are near each other
// they do not quite overlap. Fitted to 229 problems (those of the streaming steps'
// level_us and 110 others), up to two tilings of each, with and without checkpoint:
// 5 to 95% within -19 and +16%.
double res_level_us(const Lay2D &L, const ResTile &t, ResKind kind, bool band)
{
    struct Cost {
        double comp, row, rows[4], svc, xch, data, whole, mixed, way, dist;
    };
    static const Cost fwd = {0.53, 0.02, {0.067, 0.037, 0.0355, 0.0305}, 0.15, 0.0, 0.70, 0.0030, 0.007, 1.02, 0.0077};
    static const Cost sums = {0.54, 0.062, {0.070, 0.039, 0.033, 0.042}, 0.21, 0.0, 0.70, 0.0031, 0.0078, 1.12, 0.0065};
    static const Cost bwd = {0.82, 0.86, {0.167, 0.067, 0.051, 0.0}, 0.95, 0.0042, 0.62, 0.0048, 0.031, 1.29, 0.0036};
    const Cost &c = kind == RES_BWD ? bwd : (kind == RES_FWD ? fwd : sums);
    const int R = t.th / t.g, nx4 = (L.nxp + 3) / 4;
    const double edge = t.ntx * t.ntz > 1 ? t.ne * (kind == RES_BWD ? 2.0 : 1.0) : 0.0;
    const double comp = c.comp + c.row * (R - 1) + c.rows[R - 1] * ((t.w4 * t.g + 31) / 32) * R, svc = c.svc + c.xch * edge;
    double data = 0.0;
    for (int bz = 0; band && bz < t.ntz; ++bz) {
        // sponge rows and model rows of the tile row
        const int r0 = bz * t.th, r1 = std::min(L.nzp, r0 + t.th);
        const int model = std::max(0, std::min(r1, L.P + L.nz) - std::max(r0, L.P)), sponge = r1 - r0 - model;
        for (int bx = 0; bx < t.ntx; ++bx) {
            int n[4] = {0, 0, 0, 0}; // float4s of a sponge row, whole and mixed; of a model row
            for (int q = bx * t.w4; q < std::min(nx4, (bx + 1) * t.w4); ++q) {
                const int j0 = 4 * q, j1 = std::min(j0 + 4, L.nxp);
                const int cells = j1 - j0 - std::max(0, std::min(j1, L.P + L.nx) - std::max(j0, L.P));
                ++n[j1 - j0 == 4 ? 0 : 1];
                if (cells > 0) ++n[cells == 4 ? 2 : 3];
            }
            data = std::max(data, c.data + c.whole * (sponge * n[0] + model * n[2]) + c.mixed * (sponge * n[1] + model * n[3]));
        }
    }
    auto pow8 = [](double a) { return a *= a, a *= a, a * a; };
    auto norm = [&](double a, double b, double d) { return std::sqrt(std::sqrt(std::sqrt(pow8(a) + pow8(b) + pow8(d)))); };
    const int rounds = (t.per + t.s - 1) / t.s;
    const double way = comp + (t.ntx * t.ntz > 1 ? c.way : 0.4) + c.dist * edge;
    return rounds * norm(t.s * norm(comp, svc, data), way, 0.0);
}

namespace {
std::mutex g_pin_mu;
std::set<std::array<int, 4>> g_pinned;
} // namespace

void res_pin(StepKind kind, const Lay2D &L, int ns, bool pinned)
{
    std::lock_guard<std::mutex> lock(g_pin_mu);
    const std::array<int, 4> key = {kind, L.nzp, L.nxp, ns};
    if (pinned)
        g_pinned.insert(key);
    else
        g_pinned.erase(key);
}

bool res_pinned(StepKind kind, const Lay2D &L, int ns)
{
    std::lock_guard<std::mutex> lock(g_pin_mu);
    return g_pinned.count({kind, L.nzp, L.nxp, ns}) != 0;
}

void res_pin_clear()
{
    std::lock_guard<std::mutex> lock(g_pin_mu);
    g_pinned.clear();
}

cudaError_t launch_offh_images(const Lay2D &L, const float *u, long long n, int hmax, float *acc, cudaStream_t st)
{
    if (n <= 0) return cudaSuccess;
    res_prepare();
    // runs of images such that the tiles fill the SMs' 4 CTAs about twice, of at
    // least 32 images (each run adds its sums to memory once) and at most 256
    // (FP32 sums of more images lose digits that the sum over runs keeps)
    const long long tiles = (long long)((L.nz + 7) / 8) * ((L.nx + TX - 1) / TX);
    const long long runs = std::max<long long>(1, 8LL * g_res_sms / tiles);
    const int run = (int)std::max<long long>(32, std::min<long long>(256, (n + runs - 1) / runs));
    const unsigned grid = (unsigned)(tiles * ((n + run - 1) / run));
    if (hmax <= 3)
        k_offh_images<4><<<grid, TPB, 0, st>>>(u, L, n, run, hmax, acc);
    else if (hmax <= 10)
        k_offh_images<11><<<grid, TPB, 0, st>>>(u, L, n, run, hmax, acc);
    else
        k_offh_images<13><<<grid, TPB, 0, st>>>(u, L, n, run, hmax, acc);
    return cudaGetLastError();
}

cudaError_t launch_resident(const ResArgs &a, ResKind kind, cudaStream_t st)
{
    // no packet of an earlier pass may carry a level of this one
    const cudaError_t e = cudaMemsetAsync(a.xch, 0, (size_t)a.t.xch, st);
    if (e != cudaSuccess) return e;
    int n = 0;
    const ResVariant &v = res_variants(kind, n)[a.t.variant];
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(a.t.sets * a.t.ntx * a.t.ntz);
    cfg.blockDim = dim3(32 * (v.nw + RES_SVC));
    cfg.dynamicSmemBytes = (size_t)a.t.smem;
    cfg.stream = st;
    // every CTA waits on its neighbours: all of them have to be resident
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    void *params[] = {const_cast<ResArgs *>(&a)};
    return cudaLaunchKernelExC(&cfg, v.fn, params);
}

} // namespace fwi
