// fwi_resident.h -- argument block and tiling of the chip-resident 2-D time
// loops (fwi_resident2d.cu). Not part of the public ABI.
#pragma once

#include "fwi_args.h"

namespace fwi {

constexpr int RES_SMAX = 8;        // most shots in flight per CTA
constexpr int RES_SVC = 4;         // service warps per CTA
constexpr int RES_MAXE = 256;      // most receivers of one (tile, shot)
// forward passes without an illumination sum, with that of u^2, of u_tt^2; backward
enum ResKind { RES_FWD = 0, RES_FWD_U2 = 1, RES_FWD_UTT2 = 2, RES_BWD = 3 };

// How one pass is laid out over the chip: every shot in flight is cut into
// ntx x ntz tiles of 4 w4 columns by th rows, one CTA each; a CTA holds its
// tile of s shots at a time; `sets` groups of CTAs work on different shots.
struct ResTile {
    int ok;            // 0: the streaming steps are used
    int variant;       // compiled (rows per thread, warps) variant of the kind
    int w4, th, g;     // float4 columns, rows, row groups of a tile
    int ntx, ntz;      // tiles of one shot
    int sets, s;       // CTA groups; shots in flight per CTA
    int accs;          // illumination sums held apart: one per set and group of warps,
                       // so that each is added to in a fixed order
    int per;           // shots of one set over the whole pass
    int fs;            // floats of one field tile with its halo
    int ne;            // float4s of a tile's edge strips
    int smem;          // dynamic shared memory
    long long xch;     // bytes of the exchange packets
    float us;          // expected time of one level of all shots, in us
};

struct ResArgs {
    Lay2D L;
    ResTile t;
    const float *c2, *damp;
    const int2 *src_ij;
    const float *wav;      // [ns][nt]
    float src_scale;
    int ns, nt, nrec;
    int *status;
    uint2 *xch;            // packets {value, level}: [sets * s][buffer][field][ntx * ntz][ne][4]
    const int *rptr;       // receivers of (tile, shot): [ptr[t * ns + s], ptr[t * ns + s + 1])
    const int2 *rent;      // {local = row * 4 w4 + column, r}
    float *u[2];           // wavefields of even / odd levels, field layout
    float *band;           // [ns][nt][nbandp]
    // forward
    float *seis;           // [ns][nt][nrec] or null
    float *acc_illum;      // [accs][nz][nx] or null
    int save;              // the final two levels are written to u
    float *snaps;          // F32 snapshots (u^n, u^{n-1}) at n = 0, snap_k, ..., [.][2][ns] fields, or null
    int snap_k;
    float *hist;           // levels 1 .. nt - 1 of every shot ([nt - 1][ns] fields) or null
    // backward
    const float *adj;      // [nt][nent], receiver-table order, or null
    int nent;
    float adj_scale;
    float *acc_grad;       // [nzp][nxp]
};

// Packet buffer (0 or 1) of level v of a round: the parity of the exchange's number
// over all rounds, round (nt - 2) + v (levels 1 .. nt - 2 are exchanged in every
// round of both passes), see fwi_resident2d.cu
__host__ __device__ inline int res_slot(int round, int nt, int v)
{
    return (int)(((unsigned)round * (unsigned)nt + (unsigned)v) & 1u);
}

// Layout of a pass over ns shots (ok = 0 where one shot does not fit the chip)
ResTile res_plan(const Lay2D &L, int ns, ResKind kind);
// expected time (us) of one level of all shots; band: the pass keeps (forward) or
// reads (backward) the sponge checkpoint
double res_level_us(const Lay2D &L, const ResTile &t, ResKind kind, bool band);
// shapes whose streaming steps were pinned (fwi_autotune_set): no resident loop
void res_pin(StepKind kind, const Lay2D &L, int ns, bool pinned);
bool res_pinned(StepKind kind, const Lay2D &L, int ns);
void res_pin_clear();
// acc[h][x] += sum over n images (field layout, fstride apart) of u(x + h) u(x - h),
// h = 0 .. hmax, at the physical points
cudaError_t launch_offh_images(const Lay2D &L, const float *u, long long n, int hmax, float *acc, cudaStream_t st);
cudaError_t launch_resident(const ResArgs &a, ResKind kind, cudaStream_t st);

} // namespace fwi
