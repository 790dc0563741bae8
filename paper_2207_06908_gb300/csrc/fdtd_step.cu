// fdtd_step.cu -- the fused Yee time step of the GB300 FDTD library
// (sm_103a, FP32): Kuklin, arXiv 2207.06908, Sec. 2.1, Eq. fdtdhx (H half
// step) then Eq. fdtdex (E half step, loss term time-averaged), with the
// CPML of Sec. 2.2, over the whole grid in one launch.
//
// Structure (one launch per time step; fields ping-pong between buffers):
//   - Work items are (z block, 32x16 column tile) pairs in z-block-major
//     order, handed out by an atomic counter to a persistent grid of
//     (SMs x resident CTAs); all CTAs march near the same z, so the halo
//     planes one CTA loads are still in L2 when its neighbours load them.
//     Within a z block the column tiles that meet a CPML layer come first:
//     the last items of a launch are the quick ones.
//   - One producer warp streams, plane by plane, TMA boxes into two
//     shared-memory rings tracked by mbarriers: E^n (tile + 1-cell halo on
//     every side, x start rounded down to a 16-byte boundary) into a
//     4-slot ring (two planes in use, two in flight), and H^{n-1/2} (tile +
//     low halo), the class bytes and, in a CPML layer, the auxiliary fields
//     into a 3-slot ring (one in use, two in flight).  The arrays of one kind
//     are the fourth dimension of one tensor map, so a plane takes three
//     copies, five in a tile that meets an x and a y layer.
//   - Eight row warps, two neighbouring x cells per lane: warp w owns rows w
//     and w + 8 of the tile (so a y layer's rows spread over all warps).  Per
//     plane k they form H^{n+1/2}(k) of their cells, then, after the one
//     barrier a plane has, E^{n+1}(k) from that H plane and the plane before
//     it, both in shared memory.  Two more warps recompute (never exchange)
//     H^{n+1/2} of the low-y row and the low-x column of the halo meanwhile.
//   - The layers an item meets are template arguments: an item that meets
//     none runs without any CPML code, the others with one branch per layer.
// What bounds it: DRAM on grids that fill the chip, otherwise the latency of
// a plane's chain (copies landed, H, barrier, E), which a CTA cannot
// overlap with more than the ring holds: 1300 cycles alone on an SM without a
// layer, 2000 with one.  Hence few and wide instructions per plane, values
// the same for a warp in uniform registers (item by shuffle, one base
// pointer per array and plane, one 32-bit offset per lane), no choice inside
// the plane loop but whether a lane is in a layer, registers split by role (setmaxnreg) so that nothing
// spills, and few copies issued by a converged warp.  With four cells per
// lane (16-byte accesses) the plane loop has fewer instructions but half the
// warps to hide its latency, and measured slower (197 us on the 256^3 CPML
// grid at the same stage as 171); running 64-bit pointers per lane in place
// of offsets took 11 % more instructions (256^3 PEC 134 us).  Measured (us
// per step; one cell per lane, fifteen copies a plane and 16 planes per item
// before): 256^3 PEC 136.3 -> 129.8, 256^3 with a 10-cell CPML 175.9 ->
// 160.8, 512x512x384 with 12 cells 956 -> 914, 128^3 with 8 cells 42.7 ->
// 30.8, 64^3 with 8 cells 25.6 -> 9.4 (programmatic dependencies between the
// steps' kernels, fdtd_runtime.cu, included).
// DRAM traffic per cell and step: 6 FP32 reads + 6 writes + 1 class byte
// (49 B) plus the CPML auxiliaries in the layer; every halo read is an L2
// hit.  Every wait is bounded; on a timeout the kernel records an error
// flag, drains its copies in flight and returns.
#include <cuda.h>

#include <algorithm>
#include <type_traits>

#include "fdtd.h"
#include "fdtd_internal.h"

namespace fdtd {
namespace {

using geom::TX;                        // tile width
using geom::TY;                        // tile height
constexpr int GX = 2;                  // neighbouring x cells per lane of a row warp (8-byte accesses)
constexpr int LPR = TX / GX;           // lanes per tile row
constexpr int RPW = 32 / LPR;          // tile rows per row warp (w, w + NCW, ...)
constexpr int NCW = TY / RPW;          // row warps
constexpr int NHW = 2;                 // halo warps: low-y row, low-x column
constexpr int NCONS = (NCW + NHW) * 32;  // row warps + halo warps
constexpr int NTHREADS = (NCW + 4) * 32;   // + the producer warp, one warp idle: whole warpgroups
// registers: the row warps (the first warpgroups) hold their cells' state and
// take row_regs each, the halo warps and the producer aux_regs; together
// what the block is launched with (two blocks per SM)
// (the split that leaves no spills: a batch's row warps read their arguments
// from shared memory and need fewer, its producer more)
constexpr int LAUNCH_REGS = 80;
constexpr int row_regs(bool batch) { return batch ? 88 : 96; }
constexpr int aux_regs(bool batch) { return batch ? 64 : 48; }
static_assert(NCW % 4 == 0, "row warps fill warpgroups");
static_assert(NCW * row_regs(false) + 4 * aux_regs(false) <= (NCW + 4) * LAUNCH_REGS &&
              NCW * row_regs(true) + 4 * aux_regs(true) <= (NCW + 4) * LAUNCH_REGS,
              "the shares of the launch's registers");
constexpr int NE = 4;                  // E-plane ring: planes k, k+1 in use, two ahead
constexpr int NH_MAX = 3;              // H / class / CPML ring: plane k in use, up to two ahead
                                       // (a launch whose auxiliary region is large uses 2)

using geom::XO;
using geom::EBX;
using geom::EBY;
using geom::HBX;
using geom::HBY;
using geom::CXO;
using geom::CBX;
using geom::CBY;

constexpr int al128(int v) { return (v + 127) / 128 * 128; }

// Shared-memory copy of a class's coefficients: three float4 rows
// {db_x, db_y, db_z, 0}, {ca_x, ca_y, ca_z, 0}, {cb_x, cb_y, cb_z, 0}, so the
// H half step reads one 16-byte row and the E half step two (the global
// table keeps kNumCoef floats per class: ca[3], cb[3], db[3]).
constexpr int kTabStride = 12;
__device__ __forceinline__ int tab_src(int slot)
{
    const int r = slot >> 2, c = slot & 3;
    return c == 3 ? -1 : (r == 0 ? 6 + c : (r == 1 ? c : 3 + c));
}
// one array's box in a slot; the boxes of one kind lie one after the other,
// as one copy writes them (a kind starts on a 128-byte boundary)
constexpr int E_COMP = EBX * EBY * 4;
constexpr int H_COMP = HBX * HBY * 4;
constexpr int C_BYTES = al128(CBX * CBY);
constexpr int PE_BYTES = TX * TY * 4;                // E-type psi box: the tile itself
// E slot: three E boxes and a header: item, -, staged-layer flags of the
// plane, x-box start, y-box start, domain, the item's x0, y0, ka, kb
constexpr int OFF_HDR = 3 * E_COMP;
constexpr int ESLOT = al128(OFF_HDR + 40);
// H slot: three H boxes, the class box, then the staged-auxiliary region
// (grid dependent size).  In a z-layer plane the region holds the z boxes
// (2 H-type with the H box, 2 E-type with the tile box); elsewhere the x
// boxes (4, narrowed along x) followed by the y boxes (4, narrowed along y).
constexpr int OFF_H = 0;
constexpr int OFF_C = al128(3 * H_COMP);
constexpr int OFF_PSI = OFF_C + C_BYTES;
constexpr int OFF_ZE = al128(2 * H_COMP);            // the E-type z boxes in the region
constexpr int Z_BYTES = OFF_ZE + 2 * PE_BYTES;
constexpr uint32_t TX_E = 3u * EBX * EBY * 4;
constexpr uint32_t TX_H = 3u * HBX * HBY * 4 + CBX * CBY;
constexpr uint32_t TX_Z = 2u * HBX * HBY * 4 + 2u * TX * TY * 4;
constexpr int F_Z = 1, F_X = 2, F_Y = 4;              // staged-layer flags

__host__ __device__ constexpr int hslot_bytes(int region) { return al128(OFF_PSI + region); }

// block-level layout: E ring, H ring, H^{n+1/2} planes, barriers, misc,
// coefficient table, CPML profiles
constexpr int SM_EH = 0;
constexpr int SM_HH = NE * ESLOT;
constexpr int HNEW_PLANE = HBY * HBX;
constexpr int HNEW_BYTES = 2 * 3 * HNEW_PLANE * 4;     // [2][3][HBY][HBX]
constexpr int NBAR = 2 * NE + 2 * NH_MAX;             // fullE, emptyE, fullH, emptyH
// x-layer coefficients of the current item's columns: {b, c, 1/kappa} at E,
// then at H positions, TX floats each (zero outside the layer, where nothing
// uses them), and three zero coefficient rows
constexpr int XC_BYTES = (6 * TX + 12) * 4;
struct Layout {
    int hslot, hnew, xc, bar, misc, tab;
    __host__ __device__ Layout(int region, int nh)
    {
        hslot = hslot_bytes(region);
        hnew = SM_HH + nh * hslot;
        xc = hnew + HNEW_BYTES;
        bar = xc + XC_BYTES;
        misc = bar + NBAR * 8;
        tab = misc + 32;
    }
};

__host__ __device__ inline int smem_bytes(int n_classes, int d, int region, int nh)
{
    return Layout(region, nh).tab + al128(sizeof(StepArgs)) + n_classes * kTabStride * 4 + 3 * 2 * 2 * d * 16 +
           128;
}

constexpr unsigned long long kWaitNs = 2000000000ull;   // 2 s per wait

// ---- PTX helpers ----------------------------------------------------------
__device__ __forceinline__ uint32_t smem_u32(const void *p)
{
    return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ unsigned long long gtimer()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint32_t bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}

__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}

// bounded wait on one mbarrier phase; gives up on timeout (limit_ns) or when
// another warp of the CTA has already given up
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int *abort,
                                          unsigned long long limit_ns = kWaitNs)
{
    if (mbar_try(bar, parity)) return true;
    const unsigned long long t0 = gtimer();
    while (true) {
        if (mbar_try(bar, parity)) return true;
        if (*abort) return false;
        if (gtimer() - t0 > limit_ns) return false;
    }
}

// Self-test of the bounded wait: one thread waits, through mbar_wait, on an
// mbarrier phase that nothing will complete, gives up after limit_ns and
// records that in *flag (the step kernel's timeout path, without a step).
__global__ void wait_selftest_kernel(unsigned long long limit_ns, int *flag)
{
    __shared__ uint64_t bar;
    __shared__ int abort_flag;
    if (threadIdx.x == 0) {
        mbar_init(smem_u32(&bar), 1);
        abort_flag = 0;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        const bool ok = mbar_wait(smem_u32(&bar), 0, &abort_flag, limit_ns);
        *flag = ok ? 2 : 1;
    }
    __syncthreads();
    if (threadIdx.x == 0) asm volatile("mbarrier.inval.shared::cta.b64 [%0];" ::"r"(smem_u32(&bar)) : "memory");
}

__device__ int g_selftest_flag;
__device__ int g_selftest_leave[2];

// box at (x, y, z) of every array of the map
__device__ __forceinline__ void tma_load(uint32_t dst, const CUtensorMap *map, int x, int y, int z, uint32_t bar)
{
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%2, %3, %4, %5}], [%6];" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(0), "r"(bar)
        : "memory");
}

// one lane of the (converged) warp
__device__ __forceinline__ bool elect_one()
{
    uint32_t ok;
    asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}\n" : "=r"(ok));
    return ok != 0;
}

__device__ __forceinline__ void consumer_sync()
{
    asm volatile("bar.sync 1, %0;" ::"n"(NCONS) : "memory");
}

// The same barrier, telling every consumer thread whether any of them gave p:
// what they decide together (to leave a CTA whose waits gave up) comes out of
// the barrier.  Each reading the abort flag for itself after a plain barrier
// could differ, as the producer may set the flag between two warps' reads,
// and the warps that stay would wait for those that left without a limit.
__device__ __forceinline__ bool consumer_any(bool p)
{
    uint32_t any;
    asm volatile(
        "{\n .reg .pred p, q;\n setp.ne.u32 p, %1, 0;\n bar.red.or.pred q, 1, %2, p;\n selp.u32 %0, 1, 0, q;\n}\n"
        : "=r"(any)
        : "r"((uint32_t)p), "n"(NCONS)
        : "memory");
    return any != 0;
}

// Self-test of leaving together: the consumer warps of a CTA go round
// consumer_any on an abort flag that the warp after them sets at some moment,
// or until `rounds` are up.  out[0]: the largest difference, over the CTAs, of
// the rounds after which two warps left; out[1]: CTAs that left early.
__global__ void __launch_bounds__(NCONS + 32) leave_selftest_kernel(int rounds, int *out)
{
    __shared__ int abort_flag, first, last;
    if (threadIdx.x == 0) {
        abort_flag = 0;
        first = rounds;
        last = 0;
    }
    __syncthreads();
    volatile int *abort = &abort_flag;
    if (threadIdx.x < NCONS) {
        int r = 0;
        while (r < rounds && !consumer_any(*abort != 0)) ++r;
        if ((threadIdx.x & 31) == 0) {
            atomicMin(&first, r);
            atomicMax(&last, r);
        }
    } else if (threadIdx.x == NCONS) {
        const unsigned long long t0 = gtimer(), t = 1000ull + 37ull * blockIdx.x;
        while (gtimer() - t0 < t) {}
        *abort = 1;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        atomicMax(out, last - first);
        if (last < rounds) atomicAdd(out + 1, 1);
    }
}

// ---- stencil cores ----------------------------------------------------------
// Layer membership of one cell, hoisted out of the per-cell work: slab
// index per axis (-1 outside the layer) and, per axis, the cell's entry in
// the staged boxes (null when not staged: read from global memory).
struct Slab {
    int sx, sy, sz;          // slab index along x, y, z or -1
    const float *base;       // staged-auxiliary region of the plane's H slot
    int xo, yo;              // float offsets of the cell in the first x / y box, or -1
    int zo;                  // float offset in the first z H-type box, or -1
};

__device__ __forceinline__ int slab_of(int i, int n, int d) { return i < d ? i : (i >= n - d ? i - (n - 2 * d) : -1); }

// CPML convolution of the two differences along one axis (Sec. 2.2): with
// the profile b, c, 1/kappa of the cell's slab entry s,
// psi <- b psi + c dif, dif <- dif / kappa + psi.  The profile row holds
// {b, c, 1/kappa, -} per slab entry, read with one 16-byte load for both
// differences.
__device__ __forceinline__ void cpml2(float &d0, float &d1, const float4 *pr, int s, float o0, float o1)
{
    const float4 pv = pr[s];
    d0 = __fmaf_rn(d0, pv.z, __fmaf_rn(pv.x, o0, __fmul_rn(pv.y, d0)));
    d1 = __fmaf_rn(d1, pv.z, __fmaf_rn(pv.x, o1, __fmul_rn(pv.y, d1)));
}

// Element of cell (i, j, k) in the compact auxiliaries of each axis, which
// hold only the layer: x [nz][ny][px] by slab column sx, y [nz][2d][pitch]
// by slab row sy, z [2d][ny][pitch] by slab plane sz (px = 2d rounded up to
// a multiple of 4, so rows stay 16-byte aligned for TMA).
// The host keeps every compact array below 2^31 elements, so 32-bit indices.
__device__ __forceinline__ int psi_x(const StepArgs &a, int sx, int j, int k) { return (k * a.ny + j) * a.px + sx; }
__device__ __forceinline__ int psi_y(const StepArgs &a, int i, int sy, int k)
{
    return (k * (2 * a.d) + sy) * a.pitch + i;
}
// elements of the compact x, y, z arrays (extents for the bounds-checked build)
__device__ __forceinline__ long long psi_n(const StepArgs &a, int u)
{
    return u == 0 ? (long long)a.nz * a.ny * a.px : (long long)(2 * a.d) * a.pitch * (u == 1 ? a.nz : a.ny);
}

// profile row of axis u at E (h = 0) or H (h = 1) positions in the staged
// profiles: [axis][E, H][2d slab entries] x {b, c, 1/kappa, -}
__device__ __forceinline__ const float4 *prow(const float *prof, int u, int h, int d2)
{
    return reinterpret_cast<const float4 *>(prof) + (u * 2 + h) * d2;
}

// H^{n+1/2} of cell (i,j,k) from E^n around it (Eq. fdtdhx and its cyclic
// analogues): Hx += db [dEy/dz - dEz/dy], Hy += db [dEz/dx - dEx/dz],
// Hz += db [dEx/dy - dEy/dx]; differences in field units, 1/dx in db.
// One cell of the low-y row or low-x column of a tile's halo, recomputed
// and never stored; its auxiliaries are in the staged boxes, which include
// the halo.
template <bool CPML>
__device__ __forceinline__ void h_core(const StepArgs &a, const float4 *t, const float *prof, const Slab &L,
                                       float ex, float ey, float ez, float ey_x1, float ez_x1,
                                       float ex_y1, float ez_y1, float ex_z1, float ey_z1, float hx0, float hy0,
                                       float hz0, float &hx, float &hy, float &hz)
{
    float hx_z = ey_z1 - ey, hx_y = ez_y1 - ez;
    float hy_x = ez_x1 - ez, hy_z = ex_z1 - ex;
    float hz_y = ex_y1 - ex, hz_x = ey_x1 - ey;
    if (CPML) {
        const int d2 = 2 * a.d;
        if (L.sx >= 0)
            cpml2(hy_x, hz_x, prow(prof, 0, 1, d2), L.sx, L.base[L.xo], L.base[L.xo + (a.pg.xb >> 2)]);
        if (L.sy >= 0)
            cpml2(hx_y, hz_y, prow(prof, 1, 1, d2), L.sy, L.base[L.yo], L.base[L.yo + (a.pg.yb >> 2)]);
        if (L.sz >= 0)
            cpml2(hx_z, hy_z, prow(prof, 2, 1, d2), L.sz, L.base[L.zo], L.base[L.zo + H_COMP / 4]);
    }
    const float4 db = t[0];
    hx = __fmaf_rn(db.x, hx_z - hx_y, hx0);
    hy = __fmaf_rn(db.y, hy_x - hy_z, hy0);
    hz = __fmaf_rn(db.z, hz_y - hz_x, hz0);
}

// ---- two cells per lane -----------------------------------------------------
// The row warps' stencil: a lane owns two neighbouring x cells of one tile
// row, so a field box is read with one 8-byte access per component and stored
// with another, the index arithmetic and the barriers are paid once per two
// cells, and the differences and layer sums run two cells to an instruction
// (packed FP32 pairs).  The layers an item meets are template arguments and
// the lanes outside them skip them.  Every sum is written as explicit products
// and fused multiply-adds, so every instantiation of the kernel rounds alike.
using F2 = unsigned long long;           // two FP32 values
__device__ __forceinline__ F2 pk(float lo, float hi)
{
    F2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ float lo2(F2 v) { return __uint_as_float((uint32_t)v); }
__device__ __forceinline__ float hi2(F2 v) { return __uint_as_float((uint32_t)(v >> 32)); }
__device__ __forceinline__ F2 fma2(F2 a, F2 b, F2 c)
{
    F2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ F2 mul2(F2 a, F2 b)
{
    F2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

__device__ __forceinline__ F2 ld2(const float *p) { return *reinterpret_cast<const F2 *>(p); }
__device__ __forceinline__ void st2(float *p, F2 x) { *reinterpret_cast<F2 *>(p) = x; }
// a - b (the product with -1 is exact, so this is the plain difference)
__device__ __forceinline__ F2 sub2(F2 a, F2 b) { return fma2(b, pk(-1.f, -1.f), a); }
// differences along x: of the next cell and this one (e: the cell after the
// pair), of this one and the one before (w)
__device__ __forceinline__ F2 next_diff(F2 x, float e) { return pk(hi2(x) - lo2(x), e - hi2(x)); }
__device__ __forceinline__ F2 prev_diff(F2 x, float w) { return pk(lo2(x) - w, hi2(x) - lo2(x)); }
// a pair into a plane of an array (element `plane` on; the same for the
// whole warp) at the lane's element off of the plane, if `on`.  The second
// cell of a side of odd length falls into the row's padding (rows are padded
// to 16 elements), where it is zero for a field (its coefficients are) and
// never read.  n: the array's elements, for the bounds-checked build
template <typename Off>
__device__ __forceinline__ void put2(float *base, long long plane, Off off, F2 x, bool on, long long n, int site,
                                     int *bounds)
{
    float *p = base + plane;
    if (on && in_bounds(plane + off, n, site, bounds) && in_bounds(plane + off + 1, n, site, bounds)) st2(p + off, x);
}

// what a lane's pair of cells is to the layers of its item, formed once per item
enum { IN0 = 1, IN1 = 2, XM0 = 4, XM1 = 8, XM = 12, YM = 16 };
struct Pair {
    int fl;                  // IN0, IN1: the first, second cell lies inside the grid; XM0, XM1: in an x layer;
                             // YM: the row lies in a y layer
    int xo;                  // float offset of the first cell's entry in the first x box
    int yo;                  // float offset of the pair in the first y box
    const float4 *py;        // its y profile row at E positions, 2d rows before the one at H positions
    unsigned off;            // its element in a plane of the fields and z auxiliaries
    int xoff, yoff;          // of the x, y auxiliaries (a lane outside the layer: not used)
};

// one plane's auxiliaries for a pair
struct PlaneX {
    const float *base;       // staged-auxiliary region
    int sz;                  // slab plane or -1
    int zo, zeo;             // the pair's offsets in the first z H-type / E-type box
    const float *xc;         // x coefficients of the pair's columns (b; c and 1/kappa TX floats on)
};

// CPML of one difference of the pair (see cpml2): psi <- b psi + c dif,
// dif <- dif / kappa + psi
struct PX {
    F2 b, c, ki;
};
__device__ __forceinline__ PX profx(const float4 &q) { return PX{pk(q.x, q.x), pk(q.y, q.y), pk(q.z, q.z)}; }
__device__ __forceinline__ PX profx(const float *xc) { return PX{ld2(xc), ld2(xc + TX), ld2(xc + 2 * TX)}; }
__device__ __forceinline__ F2 cpmlx(F2 &dif, const PX &q, F2 o)
{
    const F2 p = fma2(q.b, o, mul2(q.c, dif));
    dif = fma2(dif, q.ki, p);
    return p;
}
// Both differences of a pair that the layer may cut: in0, in1 for its two
// cells.  A difference outside the layer stays as it is.
__device__ __forceinline__ void cpmlx_cut(F2 &d0, F2 &d1, const PX &q, F2 o0, F2 o1, bool in0, bool in1, F2 &p0, F2 &p1)
{
    p0 = fma2(q.b, o0, mul2(q.c, d0));
    p1 = fma2(q.b, o1, mul2(q.c, d1));
    float l0 = lo2(d0), h0 = hi2(d0), l1 = lo2(d1), h1 = hi2(d1);
    if (in0) {
        l0 = __fmaf_rn(l0, lo2(q.ki), lo2(p0));
        l1 = __fmaf_rn(l1, lo2(q.ki), lo2(p1));
    }
    if (in1) {
        h0 = __fmaf_rn(h0, hi2(q.ki), hi2(p0));
        h1 = __fmaf_rn(h1, hi2(q.ki), hi2(p1));
    }
    d0 = pk(l0, h0);
    d1 = pk(l1, h1);
}

// Both differences of the x layer at E (h = 0) or H (h = 1) positions.  VEC:
// every pair lies wholly in a layer or outside and its entries start on an
// 8-byte boundary (d and nx even); otherwise cell by cell (a choice made
// inside the plane loop costs more than the layer's arithmetic).  A pair
// never has members in both layers (they are two cells apart at least).
// Lanes outside a layer skip it.  Running along with coefficients of zero and
// one in place of that, they made NaNs of an infinite difference, and of an
// infinite auxiliary of the row they read; skipping is no slower (us per step:
// 64^3 with 8 cells 9.37 -> 9.36, 128^3 with 8 31.3 -> 30.8, 96^3 with 10
// 21.7 -> 21.4, 256^3 with 10 161.2 -> 160.9).  Selects or predicates on the
// sums spilled or cost up to 4 %; skipping cell by cell spilled too, so a
// pair that a layer may cut leaves out the sums.
template <bool VEC>
__device__ __forceinline__ void cpml_x(const StepArgs &a, const Pair &G, const PlaneX &P, int h, int k, F2 &d0, F2 &d1)
{
    if (VEC && !(G.fl & XM)) return;
    const int q = a.pg.xb >> 2, at = h ? 0 : 2;
    const float *b = P.base + at * q + G.xo;
    const PX pr = profx(P.xc + (h ? 3 * TX : 0));
    const F2 o0 = VEC ? ld2(b) : pk(b[0], b[1]), o1 = VEC ? ld2(b + q) : pk(b[q], b[q + 1]);
    F2 p0, p1;
    if (VEC) {
        p0 = cpmlx(d0, pr, o0);
        p1 = cpmlx(d1, pr, o1);
    } else {
        cpmlx_cut(d0, d1, pr, o0, o1, G.fl & XM0, G.fl & XM1, p0, p1);
    }
    const int pl = k * (a.ny * a.px);
    float *u0 = a.psi_out[h ? PSI_HY_X : PSI_EY_X], *u1 = a.psi_out[h ? PSI_HZ_X : PSI_EZ_X];
    const long long n = psi_n(a, 0);
    if (VEC) {
        put2(u0, pl, G.xoff, p0, true, n, 3, a.bounds);
        put2(u1, pl, G.xoff, p1, true, n, 3, a.bounds);
    } else {
        u0 += pl;
        u1 += pl;
        if ((G.fl & XM0) && in_bounds(pl + G.xoff, n, 3, a.bounds)) {
            u0[G.xoff] = lo2(p0);
            u1[G.xoff] = lo2(p1);
        }
        if ((G.fl & XM1) && in_bounds(pl + G.xoff + 1, n, 3, a.bounds)) {
            u0[G.xoff + 1] = hi2(p0);
            u1[G.xoff + 1] = hi2(p1);
        }
    }
}
// of the y layer
__device__ __forceinline__ void cpml_y(const StepArgs &a, const Pair &G, const PlaneX &P, int h, int k, F2 &d0, F2 &d1)
{
    if (!(G.fl & YM)) return;
    const int q = a.pg.yb >> 2, at = h ? 0 : 2;
    const float *b = P.base + G.yo + at * q;
    const PX pr = profx(G.py[h ? 2 * a.d : 0]);
    const F2 p0 = cpmlx(d0, pr, ld2(b)), p1 = cpmlx(d1, pr, ld2(b + q));
    const int pl = k * (2 * a.d * a.pitch);
    put2(a.psi_out[h ? PSI_HX_Y : PSI_EX_Y], pl, G.yoff, p0, true, psi_n(a, 1), 3, a.bounds);
    put2(a.psi_out[h ? PSI_HZ_Y : PSI_EZ_Y], pl, G.yoff, p1, true, psi_n(a, 1), 3, a.bounds);
}
// of the z layer
__device__ __forceinline__ void cpml_z(const StepArgs &a, const Pair &G, const PlaneX &P, const float *prof, int h,
                                       F2 &d0, F2 &d1)
{
    const float *b = P.base + (h ? P.zo : P.zeo);
    const PX pr = profx(prow(prof, 2, h, 2 * a.d)[P.sz]);
    const F2 p0 = cpmlx(d0, pr, ld2(b)), p1 = cpmlx(d1, pr, ld2(b + (h ? H_COMP : PE_BYTES) / 4));
    const int pl = P.sz * (a.ny * a.pitch);
    put2(a.psi_out[h ? PSI_HX_Z : PSI_EX_Z], pl, G.off, p0, G.fl & IN0, psi_n(a, 2), 3, a.bounds);
    put2(a.psi_out[h ? PSI_HY_Z : PSI_EY_Z], pl, G.off, p1, G.fl & IN0, psi_n(a, 2), 3, a.bounds);
}

// layers met by the cells an item updates (template bits)
constexpr int LX = 1, LY = 2, LZ = 4, LXS = 8;     // LX, LXS: the x layer in whole pairs, cell by cell

// H^{n+1/2} of a pair (h_core) from H^{n-1/2} in place; t0, t1: its cells'
// coefficient rows.
template <int L>
__device__ __forceinline__ void h_corex(const StepArgs &a, const Pair &G, const PlaneX &P, const float *prof, int k,
                                        F2 ex, F2 ey, F2 ez, F2 ex_y1, F2 ez_y1, float ey_e, float ez_e,
                                        F2 ex_z1, F2 ey_z1, const float4 *t0, const float4 *t1, F2 &hx, F2 &hy, F2 &hz)
{
    F2 hx_z = sub2(ey_z1, ey), hx_y = sub2(ez_y1, ez);
    F2 hy_x = next_diff(ez, ez_e), hy_z = sub2(ex_z1, ex);
    F2 hz_y = sub2(ex_y1, ex), hz_x = next_diff(ey, ey_e);
    if constexpr (L & (LX | LXS)) cpml_x<(L & LX) != 0>(a, G, P, 1, k, hy_x, hz_x);
    if constexpr (L & LY) cpml_y(a, G, P, 1, k, hx_y, hz_y);
    if constexpr (L & LZ) cpml_z(a, G, P, prof, 1, hx_z, hy_z);
    const F2 dx = sub2(hx_z, hx_y), dy = sub2(hy_x, hy_z), dz = sub2(hz_y, hz_x);
    const float4 b0 = t0[0], b1 = t1[0];
    hx = pk(__fmaf_rn(b0.x, lo2(dx), lo2(hx)), __fmaf_rn(b1.x, hi2(dx), hi2(hx)));
    hy = pk(__fmaf_rn(b0.y, lo2(dy), lo2(hy)), __fmaf_rn(b1.y, hi2(dy), hi2(hy)));
    hz = pk(__fmaf_rn(b0.z, lo2(dz), lo2(hz)), __fmaf_rn(b1.z, hi2(dz), hi2(hz)));
}

// Hx and Hy^{n+1/2} of a pair of the plane below an item, which the item
// reads but does not update, in place; x / y auxiliaries that are not staged
// there (flags f) come from global memory, elements gx, gy.
__device__ __forceinline__ void h_belowx(const StepArgs &a, const Pair &G, const PlaneX &P, const float *prof, int f,
                                         int gx, int gy, F2 ex, F2 ey, F2 ez, F2 ez_y1, float ez_e, F2 ex_z1, F2 ey_z1,
                                         const float4 *t0, const float4 *t1, F2 &hx, F2 &hy)
{
    F2 hx_z = sub2(ey_z1, ey), hx_y = sub2(ez_y1, ez);
    F2 hy_x = next_diff(ez, ez_e), hy_z = sub2(ex_z1, ex);
    auto far = [&](const float *arr, int g, int m, int u) {
        float o0 = 0.f, o1 = 0.f;
        if ((m & 1) && in_bounds(g, psi_n(a, u), 4, a.bounds)) o0 = __ldcg(arr + g);
        if ((m & 2) && in_bounds(g + 1, psi_n(a, u), 4, a.bounds)) o1 = __ldcg(arr + g + 1);
        return pk(o0, o1);
    };
    if (G.fl & XM) {
        F2 o;
        if (f & F_X) o = pk(G.fl & XM0 ? P.base[G.xo] : 0.f, G.fl & XM1 ? P.base[G.xo + 1] : 0.f);
        else o = far(a.psi_in[PSI_HY_X], gx, (G.fl & XM) / XM0, 0);
        F2 none = 0, p0, p1;
        cpmlx_cut(hy_x, none, profx(P.xc + 3 * TX), o, none, G.fl & XM0, G.fl & XM1, p0, p1);
    }
    if (G.fl & YM)
        cpmlx(hx_y, profx(G.py[2 * a.d]), (f & F_Y) ? ld2(P.base + G.yo) : far(a.psi_in[PSI_HX_Y], gy, G.fl & 3, 1));
    if (P.sz >= 0) {
        const PX q = profx(prow(prof, 2, 1, 2 * a.d)[P.sz]);
        cpmlx(hx_z, q, ld2(P.base + P.zo));
        cpmlx(hy_z, q, ld2(P.base + P.zo + H_COMP / 4));
    }
    const F2 dx = sub2(hx_z, hx_y), dy = sub2(hy_x, hy_z);
    const float4 b0 = t0[0], b1 = t1[0];
    hx = pk(__fmaf_rn(b0.x, lo2(dx), lo2(hx)), __fmaf_rn(b1.x, hi2(dx), hi2(hx)));
    hy = pk(__fmaf_rn(b0.y, lo2(dy), lo2(hy)), __fmaf_rn(b1.y, hi2(dy), hi2(hy)));
}

// E^{n+1} of a pair (Eq. fdtdex with sigma E time-averaged: E = ca E +
// cb [curl_h H^{n+1/2}], 1/dx in cb), in place; hz_w, hy_w: the cell before
// the pair along x.
template <int L>
__device__ __forceinline__ void e_corex(const StepArgs &a, const Pair &G, const PlaneX &P, const float *prof, int k,
                                        F2 hx, F2 hy, F2 hz, F2 hz_ym, F2 hx_ym, float hz_w, float hy_w,
                                        F2 hx_zm, F2 hy_zm, const float4 *t0, const float4 *t1, F2 &ex, F2 &ey, F2 &ez)
{
    F2 ex_y = sub2(hz, hz_ym), ex_z = sub2(hy, hy_zm);
    F2 ey_z = sub2(hx, hx_zm), ey_x = prev_diff(hz, hz_w);
    F2 ez_x = prev_diff(hy, hy_w), ez_y = sub2(hx, hx_ym);
    if constexpr (L & (LX | LXS)) cpml_x<(L & LX) != 0>(a, G, P, 0, k, ey_x, ez_x);
    if constexpr (L & LY) cpml_y(a, G, P, 0, k, ex_y, ez_y);
    if constexpr (L & LZ) cpml_z(a, G, P, prof, 0, ex_z, ey_z);
    const F2 dx = sub2(ex_y, ex_z), dy = sub2(ey_z, ey_x), dz = sub2(ez_x, ez_y);
    const float4 a0 = t0[1], a1 = t1[1], b0 = t0[2], b1 = t1[2];
    auto up = [](float ca, float e, float cb, float c) { return __fmaf_rn(ca, e, __fmul_rn(cb, c)); };
    ex = pk(up(a0.x, lo2(ex), b0.x, lo2(dx)), up(a1.x, hi2(ex), b1.x, hi2(dx)));
    ey = pk(up(a0.y, lo2(ey), b0.y, lo2(dy)), up(a1.y, hi2(ey), b1.y, hi2(dy)));
    ez = pk(up(a0.z, lo2(ez), b0.z, lo2(dz)), up(a1.z, hi2(ez), b1.z, hi2(dz)));
}

// Current sources of the grid whose edges lie in a finished work item (Sec.
// 2.1, J = I / dx^2 on one edge, I at t_{n+1/2}): E^{n+1} += coef I on each
// edge, rounded as a separate product and sum (the arithmetic of the source
// kernel's add to the stored E).  The item's consumers stored those E^{n+1}
// before the barrier that precedes this; no other CTA touches them in this
// step.  m: bit q set for each source q in the item.
__device__ __forceinline__ void add_sources(const StepArgs &a, uint32_t m)
{
    const long long n = __ldcg(a.step) + a.step_t;
    while (m) {
        const int q = __ffs(m) - 1;
        m &= m - 1;
        const SourceDesc &sd = a.src[q];
        const float I = n < sd.n_samples ? __ldg(a.samples + sd.sample_off + n) : 0.f;
        if (!in_bounds(sd.idx, (long long)a.plane * a.nz, 5, a.bounds)) continue;
        float *e = a.Eout[sd.comp] + sd.idx;
        *e = __fadd_rn(__ldcg(e), __fmul_rn(sd.coef, I));
    }
}

// sources that lie in work item `item` of launch `launch` (bit q: source q)
__device__ __forceinline__ uint32_t item_sources(const StepArgs &a, int launch, int item)
{
    uint32_t m = 0;
    for (int q = 0; q < a.n_isrc; ++q) {
        const int2 L = __ldg(a.isrc_loc + q);
        if (L.x == launch && L.y == item) m |= 1u << q;
    }
    return m;
}

// ---- shared-memory views ----------------------------------------------------
struct EView {
    char *p;
    __device__ const float *at(int c, int row, int col) const { return reinterpret_cast<const float *>(p + c * E_COMP) + row * EBX + col; }
    __device__ float e(int c, int row, int col) const { return *at(c, row, col); }
    __device__ int *hdr() const { return reinterpret_cast<int *>(p + OFF_HDR); }
};
struct HView {
    char *p;
    __device__ const float *at(int c, int row, int col) const { return reinterpret_cast<const float *>(p + OFF_H + c * H_COMP) + row * HBX + col; }
    __device__ float h(int c, int row, int col) const { return *at(c, row, col); }
    // the classes of a pair of cells, one per byte
    __device__ uint32_t cls2(int row, int col) const { return *reinterpret_cast<const uint16_t *>(p + OFF_C + row * CBX + col); }
    __device__ int cls(int row, int col) const { return reinterpret_cast<const uint8_t *>(p + OFF_C)[row * CBX + col]; }
    __device__ const float *psi() const { return reinterpret_cast<const float *>(p + OFF_PSI); }
};

// staging of one plane, copied out of its E-slot header (the E slot may be
// handed back to the producer before the plane's E half step)
struct Stg {
    int f, xs, ys;
    __device__ explicit Stg(const int *hdr) : f(hdr[2]), xs(hdr[3]), ys(hdr[4]) {}
    __device__ Stg(int f_, int xs_, int ys_) : f(f_), xs(xs_), ys(ys_) {}
};

// Offsets of cell (i, j) at H-box position (row, col) in the x / y boxes of
// an item (-1 when the cell is outside that layer or outside the box); they
// depend on the tile only, so they are formed once per item.
__device__ __forceinline__ int x_off(const StepArgs &a, const Stg &sg, int i, int row)
{
    const int sx = slab_of(i, a.nx, a.d);
    return (sx >= 0 && sx >= sg.xs && sx < sg.xs + a.pg.w) ? a.ox / 4 + row * a.pg.w + (sx - sg.xs) : -1;
}
__device__ __forceinline__ int y_off(const StepArgs &a, const Stg &sg, int x0, int i, int j)
{
    const int sy = slab_of(j, a.ny, a.d);
    return (sy >= 0 && sy >= sg.ys && sy < sg.ys + a.pg.hy) ? a.oy / 4 + (sy - sg.ys) * HBX + (i - (x0 - XO)) : -1;
}

// the staging of one plane applied to a cell's precomputed offsets
__device__ __forceinline__ Slab slab_in(const Stg &sg, const HView &hv, int sx, int sy, int sz, int xo, int yo,
                                        int zo)
{
    return Slab{sx, sy, sz, hv.psi(), (sg.f & F_X) ? xo : -1, (sg.f & F_Y) ? yo : -1, (sg.f & F_Z) ? zo : -1};
}

// x / y layer boxes of a tile (with its low halo): whether the tile touches
// the layer and where the box narrowed to the layer starts
__device__ __forceinline__ int tile_boxes(const StepArgs &a, int x0, int y0, int &xs, int &ys)
{
    // the layer cells among x0-1 .. x0+TX-1 (y0-1 .. y0+TY-1) form one run of
    // slab entries (the low layer's, then the high layer's, contiguous in
    // the compact arrays); the x box starts at the first, rounded down to a
    // 16-byte boundary, the y box at the first
    const int d = a.d;
    int f = 0;
    xs = 0;
    ys = 0;
    const int xl = max(x0 - 1, 0), xh = min(x0 + TX, a.nx) - 1;
    if (xl < d || xh >= a.nx - d) {
        f |= F_X;
        xs = slab_of(xl < d ? xl : max(xl, a.nx - d), a.nx, d) & ~3;
    }
    const int yl = max(y0 - 1, 0), yh = min(y0 + TY, a.ny) - 1;
    if (yl < d || yh >= a.ny - d) {
        f |= F_Y;
        ys = slab_of(yl < d ? yl : max(yl, a.ny - d), a.ny, d);
    }
    return f;
}

struct Item {
    int x0, y0, ka, kb;
};

__device__ __forceinline__ Item decode(const StepArgs &a, int item)
{
    const int ncols = a.ncx * a.ncy;
    const int zb = item / ncols;
    // within a z block the column tiles that meet a CPML layer (the slowest
    // items) come first, so the items handed out last in a launch are the
    // quickest and the launch's tail is short
    const int col = __ldg(a.col_order + (item - zb * ncols));
    Item it;
    it.x0 = (col % a.ncx) * TX;
    it.y0 = (col / a.ncx) * TY;
    const int nzb1 = (a.zhi - a.zlo + a.kz - 1) / a.kz;
    if (zb < nzb1) {
        it.ka = a.zlo + zb * a.kz;
        it.kb = min(it.ka + a.kz, a.zhi);
    } else {
        it.ka = a.zlo2 + (zb - nzb1) * a.kz;
        it.kb = min(it.ka + a.kz, a.zhi2);
    }
    return it;
}

// the same item with its values in uniform registers
__device__ __forceinline__ Item uniform(const Item &it)
{
    const unsigned all = 0xffffffffu;
    return Item{__shfl_sync(all, it.x0, 0), __shfl_sync(all, it.y0, 0), __shfl_sync(all, it.ka, 0),
                __shfl_sync(all, it.kb, 0)};
}

// does any cell the item updates or recomputes lie in a CPML layer
__device__ __forceinline__ bool item_in_cpml(const StepArgs &a, const Item &it)
{
    const int d = a.d;
    if (d == 0) return false;
    if (it.ka - 1 < d || it.kb - 1 >= a.nz - d) return true;
    const int xl = max(it.x0 - 1, 0), xh = min(it.x0 + TX, a.nx) - 1;
    const int yl = max(it.y0 - 1, 0), yh = min(it.y0 + TY, a.ny) - 1;
    return xl < d || xh >= a.nx - d || yl < d || yh >= a.ny - d;
}

// A consumer warp's place in the two rings: the slot of the next plane and
// the phase its full barrier is waited on, advanced slot by slot.
template <int NH>
struct Ring {
    uint32_t e = 0, ep = 0, h = 0, hp = 0;   // E slot and phase, H slot and phase
    __device__ uint32_t e_next() const { return (e + 1) % NE; }
    __device__ void pass_e()
    {
        e = (e + 1) % NE;
        ep ^= e == 0;
    }
    __device__ void pass_h()
    {
        h = h + 1 == NH ? 0 : h + 1;
        hp ^= h == 0;
    }
};

// shared state of the consumer warps
template <int NH>
struct Cons {
    const StepArgs *a;
    char *smem;
    const float *tab, *prof;
    float *hnew, *xc;
    uint64_t *bars;
    volatile int *abort;
    int warp, lane;
    int hslot;               // bytes per H slot
    __device__ uint32_t bar(int b) const { return (uint32_t)__cvta_generic_to_shared(&bars[b]); }
    __device__ const float4 *coef(int cls) const { return reinterpret_cast<const float4 *>(tab + cls * kTabStride); }
    // barriers of a slot
    __device__ uint32_t fullE(uint32_t s) const { return bar(s); }
    __device__ uint32_t emptyE(uint32_t s) const { return bar(NE + s); }
    __device__ uint32_t fullH(uint32_t s) const { return bar(2 * NE + s); }
    __device__ uint32_t emptyH(uint32_t s) const { return bar(2 * NE + NH_MAX + s); }
    __device__ EView ev(uint32_t s) const { return EView{smem + SM_EH + s * ESLOT}; }
    __device__ HView hv(uint32_t s) const { return HView{smem + SM_HH + s * hslot}; }
    __device__ float *hn(uint32_t b, int c, int row, int col) const { return hnew + (b * 3 + c) * HNEW_PLANE + row * HBX + col; }
    __device__ void arrive(uint32_t b) const
    {
        __syncwarp();
        asm volatile(
            "{\n .reg .pred p;\n setp.eq.s32 p, %1, 0;\n @p mbarrier.arrive.shared::cta.b64 _, [%0];\n}\n" ::"r"(b),
            "r"(lane)
            : "memory");
    }
    // wait for the E plane after the current one and the current H plane
    // (the same answer in every lane)
    __device__ bool wait_plane(const Ring<NH> &R) const
    {
        const uint32_t n = R.e_next();
        return __all_sync(0xffffffffu, mbar_wait(fullE(n), R.ep ^ (n == 0), abort) &&
                                           mbar_wait(fullH(R.h), R.hp, abort));
    }
};

// One work item in a row warp.  R is at the item's first plane, ka-1, on
// entry and at the next item's on return.  A wait that gives up sets *abort;
// the warp then goes through the item's remaining barriers without touching
// the slots, so no other warp is left waiting, and the CTA leaves at the
// item's end.
// L: the layers the item's own cells meet
template <int L, int NH>
__device__ __forceinline__ void run_rows(const Cons<NH> &C, const Item &it, Ring<NH> &R, uint32_t &hb)
{
    const StepArgs &a = *C.a;
    const int lane = C.lane, d = a.d;
    // the lane's pair of cells
    const int row = 1 + C.warp + (lane / LPR) * NCW, gx = GX * (lane % LPR);
    const int lx = XO + gx, clx = CXO + gx;
    const int i = it.x0 + gx, j = it.y0 + row - 1;
    const int nv = j < a.ny ? max(0, min(GX, a.nx - i)) : 0;
    Pair G;
    G.fl = (1 << nv) - 1;
    G.xo = 0;                       // a pair outside the layer reads, cell by cell, and does not use, what lies there
    G.yo = 0;
    G.py = reinterpret_cast<const float4 *>(C.prof);
    // slab entry of the pair's first cell, in the layer its members lie in, and of its row
    const int xe = i < d ? i : i - (a.nx - 2 * d), sy = d > 0 && nv > 0 ? slab_of(j, a.ny, d) : -1;
    if (d > 0) {
        Stg tb(0, 0, 0);                // the tile's x / y layer boxes
        tb.f = tile_boxes(a, it.x0, it.y0, tb.xs, tb.ys);
#pragma unroll
        for (int c = 0; c < GX; ++c)
            if (c < nv && slab_of(i + c, a.nx, d) >= 0) G.fl |= XM0 << c;
        if (G.fl & XM) G.xo = a.ox / 4 + row * a.pg.w + xe - tb.xs;
        if (sy >= 0) {
            G.fl |= YM;
            G.yo = a.oy / 4 + (sy - tb.ys) * HBX + lx;
            G.py = prow(C.prof, 1, 0, 2 * d) + sy;
        }
    }
    G.off = (unsigned)j * a.pitch + i;
    G.xoff = j * a.px + xe;
    G.yoff = sy * a.pitch + i;
    // coefficient rows of the pair's cells (a second cell outside the grid: zeros)
    const float4 *const zero = reinterpret_cast<const float4 *>(C.xc + 6 * TX);
    auto row0 = [&](uint32_t cls) { return reinterpret_cast<const float4 *>(C.tab + (cls & 255u) * kTabStride); };
    auto row1 = [&](uint32_t cls) {
        return (G.fl & 3) == IN0 ? zero : reinterpret_cast<const float4 *>(C.tab + (cls >> 8) * kTabStride);
    };
    bool ok = __all_sync(0xffffffffu, mbar_wait(C.fullH(R.h), R.hp, C.abort));
    if (!ok) *C.abort = 1;
    // Hx, Hy of the plane below, kept where that plane's would be: the lane's
    // own cells of the other H buffer
    float *const own = C.hn(0, 0, row, lx);
    F2 hx = 0, hy = 0, hz = 0;
    if (ok && it.ka > 0) {
        const EView e0 = C.ev(R.e), e1 = C.ev(R.e_next());
        const HView h0 = C.hv(R.h);
        const int k = it.ka - 1;
        const PlaneX P{h0.psi(), d > 0 ? slab_of(k, a.nz, d) : -1, row * HBX + lx, 0, C.xc + gx};
        const uint32_t cls = h0.cls2(row, clx);
        hx = ld2(h0.at(0, row, lx));
        hy = ld2(h0.at(1, row, lx));
        h_belowx(a, G, P, C.prof, Stg(e0.hdr()).f, psi_x(a, xe, j, k), psi_y(a, i, sy, k), ld2(e0.at(0, row, lx)), ld2(e0.at(1, row, lx)),
                 ld2(e0.at(2, row, lx)), ld2(e0.at(2, row + 1, lx)), e0.e(2, row, lx + GX), ld2(e1.at(0, row, lx)),
                 ld2(e1.at(1, row, lx)), row0(cls), row1(cls), hx, hy);
    }
    st2(own + (hb ^ 1) * (3 * HNEW_PLANE), hx);
    st2(own + (hb ^ 1) * (3 * HNEW_PLANE) + HNEW_PLANE, hy);
    C.arrive(C.emptyE(R.e));
    C.arrive(C.emptyH(R.h));
    R.pass_e();
    R.pass_h();
#pragma unroll 1
    for (int k = it.ka; k < it.kb; ++k) {
        ok = ok && C.wait_plane(R);
        if (!ok) *C.abort = 1;
        const EView ek = C.ev(R.e), ek1 = C.ev(R.e_next());
        const HView hk = C.hv(R.h);
        const PlaneX P{hk.psi(), (L & LZ) ? slab_of(k, a.nz, d) : -1, row * HBX + lx,
                       OFF_ZE / 4 + (row - 1) * TX + gx, C.xc + gx};
        const long long pl = k * a.plane, n = a.plane * a.nz;
        float *const cur = own + hb * (3 * HNEW_PLANE), *const old = own + (hb ^ 1) * (3 * HNEW_PLANE);
        F2 ex, ey, ez;
        uint32_t cls = 0;
        if (ok) {
            ex = ld2(ek.at(0, row, lx));
            ey = ld2(ek.at(1, row, lx));
            ez = ld2(ek.at(2, row, lx));
            cls = hk.cls2(row, clx);
            hx = ld2(hk.at(0, row, lx));
            hy = ld2(hk.at(1, row, lx));
            hz = ld2(hk.at(2, row, lx));
            h_corex<L>(a, G, P, C.prof, k, ex, ey, ez, ld2(ek.at(0, row + 1, lx)), ld2(ek.at(2, row + 1, lx)),
                       ek.e(1, row, lx + GX), ek.e(2, row, lx + GX), ld2(ek1.at(0, row, lx)),
                       ld2(ek1.at(1, row, lx)), row0(cls), row1(cls), hx, hy, hz);
            st2(cur, hx);
            st2(cur + HNEW_PLANE, hy);
            st2(cur + 2 * HNEW_PLANE, hz);
        }
        consumer_sync();            // H^{n+1/2} of plane k complete (tile + halo)
        C.arrive(C.emptyE(R.e));    // E(k) is not read again
        if (ok) {
            put2(a.Hout[0], pl, G.off, hx, G.fl & IN0, n, 1, a.bounds);
            put2(a.Hout[1], pl, G.off, hy, G.fl & IN0, n, 1, a.bounds);
            put2(a.Hout[2], pl, G.off, hz, G.fl & IN0, n, 1, a.bounds);
            e_corex<L>(a, G, P, C.prof, k, hx, hy, hz, ld2(cur + 2 * HNEW_PLANE - HBX), ld2(cur - HBX),
                       cur[2 * HNEW_PLANE - 1], cur[HNEW_PLANE - 1], ld2(old), ld2(old + HNEW_PLANE), row0(cls),
                       row1(cls), ex, ey, ez);
            put2(a.Eout[0], pl, G.off, ex, G.fl & IN0, n, 2, a.bounds);
            put2(a.Eout[1], pl, G.off, ey, G.fl & IN0, n, 2, a.bounds);
            put2(a.Eout[2], pl, G.off, ez, G.fl & IN0, n, 2, a.bounds);
        }
        C.arrive(C.emptyH(R.h));    // this warp is done with plane k's H slot
        R.pass_e();
        R.pass_h();
        hb ^= 1u;
    }
    C.arrive(C.emptyE(R.e));        // plane kb (E only)
    R.pass_e();
}

// The same item in a halo warp: H^{n+1/2} of the low-y row, cells (i, y0-1),
// or of the low-x column, cells (x0-1, y0+lane), of every plane, recomputed
// into the shared H planes.
template <bool CPML, int NH>
__device__ __forceinline__ void run_halo(const Cons<NH> &C, const Item &it, Ring<NH> &R, uint32_t &hb)
{
    const StepArgs &a = *C.a;
    const int lane = C.lane, d = a.d;
    Stg tb(0, 0, 0);
    if (CPML) tb.f = tile_boxes(a, it.x0, it.y0, tb.xs, tb.ys);
    const bool low_y = C.warp == NCW;
    const int row = low_y ? 0 : 1 + lane, col = low_y ? XO + lane : XO - 1;
    const int i = low_y ? it.x0 + lane : it.x0 - 1, j = low_y ? it.y0 - 1 : it.y0 + lane;
    const bool act = low_y || lane < TY;
    const bool in = act && i >= 0 && j >= 0 && i < a.nx && j < a.ny;
    int sx = -1, sy = -1, xo = -1, yo = -1;
    if (CPML && in) {
        sx = slab_of(i, a.nx, d);
        sy = slab_of(j, a.ny, d);
        if (tb.f & F_X) xo = x_off(a, tb, i, row);
        if (tb.f & F_Y) yo = y_off(a, tb, it.x0, i, j);
    }
    C.arrive(C.emptyE(R.e));        // the plane below the item has no halo
    C.arrive(C.emptyH(R.h));
    R.pass_e();
    R.pass_h();
    bool ok = true;
#pragma unroll 1
    for (int k = it.ka; k < it.kb; ++k) {
        ok = ok && C.wait_plane(R);
        if (!ok) *C.abort = 1;
        if (ok && act) {
            const EView ek = C.ev(R.e), ek1 = C.ev(R.e_next());
            const HView hk = C.hv(R.h);
            float hx = 0.f, hy = 0.f, hz = 0.f;
            if (in) {
                const Slab L = CPML ? slab_in(Stg(ek.hdr()), hk, sx, sy, slab_of(k, a.nz, d), xo, yo, row * HBX + col)
                                    : Slab{-1, -1, -1, nullptr, -1, -1, -1};
                h_core<CPML>(a, C.coef(hk.cls(row, col - XO + CXO)), C.prof, L, ek.e(0, row, col), ek.e(1, row, col),
                             ek.e(2, row, col), ek.e(1, row, col + 1), ek.e(2, row, col + 1), ek.e(0, row + 1, col),
                             ek.e(2, row + 1, col), ek1.e(0, row, col), ek1.e(1, row, col), hk.h(0, row, col),
                             hk.h(1, row, col), hk.h(2, row, col), hx, hy, hz);
            }
            *C.hn(hb, 0, row, col) = hx;
            *C.hn(hb, 1, row, col) = hy;
            *C.hn(hb, 2, row, col) = hz;
        }
        C.arrive(C.emptyH(R.h));    // a halo warp reads the slot in the H half step only
        consumer_sync();            // H^{n+1/2} of plane k complete (tile + halo)
        C.arrive(C.emptyE(R.e));    // E(k) is not read again
        R.pass_e();
        R.pass_h();
        hb ^= 1u;
    }
    C.arrive(C.emptyE(R.e));        // plane kb (E only)
    R.pass_e();
}

// the x-layer coefficients of an item's columns, one value per consumer thread
__device__ __forceinline__ void fill_xc(const StepArgs &a, const float *prof, float *xc, int x0, int tid)
{
    for (int q = tid; q < 6 * TX; q += NCONS) {
        const int w = q / TX, i = x0 + q - w * TX, half = w / 3, comp = w - 3 * half;
        const int s = i < a.nx ? slab_of(i, a.nx, a.d) : -1;
        xc[q] = s >= 0 ? prof[((half * 2 * a.d + s) << 2) + comp] : 0.f;
    }
}

// domain of global work item q: item_start[d] <= q < item_start[d + 1]
__device__ __forceinline__ int find_domain(const int *item_start, int n, int q)
{
    int lo = 0, hi = n - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (__ldg(item_start + mid) <= q) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

// the items of a consumer warp, in the order the producer hands them out
template <bool ROWS, bool ZL, int NH, bool BATCH>
__device__ __forceinline__ void consume(const Cons<NH> &C, const BatchArgs &B, StepArgs *sa, int *cons_e, int *cons_h)
{
    Ring<NH> R;
    uint32_t ce = 0, ch = 0, hb = 0;    // planes of the items before the current one
    uint32_t item_e = 0;                // E planes of the current item
    int cur = -1;                   // domain whose arguments are staged
    const int tid = threadIdx.x;
    while (true) {
        // first plane of the next item (or the end marker)
        if (!mbar_wait(C.fullE(R.e), R.ep, C.abort)) *C.abort = 1;
        if (consumer_any(*C.abort != 0)) break;
        ce += item_e;
        ch += max(item_e, 1u) - 1;
        const int *hdr = C.ev(R.e).hdr();
        const int item = hdr[0], dom = hdr[5];
        if (item < 0) break;
        if (BATCH && dom != cur) {
            // stage this domain's image -- its arguments, coefficient
            // table rows and CPML profile rows, which the host laid out
            // exactly as their shared-memory copy -- in one round of
            // independent 16-byte loads
            const int2 ref = __ldg(B.img_ref + (dom * 2 + B.launch) * 2 + B.parity);
            const int4 *src = B.img + ref.x;
            int4 *dst = reinterpret_cast<int4 *>(sa);
            for (int q = tid; q < ref.y; q += NCONS) dst[q] = __ldg(src + q);
            cur = dom;
            consumer_sync();
        }
        const StepArgs &a = *C.a;
        const Item it = uniform(Item{hdr[6], hdr[7], hdr[8], hdr[9]});
        const bool layer = item_in_cpml(a, it);
        if (layer) fill_xc(a, C.prof, C.xc, it.x0, tid);
        const uint32_t n = R.e_next();
        if (!mbar_wait(C.fullE(n), R.ep ^ (n == 0), C.abort)) *C.abort = 1;
        if (consumer_any(*C.abort != 0)) break;
        if constexpr (ROWS) {
            // the layers its own cells meet (its planes: all or none of them)
            const int d = a.d;
            const bool lx = d > 0 && (it.x0 < d || min(it.x0 + TX, a.nx) > a.nx - d);
            const bool ly = d > 0 && (it.y0 < d || min(it.y0 + TY, a.ny) > a.ny - d);
            constexpr int Z = ZL ? LZ : 0;
            const bool vec = ((d | a.nx) & 1) == 0;
            if (lx && ly) {
                if (vec) run_rows<LX | LY | Z, NH>(C, it, R, hb);
                else run_rows<LXS | LY | Z, NH>(C, it, R, hb);
            } else if (lx) {
                if (vec) run_rows<LX | Z, NH>(C, it, R, hb);
                else run_rows<LXS | Z, NH>(C, it, R, hb);
            } else if (ly) {
                run_rows<LY | Z, NH>(C, it, R, hb);
            } else {
                run_rows<Z, NH>(C, it, R, hb);
            }
        } else {
            if (layer) run_halo<true, NH>(C, it, R, hb);
            else run_halo<false, NH>(C, it, R, hb);
        }
        if (!BATCH && a.n_isrc > 0) {
            // current sources on the item's edges, after all its E stores
            const uint32_t m = item_sources(a, B.launch, item);
            if (m) {
                consumer_sync();
                if (ROWS && tid == 0) add_sources(a, m);
            }
        }
        item_e = (uint32_t)(it.kb - it.ka) + 2;
    }
    if (ROWS && tid == 0) {
        *cons_e = (int)ce;
        *cons_h = (int)ch;
    }
}

// BATCH = false: one domain whose arguments and descriptors are the kernel's
// own parameters (constant bank); BATCH = true: a table of domains in global
// memory, the current domain's arguments staged in shared memory.
template <bool ZL, int NH, bool BATCH>
__global__ void __launch_bounds__(NTHREADS, 2) step_tma_kernel(const __grid_constant__ SingleArgs S,
                                                              const BatchArgs B)
{
    extern __shared__ __align__(128) char smem_raw[];
    // TMA destinations are kept 128-byte aligned
    char *smem = smem_raw + ((128u - (smem_u32(smem_raw) & 127u)) & 127u);
    const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    const Layout Lo(B.region, NH);
    StepArgs *sa = reinterpret_cast<StepArgs *>(smem + Lo.tab);          // current domain's arguments
    float *tab = reinterpret_cast<float *>(smem + Lo.tab + al128(sizeof(StepArgs)));
    float *prof = tab + B.max_classes * kTabStride;  // [axis][E, H][2d] x {b, c, 1/kappa, -}, slab entries only
    float *hnew = reinterpret_cast<float *>(smem + Lo.hnew);
    float *xc = reinterpret_cast<float *>(smem + Lo.xc);
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + Lo.bar);
    volatile int *abort = reinterpret_cast<volatile int *>(smem + Lo.misc);
    int *cons_e = reinterpret_cast<int *>(smem + Lo.misc + 4);
    int *cons_h = reinterpret_cast<int *>(smem + Lo.misc + 8);
    int *iss_e = reinterpret_cast<int *>(smem + Lo.misc + 12);
    int *iss_h = reinterpret_cast<int *>(smem + Lo.misc + 16);
    Cons<NH> C{BATCH ? sa : &S.a, smem, tab, prof, hnew, xc, bars, abort, warp, lane, Lo.hslot};

    if (!BATCH) {
        // the one domain's coefficient table and CPML profiles, once
        const StepArgs &ga = S.a;
        for (int q = threadIdx.x; q < ga.n_classes * kTabStride; q += NTHREADS) {
            const int cl = q / kTabStride, src = tab_src(q - cl * kTabStride);
            tab[q] = src < 0 ? 0.f : __ldg(ga.table + cl * kNumCoef + src);
        }
        if (ga.d > 0) {
            const int d2 = 2 * ga.d, per = PR_COUNT * d2;
            for (int q = threadIdx.x; q < 3 * per; q += NTHREADS) {
                const int u = q / per, w = (q - u * per) / d2, sl = q - u * per - w * d2;
                const int n = u == 0 ? ga.nx : (u == 1 ? ga.ny : ga.nz);
                const int i = sl < ga.d ? sl : n - d2 + sl;
                prof[(((u * 2 + w / 3) * d2 + sl) << 2) + w % 3] = __ldg(ga.prof[u] + w * n + i);
            }
        }
    }
    if (threadIdx.x < 12) xc[6 * TX + threadIdx.x] = 0.f;
    if (threadIdx.x == 0) {
        for (int q = 0; q < NE; ++q) {
            mbar_init(C.fullE(q), 1);
            mbar_init(C.emptyE(q), NCW + NHW);
        }
        for (int q = 0; q < NH; ++q) {
            mbar_init(C.fullH(q), 1);
            mbar_init(C.emptyH(q), NCW + NHW);
        }
        *abort = 0;
        *cons_e = *cons_h = *iss_e = *iss_h = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();

    if (warp >= NCW) asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(aux_regs(BATCH)));
    if (warp >= NCW + NHW) {
        // ------------------------------ producer ------------------------------
        // The whole warp runs the loop, every value the same in all lanes
        // (item numbers come from lane 0 by shuffle), and one elected lane
        // issues the copies: addresses and coordinates stay in uniform
        // registers.  A plane's copies are few, one per kind of array, and
        // H(z) goes with E(z + 1): the consumers need both to start plane z.
        if (warp == NCW + NHW) {
            uint32_t qe = 0, qh = 0, se = 0, sh = 0, pe = 1, ph = 1;   // planes issued, slots, empty phases
            bool ok = true;
            auto wait = [&](uint32_t bar, uint32_t parity) {
                return __all_sync(0xffffffffu, mbar_wait(bar, parity, abort));
            };
            auto next_e = [&]() {
                ++qe;
                se = (se + 1) % NE;
                pe ^= se == 0;
            };
            // The CTA's first item is its own number (the grid has no more
            // CTAs than items), the counter hands out the ones after those:
            // nothing has to travel before the first copies but the wait for
            // the step before, and that comes when all else is ready.
            int next = blockIdx.x;
            bool first = true;
            while (ok) {
                const int gitem = __shfl_sync(0xffffffffu, next, 0);
                if (gitem >= B.nitems) break;
                const int dom = BATCH ? find_domain(B.item_start, B.n_domains, gitem) : 0;
                const StepArgs &a = BATCH ? B.doms[dom].a[B.launch][B.parity] : S.a;
                const TmaMaps &m = BATCH ? B.doms[dom].m[B.parity] : S.m;
                const int item = BATCH ? gitem - __ldg(B.item_start + dom) : gitem;
                const Item it = uniform(decode(a, item));
                const int nz = a.nz, d = a.d, ox = a.ox, oy = a.oy;
                // x / y boxes of the tile, and what they add to a plane
                int fxy = 0, xs = 0, ys = 0;
                if (d > 0) fxy = tile_boxes(a, it.x0, it.y0, xs, ys);
                const uint32_t tx_xy = ((fxy & F_X) ? 4u * a.pg.w * HBY * 4 : 0u) +
                                       ((fxy & F_Y) ? 4u * HBX * a.pg.hy * 4 : 0u);
                const bool zxy = a.zxy;
                // plane z's layers and E boxes; f: its staged-layer flags
                auto flags = [&](int z) {
                    if (d == 0 || z < 0 || z >= nz) return 0;
                    const bool zs = z < d || z >= nz - d;
                    return zs ? F_Z | (zxy ? fxy : 0) : fxy;
                };
                auto load_e = [&](int z) {
                    char *es = smem + SM_EH + se * ESLOT;
                    if (elect_one()) {
                        int *hdr = reinterpret_cast<int *>(es + OFF_HDR);
                        hdr[0] = item;
                        hdr[2] = flags(z);
                        hdr[3] = xs;
                        hdr[4] = ys;
                        hdr[5] = dom;
                        hdr[6] = it.x0;
                        hdr[7] = it.y0;
                        hdr[8] = it.ka;
                        hdr[9] = it.kb;
                        mbar_expect_tx(C.fullE(se), TX_E);
                        tma_load(smem_u32(es), &m.e, it.x0 - XO, it.y0 - 1, z, C.fullE(se));
                    }
                    __syncwarp();
                    next_e();
                };
                if (first) step_chain();
                first = false;
                if (!wait(C.emptyE(se), pe)) { ok = false; break; }
                load_e(it.ka - 1);
                for (int z = it.ka - 1; z < it.kb; ++z) {
                    if (!wait(C.emptyH(sh), ph) || !wait(C.emptyE(se), pe)) { ok = false; break; }
                    const int f = flags(z);
                    char *hs = smem + SM_HH + sh * Lo.hslot, *ps = hs + OFF_PSI;
                    const uint32_t fb = C.fullH(sh);
                    if (elect_one()) {
                        mbar_expect_tx(fb, TX_H + ((f & F_Z) ? TX_Z : 0u) + ((f & (F_X | F_Y)) ? tx_xy : 0u));
                        tma_load(smem_u32(hs + OFF_H), &m.h, it.x0 - XO, it.y0 - 1, z, fb);
                        tma_load(smem_u32(hs + OFF_C), &m.c, it.x0 - CXO, it.y0 - 1, z, fb);
                        if (f & F_Z) {
                            const int sz = z < d ? z : z - (nz - 2 * d);     // plane of the compact z arrays
                            tma_load(smem_u32(ps), &m.zh, it.x0 - XO, it.y0 - 1, sz, fb);
                            tma_load(smem_u32(ps + OFF_ZE), &m.ze, it.x0, it.y0, sz, fb);
                        }
                        if (f & F_X) tma_load(smem_u32(ps + ox), &m.x, xs, it.y0 - 1, z, fb);
                        if (f & F_Y) tma_load(smem_u32(ps + oy), &m.y, it.x0 - XO, ys, z, fb);
                    }
                    __syncwarp();
                    ++qh;
                    sh = sh + 1 == NH ? 0 : sh + 1;
                    ph ^= sh == 0;
                    load_e(z + 1);
                    // the next item's number travels while this one's last planes are issued
                    if (z == max(it.ka - 1, it.kb - 3) && lane == 0) next = gridDim.x + atomicAdd(B.work, 1);
                }
            }
            if (ok) {
                // end marker: an E slot whose header carries item -1
                if (wait(C.emptyE(se), pe)) {
                    if (elect_one()) {
                        int *hdr = reinterpret_cast<int *>(smem + SM_EH + se * ESLOT + OFF_HDR);
                        hdr[0] = -1;
                        hdr[2] = 0;
                        hdr[5] = -1;
                        mbar_arrive(C.fullE(se));
                    }
                    __syncwarp();
                    next_e();
                } else {
                    ok = false;
                }
            }
            if (lane == 0) {
                if (!ok) {
                    *abort = 1;
                    atomicExch(B.err, 1);
                }
                *iss_e = (int)qe;
                *iss_h = (int)qh;
                // the last CTA to finish handing out work resets the counters
                __threadfence();
                if (atomicAdd(B.work + 1, 1) == (int)gridDim.x - 1) {
                    B.work[0] = 0;
                    B.work[1] = 0;
                    __threadfence();
                }
            }
        }
    } else if (warp >= NCW) {
        consume<false, ZL, NH, BATCH>(C, B, sa, cons_e, cons_h);
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(row_regs(BATCH)));
        consume<true, ZL, NH, BATCH>(C, B, sa, cons_e, cons_h);
    }
    __syncthreads();
    // on an abort, wait (bounded) for copies still in flight before the
    // shared memory is given back
    if (threadIdx.x == 0 && *abort) {
        atomicExch(B.err, 1);
        const unsigned long long t0 = gtimer();
        for (int q = *cons_e; q < *iss_e; ++q)
            while (!mbar_try(C.fullE(q % NE), (q / NE) & 1))
                if (gtimer() - t0 > kWaitNs) break;
        for (int q = *cons_h; q < *iss_h; ++q)
            while (!mbar_try(C.fullH(q % NH), (q / NH) & 1))
                if (gtimer() - t0 > kWaitNs) break;
    }
}

}  // namespace

int step_tile_x() { return TX; }
int step_tile_y() { return TY; }
int step_threads() { return NTHREADS; }
int step_smem_bytes(int n_classes, int d, int region, int nh) { return smem_bytes(n_classes, d, region, nh); }
int step_tab_offset() { return al128(sizeof(StepArgs)); }

PsiGeom step_psi_geom(int d, int nx, int ny)
{
    PsiGeom pg{};
    if (d == 0) return pg;
    // the x (y) box of a tile spans the slab entries of the layer cells
    // among x0-1 .. x0+TX-1 (y0-1 .. y0+TY-1), from the first (rounded down
    // to a multiple of 4 along x) to the last: the largest span over the tiles
    auto slab = [d](int i, int n) { return i < d ? i : (i >= n - d ? i - (n - 2 * d) : -1); };
    int w = 0, hy = 0;
    for (int x0 = 0; x0 < nx; x0 += TX) {
        const int xl = std::max(x0 - 1, 0), xh = std::min(x0 + TX, nx) - 1;
        if (!(xl < d || xh >= nx - d)) continue;
        const int first = slab(xl < d ? xl : std::max(xl, nx - d), nx) & ~3;
        const int last = slab(xh >= nx - d ? xh : std::min(xh, d - 1), nx);
        w = std::max(w, (last - first + 1 + 3) / 4 * 4);
    }
    for (int y0 = 0; y0 < ny; y0 += TY) {
        const int yl = std::max(y0 - 1, 0), yh = std::min(y0 + TY, ny) - 1;
        if (!(yl < d || yh >= ny - d)) continue;
        const int first = slab(yl < d ? yl : std::max(yl, ny - d), ny);
        const int last = slab(yh >= ny - d ? yh : std::min(yh, d - 1), ny);
        hy = std::max(hy, last - first + 1);
    }
    pg.w = w;
    pg.hy = hy;
    pg.xb = pg.w * HBY * 4;
    pg.yb = HBX * pg.hy * 4;
    return pg;
}

void step_region(const PsiGeom &pg, int zxy, int *region, int *ox, int *oy)
{
    if (pg.w == 0) {
        *region = *ox = *oy = 0;
    } else if (zxy) {
        *ox = Z_BYTES;
        *oy = *ox + al128(4 * pg.xb);
        *region = *oy + al128(4 * pg.yb);
    } else {
        *ox = 0;
        *oy = al128(4 * pg.xb);
        *region = std::max(Z_BYTES, *oy + al128(4 * pg.yb));
    }
}
// the kernel of launch l (1: the z-layer planes)
using StepKernel = void (*)(SingleArgs, BatchArgs);
static StepKernel step_kernel(int l, int nh, bool batch)
{
    static const StepKernel k[2][2][2] = {{{step_tma_kernel<false, 2, false>, step_tma_kernel<false, 2, true>},
                                           {step_tma_kernel<false, 3, false>, step_tma_kernel<false, 3, true>}},
                                          {{step_tma_kernel<true, 2, false>, step_tma_kernel<true, 2, true>},
                                           {step_tma_kernel<true, 3, false>, step_tma_kernel<true, 3, true>}}};
    return k[l][nh == 3][batch];
}
const void *step_kernel_ptr(int l, int nh, bool batch) { return (const void *)step_kernel(l, nh, batch); }

// A launch with `regs` registers a thread holds both roles' shares: a
// setmaxnreg.inc beyond what the launch was given would wait without a limit.
static bool split_fits(int regs, bool batch)
{
    return (NCW + 4) * regs >= NCW * row_regs(batch) + 4 * aux_regs(batch);
}
cudaError_t check_step_kernel(int l, int nh, bool batch)
{
    cudaFuncAttributes at;
    const cudaError_t e = cudaFuncGetAttributes(&at, step_kernel_ptr(l, nh, batch));
    if (e != cudaSuccess) return e;
    return split_fits(at.numRegs, batch) ? cudaSuccess : cudaErrorLaunchOutOfResources;
}

cudaError_t launch_step(const SingleArgs &one, const BatchArgs &b, int grid, cudaStream_t s)
{
    const int smem = smem_bytes(b.max_classes, b.max_d, b.region, b.nh);
    step_kernel(b.launch, b.nh, b.doms != nullptr)<<<grid, NTHREADS, smem, s>>>(one, b);
    return cudaGetLastError();
}

}  // namespace fdtd

extern "C" int fdtd_selftest_wait(double seconds, void *cuda_stream)
{
    if (!(seconds > 0.0) || seconds > 10.0) return FDTD_EINVAL;
    int *flag = nullptr;
    cudaError_t e = cudaGetSymbolAddress(reinterpret_cast<void **>(&flag), fdtd::g_selftest_flag);
    cudaStream_t s = (cudaStream_t)cuda_stream;
    if (e == cudaSuccess) e = cudaMemsetAsync(flag, 0, sizeof(int), s);
    if (e == cudaSuccess) {
        fdtd::wait_selftest_kernel<<<1, 32, 0, s>>>((unsigned long long)(seconds * 1e9), flag);
        e = cudaGetLastError();
    }
    int v = 0;
    if (e == cudaSuccess) e = cudaMemcpyAsync(&v, flag, sizeof v, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return FDTD_ECUDA;
    return v == 1 ? FDTD_ETIMEOUT : (v == 2 ? FDTD_OK : FDTD_ECUDA);
}

extern "C" int fdtd_selftest_leave(int ctas, int rounds, int *spread, int *early, void *cuda_stream)
{
    if (ctas < 1 || ctas > 65535 || rounds < 1 || rounds > 1000000 || !spread || !early) return FDTD_EINVAL;
    int *out = nullptr;
    cudaError_t e = cudaGetSymbolAddress(reinterpret_cast<void **>(&out), fdtd::g_selftest_leave);
    cudaStream_t s = (cudaStream_t)cuda_stream;
    if (e == cudaSuccess) e = cudaMemsetAsync(out, 0, 2 * sizeof(int), s);
    if (e == cudaSuccess) {
        fdtd::leave_selftest_kernel<<<ctas, fdtd::NCONS + 32, 0, s>>>(rounds, out);
        e = cudaGetLastError();
    }
    int v[2] = {0, 0};
    if (e == cudaSuccess) e = cudaMemcpyAsync(v, out, sizeof v, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    *spread = v[0];
    *early = v[1];
    return e == cudaSuccess ? FDTD_OK : FDTD_ECUDA;
}

extern "C" int fdtd_selftest_registers(int regs)
{
    if (regs < 1 || regs > 255) return FDTD_EINVAL;
    return fdtd::split_fits(regs, false) && fdtd::split_fits(regs, true) ? FDTD_OK : FDTD_ECUDA;
}
