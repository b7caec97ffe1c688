// sweep_tma.cu -- FP32 fused red-black sweep fed by the Tensor Memory
// Accelerator, warp-specialised (sm_103a).
//
// Same schedule and arithmetic as k_rbgs_sweep (kernels.cu), and bitwise the
// same result: a CTA owns a 64 x 8 (or 32 x 16) tile and a chunk of planes, marches
// upward, computes the new red values of plane k (its tile plus a one-cell
// ring) and the new black values of plane k-1, out of place.  The roles are
// split over warps:
//   - warp 0, the producer: one thread issues, per plane, five tiled bulk
//     tensor copies (phi with a 2-cell halo, f and the three face-weight
//     arrays with a 1-cell halo, 15.5 KB) into a 6-stage shared-memory ring,
//     each stage guarded by a "full" mbarrier (the bytes landed) and an
//     "empty" one (every consumer warp has read it);
//   - warps 1..11, the consumers (8 row warps, 2 ring-row warps, 1
//     ring-column warp): they wait only on the full barriers, release a
//     plane's stage when its operands are in registers, and meet at one named
//     barrier per plane.
// A consumer's lane owns a pair of cells of a column.  Whatever of the column
// a step needs again stays in registers: the black values of planes k-1, k and
// k+1 (one load a plane serves the red update above it, beside it and below
// it), the z faces' weights, the black cell's f and weights (loaded with the red
// cell's as one vector), and the column's own red values.  That took the shared
// loads a row and plane from 27, all at a stride of two elements, to 13, half of
// them vectors (L1 wavefronts 59% -> 38% of peak at 256^3), and a step's black
// updates need no barrier after its red ones.  A step holds planes k and k+1,
// so four stages are copies in flight; 100 KB of shared memory and 72 registers
// give 2 CTAs (24 warps) per SM.  The CTAs are persistent: each walks tiles t,
// t + grid, .. of the launch order, and the producer runs on into the next tile,
// so a tile costs no pipeline ramp (a form whose CTAs took contiguous runs of
// tiles lost the L2 reuse of tile halos).  Per sweep, 512^3: 637 -> 555 us (86%
// of HBM on 24 bytes a cell), with the prolongation 801 -> 622 us; 256^3 96 ->
// 80 us.  With the step's code unrolled over the stages the same kernel took 30
// step bodies and waited for instructions (256^3: 113 us).
// Waits are bounded: a wait that gives up sets the error word and the
// threads go on (no consumer may leave the loop while the others meet at
// the named barrier); the producer stops issuing, and before it exits it
// waits, with the default bound, for every copy it issued.  A consumer that
// gave up says so in shared memory before it releases another stage: the plane
// there may still be landing, and a copy into it would open the next phase of
// its barrier over the one in flight.
//
// TMA rules kept: every copy starts at x = x0 - 4 (x0 a multiple of 32), a
// multiple of 4 floats = 16 bytes; rows are P floats with P a multiple of 8;
// shared destinations are 128-byte aligned; only loads use out-of-range
// (negative) coordinates, which read zeros.
#include <cuda.h>

#include <algorithm>
#include <mutex>

#include "kernels.h"

namespace mg {

namespace {

constexpr int kConsumers = kSweepTY + 3;   // 8 row warps, 2 ring-row warps, 1 ring-column warp
constexpr int kTmaThreads = 32 * (kConsumers + 1);

constexpr int pad128(int bytes) { return (bytes + 127) / 128 * 128; }
// Two red planes: a step writes plane k's and reads plane k-1's, and ends at a
// barrier.
constexpr int kRedPlanes = 2;

// A tile W cells wide and TY high (512 cells), and the staged copies under it.
template <int W>
struct Geo {
    static constexpr int TY = 512 / W;              // rows
    static constexpr int LP = W / 2;                // lanes (pairs) of a row
    static constexpr int TW = W + 8;                // staged columns x0 - 4 .. x0 + W + 3
    static constexpr int SrcRows = TY + 4;          // y0 - 2 .. y0 + TY + 1
    static constexpr int OpRows = TY + 2;           // y0 - 1 .. y0 + TY
    static constexpr int WyRows = TY + 3;           // y0 - 1 .. y0 + TY + 1 (faces)
    static constexpr int SrcBytes = SrcRows * TW * 4;
    static constexpr int OpBytes = OpRows * TW * 4;
    static constexpr int WyBytes = WyRows * TW * 4;
    static constexpr int FOff = pad128(SrcBytes);   // phi at 0
    static constexpr int WxOff = FOff + pad128(OpBytes);
    static constexpr int WyOff = WxOff + pad128(OpBytes);
    static constexpr int WzOff = WyOff + pad128(WyBytes);
    static constexpr unsigned TxBytes = SrcBytes + 3 * OpBytes + WyBytes;  // bytes landing per stage
    // With the prolongation fused (the first post-smoothing sweep): the coarse
    // correction under the phi tile, coarse columns x0/2 - 4 .. x0/2 + W/2 + 3
    // and rows y0/2 - 1 .. y0/2 + TY/2 of coarse plane p/2
    static constexpr int EcW = W / 2 + 8, EcRows = TY / 2 + 2;
    static constexpr int EcOff = WzOff + pad128(OpBytes);
    static constexpr int EcBytes = EcW * EcRows * 4;
    static constexpr int RedSW = W + 2, RedPlane = (TY + 2) * RedSW;   // a red plane, floats
    __host__ __device__ static constexpr int stage_bytes(bool prol) { return EcOff + (prol ? pad128(EcBytes) : 0); }
    __host__ __device__ static constexpr int smem_bytes(int ns, bool prol)
    {
        return ns * stage_bytes(prol) + pad128(kRedPlanes * RedPlane * 4) + 128;
    }
};

// the configuration the library launches: 6 stages, 2 CTAs (24 warps) per SM
constexpr int kStages = 6, kMinCtas = 2;

constexpr long long kWaitLimit = 1ll << 22;  // default try_wait polls before giving up

__device__ __forceinline__ unsigned smem_addr(const void *p)
{
    return (unsigned)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ void mbar_init(unsigned bar, unsigned count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count));
}

__device__ __forceinline__ void mbar_expect_tx(unsigned bar, unsigned bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes)
                 : "memory");
}

__device__ __forceinline__ void mbar_arrive(unsigned bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

__device__ __forceinline__ void named_barrier(int id, int threads)
{
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(unsigned bar, unsigned parity)
{
    unsigned ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}

// Bounded wait for phase `parity` of the barrier: at most `polls` polls;
// false if it gave up.
__device__ __forceinline__ bool mbar_wait(unsigned bar, unsigned parity, long long polls)
{
    for (long long i = 0; i < polls; ++i)
        if (mbar_try_wait(bar, parity)) return true;
    return false;
}

__device__ __forceinline__ void tma_load_3d(unsigned dst, const CUtensorMap *map, unsigned bar,
                                            int x, int y, int z)
{
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(dst),
        "l"(reinterpret_cast<unsigned long long>(map)), "r"(x), "r"(y), "r"(z), "r"(bar)
        : "memory");
}

__device__ __forceinline__ void tensormap_acquire(const CUtensorMap *map)
{
    asm volatile("fence.proxy.tensormap::generic.acquire.gpu [%0], 128;" ::"l"(
                     reinterpret_cast<unsigned long long>(map))
                 : "memory");
}

}  // namespace

// Tensor maps of one box at one level: phi, phi2, f, wx, wy, wz and the
// coarse level's phi (the correction; absent where it is not encoded), each
// 128-byte aligned, as CUtensorMap is.
struct SweepMaps {
    CUtensorMap m[7];
};

namespace {

// Red update of one cell from its staged operands (the plain sweep's FMA
// order): s = -f + sum of w x neighbour, times the correctly rounded 1/D.
__device__ __forceinline__ float red_update(float sw, float se, float ss, float sn, float sd,
                                           float su, float wxa, float wxb, float wya, float wyb,
                                           float wza, float wzb, float f)
{
    float s = fmaf(wxa, sw, -f);
    s = fmaf(wxb, se, s);
    s = fmaf(wya, ss, s);
    s = fmaf(wyb, sn, s);
    s = fmaf(wza, sd, s);
    s = fmaf(wzb, su, s);
    return s * __frcp_rn(((wxa + wxb) + (wya + wyb)) + (wza + wzb));
}

// The next stage a consumer takes and the phase its plane lands in.
template <int NS>
struct Ring {
    int s = 0;
    unsigned par = 0;
    __device__ __forceinline__ void next()
    {
        if (++s == NS) {
            s = 0;
            par ^= 1u;
        }
    }
};

// Element of the staged coarse tile under column (x, y).
template <int W>
__device__ __forceinline__ int coarse_at(int x, int y, int x0, int y0)
{
    return Geo<W>::EcOff / 4 + ((y >> 1) - (y0 >> 1) + 1) * Geo<W>::EcW + (x >> 1) - (x0 >> 1) + 4;
}

// PROL: the level's prolongation phi += e(parent) (the coarse correction,
// in the coarse level's phi) enters the sweep: each stage also holds the
// coarse tile under its plane, and a red update adds a neighbour's parent
// correction to the neighbour's staged value before using it, the FP32 sum
// the prolongation kernel would have stored.  A red update reads only black
// neighbours and a black update only the new red values, so the sweep's
// result is bitwise that of prolongation then sweep; the level's phi in
// memory stays unprolonged, which the out-of-place sweep never reads again.
template <int W, int NS, int MINB, bool PROL>
__global__ void __launch_bounds__(kTmaThreads, MINB)
    k_rbgs_sweep_tma(BoxSet<float> S, const SweepMaps *__restrict__ maps,
                     const int *__restrict__ active, int src_is_phi2, int *__restrict__ err,
                     long long polls)
{
    using G = Geo<W>;
    constexpr int STG = G::stage_bytes(PROL) / 4;   // stage stride, floats
    static_assert(NS >= 3, "planes k and k + 1 are held, another is in flight");
    constexpr int PHI = 0, FF = G::FOff / 4, WX = G::WxOff / 4, WY = G::WyOff / 4,
                  WZ = G::WzOff / 4, TW = G::TW, SW = G::RedSW, TY = G::TY, LP = G::LP;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    unsigned char *smem = reinterpret_cast<unsigned char *>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 127) & ~uintptr_t(127));
    float *const sm = reinterpret_cast<float *>(smem);
    float *const red = sm + NS * STG;
    __shared__ __align__(8) unsigned long long full[NS], empty[NS];
    __shared__ volatile int gave_up;

    const int *ts = S.tstart[TK_SWEEP];
    const int ntile = S.ntiles[TK_SWEEP];
    // t-th tile of this launch in the set's TK_SWEEP index space, taken backwards
    // when the source is phi2 (the sweep before, from phi, ran forwards and ended
    // with these tiles in L2: 64 boxes of 32 to 128 a side 15.67 -> 15.47 ms, 256^3
    // 8.44 -> 8.40, the same at 512^3);
    // the box it belongs to is skipped when it is not active
    struct Tile {
        int b, x0, y0, z0, z1;
        bool on;
    };
    auto tile_at = [&](int t) {
        Tile T;
        if (src_is_phi2) t = ntile - 1 - t;
        T.b = find_box(ts, S.nbox, t);
        const Box<float> &B = S.boxes[T.b];
        const int ntx = (B.nx + W - 1) / W, nty = (B.ny + TY - 1) / TY;
        int loc = t - ts[T.b];
        T.x0 = loc % ntx * W;
        loc /= ntx;
        T.y0 = loc % nty * TY;
        T.z0 = loc / nty * B.zc;
        T.z1 = min(T.z0 + B.zc, B.nz);
        T.on = !active || active[B.box];
        return T;
    };
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        gave_up = 0;
        for (int s = 0; s < NS; ++s) {
            mbar_init(smem_addr(&full[s]), 1);
            mbar_init(smem_addr(&empty[s]), kConsumers);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    asm volatile("griddepcontrol.wait;" ::: "memory");

    if (warp == 0) {
        // producer: the i-th plane of this CTA's tiles goes to stage i % NS;
        // from the NS-th on it waits until the consumers have released the
        // stage.  It runs on into the next tile while they finish this one.
        if (lane == 0) {
            int i = 0;
            bool ok = true;
            // the next tile of an active box
            auto next_tile = [&](int t, Tile &T) {
                for (; t < ntile; t += gridDim.x) {
                    T = tile_at(t);
                    if (T.on) break;
                }
                return t;
            };
            auto acquire = [&](int b) {
                for (int m = 0; m < (PROL ? 7 : 6); ++m) tensormap_acquire(&maps[b].m[m]);
            };
            Tile T, N;
            int t = next_tile(blockIdx.x, T), tn = t;
            if (t < ntile) acquire(T.b);
            for (; ok && t < ntile; t = tn, T = N) {
                const SweepMaps &M = maps[T.b];
                tn = -1;
                const CUtensorMap *msrc = &M.m[src_is_phi2 ? 1 : 0];
                const int x0 = T.x0, y0 = T.y0;
                for (int p = T.z0 - 2; p <= T.z1 + 1; ++p, ++i) {
                    const int s = i % NS;
                    if (p == min(T.z0 + NS - 2, T.z1 + 1)) {
                        // a ring of planes is in flight: look the next tile up
                        // and acquire its box's maps meanwhile
                        tn = next_tile(t + gridDim.x, N);
                        if (tn < ntile && N.b != T.b) acquire(N.b);
                    }
                    if (i >= NS &&
                        (!mbar_wait(smem_addr(&empty[s]), (unsigned)(((i / NS) - 1) & 1), polls) ||
                         gave_up)) {
                        atomicExch(err, 1);
                        ok = false;
                        break;
                    }
                    unsigned char *base = smem + s * (STG * 4);
                    const unsigned bar = smem_addr(&full[s]);
                    mbar_expect_tx(bar, G::TxBytes + (PROL ? G::EcBytes : 0));
                    const int zt = p + 1;  // tensor z of logical plane p (guard plane first)
                    tma_load_3d(smem_addr(base), msrc, bar, x0 - 4, y0 - 2, zt);
                    tma_load_3d(smem_addr(base + G::FOff), &M.m[2], bar, x0 - 4, y0 - 1, zt);
                    tma_load_3d(smem_addr(base + G::WxOff), &M.m[3], bar, x0 - 4, y0 - 1, zt);
                    tma_load_3d(smem_addr(base + G::WyOff), &M.m[4], bar, x0 - 4, y0 - 1, zt);
                    tma_load_3d(smem_addr(base + G::WzOff), &M.m[5], bar, x0 - 4, y0 - 1, zt);
                    // the coarse correction under plane p: coarse plane p >> 1
                    // (planes -1, -2: the coarse guard plane, zero)
                    if (PROL)
                        tma_load_3d(smem_addr(base + G::EcOff), &M.m[6], bar, x0 / 2 - 4,
                                    y0 / 2 - 1, (p >> 1) + 1);
                }
            }
            // every copy issued has landed before this thread exits (the
            // earlier planes' stages were waited on before their reuse)
            for (int q = max(0, i - NS); q < i; ++q)
                if (!mbar_wait(smem_addr(&full[q % NS]), (unsigned)((q / NS) & 1), kWaitLimit))
                    atomicExch(err, 1);
        }
        return;
    }

    // consumers
    const int cw = warp - 1;   // 0..7 row warps, 8 / 9 ring rows, 10 ring column
    Ring<NS> rg;
    long long left = polls;
    auto take = [&]() {   // the next plane's stage, once the plane has landed in it
        const int st = rg.s;
        if (!mbar_wait(smem_addr(&full[st]), rg.par, left)) {
            atomicExch(err, 1);
            gave_up = 1;
            left = 0;     // (a wait that gave up is not repeated)
        }
        rg.next();
        return st;
    };
    auto release = [&](int stage) {            // this warp has read the stage's plane
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_addr(&empty[stage]));
    };
    int r0 = 0;   // where the current plane's red values go

    if (cw < kSweepTY + 2) {
        // Rows y0 - 1 .. y0 + TY: lane owns the pair (xa, xa + 1), whose red cell
        // on plane k is at position q = (y + k) & 1.  A warp takes one row of 32
        // pairs, or rows r and r + 2 of 16, so q is uniform; the planes
        // alternate, so the loop holds a step for either q, with
        // every position a constant (unrolled over the stages as well, the row
        // kinds and parities made 30 step bodies, and the warps waited for
        // instructions).
        auto march = [&](auto own_tag) {
            constexpr bool OWN = decltype(own_tag)::value;   // row of the tile: black cells too
            const int lp = lane % LP;
            const int row = !OWN ? (cw == kSweepTY ? 0 : TY + 1)                // 0 .. TY + 1
                            : LP == 32 ? cw + 1 : (cw >> 1) * 4 + (cw & 1) + 2 * (lane / LP) + 1;
            const bool lane_on = OWN || lane < LP;           // (a ring row is one row)
            const int pa = (row + 1) * TW + 2 * lp + 4;      // phi region, of xa
            const int oa = row * TW + 2 * lp + 4;            // operand regions
            const int ra = row * SW + 2 * lp + 1;            // red plane
            for (int t = blockIdx.x; t < ntile; t += gridDim.x) {
            const Tile T = tile_at(t);
            if (!T.on) continue;
            const Box<float> &B = S.boxes[T.b];
            const int nx = B.nx, ny = B.ny, nz = B.nz, z0 = T.z0, z1 = T.z1;
            const long long Q = B.Q;
            const int y = T.y0 + row - 1, xa = T.x0 + 2 * lp;
            const bool vy = y >= 0 && y < ny;
            const bool v0 = vy && xa < nx, v1 = vy && xa + 1 < nx;
            const int ec = coarse_at<W>(xa, y, T.x0, T.y0), es = coarse_at<W>(xa, y - 1, T.x0, T.y0),
                      en = coarse_at<W>(xa, y + 1, T.x0, T.y0);
            const bool orow = OWN && y < ny;
            float *gdst = (src_is_phi2 ? B.phi : B.phi2) + (long long)(z0 - 2) * Q +
                          (long long)y * B.P + xa;           // plane k - 1
            const int q0 = (y + z0 - 1) & 1;
            // planes z0 - 2 and z0 - 1; then a step takes plane k + 1
            const int sA = take();
            int s0 = take();
            const float *const A = sm + sA * STG, *const A1 = sm + s0 * STG;
            // carried over the steps, all of this column: the black values of
            // planes k - 1 (under the red cell) and k (beside it), the z-face
            // weights of plane k; of plane k - 1 the black cell's f and weights,
            // and the red values of planes k - 1 and k - 2
            float dn = A[PHI + pa + q0], be = A1[PHI + pa + 1 - q0];
            if (PROL) {
                dn += A[ec];
                be += A1[ec];
            }
            float2 wz = *reinterpret_cast<const float2 *>(A1 + WZ + oa);
            float fB = 0.f, xB0 = 0.f, xB1 = 0.f, yB0 = 0.f, yB1 = 0.f, zB0 = 0.f;
            float r1 = 0.f, r2 = 0.f;
            release(sA);
            int k = z0 - 1;
            auto step = [&](auto q_tag) {
                constexpr int q = decltype(q_tag)::value;
                const int sP = take();
                const float *const S0 = sm + s0 * STG, *const SP = sm + sP * STG;
                float *const R0 = red + r0;
                const float *const R1 = red + (G::RedPlane - r0);
                // operands of plane k (the red cell's now, the black cell's on
                // the next step) and the black value above
                float up = SP[PHI + pa + q], outer = S0[PHI + pa + (q ? 2 : -1)],
                      so = S0[PHI + pa + q - TW], no = S0[PHI + pa + q + TW];
                if (PROL) {   // the neighbours as the prolongation leaves them
                    up += SP[ec];
                    outer += S0[ec + (q ? 1 : -1)];
                    so += S0[es];
                    no += S0[en];
                }
                float fR, x0w, x1w, y0w, y1w, z1w;   // the red cell's
                float fN = 0.f, x0n = 0.f, x1n = 0.f, y0n = 0.f, y1n = 0.f;   // the black cell's
                float2 wzn;
                if constexpr (OWN) {
                    const float2 f2 = *reinterpret_cast<const float2 *>(S0 + FF + oa);
                    const float2 wx = *reinterpret_cast<const float2 *>(S0 + WX + oa);
                    const float wx2 = S0[WX + oa + 2];
                    const float2 wy = *reinterpret_cast<const float2 *>(S0 + WY + oa);
                    const float2 wyu = *reinterpret_cast<const float2 *>(S0 + WY + oa + TW);
                    wzn = *reinterpret_cast<const float2 *>(SP + WZ + oa);
                    fR = q ? f2.y : f2.x;
                    x0w = q ? wx.y : wx.x;
                    x1w = q ? wx2 : wx.y;
                    y0w = q ? wy.y : wy.x;
                    y1w = q ? wyu.y : wyu.x;
                    fN = q ? f2.x : f2.y;
                    x0n = q ? wx.x : wx.y;
                    x1n = q ? wx.y : wx2;
                    y0n = q ? wy.x : wy.y;
                    y1n = q ? wyu.x : wyu.y;
                } else {
                    fR = S0[FF + oa + q];
                    x0w = S0[WX + oa + q];
                    x1w = S0[WX + oa + q + 1];
                    y0w = S0[WY + oa + q];
                    y1w = S0[WY + oa + q + TW];
                    wzn = *reinterpret_cast<const float2 *>(SP + WZ + oa);
                }
                z1w = q ? wzn.y : wzn.x;
                const float z0w = q ? wz.y : wz.x;   // also the black cell's upper face
                // the black neighbours of plane k - 1's black cell: red values
                // published by the barrier of the last step
                float ob = 0.f, sb = 0.f, nb = 0.f;
                if constexpr (OWN) {
                    ob = R1[ra + (q ? 2 : -1)];
                    sb = R1[ra + q - SW];
                    nb = R1[ra + q + SW];
                }
                release(s0);   // every operand is in registers
                // (1) the red value of plane k
                float val = red_update(q ? be : outer, q ? outer : be, so, no, dn, up, x0w, x1w,
                                       y0w, y1w, z0w, z1w, fR);
                val = (q ? v1 : v0) && k >= 0 && k < nz ? val : 0.f;
                if (lane_on) R0[ra + q] = val;
                // (2) the black value of plane k - 1, at the same position: its
                // neighbour in the pair and those above and below are this
                // thread's own red values
                if constexpr (OWN) {
                    const int km = k - 1;
                    if (orow && km >= z0 && km < z1) {
                        float bv = red_update(q ? r1 : ob, q ? ob : r1, sb, nb, r2, val, xB0, xB1,
                                              yB0, yB1, zB0, z0w, fB);
                        bv = (q ? v1 : v0) ? bv : 0.f;
                        if (v1) {
                            float2 o;
                            o.x = q ? r1 : bv;
                            o.y = q ? bv : r1;
                            *reinterpret_cast<float2 *>(gdst) = o;
                        } else if (v0) {
                            gdst[0] = q ? r1 : bv;
                        }
                    }
                    fB = fN;
                    xB0 = x0n;
                    xB1 = x1n;
                    yB0 = y0n;
                    yB1 = y1n;
                    zB0 = q ? wz.x : wz.y;   // plane k's lower face at its black cell
                    r2 = r1;
                    r1 = val;
                }
                dn = be;
                be = up;
                wz = wzn;
                named_barrier(1, 32 * kConsumers);
                s0 = sP;
                r0 = G::RedPlane - r0;
                gdst += Q;
                ++k;
            };
            bool second = q0 != 0;   // the first step's plane has q = 1
            while (true) {
                if (!second) {
                    step(std::integral_constant<int, 0>{});
                    if (k > z1) break;
                }
                second = false;
                step(std::integral_constant<int, 1>{});
                if (k > z1) break;
            }
            release(s0);   // plane z1 + 1
            }
        };
        if (cw < kSweepTY) march(std::true_type{});
        else march(std::false_type{});
        return;
    }

    // the ring columns x0 - 1 (the first TY / 2 lanes) and x0 + W (the next): a
    // lane owns the pair (yy, yy + 1), red at position q = (xc + y0 + k) & 1
    const bool on = lane < TY;
    const int cx = lane < TY / 2 ? -1 : W, cy = 2 * (lane % (TY / 2));
    const int pc = (cy + 2) * TW + cx + 4, oc = pc - TW, rc = (cy + 1) * SW + cx + 1;
    for (int t = blockIdx.x; t < ntile; t += gridDim.x) {
        const Tile T = tile_at(t);
        if (!T.on) continue;
        const Box<float> &B = S.boxes[T.b];
        const int nz = B.nz, z0 = T.z0, z1 = T.z1;
        const int xc = T.x0 + cx, yy = T.y0 + cy;
        const bool vx = on && xc >= 0 && xc < B.nx;
        const bool v0 = vx && yy < B.ny, v1 = vx && yy + 1 < B.ny;
        // (the parents of a pair's rows are one row of the coarse tile)
        const int ec = coarse_at<W>(xc, yy, T.x0, T.y0), ew = coarse_at<W>(xc - 1, yy, T.x0, T.y0),
                  ee = coarse_at<W>(xc + 1, yy, T.x0, T.y0);
        int q = (xc + T.y0 + z0 - 1) & 1;
        const int sA = take();
        int s0 = take();
        float dn = 0.f, be = 0.f;
        if (on) {
            const float *const A = sm + sA * STG, *const A1 = sm + s0 * STG;
            dn = A[PHI + pc + q * TW];
            be = A1[PHI + pc + (1 - q) * TW];
            if (PROL) {
                dn += A[ec];
                be += A1[ec];
            }
        }
        release(sA);
        for (int k = z0 - 1; k <= z1; ++k) {
            const int sP = take();
            const float *const S0 = sm + s0 * STG, *const SP = sm + sP * STG;
            float *const R0 = red + r0;
            if (on) {
                const int c = pc + q * TW, o = oc + q * TW;
                float up = SP[PHI + c];
                if (PROL) up += SP[ec];
                if (k >= z0 && k < z1) {
                    float we = S0[PHI + c - 1], ea = S0[PHI + c + 1],
                          out = S0[PHI + pc + (q ? 2 * TW : -TW)];
                    if (PROL) {
                        we += S0[ew];
                        ea += S0[ee];
                        out += S0[ec + (q ? G::EcW : -G::EcW)];
                    }
                    const float val =
                        red_update(we, ea, q ? be : out, q ? out : be, dn, up, S0[WX + o],
                                   S0[WX + o + 1], S0[WY + o], S0[WY + o + TW], S0[WZ + o],
                                   SP[WZ + o], S0[FF + o]);
                    R0[rc + q * SW] = (q ? v1 : v0) && k >= 0 && k < nz ? val : 0.f;
                }
                dn = be;
                be = up;
            }
            q ^= 1;
            release(s0);
            named_barrier(1, 32 * kConsumers);
            s0 = sP;
            r0 = G::RedPlane - r0;
        }
        release(s0);   // plane z1 + 1
    }
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *,
                                  const cuuint64_t *, const cuuint64_t *, const cuuint32_t *,
                                  const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encoder()
{
    static std::once_flag once;
    static EncodeTiledFn fn = nullptr;
    std::call_once(once, [] {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000,
                                             cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(p);
        cudaGetLastError();
    });
    return fn;
}

}  // namespace

template <int W>
static bool encode_maps(SweepMaps *out, int nx, int ny, int nz, const float *phi_base,
                        const float *phi2_base, const float *f_base, const float *wx_base,
                        const float *wy_base, const float *wz_base, const float *phic_base,
                        int cx, int cy, int cz)
{
    using G = Geo<W>;
    EncodeTiledFn fn = encoder();
    if (!fn) return false;
    const cuuint32_t ones[3] = {1, 1, 1};
    auto enc = [&](CUtensorMap *m, const float *base, int mx, int my, int mz,
                   const cuuint32_t *box) {
        const long long P = pitch_row(mx), Q = pitch_plane(mx, my);
        const cuuint64_t dims[3] = {(cuuint64_t)P, (cuuint64_t)(my + 1), (cuuint64_t)(mz + 2)};
        const cuuint64_t strides[2] = {(cuuint64_t)P * 4, (cuuint64_t)Q * 4};
        return fn(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, const_cast<float *>(base), dims,
                  strides, box, ones, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                  CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
    };
    const cuuint32_t box_src[3] = {G::TW, G::SrcRows, 1};
    const cuuint32_t box_op[3] = {G::TW, G::OpRows, 1};
    const cuuint32_t box_wy[3] = {G::TW, G::WyRows, 1};
    const float *base[6] = {phi_base, phi2_base, f_base, wx_base, wy_base, wz_base};
    const cuuint32_t *box[6] = {box_src, box_src, box_op, box_op, box_wy, box_op};
    for (int i = 0; i < 6; ++i)
        if (!enc(&out->m[i], base[i], nx, ny, nz, box[i])) return false;
    memset(&out->m[6], 0, sizeof(CUtensorMap));
    if (phic_base) {
        if (nx != 2 * cx || ny != 2 * cy) return false;
        const cuuint32_t box_ec[3] = {G::EcW, G::EcRows, 1};
        if (!enc(&out->m[6], phic_base, cx, cy, cz, box_ec)) return false;
    }
    return true;
}

// Encode the maps of a box level (arrays given by their allocation base =
// logical (0, 0, -1)): phi, phi2, f, wx, wy, wz, and with phic_base the
// coarse level's phi (cx x cy x cz cells) for the fused prolongation; width: of
// the tiles (64 or 32).
// Returns false if the driver cannot.
bool encode_sweep_maps(SweepMaps *out, int nx, int ny, int nz, const float *phi_base,
                       const float *phi2_base, const float *f_base, const float *wx_base,
                       const float *wy_base, const float *wz_base, const float *phic_base,
                       int cx, int cy, int cz, int width)
{
    return width == 32 ? encode_maps<32>(out, nx, ny, nz, phi_base, phi2_base, f_base, wx_base,
                                         wy_base, wz_base, phic_base, cx, cy, cz)
                       : encode_maps<64>(out, nx, ny, nz, phi_base, phi2_base, f_base, wx_base,
                                         wy_base, wz_base, phic_base, cx, cy, cz);
}

// The single-stage entry points take the fused prolongation only where the
// coarse rows and planes hold a whole 40 x 6 tile.
bool sweep_tma_prol_fits(int nx, int ny, int cx, int cy)
{
    return nx == 2 * cx && ny == 2 * cy && pitch_row(cx) >= Geo<64>::EcW && cy + 1 >= Geo<64>::EcRows;
}

size_t sweep_maps_size() { return sizeof(SweepMaps); }

// The ring's dynamic shared memory, and the largest shared-memory carveout so
// that two CTAs fit on an SM.  Function attributes are per device: they
// are set once on each device, the first time a launch or an occupancy
// query runs with that device current.
template <int W, int NS, int MINB, bool PROL>
static void set_smem_attributes()
{
    constexpr int kMaxDevices = 64;
    static std::mutex mu;
    static bool done[kMaxDevices] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) {
        cudaGetLastError();
        dev = -1;
    }
    std::lock_guard<std::mutex> lk(mu);
    if (dev >= 0 && done[dev]) return;
    cudaFuncSetAttribute(k_rbgs_sweep_tma<W, NS, MINB, PROL>,
                         cudaFuncAttributeMaxDynamicSharedMemorySize,
                         Geo<W>::smem_bytes(NS, PROL));
    cudaFuncSetAttribute(k_rbgs_sweep_tma<W, NS, MINB, PROL>,
                         cudaFuncAttributePreferredSharedMemoryCarveout,
                         cudaSharedmemCarveoutMaxShared);
    if (dev >= 0) done[dev] = true;
}

// (They also ask for rows and planes that hold a whole 72 x 12 copy box.)
bool sweep_tma_fits(int nx, int ny) { return pitch_row(nx) >= Geo<64>::TW && ny + 1 >= Geo<64>::SrcRows; }

int sweep_tma_ctas_per_sm()
{
    int n = 0;
    set_smem_attributes<64, kStages, kMinCtas, false>();
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_rbgs_sweep_tma<64, kStages, kMinCtas, false>,
                                                      kTmaThreads,
                                                      Geo<64>::smem_bytes(kStages, false)) != cudaSuccess) {
        cudaGetLastError();
        return 1;
    }
    return n > 0 ? n : 1;
}

// CTAs that fit on the current device at once.
static int resident_ctas()
{
    constexpr int kMaxDevices = 64;
    static std::mutex mu;
    static int known[kMaxDevices] = {};
    int dev = 0, sms = 1;
    if (cudaGetDevice(&dev) != cudaSuccess) dev = -1;
    std::lock_guard<std::mutex> lk(mu);
    if (dev >= 0 && dev < kMaxDevices && known[dev]) return known[dev];
    if (dev < 0 || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
        cudaGetLastError();
        return 1;
    }
    const int n = sms * sweep_tma_ctas_per_sm();
    if (dev < kMaxDevices) known[dev] = n;
    return n;
}

long long sweep_wait_polls(int wait_limit)
{
    return wait_limit == 0 ? kWaitLimit : wait_limit < 0 ? 0 : (long long)wait_limit;
}

cudaError_t launch_rbgs_sweep_tma(const BoxSet<float> &S, const SweepMaps *maps, const int *active,
                                  int src_is_phi2, int *err, cudaStream_t st, long long wait_polls,
                                  bool prolong)
{
    if (S.ntiles[TK_SWEEP] == 0) return cudaSuccess;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(std::min(S.ntiles[TK_SWEEP], resident_ctas()));
    cfg.blockDim = dim3(kTmaThreads);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = pdl_enabled() ? 1 : 0;
    auto go = [&](auto width, auto prol) {
        constexpr int W = decltype(width)::value;
        constexpr bool PR = decltype(prol)::value;
        set_smem_attributes<W, kStages, kMinCtas, PR>();
        cfg.dynamicSmemBytes = Geo<W>::smem_bytes(kStages, PR);
        return cudaLaunchKernelEx(&cfg, k_rbgs_sweep_tma<W, kStages, kMinCtas, PR>, S, maps,
                                  active, src_is_phi2, err, wait_polls);
    };
    const std::integral_constant<int, 64> w64;
    const std::integral_constant<int, 32> w32;
    if (S.sweep_w == 32) return prolong ? go(w32, std::true_type{}) : go(w32, std::false_type{});
    return prolong ? go(w64, std::true_type{}) : go(w64, std::false_type{});
}

}  // namespace mg
