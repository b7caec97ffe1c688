// kernels.cu -- CUDA kernels (sm_103a) of the multigrid Poisson solver.
//
// Operator (the library's reading of the paper's Sec. 1 variable-coefficient
// Poisson equation): with face weights w = beta_face / h^2,
//     (A phi)_c = sum over the 6 faces f of w_f (phi_nbr(f) - phi_c),
// phi_nbr = 0 outside the box (homogeneous Dirichlet wall h/2 from the
// centre, whose face weight carries 2 beta).  A Gauss-Seidel update solves
// row c for phi_c: phi_c = (sum_f w_f phi_nbr - f_c) / sum_f w_f.
//
// Every stencil is a 7-point, HBM-bound pass (no dense contraction, so no
// tensor cores); kernels are written for coalesced row access with the
// guarded level layout described in common.cuh.
#include "kernels.h"

#include "cluster.h"

#include <algorithm>
#include <cooperative_groups.h>
#include <type_traits>

#include <atomic>
#include <mutex>

namespace cg = cooperative_groups;

namespace mg {

static std::atomic<long long> g_launches{0};
long long launch_counter() { return g_launches.load(std::memory_order_relaxed); }
static inline cudaError_t counted(cudaError_t e)
{
    g_launches.fetch_add(1, std::memory_order_relaxed);
    return e;
}

// Programmatic dependent launch.  The kernels of the solve loop are launched
// with cudaLaunchAttributeProgrammaticStreamSerialization, so that a kernel's
// CTAs can be scheduled while its predecessor's last CTAs drain (the cycle is
// a chain of many short, dependent launches on the coarse levels); each such
// kernel first waits for the predecessor grid to complete and its writes to
// be visible.  The wait is a no-op in a plain launch.  MG_PDL=0 in the
// environment launches them plainly.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

bool pdl_enabled()
{
    static const bool on = [] {
        const char *v = getenv("MG_PDL");
        return !(v && v[0] == '0');
    }();
    return on;
}

template <typename... KArgs, typename... Args>
static cudaError_t pdl_launch(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem,
                              cudaStream_t st, Args... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = pdl_enabled() ? 1 : 0;
    return counted(cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...));
}

// ------------------------------------------------------------ helpers ----

template <class T>
__device__ __forceinline__ T fmadd(T a, T b, T c);
template <>
__device__ __forceinline__ double fmadd<double>(double a, double b, double c) { return fma(a, b, c); }
template <>
__device__ __forceinline__ float fmadd<float>(float a, float b, float c) { return fmaf(a, b, c); }

// Gauss-Seidel value of cell c from its six neighbours in src:
// (sum_f w_f src_nbr - f_c) / D_c, with -f_c as the start of the FMA chain
// (six FMAs and one multiply: GB300's FP64 pipe is the narrow resource).
// cf: the cell's element in f and invD (c, or its colour-split position).
template <class T>
__device__ __forceinline__ T gs_sum(const T *__restrict__ src, const T *__restrict__ f,
                                    const T *__restrict__ wx, const T *__restrict__ wy,
                                    const T *__restrict__ wz, long long c, long long cf, int P,
                                    long long Q)
{
    T s = fmadd(wx[c], src[c - 1], -f[cf]);
    s = fmadd(wx[c + 1], src[c + 1], s);
    s = fmadd(wy[c], src[c - P], s);
    s = fmadd(wy[c + P], src[c + P], s);
    s = fmadd(wz[c], src[c - Q], s);
    return fmadd(wz[c + Q], src[c + Q], s);
}

template <class T>
__device__ __forceinline__ T gs_value(const T *__restrict__ src, const T *__restrict__ f,
                                      const T *__restrict__ invD, const T *__restrict__ wx,
                                      const T *__restrict__ wy, const T *__restrict__ wz,
                                      long long c, long long cf, int P, long long Q)
{
    return gs_sum<T>(src, f, wx, wy, wz, c, cf, P, Q) * invD[cf];
}

// f_c - (A phi)_c = f_c + D_c phi_c - sum_f w_f phi_nbr, one FMA chain (seven
// FP64 operations with the stored D).  HAS_D: the diagonal comes from the
// stored D (FP64 levels: saves five FP64 adds on GB300's narrow FP64 pipe),
// else it is summed from the six weights.  It is a template parameter, and
// kernels branch on it once per box, because a run-time choice inside the
// stencil is if-converted and then pays for both sides.
template <class T, bool HAS_D>
__device__ __forceinline__ T residual_at(const T *__restrict__ phi, const T *__restrict__ f,
                                         const T *__restrict__ wx, const T *__restrict__ wy,
                                         const T *__restrict__ wz, const T *__restrict__ Dg,
                                         long long c, long long cf, int P, long long Q)
{
    T a = wx[c], b = wx[c + 1], d = wy[c], e = wy[c + P], g = wz[c], h = wz[c + Q];
    const T D = HAS_D ? Dg[cf] : ((a + b) + (d + e)) + (g + h);
    T s = fmadd(D, phi[c], f[cf]);
    s = fmadd(-a, phi[c - 1], s);
    s = fmadd(-b, phi[c + 1], s);
    s = fmadd(-d, phi[c - P], s);
    s = fmadd(-e, phi[c + P], s);
    s = fmadd(-g, phi[c - Q], s);
    return fmadd(-h, phi[c + Q], s);
}

template <class T>
struct Vec2;
template <>
struct Vec2<double> { typedef double2 type; };
template <>
struct Vec2<float> { typedef float2 type; };

// FP64 <-> FP32 conversions by integer moves of the IEEE 754 fields
// (binary64: sign, 11-bit exponent biased by 1023, 52-bit fraction;
// binary32: sign, 8-bit exponent biased by 127, 23-bit fraction).  GB300
// executes the conversion instructions on its narrow FP64 pipe, where one
// conversion costs as much as an FMA; these use the integer pipe.

// exact widening of a float in FP32's normal range (exponent field 1..254):
// exponent + (1023 - 127), the fraction's top 20 bits in the high word, its
// low 3 bits at the top of the low word
__device__ __forceinline__ double normal_f32_to_f64(float x)
{
    const unsigned b = __float_as_uint(x);
    return __hiloint2double((int)((b & 0x80000000u) | (((b & 0x7fffffffu) >> 3) + (896u << 20))),
                            (int)(b << 29));
}

// The conversion instruction for the values the integer path below leaves
// out (zero, subnormal results, overflow, infinity, NaN): a call, so that the
// compiler cannot run it under a predicate for every value, which would put
// one FP64-pipe conversion into each call of f64_to_f32_rn.
__device__ __noinline__ float f64_to_f32_by_cvt(double x) { return __double2float_rn(x); }

// the float nearest to x, ties to even (IEEE round-to-nearest)
__device__ __forceinline__ float f64_to_f32_rn(double x)
{
    const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
    const unsigned h = hi & 0x7fffffffu;
    // biased exponent 897..1150: FP32 exponent 1..254 (a round-up out of 254
    // carries into the exponent and gives infinity, as the rounding does)
    if (h - (897u << 20) >= (254u << 20)) return f64_to_f32_by_cvt(x);
    unsigned m = ((h - (896u << 20)) << 3) | (lo >> 29);   // truncated to 23 fraction bits
    const unsigned rest = lo & 0x1fffffffu;                 // the 29 bits dropped
    m += (rest > 0x10000000u || (rest == 0x10000000u && (m & 1u))) ? 1u : 0u;
    return __uint_as_float(m | (hi & 0x80000000u));
}

// 1/d in FP64 without an FP64 division, whose iterations occupy GB300's
// narrow FP64 pipe: Newton-Raphson for the reciprocal (Muller et al.,
// Handbook of Floating-Point Arithmetic, on iterations for 1/d) from an FP32
// seed.  The seed: d's fraction truncated to 23 bits (relative error below
// 2^-23) and its FP32 reciprocal by the approximate instruction (at most one
// FP32 ulp), widened exactly, both by integer moves; then d y0 = 1 - e with
// |e| < 2^-21.9, and one cubic step y = y0 (1 + e + e^2) = (1 - e^3) / d,
// e computed by a fused multiply-add, is within 2^-65 of 1/d before its one
// rounding, hence within one ulp (and nearly always the correctly rounded
// value).  A d outside 2^-125 <= |d| < 2^126 (so that the seed and its
// reciprocal are normal FP32 numbers; d = 0, inf, NaN) takes the division.
__device__ __forceinline__ double rcp64(double d)
{
    const unsigned hi = (unsigned)__double2hiint(d), lo = (unsigned)__double2loint(d);
    const unsigned h = hi & 0x7fffffffu;
    if ((h >> 20) - 898u > 250u) return 1.0 / d;   // FP32 exponent of d outside 2..252
    const float f = __uint_as_float((((h - (896u << 20)) << 3) | (lo >> 29)) | (hi & 0x80000000u));
    float s;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(s) : "f"(f));
    const double y = normal_f32_to_f64(s);   // s is normal: 2^-126 < |1/f| <= 2^125
    const double e = fma(-d, y, 1.0);
    return fma(fma(e, e, e), y, y);
}

// Tile of this CTA in a launch that runs its tiles backwards.  Consecutive
// kernels of a level alternate direction (red passes, restrictions and the
// norm pass forwards, black passes and prolongations backwards), so that each
// starts on what the one before left in L2 (126 MB; 64 boxes of 32 to 128 a side
// take 29.6 ms against 30.6 with every kernel forwards, a 256^3 solve 16.56
// against 16.8, 128^3 3.05 against 3.07; the same at 512^3, where L2 holds a
// twentieth of a pass).  Levels that L2 holds whole gain nothing and lose up to
// 0.05 us a launch (96^3 by launches 2.30 ms against 2.24).  No kernel reads what another tile of its own launch wrote.
__device__ __forceinline__ int tile_dir(bool back)
{
    return back ? (int)(gridDim.x - 1 - blockIdx.x) : (int)blockIdx.x;
}

// ---------------------------------------------- single-colour GS pass ----

// The value of a boundary cell into its copies in neighbouring guard cells.
// head: the first record of each face.
template <class T>
__device__ __forceinline__ void push_cell(const Box<T> &B, const PushRec<T> *head, int i, int j,
                                          int k, T v)
{
    auto face = [&](int f, int a, int b) {
        const PushRec<T> *R = head + f;
        while (true) {
            if (a >= R->a0 && a < R->a1 && b >= R->b0 && b < R->b1) R->dst[a * R->sa + b * R->sb] = v;
            if (R->next == 0) break;
            R = B.prec + R->next;
        }
    };
    if (i == 0) face(0, j, k);
    if (i == B.nx - 1) face(1, j, k);
    if (j == 0) face(2, i, k);
    if (j == B.ny - 1) face(3, i, k);
    if (k == 0) face(4, i, j);
    if (k == B.nz - 1) face(5, i, j);
}

// PUSH (levels with ghost exchanges): boundary cells also store their new
// value into the guard cells that copy them, so that the next stencil needs no
// exchange launch.  Safe inside the pass: it writes guard cells of its own
// colour (the colour is global over a coupled level, and a periodic axis that
// is smoothed is even) and reads those of the other.  32 coupled boxes of
// 64^3: 8 exchanges a cycle and level (10 us on the finest, 2 to 4 below)
// become 2 (3 on the finest).
template <class T, bool PUSH>
__global__ void __launch_bounds__(kThreads) k_rbgs_pass(BoxSet<T> S, const int *__restrict__ active,
                                                        int color)
{
    pdl_wait();
    const int t = tile_dir(color != 0);
    const int *ts = S.tstart[TK_PAIR];
    const int b = find_box(ts, S.nbox, t);
    const Box<T> &B = S.boxes[b];
    if (active && !active[B.box]) return;
    // the push records go through shared memory: loaded with the stencil's
    // operands, read after it, at no registers (held in registers they cost
    // the large levels a quarter in occupancy, loaded late the small ones
    // 2 us)
    __shared__ long long head[PUSH ? 6 * sizeof(PushRec<T>) / 8 : 1];
    if (PUSH) {
        const int tid = threadIdx.y * kTX + threadIdx.x;
        if (tid < (int)(6 * sizeof(PushRec<T>) / 8))
            head[tid] = reinterpret_cast<const long long *>(B.prec)[tid];
    }
    const int nx = B.nx, ny = B.ny, nz = B.nz, P = B.P;
    const long long Q = B.Q;
    TilePos p = tile_pos(TK_PAIR, nx, ny, nz, t - ts[b]);
    const int j = p.y, k = p.z;
    const int i = 2 * p.x + ((j + k + color + B.par) & 1);
    const bool in = j < ny && i < nx;
    if (!PUSH && !in) return;
    T v = T(0);
    if (in) {
        const long long c = (long long)k * Q + (long long)j * P + i;
        const long long cf =
            split_on(B) ? (long long)k * Q + (long long)j * P + (color ? (P >> 1) : 0) + p.x : c;
        v = gs_value<T>(B.phi, B.f, B.invD, B.wx, B.wy, B.wz, c, cf, P, Q);
        B.phi[c] = v;
    }
    if (PUSH) {
        __syncthreads();
        if (in) push_cell(B, reinterpret_cast<const PushRec<T> *>(head), i, j, k, v);
    }
}

// One colour out of place: dst = src with the cells of `color` updated (a
// thread per red-black pair along x, which holds one cell of each colour; the
// pair is read and written as one vector, the other cell copied).  The norm
// variant also sums r_c^2 over the updated cells, where
// r_c = D_c (phi_c - phi'_c) = f_c - (A src)_c (phi'_c solves row c) is
// the residual of src at c, formed as D_c src_c - s_c from the update's own
// sum s_c = sum_f w_f src_nbr - f_c (one extra FMA).  Right after a black
// pass the black residuals vanish, so a red pass with partials yields
// ||f - A src||^2 as a by-product (the cycle's convergence norm, taken at the
// start of the next cycle).
template <class T>
__device__ __forceinline__ void oop_pair(const Box<T> &B, int color, int from2, int j, int k,
                                         int x0, bool norm, double &r2)
{
    const int P = B.P;
    const long long Q = B.Q;
    const T *__restrict__ src = from2 ? B.phi2 : B.phi;
    T *__restrict__ dst = from2 ? B.phi : B.phi2;
    typedef typename Vec2<T>::type V2;
    const long long c0 = (long long)k * Q + (long long)j * P + x0;
    V2 pair = *reinterpret_cast<const V2 *>(src + c0);
    const int odd = (j + k + color + B.par) & 1;   // the pair's cell of this colour
    if (x0 + odd < B.nx) {
        const long long c = c0 + odd;
        const long long cf =
            split_on(B) ? (long long)k * Q + (long long)j * P + (color ? (P >> 1) : 0) + (x0 >> 1)
                        : c;
        const T sc = gs_sum<T>(src, B.f, B.wx, B.wy, B.wz, c, cf, P, Q);
        const T nv = sc * B.invD[cf];
        if (norm) {
            const T r = fmadd(B.D[cf], odd ? pair.y : pair.x, -sc);
            r2 = fma((double)r, (double)r, r2);
        }
        if (odd) pair.y = nv;
        else pair.x = nv;
    }
    *reinterpret_cast<V2 *>(dst + c0) = pair;
}

template <class T>
__global__ void __launch_bounds__(kThreads, 8) k_rbgs_pass_oop(BoxSet<T> S,
                                                               const int *__restrict__ active,
                                                               int color, int from2)
{
    pdl_wait();
    const int t = tile_dir(color != 0);
    const int *ts = S.tstart[TK_PAIR];
    const int b = find_box(ts, S.nbox, t);
    const Box<T> &B = S.boxes[b];
    if (active && !active[B.box]) return;
    TilePos p = tile_pos(TK_PAIR, B.nx, B.ny, B.nz, t - ts[b]);
    double unused = 0.0;
    if (p.y < B.ny && 2 * p.x < B.nx) oop_pair(B, color, from2, p.y, p.z, 2 * p.x, false, unused);
}

// The same pass with the residual norm: each thread takes its pair through a
// column of col_depth planes (TK_PCOLZ tiles), so the block reduction of the
// partial sums (FP64 adds and shuffles, costly on GB300's narrow FP64 pipe)
// is paid once per column instead of once per cell.
template <class T>
__global__ void __launch_bounds__(kThreads) k_rbgs_pass_oop_norm(BoxSet<T> S,
                                                                    const int *__restrict__ active,
                                                                    int color, int from2,
                                                                    double *__restrict__ partials)
{
    pdl_wait();
    const int t = blockIdx.x;
    const int *ts = S.tstart[TK_PCOLZ];
    const int b = find_box(ts, S.nbox, t);
    const Box<T> &B = S.boxes[b];
    if (active && !active[B.box]) return;
    TilePos p = tile_pos(TK_PCOLZ, B.nx, B.ny, B.nz, t - ts[b]);
    double r2 = 0.0;
    if (p.y < B.ny && 2 * p.x < B.nx) {
        const int cz = col_depth(B), z0 = p.z * cz, z1 = min(z0 + cz, B.nz);
#pragma unroll 1
        for (int k = z0; k < z1; ++k) oop_pair(B, color, from2, p.y, k, 2 * p.x, true, r2);
    }
    const double sum = block_sum(r2);
    if (threadIdx.x == 0 && threadIdx.y == 0) partials[t] = sum;
}

// -------------------------------------- fused red+black sweep (z-march) ----
//
// dst = black pass of (red pass of src), out of place.  The CTA owns a tile
// of 64 x kSweepTY columns and a chunk of zc planes; in row warp ty, lane tx
// owns the cell pair (x0 + 2tx, x0 + 2tx + 1) of row y0 + ty, which holds
// exactly one red and one black cell on every plane.  Marching k upward, step
// k computes the new red values of plane k (own columns, plus the red cells
// of a one-cell ring around the tile, recomputed by three ring warps because
// the neighbouring CTA's values are not visible) into a 4-plane shared ring
// buffer, then the new black values of plane k-1 from the red values of
// planes k-2, k-1, k, and stores both cells of the pair for plane k-1.
// Reading src and writing dst keeps every CTA's inputs unchanged while other
// CTAs run.
//
// Written for few instructions per cell (at 28 bytes a cell in FP32 the sweep
// is issue-bound before it is DRAM-bound): the ring is balanced over
// dedicated warps; every thread precomputes the offsets, shared-memory
// positions and validity of its cells for both colour parities, so a step
// only adds a plane offset; cells outside the box load from a harmless
// address and store 0 instead of branching; the march is unrolled by 4, so
// the ring-buffer slot and the parity are constants in each step; with 4
// slots one barrier per step suffices (a step writes the slot read two steps
// earlier, with a barrier between).  The black operands are loaded one step
// ahead; 56 registers keep 3 CTAs (33 warps) resident per SM.

// A red update's 13 operands and a black update's 7 global ones (its red
// neighbours come from shared memory).  The diagonal is the sum of the six
// face weights the update loads anyway, so its reciprocal is computed
// instead of read: 4 of 28 bytes a cell less in FP32 (the correctly rounded
// FP32 reciprocal), and for FP64 the set-up's rcp64, i.e. the stored 1/D.
template <class T>
struct SweepRed { T sw, se, ss, sn, sd, su, wxa, wxb, wya, wyb, wza, wzb, f; };
template <class T>
struct SweepBlack { T wxa, wxb, wya, wyb, wza, wzb, f; };

__device__ __forceinline__ float rcp_rn(float d) { return __frcp_rn(d); }
__device__ __forceinline__ double rcp_rn(double d) { return rcp64(d); }

// 1 / D from a cell's six face weights, summed in the set-up's order
template <class T>
__device__ __forceinline__ T inv_diag6(T wxa, T wxb, T wya, T wyb, T wza, T wzb)
{
    return rcp_rn(((wxa + wxb) + (wya + wyb)) + (wza + wzb));
}

template <class T>
__device__ __forceinline__ SweepRed<T> sweep_load_red(const T *__restrict__ src, const T *__restrict__ f,
                                          const T *__restrict__ wx,
                                          const T *__restrict__ wy, const T *__restrict__ wz,
                                          int c, int P, int Q)
{
    SweepRed<T> r;
    r.sw = src[c - 1]; r.se = src[c + 1]; r.ss = src[c - P]; r.sn = src[c + P];
    r.sd = src[c - Q]; r.su = src[c + Q];
    r.wxa = wx[c]; r.wxb = wx[c + 1]; r.wya = wy[c]; r.wyb = wy[c + P]; r.wza = wz[c]; r.wzb = wz[c + Q];
    r.f = f[c];
    return r;
}
template <class T>
__device__ __forceinline__ SweepBlack<T> sweep_load_black(const T *__restrict__ f,
                                            const T *__restrict__ wx, const T *__restrict__ wy,
                                            const T *__restrict__ wz, int c, int P, int Q)
{
    SweepBlack<T> b;
    b.wxa = wx[c]; b.wxb = wx[c + 1]; b.wya = wy[c]; b.wyb = wy[c + P]; b.wza = wz[c]; b.wzb = wz[c + Q];
    b.f = f[c];
    return b;
}
template <class T>
__device__ __forceinline__ T sweep_red_value(const SweepRed<T> &r)
{
    T s = fmadd(r.wxa, r.sw, -r.f);
    s = fmadd(r.wxb, r.se, s); s = fmadd(r.wya, r.ss, s); s = fmadd(r.wyb, r.sn, s);
    s = fmadd(r.wza, r.sd, s); s = fmadd(r.wzb, r.su, s);
    return s * inv_diag6(r.wxa, r.wxb, r.wya, r.wyb, r.wza, r.wzb);
}

template <class T>
__global__ void __launch_bounds__(kSweepThreads, sizeof(T) == 4 ? 3 : 1)
k_rbgs_sweep(BoxSet<T> S, const int *__restrict__ active, int src_is_phi2)
{
    pdl_wait();
    constexpr int W = 2 * kTX, SW = W + 2;            // smem row length
    constexpr int SROWS = kSweepTY + 2, SPLANE = SROWS * SW;
    __shared__ T red[4 * SPLANE];   // red values of 4 planes (slot = step % 4)
    const int t = blockIdx.x;
    const int *ts = S.tstart[TK_SWEEP];
    const int b = find_box(ts, S.nbox, t);
    const Box<T> &B = S.boxes[b];
    if (active && !active[B.box]) return;
    const int nx = B.nx, ny = B.ny, nz = B.nz, P = B.P;
    const int Q = (int)B.Q;
    const T *__restrict__ src = src_is_phi2 ? B.phi2 : B.phi;
    T *__restrict__ dst = src_is_phi2 ? B.phi : B.phi2;
    const T *__restrict__ f = B.f;
    const T *__restrict__ wx = B.wx;
    const T *__restrict__ wy = B.wy;
    const T *__restrict__ wz = B.wz;
    const int zc = B.zc;
    const TilePos tp = tile_pos(TK_SWEEP, nx, ny, nz, t - ts[b], zc);
    const int lane = threadIdx.x, wid = threadIdx.y;
    const int x0 = 2 * (tp.x - lane), y0 = tp.y - wid;
    const int z0 = tp.z * zc, z1 = min(z0 + zc, nz);
    const int kf = z0 - 1;                            // first step's plane
    const bool own = wid < kSweepTY;
    const bool colw = wid == kSweepTY + 2;
    const int xa = x0 + 2 * lane;

    // this thread's red cell at even (rE) and odd (rO) steps: plane offset 0
    // (the first step's plane), smem position, validity in x and y
    int rE, rO, sE, sO;
    bool vE, vO;
    bool ractive;        // updates a red cell at every step (own) or at steps with k in [z0, z1)
    if (!colw) {
        const int y = own ? y0 + wid : wid == kSweepTY ? y0 - 1 : y0 + kSweepTY;
        const int srow = own ? wid + 1 : wid == kSweepTY ? 0 : kSweepTY + 1;
        const int p0 = (y + kf) & 1;                  // red x parity at the first step
        const bool rowin = y >= 0 && y < ny;
        rE = kf * Q + y * P + xa + p0;
        rO = kf * Q + y * P + xa + (p0 ^ 1);
        sE = srow * SW + 2 * lane + 1 + p0;
        sO = srow * SW + 2 * lane + 1 + (p0 ^ 1);
        vE = rowin && xa + p0 < nx;
        vO = rowin && xa + (p0 ^ 1) < nx;
        ractive = true;
    } else {
        const int xc = lane < kSweepTY / 2 ? x0 - 1 : x0 + W;
        const int ym = y0 + 2 * (lane % (kSweepTY / 2));
        const int q0 = (xc + y0 + kf) & 1;            // red row offset at the first step
        const bool cin = lane < kSweepTY && xc >= 0 && xc < nx;
        rE = kf * Q + (ym + q0) * P + xc;
        rO = kf * Q + (ym + (q0 ^ 1)) * P + xc;
        sE = (ym + q0 - y0 + 1) * SW + xc - x0 + 1;
        sO = (ym + (q0 ^ 1) - y0 + 1) * SW + xc - x0 + 1;
        vE = cin && ym + q0 < ny;
        vO = cin && ym + (q0 ^ 1) < ny;
        ractive = lane < kSweepTY;
    }
    const bool ringonly = !own;
    // own rows: the black cell is the pair's other cell; pair store position
    const int yo = y0 + wid;
    const bool orow = own && yo < ny;
    const int pairo = kf * Q + yo * P + xa;           // pair base at the first step
    const bool full = xa + 1 < nx, half = xa < nx;
    const int srowo = (wid + 1) * SW;
    const int po = (yo + kf) & 1;                     // own rows' p0
    const int cE = srowo + 2 * lane + 1 + po, cO = srowo + 2 * lane + 1 + (po ^ 1);

    // first step's red operands
    SweepBlack<T> bc{};
    // step j of a block of 6 starting at plane kb (j compile-time: slot j % 3,
    // parity j & 1).  Red work at plane k = kb + j, black work at plane k - 1.
    auto step = [&](int kb, int boff, auto J) {
        constexpr int j = decltype(J)::value, s0 = j % 4, sm = (j + 3) % 4, smm = (j + 2) % 4;
        constexpr bool odd = j & 1;
        const int k = kb + j, off = boff + j * Q;
        const bool vc = (odd ? vO : vE) && k >= 0 && k < nz;
        const SweepRed<T> rc = sweep_load_red(src, f, wx, wy, wz, vc ? (odd ? rO : rE) + off : 0, P, Q);
        // this plane's black operands (used at the next step)
        const bool bv_ok = orow && k >= z0 && k < z1 && (odd ? vE : vO);
        const SweepBlack<T> bn = sweep_load_black(f, wx, wy, wz, bv_ok ? (odd ? rE : rO) + off : 0, P, Q);
        if (ractive && (!ringonly || (k >= z0 && k < z1))) {
            const bool v = (odd ? vO : vE) && k >= 0 && k < nz;
            const T val = sweep_red_value(rc);
            red[s0 * SPLANE + (odd ? sO : sE)] = v ? val : T(0);
        }
        __syncthreads();
        const int km = k - 1;
        if (orow && km >= z0) {
            // plane km had parity !odd: its red cell sits at the (odd ? E : O) position
            const int rpos = odd ? cE : cO;           // red cell of plane km
            const int lb = odd ? cO : cE;             // black cell of plane km
            const T rv = red[sm * SPLANE + rpos];
            T s = fmadd(bc.wxa, red[sm * SPLANE + lb - 1], -bc.f);
            s = fmadd(bc.wxb, red[sm * SPLANE + lb + 1], s);
            s = fmadd(bc.wya, red[sm * SPLANE + lb - SW], s);
            s = fmadd(bc.wyb, red[sm * SPLANE + lb + SW], s);
            s = fmadd(bc.wza, red[smm * SPLANE + lb], s);
            s = fmadd(bc.wzb, red[s0 * SPLANE + lb], s);
            const bool bvalid = odd ? vO : vE;        // black cell of plane km
            const T bval =
                bvalid ? s * inv_diag6(bc.wxa, bc.wxb, bc.wya, bc.wyb, bc.wza, bc.wzb) : T(0);
            const bool redfirst = (odd ? po : (po ^ 1)) == 0;  // red is the pair's first cell
            const T va = redfirst ? rv : bval, vb = redfirst ? bval : rv;
            const int c0 = pairo + off - Q;
            if (full) {
                typename Vec2<T>::type v2; v2.x = va; v2.y = vb;
                *reinterpret_cast<typename Vec2<T>::type *>(dst + c0) = v2;
            } else if (half) dst[c0] = va;
        }
        bc = bn;
    };
    for (int kb = kf, boff = 0; kb <= z1; kb += 4, boff += 4 * Q) {
        step(kb, boff, std::integral_constant<int, 0>{});
        if (kb + 1 <= z1) step(kb, boff, std::integral_constant<int, 1>{});
        if (kb + 2 <= z1) step(kb, boff, std::integral_constant<int, 2>{});
        if (kb + 3 <= z1) step(kb, boff, std::integral_constant<int, 3>{});
    }
}

// ------------------------------------------- residual + restriction ----

// The coarse right-hand side r of coarse cell (I, J, K) and the start of the
// coarse solution: 0, or (cinvD given) the coarse level's first red pass from
// 0 already applied: -r / D on its red cells (the value of the pass's FMA
// chain, whose products are all zero), which saves that pass: one of eight a
// cycle on every coarse level, 17 us on 128^3, 3 to 4 on the small ones.
// FOLD: some box of the set folds (else the test costs the register-bound FP32
// restriction a tenth).
template <class T, bool FOLD>
__device__ __forceinline__ void put_coarse(const Box<T> &B, int I, int J, int K, T r)
{
    const long long cf = cfidx(B, I, J, K);
    B.fc[cf] = r;
    B.phic[(long long)K * B.cQ + (long long)J * B.cP + I] =
        FOLD && B.cinvD && !((I + J + K + B.cpar) & 1) ? -r * B.cinvD[cf] : T(0);
}

// One coarse cell per thread, one tile of TK_COARSE: fc = mean over the 8
// children of f - A phi, phic its start.
template <class T, bool FC, bool FOLD>
__device__ __forceinline__ void restrict_tile(const BoxSet<T> &S, const int *__restrict__ active,
                                              int t)
{
    const int *ts = S.tstart[TK_COARSE];
    const int b = find_box(ts, S.nbox, t);
    const Box<T> &B = S.boxes[b];
    if (active && !active[B.box]) return;
    const int nx = B.nx, ny = B.ny, nz = B.nz, P = B.P;
    const long long Q = B.Q;
    TilePos p = tile_pos<FC>(TK_COARSE, nx, ny, nz, t - ts[b]);
    const int I = p.x, J = p.y, K = p.z;
    if (I >= nx / 2 || J >= ny / 2) return;
    auto children = [&](auto has_d) {
        constexpr bool HD = decltype(has_d)::value;
        T sum = T(0);
#pragma unroll
        for (int c = 0; c < 2; ++c)
#pragma unroll
            for (int bb = 0; bb < 2; ++bb)
#pragma unroll
                for (int a = 0; a < 2; ++a) {
                    const long long q =
                        (long long)(2 * K + c) * Q + (long long)(2 * J + bb) * P + 2 * I + a;
                    sum += residual_at<T, HD>(B.phi, B.f, B.wx, B.wy, B.wz, B.D, q,
                                              fidx(B, 2 * I + a, 2 * J + bb, 2 * K + c), P, Q);
                }
        return sum;
    };
    const T sum = B.D ? children(std::true_type{}) : children(std::false_type{});
    put_coarse<T, FOLD>(B, I, J, K, sum * T(0.125));
}

template <class T, bool FC, bool FOLD>
__global__ void __launch_bounds__(kThreads) k_resid_restrict(BoxSet<T> S, const int *__restrict__ active)
{
    pdl_wait();
    restrict_tile<T, FC, FOLD>(S, active, blockIdx.x);
}

// The red-children restriction of coarse cell (I, J, K); returns the sum of
// the squared red residuals when NORM.
template <class T, bool NORM, bool FOLD>
__device__ __forceinline__ T restrict_red_cell(const Box<T> &B, int I, int J, int K)
{
    const int P = B.P;
    const long long Q = B.Q;
    // red children of the 2x2x2 block at (2I, 2J, 2K): (a+b+c+par) even,
    // par the parity of the box's lower corner in the level's index space
    const long long o = (long long)(2 * K) * Q + (long long)(2 * J) * P + 2 * I;
    // colour-split f and D: a red child (i, j, k) of this block sits at
    // element I of row (j, k)'s red half
    const long long of = (long long)(2 * K) * Q + (long long)(2 * J) * P + I;
    T r2 = T(0);
    auto red4 = [&](auto has_d, auto odd) {
        constexpr bool HD = decltype(has_d)::value, OD = decltype(odd)::value;
        const long long c0 = OD ? o + 1 : o, c1 = OD ? o + P : o + P + 1,
                        c2 = OD ? o + Q : o + Q + 1, c3 = OD ? o + Q + P + 1 : o + Q + P;
        const bool sp = split_on(B);
        const long long f0 = sp ? of : c0, f1 = sp ? of + P : c1, f2 = sp ? of + Q : c2,
                        f3 = sp ? of + Q + P : c3;
        const T a0 = residual_at<T, HD>(B.phi, B.f, B.wx, B.wy, B.wz, B.D, c0, f0, P, Q);
        const T a1 = residual_at<T, HD>(B.phi, B.f, B.wx, B.wy, B.wz, B.D, c1, f1, P, Q);
        const T a2 = residual_at<T, HD>(B.phi, B.f, B.wx, B.wy, B.wz, B.D, c2, f2, P, Q);
        const T a3 = residual_at<T, HD>(B.phi, B.f, B.wx, B.wy, B.wz, B.D, c3, f3, P, Q);
        if (NORM) r2 = fmadd(a3, a3, fmadd(a2, a2, fmadd(a1, a1, a0 * a0)));
        return ((a0 + a1) + a2) + a3;
    };
    const T sum = B.D ? (B.par ? red4(std::true_type{}, std::true_type{})
                               : red4(std::true_type{}, std::false_type{}))
                      : (B.par ? red4(std::false_type{}, std::true_type{})
                               : red4(std::false_type{}, std::false_type{}));
    put_coarse<T, FOLD>(B, I, J, K, sum * T(0.125));
    return r2;
}

// After a red-black sweep every black cell satisfies its own equation (its
// residual is rounding-level), so right after smoothing the residual is
// carried by the red cells alone.  This variant restricts the residual of the
// 4 red children of each coarse cell (the black 4 count as zero): half the
// stencil work of k_resid_restrict, the same coarse right-hand side to
// rounding.  Valid only when the last operation on phi was a black pass.
// NORM: also each warp's sum of the squared red residuals into
// partials[t * kThreads / 32 + warp] (hence ||f - A phi||^2 of the smoothed
// iterate, summed per box in fixed order by the caller); no block barrier.
template <class T, bool FC, bool NORM, bool FOLD>
__device__ __forceinline__ void restrict_red_tile(const BoxSet<T> &S,
                                                  const int *__restrict__ active, int t,
                                                  double *__restrict__ partials = nullptr)
{
    const int *ts = S.tstart[TK_COARSE];
    const int b = find_box(ts, S.nbox, t);
    const Box<T> &B = S.boxes[b];
    if (active && !active[B.box]) return;   // the whole CTA: its box is skipped
    const int nx = B.nx, ny = B.ny, nz = B.nz, P = B.P;
    const long long Q = B.Q;
    TilePos p = tile_pos<FC>(TK_COARSE, nx, ny, nz, t - ts[b]);
    const int I = p.x, J = p.y, K = p.z;
    if (NORM) {
        // the warp's sum in T (for FP32 no FP64 adds on the narrow pipe; an
        // exit test's sum needs no more), widened once
        T r2 = T(0);
        if (I < nx / 2 && J < ny / 2) r2 = restrict_red_cell<T, NORM, FOLD>(B, I, J, K);
        for (int o = 16; o > 0; o >>= 1) r2 += __shfl_down_sync(0xffffffffu, r2, o);
        const int tid = threadIdx.y * kTX + threadIdx.x;
        if ((tid & 31) == 0) partials[(long long)t * (kThreads / 32) + (tid >> 5)] = (double)r2;
        return;
    }
    if (I >= nx / 2 || J >= ny / 2) return;
    restrict_red_cell<T, NORM, FOLD>(B, I, J, K);
}

template <class T, bool FC, bool NORM, bool FOLD>
__global__ void __launch_bounds__(kThreads) k_resid_restrict_red(BoxSet<T> S,
                                                                 const int *__restrict__ active,
                                                                 double *__restrict__ partials)
{
    pdl_wait();
    restrict_red_tile<T, FC, NORM, FOLD>(S, active, blockIdx.x, partials);
}

// --------------------------------------------------------- prolongation ----

// One thread per coarse cell: its correction is added to the 8 children (two
// rows of two planes, each child pair one vector store when nx allows).
template <class T, bool FC>
__device__ __forceinline__ void prolong_tile(const BoxSet<T> &S, const int *__restrict__ active,
                                             int t)
{
    const int *ts = S.tstart[TK_COARSE];
    const int b = find_box(ts, S.nbox, t);
    const Box<T> &B = S.boxes[b];
    if (active && !active[B.box]) return;
    TilePos p = tile_pos<FC>(TK_COARSE, B.nx, B.ny, B.nz, t - ts[b]);
    const int I = p.x, J = p.y, K = p.z;
    if (I >= B.nx / 2 || J >= B.ny / 2) return;
    const T e = B.phic[(long long)K * B.cQ + (long long)J * B.cP + I];
    const long long o = (long long)(2 * K) * B.Q + (long long)(2 * J) * B.P + 2 * I;
    typedef typename Vec2<T>::type V2;
#pragma unroll
    for (int c = 0; c < 2; ++c)
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            V2 *q = reinterpret_cast<V2 *>(B.phi + o + c * B.Q + r * B.P);
            V2 v = *q;
            v.x += e;
            v.y += e;
            *q = v;
        }
}

template <class T, bool FC>
__global__ void __launch_bounds__(kThreads) k_prolong(BoxSet<T> S, const int *__restrict__ active)
{
    pdl_wait();
    prolong_tile<T, FC>(S, active, tile_dir(true));
}

// -------------------------------------------------------- residual field ----

template <class T>
__global__ void __launch_bounds__(kThreads) k_residual_field(BoxSet<T> S)
{
    const int t = blockIdx.x;
    const int *ts = S.tstart[TK_CELL];
    const int b = find_box(ts, S.nbox, t);
    const Box<T> &B = S.boxes[b];
    TilePos p = tile_pos(TK_CELL, B.nx, B.ny, B.nz, t - ts[b]);
    if (p.x >= B.nx || p.y >= B.ny) return;
    const long long c = (long long)p.z * B.Q + (long long)p.y * B.P + p.x;
    const long long cf = fidx(B, p.x, p.y, p.z);
    B.phi2[c] = B.D ? residual_at<T, true>(B.phi, B.f, B.wx, B.wy, B.wz, B.D, c, cf, B.P, B.Q)
                    : residual_at<T, false>(B.phi, B.f, B.wx, B.wy, B.wz, B.D, c, cf, B.P, B.Q);
}

// ------------------------------------------------------------- norms ----

// mode 0: residual of every cell; 1: f; 2: residual of the red cells only
// (right after a red-black sweep), one thread per red-black pair so that no
// lane idles.  Each thread adds a column of col_depth planes.
template <class T>
__global__ void __launch_bounds__(kThreads) k_norm_partials(BoxSet<T> S, const int *__restrict__ active,
                                                            int mode, double *__restrict__ partials)
{
    pdl_wait();
    const int kind = mode == 2 ? TK_PCOLZ : TK_COLZ;
    const int t = blockIdx.x;
    const int *ts = S.tstart[kind];
    const int b = find_box(ts, S.nbox, t);
    const Box<T> &B = S.boxes[b];
    if (active && !active[B.box]) return;
    TilePos p = tile_pos(kind, B.nx, B.ny, B.nz, t - ts[b]);
    double v = 0.0;
    const int ex = mode == 2 ? (B.nx + 1) / 2 : B.nx;
    auto column = [&](auto has_d) {
        constexpr bool HD = decltype(has_d)::value;
        const int cz = col_depth(B), z0 = p.z * cz, z1 = min(z0 + cz, B.nz);
        for (int k = z0; k < z1; ++k) {
            const int x = mode == 2 ? 2 * p.x + ((p.y + k + B.par) & 1) : p.x;
            if (x >= B.nx) continue;
            const long long c = (long long)k * B.Q + (long long)p.y * B.P + x;
            const long long cf = fidx(B, x, p.y, k);
            const T r = mode == 1 ? B.f[cf]
                                  : residual_at<T, HD>(B.phi, B.f, B.wx, B.wy, B.wz, B.D, c, cf,
                                                       B.P, B.Q);
            v = fma((double)r, (double)r, v);
        }
    };
    if (p.x < ex && p.y < B.ny) {
        if (B.D) column(std::true_type{});
        else column(std::false_type{});
    }
    double s = block_sum(v);
    if (threadIdx.x == 0 && threadIdx.y == 0) partials[t] = s;
}

// Max norms for the solve's statistics (FP64 level 0): field 0 max |f|,
// field 1 max |f - A phi| with phi from phi2 for the boxes whose side flag is
// set.  Per TK_COLZ tile, then one CTA per box takes the max over its tiles.
__global__ void __launch_bounds__(kThreads) k_max_partials(BoxSet<double> S,
                                                           const int *__restrict__ side,
                                                           int field, double *__restrict__ partials)
{
    const int t = blockIdx.x;
    const int *ts = S.tstart[TK_COLZ];
    const int b = find_box(ts, S.nbox, t);
    const Box<double> &B = S.boxes[b];
    TilePos p = tile_pos(TK_COLZ, B.nx, B.ny, B.nz, t - ts[b]);
    const double *phi = (side && side[B.box]) ? B.phi2 : B.phi;
    double v = 0.0;
    if (p.x < B.nx && p.y < B.ny) {
        const int cz = col_depth(B), z0 = p.z * cz, z1 = min(z0 + cz, B.nz);
        for (int k = z0; k < z1; ++k) {
            const long long c = (long long)k * B.Q + (long long)p.y * B.P + p.x;
            const long long cf = fidx(B, p.x, p.y, k);
            const double r =
                field == 0 ? B.f[cf]
                           : residual_at<double, true>(phi, B.f, B.wx, B.wy, B.wz, B.D, c, cf,
                                                       B.P, B.Q);
            v = fmax(v, fabs(r));
        }
    }
    __shared__ double wmax[kThreads / 32];
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_down_sync(0xffffffffu, v, o));
    const int tid = threadIdx.y * kTX + threadIdx.x;
    if ((tid & 31) == 0) wmax[tid >> 5] = v;
    __syncthreads();
    if (tid == 0) {
        double m = 0.0;
        for (int w = 0; w < kThreads / 32; ++w) m = fmax(m, wmax[w]);
        partials[t] = m;
    }
}

__global__ void __launch_bounds__(1024) k_max_finish(BoxSet<double> S,
                                                     const double *__restrict__ partials,
                                                     double *__restrict__ out)
{
    __shared__ double wmax[32];
    const int b = blockIdx.x;
    const Box<double> &B = S.boxes[b];
    const int *ts = S.tstart[TK_COLZ];
    double m = 0.0;
    for (int q = ts[b] + (int)threadIdx.x; q < ts[b + 1]; q += 1024) m = fmax(m, partials[q]);
    for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_down_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0) wmax[threadIdx.x >> 5] = m;
    __syncthreads();
    if (threadIdx.x == 0) {
        double r = 0.0;
        for (int w = 0; w < 32; ++w) r = fmax(r, wmax[w]);
        out[B.box] = r;
    }
}

// One CTA of 1024 threads per box: thread q adds partials q, q + 1024, ...
// in order, then fixed shuffle trees.
template <class T>
__global__ void __launch_bounds__(1024) k_norm_finish(BoxSet<T> S, const int *__restrict__ active,
                                                      const double *__restrict__ partials,
                                                      double *__restrict__ out,
                                                      double *__restrict__ copy,
                                                      double *__restrict__ inv,
                                                      const double *__restrict__ mult,
                                                      const int *__restrict__ ts)
{
    pdl_wait();
    const int b = blockIdx.x;
    const Box<T> &B = S.boxes[b];
    if (active && !active[B.box]) return;
    const int lo = ts[b], hi = ts[b + 1];
    double s = 0.0;
    for (int q = lo + (int)threadIdx.x; q < hi; q += 1024) s += partials[q];
    const double tot = block_sum_1024(s);
    if (threadIdx.x == 0) {
        const double nrm = mult ? sqrt(tot) * mult[B.box] : sqrt(tot);
        out[B.box] = nrm;
        if (copy) copy[B.box] = nrm;
        if (inv) inv[B.box] = nrm > 0.0 ? 1.0 / nrm : 0.0;
    }
}

// ----------------------------------------------------- coarsest level ----

// Grid (nbox, row chunks of 32); 8 warps x 4 rows each.
template <class T>
__global__ void __launch_bounds__(kThreads) k_bottom(BoxSet<T> S, const int *__restrict__ active)
{
    __shared__ T fs[MG_BOTTOM_CELLS];
    const Box<T> &B = S.boxes[blockIdx.x];
    if (active && !active[B.box]) return;
    const int nx = B.nx, ny = B.ny, nz = B.nz;
    const int n = nx * ny * nz;
    const int tid = threadIdx.y * kTX + threadIdx.x;
    for (int q = tid; q < n; q += kThreads) {
        const int i = q % nx, j = (q / nx) % ny, k = q / (nx * ny);
        fs[q] = B.f[fidx(B, i, j, k)];
    }
    __syncthreads();
    const int lane = threadIdx.x, warp = threadIdx.y;
    for (int rr = 0; rr < 4; ++rr) {
        const int r = blockIdx.y * 32 + warp * 4 + rr;
        if (r >= n) break;
        const T *row = B.ainv + (long long)r * n;
        T acc = T(0);
        for (int q = lane; q < n; q += 32) acc = fmadd(row[q], fs[q], acc);
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
        if (lane == 0) {
            const int i = r % nx, j = (r / nx) % ny, k = r / (nx * ny);
            B.phi[(long long)k * B.Q + (long long)j * B.P + i] = acc;
        }
    }
}

// ------------------------------------- coarse V-cycle in one cluster per box ----
//
// Levels of a few ten thousand cells take well under a microsecond of work a
// stage, but a launch each; the coarse end of every box's V-cycle therefore
// runs inside one thread-block cluster per box, with its levels in shared
// memory from the first pass to the last: nu1 red/black passes and residual +
// restriction going down, the dense coarsest solve, then prolongation and nu2
// passes going up.  Same stage definitions and per-cell arithmetic as the
// per-level kernels (bitwise the same results).
//
// The first ndist levels are split over the cluster by planes of z (every
// level's split halves with the planes, so a fine pair of planes and its
// coarse plane sit in one CTA); a CTA's boundary planes are stored into the
// neighbour's halo plane as they are updated (distributed shared memory), and
// one cluster barrier ends each pass.  The levels below (at most kTailSolo
// cells) run in the cluster's first CTA alone, where a block barrier does.
// What bounds it: the dependent chain of about 20 stages per two levels, each
// a barrier (~0.4 us), the shared-memory latency and, in FP64, the narrow pipe
// (16 cycles an SM per warp instruction: 1.7 us for a pass over 32^3 on 16
// SMs; a chain of 7 dependent FP64 operations alone is 0.4 us).  Weights are
// loaded before the wait on the preceding kernel.  FP64, 32^3 and below: 60 us
// a cycle against 93 us as launches plus a one-CTA kernel below 16^3 that
// worked on global memory (the 64^3 solve 1.76 -> 1.51 ms).

constexpr int kTailThreads = 512;

// One level of a CTA's part, in shared memory (offsets from the host's plan).
// f, 1/D and D keep the level's colour split: hp > 0: a row holds its red
// cells, then (from hp) its black ones; hp = 0: in x order.
template <class T>
struct TailView {
    T *phi, *f;                  // phi: [np + 2][ny + 2][nx + 2]; f: [np][ny][fp]
    const T *wx, *wy, *wz;       // [np][ny][nx + 2], [np][ny + 1][nx], [np + 1][ny][nx]
    const T *inv, *dg;           // [np][ny][fp]; dg NULL: D is read from global memory
    int nx, ny, p, q, np, z0, par, fp, hp;
    int lo, hi, lo_top;          // ranks that own planes z0 - 1 and z0 + np (-1: a wall); halo plane of lo
};

// u / n for 0 <= u < 2^20, n >= 1 and rn = 1.0f / n: (u + 1/2) / n lies at
// least 1 / (2n) from an integer, further than the two FP32 roundings reach
// (an integer division is a chain of about 100 cycles, paid at every stage).
__device__ __forceinline__ int tail_div(int u, float rn) { return (int)(((float)u + 0.5f) * rn); }

// This thread's walk over [0, ex) x [0, ey) x [0, ez) in steps of the CTA.
struct TailWalk {
    int x, y, z, sx, sy, sz, ex, ey, ez;
    __device__ __forceinline__ TailWalk(int ex_, int ey_, int ez_) : ex(ex_), ey(ey_), ez(ez_)
    {
        const float rx = __frcp_rn((float)ex), ry = __frcp_rn((float)ey);
        const int u = threadIdx.x, r = tail_div(u, rx), r2 = tail_div(kTailThreads, rx);
        x = u - r * ex;
        z = tail_div(r, ry);
        y = r - z * ey;
        sx = kTailThreads - r2 * ex;
        sz = tail_div(r2, ry);
        sy = r2 - sz * ey;
    }
    template <class F>
    __device__ __forceinline__ void each(F fn) const
    {
        int a = x, b = y, c = z;
        while (c < ez) {
            fn(a, b, c);
            a += sx;
            b += sy;
            c += sz;
            if (a >= ex) { a -= ex; ++b; }
            if (b >= ey) { b -= ey; ++c; }
        }
    }
};

// N elements global -> shared (both aligned to N elements) without a register
// or a wait (tail_async_wait)
template <int N, class T>
__device__ __forceinline__ void tail_async(T *dst, const T *src)
{
    constexpr int bytes = N * (int)sizeof(T);
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(
                     (unsigned)__cvta_generic_to_shared(dst)),
                 "l"(src), "n"(bytes)
                 : "memory");
}
__device__ __forceinline__ void tail_async_wait()
{
    asm volatile("cp.async.wait_all;" ::: "memory");
}

template <class T>
__device__ __forceinline__ int tail_at(const TailView<T> &V, int i, int j, int z)
{
    return (z + 1) * V.q + (j + 1) * V.p + i + 1;
}
// element of f, 1/D and D
template <class T>
__device__ __forceinline__ int tail_fat(const TailView<T> &V, int i, int j, int z)
{
    const int r = (z * V.ny + j) * V.fp;
    return V.hp ? r + (((i + j + V.z0 + z + V.par) & 1) ? V.hp : 0) + (i >> 1) : r + i;
}

// v into the copies of cell (i, j, z): neighbouring CTAs' halo planes and, on
// periodic axes, the guard cells
template <class T>
__device__ __forceinline__ void tail_push(const cg::cluster_group &cl, const TailView<T> &V, int per,
                                          int i, int j, int z, int c, T v)
{
    if (z == 0 && V.lo >= 0)
        cl.map_shared_rank(V.phi, V.lo)[V.lo_top * V.q + (j + 1) * V.p + i + 1] = v;
    if (z == V.np - 1 && V.hi >= 0)
        cl.map_shared_rank(V.phi, V.hi)[(j + 1) * V.p + i + 1] = v;
    if (per & 1) {
        if (i == 0) V.phi[c + V.nx] = v;
        if (i == V.nx - 1) V.phi[c - V.nx] = v;
    }
    if (per & 2) {
        if (j == 0) V.phi[c + V.ny * V.p] = v;
        if (j == V.ny - 1) V.phi[c - V.ny * V.p] = v;
    }
}

template <class T>
__global__ void __launch_bounds__(kTailThreads, 1)
    k_coarse_vcycle(const CoarseJob<T> *__restrict__ jobs, const int *__restrict__ active, int nu1,
                    int nu2, int post_first)
{
    extern __shared__ __align__(16) char tail_smem[];
    __shared__ CoarseJob<T> J;
    __shared__ TailView<T> views[kMaxCoarse];
    const cg::cluster_group cl = cg::this_cluster();
    const int rank = (int)cl.block_rank(), CL = (int)cl.num_blocks();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    T *const sm = reinterpret_cast<T *>(tail_smem);
    {
        const int words = (int)(sizeof(CoarseJob<T>) / sizeof(int));
        const int *src = reinterpret_cast<const int *>(jobs + blockIdx.x / CL);
        int *dst = reinterpret_cast<int *>(&J);
        for (int w = tid; w < words; w += kTailThreads) dst[w] = src[w];
    }
    __syncthreads();
    const int nl = J.nlev, nd = J.ndist, per = J.per;
    const bool zero_start = J.zero != 0;
    if (tid < nl) {   // a thread per level
        const int l = tid;
        const Box<T> &B = J.lv[l];
        const TailLevel &L = J.tl[l];
        auto plane0 = [&](int r) {   // first plane of rank r
            return l < nd ? ((r * J.nzc) / CL) << (nd - 1 - l) : (r == 0 ? 0 : B.nz);
        };
        auto owner = [&](int k) {    // rank of plane k
            return l < nd ? (((k >> (nd - 1 - l)) + 1) * CL + J.nzc - 1) / J.nzc - 1 : 0;
        };
        TailView<T> V;
        V.nx = B.nx;
        V.ny = B.ny;
        V.p = B.nx + 2;
        V.q = V.p * (B.ny + 2);
        V.z0 = plane0(rank);
        V.np = plane0(rank + 1) - V.z0;
        V.par = B.par;
        V.hp = L.hp;
        V.fp = L.hp ? 2 * L.hp : B.nx;
        V.phi = sm + L.phi;
        V.f = sm + L.f;
        V.wx = sm + L.wx;
        V.wy = sm + L.wy;
        V.wz = sm + L.wz;
        V.inv = sm + L.inv;
        V.dg = L.dg >= 0 ? sm + L.dg : nullptr;
        V.lo = V.hi = -1;
        V.lo_top = 0;
        int kl = V.z0 - 1, kh = V.z0 + V.np;
        if (per & 4) {
            if (kl < 0) kl += B.nz;
            if (kh >= B.nz) kh -= B.nz;
        }
        if (kl >= 0) {
            V.lo = owner(kl);
            V.lo_top = plane0(V.lo + 1) - plane0(V.lo) + 1;
        }
        if (kh < B.nz) V.hi = owner(kh);
        views[l] = V;
    }
    __syncthreads();
    // the weights of this CTA's planes, before the wait: no kernel of a solve
    // writes them (pairs of elements; a level that is smoothed has even nx)
    for (int l = 0; l + 1 < nl; ++l) {
        const TailView<T> V = views[l];
        if (V.np == 0) continue;
        const Box<T> &B = J.lv[l];
        const long long g0 = (long long)V.z0 * B.Q;
        const int P = B.P, Q = (int)B.Q, h = V.nx >> 1;
        const T *const gx = B.wx + g0, *const gy = B.wy + g0, *const gz = B.wz + g0,
                *const gi = B.invD + g0, *const gd = B.D + g0;
        T *const sx = const_cast<T *>(V.wx), *const sy = const_cast<T *>(V.wy),
                 *const sz = const_cast<T *>(V.wz), *const si = const_cast<T *>(V.inv),
                 *const sd = const_cast<T *>(V.dg);
        const int hp2 = V.fp >> 1;   // (colour-split rows: the last pair of a half may be padding)
        TailWalk(h + 1, V.ny + 1, V.np + 1).each([&](int x, int j, int z) {
            const int r = z * Q + j * P, row = z * V.ny + j;
            const bool jy = j < V.ny, kz = z < V.np;
            if (jy && kz) tail_async<2>(sx + row * V.p + 2 * x, gx + r + 2 * x);
            if (x < h) {
                const int d = row * V.nx + 2 * x;
                if (kz) tail_async<2>(sy + d + z * V.nx, gy + r + 2 * x);
                if (jy) tail_async<2>(sz + d, gz + r + 2 * x);
            }
            if (x < hp2 && jy && kz) {
                const int q = r + (V.hp && 2 * x >= V.hp ? (P >> 1) + 2 * x - V.hp : 2 * x);
                tail_async<2>(si + row * V.fp + 2 * x, gi + q);
                if (sd) tail_async<2>(sd + row * V.fp + 2 * x, gd + q);
            }
        });
    }
    for (int l = 0; l < nl; ++l) {   // phi = 0, guards and halos too
        const TailView<T> V = views[l];
        constexpr int N = 16 / (int)sizeof(T);   // (the plan pads every array to 16 bytes)
        if (V.np > 0)
            for (int c = N * tid; c < (V.np + 2) * V.q; c += N * kTailThreads)
                *reinterpret_cast<float4 *>(V.phi + c) = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    if (J.ainv >= 0 && rank == 0) {
        const Box<T> &B = J.lv[nl - 1];
        const int n = B.nx * B.ny * B.nz;
        for (int q = tid; q < n * n; q += kTailThreads) tail_async<1>(sm + J.ainv + q, B.ainv + q);
    }
    pdl_wait();
    if (active && !active[J.box]) {        // uniform over the cluster
        tail_async_wait();                 // (no copy may land after the CTA has gone)
        return;
    }
    // (the zeros of one thread lie under cells that another copies)
    if (!zero_start) __syncthreads();
    {   // the first level's f (and phi unless it is 0)
        const Box<T> &B = J.lv[0];
        const TailView<T> V = views[0];
        const bool split = split_on(B);
        TailWalk(V.nx, V.ny, V.np).each([&](int i, int j, int z) {
            const long long g = (long long)(V.z0 + z) * B.Q + (long long)j * B.P;
            const int odd = (i + j + V.z0 + z + V.par) & 1;
            tail_async<1>(V.f + tail_fat(V, i, j, z),
                          B.f + g + (split ? (odd ? (B.P >> 1) : 0) + (i >> 1) : i));
            if (!zero_start) tail_async<1>(V.phi + tail_at(V, i, j, z), B.phi + g + i);
        });
    }
    tail_async_wait();
    if (nd > 0) cl.sync();   // every CTA's halos are zero before a neighbour writes them
    else __syncthreads();
    if (!zero_start) {
        const TailView<T> V = views[0];
        TailWalk(V.nx, V.ny, V.np).each([&](int i, int j, int z) {
            const int c = tail_at(V, i, j, z);
            tail_push(cl, V, per, i, j, z, c, V.phi[c]);
        });
        if (nd > 0) cl.sync();
        else __syncthreads();
    }
    // down the levels 0 .. nl - 2, the coarsest, and up again: one copy of
    // each stage's code (a stage runs a few times a launch, so that its
    // instruction fetches count)
    for (int step = 0; step < 2 * nl - 1; ++step) {
        const bool down = step < nl - 1;
        const int l = down ? step : 2 * (nl - 1) - step;
        const bool split = l < nd;
        if (!down && l == nd - 1) cl.sync();   // the first CTA's correction is there
        const TailView<T> V = views[l];
        if (l == nl - 1) {
            // the coarsest level: phi = A^{-1} f, a warp per row.  A large
            // inverse is read by every CTA of the cluster (567 cells in FP64
            // on one SM's pipe: 77 us), a part of the rows each.
            const Box<T> &B = J.lv[l];
            const int n = V.nx * V.ny * B.nz;
            const bool shared = CL > 1 && J.ainv < 0;
            if (!shared && rank != 0) continue;
            T *phi = V.phi;
            if (shared) {
                cl.sync();   // the first CTA's f is there
                if (rank != 0) {
                    const T *const f0 = cl.map_shared_rank(V.f, 0);
                    for (int q = tid; q < n; q += kTailThreads) V.f[q] = f0[q];
                    __syncthreads();
                    phi = cl.map_shared_rank(V.phi, 0);
                }
            }
            const float rx = __frcp_rn((float)V.nx), ry = __frcp_rn((float)V.ny);
            const int nw = kTailThreads / 32;
            for (int r = shared ? rank * nw + warp : warp; r < n; r += shared ? CL * nw : nw) {
                const T *row = (J.ainv >= 0 ? sm + J.ainv : B.ainv) + (long long)r * n;
                T acc = T(0);
                for (int q = lane; q < n; q += 32) acc = fmadd(row[q], V.f[q], acc);
                for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
                if (lane == 0) {
                    const int t = tail_div(r, rx), k = tail_div(t, ry);
                    phi[(k + 1) * V.q + (t - k * V.ny + 1) * V.p + r - t * V.nx + 1] = acc;
                }
            }
            if (shared) cl.sync();
            else __syncthreads();
            continue;
        }
        if (!split && rank != 0) continue;
        auto sync = [&]() {
            if (split) cl.sync();
            else __syncthreads();
        };
        const int nu = down ? nu1 : nu2, first = down ? 0 : post_first;
        const TailWalk W(V.nx >> 1, V.ny, V.np);
        if (!down) {
            // prolongation: a sweep's first pass reads only the other colour,
            // so only that colour takes the correction (both when no sweep
            // follows).  The coarse phi sits in this CTA or in the first.
            const TailView<T> C = views[l + 1];
            const bool away = l == nd - 1;
            const T *const pc = away ? cl.map_shared_rank(C.phi, 0) : C.phi;
            const int cz0 = away ? 0 : C.z0;
            W.each([&](int x, int j, int z) {
                const int k = V.z0 + z;
                const T e = pc[((k >> 1) - cz0 + 1) * C.q + ((j >> 1) + 1) * C.p + x + 1];
                for (int a = 0; a < 2; ++a) {
                    const int i = 2 * x + a;
                    if (nu2 > 0 && ((i + j + k + V.par) & 1) == post_first) continue;
                    const int c = tail_at(V, i, j, z);
                    const T v = V.phi[c] + e;
                    V.phi[c] = v;
                    tail_push(cl, V, per, i, j, z, c, v);
                }
            });
            sync();
        }
        for (int s = 0; s < 2 * nu; ++s) {
            const int color = (s & 1) ? 1 - first : first;
            // phi = 0 on entry: the first pass is -f / D (the chain's value)
            const bool zero = down && s == 0 && (zero_start || l > 0);
            W.each([&](int x, int j, int z) {
                const int i = 2 * x + ((j + V.z0 + z + color + V.par) & 1);
                const int c = tail_at(V, i, j, z);
                const int row = z * V.ny + j, d = row * V.nx + i, e = d + z * V.nx;
                const int fi = row * V.fp + (V.hp ? (color ? V.hp : 0) + x : i);
                T v = -V.f[fi];
                if (!zero) {
                    const T *const wx = V.wx + row * V.p + i;
                    v = fmadd(wx[0], V.phi[c - 1], v);
                    v = fmadd(wx[1], V.phi[c + 1], v);
                    v = fmadd(V.wy[e], V.phi[c - V.p], v);
                    v = fmadd(V.wy[e + V.nx], V.phi[c + V.p], v);
                    v = fmadd(V.wz[d], V.phi[c - V.q], v);
                    v = fmadd(V.wz[d + V.nx * V.ny], V.phi[c + V.q], v);
                }
                v *= V.inv[fi];
                V.phi[c] = v;
                tail_push(cl, V, per, i, j, z, c, v);
            });
            sync();
        }
        if (!down) continue;
        // residuals (of the red cells, or all), each in its cell's place of the
        // scratch array, then f of level l + 1 by the per-level kernel's sum.
        // The last split level's go to the first CTA: the two fine planes of a
        // coarse cell may sit in different CTAs there.
        const Box<T> &B = J.lv[l];
        const bool red = J.tl[l].red != 0, away = l == nd - 1;
        // (the first CTA may still read the scratch for the level above: with
        // pre-smoothing, a pass's barrier lies between)
        if (away && nu1 == 0 && l > 0) cl.sync();
        T *const res = away ? cl.map_shared_rank(sm + J.scratch, 0) : sm + J.scratch;
        const int kb = away ? V.z0 : 0, nr = red ? V.nx >> 1 : V.nx;
        const T *const gd = B.D;
        TailWalk(nr, V.ny, V.np).each([&](int x, int j, int z) {
            const int k = V.z0 + z;
            const int i = red ? 2 * x + ((j + k + V.par) & 1) : x;
            const int c = tail_at(V, i, j, z);
            const int row = z * V.ny + j, d = row * V.nx + i, e = d + z * V.nx;
            const int fi = tail_fat(V, i, j, z);
            const T *const wx = V.wx + row * V.p + i;
            const T a = wx[0], b = wx[1], g = V.wy[e], h = V.wy[e + V.nx], m = V.wz[d],
                    n = V.wz[d + V.nx * V.ny];
            T D;
            if (sizeof(T) == sizeof(float)) D = ((a + b) + (g + h)) + (m + n);
            else if (V.dg) D = V.dg[fi];
            else D = gd[fidx(B, i, j, k)];
            T r = fmadd(D, V.phi[c], V.f[fi]);
            r = fmadd(-a, V.phi[c - 1], r);
            r = fmadd(-b, V.phi[c + 1], r);
            r = fmadd(-g, V.phi[c - V.p], r);
            r = fmadd(-h, V.phi[c + V.p], r);
            r = fmadd(-m, V.phi[c - V.q], r);
            res[((kb + z) * V.ny + j) * nr + x] = fmadd(-n, V.phi[c + V.q], r);
        });
        if (away) cl.sync();
        else __syncthreads();
        if (!away || rank == 0) {
            const TailView<T> C = views[l + 1];
            const T *const src = sm + J.scratch;
            TailWalk(C.nx, C.ny, away ? J.lv[l + 1].nz : C.np).each([&](int I, int jc, int K) {
                const T *const r0 = src + (2 * K * V.ny + 2 * jc) * nr, *const r1 = r0 + nr,
                               *const r2 = r0 + V.ny * nr, *const r3 = r2 + nr;
                T sum;
                if (red) {
                    sum = ((r0[I] + r1[I]) + r2[I]) + r3[I];
                } else {
                    sum = T(0) + r0[2 * I];
                    sum += r0[2 * I + 1];
                    sum += r1[2 * I];
                    sum += r1[2 * I + 1];
                    sum += r2[2 * I];
                    sum += r2[2 * I + 1];
                    sum += r3[2 * I];
                    sum += r3[2 * I + 1];
                }
                C.f[tail_fat(C, I, jc, K)] = sum * T(0.125);
            });
            __syncthreads();
        }
    }
    {   // the first level's solution
        const Box<T> &B = J.lv[0];
        const TailView<T> V = views[0];
        TailWalk(V.nx, V.ny, V.np).each([&](int i, int j, int z) {
            B.phi[(long long)(V.z0 + z) * B.Q + (long long)j * B.P + i] =
                V.phi[tail_at(V, i, j, z)];
        });
    }
}

// ------------------------------------------------ mixed refinement step ----
//
// FP64 iterative refinement around FP32 V-cycles, in two passes per step:
//   k_refine_update:   x += c_e e, then e = 0   (in place, pointwise)
//   k_refine_residual: r = f - A64 x;  r32 = float(r) * float(1 / c_r);
//                      partial sums of r32^2 (FP32 per column, FP64 per CTA)
// so ||r|| = c_r * sqrt(sum r32^2).  Only the update, the residual and their
// conversions use the FP64 pipe (GB300 issues 2 FP64 FMA per SM per clock
// against 128 FP32): 11 FP64-pipe operations per cell.

__global__ void __launch_bounds__(kThreads) k_refine_update(BoxSet<double> S64, BoxSet<float> S32,
                                                            const int *__restrict__ active,
                                                            const double *__restrict__ c_e)
{
    pdl_wait();
    const int t = blockIdx.x;
    const int *ts = S64.tstart[TK_CELL];
    const int b = find_box(ts, S64.nbox, t);
    const Box<double> &B = S64.boxes[b];
    const Box<float> &E = S32.boxes[b];
    if (active && !active[B.box]) return;
    TilePos p = tile_pos(TK_CELL, B.nx, B.ny, B.nz, t - ts[b]);
    if (p.x >= B.nx || p.y >= B.ny) return;
    const long long c = (long long)p.z * B.Q + (long long)p.y * B.P + p.x;
    const float e = E.phi[c];
    B.phi[c] = fma(c_e[B.box], (double)e, B.phi[c]);
    E.phi[c] = 0.f;   // the next step's FP32 cycles start from e = 0
}

// X_ZERO: x = 0 (a zero initial guess), so r = f exactly (every product in
// the FMA chain is a signed zero): f is read instead of the stencil formed,
// with the same roundings and sums after it.
template <bool X_ZERO>
__global__ void __launch_bounds__(kThreads) k_refine_residual(BoxSet<double> S64, BoxSet<float> S32,
                                                              const int *__restrict__ active,
                                                              const double *__restrict__ c_r_inv,
                                                              double *__restrict__ partials)
{
    pdl_wait();
    const int t = blockIdx.x;
    const int *ts = S64.tstart[TK_COLZ];
    const int b = find_box(ts, S64.nbox, t);
    const Box<double> &B = S64.boxes[b];
    const Box<float> &E = S32.boxes[b];
    if (active && !active[B.box]) return;
    TilePos p = tile_pos(TK_COLZ, B.nx, B.ny, B.nz, t - ts[b]);
    float acc = 0.f;
    if (p.x < B.nx && p.y < B.ny) {
        const float cri = (float)c_r_inv[B.box];
        const int cz = col_depth(B), z0 = p.z * cz, z1 = min(z0 + cz, B.nz);
        auto column = [&](auto has_d) {
            constexpr bool HD = decltype(has_d)::value;
            for (int k = z0; k < z1; ++k) {
                const long long c = (long long)k * B.Q + (long long)p.y * B.P + p.x;
                const long long cf = fidx(B, p.x, p.y, k);
                const double r = X_ZERO ? B.f[cf]
                                        : residual_at<double, HD>(B.phi, B.f, B.wx, B.wy, B.wz,
                                                                  B.D, c, cf, B.P, B.Q);
                const float r32 = (float)r * cri;
                E.f[c] = r32;
                acc = fmaf(r32, r32, acc);
            }
        };
        if (B.D) column(std::true_type{});
        else column(std::false_type{});
    }
    double s = block_sum((double)acc);
    if (threadIdx.x == 0 && threadIdx.y == 0) partials[t] = s;
}

// The decision on box b (active) after cycle c, whose residual norm is nrm:
// true if it goes on.
__device__ __forceinline__ bool judge_box(int b, int c, double nrm,
                                          const double *__restrict__ normf,
                                          int *__restrict__ active, const JudgeState &J)
{
    if (c == 0) return true;
    const double rel = nrm / normf[b];
    if (c < MG_MAX_HIST) J.hist[(long long)b * MG_MAX_HIST + c] = rel;
    J.cycles[b] = c;
    int st = MG_ERR_NOT_CONVERGED;
    bool done = true;
    if (!isfinite(rel)) st = MG_ERR_NONFINITE;
    else if (rel <= *J.tol) st = MG_OK;
    else if (rel > 1e3 * fmax(J.rel0[b], *J.tol)) st = MG_ERR_DIVERGED;
    else {
        int stall = rel > 0.9 * J.best[b] ? J.stall[b] + 1 : 0;
        J.stall[b] = stall;
        J.best[b] = fmin(J.best[b], rel);
        done = (J.stall_limit > 0 && stall >= J.stall_limit) || c >= J.max_cycles;
    }
    J.status[b] = st;
    if (done) active[b] = 0;
    return !done;
}

// ----------------------------------------------- on-device convergence ----
//
// The same decision as the host loop, per active box, after each cycle:
// non-finite -> MG_ERR_NONFINITE; rel <= tol -> MG_OK; rel > 1e3 max(rel0,
// tol) -> MG_ERR_DIVERGED; stall_limit cycles in a row without a 10% gain
// over the best (V-cycles: 5; CG, whose residual is not monotone: no such
// rule), or max_cycles reached -> MG_ERR_NOT_CONVERGED.  A decided box is made
// inactive; the loop continues (graph condition 1) while any box is active.
// When the norm is taken at the start of the next cycle (look-ahead), the
// loop starts at step -1: the first call judges nothing (no cycle has run).
__global__ void __launch_bounds__(1024) k_judge(int nbox, const double *__restrict__ norm,
                                                const double *__restrict__ normf,
                                                int *__restrict__ active, JudgeState J,
                                                cudaGraphConditionalHandle handle, int use_handle)
{
    pdl_wait();
    __shared__ int any;
    if (threadIdx.x == 0) any = 0;
    __syncthreads();
    const int c = *J.step + 1;
    for (int b = threadIdx.x; b < nbox; b += blockDim.x)
        if (active[b] && judge_box(b, c, norm[b], normf, active, J)) any = 1;
    __syncthreads();
    if (threadIdx.x == 0) {
        *J.step = c;
        if (use_handle) cudaGraphSetConditional(handle, any ? 1u : 0u);
    }
}

// k_norm_finish and k_judge in one launch, for the loop of a single box that
// starts its cycles with the look-ahead norm: two launches of one CTA each,
// 3.4 + 2.4 us a cycle, most of it their start and end (a 64^3 solve of 13
// cycles 1.380 -> 1.365 ms).
__global__ void __launch_bounds__(1024) k_norm_judge(const double *__restrict__ partials,
                                                     double *__restrict__ norm,
                                                     const double *__restrict__ normf,
                                                     int *__restrict__ active, JudgeState J,
                                                     cudaGraphConditionalHandle handle,
                                                     const int *__restrict__ ts)
{
    pdl_wait();
    const bool on = active[0] != 0;
    const int c = *J.step + 1;
    double tot = 0.0;
    if (on) {
        double s = 0.0;
        for (int q = ts[0] + (int)threadIdx.x; q < ts[1]; q += 1024) s += partials[q];
        tot = block_sum_1024(s);
    }
    if (threadIdx.x == 0) {
        bool any = false;
        if (on) {
            norm[0] = sqrt(tot);
            any = judge_box(0, c, norm[0], normf, active, J);
        }
        *J.step = c;
        cudaGraphSetConditional(handle, any ? 1u : 0u);
    }
}

// ------------------------------------------------- packing and helpers ----

// The copies between the caller's packed arrays and the level layout, and
// the zeroing of a level's phi, take one thread per cell column of col_depth
// planes (TK_COLZ tiles): as many independent loads or stores in flight per
// thread instead of one per one-plane CTA.  partials (f only, or NULL): also
// the CTA's sum of f^2, as k_norm_partials in mode 1 forms it (the column's
// FMAs in plane order, then block_sum), so that ||f|| needs no pass of its own.
__global__ void __launch_bounds__(kThreads) k_pack(BoxSet<double> S, const long long *__restrict__ off,
                                                   const double *__restrict__ user, int to_f,
                                                   double *__restrict__ partials)
{
    pdl_wait();
    const int t = blockIdx.x;
    const int *ts = S.tstart[TK_COLZ];
    const int b = find_box(ts, S.nbox, t);
    const Box<double> &B = S.boxes[b];
    TilePos p = tile_pos(TK_COLZ, B.nx, B.ny, B.nz, t - ts[b]);
    double v = 0.0;
    if (p.x < B.nx && p.y < B.ny) {
        const int cz = col_depth(B), z0 = p.z * cz, z1 = min(z0 + cz, B.nz);
        const long long us = (long long)B.ny * B.nx;
        const double *src = user + off[B.box] + ((long long)z0 * B.ny + p.y) * B.nx + p.x;
#pragma unroll 4
        for (int k = z0; k < z1; ++k, src += us) {
            const double u = *src;
            if (to_f) {
                B.f[fidx(B, p.x, p.y, k)] = u;
                if (partials) v = fma(u, u, v);
            } else {
                B.phi[(long long)k * B.Q + (long long)p.y * B.P + p.x] = u;
            }
        }
    }
    if (partials) {   // uniform over the launch
        const double sum = block_sum(v);
        if (threadIdx.x == 0 && threadIdx.y == 0) partials[t] = sum;
    }
}

__global__ void __launch_bounds__(kThreads) k_unpack(BoxSet<double> S, const long long *__restrict__ off,
                                                     double *__restrict__ user,
                                                     const int *__restrict__ side)
{
    pdl_wait();
    const int t = blockIdx.x;
    const int *ts = S.tstart[TK_COLZ];
    const int b = find_box(ts, S.nbox, t);
    const Box<double> &B = S.boxes[b];
    TilePos p = tile_pos(TK_COLZ, B.nx, B.ny, B.nz, t - ts[b]);
    if (p.x >= B.nx || p.y >= B.ny) return;
    const int cz = col_depth(B), z0 = p.z * cz, z1 = min(z0 + cz, B.nz);
    const long long us = (long long)B.ny * B.nx;
    double *dst = user + off[B.box] + ((long long)z0 * B.ny + p.y) * B.nx + p.x;
    const double *src = ((side && side[B.box]) ? B.phi2 : B.phi) + (long long)z0 * B.Q +
                        (long long)p.y * B.P + p.x;
#pragma unroll 4
    for (int k = z0; k < z1; ++k, dst += us, src += B.Q) *dst = *src;
}

template <class T>
__global__ void __launch_bounds__(kThreads) k_zero(BoxSet<T> S, const int *__restrict__ active)
{
    pdl_wait();
    const int t = blockIdx.x;
    const int *ts = S.tstart[TK_COLZ];
    const int b = find_box(ts, S.nbox, t);
    const Box<T> &B = S.boxes[b];
    if (active && !active[B.box]) return;
    TilePos p = tile_pos(TK_COLZ, B.nx, B.ny, B.nz, t - ts[b]);
    if (p.x >= B.nx || p.y >= B.ny) return;
    const int cz = col_depth(B), z0 = p.z * cz, z1 = min(z0 + cz, B.nz);
    T *dst = B.phi + (long long)z0 * B.Q + (long long)p.y * B.P + p.x;
#pragma unroll 4
    for (int k = z0; k < z1; ++k, dst += B.Q) *dst = T(0);
}

__global__ void k_scales(int nbox, const int *__restrict__ active, int init,
                         const double *__restrict__ norm, const double *__restrict__ normf,
                         double *__restrict__ se, double *__restrict__ sr, double *__restrict__ sr_inv)
{
    pdl_wait();
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= nbox) return;
    if (init) {
        const double v = normf[b];
        se[b] = 0.0;
        sr[b] = v;
        sr_inv[b] = v > 0.0 ? 1.0 / v : 0.0;
    } else if (!active || active[b]) {
        const double v = norm[b];
        se[b] = sr[b];
        sr[b] = v;
        sr_inv[b] = v > 0.0 ? 1.0 / v : 0.0;
    }
}

// First stage of the inner exit test's sums: chunk c of the set (chunk
// c - cstart[b] of box b, cstart the per-box chunk prefix) sums the per-warp
// partials of its kInnerChunk restriction tiles in fixed order.
__global__ void __launch_bounds__(256) k_inner_sum(BoxSet<float> S, const int *__restrict__ active32,
                                                   const int *__restrict__ cstart,
                                                   int chunk_tiles,
                                                   const double *__restrict__ partials,
                                                   double *__restrict__ chunks)
{
    pdl_wait();
    __shared__ double wsum[8];
    const int c = blockIdx.x;
    const int b = find_box(cstart, S.nbox, c);
    if (!active32[S.boxes[b].box]) return;   // the whole CTA
    const int *ts = S.tstart[TK_COARSE];
    constexpr int W = kThreads / 32;   // partial sums per tile of the restriction
    const int t0 = ts[b] + (c - cstart[b]) * chunk_tiles;
    const int t1 = min(t0 + chunk_tiles, ts[b + 1]);
    double v = 0.0;
    for (long long q = (long long)t0 * W + threadIdx.x; q < (long long)t1 * W; q += 256)
        v += partials[q];
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) wsum[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        double tot = 0.0;
        for (int w = 0; w < 8; ++w) tot += wsum[w];
        chunks[c] = tot;
    }
}

// Exit test of the inner FP32 cycles of a refinement step (mixed precision,
// adaptive inner cycles).  The step solves A e = r32 with r32 = r_k / se
// (||r_k|| = sr, so ||r32|| = sr / se); after its update x + se e the FP64
// residual is se times the inner residual r32 - A e, up to FP32 rounding.
// Per box still in the inner cycles: ||r32 - A e|| of the just smoothed
// iterate (the red-children restriction's sums, per box and in fixed order:
// its chunk sums) against max(tol ||f|| / 2, floor_rel sr) / se: at or below
// it the update is expected to meet tol, or the step has gained the factor
// floor_rel, and the box leaves the inner cycles of this step (active32 = 0).
// floor_rel: the most one step asks of FP32 arithmetic.  One CTA per box;
// coupled (the boxes of a level solved as one domain, whose norms and scales
// are the domain's): one CTA, one decision for every box.
__global__ void __launch_bounds__(1024) k_inner_judge(BoxSet<float> S, int *__restrict__ active32,
                                                      const int *__restrict__ cstart,
                                                      const double *__restrict__ chunks,
                                                      const double *__restrict__ se,
                                                      const double *__restrict__ sr,
                                                      const double *__restrict__ normf,
                                                      const double *__restrict__ tol,
                                                      double floor_rel, int coupled)
{
    pdl_wait();
    __shared__ double wsum[32];
    const int b = blockIdx.x;
    const int id = S.boxes[b].box;
    if (!active32[id]) return;   // the whole CTA
    const int lo = coupled ? cstart[0] : cstart[b], hi = coupled ? cstart[S.nbox] : cstart[b + 1];
    double v = 0.0;
    for (int q = lo + threadIdx.x; q < hi; q += 1024) v += chunks[q];
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) wsum[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        double tot = 0.0;
        for (int w = 0; w < 32; ++w) tot += wsum[w];
        const double e = se[id];
        const double target =
            e > 0.0 ? fmax(0.5 * tol[0] * normf[id], floor_rel * sr[id]) / e : 0.0;
        if (!(sqrt(tot) > target)) {
            if (coupled)
                for (int q = 0; q < S.nbox; ++q) active32[S.boxes[q].box] = 0;
            else
                active32[id] = 0;
        }
    }
}

// Start of a refinement step's inner cycles: the inner flags are a copy of
// the step's; with a loop handle (inner cycles as a graph WHILE node) also
// the cycle counter to 0 and the loop condition to 1.  One CTA.
__global__ void __launch_bounds__(256) k_inner_begin(int nbox, const int *__restrict__ src,
                                                     int *__restrict__ dst, int *__restrict__ count,
                                                     cudaGraphConditionalHandle handle,
                                                     int use_handle)
{
    pdl_wait();
    for (int b = threadIdx.x; b < nbox; b += blockDim.x) dst[b] = src[b];
    if (threadIdx.x == 0) {
        *count = 0;
        if (use_handle) cudaGraphSetConditional(handle, 1u);
    }
}

// End of one inner cycle in the WHILE form: the loop goes on while some box
// is still in the inner cycles and fewer than max_cycles have run (the
// counter bounds the loop whatever the flags say); count[1] sums the cycles
// of the whole solve.  One CTA.
__global__ void __launch_bounds__(256) k_inner_end(int nbox, const int *__restrict__ flags,
                                                   int *__restrict__ count, int max_cycles,
                                                   cudaGraphConditionalHandle handle)
{
    pdl_wait();
    __shared__ int any;
    if (threadIdx.x == 0) any = 0;
    __syncthreads();
    for (int b = threadIdx.x; b < nbox; b += blockDim.x)
        if (flags[b]) any = 1;
    __syncthreads();
    if (threadIdx.x == 0) {
        const int c = count[0] + 1;
        count[0] = c;
        count[1] += 1;   // the solve's total, for the launch count
        cudaGraphSetConditional(handle, (any && c < max_cycles) ? 1u : 0u);
    }
}

cudaError_t launch_inner_begin(int nbox, const int *src, int *dst, int *count,
                               cudaGraphConditionalHandle handle, int use_handle, cudaStream_t st)
{
    return pdl_launch(k_inner_begin, dim3(1), dim3(256), 0, st, nbox, src, dst, count, handle,
                      use_handle);
}

cudaError_t launch_inner_end(int nbox, const int *flags, int *count, int max_cycles,
                             cudaGraphConditionalHandle handle, cudaStream_t st)
{
    return pdl_launch(k_inner_end, dim3(1), dim3(256), 0, st, nbox, flags, count, max_cycles,
                      handle);
}

// ------------------------------------------------------------- set-up ----
//
// Each set-up step is a per-position device function, called by a one-box
// kernel (the single-stage entry points) and by a set kernel that covers
// every box of a level in one launch (the solver).

// weight of a face between cells with coefficients a and b: the harmonic mean
// 2 a b / (a + b) times 1/h^2, given cb = (2 / h^2) b (the upper cell's
// factor, shared by the three faces below it), the quotient taken through
// rcp64 (within a few ulp of the correctly rounded quotient)
__device__ __forceinline__ double harmonic_w(double a, double b, double cb)
{
    return (a * cb) * rcp64(a + b);
}

// Wall w (0..5 = x-, x+, y-, y+, z-, z+) is Neumann when bit w of the mask is
// set: its faces carry no flux (weight 0); otherwise it is a Dirichlet wall
// h/2 from the cell centre (2 beta of the cell).
__device__ __forceinline__ double wall_beta(int bcm, int w, double b)
{
    return ((bcm >> w) & 1) ? 0.0 : 2.0 * b;
}

// Face weights at position (i, j, k) in [0, nx] x [0, ny] x [0, nz]: harmonic
// mean of the two cells' beta (a wall face: wall_beta) over h^2; with W32
// (mixed precision's finest level) also their FP32 roundings, the values
// the rounding step would write (a compile-time choice: a run-time test
// would cost the FP64-bound FP64 path its predicated conversions).
template <bool W32>
__device__ __forceinline__ void face_weights_at(int nx, int ny, int nz, int P, long long Q,
                                                double inv_h2, int bcm,
                                                const double *__restrict__ beta, double *wx,
                                                double *wy, double *wz, int i, int j, int k,
                                                float *wx32 = nullptr, float *wy32 = nullptr,
                                                float *wz32 = nullptr)
{
    auto bc = [&](int a, int bb, int c) { return beta[((long long)c * ny + bb) * nx + a]; };
    const long long q = (long long)k * Q + (long long)j * P + i;
    // cell (i, j, k) is the upper cell of all three faces at this position
    // (every inner face lies below a cell of the box)
    const double b = (i < nx && j < ny && k < nz) ? bc(i, j, k) : 0.0;
    const double cb = (2.0 * inv_h2) * b;
    if (j < ny && k < nz) {
        const double v = (i == 0) ? wall_beta(bcm, 0, bc(0, j, k)) * inv_h2
                       : (i == nx) ? wall_beta(bcm, 1, bc(nx - 1, j, k)) * inv_h2
                                   : harmonic_w(bc(i - 1, j, k), b, cb);
        wx[q] = v;
        if (W32) wx32[q] = f64_to_f32_rn(v);
    }
    if (i < nx && k < nz) {
        const double v = (j == 0) ? wall_beta(bcm, 2, bc(i, 0, k)) * inv_h2
                       : (j == ny) ? wall_beta(bcm, 3, bc(i, ny - 1, k)) * inv_h2
                                   : harmonic_w(bc(i, j - 1, k), b, cb);
        wy[q] = v;
        if (W32) wy32[q] = f64_to_f32_rn(v);
    }
    if (i < nx && j < ny) {
        const double v = (k == 0) ? wall_beta(bcm, 4, bc(i, j, 0)) * inv_h2
                       : (k == nz) ? wall_beta(bcm, 5, bc(i, j, nz - 1)) * inv_h2
                                   : harmonic_w(bc(i, j, k - 1), b, cb);
        wz[q] = v;
        if (W32) wz32[q] = f64_to_f32_rn(v);
    }
}

// Face weights of a coupled level's box from beta in the level layout (bl),
// whose guard cells hold the neighbouring box's beta across an interface or
// -1 on the union's boundary: an interface face takes the harmonic mean like
// any inner face (the neighbour computes the same value), a boundary face is
// a Dirichlet wall (2 beta).
__device__ __forceinline__ void face_weights_level_at(int nx, int ny, int nz, int P, long long Q,
                                                      double inv_h2, int bcm,
                                                      const double *__restrict__ bl, double *wx,
                                                      double *wy, double *wz, int i, int j, int k)
{
    const long long q = (long long)k * Q + (long long)j * P + i;
    // a below / left of the face, b = bl[q] above / right (the same cell for
    // all three faces); lo/hi: the walls on either side of axis d (their
    // Dirichlet or Neumann condition from bcm)
    const double b = bl[q];
    const double cb = (2.0 * inv_h2) * b;
    auto face = [&](double a, int d) {
        if (a < 0.0) return wall_beta(bcm, 2 * d, b) * inv_h2;
        if (b < 0.0) return wall_beta(bcm, 2 * d + 1, a) * inv_h2;
        return harmonic_w(a, b, cb);
    };
    if (j < ny && k < nz) wx[q] = face(bl[q - 1], 0);
    if (i < nx && k < nz) wy[q] = face(bl[q - P], 1);
    if (i < nx && j < ny) wz[q] = face(bl[q - Q], 2);
}

// Coarse position (I, J, K) in [0, cx] x [0, cy] x [0, cz]; coarse face
// beta = mean of the 4 fine faces, coarse h = 2h: w_c = (sum of 4 w) / 16.
template <class T>
__device__ __forceinline__ void coarsen_at(int nx, int ny, int nz, int P, long long Q,
                                           const T *__restrict__ wx, const T *__restrict__ wy,
                                           const T *__restrict__ wz, int cP, long long cQ,
                                           T *cwx, T *cwy, T *cwz, int I, int J, int K)
{
    const int cx = nx / 2, cy = ny / 2, cz = nz / 2;
    auto at = [&](int i, int j, int k) { return (long long)k * Q + (long long)j * P + i; };
    const long long cq = (long long)K * cQ + (long long)J * cP + I;
    const T q = T(0.0625);
    if (J < cy && K < cz)
        cwx[cq] = (wx[at(2 * I, 2 * J, 2 * K)] + wx[at(2 * I, 2 * J + 1, 2 * K)] +
                   wx[at(2 * I, 2 * J, 2 * K + 1)] + wx[at(2 * I, 2 * J + 1, 2 * K + 1)]) * q;
    if (I < cx && K < cz)
        cwy[cq] = (wy[at(2 * I, 2 * J, 2 * K)] + wy[at(2 * I + 1, 2 * J, 2 * K)] +
                   wy[at(2 * I, 2 * J, 2 * K + 1)] + wy[at(2 * I + 1, 2 * J, 2 * K + 1)]) * q;
    if (I < cx && J < cy)
        cwz[cq] = (wz[at(2 * I, 2 * J, 2 * K)] + wz[at(2 * I + 1, 2 * J, 2 * K)] +
                   wz[at(2 * I, 2 * J + 1, 2 * K)] + wz[at(2 * I + 1, 2 * J + 1, 2 * K)]) * q;
}

// ---- mixed precision's coarser FP32 levels, averaged in FP32
//
// Only the finest level's FP32 weights (the rounded FP64 ones) and the
// coarser FP32 levels are read by mixed precision's cycles: the coarser
// levels are averaged from the finer FP32 weights (coarsen_at<float>) and
// take their FP32 1/D from their own weights, with no FP64 coarse level.

// FP32 1/D of cell c from the level's FP32 weights.
__device__ __forceinline__ void inv_diag32_at(int P, long long Q, const float *__restrict__ wx,
                                              const float *__restrict__ wy,
                                              const float *__restrict__ wz, float *invD,
                                              long long c)
{
    invD[c] = 1.0f / (((wx[c] + wx[c + 1]) + (wy[c] + wy[c + P])) + (wz[c] + wz[c + Q]));
}

template <bool W32 = false>
__device__ __forceinline__ void inv_diag_at(int P, long long Q, const double *__restrict__ wx,
                                            const double *__restrict__ wy,
                                            const double *__restrict__ wz, double *invD,
                                            double *Dout, long long c, long long cf,
                                            float *invD32 = nullptr)
{
    const double D = ((wx[c] + wx[c + 1]) + (wy[c] + wy[c + P])) + (wz[c] + wz[c + Q]);
    if (invD) invD[cf] = rcp64(D);  // NULL: mixed precision, whose FP64 levels never smooth
    if (Dout) Dout[cf] = D;
    // mixed precision's finest level (no FP64 1/D): the FP32 1/D the
    // rounding step would write
    if (W32) invD32[c] = 1.0f / f64_to_f32_rn(D);
}

// Every stored weight (and the inverse diagonal) at position (i, j, k) in
// [0, nx] x [0, ny] x [0, nz], rounded to FP32 (the FP32 copies are in the
// natural layout; the FP64 invD and D are colour-split when rb).  Without an
// FP64 invD the FP32 one is the FP32 reciprocal of the rounded D.
__device__ __forceinline__ void round_at(int nx, int ny, int nz, int P, long long Q,
                                         const double *__restrict__ wx,
                                         const double *__restrict__ wy,
                                         const double *__restrict__ wz,
                                         const double *__restrict__ invD, float *wx32,
                                         float *wy32, float *wz32, float *invD32, int i, int j,
                                         int k, int rb = 0, int par = 0,
                                         const double *__restrict__ D = nullptr)
{
    const long long q = (long long)k * Q + (long long)j * P + i;
    if (j < ny && k < nz) wx32[q] = f64_to_f32_rn(wx[q]);
    if (i < nx && k < nz) wy32[q] = f64_to_f32_rn(wy[q]);
    if (i < nx && j < ny) wz32[q] = f64_to_f32_rn(wz[q]);
    if (i < nx && j < ny && k < nz) {
        const long long cf = rb ? split_at(i, j, k, par, P, Q) : q;
        invD32[q] = invD ? f64_to_f32_rn(invD[cf]) : 1.0f / f64_to_f32_rn(D[cf]);
    }
}

// Dense inverses of the coarsest levels: M = -A (symmetric positive definite)
// is assembled and inverted in place by Gauss-Jordan elimination without
// pivoting (M is diagonally dominant, or positive definite after the shift
// below), A^{-1} = -M^{-1}.  When every wall is Neumann (`singular`), M is only
// semi-definite with the constants as null space; c 1 1^T with c = trace(M) /
// n^2 is added, which makes it positive definite: applied to r it gives a
// solution of M x = r - mean(r) (the constant part of r, which no solution can
// match, is dropped), and the zero-mean one when r has zero mean.
//
// Only the upper triangle is kept: after pivots 0..p an entry with exactly one
// index <= p is the negative of its mirror and every other entry equals its
// mirror, so each pivot costs n^2/2 updates.  The rows are dealt out over the
// CTAs of one cluster (row i to rank i % CTAs), in shared memory when they fit
// (n <= 890 in FP64 on 16 CTAs), else in global scratch; a pivot needs its
// column, which every owner stores into every CTA as it updates it, and one
// cluster barrier.  What bounds it: n pivots of a barrier (~0.5 us) plus
// n^2/2 FMAs on the FP64 pipes of 16 SMs.  A row's updates are those of a
// single CTA in the same order, so the inverse is the same bit for bit.  One CTA
// per box took 30.5 ms for 567 cells (FP64), 1.79 ms for the 192-cell boxes of
// a batch, 181 us for 105 cells (FP32); these take 3.6 ms, 0.68 ms and 128 us.
constexpr int kInvThreads = 512;

// The rows of rank's part.  Row i = rank + ncta m holds (i, i..n-1).
template <class R>
struct InvRows {
    R *a;
    int n, rank, ncta;
    bool packed;
    __device__ __forceinline__ R *row(int m) const
    {
        const long long i = rank + (long long)ncta * m;
        return a + (packed ? (long long)m * (n - rank) - (long long)ncta * m * (m - 1) / 2 : i * n + i);
    }
    // row i if it is this rank's, else NULL
    __device__ __forceinline__ R *own(int i) const
    {
        return i % ncta == rank ? row(i / ncta) : nullptr;
    }
    __device__ __forceinline__ int count() const { return rank < n ? (n - 1 - rank) / ncta + 1 : 0; }
};

__host__ __device__ inline long long inv_rows_elems(int n, int ncta)   // rank 0's, the most
{
    const long long m = (n - 1) / ncta + 1;
    return m * n - (long long)ncta * m * (m - 1) / 2;
}

// The block of M = -A of one box, rows and columns from `at` on (the box's
// cells in C order): diagonal = sum of the six weights, -w to each later
// neighbour inside the box (the earlier ones are the mirrors).
template <class R, class W>
__device__ __forceinline__ void assemble_box_block(int nx, int ny, int nz, int P, long long Q,
                                                   const W *__restrict__ wx,
                                                   const W *__restrict__ wy,
                                                   const W *__restrict__ wz, const InvRows<R> &M,
                                                   int at)
{
    const int m = nx * ny * nz;
    for (int r = threadIdx.x; r < m; r += blockDim.x) {
        R *row = M.own(at + r);
        if (!row) continue;
        const int i = r % nx, j = (r / nx) % ny, k = r / (nx * ny);
        const long long c = (long long)k * Q + (long long)j * P + i;
        const W ww = wx[c], we = wx[c + 1], ws = wy[c], wn = wy[c + P], wd = wz[c],
                wu = wz[c + Q];
        row[0] = (R)(((ww + we) + (ws + wn)) + (wd + wu));
        if (i < nx - 1) row[1] = (R)-we;
        if (j < ny - 1) row[nx] = (R)-wn;
        if (k < nz - 1) row[nx * ny] = (R)-wu;
    }
}

// The matrix storage of a cluster's inverse: two columns and the pivot row
// first (3 n of R), then the rows if they fit in smem_bytes, else scratch.
template <class R>
__device__ __forceinline__ InvRows<R> inv_rows(const cg::cluster_group &cl, int n, R *smem,
                                               int smem_bytes, R *scratch)
{
    InvRows<R> M;
    M.n = n;
    M.rank = (int)cl.block_rank();
    M.ncta = (int)cl.num_blocks();
    M.packed = (3LL * n + inv_rows_elems(n, M.ncta)) * (long long)sizeof(R) <= smem_bytes;
    M.a = M.packed ? smem + 3 * n : scratch;
    for (int m = threadIdx.x >> 5; m < M.count(); m += kInvThreads / 32) {
        R *r = M.row(m);
        for (int j = threadIdx.x & 31; j < n - M.rank - M.ncta * m; j += 32) r[j] = R(0);
    }
    __syncthreads();
    return M;
}

// Invert the assembled rows; A^{-1} to inv64 and/or inv32 (either may be NULL).
// smem: the columns and the pivot row; ips: shared, [2].
template <class R>
__device__ __forceinline__ void gauss_jordan_cluster(const cg::cluster_group &cl,
                                                     const InvRows<R> &M, bool singular,
                                                     double *inv64, float *inv32, R *smem, R *ips)
{
    const int n = M.n, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int nw = kInvThreads / 32, rows = M.count();
    R *const rowv = smem + 2 * n;
    auto everywhere = [&](R *p, R v) {
        for (int r = 0; r < M.ncta; ++r) *cl.map_shared_rank(p, r) = v;
    };
    cl.sync();   // every CTA's shared memory is in use
    if (singular) {
        for (int m = tid; m < rows; m += kInvThreads) everywhere(smem + M.rank + M.ncta * m, M.row(m)[0]);
        cl.sync();
        if (tid == 0) {
            R tr = R(0);
            for (int r = 0; r < n; ++r) tr += smem[r];
            ips[0] = tr / ((R)n * (R)n);
        }
        __syncthreads();
        const R shift = ips[0];
        for (int m = warp; m < rows; m += nw) {
            R *r = M.row(m);
            for (int j = lane; j < n - M.rank - M.ncta * m; j += 32) r[j] += shift;
        }
        cl.sync();
    }
    if (M.rank == 0) {   // the first pivot's column is row 0
        const R *r = M.row(0);
        for (int j = tid; j < n; j += kInvThreads) everywhere(smem + j, r[j]);
        if (tid == 0) everywhere(ips, R(1) / r[0]);
    }
    cl.sync();
    for (int p = 0; p < n; ++p) {
        // column p: (i, p) for i <= p, (p, i) below the diagonal; its new row
        // p: a_pj / a_pp (a_pj for j < p is minus its stored mirror)
        const R *const col = smem + (p & 1) * n;
        R *const next = smem + ((p + 1) & 1) * n;
        const R ip = ips[p & 1];
        for (int j = tid; j < n; j += kInvThreads)
            rowv[j] = j == p ? ip : (j > p ? col[j] : -col[j]) * ip;
        __syncthreads();
        for (int m = warp; m < rows; m += nw) {
            const int i = M.rank + M.ncta * m;
            const R ci = col[i];
            R *ar = M.row(m);
            for (int j = i + lane; j < n; j += 32) {
                R v;
                if (i == p) v = rowv[j];              // row p (j >= p; j = p: 1 / a_pp)
                else if (j == p) v = -ci * ip;        // column p above the diagonal
                else v = fmadd(-ci, rowv[j], ar[j - i]);
                ar[j - i] = v;
                if (j == p + 1) {                     // column p + 1, down to its diagonal
                    everywhere(next + i, v);
                    if (i == p + 1) everywhere(ips + ((p + 1) & 1), R(1) / v);
                } else if (i == p + 1) {              // and, mirrored, from row p + 1
                    everywhere(next + j, v);
                }
            }
        }
        cl.sync();
    }
    for (int m = warp; m < rows; m += nw) {
        const int i = M.rank + M.ncta * m;
        const R *ar = M.row(m);
        for (int j = i + lane; j < n; j += 32) {
            const double v = -(double)ar[j - i];
            const long long e = (long long)i * n + j, t = (long long)j * n + i;
            if (inv64) {
                inv64[e] = v;
                inv64[t] = v;
            }
            if (inv32) {
                inv32[e] = (float)v;
                inv32[t] = (float)v;
            }
        }
    }
}

// The coarsest level's inverse of one box in precision R (double: A^{-1} to
// inv64 and its rounding to inv32; float, when no FP64 inverse is wanted: inv32
// only), by the calling cluster.
template <class R, class W>
__device__ __forceinline__ void bottom_inverse_cluster(const cg::cluster_group &cl, int nx, int ny,
                                                       int nz, int P, long long Q,
                                                       const W *__restrict__ wx,
                                                       const W *__restrict__ wy,
                                                       const W *__restrict__ wz, bool singular,
                                                       R *smem, int smem_bytes, R *scratch,
                                                       double *inv64, float *inv32, R *ips)
{
    const InvRows<R> M = inv_rows<R>(cl, nx * ny * nz, smem, smem_bytes, scratch);
    assemble_box_block(nx, ny, nz, P, Q, wx, wy, wz, M, 0);
    gauss_jordan_cluster<R>(cl, M, singular, inv64, inv32, smem, ips);
}

// ---- one box (single-stage entry points): grid over positions

__global__ void k_face_weights(int nx, int ny, int nz, int P, long long Q, double inv_h2,
                               int bcm, const double *__restrict__ beta, double *__restrict__ wx,
                               double *__restrict__ wy, double *__restrict__ wz)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y * blockDim.y + threadIdx.y;
    const int k = blockIdx.z;
    if (i > nx || j > ny || k > nz) return;
    face_weights_at<false>(nx, ny, nz, P, Q, inv_h2, bcm, beta, wx, wy, wz, i, j, k);
}

__global__ void k_coarsen(int nx, int ny, int nz, int P, long long Q, const double *__restrict__ wx,
                          const double *__restrict__ wy, const double *__restrict__ wz, int cP,
                          long long cQ, double *__restrict__ cwx, double *__restrict__ cwy,
                          double *__restrict__ cwz)
{
    const int I = blockIdx.x * blockDim.x + threadIdx.x;
    const int J = blockIdx.y * blockDim.y + threadIdx.y;
    const int K = blockIdx.z;
    if (I > nx / 2 || J > ny / 2 || K > nz / 2) return;
    coarsen_at(nx, ny, nz, P, Q, wx, wy, wz, cP, cQ, cwx, cwy, cwz, I, J, K);
}

__global__ void k_inv_diag(int nx, int ny, int nz, int P, long long Q, const double *__restrict__ wx,
                           const double *__restrict__ wy, const double *__restrict__ wz,
                           double *__restrict__ invD, double *__restrict__ Dout)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y * blockDim.y + threadIdx.y;
    const int k = blockIdx.z;
    if (i >= nx || j >= ny || k >= nz) return;
    const long long c = (long long)k * Q + (long long)j * P + i;
    inv_diag_at(P, Q, wx, wy, wz, invD, Dout, c, c);
}

__global__ void k_round_f32(int nx, int ny, int nz, int P, long long Q, const double *__restrict__ wx,
                            const double *__restrict__ wy, const double *__restrict__ wz,
                            const double *__restrict__ invD, float *__restrict__ wx32,
                            float *__restrict__ wy32, float *__restrict__ wz32,
                            float *__restrict__ invD32)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y * blockDim.y + threadIdx.y;
    const int k = blockIdx.z;
    if (i > nx || j > ny || k > nz) return;
    round_at(nx, ny, nz, P, Q, wx, wy, wz, invD, wx32, wy32, wz32, invD32, i, j, k);
}

__global__ void __launch_bounds__(kInvThreads) k_bottom_inverse(
    int nx, int ny, int nz, int P, long long Q, const double *__restrict__ wx,
    const double *__restrict__ wy, const double *__restrict__ wz, int singular,
    double *__restrict__ a, double *__restrict__ inv64, float *__restrict__ inv32, int smem_bytes)
{
    extern __shared__ __align__(16) unsigned char inv_smem[];
    __shared__ double ips[2];
    bottom_inverse_cluster<double>(cg::this_cluster(), nx, ny, nz, P, Q, wx, wy, wz, singular != 0,
                                   reinterpret_cast<double *>(inv_smem), smem_bytes, a, inv64,
                                   inv32, ips);
}

// ---- every box of a level in one launch (the solver's set-up)

__host__ __device__ constexpr int setup_kind(int step)
{
    return (step == 1 || step == 9) ? TK_CFACE
         : (step == 2 || step == 6 || step == 8) ? TK_CELL : TK_FACE;
}

// One set-up step at one position of box B (see k_setup for the steps).
template <int step>
__device__ __forceinline__ void setup_step(const SetupBox &B, const TilePos &p)
{
    if constexpr (step == 0)
        face_weights_at<false>(B.nx, B.ny, B.nz, B.P, B.Q, B.inv_h2, B.bc, B.beta, B.wx, B.wy,
                               B.wz, p.x, p.y, p.z);
    else if constexpr (step == 5)
        face_weights_at<true>(B.nx, B.ny, B.nz, B.P, B.Q, B.inv_h2, B.bc, B.beta, B.wx, B.wy,
                              B.wz, p.x, p.y, p.z, B.wx32, B.wy32, B.wz32);
    else if constexpr (step == 1)
        coarsen_at<double>(B.nx, B.ny, B.nz, B.P, B.Q, B.wx, B.wy, B.wz, B.cP, B.cQ, B.cwx,
                           B.cwy, B.cwz, p.x, p.y, p.z);
    else if constexpr (step == 2)
        inv_diag_at(B.P, B.Q, B.wx, B.wy, B.wz, B.invD, B.D,
                    (long long)p.z * B.Q + (long long)p.y * B.P + p.x,
                    B.rb ? split_at(p.x, p.y, p.z, B.par, B.P, B.Q)
                         : (long long)p.z * B.Q + (long long)p.y * B.P + p.x);
    else if constexpr (step == 6)
        inv_diag_at<true>(B.P, B.Q, B.wx, B.wy, B.wz, nullptr, B.D,
                          (long long)p.z * B.Q + (long long)p.y * B.P + p.x,
                          B.rb ? split_at(p.x, p.y, p.z, B.par, B.P, B.Q)
                               : (long long)p.z * B.Q + (long long)p.y * B.P + p.x,
                          B.invD32);
    else if constexpr (step == 4)
        face_weights_level_at(B.nx, B.ny, B.nz, B.P, B.Q, B.inv_h2, B.bc, B.betaL, B.wx, B.wy,
                              B.wz, p.x, p.y, p.z);
    else if constexpr (step == 8)
        inv_diag32_at(B.P, B.Q, B.wx32, B.wy32, B.wz32, B.invD32,
                      (long long)p.z * B.Q + (long long)p.y * B.P + p.x);
    else if constexpr (step == 9)
        coarsen_at<float>(B.nx, B.ny, B.nz, B.P, B.Q, B.wx32, B.wy32, B.wz32, B.cP, B.cQ,
                          B.cwx32, B.cwy32, B.cwz32, p.x, p.y, p.z);
    else
        round_at(B.nx, B.ny, B.nz, B.P, B.Q, B.wx, B.wy, B.wz, B.invD, B.wx32, B.wy32, B.wz32,
                 B.invD32, p.x, p.y, p.z, B.rb, B.par, B.D);
}

// step 0 faces (TK_FACE), 1 coarsen (TK_CFACE), 2 diagonal (TK_CELL),
// 3 FP32 copies (TK_FACE), 4 faces of a coupled level from betaL (TK_FACE),
// 5 faces with their FP32 copies (TK_FACE), 6 diagonal with the FP32 1/D
// (TK_CELL): 5 and 6 take the place of 0, 2 and 3 on mixed precision's
// finest level; 8 FP32 1/D (TK_CELL) and 9 FP32 coarsening (TK_CFACE) set
// up its coarser FP32 levels from the finer FP32 ones.  The step is a
// template argument: a run-time index into the set's tstart array
// (a kernel parameter) would make every thread copy the set to local memory.
template <int STEP>
__global__ void __launch_bounds__(kThreads) k_setup(SetupSet S, int t0)
{
    constexpr int kind = setup_kind(STEP);
    const int t = blockIdx.x + t0;
    const int *ts = S.tstart[kind];
    const int b = find_box(ts, S.nbox, t);
    const SetupBox &B = S.boxes[b];
    const TilePos p = tile_pos(kind, B.nx, B.ny, B.nz, t - ts[b]);
    int ex, ey, ez;
    tile_extent(kind, B.nx, B.ny, B.nz, ex, ey, ez);
    if (p.x >= ex || p.y >= ey) return;
    setup_step<STEP>(B, p);
}

// One cluster per box: the coarsest level's dense inverse, in FP64 when an FP64
// inverse is wanted, else (mixed precision, whose FP64 levels never solve) in
// FP32 straight away.
__global__ void __launch_bounds__(kInvThreads) k_setup_bottom(SetupSet S, int smem_bytes)
{
    extern __shared__ __align__(16) unsigned char inv_smem[];
    __shared__ double ips[2];
    const cg::cluster_group cl = cg::this_cluster();
    const SetupBox &B = S.boxes[blockIdx.x / cl.num_blocks()];
    const bool singular = (B.bc & 63) == 63;
    double *const sd = reinterpret_cast<double *>(inv_smem);
    float *const sf = reinterpret_cast<float *>(inv_smem), *const wf = reinterpret_cast<float *>(B.work);
    float *const ipf = reinterpret_cast<float *>(ips);
    if (B.w32src)
        // coarser FP32 levels averaged in FP32: assembled from their weights
        bottom_inverse_cluster<float>(cl, B.nx, B.ny, B.nz, B.P, B.Q, B.wx32, B.wy32, B.wz32,
                                      singular, sf, smem_bytes, wf, nullptr, B.inv32, ipf);
    else if (B.inv64)
        bottom_inverse_cluster<double>(cl, B.nx, B.ny, B.nz, B.P, B.Q, B.wx, B.wy, B.wz, singular,
                                       sd, smem_bytes, B.work, B.inv64, B.inv32, ips);
    else
        bottom_inverse_cluster<float>(cl, B.nx, B.ny, B.nz, B.P, B.Q, B.wx, B.wy, B.wz, singular,
                                      sf, smem_bytes, wf, nullptr, B.inv32, ipf);
}

// ----------------------------------------------------- projection steps ----
//
// The velocity constraint around the solve (the equation of a MAESTRO step
// enforces it): f = div(u) - S from face velocities, and after the solve
// u -= beta_face grad(phi) on every face (phi = 0 outside, wall faces with
// doubled beta), so that div(u) = S.  beta_face / h = w h with the stored
// level weights w = beta_face / h^2.  Velocity and cell arrays are in their
// natural C layouts: u (nz, ny, nx+1), v (nz, ny+1, nx), w (nz+1, ny, nx).

__global__ void k_project_rhs(int nx, int ny, int nz, double inv_h, const double *__restrict__ u,
                              const double *__restrict__ v, const double *__restrict__ w,
                              const double *__restrict__ S, double *__restrict__ f)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y * blockDim.y + threadIdx.y;
    const int k = blockIdx.z;
    if (i >= nx || j >= ny || k >= nz) return;
    const long long ux = ((long long)k * ny + j) * (nx + 1) + i;
    const long long vy = ((long long)k * (ny + 1) + j) * nx + i;
    const long long wz = ((long long)k * ny + j) * nx + i;
    const long long c = wz;
    const double d = (u[ux + 1] - u[ux]) + (v[vy + nx] - v[vy]) + (w[wz + (long long)nx * ny] - w[wz]);
    f[c] = d * inv_h - (S ? S[c] : 0.0);
}

__global__ void k_project_correct(int nx, int ny, int nz, int P, long long Q, double h,
                                  const double *__restrict__ wx, const double *__restrict__ wy,
                                  const double *__restrict__ wzf, const double *__restrict__ phi,
                                  double *__restrict__ u, double *__restrict__ v,
                                  double *__restrict__ w)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y * blockDim.y + threadIdx.y;
    const int k = blockIdx.z;
    if (i > nx || j > ny || k > nz) return;
    auto ph = [&](int a, int b, int c) -> double {
        if (a < 0 || b < 0 || c < 0 || a >= nx || b >= ny || c >= nz) return 0.0;
        return phi[((long long)c * ny + b) * nx + a];
    };
    const long long q = (long long)k * Q + (long long)j * P + i;
    if (j < ny && k < nz)
        u[((long long)k * ny + j) * (nx + 1) + i] -= wx[q] * h * (ph(i, j, k) - ph(i - 1, j, k));
    if (i < nx && k < nz)
        v[((long long)k * (ny + 1) + j) * nx + i] -= wy[q] * h * (ph(i, j, k) - ph(i, j - 1, k));
    if (i < nx && j < ny)
        w[((long long)k * ny + j) * nx + i] -= wzf[q] * h * (ph(i, j, k) - ph(i, j, k - 1));
}

// dbeta += chain of dL/dbeta_face through the harmonic mean (see mg.h),
// summed over nrhs right-hand sides (phi and lam: consecutive (nz, ny, nx)
// arrays); a Neumann wall face (bit w of bcm) has no coefficient and adds
// nothing.
//
// The face between cells c and o adds g 2 beta_o^2 / (beta_c + beta_o)^2 to c
// and g 2 beta_c^2 / (beta_c + beta_o)^2 to o, g = sum over right-hand sides of
// (lam_o - lam_c)(phi_o - phi_c) / h^2.  Bound by the FP64 pipe: 9 operations a
// cell and right-hand side, so every face's sum and its 2 / (beta_c + beta_o)^2
// (rcp64, no division) are formed once, by the thread of its lower cell, and
// handed to the upper cell through shared memory (x, y) or a register (z).  A
// CTA marches kGradZ planes; the tile's lower x and y faces are formed again by
// one warp each, its first z faces by every thread.  8 x 128^3: 540 us; one
// launch per right-hand side with six faces and FP64 divisions a cell took
// 8 x 397 us.
constexpr int kGradZ = 8;
__global__ void __launch_bounds__(kThreads) k_beta_grad(int nx, int ny, int nz, int nrhs,
                                                        double inv_h2, int bcm,
                                                        const double *__restrict__ beta,
                                                        const double *__restrict__ phi,
                                                        const double *__restrict__ lam,
                                                        double *__restrict__ dbeta)
{
    __shared__ double sx[2][kTY][kTX + 1], sy[2][kTY + 1][kTX];
    const int tx = threadIdx.x, ty = threadIdx.y;
    const int i0 = blockIdx.x * kTX, j0 = blockIdx.y * kTY;
    const int i = i0 + tx, j = j0 + ty;
    const int k0 = blockIdx.z * kGradZ, k1 = min(k0 + kGradZ, nz);
    const long long sy1 = nx, sz1 = (long long)nx * ny, cells = sz1 * nz;
    const double two = 2.0 * inv_h2;
    // the face between cell c and the upper cell c + d
    auto face = [&](long long c, long long d) {
        double g = 0.0;
        for (int r = 0; r < nrhs; ++r) {
            const double *p = phi + r * cells + c, *l = lam + r * cells + c;
            g = fma(l[d] - l[0], p[d] - p[0], g);
        }
        const double q = rcp64(beta[c] + beta[c + d]);
        return (two * g) * (q * q);
    };
    const bool in = i < nx && j < ny;
    const long long col = (long long)j * nx + i;
    double zlo = (in && k0 > 0) ? face((k0 - 1) * sz1 + col, sz1) : 0.0;
    for (int k = k0; k < k1; ++k) {
        const long long c = k * sz1 + col;
        const int s = k & 1;
        const bool ux = in && i + 1 < nx, uy = in && j + 1 < ny, uz = in && k + 1 < nz;
        double fx = 0.0, fy = 0.0, fz = 0.0, wall = 0.0;
        if (in) {   // the three upper faces, their differences shared over one read
            double gx = 0.0, gy = 0.0, gz = 0.0;
            const long long dx = ux ? 1 : 0, dy = uy ? sy1 : 0, dz = uz ? sz1 : 0;
            const bool edge = i == 0 || !ux || j == 0 || !uy || k == 0 || !uz;
            for (int r = 0; r < nrhs; ++r) {
                const double *p = phi + r * cells + c, *l = lam + r * cells + c;
                const double pc = p[0], lc = l[0];
                gx = fma(l[dx] - lc, p[dx] - pc, gx);
                gy = fma(l[dy] - lc, p[dy] - pc, gy);
                gz = fma(l[dz] - lc, p[dz] - pc, gz);
                if (edge) wall = fma(lc, pc, wall);
            }
            const double b = beta[c];
            double q = rcp64(b + beta[c + dx]);
            fx = (two * gx) * (q * q);
            q = rcp64(b + beta[c + dy]);
            fy = (two * gy) * (q * q);
            q = rcp64(b + beta[c + dz]);
            fz = (two * gz) * (q * q);
        }
        sx[s][ty][tx + 1] = fx;
        sy[s][ty + 1][tx] = fy;
        if (ty == 0 && tx < kTY) {   // the tile's lower x faces
            const int jj = j0 + tx;
            sx[s][tx][0] = (i0 > 0 && i0 < nx + 1 && jj < ny)
                               ? face(k * sz1 + (long long)jj * nx + i0 - 1, 1) : 0.0;
        }
        if (ty == 1)                 // its lower y faces
            sy[s][0][tx] = (j0 > 0 && i < nx)
                               ? face(k * sz1 + (long long)(j0 - 1) * nx + i, sy1) : 0.0;
        __syncthreads();             // (two buffers: the next plane writes the other one)
        if (in) {
            auto sq = [&](long long o) { const double b = beta[o]; return b * b; };
            const double xlo = sx[s][ty][tx], ylo = sy[s][ty][tx];
            double acc = 0.0;
            int walls = 0;
            auto one = [&](bool inside, int w, double f, long long o) {
                if (inside) acc = fma(f, sq(o), acc);
                else if (!((bcm >> w) & 1)) ++walls;
            };
            one(i > 0, 0, xlo, c - 1);
            one(ux, 1, fx, c + 1);
            one(j > 0, 2, ylo, c - sy1);
            one(uy, 3, fy, c + sy1);
            one(k > 0, 4, zlo, c - sz1);
            one(uz, 5, fz, c + sz1);
            if (walls) acc = fma((double)walls * two, wall, acc);
            dbeta[c] += acc;
        }
        zlo = fz;
    }
}

// ------------------------------------------------------ wall values ----
//
// f_out = f - the lift of non-zero wall values, one thread per cell (only
// cells on the box surface change; the others are copied; f_out may be f).  vals packs one
// value per wall face, walls in the order x-, x+, y-, y+, z-, z+; an x wall
// is (nz, ny), a y wall (nz, nx), a z wall (ny, nx), C order.  A Dirichlet
// value g (phi on the wall) lifts w_wall g, with w_wall = 2 beta_c / h^2 the
// stored weight of the wall face; a Neumann value q (outward flux
// beta dphi/dn) lifts q / h.  Walls are taken in order, as in the oracle.
__global__ void k_bc_lift(int nx, int ny, int nz, int P, long long Q, double inv_h, int bcm,
                          const double *__restrict__ wx, const double *__restrict__ wy,
                          const double *__restrict__ wz, const double *__restrict__ vals,
                          const double *f, double *fout)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y * blockDim.y + threadIdx.y;
    const int k = blockIdx.z;
    if (i >= nx || j >= ny || k >= nz) return;
    const long long u = ((long long)k * ny + j) * nx + i;
    const long long c = (long long)k * Q + (long long)j * P + i;
    double v = f[u];
    const long long ax = (long long)ny * nz, ay = (long long)nx * nz, az = (long long)nx * ny;
    const long long o[6] = {0, ax, 2 * ax, 2 * ax + ay, 2 * ax + 2 * ay, 2 * ax + 2 * ay + az};
    auto term = [&](int w, double wall_w, long long at) {
        if ((bcm >> (6 + w / 2)) & 1) return;   // periodic axis: no wall
        const double g = vals[o[w] + at];
        v -= ((bcm >> w) & 1) ? g * inv_h : wall_w * g;
    };
    if (i == 0) term(0, wx[c], (long long)k * ny + j);
    if (i == nx - 1) term(1, wx[c + 1], (long long)k * ny + j);
    if (j == 0) term(2, wy[c], (long long)k * nx + i);
    if (j == ny - 1) term(3, wy[c + P], (long long)k * nx + i);
    if (k == 0) term(4, wz[c], (long long)j * nx + i);
    if (k == nz - 1) term(5, wz[c + Q], (long long)j * nx + i);
    fout[u] = v;
}

// ------------------------------------------------------------ means ----
//
// With every wall Neumann A is singular (constants): f loses its mean before
// the solve and phi after it.  Partial sums over TK_COLZ columns (field 0 =
// f, 1 = phi), then one CTA per box sums them in a fixed order and
// subtracts the mean from every cell.
__global__ void __launch_bounds__(kThreads) k_sum_partials(BoxSet<double> S, int field,
                                                           double *__restrict__ partials)
{
    pdl_wait();
    const int t = blockIdx.x;
    const int *ts = S.tstart[TK_COLZ];
    const int b = find_box(ts, S.nbox, t);
    const Box<double> &B = S.boxes[b];
    TilePos p = tile_pos(TK_COLZ, B.nx, B.ny, B.nz, t - ts[b]);
    double v = 0.0;
    if (p.x < B.nx && p.y < B.ny) {
        const int cz = col_depth(B), z0 = p.z * cz, z1 = min(z0 + cz, B.nz);
        for (int k = z0; k < z1; ++k)
            v += field ? B.phi[(long long)k * B.Q + (long long)p.y * B.P + p.x]
                       : B.f[fidx(B, p.x, p.y, k)];
    }
    double s = block_sum(v);
    if (threadIdx.x == 0 && threadIdx.y == 0) partials[t] = s;
}

__global__ void __launch_bounds__(1024) k_mean_finish(BoxSet<double> S,
                                                      const double *__restrict__ partials,
                                                      double *__restrict__ mean)
{
    pdl_wait();
    __shared__ double wsum[32];
    const int b = blockIdx.x;
    const Box<double> &B = S.boxes[b];
    const int *ts = S.tstart[TK_COLZ];
    double s = 0.0;
    for (int q = ts[b] + (int)threadIdx.x; q < ts[b + 1]; q += 1024) s += partials[q];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) wsum[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        double tot = 0.0;
        for (int w = 0; w < 32; ++w) tot += wsum[w];
        mean[B.box] = tot / ((double)B.nx * B.ny * B.nz);
    }
}

__global__ void __launch_bounds__(kThreads) k_sub_mean(BoxSet<double> S, int field,
                                                       const double *__restrict__ mean)
{
    pdl_wait();
    const int t = blockIdx.x;
    const int *ts = S.tstart[TK_CELL];
    const int b = find_box(ts, S.nbox, t);
    const Box<double> &B = S.boxes[b];
    TilePos p = tile_pos(TK_CELL, B.nx, B.ny, B.nz, t - ts[b]);
    if (p.x >= B.nx || p.y >= B.ny) return;
    if (field) B.phi[(long long)p.z * B.Q + (long long)p.y * B.P + p.x] -= mean[B.box];
    else B.f[fidx(B, p.x, p.y, p.z)] -= mean[B.box];
}

// ------------------------------------------------- preconditioned CG ----
//
// Conjugate gradients on A x = f (A negative definite: the signs cancel in
// alpha and beta), preconditioned by one symmetric V-cycle z = V r.  Level-0
// FP64 arrays of every box: x in phi2, r in f, z in phi (the V-cycle's own
// solution), p and q in two extra arrays.  Per-box scalars in PcgScalars.

// PcgScalars (kernels.h): rz = <r, z> of the previous iteration (0 before the
// first, then of this one), beta, alpha; [nbox] each.

// A p at cell c (the operator; D stored on FP64 levels, element cf)
__device__ __forceinline__ double apply_at(const double *__restrict__ p,
                                           const Box<double> &B, long long c, long long cf)
{
    double s = fma(B.wx[c], p[c - 1], -B.D[cf] * p[c]);
    s = fma(B.wx[c + 1], p[c + 1], s);
    s = fma(B.wy[c], p[c - B.P], s);
    s = fma(B.wy[c + B.P], p[c + B.P], s);
    s = fma(B.wz[c], p[c - B.Q], s);
    return fma(B.wz[c + B.Q], p[c + B.Q], s);
}

// op 0: partials of <f, phi> (= <r, z>);
// op 1: p = z + beta p;
// op 2: q = A p, partials of <p, q> (a launch of its own: A p reads the
//       neighbours' p of op 1);
// op 3: x += alpha p, r -= alpha q, partials of <r, r>, phi = the next
//       V-cycle's start (z is dead once op 1 has used it): 0 with the first
//       red pass applied;
// op 4 (start): x = phi (the initial guess), r = f - A x, p = 0, partials
//       of <r, r>;
// op 5: phi = x (before a restart from the true residual);
// op 6: phi = the V-cycle's start (as op 3).
// The op is a template argument: a run-time one was tested for every cell.
// Partials per TK_COLZ tile (a thread per column of kColZ planes, whatever the
// size, and block_sum_ordered: on high-contrast coefficients CG turns a
// rounding of its dot products into a solution that differs by more than its
// error at the usual tolerances, so their order stays what it was).
template <int op>
__global__ void __launch_bounds__(kThreads) k_pcg(BoxSet<double> S, const int *__restrict__ active,
                                                  double *const *__restrict__ pv,
                                                  double *const *__restrict__ qv, PcgScalars sc,
                                                  double *__restrict__ partials)
{
    pdl_wait();
    const int t = blockIdx.x;
    const int *ts = S.tstart[TK_COLZ];
    const int b = find_box(ts, S.nbox, t);
    const Box<double> &B = S.boxes[b];
    if (active && !active[B.box]) return;
    TilePos p = tile_pos(TK_COLZ, B.nx, B.ny, B.nz, t - ts[b]);
    double *P = pv[B.box], *Qa = qv[B.box];
    double v = 0.0;
    if (p.x < B.nx && p.y < B.ny) {
        const int cz = col_depth(B), z0 = p.z * cz, z1 = min(z0 + cz, B.nz);
        const double be = op == 1 ? sc.beta[B.box] : 0.0, al = op == 3 ? sc.alpha[B.box] : 0.0;
        // the V-cycle's zero start with its first red pass applied (put_coarse)
        auto start = [&](int i, int j, int k, double r, long long cf) {
            return ((i + j + k + B.par) & 1) ? 0.0 : -r * B.invD[cf];
        };
        // a few planes' loads in flight before the first of their stores
        constexpr int N = op == 2 || op == 4 ? 2 : 4;
        for (int k0 = z0; k0 < z1; k0 += N) {
            double x0[N], x1[N], x2[N];
#pragma unroll
            for (int u = 0; u < N; ++u) {
                const int k = k0 + u;
                if (k >= z1) break;
                const long long c = (long long)k * B.Q + (long long)p.y * B.P + p.x;
                const long long cf = fidx(B, p.x, p.y, k);
                if (op == 0) {
                    x0[u] = B.f[cf];
                    x1[u] = B.phi[c];
                } else if (op == 1) {
                    x0[u] = P[c];
                    x1[u] = B.phi[c];
                } else if (op == 2) {
                    x0[u] = apply_at(P, B, c, cf);
                    x1[u] = P[c];
                } else if (op == 3) {
                    x0[u] = fma(al, P[c], B.phi2[c]);
                    x1[u] = fma(-al, Qa[c], B.f[cf]);
                    x2[u] = start(p.x, p.y, k, x1[u], cf);
                } else if (op == 4) {
                    x0[u] = B.phi[c];
                    x1[u] = residual_at<double, true>(B.phi, B.f, B.wx, B.wy, B.wz, B.D, c, cf,
                                                      B.P, B.Q);
                } else if (op == 5) {
                    x0[u] = B.phi2[c];
                } else {
                    x0[u] = start(p.x, p.y, k, B.f[cf], cf);
                }
            }
#pragma unroll
            for (int u = 0; u < N; ++u) {
                const int k = k0 + u;
                if (k >= z1) break;
                const long long c = (long long)k * B.Q + (long long)p.y * B.P + p.x;
                const long long cf = fidx(B, p.x, p.y, k);
                if (op == 0) {
                    v = fma(x0[u], x1[u], v);
                } else if (op == 1) {
                    P[c] = fma(be, x0[u], x1[u]);
                } else if (op == 2) {
                    Qa[c] = x0[u];
                    v = fma(x1[u], x0[u], v);
                } else if (op == 3) {
                    B.phi2[c] = x0[u];
                    B.f[cf] = x1[u];
                    B.phi[c] = x2[u];
                    v = fma(x1[u], x1[u], v);
                } else if (op == 4) {
                    B.phi2[c] = x0[u];
                    B.f[cf] = x1[u];
                    P[c] = 0.0;
                    v = fma(x1[u], x1[u], v);
                } else {
                    B.phi[c] = x0[u];
                }
            }
        }
    }
    if (op != 1 && op < 5) {
        const double sum = block_sum_ordered(v);
        if (threadIdx.x == 0 && threadIdx.y == 0) partials[t] = sum;
    }
}

// Mixed-precision preconditioner (the FP32 V-cycle applied to the FP64 r):
// op 0: the FP32 right-hand side r / ||r|| and the FP32 cycle's start;
// op 1: z = ||r|| e, the FP32 solution scaled back into the FP64 phi.
// nrm: ||r|| per box (the last CG update's, or the start's).
__global__ void __launch_bounds__(kThreads) k_pcg_mixed(BoxSet<double> S64, BoxSet<float> S32,
                                                        const int *__restrict__ active, int op,
                                                        const double *__restrict__ nrm)
{
    pdl_wait();
    const int t = blockIdx.x;
    const int *ts = S64.tstart[TK_CELL];
    const int b = find_box(ts, S64.nbox, t);
    const Box<double> &B = S64.boxes[b];
    const Box<float> &E = S32.boxes[b];
    if (active && !active[B.box]) return;
    TilePos p = tile_pos(TK_CELL, B.nx, B.ny, B.nz, t - ts[b]);
    if (p.x >= B.nx || p.y >= B.ny) return;
    const long long c = (long long)p.z * B.Q + (long long)p.y * B.P + p.x;
    const double s = nrm[B.box];
    if (op == 0) {
        const float r = s > 0.0 ? (float)(B.f[fidx(B, p.x, p.y, p.z)] / s) : 0.0f;
        E.f[c] = r;
        // (the zero start with its first red pass applied, as in k_pcg)
        E.phi[c] = ((p.x + p.y + p.z + E.par) & 1) ? 0.0f : -r * E.invD[c];
    } else {
        B.phi[c] = s * (double)E.phi[c];
    }
}

// One CTA per box: the sum of the box's partials (fixed order) and what the
// iteration takes from it.  op 0: <r, z>, so beta = it / rz (0 on the first
// iteration) and rz = it; op 2: <p, q>, alpha = rz / it; op 3, 4: out = its
// square root.
template <int op>
__global__ void __launch_bounds__(1024) k_pcg_finish(BoxSet<double> S, const int *__restrict__ active,
                                                     const double *__restrict__ partials,
                                                     PcgScalars sc, double *__restrict__ out)
{
    pdl_wait();
    const int b = blockIdx.x;
    const int box = S.boxes[b].box;
    if (active && !active[box]) return;
    const int *ts = S.tstart[TK_COLZ];
    double s = 0.0;
    for (int q = ts[b] + (int)threadIdx.x; q < ts[b + 1]; q += 1024) s += partials[q];
    // (the order of the sums is fixed for good: see block_sum_ordered)
    __shared__ double wsum[32];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) wsum[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x != 0) return;
    double tot = 0.0;
    for (int w = 0; w < 32; ++w) tot += wsum[w];
    if (op == 0) {
        const double rz = sc.rz[box];
        sc.beta[box] = rz != 0.0 ? tot / rz : 0.0;
        sc.rz[box] = tot;
    } else if (op == 2) {
        sc.alpha[box] = tot != 0.0 ? sc.rz[box] / tot : 0.0;
    } else {
        out[box] = sqrt(tot);
    }
}

// ---------------------------------------------------- coupled levels ----
//
// The boxes of a coupled level (one MultiFAB level, paper Sec. 2, solved as
// one domain) keep their arrays in the wide layout.  Before every kernel
// that reads a neighbour of a box's cell, the guard cells that face another
// box receive that box's current values (ghost exchange, one CTA per
// intersection patch); the other guard cells stay 0, the Dirichlet walls of
// the union.

template <class T>
__global__ void __launch_bounds__(kThreads) k_exchange(BoxSet<T> S, const int *__restrict__ active,
                                                       const ExchRec *__restrict__ rec, int second)
{
    pdl_wait();
    if (active && !active[0]) return;   // one decision for the whole level
    const ExchRec R = rec[blockIdx.x];
    const Box<T> &D = S.boxes[R.dst];
    const Box<T> &F = S.boxes[R.src];
    T *__restrict__ dphi = second ? D.phi2 : D.phi;          // second: the phi2 arrays
    const T *__restrict__ fphi = second ? F.phi2 : F.phi;
    const int n = R.ex * R.ey * R.ez;
    const int stride = kThreads * gridDim.y;  // a record's cells over gridDim.y CTAs
    for (int e = blockIdx.y * kThreads + threadIdx.y * kTX + threadIdx.x; e < n; e += stride) {
        const int a = e % R.ex, r = e / R.ex;
        const int bb = r % R.ey, c = r / R.ey;
        dphi[(long long)(R.dk + c) * D.Q + (long long)(R.dj + bb) * D.P + R.di + a] =
            fphi[(long long)(R.sk + c) * F.Q + (long long)(R.sj + bb) * F.P + R.si + a];
    }
}

// The guard cells of the six faces of every box (CTA (box, face)) = v.
template <class T>
__global__ void __launch_bounds__(kThreads) k_guard_fill(BoxSet<T> S, T v)
{
    const Box<T> &B = S.boxes[blockIdx.x];
    const int face = blockIdx.y;
    const int nx = B.nx, ny = B.ny, nz = B.nz;
    const int ea = face < 2 ? ny : nx, eb = face < 4 ? nz : ny;
    for (int e = threadIdx.y * kTX + threadIdx.x; e < ea * eb; e += kThreads) {
        const int a = e % ea, b = e / ea;
        int i, j, k;
        if (face < 2) { i = face ? nx : -1; j = a; k = b; }
        else if (face < 4) { i = a; j = face == 3 ? ny : -1; k = b; }
        else { i = a; j = b; k = face == 5 ? nz : -1; }
        B.phi[(long long)k * B.Q + (long long)j * B.P + i] = v;
    }
}

// Dense inverse of the union of the boxes' coarsest levels (one cluster): each
// box's block as for a single box, plus -w between a box's cell and the cell
// of the neighbouring box (or, on a periodic axis, of the box itself) across
// every exchanged face (from the coarsest level's exchange records: guard
// cell of dst <-> cell of src), then Gauss-Jordan (with the constant shift
// when A is singular).  S: the coarsest level of every box, in union order.
__global__ void __launch_bounds__(kInvThreads) k_union_inverse(SetupSet S, UnionBottom U, double *a,
                                                               double *inv64, float *inv32,
                                                               int smem_bytes)
{
    extern __shared__ __align__(16) unsigned char inv_smem[];
    __shared__ double ips[2];
    const cg::cluster_group cl = cg::this_cluster();
    double *const sd = reinterpret_cast<double *>(inv_smem);
    const InvRows<double> M = inv_rows<double>(cl, U.n, sd, smem_bytes, a);
    for (int b = 0; b < U.nbox; ++b) {
        const SetupBox &B = S.boxes[b];
        assemble_box_block(B.nx, B.ny, B.nz, B.P, B.Q, B.wx, B.wy, B.wz, M, U.off[b]);
    }
    __syncthreads();
    for (int q = 0; q < U.nrec; ++q) {
        const ExchRec R = U.rec[q];
        const SetupBox &D = S.boxes[R.dst];
        const SetupBox &F = S.boxes[R.src];
        const int m = R.ex * R.ey * R.ez;
        for (int e = threadIdx.x; e < m; e += blockDim.x) {
            const int x = e % R.ex, r = e / R.ex;
            const int y = r % R.ey, z = r / R.ey;
            int gi = R.di + x, gj = R.dj + y, gk = R.dk + z;  // guard cell of dst
            const int si = R.si + x, sj = R.sj + y, sk = R.sk + z;
            // the dst cell next to the guard, and the weight of the face between
            int ci = min(max(gi, 0), D.nx - 1), cj = min(max(gj, 0), D.ny - 1),
                ck = min(max(gk, 0), D.nz - 1);
            const long long c = (long long)ck * D.Q + (long long)cj * D.P + ci;
            double w;
            if (gi < 0) w = D.wx[c];
            else if (gi >= D.nx) w = D.wx[c + 1];
            else if (gj < 0) w = D.wy[c];
            else if (gj >= D.ny) w = D.wy[c + D.P];
            else if (gk < 0) w = D.wz[c];
            else w = D.wz[c + D.Q];
            const int row = U.off[R.dst] + (ck * D.ny + cj) * D.nx + ci;
            const int col = U.off[R.src] + (sk * F.ny + sj) * F.nx + si;
            // added, not set: across a periodic axis of 2 cells the same two
            // cells are also neighbours through the inner face
            if (col >= row) {
                double *r = M.own(row);
                if (r) r[col - row] -= w;
            }
        }
        __syncthreads();
    }
    gauss_jordan_cluster<double>(cl, M, U.singular != 0, inv64, inv32, sd, ips);
}

// Coarsest solve of a coupled level: phi = Ainv f over the union, rows in
// chunks of 32 per CTA (grid y).  S: coarsest level of every box in union
// order.
template <class T>
__global__ void __launch_bounds__(kThreads) k_union_bottom(BoxSet<T> S, UnionBottom U,
                                                           const T *__restrict__ ainv,
                                                           const int *__restrict__ active)
{
    pdl_wait();
    __shared__ T fs[MG_BOTTOM_CELLS];
    if (active && !active[0]) return;
    const int n = U.n;
    const int tid = threadIdx.y * kTX + threadIdx.x;
    auto locate = [&](int q, int &b, long long &c, long long &cf) {
        b = find_box(U.off, U.nbox, q);
        const Box<T> &B = S.boxes[b];
        const int r = q - U.off[b];
        const int i = r % B.nx, j = (r / B.nx) % B.ny, k = r / (B.nx * B.ny);
        c = (long long)k * B.Q + (long long)j * B.P + i;
        cf = fidx(B, i, j, k);
    };
    for (int q = tid; q < n; q += kThreads) {
        int b;
        long long c, cf;
        locate(q, b, c, cf);
        fs[q] = S.boxes[b].f[cf];
    }
    __syncthreads();
    const int lane = threadIdx.x, warp = threadIdx.y;
    for (int rr = 0; rr < 4; ++rr) {
        const int r = blockIdx.x * 32 + warp * 4 + rr;
        if (r >= n) break;
        const T *row = ainv + (long long)r * n;
        T acc = T(0);
        for (int q = lane; q < n; q += 32) acc = fmadd(row[q], fs[q], acc);
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
        if (lane == 0) {
            int b;
            long long c, cf;
            locate(r, b, c, cf);
            S.boxes[b].phi[c] = acc;
        }
    }
}

// A coupled level has one residual norm: norm[b] <- sqrt(sum over boxes of
// norm[b]^2) for every box (a fixed-order sum by one thread).
__global__ void k_norm_combine(int nbox, double *__restrict__ norm)
{
    pdl_wait();
    __shared__ double tot;
    if (threadIdx.x == 0) {
        double s = 0.0;
        for (int b = 0; b < nbox; ++b) s += norm[b] * norm[b];
        tot = sqrt(s);
    }
    __syncthreads();
    for (int b = threadIdx.x; b < nbox; b += blockDim.x) norm[b] = tot;
}

// ------------------------------------ right-hand sides of one box ----
//
// A batch whose boxes are right-hand sides of one box (mg_solve_multi,
// mg_adjoint with several right-hand sides) has one set of weights, 1/D and
// D for all of them.  These pass variants take a tile of box 0's index
// space and update the same cells in every active right-hand side, so the
// six weights and 1/D of a cell are read once for all of them: an FP64 pass
// then moves 16 + 28 / nrhs bytes a cell and right-hand side (phi's sectors,
// half of f, half of phi written) instead of 44.  The arithmetic per cell is
// that of k_rbgs_pass / k_rbgs_pass_oop, in the same order.

template <class T>
__global__ void __launch_bounds__(kThreads) k_rbgs_pass_multi(BoxSet<T> S,
                                                              const int *__restrict__ active,
                                                              int color)
{
    pdl_wait();
    const Box<T> &B0 = S.boxes[0];
    const int P = B0.P;
    const long long Q = B0.Q;
    const TilePos p = tile_pos(TK_PAIR, B0.nx, B0.ny, B0.nz, tile_dir(color != 0));
    const int j = p.y, k = p.z;
    const int i = 2 * p.x + ((j + k + color + B0.par) & 1);
    if (j >= B0.ny || i >= B0.nx) return;
    const long long c = (long long)k * Q + (long long)j * P + i;
    const long long cf =
        split_on(B0) ? (long long)k * Q + (long long)j * P + (color ? (P >> 1) : 0) + p.x : c;
    const T wxa = B0.wx[c], wxb = B0.wx[c + 1], wya = B0.wy[c], wyb = B0.wy[c + P],
            wza = B0.wz[c], wzb = B0.wz[c + Q], id = B0.invD[cf];
#pragma unroll 2
    for (int r = 0; r < S.nbox; ++r) {
        const Box<T> &B = S.boxes[r];
        if (active && !active[B.box]) continue;
        const T *__restrict__ ph = B.phi;
        T s = fmadd(wxa, ph[c - 1], -B.f[cf]);
        s = fmadd(wxb, ph[c + 1], s);
        s = fmadd(wya, ph[c - P], s);
        s = fmadd(wyb, ph[c + P], s);
        s = fmadd(wza, ph[c - Q], s);
        B.phi[c] = fmadd(wzb, ph[c + Q], s) * id;
    }
}

// One colour out of place (as k_rbgs_pass_oop) in every right-hand side.
template <class T>
__global__ void __launch_bounds__(kThreads) k_rbgs_pass_oop_multi(BoxSet<T> S,
                                                                  const int *__restrict__ active,
                                                                  int color, int from2)
{
    pdl_wait();
    const Box<T> &B0 = S.boxes[0];
    const int P = B0.P;
    const long long Q = B0.Q;
    const TilePos p = tile_pos(TK_PAIR, B0.nx, B0.ny, B0.nz, tile_dir(color != 0));
    const int j = p.y, k = p.z, x0 = 2 * p.x;
    if (j >= B0.ny || x0 >= B0.nx) return;
    typedef typename Vec2<T>::type V2;
    const long long c0 = (long long)k * Q + (long long)j * P + x0;
    const int odd = (j + k + color + B0.par) & 1;
    const bool upd = x0 + odd < B0.nx;
    const long long c = c0 + odd;
    const long long cf =
        split_on(B0) ? (long long)k * Q + (long long)j * P + (color ? (P >> 1) : 0) + (x0 >> 1)
                     : c;
    T wxa = 0, wxb = 0, wya = 0, wyb = 0, wza = 0, wzb = 0, id = 0;
    if (upd) {
        wxa = B0.wx[c];
        wxb = B0.wx[c + 1];
        wya = B0.wy[c];
        wyb = B0.wy[c + P];
        wza = B0.wz[c];
        wzb = B0.wz[c + Q];
        id = B0.invD[cf];
    }
#pragma unroll 2
    for (int r = 0; r < S.nbox; ++r) {
        const Box<T> &B = S.boxes[r];
        if (active && !active[B.box]) continue;
        const T *__restrict__ src = from2 ? B.phi2 : B.phi;
        T *__restrict__ dst = from2 ? B.phi : B.phi2;
        V2 pair = *reinterpret_cast<const V2 *>(src + c0);
        if (upd) {
            T s = fmadd(wxa, src[c - 1], -B.f[cf]);
            s = fmadd(wxb, src[c + 1], s);
            s = fmadd(wya, src[c - P], s);
            s = fmadd(wyb, src[c + P], s);
            s = fmadd(wza, src[c - Q], s);
            s = fmadd(wzb, src[c + Q], s);
            const T nv = s * id;
            if (odd) pair.y = nv;
            else pair.x = nv;
        }
        *reinterpret_cast<V2 *>(dst + c0) = pair;
    }
}

// ------------------------------------------- persistent level sweeps ----
//
// The many boxes of a batch (the grids of one MultiFAB level, paper Sec. 2)
// walk a level's stages together.  Instead of one launch per stage, a level
// is smoothed by one launch going down (the pre-smoothing passes, then the
// residual and restriction) and one coming up (prolongation, then the
// post-smoothing passes).  The launch is persistent: its grid is at most the
// number of CTAs that can be resident at once (a cooperative launch, so the
// runtime refuses a grid that could not be), each CTA walks the tiles of
// every active box of a stage with a grid-sized stride, and a grid-wide
// barrier separates consecutive stages.  The barrier is bounded: a CTA that
// has polled it `polls` times without seeing it complete sets the error
// word and returns, so a failure (or a forced time-out) ends the launch with
// an error the host reports as MG_ERR_TIMEOUT, never a hang.

// The barrier (GridSync, kernels.h): one 32-bit word in device memory, zero
// when a solve starts.  Every CTA adds 1 except CTA 0, which adds
// 2^31 - (G - 1): when all G have arrived the word has grown by exactly
// 2^31, so its top bit has flipped and its low bits are back where they
// were -- the next barrier starts from there without a reset.
__device__ __forceinline__ bool grid_sync(const GridSync &g)
{
    __shared__ int ok_s;
    __syncthreads();
    if (threadIdx.x == 0 && threadIdx.y == 0) {
        const unsigned add = blockIdx.x == 0 ? 0x80000000u - (gridDim.x - 1u) : 1u;
        __threadfence();   // this CTA's stage results before its arrival
        const unsigned old = atomicAdd(g.word, add);
        const volatile unsigned *w = g.word;
        int ok = 1;
        long long i = 0;
        while (((old ^ *w) & 0x80000000u) == 0u) {
            if (i++ >= g.polls) {
                ok = 0;
                atomicExch(g.err, 1);
                break;
            }
            __nanosleep(32);
        }
        __threadfence();   // the other CTAs' results after the barrier
        ok_s = ok;
    }
    __syncthreads();
    return ok_s != 0;
}

// One tile of an in-place single-colour pass (as k_rbgs_pass).
template <class T>
__device__ __forceinline__ void pass_tile(const BoxSet<T> &S, const int *__restrict__ active,
                                          int color, int t)
{
    const int *ts = S.tstart[TK_PAIR];
    const int b = find_box(ts, S.nbox, t);
    const Box<T> &B = S.boxes[b];
    if (active && !active[B.box]) return;
    const int P = B.P;
    const long long Q = B.Q;
    const TilePos p = tile_pos(TK_PAIR, B.nx, B.ny, B.nz, t - ts[b]);
    const int j = p.y, k = p.z;
    const int i = 2 * p.x + ((j + k + color + B.par) & 1);
    if (j >= B.ny || i >= B.nx) return;
    const long long c = (long long)k * Q + (long long)j * P + i;
    const long long cf =
        split_on(B) ? (long long)k * Q + (long long)j * P + (color ? (P >> 1) : 0) + p.x : c;
    B.phi[c] = gs_value<T>(B.phi, B.f, B.invD, B.wx, B.wy, B.wz, c, cf, P, Q);
}

// One tile of the black pass out of place, phi2 -> phi (the rest of the
// finest level's first sweep after the look-ahead red pass).
template <class T>
__device__ __forceinline__ void pass_oop_tile(const BoxSet<T> &S, const int *__restrict__ active,
                                              int t)
{
    const int *ts = S.tstart[TK_PAIR];
    const int b = find_box(ts, S.nbox, t);
    const Box<T> &B = S.boxes[b];
    if (active && !active[B.box]) return;
    const TilePos p = tile_pos(TK_PAIR, B.nx, B.ny, B.nz, t - ts[b]);
    double unused = 0.0;
    if (p.y < B.ny && 2 * p.x < B.nx) oop_pair(B, 1, 1, p.y, p.z, 2 * p.x, false, unused);
}

// Work item q of a ghost exchange: record q % nrec, chunk q / nrec of
// `chunks` (as k_exchange with gridDim.y = chunks).
template <class T>
__device__ __forceinline__ void exchange_item(const BoxSet<T> &S, const ExchRec *__restrict__ rec,
                                              int nrec, int chunks, int q, int second)
{
    const ExchRec R = rec[q % nrec];
    const int chunk = q / nrec;
    const Box<T> &D = S.boxes[R.dst];
    const Box<T> &F = S.boxes[R.src];
    T *__restrict__ dphi = second ? D.phi2 : D.phi;
    const T *__restrict__ fphi = second ? F.phi2 : F.phi;
    const int n = R.ex * R.ey * R.ez;
    const int stride = kThreads * chunks;
    for (int e = chunk * kThreads + threadIdx.y * kTX + threadIdx.x; e < n; e += stride) {
        const int a = e % R.ex, r = e / R.ex;
        const int bb = r % R.ey, c = r / R.ey;
        dphi[(long long)(R.dk + c) * D.Q + (long long)(R.dj + bb) * D.P + R.di + a] =
            fphi[(long long)(R.sk + c) * F.Q + (long long)(R.sj + bb) * F.P + R.si + a];
    }
}

// A launch that finds the error word set (a barrier of an earlier launch in
// this solve gave up, leaving the barrier word mid-count) does nothing.
__device__ __forceinline__ bool grid_failed(const GridSync &g)
{
    return *reinterpret_cast<const volatile int *>(g.err) != 0;
}

template <class T>
__global__ void __launch_bounds__(kThreads, 3) k_level_down(BoxSet<T> S, const int *__restrict__ active,
                                                         LevelOps op, GridSync g)
{
    if (grid_failed(g)) return;
    auto each = [&](int n, auto &&work) {
        for (int t = blockIdx.x; t < n; t += gridDim.x) work(t);
    };
    auto exchange = [&](int second) -> bool {
        if (op.nrec == 0) return true;
        each(op.nrec * op.chunks,
             [&](int q) { exchange_item(S, op.rec, op.nrec, op.chunks, q, second); });
        return grid_sync(g);
    };
    const int npair = S.ntiles[TK_PAIR];
    int sweeps = op.nu;
    if (op.head_done) {
        if (!exchange(1)) return;
        each(npair, [&](int t) { pass_oop_tile(S, active, t); });
        if (!grid_sync(g)) return;
        --sweeps;
    }
    for (int sw = 0; sw < sweeps; ++sw)
        for (int color = 0; color < 2; ++color) {
            if (op.red_done && sw == 0 && color == 0) continue;
            if (!exchange(0)) return;
            each(npair, [&](int t) { pass_tile(S, active, color, t); });
            if (!grid_sync(g)) return;
        }
    if (!exchange(0)) return;
    const int nc = S.ntiles[TK_COARSE];
    if (op.red && op.partials) {
        if (op.flat) each(nc, [&](int t) { restrict_red_tile<T, true, true, true>(S, active, t, op.partials); });
        else each(nc, [&](int t) { restrict_red_tile<T, false, true, true>(S, active, t, op.partials); });
    } else if (op.red) {
        if (op.flat) each(nc, [&](int t) { restrict_red_tile<T, true, false, true>(S, active, t); });
        else each(nc, [&](int t) { restrict_red_tile<T, false, false, true>(S, active, t); });
    } else {
        if (op.flat) each(nc, [&](int t) { restrict_tile<T, true, true>(S, active, t); });
        else each(nc, [&](int t) { restrict_tile<T, false, true>(S, active, t); });
    }
}

template <class T>
__global__ void __launch_bounds__(kThreads, 4) k_level_up(BoxSet<T> S, const int *__restrict__ active,
                                                       LevelOps op, GridSync g)
{
    if (grid_failed(g)) return;
    auto each = [&](int n, auto &&work) {
        for (int t = blockIdx.x; t < n; t += gridDim.x) work(t);
    };
    const int nc = S.ntiles[TK_COARSE];
    if (op.flat) each(nc, [&](int t) { prolong_tile<T, true>(S, active, t); });
    else each(nc, [&](int t) { prolong_tile<T, false>(S, active, t); });
    const int npair = S.ntiles[TK_PAIR];
    for (int sw = 0; sw < op.nu; ++sw)
        for (int c = 0; c < 2; ++c) {
            if (!grid_sync(g)) return;
            if (op.nrec) {
                each(op.nrec * op.chunks,
                     [&](int q) { exchange_item(S, op.rec, op.nrec, op.chunks, q, 0); });
                if (!grid_sync(g)) return;
            }
            const int color = op.reverse ? 1 - c : c;
            each(npair, [&](int t) { pass_tile(S, active, color, t); });
        }
}

// ----------------------------------- coarsest level by conjugate gradients ----
//
// A box whose halving stops at a level too large for a dense inverse (more
// than MG_MAX_BOTTOM cells: a 33^3 box, or 100^3, whose coarsest level is
// 25^3) solves that level by conjugate gradients preconditioned with its
// diagonal, on M = -A (symmetric positive definite): x = phi, r = phi2, and
// two more level arrays p, q.  One persistent cooperative launch runs the
// whole iteration; each of its three stages per iteration ends at the
// bounded grid barrier of the persistent level sweeps, and every dot product
// is summed in a fixed order (per-CTA partial sums, then each CTA adds the
// partials 0 .. G-1), so every CTA takes the same decisions and the result
// is reproducible.  It stops when <r, D^-1 r> has fallen by tol^2, after
// maxit iterations, when 200 iterations in a row have not lowered it below
// its smallest value so far (rounding has stalled it), or if <p, M p> is
// not positive.

// (M v)_c = D_c v_c - sum_f w_f v_nbr: minus the operator, zero outside.
template <class T>
__device__ __forceinline__ T neg_apply(const Box<T> &B, const T *__restrict__ v, long long c,
                                       long long cf)
{
    const T a = B.wx[c], b = B.wx[c + 1], d = B.wy[c], e = B.wy[c + B.P], g = B.wz[c],
            h = B.wz[c + B.Q];
    const T D = B.D ? B.D[cf] : ((a + b) + (d + e)) + (g + h);
    T s = D * v[c];
    s = fmadd(-a, v[c - 1], s);
    s = fmadd(-b, v[c + 1], s);
    s = fmadd(-d, v[c - B.P], s);
    s = fmadd(-e, v[c + B.P], s);
    s = fmadd(-g, v[c - B.Q], s);
    return fmadd(-h, v[c + B.Q], s);
}

// Fixed-order sum of the G partials (every CTA gets the same bits).
__device__ __forceinline__ double sum_partials(const double *__restrict__ part, int G)
{
    __shared__ double tot;
    double v = 0.0;
    if (threadIdx.y == 0) {
        for (int i = threadIdx.x; i < G; i += kTX) v += part[i];
        for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
        if (threadIdx.x == 0) tot = v;
    }
    __syncthreads();
    const double r = tot;
    __syncthreads();
    return r;
}

template <class T>
__global__ void __launch_bounds__(kThreads) k_cg_bottom(BoxSet<T> S, const int *__restrict__ active,
                                                        T *p, T *q, double *part, GridSync g,
                                                        double tol, int maxit)
{
    const Box<T> &B = S.boxes[0];
    if ((active && !active[B.box]) || grid_failed(g)) return;
    const int nt = S.ntiles[TK_CELL], G = gridDim.x;
    double *pa = part, *pb = part + G;
    const int nx = B.nx, ny = B.ny, nz = B.nz;
    T *__restrict__ x = B.phi;
    T *__restrict__ r = B.phi2;
    // each stage walks the level's cells tile by tile
    auto cells = [&](auto &&body) {
        for (int t = blockIdx.x; t < nt; t += G) {
            const TilePos tp = tile_pos(TK_CELL, nx, ny, nz, t);
            if (tp.x < nx && tp.y < ny)
                body((long long)tp.z * B.Q + (long long)tp.y * B.P + tp.x, fidx(B, tp.x, tp.y, tp.z));
        }
    };
    auto put = [&](double *dst, double v) {
        const double bs = block_sum_ordered(v);
        if (threadIdx.x == 0 && threadIdx.y == 0) dst[blockIdx.x] = bs;
    };
    // x = 0, r = -f, p = D^-1 r, partial <r, D^-1 r>
    double acc = 0.0;
    cells([&](long long c, long long cf) {
        const T rv = -B.f[cf];
        const T zv = rv * B.invD[cf];
        x[c] = T(0);
        r[c] = rv;
        p[c] = zv;
        acc += (double)rv * (double)zv;
    });
    put(pb, acc);
    if (!grid_sync(g)) return;
    double rz = sum_partials(pb, G);
    const double rz0 = rz, stop = tol * tol * rz0;
    if (!(rz0 > 0.0)) return;   // f = 0 on this level: x = 0
    double best = rz0;
    int since = 0;
    for (int it = 0; it < maxit; ++it) {
        // q = M p, partial <p, q>
        acc = 0.0;
        cells([&](long long c, long long cf) {
            const T qv = neg_apply(B, p, c, cf);
            q[c] = qv;
            acc += (double)p[c] * (double)qv;
        });
        put(pa, acc);
        if (!grid_sync(g)) return;
        const double pq = sum_partials(pa, G);
        if (!(pq > 0.0)) return;
        const T alpha = (T)(rz / pq);
        // x += alpha p, r -= alpha q, partial <r, D^-1 r>
        acc = 0.0;
        cells([&](long long c, long long cf) {
            x[c] = fmadd(alpha, p[c], x[c]);
            const T rv = fmadd(-alpha, q[c], r[c]);
            r[c] = rv;
            acc += (double)rv * (double)(rv * B.invD[cf]);
        });
        put(pb, acc);
        if (!grid_sync(g)) return;
        const double rz1 = sum_partials(pb, G);
        if (rz1 <= stop) return;
        if (rz1 < best) {
            best = rz1;
            since = 0;
        } else if (++since >= 200) {
            return;
        }
        const T beta = (T)(rz1 / rz);
        rz = rz1;
        // p = D^-1 r + beta p
        cells([&](long long c, long long cf) { p[c] = fmadd(beta, p[c], r[c] * B.invD[cf]); });
        if (!grid_sync(g)) return;
    }
}

// The same iteration, the same bits, by one cluster when the level has at most
// 16 x 2 cell tiles: a thread holds its cell's x, r, weights and 1/D in
// registers through the solve, only p is in memory, a tile's partial sums go
// into every CTA through distributed shared memory, and the three barriers of
// an iteration are the cluster's.  What bounds it: the barriers, the dependent
// FP64 sums (8 + 5 + 5 of ~100 cycles), p's round trip through L2 and the
// FP64 pipes of 16 SMs, which set the line: FP64 solves of 36 x 52 x 44 cells
// (11 tiles) 7.1 -> 4.0 ms, 13 x 9 x 9 (13) 0.74 -> 0.46, 104 x 120 x 152 (26)
// 13.1 -> 10.6; with four tiles a CTA 168 x 176 x 240 (60 tiles) took 26.8 ms
// against 24.6 and 64 x 17 x 15 (64) 2.2 against 1.8.
constexpr int kCgCtas = 16, kCgGroups = 2;

template <class T>
__global__ void __launch_bounds__(kThreads *kCgGroups)
    k_cg_bottom_cluster(BoxSet<T> S, const int *__restrict__ active, T *p, double tol, int maxit)
{
    const cg::cluster_group cl = cg::this_cluster();
    const Box<T> &B = S.boxes[0];
    if (active && !active[B.box]) return;
    __shared__ double wpart[kThreads / 32 * kCgGroups], part[2][kCgCtas * kCgGroups], tot;
    const int nt = S.ntiles[TK_CELL], CL = (int)cl.num_blocks();
    const int t = (int)threadIdx.z * CL + (int)cl.block_rank();
    const int warp = (int)threadIdx.z * kTY + (int)threadIdx.y, lane = threadIdx.x;
    const TilePos tp = tile_pos(TK_CELL, B.nx, B.ny, B.nz, t);
    const bool on = t < nt && tp.x < B.nx && tp.y < B.ny;
    const int P = B.P;
    const long long Q = B.Q;
    const long long c = on ? (long long)tp.z * Q + (long long)tp.y * P + tp.x : 0;
    // the sum over all cells of v, in the order of the cooperative launch with
    // one tile a CTA (w: which of two buffers, used in turn)
    auto total = [&](double v, int w) {
        for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
        if (lane == 0) wpart[warp] = v;
        __syncthreads();
        if (threadIdx.y == 0 && t < nt) {
            double s = 0.0;
            for (int i = 0; i < kThreads / 32; ++i) s += wpart[warp + i];
            if (lane < CL) cl.map_shared_rank(&part[w][0], lane)[t] = s;
        }
        cl.sync();
        if (warp == 0) {
            double s = 0.0;
            for (int i = lane; i < nt; i += 32) s += part[w][i];
            for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
            if (lane == 0) tot = s;
        }
        __syncthreads();
        return tot;
    };
    T wxa = 0, wxb = 0, wya = 0, wyb = 0, wza = 0, wzb = 0, D = 0, id = 0, x = 0, r = 0, pc = 0;
    if (on) {
        const long long cf = fidx(B, tp.x, tp.y, tp.z);
        wxa = B.wx[c];
        wxb = B.wx[c + 1];
        wya = B.wy[c];
        wyb = B.wy[c + P];
        wza = B.wz[c];
        wzb = B.wz[c + Q];
        D = B.D ? B.D[cf] : ((wxa + wxb) + (wya + wyb)) + (wza + wzb);
        id = B.invD[cf];
        r = -B.f[cf];
        pc = r * id;
        p[c] = pc;
    }
    cl.sync();   // every CTA runs before its shared memory is written
    double rz = total((double)r * (double)pc, 1);
    const double stop = tol * tol * rz;
    double best = rz;
    int since = 0;
    for (int it = 0; it < maxit && rz > 0.0; ++it) {
        T q = 0;
        if (on) {
            q = D * pc;
            q = fmadd(-wxa, __ldcg(p + c - 1), q);
            q = fmadd(-wxb, __ldcg(p + c + 1), q);
            q = fmadd(-wya, __ldcg(p + c - P), q);
            q = fmadd(-wyb, __ldcg(p + c + P), q);
            q = fmadd(-wza, __ldcg(p + c - Q), q);
            q = fmadd(-wzb, __ldcg(p + c + Q), q);
        }
        const double pq = total((double)pc * (double)q, 0);
        if (!(pq > 0.0)) break;
        const T alpha = (T)(rz / pq);
        x = fmadd(alpha, pc, x);
        r = fmadd(-alpha, q, r);
        const double rz1 = total((double)r * (double)(r * id), 1);
        if (rz1 <= stop) break;
        if (rz1 < best) {
            best = rz1;
            since = 0;
        } else if (++since >= 200) {
            break;
        }
        const T beta = (T)(rz1 / rz);
        rz = rz1;
        pc = fmadd(beta, pc, r * id);
        if (on) p[c] = pc;
        cl.sync();
    }
    if (on) B.phi[c] = x;
}

// ----------------------------------------------------------- launchers ----

static inline dim3 block2d() { return dim3(kTX, kTY); }

template <class T>
cudaError_t launch_rbgs_pass_oop(const BoxSet<T> &S, const int *active, int color, int from2,
                                 double *partials, cudaStream_t st)
{
    if (partials) {
        if (S.ntiles[TK_PCOLZ] == 0) return cudaSuccess;
        return pdl_launch(k_rbgs_pass_oop_norm<T>, dim3(S.ntiles[TK_PCOLZ]), block2d(), 0, st, S,
                          active, color, from2, partials);
    }
    if (S.ntiles[TK_PAIR] == 0) return cudaSuccess;
    return pdl_launch(k_rbgs_pass_oop<T>, dim3(S.ntiles[TK_PAIR]), block2d(), 0, st, S, active,
                      color, from2);
}

template <class T>
cudaError_t launch_rbgs_pass(const BoxSet<T> &S, const int *active, int color, cudaStream_t st,
                             bool push)
{
    if (S.ntiles[TK_PAIR] == 0) return cudaSuccess;
    return pdl_launch(push ? k_rbgs_pass<T, true> : k_rbgs_pass<T, false>, dim3(S.ntiles[TK_PAIR]), block2d(), 0, st, S, active, color);
}

template <class T>
int sweep_ctas_per_sm()
{
    int n = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_rbgs_sweep<T>, kSweepThreads, 0) !=
        cudaSuccess) {
        cudaGetLastError();
        return 4;
    }
    return n > 0 ? n : 1;
}
template int sweep_ctas_per_sm<double>();
template int sweep_ctas_per_sm<float>();

template <class T>
cudaError_t launch_rbgs_sweep(const BoxSet<T> &S, const int *active, int src_is_phi2,
                              cudaStream_t st)
{
    if (S.ntiles[TK_SWEEP] == 0) return cudaSuccess;
    return pdl_launch(k_rbgs_sweep<T>, dim3(S.ntiles[TK_SWEEP]), dim3(kTX, kSweepWarps), 0, st, S,
                      active, src_is_phi2);
}

template <class T>
cudaError_t launch_resid_restrict(const BoxSet<T> &S, const int *active, cudaStream_t st)
{
    if (S.ntiles[TK_COARSE] == 0) return cudaSuccess;
    const bool flat = S.flat & (1 << TK_COARSE);
    auto k = flat ? (S.fold ? k_resid_restrict<T, true, true> : k_resid_restrict<T, true, false>)
                  : (S.fold ? k_resid_restrict<T, false, true> : k_resid_restrict<T, false, false>);
    return pdl_launch(k, dim3(S.ntiles[TK_COARSE]), block2d(), 0, st, S, active);
}

template <class T>
cudaError_t launch_resid_restrict_red(const BoxSet<T> &S, const int *active, cudaStream_t st,
                                      double *partials)
{
    if (S.ntiles[TK_COARSE] == 0) return cudaSuccess;
    const bool flat = S.flat & (1 << TK_COARSE);
    auto pick = [&](auto norm, auto fold) {
        constexpr bool N = decltype(norm)::value, F = decltype(fold)::value;
        return flat ? k_resid_restrict_red<T, true, N, F> : k_resid_restrict_red<T, false, N, F>;
    };
    const std::true_type yes;
    const std::false_type no;
    auto k = partials ? (S.fold ? pick(yes, yes) : pick(yes, no))
                      : (S.fold ? pick(no, yes) : pick(no, no));
    return pdl_launch(k, dim3(S.ntiles[TK_COARSE]), block2d(), 0, st, S, active, partials);
}

cudaError_t launch_inner_judge(const BoxSet<float> &S, int *active32, const double *partials,
                               const int *cstart, int nchunks, int chunk_tiles, double *chunks,
                               const double *se, const double *sr, const double *normf,
                               const double *tol, double floor_rel, int coupled, cudaStream_t st)
{
    if (S.nbox == 0 || nchunks == 0) return cudaSuccess;
    cudaError_t e = pdl_launch(k_inner_sum, dim3(nchunks), dim3(256), 0, st, S, active32, cstart,
                               chunk_tiles, partials, chunks);
    if (e != cudaSuccess) return e;
    return pdl_launch(k_inner_judge, dim3(coupled ? 1 : S.nbox), dim3(1024), 0, st, S, active32,
                      cstart, chunks, se, sr, normf, tol, floor_rel, coupled);
}

template <class T>
cudaError_t launch_prolong(const BoxSet<T> &S, const int *active, cudaStream_t st)
{
    if (S.ntiles[TK_COARSE] == 0) return cudaSuccess;
    if (S.flat & (1 << TK_COARSE))
        return pdl_launch(k_prolong<T, true>, dim3(S.ntiles[TK_COARSE]), block2d(), 0, st,
                          S, active);
    return pdl_launch(k_prolong<T, false>, dim3(S.ntiles[TK_COARSE]), block2d(), 0, st, S,
                      active);
}

template <class T>
cudaError_t launch_residual_field(const BoxSet<T> &S, cudaStream_t st)
{
    if (S.ntiles[TK_CELL] == 0) return cudaSuccess;
    k_residual_field<T><<<S.ntiles[TK_CELL], block2d(), 0, st>>>(S);
    return counted(cudaGetLastError());
}

template <class T>
cudaError_t launch_norm_partials(const BoxSet<T> &S, const int *active, int mode, double *partials,
                                 cudaStream_t st)
{
    const int kind = mode == 2 ? TK_PCOLZ : TK_COLZ;
    if (S.ntiles[kind] == 0) return cudaSuccess;
    return pdl_launch(k_norm_partials<T>, dim3(S.ntiles[kind]), block2d(), 0, st, S, active, mode,
                      partials);
}

template <class T>
cudaError_t launch_norm_finish(const BoxSet<T> &S, const int *active, const double *partials,
                               double *out, double *copy, double *inv, cudaStream_t st,
                               const double *mult, int mode)
{
    if (S.nbox == 0) return cudaSuccess;
    // the partials' tile starts (the host picks the kind: a run-time index
    // into the kernel's parameter set would copy it to local memory)
    const int *ts = S.tstart[mode == 2 ? TK_PCOLZ : TK_COLZ];
    return pdl_launch(k_norm_finish<T>, dim3(S.nbox), dim3(1024), 0, st, S, active, partials, out,
                      copy, inv, mult, ts);
}

template <class T>
cudaError_t launch_bottom(const BoxSet<T> &S, const int *active, int max_cells, cudaStream_t st)
{
    if (S.nbox == 0) return cudaSuccess;
    dim3 grid(S.nbox, (max_cells + 31) / 32);
    k_bottom<T><<<grid, block2d(), 0, st>>>(S, active);
    return counted(cudaGetLastError());
}

// Clusters of cl CTAs of a kernel that can be resident at once (0: none); also
// allows the kernel such clusters and smem bytes of dynamic shared memory.
template <class K>
static int resident_clusters(K *k, int cl, dim3 block, size_t smem)
{
    if (cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess ||
        (smem > 0 && cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                          (int)smem) != cudaSuccess)) {
        cudaGetLastError();
        return 0;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(cl);
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = cl;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, k, &cfg) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return n;
}

template <class T>
int tail_clusters(int cl, size_t smem)
{
    return resident_clusters(k_coarse_vcycle<T>, cl, dim3(kTailThreads), smem);
}
template int tail_clusters<double>(int, size_t);
template int tail_clusters<float>(int, size_t);

template <class T>
cudaError_t launch_coarse_vcycle(const CoarseJob<T> *jobs, int njobs, int cl, size_t smem,
                                 const int *active, int nu1, int nu2, cudaStream_t st,
                                 int post_first)
{
    if (njobs == 0) return cudaSuccess;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(njobs * cl);
    cfg.blockDim = dim3(kTailThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = cl;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = pdl_enabled() ? 2 : 1;
    return counted(cudaLaunchKernelEx(&cfg, k_coarse_vcycle<T>, jobs, active, nu1, nu2, post_first));
}

cudaError_t launch_refine_update(const BoxSet<double> &S64, const BoxSet<float> &S32,
                                 const int *active, const double *c_e, cudaStream_t st)
{
    if (S64.ntiles[TK_CELL] == 0) return cudaSuccess;
    return pdl_launch(k_refine_update, dim3(S64.ntiles[TK_CELL]), block2d(), 0, st, S64, S32,
                      active, c_e);
}

cudaError_t launch_refine_residual(const BoxSet<double> &S64, const BoxSet<float> &S32,
                                   const int *active, const double *c_r_inv, double *partials,
                                   cudaStream_t st, bool x_zero)
{
    if (S64.ntiles[TK_COLZ] == 0) return cudaSuccess;
    if (x_zero)
        return pdl_launch(k_refine_residual<true>, dim3(S64.ntiles[TK_COLZ]), block2d(), 0, st,
                          S64, S32, active, c_r_inv, partials);
    return pdl_launch(k_refine_residual<false>, dim3(S64.ntiles[TK_COLZ]), block2d(), 0, st, S64,
                      S32, active, c_r_inv, partials);
}

cudaError_t launch_judge(int nbox, const double *norm, const double *normf, int *active,
                         const JudgeState &J, cudaGraphConditionalHandle handle, int use_handle,
                         cudaStream_t st)
{
    const int threads = nbox < 1024 ? ((nbox + 31) / 32) * 32 : 1024;
    return pdl_launch(k_judge, dim3(1), dim3(threads), 0, st, nbox, norm, normf, active, J,
                      handle, use_handle);
}

cudaError_t launch_norm_judge(const BoxSet<double> &S, const double *partials, double *norm,
                              const double *normf, int *active, const JudgeState &J,
                              cudaGraphConditionalHandle handle, cudaStream_t st)
{
    return pdl_launch(k_norm_judge, dim3(1), dim3(1024), 0, st, partials, norm, normf, active, J,
                      handle, S.tstart[TK_PCOLZ]);
}

cudaError_t launch_pack(const BoxSet<double> &S, const long long *off, const double *user,
                        int to_f, cudaStream_t st, double *partials)
{
    if (S.ntiles[TK_COLZ] == 0) return cudaSuccess;
    return pdl_launch(k_pack, dim3(S.ntiles[TK_COLZ]), block2d(), 0, st, S, off, user, to_f,
                      to_f ? partials : nullptr);
}

cudaError_t launch_unpack(const BoxSet<double> &S, const long long *off, double *user,
                          const int *side, cudaStream_t st)
{
    if (S.ntiles[TK_COLZ] == 0) return cudaSuccess;
    return pdl_launch(k_unpack, dim3(S.ntiles[TK_COLZ]), block2d(), 0, st, S, off, user, side);
}

template <class T>
cudaError_t launch_zero(const BoxSet<T> &S, const int *active, cudaStream_t st)
{
    if (S.ntiles[TK_COLZ] == 0) return cudaSuccess;
    return pdl_launch(k_zero<T>, dim3(S.ntiles[TK_COLZ]), block2d(), 0, st, S, active);
}

cudaError_t launch_scales(int nbox, const int *active, int init, const double *norm,
                          const double *normf, double *se, double *sr, double *sr_inv,
                          cudaStream_t st)
{
    return pdl_launch(k_scales, dim3((nbox + 127) / 128), dim3(128), 0, st, nbox, active, init,
                      norm, normf, se, sr, sr_inv);
}

static inline dim3 grid3(int ex, int ey, int ez)
{
    return dim3((ex + kTX - 1) / kTX, (ey + kTY - 1) / kTY, ez);
}

cudaError_t launch_face_weights(int nx, int ny, int nz, double inv_h2, int bcm, const double *beta,
                                double *wx, double *wy, double *wz, cudaStream_t st)
{
    k_face_weights<<<grid3(nx + 1, ny + 1, nz + 1), block2d(), 0, st>>>(
        nx, ny, nz, (int)pitch_row(nx), pitch_plane(nx, ny), inv_h2, bcm, beta, wx, wy, wz);
    return counted(cudaGetLastError());
}

cudaError_t launch_coarsen(int nx, int ny, int nz, const double *wx, const double *wy,
                           const double *wz, double *cwx, double *cwy, double *cwz, cudaStream_t st)
{
    const int cx = nx / 2, cy = ny / 2, cz = nz / 2;
    k_coarsen<<<grid3(cx + 1, cy + 1, cz + 1), block2d(), 0, st>>>(
        nx, ny, nz, (int)pitch_row(nx), pitch_plane(nx, ny), wx, wy, wz, (int)pitch_row(cx),
        pitch_plane(cx, cy), cwx, cwy, cwz);
    return counted(cudaGetLastError());
}

cudaError_t launch_inv_diag(int nx, int ny, int nz, const double *wx, const double *wy,
                            const double *wz, double *invD, double *D, cudaStream_t st)
{
    k_inv_diag<<<grid3(nx, ny, nz), block2d(), 0, st>>>(nx, ny, nz, (int)pitch_row(nx),
                                                        pitch_plane(nx, ny), wx, wy, wz, invD, D);
    return counted(cudaGetLastError());
}

cudaError_t launch_round_f32(int nx, int ny, int nz, const double *wx, const double *wy,
                             const double *wz, const double *invD, float *wx32, float *wy32,
                             float *wz32, float *invD32, cudaStream_t st)
{
    k_round_f32<<<grid3(nx + 1, ny + 1, nz + 1), block2d(), 0, st>>>(
        nx, ny, nz, (int)pitch_row(nx), pitch_plane(nx, ny), wx, wy, wz, invD, wx32, wy32, wz32,
        invD32);
    return counted(cudaGetLastError());
}

// CTAs of the cluster that inverts an n x n matrix (nbox of them at once), and
// the shared memory of each: short matrices are a chain of barriers, which one
// CTA passes fastest.
static int inv_ctas(int n, int nbox, int limit)
{
    const int c = std::min(n >= 128 ? 16 : n >= 48 ? 8 : 1, limit);
    return cluster_step_down(c, [&](int k) { return (long long)k * nbox <= 304; });   // (two waves)
}
// The largest cluster of an inverse kernel that the current device can hold
// with the most shared memory it takes; asked once a device.
template <class K>
static int inv_limit(K *kernel, int which)
{
    constexpr int kMaxDevices = 64;
    static std::mutex mu;
    static int known[3][kMaxDevices] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) {
        cudaGetLastError();
        dev = -1;
    }
    std::lock_guard<std::mutex> lk(mu);
    if (dev >= 0 && known[which][dev]) return known[which][dev];
    const int c = cluster_step_down(16, [&](int k) {
        return resident_clusters(kernel, k, dim3(kInvThreads), kTailSmem) > 0;
    });
    if (dev >= 0) known[which][dev] = c;
    return c;
}
static int inv_bytes(int n, int ctas, bool fp64)
{
    const long long e = fp64 ? 8 : 4, rows = (3LL * n + inv_rows_elems(n, ctas)) * e;
    return (int)(rows <= kTailSmem ? rows : 3LL * n * e);
}

template <class K, class... Args>
static cudaError_t inv_launch(K kernel, int clusters, int ctas, int smem, cudaStream_t st, Args... args)
{
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kTailSmem);
    if (e == cudaSuccess && ctas > 8)
        e = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(clusters * ctas);
    cfg.blockDim = dim3(kInvThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = ctas;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return counted(cudaLaunchKernelEx(&cfg, kernel, args...));
}

cudaError_t launch_bottom_inverse(int nx, int ny, int nz, const double *wx, const double *wy,
                                  const double *wz, int singular, double *work, double *inv64,
                                  float *inv32, cudaStream_t st)
{
    const int n = nx * ny * nz, c = inv_ctas(n, 1, inv_limit(k_bottom_inverse, 0)),
              smem = inv_bytes(n, c, true);
    return inv_launch(k_bottom_inverse, 1, c, smem, st, nx, ny, nz, (int)pitch_row(nx),
                      (long long)pitch_plane(nx, ny), wx, wy, wz, singular, work, inv64, inv32, smem);
}

cudaError_t launch_setup_tiles(const SetupSet &S, int step, int t0, int t1, cudaStream_t st)
{
    if (t1 <= t0) return cudaSuccess;
    const dim3 g(t1 - t0), b = block2d();
    switch (step) {
    case 0: k_setup<0><<<g, b, 0, st>>>(S, t0); break;
    case 1: k_setup<1><<<g, b, 0, st>>>(S, t0); break;
    case 2: k_setup<2><<<g, b, 0, st>>>(S, t0); break;
    case 3: k_setup<3><<<g, b, 0, st>>>(S, t0); break;
    case 4: k_setup<4><<<g, b, 0, st>>>(S, t0); break;
    case 5: k_setup<5><<<g, b, 0, st>>>(S, t0); break;
    case 6: k_setup<6><<<g, b, 0, st>>>(S, t0); break;
    case 8: k_setup<8><<<g, b, 0, st>>>(S, t0); break;
    case 9: k_setup<9><<<g, b, 0, st>>>(S, t0); break;
    default: return cudaErrorInvalidValue;
    }
    return counted(cudaGetLastError());
}

cudaError_t launch_setup(const SetupSet &S, int step, cudaStream_t st)
{
    if (step < 0 || step > 9 || step == 7) return cudaErrorInvalidValue;
    return launch_setup_tiles(S, step, 0, S.ntiles[setup_kind(step)], st);
}

cudaError_t launch_setup_bottom(const SetupSet &S, int max_cells, bool fp64, cudaStream_t st)
{
    if (S.nbox == 0) return cudaSuccess;
    const int c = inv_ctas(max_cells, S.nbox, inv_limit(k_setup_bottom, 1)),
              smem = inv_bytes(max_cells, c, fp64);
    return inv_launch(k_setup_bottom, S.nbox, c, smem, st, S, smem);
}

cudaError_t launch_project_rhs(int nx, int ny, int nz, double h, const double *u, const double *v,
                               const double *w, const double *S, double *f, cudaStream_t st)
{
    k_project_rhs<<<grid3(nx, ny, nz), block2d(), 0, st>>>(nx, ny, nz, 1.0 / h, u, v, w, S, f);
    return counted(cudaGetLastError());
}

cudaError_t launch_project_correct(int nx, int ny, int nz, double h, const double *wx,
                                   const double *wy, const double *wz, const double *phi,
                                   double *u, double *v, double *w, cudaStream_t st, bool wide)
{
    k_project_correct<<<grid3(nx + 1, ny + 1, nz + 1), block2d(), 0, st>>>(
        nx, ny, nz, (int)pitch_row(nx, wide), pitch_plane(nx, ny, wide), h, wx, wy, wz, phi, u,
        v, w);
    return counted(cudaGetLastError());
}

cudaError_t launch_beta_grad(int nx, int ny, int nz, int nrhs, double inv_h2, int bcm,
                             const double *beta, const double *phi, const double *lam,
                             double *dbeta, cudaStream_t st)
{
    k_beta_grad<<<grid3(nx, ny, (nz + kGradZ - 1) / kGradZ), block2d(), 0, st>>>(
        nx, ny, nz, nrhs, inv_h2, bcm, beta, phi, lam, dbeta);
    return counted(cudaGetLastError());
}

cudaError_t launch_bc_lift(int nx, int ny, int nz, double inv_h, int bcm, const double *wx,
                           const double *wy, const double *wz, const double *vals,
                           const double *f, double *fout, cudaStream_t st, bool wide)
{
    k_bc_lift<<<grid3(nx, ny, nz), block2d(), 0, st>>>(nx, ny, nz, (int)pitch_row(nx, wide),
                                                       pitch_plane(nx, ny, wide), inv_h, bcm, wx,
                                                       wy, wz, vals, f, fout);
    return counted(cudaGetLastError());
}

cudaError_t launch_remove_mean(const BoxSet<double> &S, int field, double *partials, double *mean,
                               cudaStream_t st)
{
    if (S.ntiles[TK_COLZ] == 0) return cudaSuccess;
    cudaError_t e = pdl_launch(k_sum_partials, dim3(S.ntiles[TK_COLZ]), block2d(), 0, st, S, field,
                               partials);
    if (e != cudaSuccess) return e;
    e = pdl_launch(k_mean_finish, dim3(S.nbox), dim3(1024), 0, st, S, partials, mean);
    if (e != cudaSuccess) return e;
    return pdl_launch(k_sub_mean, dim3(S.ntiles[TK_CELL]), block2d(), 0, st, S, field, mean);
}

template <class T>
cudaError_t launch_exchange(const BoxSet<T> &S, const int *active, const ExchRec *rec, int nrec,
                            int max_cells, cudaStream_t st, int second)
{
    if (nrec == 0) return cudaSuccess;
    // about 4 cells per thread on the largest record (a 256^2 face: 64 CTAs)
    const int chunks = std::max(1, std::min(1024, (max_cells + 4 * kThreads - 1) / (4 * kThreads)));
    return pdl_launch(k_exchange<T>, dim3(nrec, chunks), block2d(), 0, st, S, active, rec, second);
}

template <class T>
cudaError_t launch_rbgs_pass_multi(const BoxSet<T> &S, const int *active, int color, int oop,
                                   int from2, cudaStream_t st)
{
    if (S.nbox == 0 || S.ntiles[TK_PAIR] == 0) return cudaSuccess;
    const int per = S.ntiles[TK_PAIR] / S.nbox;   // tiles of one right-hand side
    if (oop)
        return pdl_launch(k_rbgs_pass_oop_multi<T>, dim3(per), block2d(), 0, st, S, active, color,
                          from2);
    return pdl_launch(k_rbgs_pass_multi<T>, dim3(per), block2d(), 0, st, S, active, color);
}
template cudaError_t launch_rbgs_pass_multi<double>(const BoxSet<double> &, const int *, int, int,
                                                    int, cudaStream_t);
template cudaError_t launch_rbgs_pass_multi<float>(const BoxSet<float> &, const int *, int, int,
                                                   int, cudaStream_t);

template <class T>
int level_ctas_per_sm()
{
    int n = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_level_down<T>, kThreads, 0) !=
        cudaSuccess) {
        cudaGetLastError();
        return 1;
    }
    int m = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&m, k_level_up<T>, kThreads, 0) !=
        cudaSuccess) {
        cudaGetLastError();
        return 1;
    }
    return std::max(1, std::min(n, m));
}
template int level_ctas_per_sm<double>();
template int level_ctas_per_sm<float>();

template <class T>
cudaError_t launch_level(const BoxSet<T> &S, const int *active, int up, const LevelOps &op,
                         const GridSync &g, int grid, cudaStream_t st)
{
    if (S.nbox == 0 || grid < 1) return cudaSuccess;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = block2d();
    cfg.dynamicSmemBytes = 0;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;   // every CTA resident at once
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return counted(up ? cudaLaunchKernelEx(&cfg, k_level_up<T>, S, active, op, g)
                      : cudaLaunchKernelEx(&cfg, k_level_down<T>, S, active, op, g));
}
template cudaError_t launch_level<double>(const BoxSet<double> &, const int *, int,
                                          const LevelOps &, const GridSync &, int, cudaStream_t);
template cudaError_t launch_level<float>(const BoxSet<float> &, const int *, int,
                                         const LevelOps &, const GridSync &, int, cudaStream_t);

template <class T>
int cg_bottom_ctas_per_sm()
{
    int n = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_cg_bottom<T>, kThreads, 0) !=
        cudaSuccess) {
        cudaGetLastError();
        return 1;
    }
    return std::max(1, n);
}
template int cg_bottom_ctas_per_sm<double>();
template int cg_bottom_ctas_per_sm<float>();

template <class T>
cudaError_t launch_cg_bottom(const BoxSet<T> &S, const int *active, T *p, T *q, double *part,
                             const GridSync &g, int grid, double tol, int maxit, cudaStream_t st,
                             bool cluster)
{
    if (S.nbox == 0 || grid < 1) return cudaSuccess;
    cudaLaunchConfig_t cfg = {};
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (cluster) {
        auto *const k = k_cg_bottom_cluster<T>;
        cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        if (e != cudaSuccess) return e;
        cfg.gridDim = dim3(kCgCtas);
        cfg.blockDim = dim3(kTX, kTY, (S.ntiles[TK_CELL] + kCgCtas - 1) / kCgCtas);
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = kCgCtas;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        return counted(cudaLaunchKernelEx(&cfg, k, S, active, p, tol, maxit));
    }
    cfg.gridDim = dim3(grid);
    cfg.blockDim = block2d();
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    return counted(cudaLaunchKernelEx(&cfg, k_cg_bottom<T>, S, active, p, q, part, g, tol, maxit));
}
template cudaError_t launch_cg_bottom<double>(const BoxSet<double> &, const int *, double *,
                                              double *, double *, const GridSync &, int, double,
                                              int, cudaStream_t, bool);
template cudaError_t launch_cg_bottom<float>(const BoxSet<float> &, const int *, float *, float *,
                                             double *, const GridSync &, int, double, int,
                                             cudaStream_t, bool);

// The cluster takes levels of at most kCgCtas x kCgGroups tiles (a thread a
// cell; see the kernel) where a cluster of that size can be resident.
template <class T>
bool cg_cluster_fits(long long tiles)
{
    return tiles <= kCgCtas * kCgGroups &&
           resident_clusters(k_cg_bottom_cluster<T>, kCgCtas, dim3(kTX, kTY, kCgGroups), 0) > 0;
}
template bool cg_cluster_fits<double>(long long);
template bool cg_cluster_fits<float>(long long);

template <class T>
cudaError_t launch_guard_fill(const BoxSet<T> &S, T v, cudaStream_t st)
{
    if (S.nbox == 0) return cudaSuccess;
    k_guard_fill<T><<<dim3(S.nbox, 6), block2d(), 0, st>>>(S, v);
    return counted(cudaGetLastError());
}

cudaError_t launch_union_inverse(const SetupSet &S, const UnionBottom &U, double *work,
                                 double *inv64, float *inv32, cudaStream_t st)
{
    const int c = inv_ctas(U.n, 1, inv_limit(k_union_inverse, 2)),
              smem = inv_bytes(U.n, c, true);
    return inv_launch(k_union_inverse, 1, c, smem, st, S, U, work, inv64, inv32, smem);
}

template <class T>
cudaError_t launch_union_bottom(const BoxSet<T> &S, const UnionBottom &U, const T *ainv,
                                const int *active, cudaStream_t st)
{
    return pdl_launch(k_union_bottom<T>, dim3((U.n + 31) / 32), block2d(), 0, st, S, U, ainv,
                      active);
}

cudaError_t launch_norm_combine(int nbox, double *norm, cudaStream_t st)
{
    return pdl_launch(k_norm_combine, dim3(1), dim3(256), 0, st, nbox, norm);
}

cudaError_t launch_pcg(const BoxSet<double> &S, const int *active, int op, double *const *pv,
                       double *const *qv, const PcgScalars &sc, double *partials,
                       double *norm_out, cudaStream_t st)
{
    if (S.ntiles[TK_COLZ] == 0) return cudaSuccess;
    auto go = [&](auto tag) {
        constexpr int OP = decltype(tag)::value;
        cudaError_t e = pdl_launch(k_pcg<OP>, dim3(S.ntiles[TK_COLZ]), block2d(), 0, st, S, active,
                                   pv, qv, sc, partials);
        if (e != cudaSuccess || OP == 1 || OP >= 5) return e;
        return pdl_launch(k_pcg_finish<OP>, dim3(S.nbox), dim3(1024), 0, st, S, active, partials,
                          sc, norm_out);
    };
    switch (op) {
    case 0: return go(std::integral_constant<int, 0>{});
    case 1: return go(std::integral_constant<int, 1>{});
    case 2: return go(std::integral_constant<int, 2>{});
    case 3: return go(std::integral_constant<int, 3>{});
    case 4: return go(std::integral_constant<int, 4>{});
    case 5: return go(std::integral_constant<int, 5>{});
    default: return go(std::integral_constant<int, 6>{});
    }
}

cudaError_t launch_max_norm(const BoxSet<double> &S, const int *side, int field,
                            double *partials, double *out, cudaStream_t st)
{
    if (S.ntiles[TK_COLZ] == 0) return cudaSuccess;
    k_max_partials<<<S.ntiles[TK_COLZ], block2d(), 0, st>>>(S, side, field, partials);
    cudaError_t e = counted(cudaGetLastError());
    if (e != cudaSuccess) return e;
    k_max_finish<<<S.nbox, 1024, 0, st>>>(S, partials, out);
    return counted(cudaGetLastError());
}

cudaError_t launch_pcg_mixed(const BoxSet<double> &S64, const BoxSet<float> &S32, const int *active,
                             int op, const double *nrm, cudaStream_t st)
{
    if (S64.ntiles[TK_CELL] == 0) return cudaSuccess;
    return pdl_launch(k_pcg_mixed, dim3(S64.ntiles[TK_CELL]), block2d(), 0, st, S64, S32, active,
                      op, nrm);
}

#define MG_INSTANTIATE(T)                                                                        \
    template cudaError_t launch_rbgs_pass<T>(const BoxSet<T> &, const int *, int, cudaStream_t,    \
                                             bool);                                              \
    template cudaError_t launch_rbgs_pass_oop<T>(const BoxSet<T> &, const int *, int, int, double *, \
                                                 cudaStream_t);                                      \
    template cudaError_t launch_rbgs_sweep<T>(const BoxSet<T> &, const int *, int, cudaStream_t); \
    template cudaError_t launch_resid_restrict<T>(const BoxSet<T> &, const int *, cudaStream_t);  \
    template cudaError_t launch_resid_restrict_red<T>(const BoxSet<T> &, const int *,             \
                                                      cudaStream_t, double *);                    \
    template cudaError_t launch_prolong<T>(const BoxSet<T> &, const int *, cudaStream_t);         \
    template cudaError_t launch_residual_field<T>(const BoxSet<T> &, cudaStream_t);               \
    template cudaError_t launch_norm_partials<T>(const BoxSet<T> &, const int *, int, double *,   \
                                                 cudaStream_t);                                   \
    template cudaError_t launch_norm_finish<T>(const BoxSet<T> &, const int *, const double *,    \
                                               double *, double *, double *, cudaStream_t,        \
                                               const double *, int);                              \
    template cudaError_t launch_bottom<T>(const BoxSet<T> &, const int *, int, cudaStream_t);   \
    template cudaError_t launch_zero<T>(const BoxSet<T> &, const int *, cudaStream_t);          \
    template cudaError_t launch_coarse_vcycle<T>(const CoarseJob<T> *, int, int, size_t,            \
                                                 const int *, int, int, cudaStream_t, int);         \
    template cudaError_t launch_exchange<T>(const BoxSet<T> &, const int *, const ExchRec *, int,  \
                                            int, cudaStream_t, int);                                         \
    template cudaError_t launch_guard_fill<T>(const BoxSet<T> &, T, cudaStream_t);                 \
    template cudaError_t launch_union_bottom<T>(const BoxSet<T> &, const UnionBottom &, const T *, \
                                                const int *, cudaStream_t);

MG_INSTANTIATE(double)
MG_INSTANTIATE(float)

}  // namespace mg
