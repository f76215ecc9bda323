// Internal definitions shared by the translation units of libsplatloam (not part of the ABI).
#pragma once

#include <atomic>
#include <cmath>
#include <cstdint>
#include <cuda_runtime.h>

#include "../../include/splatloam.h"

namespace splat {

constexpr int kMaxViews = 64;
constexpr int kBlock = 256;          // threads per render CTA = pixels per tile

// ---------------------------------------------------------------------------------------------
// chained launches: the stages of a call are short kernels that each need the one before.  A
// kernel launched with launch_chained(true, ...) may be scheduled while its predecessor still runs
// (programmatic stream serialisation) and begins with chain_wait(), which returns when the
// predecessor has completed and its writes are visible, and then lets the next kernel be
// scheduled.  Every kernel that is launched so has to call it first.  It pays where kernels are as
// short as the gaps between them (render of 2,000 primitives 44 -> 36 us, 64x1024 over 100,000 with
// autograd 329 -> 313 us, three scans over 83,000 336 -> 323 us) and costs where they fill the SMs,
// since a kernel scheduled early crowds onto the SMs that come free first (1 M primitives 664 ->
// 681 us, 12 x 500,000 2,209 -> 2,238 us): calls of up to kChainPairs pairs are chained.  The last
// kernel of a backward, the parameter gradients, has no view loop and goes by the primitives
// alone: the compositing kernel before it leaves no room on its SMs, so that being scheduled early
// only hides the launch (render and backward of 4 x 200,000 primitives 394.1 -> 392.8 us, 8 x
// 400,000 1,008.5 -> 1,005.5).
// ---------------------------------------------------------------------------------------------
__device__ __forceinline__ void chain_wait()
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

constexpr int64_t kChainPairs = int64_t{1} << 19;
inline bool chained_size(int64_t pairs) { return pairs <= kChainPairs; }

template <typename... P, typename... A>
cudaError_t launch_cluster(bool chain, int cluster, void (*kernel)(P...), dim3 grid, unsigned block,
                           size_t smem, cudaStream_t st, const A &...args)
{
    cudaLaunchAttribute attr[2] = {};
    unsigned n = 0;
    if (chain) {
        attr[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[n++].val.programmaticStreamSerializationAllowed = 1;
    }
    if (cluster > 1) {
        attr[n].id = cudaLaunchAttributeClusterDimension;
        attr[n].val.clusterDim.x = static_cast<unsigned>(cluster);
        attr[n].val.clusterDim.y = attr[n].val.clusterDim.z = 1;
        ++n;
    }
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = attr;
    cfg.numAttrs = n;
    return cudaLaunchKernelEx(&cfg, kernel, P(args)...);
}

template <typename... P, typename... A>
cudaError_t launch_chained(bool chain, void (*kernel)(P...), dim3 grid, unsigned block, size_t smem,
                           cudaStream_t st, const A &...args)
{
    return launch_cluster(chain, 1, kernel, grid, block, smem, st, args...);
}

// Raises a kernel's dynamic shared memory limit above the default 48 KB, once on each device: the
// attribute belongs to the current device's copy of the kernel.  Called where a context, or the
// call without one, is set up, not at every launch.  carveout (percent, negative for the driver's
// choice): how much of an SM's memory is shared, the rest is L1.  One static object per kernel; a
// failed call is tried again by the next one.
class SharedLimit {
public:
    template <typename Kernel>
    cudaError_t raise(Kernel *kernel, size_t bytes, int carveout = -1)
    {
        int dev = 0;
        cudaError_t e = cudaGetDevice(&dev);
        if (e != cudaSuccess) return e;
        const bool known = dev >= 0 && dev < kDevices;
        if (known && done_[dev].load(std::memory_order_acquire)) return cudaSuccess;
        e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 static_cast<int>(bytes));
        if (e == cudaSuccess && carveout >= 0)
            e = cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout,
                                     carveout);
        if (e == cudaSuccess && known) done_[dev].store(true, std::memory_order_release);
        return e;
    }

private:
    static constexpr int kDevices = 64;
    std::atomic<bool> done_[kDevices] = {};
};

// ---------------------------------------------------------------------------------------------
// per-view descriptor (device)
// ---------------------------------------------------------------------------------------------
struct ViewDesc {
    // T^c_w as float pairs (hi = nearest float of the FP64 value, lo = nearest float of the rest)
    float R_hi[9], R_lo[9];       // row-major
    float t_hi[3], t_lo[3];
    int32_t rows, cols;
    float elev_min, elev_max;
    float kr;                     // binary32 (rows - 1) / (elev_max - elev_min): contract rows
    float dgamma;                 // 2 pi / cols  (nearest float)
    float dtheta;                 // (elev_max - elev_min) / (rows - 1)  (nearest float)
    int32_t tiles_r, tiles_c;     // tile rows / columns of this view
    int64_t tile_offset;          // first global tile id of the view
    int64_t pixel_offset;         // first pixel of the view in the packed buffers
    int32_t pix_offset;           // into the pixel-frame table: tiles_r x 256 entries
    // cones two rows (and a milliradian) beyond the top and bottom rows: z = t |xy|, with
    // l = sqrt(1 + t^2) the Lipschitz constant of z - t |xy| (l = inf: no cone)
    float cull_t_top, cull_l_top, cull_t_bot, cull_l_bot;
};

// Row and column of pixel `local` of a view: a view has at most 32,767^2 pixels, so the quotient
// is a 32-bit one (a 64-bit one costs about four times the instructions).
__device__ __forceinline__ void row_col(int64_t local, int cols, int &r, int &c)
{
    const uint32_t l = static_cast<uint32_t>(local), w = static_cast<uint32_t>(cols);
    const uint32_t q = l / w;
    r = static_cast<int>(q);
    c = static_cast<int>(l - q * w);
}

// Pixel-centre ray of pixel (r, c) of a view (Sec. 3.1), binary32.
__device__ __forceinline__ float3 pixel_ray(const ViewDesc &vd, int r, int c)
{
    const float g = 3.14159265358979f - vd.dgamma * (static_cast<float>(c) + 0.5f);
    const float th = vd.rows > 1 ? vd.elev_max - vd.dtheta * static_cast<float>(r) : vd.elev_max;
    float sg, cg, st, ct;
    sincosf(g, &sg, &cg);
    sincosf(th, &st, &ct);
    return make_float3(ct * cg, ct * sg, st);
}

// Philox-4x32-10 (Salmon, Moraes, Dror, Shaw, SC 2011), from its definition: a round maps
// (c0, c1, c2, c3) to (hi(M1 c2) ^ c1 ^ k0, lo(M1 c2), hi(M0 c0) ^ c3 ^ k1, lo(M0 c0)); the key
// is bumped by the Weyl constants between rounds.
__device__ __forceinline__ uint4 philox4x32_10(uint4 c, uint2 k)
{
    constexpr uint32_t M0 = 0xD2511F53u, M1 = 0xCD9E8D57u, W0 = 0x9E3779B9u, W1 = 0xBB67AE85u;
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        const uint32_t hi0 = __umulhi(M0, c.x), lo0 = M0 * c.x;
        const uint32_t hi1 = __umulhi(M1, c.z), lo1 = M1 * c.z;
        c = make_uint4(hi1 ^ c.y ^ k.x, lo1, hi0 ^ c.w ^ k.y, lo0);
        if (r < 9) {
            k.x += W0;
            k.y += W1;
        }
    }
    return c;
}

// Keyframe sampling (Sec. 3.3): draws j < draws of refinement step *step take the first word x of
// Philox-4x32-10((j, step, 0, 0), (seed lo, seed hi)); the drawn view is n_views - 1 - #{a :
// x >= thr[a]} (thr: n_views - 1 integer thresholds of the cumulative law); active[v] = 1 for a
// view drawn at least once, 0 otherwise; *step then advances by one.
cudaError_t launch_sample_views(int n_views, int draws, const uint32_t *thr, uint32_t seed_lo,
                                uint32_t seed_hi, uint32_t *step, uint8_t *active,
                                cudaStream_t st);

// Back-projection of the packed range images of the registered views to world-frame points
// (3 x n_pixels planar, NaN where O < o_min).
cudaError_t launch_backproject(const ViewDesc *views, int n_views, int64_t n_pixels,
                               const float *depth, const float *alpha, float o_min, float *points,
                               cudaStream_t st);

// Map growth (Sec. 3.3.1, 3.3.2): mask, range-gradient weights and a systematic draw of n_d
// pixels over the packed pixels of the views; slot j of the new primitives takes the pixel that
// holds sample j first, or is written empty.
constexpr int kGrowMaxGrid = 1024;
struct GrowArgs {
    const ViewDesc *views;
    int n_views;
    int64_t n_pixels;
    const float *t_depth, *depth, *alpha;   // depth, alpha: used when refine != 0
    int refine;
    float lambda_do, lambda_de, w0, w_cap, scale_k, logit, empty_logit;
    uint32_t seed_lo, seed_hi;
    uint32_t *call;                         // device counter of draws, advanced per call
    uint32_t *q;                            // scratch, n_pixels
    unsigned long long *block_sums;         // scratch, kGrowMaxGrid + 2
    float4 *pos_logit, *quat;               // the n_d new slots
    float2 *log_scale;
    int64_t n_d;
    int grid;                               // set by launch_grow
    int64_t chunk;
};
cudaError_t launch_grow(GrowArgs a, cudaStream_t st);

// Photometric residual of one view against a query range image and its Gauss-Newton normal
// equations (Sec. 3.3.3): out[29] = H upper triangle (21, row-major), g (6), Huber cost, count;
// per_pixel (nullable) = 8 x P planar: r, w, J (6).  T: device binary32 3 x 4 render -> query.
cudaError_t launch_photometric(const ViewDesc &vd, const float *depth, const float *alpha,
                               const float *qdepth, const float *T, float o_min, float delta,
                               double *out, float *per_pixel, int sms, cudaStream_t st);

// the culling cones of a view (host)
inline void set_cull_cones(ViewDesc &vd, double emin, double emax, double dtheta)
{
    const double m = 2.0 * dtheta + 1e-3;
    const double top = emax + m, bot = emin - m, lim = 1.5;   // well inside +-pi/2
    vd.cull_t_top = top < lim ? static_cast<float>(std::tan(top)) : 0.0f;
    vd.cull_l_top = top < lim ? static_cast<float>(std::sqrt(1.0 + std::tan(top) * std::tan(top)) *
                                                   1.0001)
                              : INFINITY;
    vd.cull_t_bot = bot > -lim ? static_cast<float>(std::tan(bot)) : 0.0f;
    vd.cull_l_bot = bot > -lim ? static_cast<float>(std::sqrt(1.0 + std::tan(bot) * std::tan(bot)) *
                                                    1.0001)
                               : INFINITY;
}

// Pixel ray planes of one pixel in its tile's frame (FP64 values as float pairs): h_x, h_y
// (hi parts and the remainders) and the ray direction v (hi only).  One entry per (view, tile
// row, pixel of the tile), 64 bytes.
struct PixFrame {
    float hx[3], hy[3], v[3];
    float hx_lo[3], hy_lo[3];
    float pad;
};
static_assert(sizeof(PixFrame) == 64, "PixFrame is 64 bytes");

// Per-tile frame and addressing, computed on the host in FP64 when the views are registered.
// The tile frame Q has rows e1 = v(theta0, gamma0) (the ray through the tile centre),
// e2 = h_x(gamma0), e3 = h_y(theta0, gamma0); M = Q R^c_w and u = Q t^c_w as float pairs,
// R^c_w rounded (normals are produced in the sensor frame).  192 bytes.
struct TileInfo {
    float M_hi[9], M_lo[9];
    float u_hi[3], u_lo[3];
    float R[9];
    int32_t view, tr, tc, cols;      // cols: the view's width (row stride and cyclic period)
    int32_t valid_r, valid_c;        // pixels of this tile inside the image
    int32_t pix_base;                // first PixFrame entry of this tile row
    int64_t out_base;                // packed index of the tile's top-left pixel
    int32_t pad[6];
};
static_assert(sizeof(TileInfo) == 192, "TileInfo is 192 bytes");

// Per (view, primitive) projection record, 16 bytes.
struct PairRec {
    int16_t r0, r1;   // pixel rows [r0, r1]
    int16_t c0, nc;   // cyclic pixel columns [c0, c0 + nc) mod cols
    float kappa;      // binary32 centre range |b_c|
    uint32_t cf;      // bits 0-29: tiles touched; bit 30: normal flipped; bit 31: invalid input
};
static_assert(sizeof(PairRec) == 16, "PairRec is 16 bytes");

enum : uint32_t { kPairFlip = 1u << 30, kPairInvalid = 1u << 31 };

// ---------------------------------------------------------------------------------------------
// tile geometry shared by the binning and the render kernels
// ---------------------------------------------------------------------------------------------

// A pair's pixel rectangle and normal-flip bit in one word: r0 | flip << 15, r1, c0, nc, 16 bits
// each (rows and columns are below 2^15); 0 for a pair that touches no tile (nc >= 1 otherwise)
__host__ __device__ inline uint64_t pack_pixel_rect(const PairRec &rec)
{
    const uint32_t r0 = static_cast<uint16_t>(rec.r0) | ((rec.cf & kPairFlip) ? 0x8000u : 0u);
    return static_cast<uint64_t>(r0) | static_cast<uint64_t>(static_cast<uint16_t>(rec.r1)) << 16 |
           static_cast<uint64_t>(static_cast<uint16_t>(rec.c0)) << 32 |
           static_cast<uint64_t>(static_cast<uint16_t>(rec.nc)) << 48;
}

__host__ __device__ inline PairRec unpack_pixel_rect(uint64_t w)
{
    PairRec rec;
    rec.r0 = static_cast<int16_t>(w & 0x7FFFu);
    rec.r1 = static_cast<int16_t>((w >> 16) & 0xFFFFu);
    rec.c0 = static_cast<int16_t>((w >> 32) & 0xFFFFu);
    rec.nc = static_cast<int16_t>(w >> 48);
    rec.kappa = 0.0f;
    rec.cf = (w & 0x8000u) ? kPairFlip : 0u;
    return rec;
}

// A pair's tile rectangle: first tile row and column, rows and columns, the columns cyclic modulo
// the view's tile columns.
struct TileRect {
    int r0, nr, c0, nc;
};

// Blocks of primitives: the projection's CTAs, and the segments of its touching pairs.  Larger
// maps take blocks of 1,024, so that the pairs a CTA has to box exactly fill more warps; smaller
// ones of 256, so that there are CTAs for every SM.
constexpr int kSmallBlock = 256, kLargeBlock = 1024;
inline int block_prims(int64_t n) { return n < int64_t{1} << 18 ? kSmallBlock : kLargeBlock; }
inline int64_t project_blocks(int64_t n)
{
    return (n + block_prims(n) - 1) / block_prims(n);
}
// the most blocks of any map of up to n primitives
inline int64_t max_project_blocks(int64_t n)
{
    const int64_t small = n < int64_t{1} << 18 ? n : int64_t{1} << 18;
    const int64_t a = small / kSmallBlock + 1, b = n / kLargeBlock + 1;
    return a > b ? a : b;
}

// A touching pair in its block's segment: its tile rectangle and its primitive's place in the
// block, in two 32-bit words.  Images have at most 32,767 rows and columns and tiles at least 4
// rows and 8 columns: at most 8,192 tile rows and 4,096 tile columns.
__device__ __forceinline__ uint2 pack_touch(const TileRect &t, uint32_t local)
{
    return make_uint2(static_cast<uint32_t>(t.r0) | static_cast<uint32_t>(t.nr) << 13 | local << 27,
                      static_cast<uint32_t>(t.c0) | static_cast<uint32_t>(t.nc) << 12 |
                          local >> 5 << 25);
}

__device__ __forceinline__ TileRect unpack_touch(uint2 w, uint32_t &local)
{
    local = w.x >> 27 | w.y >> 25 << 5;
    return TileRect{static_cast<int>(w.x & 0x1FFFu), static_cast<int>(w.x >> 13 & 0x3FFFu),
                    static_cast<int>(w.y & 0xFFFu), static_cast<int>(w.y >> 12 & 0x1FFFu)};
}

// the tiles a record's pixel rectangle meets: columns c0 .. c0 + nc - 1 (mod W), wrapping past
// the last tile; tile sides are powers of two and every index here is non-negative, so shifts
// divide
__device__ __forceinline__ TileRect tile_rect(const PairRec &rec, int W, int tiles_c, int th_shift,
                                              int tw_shift)
{
    TileRect t;
    t.r0 = rec.r0 >> th_shift;
    t.nr = (rec.r1 >> th_shift) - t.r0 + 1;
    if (rec.nc >= W) {
        t.c0 = 0;
        t.nc = tiles_c;
    } else {
        const int cl = rec.c0 + rec.nc - 1;
        const int b = cl < W ? cl >> tw_shift : tiles_c + ((cl - W) >> tw_shift);
        t.c0 = rec.c0 >> tw_shift;
        t.nc = b - t.c0 + 1;
        if (t.nc >= tiles_c) {
            t.c0 = 0;
            t.nc = tiles_c;
        }
    }
    return t;
}

// ---------------------------------------------------------------------------------------------
// float-pair ("double-float") arithmetic, used where the sensor-frame centre of a primitive
// must keep more than 24 bits (the lateral offset of a far splat from a ray).
// ---------------------------------------------------------------------------------------------
struct f2 {
    float h, l;
};

__device__ __forceinline__ void two_sum(float a, float b, float &s, float &e)
{
    s = __fadd_rn(a, b);
    float bb = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}

__device__ __forceinline__ f2 f2_mul(f2 a, f2 b)
{
    float p = __fmul_rn(a.h, b.h);
    float e = __fmaf_rn(a.h, b.h, -p);
    e = __fmaf_rn(a.h, b.l, e);
    e = __fmaf_rn(a.l, b.h, e);
    f2 r;
    two_sum(p, e, r.h, r.l);
    return r;
}

__device__ __forceinline__ f2 f2_add(f2 a, f2 b)
{
    float s, e;
    two_sum(a.h, b.h, s, e);
    e = __fadd_rn(e, __fadd_rn(a.l, b.l));
    f2 r;
    two_sum(s, e, r.h, r.l);
    return r;
}

// Sum_j M_j x_j + u in float-pair arithmetic, rounded to one float (x exact floats).
__device__ __forceinline__ float f2_dot3_add(f2 m0, f2 m1, f2 m2, float x0, float x1, float x2,
                                             f2 u)
{
    float p0 = __fmul_rn(m0.h, x0), e0 = __fmaf_rn(m0.h, x0, -p0);
    float p1 = __fmul_rn(m1.h, x1), e1 = __fmaf_rn(m1.h, x1, -p1);
    float p2 = __fmul_rn(m2.h, x2), e2 = __fmaf_rn(m2.h, x2, -p2);
    float s1, t1, s2, t2, s3, t3;
    two_sum(p0, p1, s1, t1);
    two_sum(s1, p2, s2, t2);
    two_sum(s2, u.h, s3, t3);
    float err = __fadd_rn(__fadd_rn(e0, e1), e2);
    err = __fadd_rn(err, __fadd_rn(__fadd_rn(t1, t2), t3));
    err = __fmaf_rn(m0.l, x0, err);
    err = __fmaf_rn(m1.l, x1, err);
    err = __fmaf_rn(m2.l, x2, err);
    err = __fadd_rn(err, u.l);
    return __fadd_rn(s3, err);
}

// The same sum returned as a normalised float pair (hi = the rounded sum, lo = the rest).
__device__ __forceinline__ f2 f2_dot3_add2(f2 m0, f2 m1, f2 m2, float x0, float x1, float x2,
                                           f2 u)
{
    float p0 = __fmul_rn(m0.h, x0), e0 = __fmaf_rn(m0.h, x0, -p0);
    float p1 = __fmul_rn(m1.h, x1), e1 = __fmaf_rn(m1.h, x1, -p1);
    float p2 = __fmul_rn(m2.h, x2), e2 = __fmaf_rn(m2.h, x2, -p2);
    float s1, t1, s2, t2, s3, t3;
    two_sum(p0, p1, s1, t1);
    two_sum(s1, p2, s2, t2);
    two_sum(s2, u.h, s3, t3);
    float err = __fadd_rn(__fadd_rn(e0, e1), e2);
    err = __fadd_rn(err, __fadd_rn(__fadd_rn(t1, t2), t3));
    err = __fmaf_rn(m0.l, x0, err);
    err = __fmaf_rn(m1.l, x1, err);
    err = __fmaf_rn(m2.l, x2, err);
    err = __fadd_rn(err, u.l);
    f2 r;
    two_sum(s3, err, r.h, r.l);
    return r;
}

// K7 for one primitive: world-frame accumulators (dL/dmu, dL/do | dL/dt_a, dL/dlog s_a |
// dL/dt_b, dL/dlog s_b | dL/dt_n) -> gradients of (mu, logit), of the unnormalised quaternion
// (through R(q/|q|)) and of the log-scales.
__device__ __forceinline__ void chain_params(const float4 pl, const float4 q, const float4 *wg,
                                             float4 &g_pl, float4 &g_q, float2 &g_ls)
{
    const float4 a0 = wg[0], a1 = wg[1], a2 = wg[2], a3 = wg[3];
    const float qn2 = q.x * q.x + q.y * q.y + q.z * q.z + q.w * q.w;
    const float rn = rsqrtf(qn2);
    const float w = q.x * rn, x = q.y * rn, y = q.z * rn, z = q.w * rn;
    // G[r][c] = dL/dR[r][c]; column c of R is t_a, t_b, t_n
    const float G00 = a1.x, G10 = a1.y, G20 = a1.z;
    const float G01 = a2.x, G11 = a2.y, G21 = a2.z;
    const float G02 = a3.x, G12 = a3.y, G22 = a3.z;
    const float gw = 2.0f * (z * (G10 - G01) + y * (G02 - G20) + x * (G21 - G12));
    const float gx = 2.0f * (y * (G01 + G10) + z * (G02 + G20) + w * (G21 - G12)) -
                     4.0f * x * (G11 + G22);
    const float gy = 2.0f * (x * (G01 + G10) + w * (G02 - G20) + z * (G12 + G21)) -
                     4.0f * y * (G00 + G22);
    const float gz = 2.0f * (w * (G10 - G01) + x * (G02 + G20) + y * (G12 + G21)) -
                     4.0f * z * (G00 + G11);
    const float dotq = w * gw + x * gx + y * gy + z * gz;
    g_q = make_float4((gw - w * dotq) * rn, (gx - x * dotq) * rn, (gy - y * dotq) * rn,
                      (gz - z * dotq) * rn);
    const float o = 1.0f / (1.0f + __expf(-pl.w));
    g_pl = make_float4(a0.x, a0.y, a0.z, a0.w * o * (1.0f - o));
    g_ls = make_float2(a1.w, a2.w);
}

// ---------------------------------------------------------------------------------------------
// kernel launchers (defined in the .cu files)
// ---------------------------------------------------------------------------------------------
// Record the text of a failed CUDA call for splat_last_cuda_error (thread-local) and return
// SPLAT_ERR_CUDA.
int cuda_fail(cudaError_t e, const char *what);

// What the compositing kernels stage of a primitive, kPrimRow float4 written by the projection:
// (s_a t_a, o), (s_b t_b, 1 or 0 for an invalid primitive), (t_n, 0), (mu, 0), in the world frame
constexpr int kPrimRow = 4;

// What a backward starts from zero, and a refinement step's own: all nullable.  A refinement step
// has the layout kernel set them (and count the step); a backward on its own starts with
// launch_backward_start.
struct RefineStart {
    uint32_t *queue;             // work counter of the backward
    unsigned long long *evals;   // its evaluation counter
    float *pose;                 // pose gradients
    int n_pose;
    double *loss;
    int32_t *step;               // advanced by one
};

struct ProjectArgs {
    const float4 *pos_logit, *quat;
    const float2 *log_scale;
    int64_t n;
    const ViewDesc *views;
    int n_views;
    float sigma, alpha_min;
    int tile_h, tile_w, flip_normals;
    uint64_t *prect;        // per pair: pack_pixel_rect, 0 when it touches no tile
    int block_prims;        // set by the launcher
    // per (view, block): its touching pairs from place view * n + block's first primitive on,
    // their range keys, and how many there are (view * project_blocks(n) + block)
    uint2 *touch;
    float *kappa;
    uint32_t *touch_count;
    float4 *prim;
    float4 *wgrad;          // nullable: the primitives' gradient accumulators, zeroed on the way
    uint32_t *status;
    unsigned long long *n_rows;   // zeroed before: rows of 8 pixels of the blocks the pairs meet
    uint32_t *n_valid;      // zeroed before: pairs that touch a tile
    const uint8_t *active;  // per view (nullable): drawn for this step
};
cudaError_t launch_project(const ProjectArgs &a, cudaStream_t st);
cudaError_t launch_records(int64_t n, int n_views, const ViewDesc *views, int flip_normals,
                           int tile_h, int tile_w, const float4 *prim, const uint64_t *prect,
                           const uint8_t *active, PairRec *recs, cudaStream_t st);

// Binning (splat_sort.cu): from the projection's pixel rectangles to the per-tile lists in
// (range, id) order, [start, end) per tile and the work order.  A list of kListCap entries or more
// is cut into segments of at most kListCap before it is sorted, one of kHugeList or more by a
// cluster of kSplitCluster CTAs: one list of 1 M entries 0.794 -> 0.221 ms (clusters of two 0.406,
// of eight 0.146), sixteen of 68,000 0.065 -> 0.036 (0.042, 0.098: clusters of eight do not all fit
// on the chip at once, which also costs frames without such lists 6 us; of four nothing).
constexpr int kListCap = 4096;
constexpr int kSegTarget = kListCap / 2;
constexpr int kHugeList = 32768, kSplitCluster = 4;
constexpr int kSplitLevels = 6;   // cuts of one list, at most (split_list)
struct ListSegment {
    uint32_t start, len, tile;
    uint32_t in_entries;   // its keys lie in BinArgs::entries (1) or entries2 (0)
};
// A cut of len entries leaves at most len / kSegTarget + 1 stretches and one more segment for each
// bin above kSegTarget; at every level the lists and segments that are cut have kListCap entries
// or more.
constexpr int64_t max_segments(int64_t max_pairs)
{
    return kSplitLevels * (2 * (max_pairs / kSegTarget) + max_pairs / kListCap + 4);
}
struct BinArgs {
    const ViewDesc *views;
    int n_views;
    const uint8_t *active;      // nullable: views drawn for this step
    int64_t n;                  // primitives per view
    int tile_h, tile_w;
    int64_t n_tiles;
    const TileInfo *tiles;
    const uint64_t *prect;
    const uint2 *touch;
    const float *kappa;
    const uint32_t *touch_count;
    int64_t max_pairs;
    int bands, max_active_bands;   // of all views; of the views drawn, at most
    int max_band_tiles;         // most tiles of one band
    uint32_t *tile_count;       // zeroed before; counted, then counted down by the emission
    uint32_t *cta_count;        // cta_count_words(...): the counts of every counting CTA
    uint2 *ranges;
    uint32_t *order;            // tiles by decreasing bucket of list length, four an octave
    uint64_t *entries;          // emitted (range key << 32 | pair id), then the sorted entries
    uint64_t *entries2;         // scratch of the same size (needed when n >= kListCap)
    uint8_t *entry_blocks;
    ListSegment *segments;      // max_segments(max_pairs)
    uint32_t *d_count;          // out: list entries
    uint32_t *status;
    uint32_t *bin;              // kBinWords counters (written by the layout kernel)
    // work split of the compositing kernels: their warps, the record pool (0: no records are kept)
    uint32_t warps, rec_cap;
    const unsigned long long *n_rows;
    RefineStart refine;
    int sms;
    int block_prims, blocks;    // the projection's blocks; these and chunk (blocks a counting CTA
    int chunk;                  // takes) are set by the launchers
};
constexpr int kBinCtas = 4;              // counting and emitting CTAs per SM
constexpr int kMinChunk = kLargeBlock;   // primitives each takes at least
// A view's tiles are counted and emitted band by band, each a run of whole tile rows of at most
// kMaxSharedTiles tiles (the counters of one CTA, 48 KB).  Views have up to 4,096 tile columns, so
// that every band but a view's last has more than 8,192 tiles.
constexpr int kMaxSharedTiles = 12288;
__host__ __device__ inline int band_rows(int tiles_c) { return kMaxSharedTiles / tiles_c; }
__host__ __device__ inline int view_bands(int tiles_r, int tiles_c)
{
    return (tiles_r + band_rows(tiles_c) - 1) / band_rows(tiles_c);
}
inline int64_t cta_count_words(int sms, int max_views, int64_t max_tiles)
{
    return (int64_t{kBinCtas} * sms + max_views + max_tiles / 8192) *
           (max_tiles < kMaxSharedTiles ? max_tiles : kMaxSharedTiles);
}
// kBinHuge, kBinLong, kBinMid: tiles (in work order) with at least kHugeList, kListCap and 256
// entries; kBinSplit4, kBinSplit2: RenderArgs::split; kBinOver: the entries exceed the capacity
enum {
    kBinLong = 0, kBinMid, kBinSegments, kBinQueueSeg, kBinSplit4, kBinSplit2, kBinOver, kBinHuge,
    kBinWords
};
cudaError_t prepare_lists();    // once per device, before its first launch_lists
int bin_launches(int64_t n);    // kernels these three run for n primitives
cudaError_t launch_bin_counts(const BinArgs &a, cudaStream_t st);   // count and layout
cudaError_t launch_emit(const BinArgs &a, cudaStream_t st);
cudaError_t launch_lists(const BinArgs &a, cudaStream_t st);

// Pixel rectangle of a (view, primitive) record inside the tile_h x tile_w tile with first row rb
// and column cb, packed as 4 bytes (r_lo, r_hi, c_lo, c_hi) with the record's normal-flip bit in
// bit 31; the record's columns are cyclic modulo the image width W.  0xFF (r_lo > r_hi) when empty.
constexpr uint32_t kRectFlip = 0x80000000u;

__device__ __forceinline__ uint32_t tile_local_rect(const PairRec &rec, int rb, int cb, int W,
                                                    int tile_h, int tile_w)
{
    const int r_lo = max(rec.r0 - rb, 0), r_hi = min(rec.r1 - rb, tile_h - 1);
    const int nc = rec.nc;
    int c_lo, c_hi;
    if (rec.c0 + nc <= W) {   // the columns do not wrap
        c_lo = max(rec.c0 - cb, 0);
        c_hi = min(rec.c0 + nc - 1 - cb, tile_w - 1);
    } else {
        // c0 .. W - 1 and 0 .. last; a tile that both ends meet is taken whole
        const int last = rec.c0 + nc - 1 - W;
        const bool head = rec.c0 < cb + tile_w, tail = cb <= last;
        c_lo = tail ? 0 : max(rec.c0 - cb, 0);
        c_hi = head ? tile_w - 1 : (tail ? min(last - cb, tile_w - 1) : -1);
    }
    if (r_lo > r_hi || c_lo > c_hi) return 0xFFu;
    return static_cast<uint32_t>(r_lo) | (static_cast<uint32_t>(r_hi) << 8) |
           (static_cast<uint32_t>(c_lo) << 16) | (static_cast<uint32_t>(c_hi) << 24) |
           ((rec.cf & kPairFlip) ? kRectFlip : 0u);
}

// Which of a tile's 4 x 8 pixel blocks (bit (row block) * tile_w / 8 + column block) a rectangle
// inside the tile (tile_local_rect) meets.
__device__ __forceinline__ uint32_t rect_blocks(uint32_t rect, int tile_h, int tile_w)
{
    const int r_lo = rect & 0xFF, r_hi = (rect >> 8) & 0xFF;
    const int c_lo = (rect >> 16) & 0x3F, c_hi = (rect >> 24) & 0x3F;
    if (r_lo > r_hi || r_hi >= tile_h) return 0u;
    const uint32_t cols = ((2u << (c_hi >> 3)) - 1u) & ~((1u << (c_lo >> 3)) - 1u);
    const uint32_t rows = ((2u << (r_hi >> 2)) - 1u) & ~((1u << (r_lo >> 2)) - 1u);
    // the row bits spread tile_w / 8 apart, each times the column bits
    if (tile_w == 8) return rows;
    if (tile_w == 16)
        return cols * ((rows & 1u) | (rows & 2u) << 1 | (rows & 4u) << 2 | (rows & 8u) << 3);
    if (tile_w == 32) return cols * ((rows & 1u) | (rows & 2u) << 3);
    return cols;
}

struct RenderArgs {
    bool chain;                   // launch_chained
    const float4 *prim;           // per primitive, kPrimRow float4 written by the projection
    int64_t n;                    // primitives per view (pair id = view * n + i)
    const TileInfo *tiles;        // global tile -> frame and addressing
    const PixFrame *pixframes;
    const uint2 *ranges;          // global tile -> [start, end)
    const uint32_t *tile_order;   // tiles in decreasing order of list length (work order)
    // per list entry, in (tile, range, id) order: pair id, pixel rectangle inside its tile with
    // the flip bit
    const uint2 *entries;
    const uint8_t *entry_blocks;  // per list entry: the 4 x 8 blocks of its tile it meets
    int64_t n_tiles;
    const uint32_t *split;        // leading tiles of the order whose blocks go to 4 warps, to 2
    float alpha_min, alpha_max, t_min, sigma;
    // forward outputs (packed pixels)
    float *depth, *normal, *alpha;
    int64_t n_pixels;
    float *t_final;
    int32_t *n_last;
    // backward inputs / outputs
    const float *g_depth, *g_normal, *g_alpha;
    float4 *wgrad;                // per primitive 4 x float4 (world-frame accumulators)
    float *pose_grad;             // per view (dL/drho, dL/domega), or null
    uint32_t *queue;              // work counter (zeroed before each launch)
    // contributor records (forward writes, backward reads; see splat_render.cu)
    uint2 *rec;                   // pool of 32-record chunks, or null (no records)
    uint32_t *rec_prev;           // per chunk: the item's previous chunk
    uint32_t *rec_alloc;          // chunks taken (zeroed before the forward)
    uint32_t rec_cap;             // chunks in the pool
    uint32_t *rec_head, *rec_fill;   // per work item: last chunk and its fill
    uint32_t *status;             // status bits
    unsigned long long *evals;    // evaluation counter
};

cudaError_t launch_render_fwd(const RenderArgs &a, int tile_h, int tile_w, int grid,
                              cudaStream_t st);
cudaError_t launch_render_bwd(const RenderArgs &a, int tile_h, int tile_w, int grid,
                              cudaStream_t st);
// once per device, before the first launch on it; *ctas: how many an SM takes
cudaError_t prepare_render_fwd(int tile_h, int tile_w, int *ctas);
cudaError_t prepare_render_bwd(int tile_h, int tile_w, int *ctas);

cudaError_t launch_param_grads(const float4 *pos_logit, const float4 *quat, const float2 *log_scale,
                               const float4 *wgrad, int64_t n, float4 *g_pos_logit, float4 *g_quat,
                               float2 *g_log_scale, int accumulate, cudaStream_t st);

// active (nullable): pixels of views with active[v] == 0 count as invalid (views: the registered
// views, for the pixel -> view lookup).  normal_mode 0: normal term against t_normal; 1:
// self-regularised against the normals of the rendered range map (needs views; t_normal unused)
cudaError_t launch_loss(const float *depth, const float *normal, const float *alpha,
                        const float *t_depth, const float *t_normal, int64_t n_pixels,
                        float lambda_n, float lambda_o, float o_eps, float rho_exp,
                        float *g_depth, float *g_normal, float *g_alpha, double *loss_out,
                        cudaStream_t st, bool chain, const ViewDesc *views = nullptr,
                        int n_views = 0, const uint8_t *active = nullptr, int normal_mode = 0);

struct AdamArgs {
    bool chain;   // launch_chained (fused form)
    float4 *pos_logit;
    float4 *quat;
    float2 *log_scale;
    float4 *m_pl, *m_q;
    float2 *m_ls;
    float4 *v_pl, *v_q;
    float2 *v_ls;
    int32_t *step;
    int64_t n;
    float lr_pos, lr_opacity, lr_rot, lr_scale, beta1, beta2, eps;
    // scale term (fused form only): lambda_s max(0, max(s_a, s_b) - tau_s), added to *loss_out
    float lambda_s, tau_s;
    double *loss_out;
};

// Adam from explicit parameter gradients
cudaError_t launch_adam(const AdamArgs &a, const float4 *g_pl, const float4 *g_q,
                        const float2 *g_ls, cudaStream_t st);
// Adam with the chain rule from the world-frame accumulators fused in; *a.step already counts this
// step
cudaError_t launch_adam_fused(const AdamArgs &a, const float4 *wgrad, cudaStream_t st);
cudaError_t launch_step_inc(int32_t *step, cudaStream_t st);
// zero the accumulators of n primitives and what s names
cudaError_t launch_backward_start(const RefineStart &s, float4 *wgrad, int64_t n, bool chain,
                                  cudaStream_t st);

}  // namespace splat
