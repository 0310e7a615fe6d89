// Differentiable plane sweep: soft-argmin depth over the plane hypotheses
// and its gradient with respect to the images and the matching cameras'
// poses.  Not in the paper: the winner-take-all depth (Sec. III-A) is
// piecewise constant, so for gradients the planes are averaged with softmax
// weights of their aggregated costs:
//   s_k = exp(-C_k / T) / sum over valid k' of exp(-C_k' / T)
//   range = 1 / sum_k s_k rho_k,   rho_k = (n_k . r) / d_k,
// and the soft minimum S = -T log sum_k exp(-C_k / T) is a second output.
// C_k = min over the matching cameras of (1 - ZNCC) / 2 (lowest camera index
// on a tie), exactly the sweep's cost but on real-valued images.
//
// Kernels (planes in pairs on packed FP32):
//   soft_fwd_kernel  32 x 16 output pixels: per pair of planes and camera,
//                    warp the tile + window halo into shared memory; two-pass
//                    window ZNCC, two pixels per thread so that they share the
//                    window rows they load; minimum over cameras; online
//                    softmax over planes.
//   soft_bwd_kernel  16 x 16 output pixels: recomputes the same costs (bit-
//                    identical), forms dL/dC_k, spreads dL/dZNCC over both
//                    windows as separable box sums of per-pixel coefficients,
//                    then per warped halo sample with a gradient warps it
//                    again with its derivative, scatters dL/dI to the 4
//                    bilinear texels and adds dL/dw times the sample's pose
//                    derivative to a left perturbation (w, v) of each
//                    ref_to_cam pose (CTA reduction, FP64 atomics).
// Both are bound by instruction issue and latency (DRAM holds the images and
// ray table once).  A forward and backward pass through autograd, 640 x 512,
// 128 planes, 2 cameras: 5.93 -> 3.87 ms (device time of the backward kernel
// 4.22 -> 2.57 ms on a street scene, 2.77 ms on textured rectangles: samples
// without a gradient are skipped); 96 x 80, 32 planes: 686 -> 537 us.
// Before: one pixel per thread, general divisions and square roots (their
// slow-path branches serialise a thread's samples), the reference window's
// sums repeated per plane, and a backward of one plane at a time with seven
// barriers and its chain data in shared memory.
//
// Low-texture windows have coefficients so large that a changed rounding of a
// cost or a coefficient shows in the image gradients (2e-5 .. 7e-5 of their
// norm in a build that merged coefficient fields and softmax parts), so costs,
// softmax, box sums and the pose accumulators keep one order whatever the
// tiling.
#include <algorithm>
#include <cfloat>
#include <cmath>
#include <cstring>
#include <type_traits>
#include <vector>

#include "sweep_dev.cuh"

namespace ps {
int build_rays(const ps_camera& cam, float4* rays, double* max_angle);

namespace {

struct DiffCam {
    int width, height;
    const float* img;
    float r2_max;
    // projection constants, and those of its derivative, as (value, value) pairs
    float2 R2[9], t2[3], xi, fx, fy, cx, cy, k1, k2, k2x2, p1, p1x2, p1x6, p2, p2x2, p2x6, lim;
    float u_max, v_max;  // largest coordinates inside the image (read for wide images)
};

struct DiffP {
    int W, H, rho, K, n_cams;
    float T;
    const float4* rays;
    const PlaneD* planes;
    const float* ref;
    DiffCam cams[PS_MAX_CAMS];
};

// n . r of a plane and a ray.  The plane's offset along the ray, and the
// bilinear blend below, are written with explicit roundings so that every
// kernel computes the same samples (the costs decide integers: a camera, a
// plane) whatever contractions the compiler would choose in each.
__device__ __forceinline__ float plane_dot(const PlaneD& pl, const float4& r) {
    return __fmaf_rn(pl.nz, r.z, __fmaf_rn(pl.ny, r.y, __fmul_rn(pl.nx, r.x)));
}

__device__ __forceinline__ float bilerp(float ax, float ay, float i00, float i10, float i01, float i11) {
    const float bx = __fsub_rn(1.0f, ax), by = __fsub_rn(1.0f, ay);
    const float top = __fmaf_rn(ax, i10, __fmul_rn(bx, i00));
    const float bot = __fmaf_rn(ax, i11, __fmul_rn(bx, i01));
    return __fmaf_rn(ay, bot, __fmul_rn(by, top));
}

// Halo position r (its ray) through the planes p0 (lane x) and p1 (lane y)
// into camera C: the point in the camera frame, the projection (unified
// model, then distortion) with its intermediate values, and whether each
// lane projects (plane before the ray, sphere side, distortion range).
struct Proj {
    float2 X, Y, Z, n, inv, mx, my, r2, rad, u, v;
    bool ok0, ok1;
};
__device__ __forceinline__ Proj project_pair(const DiffCam& C, const PlaneD& p0, const PlaneD& p1, const float4& r) {
    Proj o;
    const float2 nr = make_float2(plane_dot(p0, r), plane_dot(p1, r));
    const float2 lam = div_rn2(make_float2(p0.d, p1.d), nr, rcp_rn2(nr));
    const float2 x = mul2(lam, dup2(r.x)), y = mul2(lam, dup2(r.y)), z = mul2(lam, dup2(r.z));
    o.X = fma2(C.R2[0], x, fma2(C.R2[1], y, fma2(C.R2[2], z, C.t2[0])));
    o.Y = fma2(C.R2[3], x, fma2(C.R2[4], y, fma2(C.R2[5], z, C.t2[1])));
    o.Z = fma2(C.R2[6], x, fma2(C.R2[7], y, fma2(C.R2[8], z, C.t2[2])));
    o.n = sqrt_rn2(fma2(o.X, o.X, fma2(o.Y, o.Y, mul2(o.Z, o.Z))));
    o.inv = rcp_rn2(fma2(C.xi, o.n, o.Z));
    o.mx = mul2(o.X, o.inv);
    o.my = mul2(o.Y, o.inv);
    o.r2 = fma2(o.mx, o.mx, mul2(o.my, o.my));
    o.rad = fma2(o.r2, fma2(C.k2, o.r2, C.k1), dup2(1.0f));
    const float2 mxy = mul2(o.mx, o.my);
    const float2 xd = fma2(o.mx, o.rad, fma2(C.p1x2, mxy, mul2(C.p2, fma2(add2(o.mx, o.mx), o.mx, o.r2))));
    const float2 yd = fma2(o.my, o.rad, fma2(C.p1, fma2(add2(o.my, o.my), o.my, o.r2), mul2(C.p2x2, mxy)));
    o.u = fma2(C.fx, xd, C.cx);
    o.v = fma2(C.fy, yd, C.cy);
    const float2 ln = mul2(C.lim, o.n);
    o.ok0 = nr.x > 0.0f && o.Z.x > ln.x && o.r2.x <= C.r2_max;
    o.ok1 = nr.y > 0.0f && o.Z.y > ln.y && o.r2.y <= C.r2_max;
    return o;
}

// The bilinear cell of camera C at (u, v), clamped into the image: corner
// offsets and weights; false when (u, v) lies outside [0, W-1] x [0, H-1].
// WIDE: images of 2^31 texels or more, or of a side above 2^24, whose offsets
// take 64 bits and whose last coordinate may be no float (64 bits for every
// image: 640 x 512, 128 planes, 2 cameras 1250 -> 1280 us forward, 2475 ->
// 2518 backward; an index per row more still).
template <bool WIDE>
struct Cell {
    std::conditional_t<WIDE, long long, int> i00, i10, i01, i11;
    float ax, ay;
};
template <bool WIDE>
__device__ __forceinline__ bool cell_at(const DiffCam& C, float u, float v, Cell<WIDE>& c) {
    const float uc = fminf(fmaxf(u, 0.0f), WIDE ? C.u_max : (float)(C.width - 1)),
                vc = fminf(fmaxf(v, 0.0f), WIDE ? C.v_max : (float)(C.height - 1));
    int x = (int)uc, y = (int)vc;
    if (!PS_DCHECK(x >= 0 && y >= 0 && x < C.width && y < C.height, CHK_GATHER)) x = y = 0;
    const int dx = x < C.width - 1 ? 1 : 0, dy = y < C.height - 1 ? C.width : 0;
    c.i00 = static_cast<decltype(c.i00)>(y) * C.width + x;
    c.i10 = c.i00 + dx;
    c.i01 = c.i00 + dy;
    c.i11 = c.i01 + dx;
    c.ax = uc - (float)x;
    c.ay = vc - (float)y;
    return uc == u && vc == v;
}

// Samples of camera C at a halo position through two planes (lane x: p0, lane
// y: p1); NaN where invalid (no ray, plane behind the ray, no projection,
// outside the image).  The gathers are clamped into the image and always
// issued, so nothing branches and a thread's positions overlap.
template <bool WIDE>
__device__ __forceinline__ float2 warp_pair(const DiffCam& C, const PlaneD& p0, const PlaneD& p1, const float4& r) {
    const float nan = __int_as_float(0x7fc00000);
    const Proj o = project_pair(C, p0, p1, r);
    Cell<WIDE> a, b;
    const bool in0 = cell_at(C, o.u.x, o.v.x, a), in1 = cell_at(C, o.u.y, o.v.y, b);
    const float* I = C.img;
    const float w0 = bilerp(a.ax, a.ay, I[a.i00], I[a.i10], I[a.i01], I[a.i11]);
    const float w1 = bilerp(b.ax, b.ay, I[b.i00], I[b.i10], I[b.i01], I[b.i11]);
    return make_float2(o.ok0 && in0 ? w0 : nan, o.ok1 && in1 ? w1 : nan);
}

// ----------------------------------------------------------------- tiles
//
// A CTA of ST threads works on SW columns of output pixels: thread t owns the
// PX pixels of column t % SW from row PX (t / SW), so that a window row that
// several of them hold is loaded once.  Planes go in pairs (lane x: the first
// plane, lane y: the second) on packed FP32.
constexpr int ST = 256;  // threads per CTA

template <int RHO_, int SW_, int PX_>
struct Tile {
    static constexpr int RHO = RHO_, SW = SW_, PX = PX_;
    static constexpr int TH = ST / SW * PX;                // output rows
    static constexpr int HWC = SW + 2 * RHO, HH = TH + 2 * RHO, NPOS = HWC * HH;
    static constexpr int RPT = (NPOS + ST - 1) / ST;       // halo positions per thread
    static constexpr int N = (2 * RHO + 1) * (2 * RHO + 1);
    // row stride of the reference samples: 16 mod 32 where a warp covers two
    // rows of 16, so that they reach distinct banks
    static constexpr int RS = SW == 16 ? 48 : HWC;
};

// Mean and sum of squared deviations of the reference windows of a thread's
// PX pixels (R: halo layout, the first pixel's window at lx, ly).  One pass
// each in row-major window order.
template <class G>
__device__ __forceinline__ void ref_windows(const float* R, int lx, int ly, float (&ma)[G::PX], float (&va)[G::PX]) {
    constexpr int RHO = G::RHO, PX = G::PX;
#pragma unroll
    for (int i = 0; i < PX; ++i) {
        float s = 0.f;
        for (int dy = 0; dy <= 2 * RHO; ++dy)
#pragma unroll
            for (int dx = 0; dx <= 2 * RHO; ++dx) s += R[(ly + i + dy) * G::RS + lx + dx];
        const float m = s / (float)G::N;
        float v = 0.f;
        for (int dy = 0; dy <= 2 * RHO; ++dy)
#pragma unroll
            for (int dx = 0; dx <= 2 * RHO; ++dx) {
                const float e = R[(ly + i + dy) * G::RS + lx + dx] - m;
                v = fmaf(e, e, v);
            }
        ma[i] = m;
        va[i] = v;
    }
}

// Two-pass ZNCC sums of both planes for a thread's PX pixels under each
// other: warped pairs W, reference R (halo layout).  Per pixel and plane the
// sums run over the window in row-major order; a window row shared by
// several pixels is loaded once.  An invalid sample is NaN and makes the
// mean NaN.
template <class G>
__device__ __forceinline__ void pair_windows(const float* R, const float2* W, int lx, int ly, const float (&ma)[G::PX],
                                             float2 (&mb)[G::PX], float2 (&cov)[G::PX], float2 (&vb)[G::PX]) {
    constexpr int RHO = G::RHO, PX = G::PX;
#pragma unroll
    for (int i = 0; i < PX; ++i) mb[i] = cov[i] = vb[i] = dup2(0.f);
#pragma unroll
    for (int y = 0; y < 2 * RHO + PX; ++y)
#pragma unroll
        for (int dx = 0; dx <= 2 * RHO; ++dx) {
            const float2 b = W[(ly + y) * G::HWC + lx + dx];
#pragma unroll
            for (int i = 0; i < PX; ++i)
                if (y - i >= 0 && y - i <= 2 * RHO) mb[i] = add2(mb[i], b);
        }
    float2 nmb[PX];
#pragma unroll
    for (int i = 0; i < PX; ++i) {
        mb[i] = div_rn2(mb[i], dup2((float)G::N), dup2(1.0f / (float)G::N));
        nmb[i] = neg2(mb[i]);
    }
    asm volatile("" ::: "memory");  // the second pass loads again: keeping the window in registers would spill
#pragma unroll
    for (int y = 0; y < 2 * RHO + PX; ++y)
#pragma unroll
        for (int dx = 0; dx <= 2 * RHO; ++dx) {
            const float2 b = W[(ly + y) * G::HWC + lx + dx];
            const float a = R[(ly + y) * G::RS + lx + dx];
#pragma unroll
            for (int i = 0; i < PX; ++i)
                if (y - i >= 0 && y - i <= 2 * RHO) {
                    const float2 ea = dup2(a - ma[i]), eb = add2(b, nmb[i]);
                    cov[i] = fma2(ea, eb, cov[i]);
                    vb[i] = fma2(eb, eb, vb[i]);
                }
        }
}

// ZNCC of both planes from the window sums, and the root of the variances'
// product that divides it.  Variances whose product overflows have an infinite
// root, and no correlation.
struct Corr {
    float2 z, s;
};
__device__ __forceinline__ Corr correlation(float va, float2 vb, float2 cov) {
    const float inf = __int_as_float(0x7f800000);
    const float2 p = mul2(dup2(va), vb);
    Corr o;
    o.s = sqrt_rn2(p);
    o.z = div_rn2(cov, o.s, rcp_rn2(o.s));
    if (p.x == inf) o.s.x = inf, o.z.x = __fmul_rn(cov.x, 0.f);
    if (p.y == inf) o.s.y = inf, o.z.y = __fmul_rn(cov.y, 0.f);
    return o;
}

// The tile's reference samples (zero outside the image).
template <class G>
__device__ __forceinline__ void load_ref(const DiffP& P, int x0, int y0, float* R) {
    for (int p = threadIdx.x; p < G::NPOS; p += blockDim.x) {
        const int hy = p / G::HWC, hx = p - hy * G::HWC, x = x0 + hx, y = y0 + hy;
        R[hy * G::RS + hx] = (x >= 0 && y >= 0 && x < P.W && y < P.H) ? P.ref[(size_t)y * P.W + x] : 0.0f;
    }
}

// Ray of image position (x, y), NaN outside the image.
__device__ __forceinline__ float4 ray_at(const DiffP& P, int x, int y) {
    const float nan = __int_as_float(0x7fc00000);
    return x >= 0 && y >= 0 && x < P.W && y < P.H ? P.rays[(size_t)y * P.W + x] : make_float4(nan, nan, nan, 0.f);
}

// Warped sample pairs of the halo, every camera, by the ST threads tid.
template <class G, bool WIDE>
__device__ __forceinline__ void warp_tile(const DiffP& P, const PlaneD& pl0, const PlaneD& pl1, int x0, int y0, int tid,
                                          float2* W2) {
    for (int j = 0; j < P.n_cams; ++j)
#pragma unroll
        for (int i = 0; i < G::RPT; ++i) {
            const int p = tid + i * ST;
            if (p < G::NPOS) W2[j * G::NPOS + p] = warp_pair<WIDE>(P.cams[j], pl0, pl1, ray_at(P, x0 + p % G::HWC, y0 + p / G::HWC));
        }
}

// The forward's CTA: FG groups of ST threads share a tile and take alternate
// pairs of planes; each pixel's costs of a round of ROUND planes wait in
// shared memory, then every thread goes over them in plane order for the
// pixels it owns there.  The online softmax thus adds the planes one by one
// in plane order, while two groups halve the time of a tile: 640 tiles of 32
// x 16 pixels (640 x 512) are 4.2 waves of one 512-thread CTA per SM instead
// of 2.1 waves of two of 256 threads.
constexpr int FG = 2;
constexpr int ROUND = 16;

template <class G, bool WIDE>
__global__ void __launch_bounds__(FG * ST, 1) soft_fwd_kernel(const __grid_constant__ DiffP P, float* range, float* cost,
                                                              float* aux) {
    constexpr int RHO = G::RHO, PX = G::PX, SW = G::SW, NPIX = ST * PX;
    constexpr int OWN = (NPIX + FG * ST - 1) / (FG * ST);             // pixels a thread owns in the softmax
    extern __shared__ __align__(16) float sm[];
    float* Cs = sm;                                                   // [ROUND][NPIX] costs (inf = invalid)
    const int group = threadIdx.x / ST, tid = threadIdx.x % ST;
    float2* W2 = reinterpret_cast<float2*>(Cs + ROUND * NPIX) + group * P.n_cams * G::NPOS;  // [n_cams][NPOS] warped pairs
    float* R = Cs + ROUND * NPIX + 2 * FG * P.n_cams * G::NPOS;       // [NPOS] reference
    const int lx = tid % SW, ly = tid / SW * PX;
    const int bx = blockIdx.x * SW, by = blockIdx.y * G::TH;
    load_ref<G>(P, bx - RHO, by - RHO, R);
    __syncthreads();
    float ma[PX], va[PX];
    ref_windows<G>(R, lx, ly, ma, va);
    const float inf = __int_as_float(0x7f800000);
    const float lim = (float)G::N * 1e-8f, inv_T = __frcp_rn(P.T);
    float cmin[OWN], Z[OWN], Nr[OWN];
#pragma unroll
    for (int i = 0; i < OWN; ++i) {
        cmin[i] = inf;
        Z[i] = Nr[i] = 0.f;
    }
    for (int base = 0; base < P.K; base += ROUND) {
        const int n = min(P.K - base, ROUND);
        for (int k0 = 0; k0 < n; k0 += 2 * FG) {
            // a group past the round's end repeats its last plane and stores nothing
            const int k = k0 + 2 * group, np = max(0, min(2, n - k));
            const PlaneD pl0 = P.planes[base + min(k, n - 1)], pl1 = P.planes[base + min(k + 1, n - 1)];
            __syncthreads();  // the previous pairs' windows are done
            warp_tile<G, WIDE>(P, pl0, pl1, bx - RHO, by - RHO, tid, W2);
            __syncthreads();
            float2 best[PX];
#pragma unroll
            for (int i = 0; i < PX; ++i) best[i] = dup2(inf);
            for (int j = 0; j < P.n_cams; ++j) {
                float2 mb[PX], cov[PX], vb[PX];
                pair_windows<G>(R, W2 + j * G::NPOS, lx, ly, ma, mb, cov, vb);
#pragma unroll
                for (int i = 0; i < PX; ++i) {
                    const bool ok0 = !isnan(mb[i].x) && !(va[i] < lim || vb[i].x < lim);
                    const bool ok1 = !isnan(mb[i].y) && !(va[i] < lim || vb[i].y < lim);
                    const float2 z = correlation(va[i], vb[i], cov[i]).z;
                    const float c0 = 0.5f * (1.0f - z.x), c1 = 0.5f * (1.0f - z.y);
                    if (ok0 && c0 < best[i].x) best[i].x = c0;
                    if (ok1 && c1 < best[i].y) best[i].y = c1;
                }
            }
#pragma unroll
            for (int i = 0; i < PX; ++i) {
                float* c = Cs + k * NPIX + (ly + i) * SW + lx;
                if (np > 0) c[0] = best[i].x;
                if (np > 1) c[NPIX] = best[i].y;
            }
        }
        __syncthreads();
#pragma unroll
        for (int i = 0; i < OWN; ++i) {
            const int px = threadIdx.x + i * FG * ST;
            if (px >= NPIX) continue;
            const float4 ray = ray_at(P, bx + px % SW, by + px / SW);
            for (int k = 0; k < n; ++k) {
                const PlaneD pl = P.planes[base + k];
                const float bq = Cs[k * NPIX + px];
                const float rho_k = div_rn(plane_dot(pl, ray), pl.d, rcp_rn(pl.d));
                // the smaller of the old minimum and bq becomes the new one; the
                // other side's weight is exp(-|difference| / T), its own 1
                const bool on = bq < inf, lt = on && bq < cmin[i];
                const float x = lt ? cmin[i] - bq : bq - cmin[i];
                const float f = x < inf ? __expf(-div_rn(x, P.T, inv_T)) : 0.f;
                const float z = lt ? __fadd_rn(__fmul_rn(Z[i], f), 1.0f) : __fadd_rn(Z[i], f);
                const float w = lt ? __fmaf_rn(1.0f, rho_k, __fmul_rn(Nr[i], f)) : __fmaf_rn(f, rho_k, Nr[i]);
                Z[i] = on ? z : Z[i];
                Nr[i] = on ? w : Nr[i];
                cmin[i] = fminf(cmin[i], bq);
            }
        }
        __syncthreads();  // the costs stay until they are read
    }
#pragma unroll
    for (int i = 0; i < OWN; ++i) {
        const int px = threadIdx.x + i * FG * ST;
        const int gx = bx + px % SW, gy = by + px / SW;
        if (px >= NPIX || gx >= P.W || gy >= P.H) continue;
        const size_t o = (size_t)gy * P.W + gx;
        const bool use = gx >= RHO && gy >= RHO && gx < P.W - RHO && gy < P.H - RHO && !isnan(P.rays[o].x);
        const bool ok = use && cmin[i] < inf;
        range[o] = ok ? Z[i] / Nr[i] : 0.f;
        if (cost) cost[o] = ok ? cmin[i] - P.T * logf(Z[i]) : 0.f;
        if (aux) {
            aux[3 * o] = ok ? cmin[i] : inf;
            aux[3 * o + 1] = use ? Z[i] : 0.f;
            aux[3 * o + 2] = ok ? Nr[i] / Z[i] : 0.f;
        }
    }
}

struct GradOut {
    float* cam[PS_MAX_CAMS];
};

// Shared memory of the backward kernel, in floats, for nc matching cameras
// and nf = 4 nc + 3 coefficient fields (all of them pairs).
template <int RHO, int MC>
struct BwdLayout {
    using G = Tile<RHO, 16, 1>;
    // Zeros on either side of the direction that is summed, so that no sum tests
    // its bounds (written once; with the reference stride RS 2837 -> 2782 us at
    // 640 x 512, 128 planes, 2 cameras): PF columns of the fields, PH rows of the
    // horizontal sums.  Two CTAs per SM are worth more than the tests, so 3 and
    // 4 cameras, and the fields of the widest window, go without.
    static constexpr int PH = MC == 2 ? 2 * RHO : 0, PF = MC == 2 && RHO < 4 ? 2 * RHO : 0;
    static constexpr int HR = G::TH + 2 * PH;        // horizontal sums' rows
    static constexpr int RO = (G::HWC + 3) / 4;      // outputs of a horizontal item
    // Row strides in pairs (16 of them span the banks).  HS = HWC: consecutive
    // halo positions are consecutive words, so the vertical sums, most of the
    // traffic, have no conflict and need no row index.  A half-warp of the
    // horizontal sums takes 4 parts of 4 rows: with 5 outputs a part and strides
    // of 4 or 12 mod 16 (window 5) all 16 words differ.
    // Odd strides and a warp per part before: 2780 -> 2567 us (as above).
    static constexpr int HS = G::HWC;
    static constexpr int FS = RO != 5 ? G::SW + 2 * PF + 1 : PF ? 28 : 20;
    static_assert(FS >= G::SW + 2 * PF && 4 * RO >= G::HWC, "rows hold their margins");
    __host__ __device__ static constexpr int nf(int nc) { return 4 * nc + 3; }
    // warped pairs [nc][NPOS], fields [nf][TH][FS], horizontal sums [nf][HR][HS], reference [HH][RS]
    __host__ __device__ static constexpr size_t floats(int nc) {
        return 2 * ((size_t)nc * G::NPOS + (size_t)nf(nc) * (G::TH * FS + HR * HS)) + G::HH * G::RS;
    }
};

// Chain of one halo position's samples of both planes in one camera: gw =
// dL/dw per plane goes to the image's four texels (global atomics, img may be
// NULL); m receives (X x g, g) with g = J^T (dw/du, dw/dv), J the 2 x 3
// projection Jacobian at X (camera frame): gw m is the samples' contribution
// to the gradient of a left perturbation (w, v) of ref_to_cam.
// The warp is the forward's; g comes from reverse-mode differentiation of the
// projection: the adjoints of the distorted point, of the normalised point
// (mx, my), then of X through mx = X / den, my = Y / den, den = xi |X| + Z.
template <bool WIDE>
__device__ __forceinline__ void chain_pair(const DiffCam& C, const PlaneD& p0, const PlaneD& p1, const float4& r,
                                           float2 gw, float* img, float2 (&m)[6]) {
    const Proj o = project_pair(C, p0, p1, r);
    Cell<WIDE> c[2];
    cell_at(C, o.u.x, o.v.x, c[0]);
    cell_at(C, o.u.y, o.v.y, c[1]);
    float2 gu, gv;
    const float* I = C.img;
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const float i00 = I[c[q].i00], i10 = I[c[q].i10], i01 = I[c[q].i01], i11 = I[c[q].i11];
        const float ax = c[q].ax, ay = c[q].ay;
        (q ? gu.y : gu.x) = __fmaf_rn(1.f - ay, i10 - i00, __fmul_rn(ay, i11 - i01));
        (q ? gv.y : gv.x) = __fmaf_rn(1.f - ax, i01 - i00, __fmul_rn(ax, i11 - i10));
    }
    const float2 drad = fma2(C.k2x2, o.r2, C.k1);
    // d(xd, yd)/d(mx, my) = [[a, b], [b, d]]
    const float2 mx = o.mx, my = o.my, mx2 = add2(mx, mx), my2 = add2(my, my);
    const float2 a = fma2(C.p2x6, mx, fma2(C.p1x2, my, fma2(mul2(mx2, mx), drad, o.rad)));
    const float2 b = fma2(C.p2x2, my, fma2(mul2(mx2, my), drad, mul2(C.p1x2, mx)));
    const float2 d = fma2(C.p2x2, mx, fma2(C.p1x6, my, fma2(mul2(my2, my), drad, o.rad)));
    const float2 gxd = mul2(gu, C.fx), gyd = mul2(gv, C.fy);
    const float2 gmx = fma2(gxd, a, mul2(gyd, b)), gmy = fma2(gxd, b, mul2(gyd, d));
    const float2 gden = neg2(mul2(fma2(gmx, mx, mul2(gmy, my)), o.inv));  // dL/dden
    const float2 xn = div_rn2(C.xi, o.n, rcp_rn2(o.n));                   // d(xi n)/dX = xi X / n
    const float2 gx = mul2(gden, xn);
    const float2 g0 = fma2(gmx, o.inv, mul2(gx, o.X)), g1 = fma2(gmy, o.inv, mul2(gx, o.Y));
    const float2 g2 = mul2(gden, fma2(xn, o.Z, dup2(1.0f)));
    m[0] = fma2(o.Y, g2, neg2(mul2(o.Z, g1)));
    m[1] = fma2(o.Z, g0, neg2(mul2(o.X, g2)));
    m[2] = fma2(o.X, g1, neg2(mul2(o.Y, g0)));
    m[3] = g0;
    m[4] = g1;
    m[5] = g2;
    if (img) {
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const float g = q ? gw.y : gw.x, ax = c[q].ax, ay = c[q].ay;
            if (g == 0.f) continue;
            if (!PS_DCHECK(c[q].i00 >= 0 && (long long)c[q].i11 < (long long)C.width * C.height, CHK_GATHER)) continue;
            atomicAdd(&img[c[q].i00], g * (1.f - ax) * (1.f - ay));
            atomicAdd(&img[c[q].i10], g * ax * (1.f - ay));
            atomicAdd(&img[c[q].i01], g * (1.f - ax) * ay);
            atomicAdd(&img[c[q].i11], g * ax * ay);
        }
    }
}

// Backward of the soft sweep for one 16 x 16 tile.  Per pair of planes:
//  1. warp the halo for every camera, as in the forward;
//  2. per pixel and plane, the cost and winning camera jb as in the forward,
//     dL/dC, and the ZNCC gradient coefficients ka = gz / sqrt(va vb),
//     kz_a = gz z / va, kz_b = gz z / vb (gz = dL/dZNCC);
//  3. window gradients as box sums.  For a window sample q of pixel p,
//       dZNCC/da_q = (b_q - mb) / sqrt(va vb) - z (a_q - ma) / va   (a: ref)
//       dZNCC/db_q = (a_q - ma) / sqrt(va vb) - z (b_q - mb) / vb   (b: camera jb)
//     so, summed over the pixels whose window holds q,
//       gW_j(q) = a_q A1_j - A2_j - b_q A3_j + A4_j
//       gR(q)  += sum_j b_j(q) A1_j - B1 - a_q B2 + B3
//     with A1_j..A4_j the (2 RHO + 1)^2 box sums of ka, ka ma, kz_b, kz_b mb
//     over pixels with jb = j, and B1..B3 those of ka mb, kz_a, kz_a ma.
//     Intensities are taken relative to a per-tile centre (a) and a
//     per-plane, per-camera centre (b), which leaves every difference
//     unchanged and keeps the products small.  The box sums are separable
//     (rows, then columns) in shared memory: no atomics;
//  4. chain every sample with dL/dw != 0 (chain_pair: the warp of such a
//     sample is computed again rather than kept from step 1).
// After the planes: dL/dref of the halo (global atomics) and the CTA's pose
// gradient (FP64 atomics).  MC: most cameras (their pose accumulators are
// registers).
template <int RHO, int MC, bool WIDE>
__global__ void __launch_bounds__(ST, 2) soft_bwd_kernel(const __grid_constant__ DiffP P, const float* aux,
                                                         const float* g_range, const float* g_cost, float* g_ref,
                                                         const __grid_constant__ GradOut GO, double* g_pose) {
    using BL = BwdLayout<RHO, MC>;
    using G = typename BL::G;
    constexpr int HWC = G::HWC, NPOS = G::NPOS, TH = G::TH, SW = G::SW, FS = BL::FS, HS = BL::HS, HR = BL::HR, RO = BL::RO, PF = BL::PF,
                  PH = BL::PH, N = G::N, RPT = G::RPT;
    constexpr int PX = 1;
    const int nc = P.n_cams, nf = BL::nf(nc);
    extern __shared__ __align__(16) float sm[];
    float2* W2 = reinterpret_cast<float2*>(sm);
    float2* F = W2 + nc * NPOS;
    float2* Hx = F + nf * TH * FS;
    float* R = reinterpret_cast<float*>(Hx + nf * HR * HS);
    __shared__ float red[ST / 32][6 * MC];
    const int tid = threadIdx.x, lx = tid % SW, ly = tid / SW * PX;
    const int bx = blockIdx.x * SW, by = blockIdx.y * TH, x0 = bx - RHO, y0 = by - RHO;
    load_ref<G>(P, x0, y0, R);
    for (int i = tid; i < nf * (TH * FS + HR * HS); i += ST) F[i] = dup2(0.f);  // fields and horizontal sums
    __syncthreads();
    float ma[PX], va[PX];
    ref_windows<G>(R, lx, ly, ma, va);
    const float inf = __int_as_float(0x7f800000);
    const float lim = (float)N * 1e-8f, inv_T = __frcp_rn(P.T);
    float cmin[PX], Z[PX], E[PX], gE[PX], gs[PX];
    bool use[PX];
#pragma unroll
    for (int i = 0; i < PX; ++i) {
        const int gx = bx + lx, gy = by + ly + i;
        const bool in = gx >= RHO && gy >= RHO && gx < P.W - RHO && gy < P.H - RHO;
        const size_t o = in ? (size_t)gy * P.W + gx : 0;
        cmin[i] = in ? aux[3 * o] : inf;
        Z[i] = in ? aux[3 * o + 1] : 1.f;
        E[i] = in ? aux[3 * o + 2] : 0.f;
        const float gr = in && g_range ? g_range[o] : 0.f;
        gs[i] = in && g_cost ? g_cost[o] : 0.f;
        use[i] = in && !isnan(P.rays[o].x) && cmin[i] < inf && (gr != 0.f || gs[i] != 0.f);
        gE[i] = use[i] ? -gr / (E[i] * E[i]) : 0.f;
    }
    float pose_acc[MC][6];
#pragma unroll
    for (int j = 0; j < MC; ++j)
#pragma unroll
        for (int i = 0; i < 6; ++i) pose_acc[j][i] = 0.f;
    float gR[RPT];
#pragma unroll
    for (int i = 0; i < RPT; ++i) gR[i] = 0.f;
    const int qc = (RHO + TH / 2) * HWC + RHO + SW / 2;  // centre of the tile
    auto finite = [&](float v) { return fabsf(v) < inf ? v : 0.f; };  // a centre that is none must not reach all of the tile
    const float ca = finite(R[(RHO + TH / 2) * G::RS + RHO + SW / 2]);
    for (int k = 0; k < P.K; k += 2) {
        const int np = min(2, P.K - k);
        const PlaneD pl0 = P.planes[k], pl1 = P.planes[k + np - 1];
        __syncthreads();  // the previous pair's chain is done with the samples and sums
        warp_tile<G, WIDE>(P, pl0, pl1, x0, y0, tid, W2);
        __syncthreads();
        // the per-camera centre of this pair's warped samples (a broadcast read)
        auto centre = [&](int j) {
            const float2 c = W2[j * NPOS + qc];
            return make_float2(finite(c.x), finite(c.y));
        };
        // 2. cost, camera and coefficients
        float best[PX][2], z[PX][2], mb[PX][2], vb[PX][2], sab[PX][2];
        int jb[PX][2];
#pragma unroll
        for (int i = 0; i < PX; ++i)
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                best[i][q] = inf;
                z[i][q] = mb[i][q] = 0.f;
                vb[i][q] = sab[i][q] = 1.f;
                jb[i][q] = -1;
            }
        for (int j = 0; j < nc; ++j) {
            float2 m2[PX], c2[PX], v2[PX];
            pair_windows<G>(R, W2 + j * NPOS, lx, ly, ma, m2, c2, v2);
            float2 ss[PX], zz[PX];
#pragma unroll
            for (int i = 0; i < PX; ++i) {
                const Corr o = correlation(va[i], v2[i], c2[i]);
                ss[i] = o.s;
                zz[i] = o.z;
            }
#pragma unroll
            for (int i = 0; i < PX; ++i)
#pragma unroll
                for (int q = 0; q < 2; ++q) {
                    const float m = q ? m2[i].y : m2[i].x, v = q ? v2[i].y : v2[i].x;
                    const bool ok = use[i] && q < np && !isnan(m) && !(va[i] < lim || v < lim);
                    const float c = 0.5f * (1.0f - (q ? zz[i].y : zz[i].x));
                    if (ok && c < best[i][q]) {
                        best[i][q] = c;
                        jb[i][q] = j;
                        z[i][q] = q ? zz[i].y : zz[i].x;
                        mb[i][q] = m;
                        vb[i][q] = v;
                        sab[i][q] = q ? ss[i].y : ss[i].x;
                    }
                }
        }
#pragma unroll
        for (int i = 0; i < PX; ++i) {
            const float4 ray = P.rays[use[i] ? (size_t)(by + ly + i) * P.W + bx + lx : 0];
            // all of them zero where no camera wins: a window that holds a sample
            // that is no number must not pass it on to its neighbours' sums
            float ka[2], kza[2], kzb[2], mac[2], mbc[2];
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const PlaneD& pl = q == 0 ? pl0 : pl1;
                const float2 cb = centre(max(jb[i][q], 0));
                // (a square root or quotient of a window that is not used may be NaN)
                const float ez = __expf(div_rn(-(best[i][q] - cmin[i]), P.T, inv_T));
                const float s = div_rn(ez, Z[i], rcp_rn(Z[i]));
                const float rho_k = div_rn(plane_dot(pl, ray), pl.d, rcp_rn(pl.d));
                const float gC = gE[i] * div_rn(-s * (rho_k - E[i]), P.T, inv_T) + gs[i] * s;
                const float gz = -0.5f * gC, gzz = gz * z[i][q];
                const bool on = jb[i][q] >= 0;
                const bool finite = on && sab[i][q] < inf;  // (otherwise all three are zero)
                ka[q] = finite ? div_rn(gz, sab[i][q], rcp_rn(sab[i][q])) : 0.f;
                kza[q] = finite ? div_rn(gzz, va[i], rcp_rn(va[i])) : 0.f;
                kzb[q] = finite ? div_rn(gzz, vb[i][q], rcp_rn(vb[i][q])) : 0.f;
                mac[q] = on ? ma[i] - ca : 0.f;
                mbc[q] = on ? mb[i][q] - (q ? cb.y : cb.x) : 0.f;
            }
            float2* f = F + (ly + i) * FS + PF + lx;
            for (int j = 0; j < nc; ++j) {
                const bool m0 = jb[i][0] == j, m1 = jb[i][1] == j;
                f[(4 * j + 0) * TH * FS] = make_float2(m0 ? ka[0] : 0.f, m1 ? ka[1] : 0.f);
                f[(4 * j + 1) * TH * FS] = make_float2(m0 ? ka[0] * mac[0] : 0.f, m1 ? ka[1] * mac[1] : 0.f);
                f[(4 * j + 2) * TH * FS] = make_float2(m0 ? kzb[0] : 0.f, m1 ? kzb[1] : 0.f);
                f[(4 * j + 3) * TH * FS] = make_float2(m0 ? kzb[0] * mbc[0] : 0.f, m1 ? kzb[1] * mbc[1] : 0.f);
            }
            f[(4 * nc + 0) * TH * FS] = make_float2(ka[0] * mbc[0], ka[1] * mbc[1]);
            f[(4 * nc + 1) * TH * FS] = make_float2(kza[0], kza[1]);
            f[(4 * nc + 2) * TH * FS] = make_float2(kza[0] * mac[0], kza[1] * mac[1]);
        }
        __syncthreads();
        // 3a. horizontal box sums: halo column c collects pixels c - 2 RHO .. c of
        // the row.  Direct sums, not running ones: coefficients of low-texture
        // windows are large, and a running sum would leave their rounding residue
        // where the exact sum is zero
        for (int it = tid; it < 4 * nf * TH; it += ST) {
            const int fr = it / 4, c0 = it % 4 * RO;
            const float2* in = F + fr * FS + c0 + PF - 2 * RHO;
            float2* out = Hx + (fr / TH * HR + PH + fr % TH) * HS + c0;
            float2 v[RO + 2 * RHO];
#pragma unroll
            for (int t = 0; t < RO + 2 * RHO; ++t) {
                const int x = c0 - 2 * RHO + t;
                v[t] = PF || (x >= 0 && x < SW) ? in[t] : dup2(0.f);
            }
#pragma unroll
            for (int c = 0; c < RO; ++c) {
                float2 s = v[c];
#pragma unroll
                for (int t = 1; t <= 2 * RHO; ++t) s = add2(s, v[c + t]);
                if (c0 + c < HWC) out[c] = s;
            }
        }
        __syncthreads();
        // 3b, 4. vertical box sums at this thread's halo positions, dL/dw and the chain.
        // The pose accumulators take the first plane's samples of every position,
        // then the second's: the order of one plane at a time
        auto column = [&](int f, int p) {  // sum of field f over rows y - 2 RHO .. y at halo position p
            const int y = p / HWC - 2 * RHO;
            const float2* in = Hx + f * (HR * HS) + (PH - 2 * RHO) * HS + p;
            float2 s = dup2(0.f);
#pragma unroll
            for (int t = 0; t <= 2 * RHO; ++t) {
                const float2 v = PH || (y + t >= 0 && y + t < TH) ? in[t * HS] : dup2(0.f);
                s = t == 0 ? v : add2(s, v);
            }
            return s;
        };
        float2 g[RPT];  // dL/dref of this pair
#pragma unroll
        for (int i = 0; i < RPT; ++i) {
            const int p = tid + i * ST;
            g[i] = dup2(0.f);
            if (p < NPOS) {
                const float a = R[p / HWC * G::RS + p % HWC] - ca;
                g[i] = add2(fma2(dup2(-a), column(4 * nc + 1, p), neg2(column(4 * nc, p))), column(4 * nc + 2, p));
            }
        }
#pragma unroll
        for (int j = 0; j < MC; ++j) {
            if (j >= nc) break;
            const float2 cb = centre(j);
            float2 gw[RPT], m[RPT][6];
#pragma unroll
            for (int i = 0; i < RPT; ++i) {
                const int p = tid + i * ST;
                gw[i] = dup2(0.f);
#pragma unroll
                for (int t = 0; t < 6; ++t) m[i][t] = dup2(0.f);
                if (p < NPOS) {
                    const float a = R[p / HWC * G::RS + p % HWC] - ca;
                    const float2 w = W2[j * NPOS + p], b = add2(w, neg2(cb)), a1 = column(4 * j, p);
                    float2 v = fma2(dup2(a), a1, neg2(column(4 * j + 1, p)));
                    v = add2(fma2(neg2(b), column(4 * j + 2, p), v), column(4 * j + 3, p));
                    const float2 gb = fma2(b, a1, g[i]);
                    // an invalid sample is in no used window: all its sums are zero
                    if (!isnan(w.x)) {
                        gw[i].x = v.x;
                        g[i].x = gb.x;
                    }
                    if (!isnan(w.y)) {
                        gw[i].y = v.y;
                        g[i].y = gb.y;
                    }
                    if (gw[i].x != 0.f || gw[i].y != 0.f)
                        chain_pair<WIDE>(P.cams[j], pl0, pl1, ray_at(P, x0 + p % HWC, y0 + p / HWC), gw[i], GO.cam[j], m[i]);
                }
            }
            // (a plane with gw = 0 may hold a sample that does not project)
#pragma unroll
            for (int i = 0; i < RPT; ++i)
                if (gw[i].x != 0.f)
#pragma unroll
                    for (int t = 0; t < 6; ++t) pose_acc[j][t] = fmaf(gw[i].x, m[i][t].x, pose_acc[j][t]);
#pragma unroll
            for (int i = 0; i < RPT; ++i)
                if (gw[i].y != 0.f)
#pragma unroll
                    for (int t = 0; t < 6; ++t) pose_acc[j][t] = fmaf(gw[i].y, m[i][t].y, pose_acc[j][t]);
        }
#pragma unroll
        for (int i = 0; i < RPT; ++i) gR[i] = (gR[i] + g[i].x) + g[i].y;
    }
    if (g_ref) {
#pragma unroll
        for (int i = 0; i < RPT; ++i) {
            const int p = tid + i * ST, x = x0 + p % HWC, y = y0 + p / HWC;
            // (outside the image gR is zero, or no number where an intensity is infinite)
            if (p < NPOS && gR[i] != 0.f && x >= 0 && y >= 0 && x < P.W && y < P.H)
                atomicAdd(&g_ref[(size_t)y * P.W + x], gR[i]);
        }
    }
    if (g_pose) {
        const int lane = tid & 31, wid = tid >> 5;
#pragma unroll
        for (int j = 0; j < MC; ++j)
#pragma unroll
            for (int i = 0; i < 6; ++i) {
                float v = pose_acc[j][i];
                for (int off = 16; off > 0; off >>= 1) v += __shfl_down_sync(0xffffffffu, v, off);
                if (lane == 0) red[wid][6 * j + i] = v;
            }
        __syncthreads();
        if (tid < 6 * nc) {
            double s = 0.0;
            for (int w = 0; w < ST / 32; ++w) s += (double)red[w][tid];
            atomicAdd(&g_pose[tid], s);
        }
    }
}

}  // namespace
}  // namespace ps

using namespace ps;

struct psdiff_s {
    ps_camera ref;
    int n_cams = 0;
    ps_camera cams[PS_MAX_CAMS];
    int rho = 0, K = 0;
    double T = 0.05;
    float4* rays = nullptr;
    PlaneD* planes = nullptr;
    int sms = 0;
};

namespace {

void free_diff(psdiff_t* h) {
    if (!h) return;
    cudaFree(h->rays);
    cudaFree(h->planes);
    delete h;
}

// Largest float not above n - 1.
float last_coordinate(int n) {
    const float x = (float)(n - 1);
    return (double)x > (double)(n - 1) ? std::nextafter(x, 0.0f) : x;
}

// A matching image whose offsets do not fit 32 bits, or whose coordinates are not all floats.
bool wide(const psdiff_t* h) {
    for (int j = 0; j < h->n_cams; ++j) {
        const ps_camera& c = h->cams[j];
        if ((long long)c.width * c.height > INT32_MAX || c.width > 1 << 24 || c.height > 1 << 24) return true;
    }
    return false;
}

int fill_params(const psdiff_t* h, const float* const* images, const ps_pose* ref_to_cam, DiffP& P) {
    std::memset(&P, 0, sizeof(P));
    P.W = h->ref.width;
    P.H = h->ref.height;
    P.rho = h->rho;
    P.K = h->K;
    P.n_cams = h->n_cams;
    P.T = std::max((float)h->T, FLT_MIN);  // (1 / T of a subnormal one overflows; both leave one plane's weight alone)
    P.rays = h->rays;
    P.planes = h->planes;
    PS_ARG(images != nullptr && images[0] != nullptr, "psdiff: images[0] is NULL");
    PS_ARG(ref_to_cam != nullptr, "psdiff: ref_to_cam is NULL");
    P.ref = images[0];
    for (int j = 0; j < h->n_cams; ++j) {
        PS_ARG(images[1 + j] != nullptr, "psdiff: images[%d] is NULL", 1 + j);
        for (int i = 0; i < 12; ++i)
            PS_ARG(std::isfinite(i < 9 ? ref_to_cam[j].R[i] : ref_to_cam[j].t[i - 9]), "psdiff: pose %d not finite", j);
        DiffCam& D = P.cams[j];
        const CamF c = to_camf(h->cams[j]);
        auto two = [](float v) { return make_float2(v, v); };
        for (int i = 0; i < 9; ++i) D.R2[i] = two((float)ref_to_cam[j].R[i]);
        for (int i = 0; i < 3; ++i) D.t2[i] = two((float)ref_to_cam[j].t[i]);
        D.xi = two(c.xi); D.fx = two(c.fx); D.fy = two(c.fy); D.cx = two(c.cx); D.cy = two(c.cy);
        D.k1 = two(c.k1); D.k2 = two(c.k2); D.k2x2 = two(2.0f * c.k2);
        D.p1 = two(c.p1); D.p1x2 = two(2.0f * c.p1); D.p1x6 = two(6.0f * c.p1);
        D.p2 = two(c.p2); D.p2x2 = two(2.0f * c.p2); D.p2x6 = two(6.0f * c.p2);
        D.lim = two(c.lim);
        D.r2_max = c.r2_max;
        D.width = c.width;
        D.height = c.height;
        D.u_max = last_coordinate(c.width);
        D.v_max = last_coordinate(c.height);
        D.img = images[1 + j];
    }
    return PS_OK;
}

}  // namespace

namespace {

// A kernel's shared-memory limit belongs to the process: every call sets the
// same one, that of the most cameras, so that calls of several threads never
// lower each other's between the attribute and the launch.
template <class G, bool WIDE>
int launch_fwd(const DiffP& P, float* range, float* cost, float* aux, cudaStream_t s) {
    auto smem = [](int nc) { return sizeof(float) * (ROUND * ST * G::PX + 2 * FG * nc * G::NPOS + G::HH * G::RS); };
    auto* kernel = soft_fwd_kernel<G, WIDE>;
    PS_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem(PS_MAX_CAMS)));
    kernel<<<dim3((P.W + G::SW - 1) / G::SW, (P.H + G::TH - 1) / G::TH), FG * ST, smem(P.n_cams), s>>>(P, range, cost, aux);
    PS_CUDA(cudaGetLastError());
    return PS_OK;
}

// Tiles of 32 x 16 pixels, two under each other per thread; images of too few
// of them for the SMs take twice as many of 16 x 16.  (Wide images, whose
// time is their own size, have the small tiles and the four-camera layout.)
template <int RHO>
int forward(const psdiff_t* h, const DiffP& P, float* range, float* cost, float* aux, cudaStream_t s) {
    using Wide = Tile<RHO, 32, 2>;
    const long long tiles = (long long)((P.W + Wide::SW - 1) / Wide::SW) * ((P.H + Wide::TH - 1) / Wide::TH);
    if (wide(h)) return launch_fwd<Tile<RHO, 16, 1>, true>(P, range, cost, aux, s);
    return tiles >= h->sms ? launch_fwd<Wide, false>(P, range, cost, aux, s)
                           : launch_fwd<Tile<RHO, 16, 1>, false>(P, range, cost, aux, s);
}

template <int RHO, int MC, bool WIDE>
int launch_bwd(const psdiff_t* h, const DiffP& P, const float* aux, const float* g_range, const float* g_cost, float* g_ref,
               const GradOut& G, double* g_pose, cudaStream_t s) {
    using T = typename BwdLayout<RHO, MC>::G;
    // at most 122 KB (window 9, 4 cameras); the limit as in launch_fwd
    auto smem = [](int nc) { return sizeof(float) * BwdLayout<RHO, MC>::floats(nc); };
    auto* kernel = soft_bwd_kernel<RHO, MC, WIDE>;
    PS_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem(MC)));
    kernel<<<dim3((P.W + T::SW - 1) / T::SW, (P.H + T::TH - 1) / T::TH), ST, smem(P.n_cams), s>>>(P, aux, g_range, g_cost,
                                                                                                 g_ref, G, g_pose);
    PS_CUDA(cudaGetLastError());
    return PS_OK;
}

}  // namespace

extern "C" int psdiff_create(const ps_diff_desc* d, psdiff_t** out) {
    clear_error();
    PS_ARG(out != nullptr, "psdiff_create: out is NULL");
    *out = nullptr;
    PS_ARG(d != nullptr && d->cams != nullptr, "psdiff_create: desc or cams is NULL");
    PS_ARG(d->n_cams >= 1 && d->n_cams <= PS_MAX_CAMS, "psdiff_create: n_cams must be in 1..%d", PS_MAX_CAMS);
    PS_ARG(d->ref.width > 0 && d->ref.height > 0 && d->ref.width <= 16384 && d->ref.height <= 16384 &&
               d->ref.fx > 0 && d->ref.fy > 0 && d->ref.xi >= 0,
           "psdiff_create: bad reference camera");
    for (int j = 0; j < d->n_cams; ++j)
        PS_ARG(d->cams[j].width > 1 && d->cams[j].height > 1 && d->cams[j].fx > 0 && d->cams[j].fy > 0 &&
                   d->cams[j].xi >= 0,
               "psdiff_create: bad matching camera %d", j);
    const ps_level& L = d->level;
    PS_ARG(L.kind == PS_LEVEL_DOWNSAMPLE && L.factor == 1, "psdiff_create: one full-resolution level (factor 1)");
    PS_ARG(L.window == 5 || L.window == 7 || L.window == 9, "psdiff_create: window must be 5, 7 or 9");
    PS_ARG(L.n_sets >= 1 && L.n_sets <= PS_MAX_SETS, "psdiff_create: n_sets must be in 1..%d", PS_MAX_SETS);
    PS_ARG(d->temperature > 0 && std::isfinite(d->temperature), "psdiff_create: temperature must be > 0");
    std::vector<PlaneD> planes;
    for (int s = 0; s < L.n_sets; ++s) {
        const ps_plane_set& S = L.sets[s];
        PS_ARG(S.count >= 1 && S.count <= 4096 && S.a > 0 && S.b >= S.a, "psdiff_create: bad plane set %d", s);
        PS_ARG(S.family == PS_PLANES_FRONTO || S.family == PS_PLANES_GROUND, "psdiff_create: bad family");
        double n[3] = {0, 0, 1};
        if (S.family == PS_PLANES_GROUND) {
            double nn = std::sqrt(S.n[0] * S.n[0] + S.n[1] * S.n[1] + S.n[2] * S.n[2]);
            PS_ARG(nn > 0, "psdiff_create: ground normal is zero");
            for (int i = 0; i < 3; ++i) n[i] = S.n[i] / nn;
        }
        for (int i = 0; i < S.count; ++i) {
            double t = S.count > 1 ? (double)i / (S.count - 1) : 0.0;
            double dd = S.family == PS_PLANES_FRONTO ? 1.0 / (1.0 / S.b + t * (1.0 / S.a - 1.0 / S.b))
                                                     : S.a + t * (S.b - S.a);
            planes.push_back({(float)n[0], (float)n[1], (float)n[2], (float)dd});
        }
    }
    psdiff_t* h = new psdiff_t();
    h->ref = d->ref;
    h->n_cams = d->n_cams;
    for (int j = 0; j < d->n_cams; ++j) h->cams[j] = d->cams[j];
    h->rho = L.window / 2;
    h->K = (int)planes.size();
    h->T = d->temperature;
    const size_t npx = (size_t)d->ref.width * d->ref.height;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&h->sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaMalloc(&h->rays, sizeof(float4) * npx);
    if (e == cudaSuccess) e = cudaMalloc(&h->planes, sizeof(PlaneD) * planes.size());
    if (e == cudaSuccess)
        e = cudaMemcpy(h->planes, planes.data(), sizeof(PlaneD) * planes.size(), cudaMemcpyHostToDevice);
    if (e != cudaSuccess) {
        free_diff(h);
        set_error("psdiff_create: %s", cudaGetErrorString(e));
        return e == cudaErrorMemoryAllocation ? PS_ERR_OOM : PS_ERR_CUDA;
    }
    if (build_rays(d->ref, h->rays, nullptr) != PS_OK || cudaDeviceSynchronize() != cudaSuccess) {
        free_diff(h);
        return PS_ERR_CUDA;
    }
    *out = h;
    return PS_OK;
}

extern "C" void psdiff_destroy(psdiff_t* h) { free_diff(h); }

extern "C" int psdiff_forward(psdiff_t* h, const float* const* images, const ps_pose* ref_to_cam, float* range,
                              float* cost, float* aux, void* stream) {
    clear_error();
    PS_ARG(h != nullptr && range != nullptr, "psdiff_forward: handle or range is NULL");
    DiffP P;
    int st = fill_params(h, images, ref_to_cam, P);
    if (st) return st;
    cudaStream_t s = (cudaStream_t)stream;
    if (P.rho == 2) return forward<2>(h, P, range, cost, aux, s);
    if (P.rho == 3) return forward<3>(h, P, range, cost, aux, s);
    return forward<4>(h, P, range, cost, aux, s);
}

extern "C" int psdiff_backward(psdiff_t* h, const float* const* images, const ps_pose* ref_to_cam, const float* aux,
                               const float* g_range, const float* g_cost, float* const* g_images, double* g_pose,
                               void* stream) {
    clear_error();
    PS_ARG(h != nullptr && aux != nullptr, "psdiff_backward: handle or aux is NULL");
    DiffP P;
    int st = fill_params(h, images, ref_to_cam, P);
    if (st) return st;
    float* g_ref = g_images ? g_images[0] : nullptr;
    GradOut G;
    for (int j = 0; j < PS_MAX_CAMS; ++j) G.cam[j] = (g_images && j < h->n_cams) ? g_images[1 + j] : nullptr;
    cudaStream_t s = (cudaStream_t)stream;
    if (wide(h)) {
        auto go = P.rho == 2 ? launch_bwd<2, 4, true> : P.rho == 3 ? launch_bwd<3, 4, true> : launch_bwd<4, 4, true>;
        return go(h, P, aux, g_range, g_cost, g_ref, G, g_pose, s);
    }
    auto go = h->n_cams <= 2 ? (P.rho == 2   ? launch_bwd<2, 2, false>
                                : P.rho == 3 ? launch_bwd<3, 2, false>
                                             : launch_bwd<4, 2, false>)
                             : (P.rho == 2   ? launch_bwd<2, 4, false>
                                : P.rho == 3 ? launch_bwd<3, 4, false>
                                             : launch_bwd<4, 4, false>);
    return go(h, P, aux, g_range, g_cost, g_ref, G, g_pose, s);
}

namespace ps {
PS_DEFINE_CHECK_READER(check_bits_diff)
}  // namespace ps
