// The scatter sum of the model rows on a grid of detector positions and
// energies (large event lists).
//
// For one detector angle and one support pixel n, the scatter part of p_jn
// (paper Eq. 2 with Eq. 4),
//     S_n(u, E) = sum_m U(u; m) W_a(n, m) phi(E; E'_a(n, m), sigma_E(E')),
// is a function of the event's position and energy alone, and a sum of
// Gaussians whose widths are known: sigma_u of the collimator and sigma_E of
// the energy response.  Once an angle holds more events than S_n has degrees
// of freedom, it is cheaper to evaluate S_n on a grid that resolves those
// Gaussians and to interpolate it at every event than to form the sum per
// event.  The grid is uniform in u (step at most 0.415 of the narrowest sigma_u)
// and in x = 2 sqrt(E / kappa) (sigma_E^2 = kappa E, so every Gaussian has unit
// width in x; step 0.25), with 12 x 8 point stencils.
//
// On the grid the sum is a matrix product per angle and energy node,
//     T[k][i][n] = sum_m U[i][m] G_k[n][m],  G_k = W phi(E_k; E', sigma_E),
// done on the tensor cores (k_grid_sum) with both factors split into two FP16
// parts (22 bits; three products), U tabulated per angle and G formed on the
// fly from two tabulated values per (n, m).
#include <cuda_fp16.h>
#include <math.h>

#include <algorithm>

#include "lmosem_internal.cuh"

namespace lmosem {

namespace {

constexpr int kPU = 12, kPE = 8;            // stencil points in u and in x
constexpr double kRhoX = 0.25;              // x step in units of sigma
constexpr double kRhoUMin = 0.30, kRhoUMax = 0.415;  // u step in units of the narrowest sigma_u
constexpr double kWideX = 1.3, kWideU = 2.0;  // width of the interpolation kernel / that sigma
constexpr double kFarSigma = 5.5;           // reach of the widest responses (see grid_plan)
constexpr double kEdgeSigma = 3.0;          // events farther outside the object or E0 are summed directly
constexpr int kWin = 96;                    // nodes one subgroup of scatter pixels reaches (product N)
constexpr int kSub = 64, kChunk = 16, kChunks = kSub / kChunk;  // scatter pixels per subgroup, per product
constexpr uint32_t kUHalf = kWin * kChunk * 2;      // bytes of one FP16 part of U of one chunk
constexpr uint32_t kUStage = kChunks * 2 * kUHalf;  // bytes of one subgroup
constexpr int kStages = 4;
constexpr int kASlots = 8;                  // one per chunk and energy node
// TMEM columns: main[2] (kWin each), partial[2] (kWin each), A slots of 16
constexpr uint32_t kColMain = 0, kColPart = 2 * kWin, kColA = 4 * kWin;
static_assert(kColA + kASlots * 16 == 512, "tensor memory columns");
constexpr int kGenWarps = 16, kEpiWarps = 8, kMmaWarp = 24, kLoadWarp = 25, kGridThreads = 26 * 32;
constexpr int kEpi = 16;                     // columns per step of the epilogue
static_assert(kSub == 64, "two ballots");
static_assert(kEpi == 16 && kWin % kEpi == 0 && kWin % 16 == 0, "whole steps");
constexpr int kEGroup = 8;                  // energy nodes per CTA: 4 lane groups x 2
constexpr int kNTile = 32;                  // support pixels per CTA

// ---------------------------------------------------------------- plan

// rank of every scatter pixel by its projected position (ties by index)
__global__ void __launch_bounds__(256) k_grid_rank(const float4* __restrict__ mpar, int n_scat, int32_t* __restrict__ order) {
    __shared__ float su[1024];
    const int a = blockIdx.y, m = blockIdx.x * blockDim.x + threadIdx.x;
    const float4* mp = mpar + (size_t)a * n_scat;
    const float um = m < n_scat ? mp[m].x : 0.0f;
    int rank = 0;
    for (int b = 0; b < n_scat; b += 1024) {
        __syncthreads();
        for (int k = threadIdx.x; k < 1024; k += blockDim.x) su[k] = b + k < n_scat ? mp[b + k].x : INFINITY;
        __syncthreads();
        const int ne = min(1024, n_scat - b);
        for (int k = 0; k < ne; ++k) rank += su[k] < um || (su[k] == um && b + k < m);
    }
    if (m < n_scat) order[(size_t)a * n_scat + rank] = m;
}

// Subgroups of at most kSub scatter pixels, consecutive in position and within
// `span` of each other; slot_m lists a subgroup's pixels (-1: unused), i0 the
// first node (a multiple of 8) its pixels reach.  One block per angle.
__global__ void k_grid_groups(const float4* __restrict__ mpar, const int32_t* __restrict__ order, int n_scat,
                              int max_sub, float span, float cut_max, float u_node0, float inv_hu,
                              int32_t* __restrict__ slot_m, int32_t* __restrict__ i0, int32_t* __restrict__ n_sub,
                              float2* __restrict__ urange) {
    extern __shared__ float su[];  // positions in order, then the subgroup starts
    int* start = reinterpret_cast<int*>(su + n_scat);
    __shared__ int ns;
    const int a = blockIdx.x;
    const int32_t* o = order + (size_t)a * n_scat;
    for (int r = threadIdx.x; r < n_scat; r += blockDim.x) su[r] = mpar[(size_t)a * n_scat + o[r]].x;
    for (int r = threadIdx.x; r < max_sub * kSub; r += blockDim.x) slot_m[(size_t)a * max_sub * kSub + r] = -1;
    __syncthreads();
    if (threadIdx.x < 32) {  // one warp walks the starts, testing kSub = 64 pixels at a time
        const int lane = threadIdx.x;
        int g = 0;
        for (int r = 0; r < n_scat && g < max_sub; ++g) {
            if (lane == 0) start[g] = r;
            const float lim = su[r] + span;
            const unsigned b0 = __ballot_sync(0xffffffffu, r + lane < n_scat && su[min(r + lane, n_scat - 1)] <= lim);
            const unsigned b1 =
                __ballot_sync(0xffffffffu, r + 32 + lane < n_scat && su[min(r + 32 + lane, n_scat - 1)] <= lim);
            r += __popc(b0) + __popc(b1);  // sorted: the positions within the span are the first ones
        }
        if (lane == 0) {
            start[g] = n_scat;
            ns = g;
            n_sub[a] = g;
            urange[a] = make_float2(su[0], su[n_scat - 1]);
        }
    }
    __syncthreads();
    for (int g = threadIdx.x; g < ns; g += blockDim.x) {
        const int k = max(0, (int)floorf((su[start[g]] - cut_max - u_node0) * inv_hu));
        i0[(size_t)a * max_sub + g] = k / 8 * 8;
    }
    for (int g = threadIdx.x >> 5; g < ns; g += blockDim.x >> 5)
        for (int k = threadIdx.x & 31; k < start[g + 1] - start[g]; k += 32)
            slot_m[((size_t)a * max_sub + g) * kSub + k] = o[start[g] + k];
}

// ---------------------------------------------------------------- tables

__device__ __forceinline__ uint32_t pack_half2(float lo, float hi) {
    __half2 h = __floats2half2_rn(lo, hi);
    return *reinterpret_cast<uint32_t*>(&h);
}

// U of one angle's chunks as the product's B operand: node rows of 16 scatter
// pixels (K-major core matrices of 8 rows x 16 B), high then low FP16 parts.
// The position of the scatter pixel is formed in FP64.
struct UArgs {
    const float4* mpar;
    const float4* scat_geo;
    const float2* trig;
    const int32_t* slot_m;
    const int32_t* i0;
    const int32_t* n_sub;
    const int32_t* slot_angle;
    int s0, n_scat, max_sub;
    double angle0, dtheta, u_node0, hu;
    float cut;
    float scale;  // log2 of the scale of U
    unsigned char* out;  // [angle of the group][chunk][2][kUHalf]
};

__global__ void __launch_bounds__(2 * kWin) k_grid_u(UArgs A) {
    const int a = A.slot_angle[A.s0 + blockIdx.y];
    const int chunk = blockIdx.x, g = chunk / kChunks;
    if (g >= A.n_sub[a]) return;
    __shared__ float4 smp[kChunk];
    __shared__ double sum_[kChunk];
    const int32_t* sm = A.slot_m + (size_t)a * A.max_sub * kSub + chunk * kChunk;
    if (threadIdx.x < kChunk) {
        const int m = sm[threadIdx.x];
        smp[threadIdx.x] = m >= 0 ? A.mpar[(size_t)a * A.n_scat + m] : make_float4(0.0f, 0.0f, 0.0f, -1.0f);
        double u = 0.0;
        if (m >= 0) {
            const float4 gm = A.scat_geo[m];
            double sn, cs;
            sincos(A.angle0 + A.dtheta * a, &sn, &cs);
            u = -(double)gm.x * sn + (double)gm.y * cs;
        }
        sum_[threadIdx.x] = u;
    }
    __syncthreads();
    const int r = threadIdx.x >> 1, kg = threadIdx.x & 1;  // node of the window, 8-pixel group
    const double un = A.u_node0 + (A.i0[(size_t)a * A.max_sub + g] + r) * A.hu;
    uint32_t hi[4], lo[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        float v[2];
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const float4 q = smp[kg * 8 + 2 * k + j];
            const float d = (float)(un - sum_[kg * 8 + 2 * k + j]);
            const float z = d * q.y;
            v[j] = fabsf(d) <= fminf(q.w, A.cut) ? ex2_approx(fmaf(-z, z, q.z + A.scale)) : 0.0f;
        }
        hi[k] = pack_half2(v[0], v[1]);
        const __half2 h = *reinterpret_cast<__half2*>(&hi[k]);
        lo[k] = pack_half2(v[0] - __low2float(h), v[1] - __high2float(h));
    }
    unsigned char* dst = A.out + ((size_t)blockIdx.y * A.max_sub * kChunks + chunk) * 2 * kUHalf +
                         (r >> 3) * 256 + kg * 128 + (r & 7) * 16;
    *reinterpret_cast<uint4*>(dst) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
    *reinterpret_cast<uint4*>(dst + kUHalf) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
}

// (cE^2 E', -log2 of the scaled path weight over sigma_E) of every (n, slot):
// [angle of the group][32-pixel tile][slot pair][32] as (E'_0, E'_1, w_0, w_1)
struct PlaneArgs {
    int nx, ny, npix, n_sup, ld, n_scat, max_sub;
    float dpx, eps0, inv_kbar, e0, w_const, cE2, scale;
    const int32_t* sup;
    const float4* scat_geo;
    const float2* trig;
    const float* l_edge;
    const float* l_pair;
    const float2* compton;
    const int32_t* slot_m;
    const int32_t* n_sub;
    const int32_t* slot_angle;
    int s0;
    float4* out;
};
constexpr int kPlanePairs = 8;

__global__ void __launch_bounds__(128) k_grid_planes(PlaneArgs A) {
    const int n = blockIdx.x * blockDim.x + threadIdx.x;
    const int a = A.slot_angle[A.s0 + blockIdx.z];
    const int p0 = blockIdx.y * kPlanePairs;
    if (n >= A.ld || 2 * p0 >= A.n_sub[a] * kSub) return;
    const bool real = n < A.n_sup;
    const int pn = real ? A.sup[n] : 0;
    const float xn = pixel_x(pn, A.nx, A.dpx), yn = pixel_y(pn, A.nx, A.ny, A.dpx);
    const float2 trig = A.trig[a];
    const int32_t* sm = A.slot_m + (size_t)a * A.max_sub * kSub;
    float4* out = A.out + (((size_t)blockIdx.z * (A.ld / kNTile) + n / kNTile) * (A.max_sub * kSub / 2) + p0) * kNTile +
                  n % kNTile;
#pragma unroll 2
    for (int p = 0; p < kPlanePairs; ++p) {
        float e[2], w[2];
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const int m = sm[2 * (p0 + p) + j];
            e[j] = A.e0 * A.cE2;
            w[j] = INFINITY;
            if (m >= 0 && real) {
                const float4 gm = __ldg(A.scat_geo + m);
                const int pm = __float_as_int(gm.w);
                float cpsi, rinv;
                if (path_geometry_xy(xn, yn, gm.x, gm.y, pn == pm, trig, &cpsi, &rinv)) {
                    float P, kt;
                    compton(cpsi, A.eps0, A.inv_kbar, &P, &kt);
                    const float e1 = A.e0 * P;
                    const float ratio = compton_lookup(A.compton, cpsi).x;
                    const float att = fmaf(ratio, __ldg(A.l_edge + (size_t)a * A.npix + pm),
                                           A.l_pair[(size_t)m * A.n_sup + n]);
                    w[j] = fmaf(att, kLog2e, -__log2f(A.w_const * gm.z * kt * rinv * rsqrtf(e1))) - A.scale;
                    e[j] = e1 * A.cE2;
                }
            }
        }
        out[p * kNTile] = make_float4(e[0], e[1], w[0], w[1]);
    }
}

// ---------------------------------------------------------------- the sum on the grid

__device__ __forceinline__ uint32_t su32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ uint64_t smem_desc(uint32_t saddr) {  // LBO 128, SBO 256, no swizzle
    return (uint64_t)((saddr & 0x3FFFFu) >> 4) | (uint64_t)(128 >> 4) << 16 | (uint64_t)(256 >> 4) << 32 |
           (uint64_t)1 << 46;
}
// D (TMEM) (+)= A (TMEM, FP16) B (shared memory, FP16), M = 128, N = kWin, K = 16
__device__ __forceinline__ void mma_ts(uint32_t d, uint32_t a, uint64_t b, uint32_t accumulate) {
    constexpr uint32_t idesc = (1u << 4) | ((uint32_t)(kWin >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}" ::"r"(d),
        "r"(a), "l"(b), "r"(idesc), "r"(accumulate)
        : "memory");
}
__device__ __forceinline__ void mma_commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(bar)
                 : "memory");
}
__device__ __forceinline__ void bar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void bar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool bar_try(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}
__device__ __noinline__ bool bar_wait_slow(uint32_t bar, uint32_t parity, long long budget,
                                           const volatile int* abort_flag) {
    const long long t0 = clock64();
    while (true) {
        if (bar_try(bar, parity)) return true;  // suspends the thread for a while: no issue slots lost to spinning
        if ((abort_flag && *abort_flag) || clock64() - t0 > budget) return false;
    }
}
// bounded wait for the phase of the given parity; false when the budget ran
// out or another warp has given up
__device__ __forceinline__ bool bar_wait(uint32_t bar, uint32_t parity, long long budget,
                                         const volatile int* abort_flag) {
    if (bar_try(bar, parity)) return true;
    return bar_wait_slow(bar, parity, budget, abort_flag);
}
__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(bar), "r"(bytes)
                 : "memory");
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(dst),
        "l"(src), "r"(bytes), "r"(bar)
        : "memory");
}
__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory"); }
__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory"); }

__device__ __forceinline__ void tmem_st16(uint32_t a, const uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};\n" ::"r"(a),
        "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]),
        "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
        : "memory");
}
__device__ __forceinline__ void tmem_st8(uint32_t a, const uint32_t* r) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};\n" ::"r"(a), "r"(r[0]),
                 "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7])
                 : "memory");
}
__device__ __forceinline__ void tmem_ld8(uint32_t a, uint32_t* r) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(a));
}
// waits for this thread's tensor-memory loads; r (what they wrote) passes
// through, so that no use is scheduled before it
__device__ __forceinline__ void tmem_wait_ld8(uint32_t* r) {
    asm volatile("tcgen05.wait::ld.sync.aligned;\n"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7])
                 :
                 : "memory");
}
__device__ __forceinline__ void tmem_ld16(uint32_t a, uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(a));
}
__device__ __forceinline__ void tmem_wait_ld(uint32_t (&x)[16], uint32_t (&y)[16]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;\n"
                 : "+r"(x[0]), "+r"(x[1]), "+r"(x[2]), "+r"(x[3]), "+r"(x[4]), "+r"(x[5]), "+r"(x[6]), "+r"(x[7]),
                   "+r"(x[8]), "+r"(x[9]), "+r"(x[10]), "+r"(x[11]), "+r"(x[12]), "+r"(x[13]), "+r"(x[14]),
                   "+r"(x[15]), "+r"(y[0]), "+r"(y[1]), "+r"(y[2]), "+r"(y[3]), "+r"(y[4]), "+r"(y[5]), "+r"(y[6]),
                   "+r"(y[7]), "+r"(y[8]), "+r"(y[9])
                 :
                 : "memory");
    asm volatile("" : "+r"(y[10]), "+r"(y[11]), "+r"(y[12]), "+r"(y[13]), "+r"(y[14]), "+r"(y[15]) : : "memory");
}
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;\n" ::: "memory"); }

__device__ __forceinline__ float2 mul2(float2 a, float2 b) {
    float2 d;
    asm("{\n\t.reg .b64 ra, rb, rd;\n\tmov.b64 ra, {%2, %3};\n\tmov.b64 rb, {%4, %5};\n\t"
        "mul.rn.f32x2 rd, ra, rb;\n\tmov.b64 {%0, %1}, rd;\n\t}"
        : "=f"(d.x), "=f"(d.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return d;
}
__device__ __forceinline__ float2 add2(float2 a, float2 b) {
    float2 d;
    asm("{\n\t.reg .b64 ra, rb, rd;\n\tmov.b64 ra, {%2, %3};\n\tmov.b64 rb, {%4, %5};\n\t"
        "add.rn.f32x2 rd, ra, rb;\n\tmov.b64 {%0, %1}, rd;\n\t}"
        : "=f"(d.x), "=f"(d.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return d;
}
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
    float2 d;
    asm("{\n\t.reg .b64 ra, rb, rc, rd;\n\tmov.b64 ra, {%2, %3};\n\tmov.b64 rb, {%4, %5};\n\tmov.b64 rc, {%6, %7};\n\t"
        "fma.rn.f32x2 rd, ra, rb, rc;\n\tmov.b64 {%0, %1}, rd;\n\t}"
        : "=f"(d.x), "=f"(d.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
    return d;
}
__device__ __forceinline__ float rsqrt_approx(float x) {
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
// the FP16 parts of two values: columns of the high and of the low operand
__device__ __forceinline__ void split2(float2 v, uint32_t* hi, uint32_t* lo) {
    const __half2 h = __floats2half2_rn(v.x, v.y);
    const float2 f = __half22float2(h);
    const float2 r = fma2(f, make_float2(-1.0f, -1.0f), v);
    const __half2 l = __floats2half2_rn(r.x, r.y);
    *hi = *reinterpret_cast<const uint32_t*>(&h);
    *lo = *reinterpret_cast<const uint32_t*>(&l);
}

struct SumArgs {
    const float4* planes;        // [angle of the group][32-pixel tile][slot pair][32]
    const unsigned char* ublob;  // [angle of the group][chunk][2][kUHalf]
    const int32_t* i0;           // [angle][max_sub]
    const int32_t* n_sub;        // [angle]
    const int32_t* slot_angle;
    int s0, ld, max_sub, ne, nu, n_nt;
    const float4* enode;         // node pairs: cE^2 E_2k (high, low part), cE^2 (E_2k+1 - E_2k)
    float out_scale;
    float* T;                    // [angle of the group][column tile][ne][nu][kTCols]
    int* status;
    long long budget;
};

constexpr int kTCols = 128;  // columns per tile of T
// first element of (angle of the group, energy node k, position node 0) of the
// 32-column slice nt
__device__ __forceinline__ size_t t_index(const SumArgs& A, int ai, int k, int nt) {
    const int n_tiles = (A.ld + kTCols - 1) / kTCols;
    return (((size_t)ai * n_tiles + nt / (kTCols / kNTile)) * A.ne + k) * A.nu * kTCols +
           (nt % (kTCols / kNTile)) * kNTile;
}

constexpr int kPlaneStages = 4;
constexpr uint32_t kPlaneStage = kSub / 2 * kNTile * 16;  // tabulated values of a subgroup and 32 pixels
constexpr uint32_t kSmPlane = kStages * kUStage;
constexpr uint32_t kSmBar = kSmPlane + kPlaneStages * kPlaneStage;
constexpr int kBars = 2 * kStages + 2 * kPlaneStages + 2 * kASlots + 4 + 1;
constexpr uint32_t kSmMisc = kSmBar + kBars * 8;
constexpr uint32_t kSmBytes = kSmMisc + 16;

// One CTA: 32 support pixels x 8 energy nodes of one angle, every grid
// position.  Lane quarter q of the tensor memory holds the energy nodes
// 8 eg + 2 q (accumulator 0) and + 1 (accumulator 1) of the 32 pixels.
// The scatter pixels come in order of their projected position, 64 at a time
// (a subgroup), which reach the kWin nodes from i0 on: so the columns of the
// accumulators are a ring of kWin nodes that slides along u, a node's value
// being complete (and stored) once i0 has passed it.
//  * 16 generator warps (4 lane quarters x 4 chunks of 16 scatter pixels) form
//    G of their chunk for both energy nodes of their quarter and write its FP16
//    parts to tensor memory;
//  * the load warp brings U by bulk copies;
//  * the MMA warp sums the 4 chunks of a subgroup into a partial accumulator
//    (3 products per chunk: low x high, high x low, high x high);
//  * 8 epilogue warps add the partial sums to the main accumulators in FP32:
//    the tensor core truncates its running sum (measured: -8e-8 relative per
//    product of a growing sum, -5e-6 after 64), so chains are kept to one
//    subgroup and the long sum is rounded to nearest.
// What bounds it: issue.  A subgroup takes 2,280 cycles per CTA at 128 x 128,
// of which its 24 products need 1,152 on the tensor cores; the generators' and
// the epilogue's 1,590 instructions per scheduler (exponentials, FP16 splits,
// tensor-memory loads, FP32 adds) keep the schedulers 65-70% busy, and the
// hand-over of a chunk between the roles takes the rest.  Measured at 128 x
// 128: three products of N = 112 take 213 cycles when lane 0 issues them, 168
// with elect.sync; plane values by __ldg made a subgroup 3,450 to 5,600 cycles,
// by bulk copies 2,700; a slot of A for every chunk and node and windows of 96
// nodes took an angle from 1.10 to 0.98 ms; two issuing warps 1.00.
__global__ void __launch_bounds__(kGridThreads, 1) k_grid_sum(SumArgs A) {
    extern __shared__ __align__(1024) unsigned char sm[];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    // mbarriers (shared-memory addresses, 8 bytes each)
    const uint32_t base = su32(sm);
    const uint32_t bfull = base + kSmBar, bempty = bfull + 8 * kStages, afull = bempty + 8 * kStages,
                   aempty = afull + 8 * kASlots, pfull = aempty + 8 * kASlots, pempty = pfull + 16,
                   gfull = pempty + 16, gempty = gfull + 8 * kPlaneStages, drain = gempty + 8 * kPlaneStages;
    uint32_t* tslot = reinterpret_cast<uint32_t*>(sm + kSmMisc);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(sm + kSmMisc + 4);
    const int n_eg = A.ne / kEGroup;
    int idx = blockIdx.x;
    const int eg = idx % n_eg;
    idx /= n_eg;
    const int nt = idx % A.n_nt, ai = idx / A.n_nt;
    const int a = A.slot_angle[A.s0 + ai];
    const int ns = A.n_sub[a];
    const int32_t* i0 = A.i0 + (size_t)a * A.max_sub;

    if (warp == kMmaWarp) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;\n" ::"r"(su32(tslot))
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
    }
    if (tid == 0) {
        for (int i = 0; i < kStages; ++i) {
            bar_init(bfull + 8 * i, 1);
            bar_init(bempty + 8 * i, 1);
        }
        for (int i = 0; i < kASlots; ++i) {
            bar_init(afull + 8 * i, 4);
            bar_init(aempty + 8 * i, 1);
        }
        for (int i = 0; i < 2; ++i) {
            bar_init(pfull + 8 * i, 1);
            bar_init(pempty + 8 * i, 4);
        }
        for (int i = 0; i < kPlaneStages; ++i) {
            bar_init(gfull + 8 * i, 1);
            bar_init(gempty + 8 * i, kGenWarps);
        }
        bar_init(drain, 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem = *tslot;
    uint32_t n_loaded = 0;  // subgroups the load warp has issued (for the drain after an abort)

    if (warp < kGenWarps) {
        // ---------------- generators: warp group x takes chunk x of every subgroup
        const int q = warp & 3, x = warp >> 2;
        const uint32_t arow = tmem + kColA + (uint32_t)(x * 16) + ((uint32_t)(32 * q) << 16);
        const float4* pl = reinterpret_cast<const float4*>(sm + kSmPlane) + x * (kChunk / 2) * kNTile + lane;
        const float4 en = A.enode[eg * (kEGroup / 2) + q];
        const float2 E2 = make_float2(en.x, en.x), El2 = make_float2(en.y, en.y), dE2 = make_float2(en.z, en.z);
        const float2 m1 = make_float2(-1.0f, -1.0f);
        float2 Z[8];
        uint32_t stage = 0, sphase = 0;
        bool ok = true;
        for (int g = 0; g < ns && ok; ++g) {
            ok = bar_wait(gfull + 8 * stage, sphase, A.budget, abort_flag);
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                uint32_t r[16];
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    float2 z;  // G = 2^-z
                    if (e == 0) {
                        const float4 p = pl[stage * (kPlaneStage / 16) + k * kNTile];
                        const float2 nlw = make_float2(p.z, p.w);
                        const float2 d = add2(fma2(make_float2(p.x, p.y), m1, E2), El2);
                        const float2 s = make_float2(rsqrt_approx(p.x), rsqrt_approx(p.y));
                        const float2 t = mul2(d, s);
                        z = fma2(t, t, nlw);
                        const float2 t1 = fma2(dE2, s, t);  // the next energy node
                        Z[k] = fma2(t1, t1, nlw);
                    } else {
                        z = Z[k];
                    }
                    split2(make_float2(ex2_approx(-z.x), ex2_approx(-z.y)), &r[k], &r[8 + k]);
                }
                if (e == 0) {  // the stage's values are read
                    __syncwarp();
                    if (lane == 0) bar_arrive(gempty + 8 * stage);
                }
                if (g > 0) {
                    ok = bar_wait(aempty + 8 * (kChunks * e + x), (uint32_t)(g - 1) & 1u, A.budget, abort_flag);
                    ok = __all_sync(0xffffffffu, ok);
                    if (!ok) break;
                    fence_after();
                }
                tmem_st16(arow + 16 * kChunks * e, r);
                tmem_wait_st();
                fence_before();
                __syncwarp();
                if (lane == 0) bar_arrive(afull + 8 * (kChunks * e + x));
            }
            if (++stage == kPlaneStages) {
                stage = 0;
                sphase ^= 1u;
            }
        }
        if (!ok) *abort_flag = 1;
    } else if (warp < kGenWarps + kEpiWarps) {
        // ---------------- epilogue of energy node e: main += partial, finished nodes to T
        const int q = warp & 3, e = (warp - kGenWarps) >> 2;
        const uint32_t row = (uint32_t)(32 * q) << 16;
        const uint32_t tmain = tmem + kColMain + e * kWin + row, tpart = tmem + kColPart + e * kWin + row;
        float* T = A.T + t_index(A, ai, eg * kEGroup + 2 * q + e, nt) + lane;
        uint32_t zero[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) zero[k] = 0u;
        for (int b = 0; b < kWin / 8; ++b) tmem_st8(tmain + b * 8, zero);
        tmem_wait_st();
        int cur = 0;                 // first node of the ring (multiple of 8)
        uint32_t ring = 0;           // its column
        // nodes [cur, to) are complete: store them and clear their columns
        auto retire = [&](int to) {
            while (cur < to) {
                uint32_t v[8];
                tmem_ld8(tmain + ring, v);
                tmem_wait_ld8(v);
                float* t = T + (size_t)cur * kTCols;
#pragma unroll
                for (int k = 0; k < 8; ++k)
                    if (cur + k < A.nu) t[k * kTCols] = __uint_as_float(v[k]) * A.out_scale;
                tmem_st8(tmain + ring, zero);
                cur += 8;
                ring = ring + 8 == kWin ? 0 : ring + 8;
            }
            tmem_wait_st();
        };
        bool ok = true;
        for (int g = 0; g < ns; ++g) {
            const int first = min(__ldg(i0 + g), (A.nu + 7) / 8 * 8);
            if (first > cur) retire(first);
            ok = bar_wait(pfull + 8 * e, (uint32_t)g & 1u, A.budget, abort_flag);
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
            fence_after();
            uint32_t col = ring;
#pragma unroll
            for (int b = 0; b < kWin / kEpi; ++b) {
                uint32_t x[kEpi], y[kEpi];
                uint32_t c1 = col + 8;
                if (c1 == kWin) c1 = 0;
                tmem_ld16(tpart + b * kEpi, x);
                tmem_ld8(tmain + col, y);
                tmem_ld8(tmain + c1, y + 8);
                tmem_wait_ld(x, y);
#pragma unroll
                for (int k = 0; k < kEpi; k += 2) {
                    const float2 v = add2(make_float2(__uint_as_float(x[k]), __uint_as_float(x[k + 1])),
                                          make_float2(__uint_as_float(y[k]), __uint_as_float(y[k + 1])));
                    y[k] = __float_as_uint(v.x);
                    y[k + 1] = __float_as_uint(v.y);
                }
                tmem_st8(tmain + col, y);
                tmem_st8(tmain + c1, y + 8);
                col = c1 + 8;
                if (col == kWin) col = 0;
            }
            fence_before();  // the partial sums are read: the next chain may overwrite them
            __syncwarp();
            if (lane == 0) bar_arrive(pempty + 8 * e);
            tmem_wait_st();
        }
        if (ok) retire((A.nu + 7) / 8 * 8);
        else *abort_flag = 1;
    } else if (warp == kMmaWarp) {
        // ---------------- products: per subgroup, the 4 chunks of energy node 0, then of node 1.
        // (A warp per energy node was slower: 1.00 against 0.98 ms per angle at 128 x 128.)
        if (elect_one()) {
            bool ok = true;
            uint32_t stage = 0, sphase = 0;
            const uint64_t desc0 = smem_desc(base);
            for (int g = 0; g < ns && ok; ++g) {
                ok = bar_wait(bfull + 8 * stage, sphase, A.budget, abort_flag);
                const uint64_t desc = desc0 + (uint64_t)(stage * (kUStage >> 4));
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const uint32_t d = tmem + kColPart + (uint32_t)e * kWin;
                    if (g > 0) ok = ok && bar_wait(pempty + 8 * e, (uint32_t)(g - 1) & 1u, A.budget, abort_flag);
#pragma unroll
                    for (int x = 0; x < kChunks; ++x) {
                        ok = ok && bar_wait(afull + 8 * (kChunks * e + x), (uint32_t)g & 1u, A.budget, abort_flag);
                        if (!ok) break;
                        fence_after();
                        const uint64_t bh = desc + (uint64_t)(x * (2 * kUHalf >> 4));
                        const uint32_t ah = tmem + kColA + (uint32_t)(kChunks * e + x) * 16;
                        mma_ts(d, ah + 8, bh, x > 0);
                        mma_ts(d, ah, bh + (kUHalf >> 4), 1u);
                        mma_ts(d, ah, bh, 1u);
                        mma_commit(aempty + 8 * (kChunks * e + x));
                    }
                    if (ok) mma_commit(pfull + 8 * e);
                }
                if (ok) mma_commit(bempty + 8 * stage);
                if (++stage == kStages) {
                    stage = 0;
                    sphase ^= 1u;
                }
            }
            if (!ok) *abort_flag = 1;
        }
        __syncwarp();
    } else {
        // ---------------- tabulated values and U of the subgroups
        if (elect_one()) {
            const unsigned char* us = A.ublob + (size_t)ai * A.max_sub * kUStage;
            const unsigned char* ps = reinterpret_cast<const unsigned char*>(A.planes) +
                                      ((size_t)ai * (A.ld / kNTile) + nt) * A.max_sub * kPlaneStage;
            bool ok = true;
            for (int g = 0; g < ns; ++g) {
                const uint32_t pst = (uint32_t)g % kPlaneStages, ust = (uint32_t)g % kStages;
                if ((g >= kPlaneStages &&
                     !bar_wait(gempty + 8 * pst, ((uint32_t)g / kPlaneStages - 1) & 1u, A.budget, abort_flag)) ||
                    (g >= kStages && !bar_wait(bempty + 8 * ust, ((uint32_t)g / kStages - 1) & 1u, A.budget, abort_flag))) {
                    ok = false;
                    break;
                }
                bulk_load(base + kSmPlane + pst * kPlaneStage, ps + (size_t)g * kPlaneStage, kPlaneStage, gfull + 8 * pst);
                bulk_load(base + ust * kUStage, us + (size_t)g * kUStage, kUStage, bfull + 8 * ust);
                ++n_loaded;
            }
            if (!ok) *abort_flag = 1;
        }
        __syncwarp();
    }
    __syncthreads();
    if (*abort_flag) {
        constexpr long long kDrainCycles = 1LL << 31;
        // products in flight finish before the tensor memory is freed
        if (warp == kMmaWarp && elect_one()) {
            mma_commit(drain);
            bar_wait(drain, 0u, kDrainCycles, nullptr);
        }
        if (warp == kLoadWarp && n_loaded > 0) {  // (the lane that issued them) and the last copy of every stage lands
            for (uint32_t s = 0; s < (uint32_t)kStages; ++s) {
                const uint32_t n = n_loaded / kStages + (s < n_loaded % kStages ? 1u : 0u);
                if (n > 0) bar_wait(bfull + 8 * s, (n - 1) & 1u, kDrainCycles, nullptr);
            }
            for (uint32_t s = 0; s < (uint32_t)kPlaneStages; ++s) {
                const uint32_t n = n_loaded / kPlaneStages + (s < n_loaded % kPlaneStages ? 1u : 0u);
                if (n > 0) bar_wait(gfull + 8 * s, (n - 1) & 1u, kDrainCycles, nullptr);
            }
        }
        if (tid == 0) atomicExch(A.status, 1);
    }
    fence_before();
    __syncthreads();
    if (warp == kMmaWarp) {
        fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;\n" ::"r"(tmem));
    }
}

// ---------------------------------------------------------------- events

// Interpolation weights of the kernel exp(-(x - y)^2 / (4 s^2)) on equispaced
// nodes h = rho s apart.  On such nodes the interpolant is exp(-x^2 / (4 s^2))
// times a polynomial of degree P - 1 in w = exp(x h / (2 s^2)), so the weights
// are Lagrange's in w with that factor.
template <int P>
struct Stencil {
    double w[P], norm[P], c1, c2;  // w_j; e^{x_j^2/4}/prod (w_j - w_k); rho^2 / 2; rho^2 / 4
};
template <int P>
Stencil<P> make_stencil(double rho) {
    Stencil<P> s;
    const int off = P / 2 - 1;
    s.c1 = 0.5 * rho * rho;
    s.c2 = 0.25 * rho * rho;
    for (int j = 0; j < P; ++j) s.w[j] = exp(s.c1 * (j - off));
    for (int j = 0; j < P; ++j) {
        double d = 1.0;
        for (int k = 0; k < P; ++k)
            if (k != j) d *= s.w[j] - s.w[k];
        s.norm[j] = exp(s.c2 * (j - off) * (j - off)) / d;
    }
    return s;
}
template <int P>
__device__ __forceinline__ void stencil_weights(const Stencil<P>& s, double xi, float* out) {
    const double w = exp(s.c1 * xi), f = exp(-s.c2 * xi * xi);
    double pre[P];
    pre[0] = f;
#pragma unroll
    for (int j = 1; j < P; ++j) pre[j] = pre[j - 1] * (w - s.w[j - 1]);
    double suf = 1.0;
#pragma unroll
    for (int j = P - 1; j >= 0; --j) {
        out[j] = (float)(pre[j] * suf * s.norm[j]);
        suf *= w - s.w[j];
    }
}

struct CellArgs {
    const int32_t* a_s;
    const float* u_s;
    const float* e_s;
    int64_t J;
    const int32_t* angle_slot;
    const float2* urange;  // per angle: positions of the outermost scatter pixels
    float edge;            // events farther outside are summed directly
    float e_min, e_max;
    double u_lo, inv_hu, x_lo, inv_hx, inv_kappa;
    int nce, ncu, n_slots;
    int nbx, nbu;          // blocks of 2 x 2 cells
};
// block of 2 x 2 cells of an event (*sub: its cell, 2 in x + in u); events
// outside the grid's region: n_slots nbx nbu + slot
__device__ __forceinline__ int grid_block(const CellArgs& A, int64_t r, double* fu, double* fx, int* sub) {
    const int a = A.a_s[r], s = A.angle_slot[a];
    const float u = A.u_s[r], e = A.e_s[r];
    const float2 ur = A.urange[a];
    const int out = A.n_slots * A.nbx * A.nbu + s;
    if (!(u >= ur.x - A.edge && u <= ur.y + A.edge && e >= A.e_min && e <= A.e_max)) return out;
    const double pu = ((double)u - A.u_lo) * A.inv_hu, px = (2.0 * sqrt((double)e * A.inv_kappa) - A.x_lo) * A.inv_hx;
    const int cu = (int)floor(pu), cx = (int)floor(px);
    if (cu < 0 || cu >= A.ncu || cx < 0 || cx >= A.nce) return out;
    *fu = pu - cu;
    *fx = px - cx;
    *sub = 2 * (cx & 1) + (cu & 1);
    return (s * A.nbx + (cx >> 1)) * A.nbu + (cu >> 1);
}
__global__ void k_grid_count(CellArgs A, int32_t* __restrict__ cnt) {
    const int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    double fu, fx;
    int sub;
    if (r < A.J) atomicAdd(cnt + grid_block(A, r, &fu, &fx, &sub), 1);
}
// events of the input outside the grid's region (before the sort)
__global__ void k_grid_outside(CellArgs A, int32_t* __restrict__ n) {
    const int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    bool out = false;
    if (r < A.J) {
        const int a = A.a_s[r];
        if (a >= 0 && a < A.n_slots) {
            double fu, fx;
            int sub;
            out = grid_block(A, r, &fu, &fx, &sub) >= A.n_slots * A.nbx * A.nbu;
        }
    }
    const unsigned b = __ballot_sync(0xffffffffu, out);
    if (b && (threadIdx.x & 31) == 0) atomicAdd(n, __popc(b));
}

// an event in block order: its row, cell (4 x block + cell of the block; outside
// the grid the key itself), position and energy, and its weights
struct __align__(16) GridEvent {
    int32_t row, cell;
    float u, e;
    float we[kPE], wu[kPU];
};
static_assert(sizeof(GridEvent) == 96, "six 16-byte words");

__global__ void k_grid_place(CellArgs A, Stencil<kPU> su, Stencil<kPE> sx, const int32_t* __restrict__ off,
                             int32_t* __restrict__ fill, GridEvent* __restrict__ out) {
    const int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= A.J) return;
    double fu = 0.0, fx = 0.0;
    int sub = 0;
    const int c = grid_block(A, r, &fu, &fx, &sub);
    GridEvent ev;
    ev.row = (int32_t)r;
    ev.cell = c < A.n_slots * A.nbx * A.nbu ? 4 * c + sub : c;
    ev.u = A.u_s[r];
    ev.e = A.e_s[r];
    stencil_weights<kPU>(su, fu, ev.wu);
    stencil_weights<kPE>(sx, fx, ev.we);
    // the order inside a block does not matter: every row is formed by itself
    out[off[c] + atomicAdd(fill + c, 1)] = ev;
}

struct RowArgs {
    const GridEvent* ev;
    const int32_t* off;          // first event of every block
    int cell0, cell1;            // blocks of the group
    int nbx, nbu, ne, nu, s0;
    const int32_t* slot_angle;
    const float* T;
    int n_sup, ld;
    const float4* ppar;
    int ld_w;
    float e0, sE0, lE0;
    float* out;
    int64_t ld_out, row_base;
};

// Rows of 64 events (in block order) x 128 support pixels: the 13 x 9 grid
// values around a block of 2 x 2 cells are loaded once for all of its events.
// The values take 166 registers, so 12 warps per SM; what bounds the kernel is
// each warp's own chain: 47% of the issue slots are used, 2.2 cycles per
// instruction go to fixed latencies and 0.9 to loads.  Fewer instructions per
// event shorten it: blocks of 2 x 2
// cells hold about twice the events of a cell for 1.2 times the values (per 33k
// events at 128 x 128 1.97 -> 1.78 ms), and an odd cell shifts its 12 weights
// instead of 96 values (model build of 250k events at 128 x 128 50.0 -> 48.7 ms,
// of 450k at 64 x 64 9.20 -> 8.57), and the sum over the energy nodes comes
// first, packed throughout (48.7 -> 48.4, 8.57 -> 8.40).  Slower: larger blocks (53.6 to 54.9 ms; 174
// to 192 registers), two lanes per pixel (53.3; 20 warps per SM instead of 12),
// the values of 8 blocks in shared memory (2.40 ms per 33k), those of a
// neighbouring block moved up in registers (2.20), the next block's lines
// prefetched to L1 (2.25).
constexpr int kRowEvents = 64;
template <int OX, int OU>
__device__ __forceinline__ float stencil_sum(const float (&tv)[kPE + 1][kPU + 1], const float (&we)[kPE],
                                             const float (&wu)[kPU]) {
    // pairs of values as they lie in the registers; OU = 1 shifts the weights
    float2 w[kPU / 2];
#pragma unroll
    for (int k = 0; k < kPU; k += 2)
        w[k / 2] = OU ? make_float2(k ? wu[k - 1] : 0.0f, wu[k]) : make_float2(wu[k], wu[k + 1]);
    // over the energy nodes first: a position's chain is packed throughout
    float2 v[kPU / 2];
    float last = 0.0f;
#pragma unroll
    for (int k = 0; k < kPU / 2; ++k) v[k] = make_float2(0.0f, 0.0f);
#pragma unroll
    for (int q = 0; q < kPE; ++q) {
        const float* t = tv[q + OX];
        const float2 e = make_float2(we[q], we[q]);
#pragma unroll
        for (int k = 0; k < kPU; k += 2) v[k / 2] = fma2(e, make_float2(t[k], t[k + 1]), v[k / 2]);
        if (OU) last = fmaf(we[q], t[kPU], last);
    }
    float2 acc = make_float2(OU ? wu[kPU - 1] * last : 0.0f, 0.0f);
#pragma unroll
    for (int k = 0; k < kPU / 2; ++k) acc = fma2(w[k], v[k], acc);
    return acc.x + acc.y;
}
__global__ void __launch_bounds__(128) k_grid_rows(RowArgs A) {
    __shared__ float4 sev[kRowEvents * 6];
    const int p0 = A.off[A.cell0] + blockIdx.x * kRowEvents, p1 = min(A.off[A.cell1], p0 + kRowEvents);
    if (p0 >= p1) return;
    const float4* src = reinterpret_cast<const float4*>(A.ev + p0);
    for (int k = threadIdx.x; k < (p1 - p0) * 6; k += 128) sev[k] = src[k];
    __syncthreads();
    const int n = blockIdx.y * 128 + threadIdx.x;
    if (n >= A.ld) return;
    const bool real = n < A.n_sup;
    float tv[kPE + 1][kPU + 1];
    float4 pp = make_float4(0.0f, 0.0f, -INFINITY, 0.0f);
    int block = -1;
    for (int p = 0; p < p1 - p0; ++p) {
        const float4 h = sev[p * 6];
        const int row = __float_as_int(h.x), c = __float_as_int(h.y);
        if ((c >> 2) != block) {
            block = c >> 2;
            const int cu = 2 * (block % A.nbu), cx = 2 * ((block / A.nbu) % A.nbx), s = block / (A.nbu * A.nbx);
            const float* t = A.T + ((((size_t)(s - A.s0) * gridDim.y + blockIdx.y) * A.ne + cx) * A.nu + cu) * kTCols +
                             threadIdx.x;
#pragma unroll
            for (int q = 0; q <= kPE; ++q) {
                if (q == kPE && cx + q >= A.ne) break;  // the last block may hold one row of cells only
#pragma unroll
                for (int k = 0; k <= kPU; ++k) tv[q][k] = __ldg(t + k * kTCols);
                t += (size_t)A.nu * kTCols;
            }
            if (real) pp = __ldg(A.ppar + (size_t)A.slot_angle[s] * A.ld_w + n);
        }
        float we[kPE], wu[kPU];
#pragma unroll
        for (int k = 0; k < (kPE + kPU) / 4; ++k) {
            const float4 v = sev[p * 6 + 1 + k];
            float* w = k < kPE / 4 ? we + 4 * k : wu + 4 * (k - kPE / 4);
            w[0] = v.x;
            w[1] = v.y;
            w[2] = v.z;
            w[3] = v.w;
        }
        float acc;
        if (c & 2) acc = (c & 1) ? stencil_sum<1, 1>(tv, we, wu) : stencil_sum<1, 0>(tv, we, wu);
        else acc = (c & 1) ? stencil_sum<0, 1>(tv, we, wu) : stencil_sum<0, 0>(tv, we, wu);
        const float te = (h.w - A.e0) * A.sE0, tu = (h.z - pp.x) * pp.y;
        const float prim = ex2_approx(fmaf(-tu, tu, pp.z + fmaf(-te, te, A.lE0)));
        // the sum is never negative; an interpolated zero may be, by its rounding
        A.out[(row - A.row_base) * A.ld_out + n] = real ? fmaxf(acc, 0.0f) + prim : 0.0f;
    }
}

// The interpolation's error is absolute: about 4e-7 of the largest of the grid
// values that it combines.  Where S_n falls steeply for every n (energies above
// every Compton energy that reaches a position, positions that no scatter pixel
// looks at) and no primary covers it, that is no longer small against the row:
// for a unit Gaussian 1.3e-6 of the value 2 sigma out, 5e-6 at 2.5, 1.3e-5 at 3,
// 3e-4 at 4.  Such rows are summed path by path.  An event's row is taken to be
// steep when its largest value (of S_n over the support, interpolated in the
// logarithm, or of the primary) is below 1 / kSteep of the largest S_n 4 nodes
// away along one of the axes (1 sigma in x, 1.7 of the narrowest sigma in u):
// from 2.6 sigma on in x, and in u from 2.1 sigma of the narrowest response on
// and 3.5 of one twice as wide, which the grid resolves better.
constexpr float kSteepLog2 = 3.0f;
constexpr int kTopStep = 4;      // nodes between those where the largest S_n is taken

// log2 of the largest S_n over the support at every kTopStep-th node of either
// axis, 4 warps per node: a sixteenth of T is read, which bounds it.  (Taken in
// the sum's epilogue it cost 1.5 to 3% of the sum.)  Also keeps the length of
// the list of directly summed rows before this group.
__global__ void __launch_bounds__(128) k_grid_top(const float* __restrict__ T, int ne, int nu, int ld,
                                                  float* __restrict__ top, const int32_t* n_list, int32_t* n_list0) {
    __shared__ float sh[4];
    if (blockIdx.x + blockIdx.y + blockIdx.z == 0 && threadIdx.x == 0) *n_list0 = *n_list;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, n_full = ld / kTCols, n_tiles = (ld + kTCols - 1) / kTCols;
    const float* t = T + (((size_t)blockIdx.z * n_tiles * ne + kTopStep * blockIdx.y) * nu + kTopStep * blockIdx.x) * kTCols +
                     4 * lane;
    float mx = 0.0f;
    auto take = [&](int k) {
        const float4 v = *reinterpret_cast<const float4*>(t + (size_t)k * ne * nu * kTCols);
        mx = fmaxf(fmaxf(mx, fmaxf(v.x, v.y)), fmaxf(v.z, v.w));
    };
#pragma unroll 4
    for (int k = warp; k < n_full; k += 4) take(k);
    if (warp == n_full % 4 && n_full * kTCols + 4 * lane < ld) take(n_full);  // (columns past ld are not written)
    for (int o = 16; o; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if (lane == 0) sh[warp] = mx;
    __syncthreads();
    if (threadIdx.x == 0)
        top[((size_t)blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x] =
            __log2f(fmaxf(fmaxf(fmaxf(sh[0], sh[1]), fmaxf(sh[2], sh[3])), 1e-37f));
}

struct TailArgs {
    const GridEvent* ev;
    const int32_t* off;
    int cell0, cell1;            // blocks of the group
    int per_slot, s0;            // per_slot: blocks of cells
    int nx, nm;                  // nodes of top
    const float* top;            // [angle of the group][nx][nm]
    const float* pmax;           // [slot][nm]: log2 of the largest primary, without its energy factor
    float u_lo, inv_hu, x_lo, inv_hx, inv_kappa;
    float e0, sE0, lE0;
    int max_list;
    int32_t* list;               // places in ev of the rows to be summed directly
    int32_t* n_list;             // rows found so far, those of earlier groups included
};
__global__ void __launch_bounds__(256) k_grid_tails(TailArgs A) {
    const int p = A.off[A.cell0] + blockIdx.x * 256 + threadIdx.x;
    if (p >= A.off[A.cell1]) return;
    const float4 h = *reinterpret_cast<const float4*>(A.ev + p);
    const int s = (__float_as_int(h.y) >> 2) / A.per_slot;
    // place among the nodes, and among those of top
    const float iu = fmaxf((h.z - A.u_lo) * A.inv_hu, 0.0f) + (kPU / 2 - 1);
    const float ix = fmaxf((2.0f * sqrtf(h.w * A.inv_kappa) - A.x_lo) * A.inv_hx, 0.0f) + (kPE / 2 - 1);
    const int ju = (int)(iu / kTopStep), jx = (int)(ix / kTopStep);
    const float fu = iu / kTopStep - ju, fx = ix / kTopStep - jx;
    const float* t = A.top + (size_t)(s - A.s0) * A.nx * A.nm;
    auto at = [&](int dx, int du) {  // dx, du nodes of top from the event
        const int x0 = min(max(jx + dx, 0), A.nx - 1), x1 = min(max(jx + dx + 1, 0), A.nx - 1);
        const int u0 = min(max(ju + du, 0), A.nm - 1), u1 = min(max(ju + du + 1, 0), A.nm - 1);
        const float a = t[x0 * A.nm + u0], b = t[x0 * A.nm + u1], c = t[x1 * A.nm + u0], d = t[x1 * A.nm + u1];
        const float lo = fmaf(fu, b - a, a), hi = fmaf(fu, d - c, c);
        return fmaf(fx, hi - lo, lo);
    };
    const float around = fmaxf(fmaxf(at(-1, 0), at(1, 0)), fmaxf(at(0, -1), at(0, 1)));
    const float te = (h.w - A.e0) * A.sE0;
    const float* pm = A.pmax + (size_t)s * A.nm;
    const float p0 = pm[min(ju, A.nm - 1)], p1 = pm[min(ju + 1, A.nm - 1)];
    const float row = fmaxf(at(0, 0), fmaf(fu, p1 - p0, p0) + fmaf(-te, te, A.lE0));
    if (row + kSteepLog2 >= around) return;
    const int k = atomicAdd(A.n_list, 1);
    if (k < A.max_list) A.list[k] = p;
}
// log2 of the largest primary over the support at every kTopStep-th position
// node, without the energy factor
__global__ void __launch_bounds__(128) k_grid_prim(const float4* __restrict__ ppar, const int32_t* __restrict__ slot_angle,
                                                   int ld_w, int n_sup, double u_node0, double step,
                                                   float* __restrict__ pmax) {
    __shared__ float sh[4];
    const float4* pp = ppar + (size_t)slot_angle[blockIdx.y] * ld_w;
    const float u = (float)(u_node0 + blockIdx.x * step);
    float mx = -INFINITY;
    for (int n = threadIdx.x; n < n_sup; n += 128) {
        const float4 q = __ldg(pp + n);
        const float t = (u - q.x) * q.y;
        mx = fmaxf(mx, fmaf(-t, t, q.z));
    }
    for (int o = 16; o; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = mx;
    __syncthreads();
    if (threadIdx.x == 0)
        pmax[(size_t)blockIdx.y * gridDim.x + blockIdx.x] =
            fmaxf(fmaxf(fmaxf(sh[0], sh[1]), fmaxf(sh[2], sh[3])), -1000.0f);
}

// Rows of the events outside the grid's region and of the steep rows, summed
// path by path, nothing shared between them.
struct DirectArgs {
    const GridEvent* ev;
    const int32_t* off;
    int key0, key1;              // keys of the group's events outside the grid
    const int32_t* list;         // places in ev of the steep rows:
    const int32_t* list0;        // the group's first one
    const int32_t* n_list;       // all found so far; none is summed here once there are more than max_list
    int max_list, per_slot;      // per_slot: blocks of cells
    int ncells, s0;
    const int32_t* slot_angle;
    const float4* planes;
    const int32_t* slot_m;
    const int32_t* n_sub;
    const float4* mpar;
    int n_scat, max_sub;
    float cE2, inv_scale;
    int n_sup, ld;
    const float4* ppar;
    int ld_w;
    float e0, sE0, lE0;
    float* out;
    int64_t ld_out, row_base;
};
// One CTA per (128 columns, row): 128 scatter pixels at a time, those within
// their cut listed in shared memory, so that the table values of several of
// them are in flight (a group with one row at 64 x 64: 40 us, about 350 with the
// test and the loads of one pixel after the other).
__global__ void __launch_bounds__(128) k_grid_direct(DirectArgs A) {
    __shared__ float2 near[128];  // (slot, U) of the pixels within their cut, in slot order
    __shared__ int cnt[4];
    const int n = blockIdx.x * 128 + threadIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const bool col = n < A.ld, real = n < A.n_sup;
    const int out0 = A.off[A.key0], n_out = A.off[A.key1] - out0;
    const int l0 = *A.list0, n_list = *A.n_list <= A.max_list ? *A.n_list - l0 : 0;
    for (int j = blockIdx.y; j < n_out + n_list; j += gridDim.y) {
        const GridEvent* ev = A.ev + (j < n_out ? out0 + j : A.list[l0 + j - n_out]);
        const int s = j < n_out ? ev->cell - A.ncells : (ev->cell >> 2) / A.per_slot, a = A.slot_angle[s];
        const float u = ev->u, e = ev->e, E = e * A.cE2, El = fmaf(e, A.cE2, -E);
        const int nc = col ? n : 0;  // threads past the row join the lists only
        const float4* pl =
            A.planes + ((size_t)(s - A.s0) * (A.ld / kNTile) + nc / kNTile) * (A.max_sub * kSub / 2) * kNTile + nc % kNTile;
        const int32_t* sm = A.slot_m + (size_t)a * A.max_sub * kSub;
        const int n_slots = A.n_sub[a] * kSub;
        float acc = 0.0f;
        for (int b = 0; b < n_slots; b += 128) {
            const int k = b + threadIdx.x, m = k < n_slots ? __ldg(sm + k) : -1;
            bool in = false;
            float U = 0.0f;
            if (m >= 0) {
                const float4 q = __ldg(A.mpar + (size_t)a * A.n_scat + m);
                const float d = u - q.x, z = d * q.y;
                in = fabsf(d) <= q.w;
                U = ex2_approx(fmaf(-z, z, q.z));
            }
            const unsigned bal = __ballot_sync(0xffffffffu, in);
            __syncthreads();  // the last list is read
            if (lane == 0) cnt[warp] = __popc(bal);
            __syncthreads();
            int first = 0, total = 0;
#pragma unroll
            for (int w = 0; w < 4; ++w) {
                if (w < warp) first += cnt[w];
                total += cnt[w];
            }
            if (in) near[first + __popc(bal & ((1u << lane) - 1u))] = make_float2(__int_as_float(k), U);
            __syncthreads();
#pragma unroll 8
            for (int i = 0; i < total; ++i) {
                const float2 q = near[i];
                const int kk = __float_as_int(q.x);
                const float* v = reinterpret_cast<const float*>(pl + (kk >> 1) * kNTile);
                const float e1 = __ldg(v + (kk & 1)), w = __ldg(v + 2 + (kk & 1)), t = (E - e1 + El) * rsqrt_approx(e1);
                acc = fmaf(q.y, ex2_approx(-fmaf(t, t, w)), acc);
            }
        }
        if (!col) continue;
        const float4 pp = A.ppar[(size_t)a * A.ld_w + n];
        const float te = (e - A.e0) * A.sE0, tu = (u - pp.x) * pp.y;
        const float prim = ex2_approx(fmaf(-tu, tu, pp.z + fmaf(-te, te, A.lE0)));
        A.out[(ev->row - A.row_base) * A.ld_out + n] = real ? fmaf(acc, A.inv_scale, prim) : 0.0f;
    }
}

double kappa_of(const lmosem_ctx* c) {
    const double fw2s = 1.0 / (2.0 * sqrt(2.0 * log(2.0)));
    return pow(c->fwhm_frac * fw2s, 2.0) * c->e0;  // sigma_E^2 = kappa E
}

CellArgs cell_args(const lmosem_ctx* c, const int32_t* a, const float* u, const float* e, int64_t n) {
    const GridPlan& G = c->grid;
    CellArgs A;
    A.a_s = a;
    A.u_s = u;
    A.e_s = e;
    A.J = n;
    A.angle_slot = G.d_angle_slot;
    A.urange = G.d_urange;
    A.edge = (float)G.edge;
    A.e_min = (float)G.e_min;
    A.e_max = (float)G.e_max;
    A.u_lo = G.u_lo;
    A.inv_hu = 1.0 / G.hu;
    A.x_lo = G.x_lo;
    A.inv_hx = 1.0 / kRhoX;
    A.inv_kappa = 1.0 / kappa_of(c);
    A.nce = G.nce;
    A.ncu = G.ncu;
    A.n_slots = c->n_angles;
    A.nbx = (G.nce + 1) / 2;
    A.nbu = (G.ncu + 1) / 2;
    return A;
}

}  // namespace

// Whether n events of this problem are worth the grid, and its plan.
//
// Both costs in seconds on GB300, as measured (the grid at 50, 64 and 128
// pixels across, the path sum at 50 to 128):
//  * the grid, per angle: k_grid_sum takes 2,300 cycles per subgroup and CTA
//    (and 9,000 per CTA) on 152 CTAs at a time, k_grid_rows about 400 cycles
//    per event and 128 columns, the tables and launches a few microseconds;
//  * the path sum: 5.5e12 terms per second, 0.8 of the position strip's terms
//    being kept by the energy cut.
// They meet near 500 events per angle at 128 x 128 (6,000 pixels) and near
// 1,000 at 64 x 64 (1,540); the grid has to win by a tenth, with every row that
// is summed directly (k_grid_direct) counted as kDirectCost of the path sum's.
// (Measured: 2.5 path-sum rows each for 1,000 at the edge of the object at 64 x
// 64, more inside it, and the latency of one per group, 40 us.)
lmosem_status grid_plan(lmosem_ctx* c, int64_t n, bool* use) {
    *use = false;
    if (n < (int64_t)64 * c->n_angles || c->n_scat < 2 * kSub || c->n_scat > 16384) return LMOSEM_OK;
    // Only for the default cuts.  Narrower ones leave steps in S_n; a wider position cut asks for terms beyond
    // kFarSigma of the widest response, which the window of nodes does not hold; no energy cut asks for the exact
    // sum.  (A wider energy cut drops fewer terms than the default, and the grid drops none by energy.)
    if (c->k_sigma != 6.0f || c->e_sigma < 6.0f) return LMOSEM_OK;
    GridPlan& G = c->grid;
    if (G.state == 0) {
        G.state = 1;  // not usable unless set below
        // widths over the scatter pixels' disc, positions over every angle
        double rmax = 0.0;
        for (int m : c->h_scat) {
            const double x = (m % c->nx + 0.5 - 0.5 * c->nx) * c->dpx, y = (m / c->nx + 0.5 - 0.5 * c->ny) * c->dpx;
            rmax = std::max(rmax, x * x + y * y);
        }
        rmax = sqrt(rmax);
        const double f2s = 0.42466090014400953;
        const double s_min = (c->fwhm0 + c->fwhm_slope * (c->radius - rmax)) * f2s;
        const double s_max = (c->fwhm0 + c->fwhm_slope * (c->radius + rmax)) * f2s;
        const double s_lat = (c->fwhm0 + c->fwhm_slope * c->radius) * f2s;  // of the outermost pixels
        const double half = 0.5 * c->n_bins * c->bin_mm, cut = kFarSigma * s_max;
        // The window of nodes has to hold the widest response.  A scatter pixel whose k_sigma cut is longer than
        // kFarSigma of the widest (the last few centimetres of depth) is cut there instead: what is left out is
        // below 4e-8 of its response's mass.  The pixels that bound the object sideways keep their whole cut.
        G.cut = cut;
        // window of a subgroup: 2 cut + span, rounded down to a multiple of 8 nodes
        const double span = std::min((kWin - 9) * kRhoUMax * s_min - 2.0 * cut, 1.25 * kSub * 2.0 * rmax / c->n_scat);
        if (!(span > 0.0) || span < 0.25 * 1.25 * kSub * 2.0 * rmax / c->n_scat) return LMOSEM_OK;
        G.hu = std::max((2.0 * cut + span) / (kWin - 9), kRhoUMin * s_min);
        if (!(G.hu <= 1.001 * kRhoUMax * s_min)) return LMOSEM_OK;
        G.rho_u = G.hu / (kWideU * s_min);
        G.edge = kEdgeSigma * s_lat;
        const double ext = std::min(half, rmax + G.edge);
        G.u_lo = -ext;
        G.ncu = (int)floor(2.0 * ext / G.hu) + 1;
        G.nu = (G.ncu + 1) / 2 * 2 + kPU - 1;  // whole blocks of 2 cells
        const double kappa = kappa_of(c), e_min = c->e0 / (1.0 + 2.0 * c->e0 / kMec2Kev);
        G.e_min = std::max(c->e_lo, e_min - 1.5 * sqrt(kappa * e_min));
        G.e_max = std::min(c->e_hi, c->e0 + kEdgeSigma * sqrt(kappa * c->e0));
        if (!(G.e_max > G.e_min)) return LMOSEM_OK;
        G.x_lo = 2.0 * sqrt(G.e_min / kappa);
        if (!(G.x_lo > 2.0 * kPE * kRhoX)) return LMOSEM_OK;  // nodes at positive energies
        G.nce = (int)floor((2.0 * sqrt(G.e_max / kappa) - G.x_lo) / kRhoX) + 1;
        G.ne = (G.nce + kPE - 1 + kEGroup - 1) / kEGroup * kEGroup;
        if (G.ne > 128 || (int64_t)c->n_angles * G.nce * G.ncu > (int64_t(1) << 28)) return LMOSEM_OK;
        G.max_sub = (c->n_scat + kSub - 1) / kSub + (int)ceil(2.0 * rmax / span) + 2;
        // scales that keep the FP16 parts in range: G <= D mu / (2 pi Kbar) / (sigma_E sqrt(2 pi)), U <= 1 / (sigma_u sqrt(2 pi))
        const double gb = c->dpx * c->mu_max / (2.0 * kPi * c->kbar) / sqrt(2.0 * kPi * kappa * e_min);
        const double ub = 1.0 / (s_min * sqrt(2.0 * kPi));
        G.log_g = (float)(14 - (int)ceil(log2(gb)));
        G.log_u = (float)(14 - (int)ceil(log2(ub)));
        if (!(fabs(G.log_g) < 60.0f && fabs(G.log_u) < 30.0f)) return LMOSEM_OK;

        G.span = span;
        G.n_sub = 1 + (int)(1.1 * std::max((double)c->n_scat / kSub, 2.0 * rmax / span));
        G.strip = std::min(1.0, 1.2 * c->k_sigma * s_lat / rmax);
        G.state = 2;  // parameters known, tables not made
    }
    if (G.state < 2) return LMOSEM_OK;
    const double per_s = 152.0 * 1.92e9, tiles = (c->n_sup + 127) / 128;
    const double t_grid = c->n_angles * ((c->n_sup + kNTile - 1) / kNTile * (G.ne / kEGroup) * (2300.0 * G.n_sub + 9000.0) / per_s +
                                         tiles * G.n_sub * 25e-9) + n * tiles * 400.0 / per_s + 60e-6;
    const double t_path = n * (0.8 * G.strip * c->n_scat * c->n_sup) / 5.5e12;
    G.ratio = t_grid / t_path;
    if (!(G.ratio < kGridGain)) return LMOSEM_OK;
    *use = true;
    if (G.state == 3) return LMOSEM_OK;
    const double kappa = kappa_of(c);
    lmosem_status st;
    const size_t na = c->n_angles;
    int32_t* order = nullptr;
    Scratch tmp(c);
    if ((st = tmp.alloc(&order, na * c->n_scat)) || (st = dev_alloc(c, &G.d_slot_m, na * G.max_sub * kSub)) ||
        (st = dev_alloc(c, &G.d_i0, na * G.max_sub)) || (st = dev_alloc(c, &G.d_n_sub, na)) ||
        (st = dev_alloc(c, &G.d_urange, na)) || (st = dev_alloc(c, &G.d_enode, G.ne / 2)) ||
        (st = dev_alloc(c, &G.d_angle_slot, na)))
        return st;
    std::vector<float4> en(G.ne / 2);
    const double cE2 = (float)(1.4426950408889634 / (2.0 * kappa));  // as the tables' FP32 factor
    auto node = [&](int k) {
        const double x = G.x_lo + (k - (kPE / 2 - 1)) * kRhoX;
        return cE2 * kappa * 0.25 * x * x;
    };
    for (int k = 0; k < G.ne / 2; ++k) {
        const double e0 = node(2 * k);
        const float hi = (float)e0;
        en[k] = make_float4(hi, (float)(e0 - hi), (float)(node(2 * k + 1) - e0), 0.0f);
    }
    LMOSEM_CK(c, cudaMemcpyAsync(G.d_enode, en.data(), en.size() * sizeof(float4), cudaMemcpyHostToDevice, c->stream));
    LMOSEM_PROF_BEGIN(c);
    k_grid_rank<<<dim3((c->n_scat + 255) / 256, c->n_angles), 256, 0, c->stream>>>(c->d_mpar, c->n_scat, order);
    LMOSEM_LAUNCHED(c, LMOSEM_K_TABLES);
    const size_t smem = sizeof(float) * ((size_t)c->n_scat + G.max_sub + 1);
    if ((st = opt_in_smem(c, k_grid_groups))) return st;
    LMOSEM_PROF_BEGIN(c);
    k_grid_groups<<<c->n_angles, 256, smem, c->stream>>>(
        c->d_mpar, order, c->n_scat, G.max_sub, (float)G.span, (float)G.cut,
        (float)(G.u_lo - (kPU / 2 - 1) * G.hu), (float)(1.0 / G.hu), G.d_slot_m, G.d_i0, G.d_n_sub, G.d_urange);
    LMOSEM_LAUNCHED(c, LMOSEM_K_TABLES);
    G.state = 3;
    return LMOSEM_OK;
}

void grid_free(lmosem_ctx* c) {
    dev_free(c, &c->grid.d_slot_m);
    dev_free(c, &c->grid.d_i0);
    dev_free(c, &c->grid.d_n_sub);
    dev_free(c, &c->grid.d_urange);
    dev_free(c, &c->grid.d_enode);
    dev_free(c, &c->grid.d_angle_slot);
}

// events (unsorted, already known to be in range) outside the grid's region
lmosem_status grid_count_outside(lmosem_ctx* c, const int32_t* a, const float* u, const float* e, int64_t n,
                                 int32_t* d_n) {
    CellArgs A = cell_args(c, a, u, e, n);
    // any slot order counts alike: the angle itself stands for it
    std::vector<int32_t> ident(c->n_angles);
    for (int k = 0; k < c->n_angles; ++k) ident[k] = k;
    LMOSEM_CK(c, cudaMemcpyAsync(c->grid.d_angle_slot, ident.data(), ident.size() * sizeof(int32_t),
                                 cudaMemcpyHostToDevice, c->stream));
    LMOSEM_PROF_BEGIN(c);
    k_grid_outside<<<(unsigned)((n + 255) / 256), 256, 0, c->stream>>>(A, d_n);
    LMOSEM_LAUNCHED(c, LMOSEM_K_SORT);
    return LMOSEM_OK;
}

// Rows of every sorted event (scaled forms: staged as FP32 per group and
// rounded), angle group by angle group within the table budget.  ratio: the
// list's cost here over the path sum's, before any row is known to be steep.
// *done = false: so many rows are steep that the path sum forms the whole list
// faster than what is left to do here (looked at once, after the first group),
// or than their direct sums (at the end).
lmosem_status build_model_rows_grid(lmosem_ctx* c, const std::vector<int32_t>& slot_angle, double ratio, bool* done) {
    const GridPlan& G = c->grid;
    *done = false;
    lmosem_status st;
    if ((st = ensure_status(c))) return st;
    const int ns = (int)slot_angle.size(), ld = (int)c->ld_model;
    const int64_t J = c->J;
    const double kappa = kappa_of(c), se0 = sqrt(kappa * c->e0);
    const int nbx = (G.nce + 1) / 2, nbu = (G.ncu + 1) / 2;
    const int64_t ncells = (int64_t)ns * nbx * nbu, nkeys = ncells + ns;

    // ---- events in cell order, with their weights
    std::vector<int32_t> slots(2 * ns);
    for (int s = 0; s < ns; ++s) {
        slots[s] = slot_angle[s];
        slots[ns + slot_angle[s]] = s;
    }
    int32_t *d_slot = nullptr, *off = nullptr, *fill = nullptr, *tot = nullptr;
    GridEvent* ev = nullptr;
    Scratch tmp(c);
    if ((st = tmp.alloc(&d_slot, ns)) || (st = tmp.alloc(&off, nkeys + 1)) || (st = tmp.alloc(&fill, nkeys)) ||
        (st = tmp.alloc(&tot, scan_blocks(nkeys + 1))) || (st = tmp.alloc(&ev, J)))
        return st;
    LMOSEM_CK(c, cudaMemcpyAsync(d_slot, slots.data(), ns * sizeof(int32_t), cudaMemcpyHostToDevice, c->stream));
    LMOSEM_CK(c, cudaMemcpyAsync(G.d_angle_slot, slots.data() + ns, ns * sizeof(int32_t), cudaMemcpyHostToDevice,
                                 c->stream));
    LMOSEM_CK(c, cudaMemsetAsync(off, 0, sizeof(int32_t) * (nkeys + 1), c->stream));
    LMOSEM_CK(c, cudaMemsetAsync(fill, 0, sizeof(int32_t) * nkeys, c->stream));
    const CellArgs C = cell_args(c, c->d_a_s, c->d_u_s, c->d_e_s, J);
    LMOSEM_PROF_BEGIN(c);
    k_grid_count<<<(unsigned)((J + 255) / 256), 256, 0, c->stream>>>(C, off);
    LMOSEM_LAUNCHED(c, LMOSEM_K_SORT);
    if ((st = exclusive_scan(c, off, nkeys + 1, tot))) return st;
    LMOSEM_PROF_BEGIN(c);
    k_grid_place<<<(unsigned)((J + 255) / 256), 256, 0, c->stream>>>(C, make_stencil<kPU>(G.rho_u),
                                                                     make_stencil<kPE>(kRhoX / kWideX), off, fill, ev);
    LMOSEM_LAUNCHED(c, LMOSEM_K_SORT);

    // ---- angle groups
    const int64_t pairs = (int64_t)G.max_sub * kSub / 2;
    const int64_t plane_n = pairs * ld, t_n = (int64_t)G.ne * G.nu * ((ld + kTCols - 1) / kTCols * kTCols), u_n = (int64_t)G.max_sub * kUStage;
    const int64_t per_angle = plane_n * 16 + t_n * 4 + u_n;
    const int top_x = (G.ne + kTopStep - 1) / kTopStep, top_u = (G.nu + kTopStep - 1) / kTopStep;
    // groups of at most 2 GiB: the pool maps fresh memory at about 0.7 ms per GB (64 x 64 with 200k events: build
    // 17.3 ms at 2 GiB, 18.2 at 1 GiB, 19.1 at 4 GiB)
    int gsz = (int)std::max<int64_t>(
        1, std::min<int64_t>(ns, std::min<int64_t>(c->table_budget, int64_t(2) << 30) / per_angle));
    // a support that leaves scatter pixels out is where steep rows are met: the first group shows it early
    if (c->partial_support) gsz = std::min(gsz, std::max(1, ns / 8));
    float4* planes = nullptr;
    float* T = nullptr;
    unsigned char* ublob = nullptr;
    const int max_list = (int)(J / kDirectCost);
    const int n_groups = (ns + gsz - 1) / gsz;
    int32_t *list = nullptr, *n_list = nullptr;  // n_list[0]: rows found; [1 + gi]: before group gi
    float *pmax = nullptr, *top = nullptr;
    if ((st = tmp.alloc(&planes, (size_t)gsz * plane_n)) || (st = tmp.alloc(&T, (size_t)gsz * t_n)) ||
        (st = tmp.alloc(&ublob, (size_t)gsz * u_n)) || (st = tmp.alloc(&top, (size_t)gsz * top_x * top_u)) ||
        (st = tmp.alloc(&pmax, (size_t)ns * top_u)) || (st = tmp.alloc(&list, max_list)) ||
        (st = tmp.alloc(&n_list, 1 + n_groups)))
        return st;
    const double u_node0 = G.u_lo - (kPU / 2 - 1) * G.hu;
    LMOSEM_CK(c, cudaMemsetAsync(n_list, 0, sizeof(int), c->stream));
    LMOSEM_PROF_BEGIN(c);
    k_grid_prim<<<dim3(top_u, ns), 128, 0, c->stream>>>(c->d_ppar, d_slot, c->ld_w, c->n_sup, u_node0, kTopStep * G.hu,
                                                        pmax);
    LMOSEM_LAUNCHED(c, LMOSEM_K_WTABLE);
    const bool scaled = c->fmt != LMOSEM_MODEL_FP32;
    std::vector<int64_t> g_rows, g_row0;
    for (int s0 = 0; s0 < ns; s0 += gsz) {
        int64_t rows = 0, row0 = -1;
        for (int r = 0; r < c->n_real; ++r)
            for (int s = s0; s < std::min(ns, s0 + gsz); ++s) {
                const size_t k = (size_t)r * c->n_angles + slot_angle[s];
                if (c->h_angle_cnt[k] > 0 && row0 < 0) row0 = c->h_angle_row0[k];
                rows += c->h_angle_cnt[k];
            }
        g_rows.push_back(rows);
        g_row0.push_back(row0);
    }
    if (scaled && (st = dev_alloc(c, &c->d_stage, (size_t)std::max<int64_t>(
                                                       1, *std::max_element(g_rows.begin(), g_rows.end())) * ld)))
        return st;
    if ((st = opt_in_smem(c, k_grid_sum))) return st;
    const float cE2 = (float)(1.4426950408889634 / (2.0 * kappa));
    int64_t rows_done = 0;
    bool looked = false;
    int found = 0;
    for (int s0 = 0, gi = 0; s0 < ns; s0 += gsz, ++gi) {
        const int na = std::min(gsz, ns - s0);
        if (g_rows[gi] == 0) continue;
        UArgs U;
        U.mpar = c->d_mpar;
        U.scat_geo = c->d_scat_geo;
        U.trig = c->d_trig;
        U.slot_m = G.d_slot_m;
        U.i0 = G.d_i0;
        U.n_sub = G.d_n_sub;
        U.slot_angle = d_slot;
        U.s0 = s0;
        U.n_scat = c->n_scat;
        U.max_sub = G.max_sub;
        U.angle0 = c->angle0;
        U.dtheta = 2.0 * kPi / c->n_angles;
        U.u_node0 = u_node0;
        U.hu = G.hu;
        U.cut = (float)G.cut;
        U.scale = G.log_u;
        U.out = ublob;
        LMOSEM_PROF_BEGIN(c);
        k_grid_u<<<dim3(G.max_sub * kChunks, na), 2 * kWin, 0, c->stream>>>(U);
        LMOSEM_LAUNCHED(c, LMOSEM_K_WTABLE);
        PlaneArgs P;
        P.nx = c->nx;
        P.ny = c->ny;
        P.npix = c->npix;
        P.n_sup = c->n_sup;
        P.ld = ld;
        P.n_scat = c->n_scat;
        P.max_sub = G.max_sub;
        P.dpx = (float)c->dpx;
        P.eps0 = (float)(c->e0 / kMec2Kev);
        P.inv_kbar = (float)(1.0 / c->kbar);
        P.e0 = (float)c->e0;
        P.w_const = (float)(c->dpx * c->dpx / (2.0 * kPi * sqrt(2.0 * kPi * kappa)));
        P.cE2 = cE2;
        P.scale = G.log_g;
        P.sup = c->d_sup;
        P.scat_geo = c->d_scat_geo;
        P.trig = c->d_trig;
        P.l_edge = c->d_l_edge;
        P.l_pair = c->d_l_pair;
        P.compton = c->d_compton;
        P.slot_m = G.d_slot_m;
        P.n_sub = G.d_n_sub;
        P.slot_angle = d_slot;
        P.s0 = s0;
        P.out = planes;
        LMOSEM_PROF_BEGIN(c);
        k_grid_planes<<<dim3((ld + 127) / 128, (unsigned)(pairs / kPlanePairs), na), 128, 0, c->stream>>>(P);
        LMOSEM_LAUNCHED(c, LMOSEM_K_WTABLE);
        SumArgs S;
        S.planes = planes;
        S.ublob = ublob;
        S.i0 = G.d_i0;
        S.n_sub = G.d_n_sub;
        S.slot_angle = d_slot;
        S.s0 = s0;
        S.ld = ld;
        S.max_sub = G.max_sub;
        S.ne = G.ne;
        S.nu = G.nu;
        S.n_nt = ld / kNTile;
        S.enode = G.d_enode;
        S.out_scale = (float)exp2(-(double)G.log_g - (double)G.log_u);
        S.T = T;
        S.status = c->d_status;
        S.budget = c->wait_budget;
        LMOSEM_PROF_BEGIN(c);
        k_grid_sum<<<(unsigned)(na * S.n_nt * (G.ne / kEGroup)), kGridThreads, kSmBytes, c->stream>>>(S);
        LMOSEM_LAUNCHED(c, LMOSEM_K_PATHSUM);
        RowArgs R;
        R.ev = ev;
        R.off = off;
        R.cell0 = s0 * nbx * nbu;
        R.cell1 = (s0 + na) * nbx * nbu;
        R.nbx = nbx;
        R.nbu = nbu;
        R.ne = G.ne;
        R.nu = G.nu;
        R.s0 = s0;
        R.slot_angle = d_slot;
        R.T = T;
        R.n_sup = c->n_sup;
        R.ld = ld;
        R.ppar = c->d_ppar;
        R.ld_w = c->ld_w;
        R.e0 = (float)c->e0;
        R.sE0 = (float)(0.8493218002880191 / se0);
        R.lE0 = (float)(-log2(se0 * sqrt(2.0 * kPi)));
        R.out = scaled ? c->d_stage : reinterpret_cast<float*>(c->d_model);
        R.ld_out = ld;
        R.row_base = scaled ? g_row0[gi] : 0;
        LMOSEM_PROF_BEGIN(c);
        k_grid_rows<<<dim3((unsigned)((g_rows[gi] + kRowEvents - 1) / kRowEvents), (unsigned)((ld + 127) / 128)), 128, 0,
                      c->stream>>>(R);
        LMOSEM_LAUNCHED(c, LMOSEM_K_PATHSUM);
        LMOSEM_PROF_BEGIN(c);
        k_grid_top<<<dim3(top_u, top_x, na), 128, 0, c->stream>>>(T, G.ne, G.nu, ld, top, n_list, n_list + 1 + gi);
        LMOSEM_LAUNCHED(c, LMOSEM_K_PATHSUM);
        TailArgs Q;
        Q.ev = ev;
        Q.off = off;
        Q.cell0 = R.cell0;
        Q.cell1 = R.cell1;
        Q.per_slot = nbx * nbu;
        Q.s0 = s0;
        Q.nx = top_x;
        Q.nm = top_u;
        Q.u_lo = (float)C.u_lo;
        Q.inv_hu = (float)C.inv_hu;
        Q.x_lo = (float)C.x_lo;
        Q.inv_hx = (float)C.inv_hx;
        Q.inv_kappa = (float)C.inv_kappa;
        Q.top = top;
        Q.pmax = pmax;
        Q.e0 = R.e0;
        Q.sE0 = R.sE0;
        Q.lE0 = R.lE0;
        Q.max_list = max_list;
        Q.list = list;
        Q.n_list = n_list;
        LMOSEM_PROF_BEGIN(c);
        k_grid_tails<<<(unsigned)((g_rows[gi] + 255) / 256), 256, 0, c->stream>>>(Q);
        LMOSEM_LAUNCHED(c, LMOSEM_K_PATHSUM);
        DirectArgs D;
        D.ev = ev;
        D.off = off;
        D.key0 = (int)(ncells + s0);
        D.key1 = (int)(ncells + s0 + na);
        D.list = list;
        D.list0 = n_list + 1 + gi;
        D.n_list = n_list;
        D.max_list = max_list;
        D.per_slot = nbx * nbu;
        D.ncells = (int)ncells;
        D.s0 = s0;
        D.slot_angle = d_slot;
        D.planes = planes;
        D.slot_m = G.d_slot_m;
        D.n_sub = G.d_n_sub;
        D.mpar = c->d_mpar;
        D.n_scat = c->n_scat;
        D.max_sub = G.max_sub;
        D.cE2 = cE2;
        D.inv_scale = (float)exp2(-(double)G.log_g);
        D.n_sup = c->n_sup;
        D.ld = ld;
        D.ppar = c->d_ppar;
        D.ld_w = c->ld_w;
        D.e0 = R.e0;
        D.sE0 = R.sE0;
        D.lE0 = R.lE0;
        D.out = R.out;
        D.ld_out = ld;
        D.row_base = R.row_base;
        LMOSEM_PROF_BEGIN(c);
        k_grid_direct<<<dim3((unsigned)((ld + 127) / 128), 64), 128, 0, c->stream>>>(D);
        LMOSEM_LAUNCHED(c, LMOSEM_K_PATHSUM);
        if (scaled && (st = quantize_rows(c, g_rows[gi], g_row0[gi]))) return st;
        rows_done += g_rows[gi];
        if (rows_done < J && !looked) {  // the first group with events, if others follow
            looked = true;
            LMOSEM_CK(c, cudaMemcpyAsync(&found, n_list, sizeof(int), cudaMemcpyDeviceToHost, c->stream));
            LMOSEM_CK(c, cudaStreamSynchronize(c->stream));
            const double f = (double)rows_done / (double)J;
            if (found > 32 && (1.0 - f) * ratio + kDirectCost * found / (f * J) > 1.0) break;
        }
    }
    dev_free(c, &c->d_stage);
    LMOSEM_CK(c, cudaMemcpyAsync(&found, n_list, sizeof(int), cudaMemcpyDeviceToHost, c->stream));
    st = take_status(c);  // a bounded wait that ran out; synchronises
    *done = rows_done == J && found <= max_list;
    return st;
}

}  // namespace lmosem
