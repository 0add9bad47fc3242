// One explicit UGKS step on the global velocity mesh (paper Sec. 2.3, with
// the explicit readings R1-R4), as four kernels.
//
// k_foot_f2 (FP32 form) / k_foot (FP64 form): per cell and node, the limited
//   least-squares gradient L grad phi (Sec. 2.3.3: weights 1/|d|^2,
//   Venkatakrishnan limiter with epsilon^2 = (K dx)^3 phi_C^2), kept in
//   registers, and the foot values phi_C + (L grad phi)_C . (x_f - xi h - x_C)
//   of every face of the cell at the nodes where the cell is upwind (sign of
//   xi . An), written to the face's row: each face node gets its foot value
//   exactly once.
//
// k_face32 (avs_step32.cu) / k_face: the raw velocity moments of a face's foot
//   values (interface W of Eq. w_interface and heat flux), the interface
//   Shakhov state (Eqs. 3, equ28, R4), then the interface distribution
//   phi_ij = tau/(tau+h) phi_bar + h/(tau+h) g_ij per node.  Writes the
//   per-node flux (xi . An) phi_ij over the foot values and the face's
//   area-weighted flux of W.  Boundaries: diffuse wall with zero net mass
//   flux, far-field Maxwellian (R8).
//
// k_cell_state: one thread per cell.  Lagged heat flux from the moments of f^n
//   (R3), W~ = W - dt/|V| sum_j A F_j (R2), the cell's Shakhov state.
// k_cell32 (avs_step32.cu) / k_cell: the collision update of every node of a
//   cell from the net flux of its faces (diagonal of Eq. SGS_phi, R1).
//
// Every face is evaluated once, so the two cells of a face see the same flux
// and W telescopes exactly.  f^n and W^n are read-only during the step; no
// block waits on another.  Sums in the FP32 form: FP32 over a thread's nodes
// and over the warp; FP64 over the warps of a block and, in the cell kernels, over
// runs of eight quads of a thread (a face group of one warp sums its row, of 1024
// nodes at most, in FP32; a face's FP32 chains are a 1/128 of rows to 48 KB, a 1/256
// of longer ones).  Interface and cell states: FP32 formulas on these sums, the
// balance of W in FP64.  The limited-gradient kernel k_grad (gradients stored next
// to f) serves the FP64 form of the Rykov model.
#include <algorithm>
#include <type_traits>

#include "avs_dev.cuh"
#include "avs_internal.h"
#include "avs_step32.h"

namespace avs {

// nodes per thread per iteration: 16-byte vector loads along the node index
template <typename T> struct VW { static constexpr int v = 16 / sizeof(T); };

template <typename T, int V>
__device__ __forceinline__ void ldv(const T* __restrict__ p, T* o)
{
    if constexpr (sizeof(T) == 8 && V == 2) {
        const double2 q = *reinterpret_cast<const double2*>(p);
        o[0] = q.x; o[1] = q.y;
    } else {
#pragma unroll
        for (int v = 0; v < V; ++v) o[v] = p[v];
    }
}

// ldv through L2 only (values this block reads once)
template <typename T, int V>
__device__ __forceinline__ void ldv_cg(const T* __restrict__ p, T* o)
{
    if constexpr (sizeof(T) == 8 && V == 2) {
        const double2 q = __ldcg(reinterpret_cast<const double2*>(p));
        o[0] = q.x; o[1] = q.y;
    } else {
#pragma unroll
        for (int v = 0; v < V; ++v) o[v] = __ldcg(p + v);
    }
}

template <typename T, int V>
__device__ __forceinline__ void stv(T* p, const T* o)
{
    if constexpr (sizeof(T) == 8 && V == 2) {
        *reinterpret_cast<double2*>(p) = make_double2(o[0], o[1]);
    } else {
#pragma unroll
        for (int v = 0; v < V; ++v) p[v] = o[v];
    }
}

// N consecutive elements (N * sizeof(T) a multiple of 16 bytes, 16-byte
// aligned) as 16-byte vector loads / stores.
template <typename T, int N>
__device__ __forceinline__ void ldvn(const T* __restrict__ p, T* o)
{
    constexpr int W = 16 / sizeof(T);
#pragma unroll
    for (int j = 0; j < N / W; ++j) ldv<T, W>(p + j * W, o + j * W);
}

template <typename T, int N>
__device__ __forceinline__ void stvn(T* p, const T* o)
{
    constexpr int W = 16 / sizeof(T);
#pragma unroll
    for (int j = 0; j < N / W; ++j) stv<T, W>(p + j * W, o + j * W);
}

// ------------------------------------------------------------------ k_grad
// G[i][a][d][k] = L * (grad phi)_d of array a of cell i at node k.  Each
// thread handles VG consecutive nodes (rows are padded to 32 nodes, so the
// vector stays inside the row) to keep more loads in flight.  NS: face slots
// unrolled (4 when every cell of a 2D mesh has at most 4 faces, else 6).
// NA: arrays per cell (2 or 1 for the monatomic gas, 3 or 2 for the Rykov model).
template <int D, typename T, int VG, int NS, int NA>
__global__ void __launch_bounds__(256) k_grad(int Nv, int Nvp, int limiter, const T* __restrict__ f,
                                              T* __restrict__ G, CellGeo<T> geo)
{
    static_assert((VG * sizeof(T)) % 16 == 0, "whole 16-byte vectors per thread");
    const int i = blockIdx.x;
    const int k0 = (blockIdx.y * blockDim.x + threadIdx.x) * VG;
    if (k0 >= Nv) return;
    const size_t cstride = (size_t)NA * Nvp;
    const int ns = geo.ns[i];
    // slots without a neighbour read the cell itself (difference 0) and have
    // zero weights and offsets, so they add nothing and need no branch
    int nb[NS];
    T cg[NS][D], rr[NS][D];
#pragma unroll
    for (int s = 0; s < NS; ++s) {
        const int n = s < ns ? geo.nbr[i * AVS_MAXS + s] : -1;
        nb[s] = n >= 0 ? n : i;
#pragma unroll
        for (int d = 0; d < D; ++d) {
            cg[s][d] = s < ns ? geo.cg[(size_t)(i * AVS_MAXS + s) * D + d] : T(0);
            rr[s][d] = s < ns ? geo.r[(size_t)(i * AVS_MAXS + s) * D + d] : T(0);
        }
    }
    const T e2 = geo.eps2[i];
#pragma unroll
    for (int a = 0; a < NA; ++a) {
        const T* fa = f + (size_t)a * Nvp + k0;
        T phi[VG], nv[NS][VG];
        ldvn<T, VG>(fa + (size_t)i * cstride, phi);
#pragma unroll
        for (int s = 0; s < NS; ++s) ldvn<T, VG>(fa + (size_t)nb[s] * cstride, nv[s]);
        T* o = G + ((size_t)i * NA + a) * D * Nvp + k0;
        T out[D][VG];
#pragma unroll
        for (int v = 0; v < VG; ++v) {
            T g[D];
#pragma unroll
            for (int d = 0; d < D; ++d) g[d] = T(0);
            T dmax = T(0), dmin = T(0);
#pragma unroll
            for (int s = 0; s < NS; ++s) {
                const T dd = nv[s][v] - phi[v];
#pragma unroll
                for (int d = 0; d < D; ++d) g[d] += cg[s][d] * dd;
                dmax = dd > dmax ? dd : dmax;
                dmin = dd < dmin ? dd : dmin;
            }
            T L = T(1);
            if (limiter == 1) {
                T p = T(0), n = T(0);
#pragma unroll
                for (int s = 0; s < NS; ++s) {
                    T d2 = g[0] * rr[s][0];
#pragma unroll
                    for (int d = 1; d < D; ++d) d2 += g[d] * rr[s][d];
                    p = d2 > p ? d2 : p;
                    n = d2 < n ? d2 : n;
                }
                // epsilon^2 = (K dx)^3 phi_C^2: scaled to the limited value (R6)
                const T e2p = e2 * phi[v] * phi[v];
                if (p > T(0)) { const T t = venkat(dmax, p, e2p); L = t < L ? t : L; }
                if (n < T(0)) { const T t = venkat(dmin, n, e2p); L = t < L ? t : L; }
            }
#pragma unroll
            for (int d = 0; d < D; ++d) out[d][v] = L * g[d];
        }
#pragma unroll
        for (int d = 0; d < D; ++d) stvn<T, VG>(o + (size_t)d * Nvp, out[d]);
    }
}

// The cell's geometry from its record (Geo32): per slot least-squares weights
// and neighbour cell, face offset and face, outward normal and upwind threshold
// as three 16-byte vectors, copied once per block to shared memory.
template <int NS>
__device__ __forceinline__ void load_geo32(const float4* __restrict__ geo, int i, float4* gs)
{
    if (threadIdx.x < 3 * NS) gs[threadIdx.x] = geo[(size_t)i * (3 * AVS_MAXS) + threadIdx.x];
    __syncthreads();
}
template <int D>
__device__ __forceinline__ void vec3(const float4& v, float (&o)[D])
{
    o[0] = v.x;
    o[1] = v.y;
    if constexpr (D == 3) o[2] = v.z;
}

// ------------------------------------------------------------------ k_foot
// Cell-centric reconstruction (Sec. 2.3.3), FP64 form.  Thread block (cell i,
// nodes of one chunk, two per thread and iteration): the limited gradient of
// every array of cell i (as k_grad, kept in registers), then for every face
// slot s of the cell the foot values
//   phi_bar = phi_i + (L grad phi)_i . (x_f - x_i - xi h)
//           = phi_i - h L (g . xi) + L (g . r_s)
// at the nodes where i is that face's upwind cell (xi . An >= 0 for the face's
// L cell, < 0 for its R cell; xi . An summed without contraction, the same
// value the face kernel tests), written to the face's row of
// FB [face][array][Nvp].  Every node of an interior face is written exactly
// once, by its upwind cell; of a boundary face only the outgoing half.  The
// gradient itself is never stored.
//
// The FP64 pipe is the bound (one warp instruction in 16 cycles of an SM, 1/32
// of the integer and FP32 rates), so what need not run on it does not: the
// extremes compare bit patterns as integers, the upwind choice is an FP32 dot
// product unless that lies within its rounding bound of zero, and g . r_s
// serves the limiter and the foot value.  160 -> about 90 FP64 instructions
// per cell and node in 3D; per step 181 -> 99 us on the 32 x 32 cavity (298
// nodes), 4.30 -> 2.24 ms on 1000 cells x 13824 nodes in 3D, where the pipe is
// full.
// Largest value of v[0..N-1] and 0, and smallest of them and 0, by integer
// comparison: as signed integers the positive doubles order as their values
// and negative ones lie below zero; as unsigned integers the negative ones
// order by magnitude, above every positive one.
template <int N>
__device__ __forceinline__ void ext_bits(const double* v, double& mx, double& mn)
{
    long long hi = 0;
    unsigned long long lo = 0;
#pragma unroll
    for (int s = 0; s < N; ++s) {
        const long long b = __double_as_longlong(v[s]);
        hi = b > hi ? b : hi;
        lo = (unsigned long long)b > lo ? (unsigned long long)b : lo;
    }
    mx = __longlong_as_double(hi);
    mn = (long long)lo < 0 ? __longlong_as_double((long long)lo) : 0.0;
}

template <int D, int NS, int NA>
__global__ void __launch_bounds__(128) k_foot(int Nv, int Nvp, int chunk, int limiter, double h,
                                              const double* __restrict__ f, double* __restrict__ FB,
                                              CellGeo<double> geo, const double* __restrict__ An, const double* __restrict__ xi,
                                              const float4* __restrict__ geo32, const float* __restrict__ xs,
                                              size_t xstride)
{
    constexpr int VG = 2;
    __shared__ double sc[NS][D], sr[NS][D];      // least-squares weights, face offsets
    __shared__ float4 g32[3 * NS];               // FP32 record: neighbours, faces, outward normals
    const int i = blockIdx.x;
    for (int e = threadIdx.x; e < NS * D; e += blockDim.x) {
        const int q = e / D, d = e % D;
        const bool on = q < geo.ns[i];
        sc[q][d] = on ? geo.cg[(size_t)(i * AVS_MAXS + q) * D + d] : 0.0;
        sr[q][d] = on ? geo.r[(size_t)(i * AVS_MAXS + q) * D + d] : 0.0;
    }
    load_geo32<NS>(geo32, i, g32);
    const size_t cstride = (size_t)NA * Nvp;
    const double e2 = geo.eps2[i];
    const int kend = min(Nv, (int)(blockIdx.y + 1) * chunk);
#pragma unroll 1
    for (int k0 = blockIdx.y * chunk + threadIdx.x * VG; k0 < kend; k0 += blockDim.x * VG) {
        double phi[NA][VG], L[NA][VG], dr[NA][VG][NS], A[NA][VG], x[VG][D];
        ldvn<double, VG * D>(xi + (size_t)k0 * D, &x[0][0]);
#pragma unroll
        for (int a = 0; a < NA; ++a) {
            const double* fa = f + (size_t)a * Nvp + k0;
            double nv[NS][VG];
            ldvn<double, VG>(fa + (size_t)i * cstride, phi[a]);
#pragma unroll
            for (int q = 0; q < NS; ++q)
                ldvn<double, VG>(fa + (size_t)__float_as_int(g32[3 * q].w) * cstride, nv[q]);
#pragma unroll
            for (int v = 0; v < VG; ++v) {
                double g[D], dd[NS];
#pragma unroll
                for (int d = 0; d < D; ++d) g[d] = 0.0;
#pragma unroll
                for (int q = 0; q < NS; ++q) {
                    dd[q] = nv[q][v] - phi[a][v];
#pragma unroll
                    for (int d = 0; d < D; ++d) g[d] += sc[q][d] * dd[q];
                }
#pragma unroll
                for (int q = 0; q < NS; ++q) {
                    dr[a][v][q] = g[0] * sr[q][0];
#pragma unroll
                    for (int d = 1; d < D; ++d) dr[a][v][q] += g[d] * sr[q][d];
                }
                double l = limiter == 0 ? 0.0 : 1.0;       // first order: phi_bar = phi_C
                if (limiter == 1) {
                    // extremes of the neighbour differences and of the face
                    // projections g . r_s (both include 0: the cell itself)
                    double dmax, dmin, p, n;
                    ext_bits<NS>(dd, dmax, dmin);
                    ext_bits<NS>(dr[a][v], p, n);
                    // epsilon^2 = (K dx)^3 phi_C^2: scaled to the limited value (R6)
                    const double e2p = e2 * phi[a][v] * phi[a][v];
                    // the ratios are >= 0 or NaN (0/0), whose bits are above those of 1
                    unsigned long long b = (unsigned long long)__double_as_longlong(1.0);
                    if (__double_as_longlong(p) > 0) {
                        const unsigned long long t = (unsigned long long)__double_as_longlong(venkat_ratio(dmax, p, e2p));
                        b = t < b ? t : b;
                    }
                    if (__double_as_longlong(n) < 0) {
                        const unsigned long long t = (unsigned long long)__double_as_longlong(venkat_ratio(dmin, n, e2p));
                        b = t < b ? t : b;
                    }
                    l = __longlong_as_double((long long)b);
                }
                double gx = g[0] * x[v][0];
#pragma unroll
                for (int d = 1; d < D; ++d) gx += g[d] * x[v][d];
                L[a][v] = l;
                A[a][v] = phi[a][v] - (h * l) * gx;
            }
        }
        float2 x32[D];
#pragma unroll
        for (int d = 0; d < D; ++d) x32[d] = *reinterpret_cast<const float2*>(xs + d * xstride + k0);
#pragma unroll
        for (int q = 0; q < NS; ++q) {
            const int fc = __float_as_int(g32[3 * q + 1].w);
            if (fc < 0) break;                   // no further faces
            const float4 n4 = g32[3 * q + 2];
            const float na[3] = {n4.x, n4.y, n4.z};
            bool up[VG];
#pragma unroll
            for (int v = 0; v < VG; ++v) {
                float xv[D], sn = 0.0f;
#pragma unroll
                for (int d = 0; d < D; ++d) {
                    xv[d] = v ? x32[d].y : x32[d].x;
                    sn = fmaf(xv[d], na[d], sn);
                }
                if (upwind_sure<D>(xv, na, sn)) up[v] = sn > 0.0f;
                else if (upwind_zero<D>(xv, na)) up[v] = n4.w == 0.0f;
                else up[v] = upwind_exact<D>(x[v], An + (size_t)fc * D, n4.w != 0.0f);
            }
            if (!up[0] && !up[1]) continue;
            double* row = FB + (size_t)fc * NA * Nvp + k0;
#pragma unroll
            for (int a = 0; a < NA; ++a) {
                double o[VG];
#pragma unroll
                for (int v = 0; v < VG; ++v) o[v] = A[a][v] + L[a][v] * dr[a][v][q];
                if (up[0] && up[1]) {
                    stvn<double, VG>(row + (size_t)a * Nvp, o);
                } else {
#pragma unroll
                    for (int v = 0; v < VG; ++v)
                        if (up[v]) row[(size_t)a * Nvp + v] = o[v];
                }
            }
        }
    }
}

// The FP32 form of the reconstruction, in packed two-lane arithmetic: four nodes
// per thread as two pairs.  Each lane rounds as the scalar operation would; the
// upwind choice is the sign of the FP32 xi . An, the same for both cells of a face
// (or, EXACT, the FP64 one), and both sides of the limiter are evaluated always.
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return fma2(b, bc2(-1.0f), a); }   // a - b, one rounding

template <int NS>
__device__ __forceinline__ void ext4(const float* v, float& mx, float& mn)
{
    if constexpr (NS == 6) {
        mx = max3f(max3f(v[0], v[1], v[2]), max3f(v[3], v[4], v[5]), 0.0f);
        mn = min3f(min3f(v[0], v[1], v[2]), min3f(v[3], v[4], v[5]), 0.0f);
    } else if constexpr (NS == 4) {
        mx = max3f(max3f(v[0], v[1], v[2]), v[3], 0.0f);
        mn = min3f(min3f(v[0], v[1], v[2]), v[3], 0.0f);
    } else {
        mx = mn = 0.0f;
#pragma unroll
        for (int s = 0; s < NS; ++s) {
            mx = fmaxf(mx, v[s]);
            mn = fminf(mn, v[s]);
        }
    }
}

// Venkatakrishnan ratio of venkat() in two lanes, uncapped: (d1^2 + eps2 +
// 2 d1 d2) / (d1^2 + 2 d2^2 + d1 d2 + eps2).  All terms are >= 0 (d1 and d2 have
// one sign).  The division (a reciprocal and a product, like fdiv) keeps
// subnormal denominators, so the ratio holds down to |f| of about 1e-20 and with
// fewer bits to 1e-22, where the squares vanish and limit2 takes 1; it holds up to
// 9e18.  (A reciprocal that flushes them, off from 1e-19 down, would save 0.8 % of
// a step on the cylinder, 12288 cells x 3522 nodes: 8.35 against 8.42 ms for ten.)
__device__ __forceinline__ float2 venkat2(float2 d1, float2 d2, float2 eps2)
{
    const float2 u = fma2(d1, d1, eps2), v = mul2(d1, d2);
    const float2 num = fma2(bc2(2.0f), v, u);
    const float2 den = fma2(mul2(bc2(2.0f), d2), d2, add2(u, v));
    return make_float2(__fdividef(num.x, den.x), __fdividef(num.y, den.y));
}

// Limiter of a node pair: the smaller of the two sides' ratios, capped at 1.
// A side without a projection (pp = 0 or nn = 0) has equal numerator and
// denominator, so it needs no test; NaN (0/0 in the tails) loses to 1 in the
// three-input minimum.  Against a compare and two selects per side and lane
// this takes one instruction per lane of the ALU pipe, the kernel's busiest.
__device__ __forceinline__ float2 limit2(float2 dmax, float2 dmin, float2 pp, float2 nn, float2 eps2)
{
    const float2 tp = venkat2(dmax, pp, eps2), tn = venkat2(dmin, nn, eps2);
    return make_float2(min3f(tp.x, tn.x, 1.0f), min3f(tp.y, tn.y, 1.0f));
}

// Thread block (cell i, nodes of one chunk), the thread's quads one after the
// other: the block's start (launch, geometry, barrier) is paid once for them.
// Bounded by the latency of the rows' loads at the warps that the registers
// allow: all rows of a quad are loaded before its arithmetic (12288 cells x 3522
// nodes, 2D: array by array 294 us, all at once 270; Rykov, 3216 nodes, 476 and
// 398), seven blocks of 128 threads per SM in 2D, 18 of 64 in 3D; rings of
// copies in shared memory as in the face kernel leave too few warps (311 us).
// EXACT: the upwind choice is the FP64 one; only a quad with a normal velocity
// within one bound of zero recomputes it (a bound per node cost the Rykov
// cylinder 90 us more).
// Warps per SM, by arrays and face slots: the most of 16, 20, 24, 28, 32 and 36 at
// which ptxas spills at most 24 bytes a thread.  One step further it spills 48 (2D,
// two arrays, four slots), 120 (six slots), 100 and 128 (three arrays) and 112 bytes
// (3D, two arrays).  2D, two arrays, four slots: 20 warps 322 us, 24 292, 28 270, 36
// 369, 40 475.
constexpr int foot_warps(int D, int NS, int NA)
{
    if (D == 3) return NA == 1 ? 36 : 16;
    if (NS == 4) return NA == 2 ? 28 : 24;
    return NA == 2 ? 20 : 16;
}
template <int D, int NS, int NA, bool EXACT>
__global__ void __launch_bounds__(D == 3 ? 64 : 128, foot_warps(D, NS, NA) / (D == 3 ? 2 : 4)) k_foot_f2(int Nv, int Nvp, int chunk, int limiter, float h,
                                                    const float* __restrict__ f, float* __restrict__ FB,
                                                    const float4* __restrict__ geo, const float* __restrict__ eps2,
                                                    const float* __restrict__ xs, size_t xstride,
                                                    const double* __restrict__ xi, const double* __restrict__ An)
{
    constexpr int VG = 4;
    __shared__ float4 gs[3 * NS];
    const int i = blockIdx.x;
    load_geo32<NS>(geo, i, gs);
    const size_t cstride = (size_t)NA * Nvp;
    const float e2 = eps2[i];
    const int kend = min(Nv, (int)(blockIdx.y + 1) * chunk);
#pragma unroll 1
    for (int k0 = blockIdx.y * chunk + threadIdx.x * VG; k0 < kend; k0 += blockDim.x * VG) {
        float2 phi[NA][2], G[NA][D][2];
        float4 n4a[NA][NS];
        float4 c4a[NA];
#pragma unroll
        for (int a = 0; a < NA; ++a) {
            const float* fa = f + (size_t)a * Nvp + k0;
            c4a[a] = __ldg(reinterpret_cast<const float4*>(fa + (size_t)i * cstride));
#pragma unroll
            for (int s = 0; s < NS; ++s) n4a[a][s] = __ldg(reinterpret_cast<const float4*>(fa + (size_t)__float_as_int(gs[3 * s].w) * cstride));
        }
#pragma unroll
        for (int a = 0; a < NA; ++a) {
            phi[a][0] = lo2(c4a[a]);
            phi[a][1] = hi2(c4a[a]);
            float4* n4 = n4a[a];
#pragma unroll
            for (int p = 0; p < 2; ++p) {
                float2 g[D], dd[NS];
#pragma unroll
                for (int d = 0; d < D; ++d) g[d] = bc2(0.0f);
#pragma unroll
                for (int s = 0; s < NS; ++s) {
                    float cg[D];
                    vec3<D>(gs[3 * s], cg);
                    dd[s] = sub2(p ? hi2(n4[s]) : lo2(n4[s]), phi[a][p]);
#pragma unroll
                    for (int d = 0; d < D; ++d) g[d] = fma2(bc2(cg[d]), dd[s], g[d]);
                }
                float2 L = bc2(1.0f);
                if (limiter == 1) {
                    float2 d2[NS];
#pragma unroll
                    for (int s = 0; s < NS; ++s) {
                        float rr[D];
                        vec3<D>(gs[3 * s + 1], rr);
                        d2[s] = mul2(g[0], bc2(rr[0]));
#pragma unroll
                        for (int d = 1; d < D; ++d) d2[s] = fma2(g[d], bc2(rr[d]), d2[s]);
                    }
                    float dx[NS], dy[NS], ex[NS], ey[NS];
#pragma unroll
                    for (int s = 0; s < NS; ++s) {
                        dx[s] = dd[s].x; dy[s] = dd[s].y;
                        ex[s] = d2[s].x; ey[s] = d2[s].y;
                    }
                    float2 dmax, dmin, pp, nn;
                    ext4<NS>(dx, dmax.x, dmin.x);
                    ext4<NS>(dy, dmax.y, dmin.y);
                    ext4<NS>(ex, pp.x, nn.x);
                    ext4<NS>(ey, pp.y, nn.y);
                    // epsilon^2 = (K dx)^3 phi_C^2: scaled to the limited value (R6)
                    const float2 e2p = mul2(mul2(bc2(e2), phi[a][p]), phi[a][p]);
                    L = limit2(dmax, dmin, pp, nn, e2p);
                }
                if (limiter == 0) L = bc2(0.0f);     // first order: phi_bar = phi_C
#pragma unroll
                for (int d = 0; d < D; ++d) G[a][d][p] = mul2(L, g[d]);
            }
        }
        // node coordinates of the thread's nodes, as lane pairs
        float2 X[2][D];
#pragma unroll
        for (int d = 0; d < D; ++d) {
            const float4 v = __ldg(reinterpret_cast<const float4*>(xs + d * xstride + k0));
            X[0][d] = lo2(v);
            X[1][d] = hi2(v);
        }
        float xmax = 0.0f;
        if constexpr (EXACT) {
#pragma unroll
            for (int p = 0; p < 2; ++p)
#pragma unroll
                for (int d = 0; d < D; ++d) xmax = max3f(xmax, fabsf(X[p][d].x), fabsf(X[p][d].y));
        }
        // phi_bar = A + G . r_s with A = phi - h G . xi, the part common to the faces
        float2 A[NA][2];
#pragma unroll
        for (int a = 0; a < NA; ++a)
#pragma unroll
            for (int p = 0; p < 2; ++p) {
                float2 gx = mul2(G[a][0][p], X[p][0]);
#pragma unroll
                for (int d = 1; d < D; ++d) gx = fma2(G[a][d][p], X[p][d], gx);
                A[a][p] = fma2(bc2(-h), gx, phi[a][p]);
            }
#pragma unroll
        for (int s = 0; s < NS; ++s) {
            const float4 r4 = gs[3 * s + 1], an = gs[3 * s + 2];
            const int fc = __float_as_int(r4.w);
            if (fc < 0) break;                       // no further faces
            float rr[D];
            vec3<D>(r4, rr);
            bool up[4];
            float near = INFINITY;
#pragma unroll
            for (int p = 0; p < 2; ++p) {
                // xi . An as in k_foot: a product, then fused multiply-adds; the
                // normal points out of the cell (an exact sign change), so the
                // face's L cell is upwind at >= 0 and its R cell at > 0, that is,
                // at or above the smallest subnormal (an.w)
                float2 sn = fma2(X[p][1], bc2(an.y), mul2(X[p][0], bc2(an.x)));
                if constexpr (D == 3) sn = fma2(X[p][2], bc2(an.z), sn);
                up[2 * p] = sn.x >= an.w;
                up[2 * p + 1] = sn.y >= an.w;
                if constexpr (EXACT) near = min3f(near, fabsf(sn.x), fabsf(sn.y));
            }
            if constexpr (EXACT) {
                // one bound for the quad: 2^-20 max |xi| sum |An_d| is above every node's in upwind_sure
                float na = fabsf(an.x) + fabsf(an.y);
                if constexpr (D == 3) na += fabsf(an.z);
                if (!(near > fmaf(xmax * 0x1p-20f, na, 0x1p-100f))) {
#pragma unroll
                    for (int z = 0; z < 4; ++z) {
                        float xz[D], nz[D], sn = 0.0f;
                        vec3<D>(an, nz);
#pragma unroll
                        for (int d = 0; d < D; ++d) {
                            xz[d] = z & 1 ? X[z >> 1][d].y : X[z >> 1][d].x;
                            sn = d == 0 ? xz[0] * nz[0] : fmaf(xz[d], nz[d], sn);
                        }
                        if (!upwind_sure<D>(xz, nz, sn) && !upwind_zero<D>(xz, nz) && k0 + z < Nv)
                            up[z] = upwind_exact<D>(xi + (size_t)(k0 + z) * D, An + (size_t)fc * D, an.w != 0.0f);
                    }
                }
            }
            const bool all = up[0] && up[1] && up[2] && up[3];
            const bool any = up[0] || up[1] || up[2] || up[3];
            if (!any) continue;
            float* row = FB + (size_t)fc * NA * Nvp + k0;
#pragma unroll
            for (int a = 0; a < NA; ++a) {
                float2 o[2];
#pragma unroll
                for (int p = 0; p < 2; ++p) {
                    float2 val = A[a][p];
#pragma unroll
                    for (int d = 0; d < D; ++d) val = fma2(G[a][d][p], bc2(rr[d]), val);
                    o[p] = val;
                }
                float* ra = row + (size_t)a * Nvp;
                if (all) {
                    *reinterpret_cast<float4*>(ra) = make_float4(o[0].x, o[0].y, o[1].x, o[1].y);
                } else {
                    if (up[0]) ra[0] = o[0].x;
                    if (up[1]) ra[1] = o[0].y;
                    if (up[2]) ra[2] = o[1].x;
                    if (up[3]) ra[3] = o[1].y;
                }
            }
        }
    }
}

template <typename A>
__device__ __forceinline__ A tau_vhs(A rho, A RT, A R, A mu_ref, A T_ref, A omega)
{
    const A T = fdiv(RT, R);
    return fdiv(mu_ref * powa(fdiv(T, T_ref), omega), rho * RT);
}

template <int D, int V, typename T, typename PP>
__device__ __forceinline__ void load_nodes(const PP& P, int k0, T (*x)[D], T* w)
{
    T xx[V * D];
    if constexpr ((V * D * sizeof(T)) % 16 == 0) {
        constexpr int PER = 16 / sizeof(T);
#pragma unroll
        for (int j = 0; j < V * D / PER; ++j) ldv<T, PER>(P.xi + (size_t)k0 * D + j * PER, xx + j * PER);
    } else {
#pragma unroll
        for (int j = 0; j < V * D; ++j) xx[j] = P.xi[(size_t)k0 * D + j];
    }
#pragma unroll
    for (int v = 0; v < V; ++v)
#pragma unroll
        for (int d = 0; d < D; ++d) x[v][d] = xx[v * D + d];
    ldv<T, V>(P.w + k0, w);
}

// ------------------------------------------------------------------ k_face
template <int D>
struct FaceP {
    int Nv, Nvp;
    size_t cstride;          // elements per cell in f: NA * Nvp
    double hd;
    double R, Pr, omega, mu_ref, T_ref;
    double* FB;                     // [face][array][Nvp]: foot values phi_bar (k_foot) in,
                               // per-node flux (xi . An) phi_ij out (pass B overwrites in place)
    double* __restrict__ AF;   // [face][D+2] area-weighted flux of W
    const double* __restrict__ Win;
    const double* __restrict__ xi;
    const double* __restrict__ w;
    const int* __restrict__ order;
    const int* __restrict__ faceL;
    const int* __restrict__ faceR;
    const double* __restrict__ An;
    const double* __restrict__ bc;
    int* err;
};

struct FaceSt {
    int kind, L, R;          // kind: 0 interior, 1 wall, 2 far field
    double An[3];
    double V[3];             // reference velocity of the moment sums
    EqPar<double> eq;             // interface equilibrium / incoming Maxwellian
    double wa, wb;
};

// The face stage in pieces.  One face, nodes [kb, ke) (thread t of NT owns
// nodes k = kb + tV.., kb + tV + NT V.., V = 2 nodes per iteration):
//   face_setup   (one thread) cells, geometry, reference velocity V of the
//                moment sums (mean of the two cells' velocities), and for a
//                boundary face the incoming Maxwellian (unit density at a wall);
//   face_pass_a  interior: raw moments about V of the foot distribution
//                phi_bar (upwind cell by the sign of xi . An), the foot values
//                kept in shared memory when CACHE; boundary: flux moments of
//                the outgoing foot values and of the incoming Maxwellian;
//   face_state   (one thread, from the summed pass-A moments) the interface
//                state: tau (Eq. 3), q_ij (R4), Shakhov parameters, weights
//                tau/(tau+h), h/(tau+h) (Eq. equ28); wall density from zero
//                net mass flux (R8) and the boundary face's A F;
//   face_pass_b  interior: phi_ij = wa phi_bar + wb g_ij per node, its flux
//                (xi . An) phi_ij and the flux moments
//                sum_k w (xi . An) psi phi_ij; boundary: outgoing foot value /
//                incoming Maxwellian.
// k_face runs them all in one block per face.
template <int D>
__device__ __forceinline__ void face_setup(const FaceP<D>& P, int f, FaceSt& S)
{
    constexpr int NW = D + 2;
    S.L = P.faceL[f];
    S.R = P.faceR[f];
    S.kind = S.R >= 0 ? 0 : (int)P.bc[(size_t)(-1 - S.R) * 6];
    for (int d = 0; d < 3; ++d) {
        S.An[d] = d < D ? P.An[(size_t)f * D + d] : 0.0;
        double v = 0.0;
        if (d < D) {
            v = P.Win[(size_t)S.L * NW + 1 + d] / P.Win[(size_t)S.L * NW];
            if (S.R >= 0) v = 0.5 * (v + P.Win[(size_t)S.R * NW + 1 + d] / P.Win[(size_t)S.R * NW]);
        }
        S.V[d] = v;
    }
    if (S.kind != 0) {
        const double* B = P.bc + (size_t)(-1 - S.R) * 6;
        const double Ub[3] = {B[2], B[3], B[4]};
        S.eq = make_eq<D, double>(S.kind == 1 ? 1.0 : B[1], Ub, P.R * B[5], nullptr, P.Pr);
    }
}

// number of pass-A sums per face: NM raw moments (interior) or 2 (D+2) flux
// moments (boundary: outgoing, incoming)
template <int D>
struct FaceNR {
    static constexpr int NM = NMom<D>::v, NW = D + 2;
    static constexpr int v = (NM > 2 * NW) ? NM : 2 * NW;
};

template <int D, int NT, bool CACHE, int V>
__device__ __forceinline__ void face_pass_a(const FaceP<D>& P, const FaceSt& S, double* fc, int kb, int ke,
                                            double* acc, int tid, int f)
{
    constexpr int NA = NArr<D>::v, NW = D + 2;
    constexpr int NR = FaceNR<D>::v;
    const bool inter = S.kind == 0;
    double An[D], Vt[D];
#pragma unroll
    for (int d = 0; d < D; ++d) {
        An[d] = S.An[d];
        Vt[d] = S.V[d];
    }
    const int Nvp = P.Nvp;
    const double* fb = P.FB + (size_t)f * NA * Nvp;          // the face's foot values
#pragma unroll
    for (int m = 0; m < NR; ++m) acc[m] = 0.0;
    if (inter) {
#pragma unroll 2
        for (int k0 = kb + tid * V; k0 < ke; k0 += NT * V) {
            double x[V][D], wv[V];
            load_nodes<D, V>(P, k0, x, wv);      // pad nodes carry w = 0 and contribute nothing
            double fv[NA][V];
#pragma unroll
            for (int a = 0; a < NA; ++a) {
                ldv<double, V>(fb + (size_t)a * Nvp + k0, fv[a]);
                if constexpr (CACHE) stv<double, V>(fc + a * Nvp + k0, fv[a]);
            }
#pragma unroll
            for (int v = 0; v < V; ++v) {
                double xs[D];
#pragma unroll
                for (int d = 0; d < D; ++d) xs[d] = x[v][d] - Vt[d];
                raw_acc<D>(acc, xs, wv[v] * fv[0][v], NA == 2 ? wv[v] * fv[NA - 1][v] : 0.0);
            }
        }
    } else {
#pragma unroll 2
        for (int k0 = kb + tid * V; k0 < ke; k0 += NT * V) {
            double x[V][D], wv[V], sn[V];
            load_nodes<D, V>(P, k0, x, wv);
            double fv[NA][V];
#pragma unroll
            for (int a = 0; a < NA; ++a) ldv<double, V>(fb + (size_t)a * Nvp + k0, fv[a]);
#pragma unroll
            for (int v = 0; v < V; ++v) {
                sn[v] = dot_rn<D>(x[v], An);
                const bool out = sn[v] >= 0.0;
                double g0 = fv[0][v], g1 = NA == 2 ? fv[NA - 1][v] : 0.0;
                if (!out) eq_eval<D>(S.eq, x[v], g0, g1);
                const double t = wv[v] * sn[v];
                double x2 = 0.0;
#pragma unroll
                for (int d = 0; d < D; ++d) x2 += x[v][d] * x[v][d];
                double mm[NW];
                mm[0] = t * g0;
#pragma unroll
                for (int d = 0; d < D; ++d) mm[1 + d] = t * g0 * x[v][d];
                mm[D + 1] = t * 0.5 * (x2 * g0 + g1);
#pragma unroll
                for (int c = 0; c < NW; ++c) {
                    acc[c] += out ? mm[c] : 0.0;
                    acc[NW + c] += out ? 0.0 : mm[c];
                }
            }
        }
    }
}

// Interface state from the summed pass-A moments red[]; writes S.eq, S.wa,
// S.wb and, for a boundary face, its area-weighted flux AF[0..D+1].
template <int D>
__device__ __forceinline__ void face_state(const FaceP<D>& P, FaceSt& S, const double* red, double* AF)
{
    constexpr int NW = D + 2;
    if (S.kind == 0) {
        double rho, U[3], RT, qb[3];
        state_from_raw<D, double>(red, S.V, rho, U, RT, qb);
        if (!(rho > 0.0) || !(RT > 0.0)) atomicOr(P.err, 1);
        const double tau = tau_vhs<double>(rho, RT, P.R, P.mu_ref, P.T_ref, P.omega);
        const double hh = P.hd;
        double qf[3] = {0.0, 0.0, 0.0};
        const double qs = fdiv(tau, tau + hh * P.Pr);
        for (int d = 0; d < D; ++d) qf[d] = qs * qb[d];
        S.eq = make_eq_a<D, double, double>(rho, U, RT, qf, P.Pr);
        S.wa = fdiv(tau, tau + hh);
        S.wb = fdiv(hh, tau + hh);
    } else if (S.kind == 1) {
        const double Sin = -red[NW];          // incoming mass flux of the unit-density wall Maxwellian
        const double rw = Sin > 0.0 ? red[0] / Sin : 0.0;
        for (int m = 0; m < NW; ++m) AF[m] = red[m] + rw * red[NW + m];
        const double* B = P.bc + (size_t)(-1 - S.R) * 6;
        const double Ub[3] = {B[2], B[3], B[4]};
        S.eq = make_eq<D, double>(rw, Ub, P.R * B[5], nullptr, P.Pr);
    } else {
        for (int m = 0; m < NW; ++m) AF[m] = red[m] + red[NW + m];
    }
}

// Pass B over nodes [kb, ke): writes the per-node flux over the face's foot
// values in FB (in place) and, for an interior face, returns the per-thread
// flux-moment partial sums in acc[D+2] (element type).
template <int D, int NT, bool CACHE, int V>
__device__ __forceinline__ void face_pass_b(const FaceP<D>& P, const FaceSt& S, const double* fc, int kb, int ke,
                                            double* acc, int tid, int f)
{
    constexpr int NA = NArr<D>::v, NW = D + 2;
    const bool inter = S.kind == 0;
    double An[D];
#pragma unroll
    for (int d = 0; d < D; ++d) An[d] = S.An[d];
    const int Nvp = P.Nvp;
    double* Fo = P.FB + (size_t)f * NA * Nvp;                // foot values in, flux out
#pragma unroll
    for (int m = 0; m < NW; ++m) acc[m] = 0.0;
    if (inter) {
        const double wa = S.wa, wb = S.wb;
#pragma unroll 2
        for (int k0 = kb + tid * V; k0 < ke; k0 += NT * V) {
            double x[V][D], wv[V], sn[V];
            load_nodes<D, V>(P, k0, x, wv);
#pragma unroll
            for (int v = 0; v < V; ++v) sn[v] = dot_rn<D>(x[v], An);
            double fv[NA][V];
#pragma unroll
            for (int a = 0; a < NA; ++a) {
                if constexpr (CACHE) ldv<double, V>(fc + a * Nvp + k0, fv[a]);
                else ldv<double, V>(Fo + (size_t)a * Nvp + k0, fv[a]);
            }
            double o[NA][V];
#pragma unroll
            for (int v = 0; v < V; ++v) {
                double gG, gH;
                eq_eval<D>(S.eq, x[v], gG, gH);
                const double pG = wa * fv[0][v] + wb * gG;
                const double pH = NA == 2 ? wa * fv[NA - 1][v] + wb * gH : 0.0;
                const double t = wv[v] * sn[v];
                double x2 = 0.0;
#pragma unroll
                for (int d = 0; d < D; ++d) x2 += x[v][d] * x[v][d];
                acc[0] += t * pG;
#pragma unroll
                for (int d = 0; d < D; ++d) acc[1 + d] += t * pG * x[v][d];
                acc[D + 1] += t * 0.5 * (x2 * pG + pH);
                o[0][v] = sn[v] * pG;
                if (NA == 2) o[NA - 1][v] = sn[v] * pH;
            }
#pragma unroll
            for (int a = 0; a < NA; ++a) stv<double, V>(Fo + (size_t)a * Nvp + k0, o[a]);
        }
    } else {
#pragma unroll 2
        for (int k0 = kb + tid * V; k0 < ke; k0 += NT * V) {
            double x[V][D], wv[V], sn[V];
            load_nodes<D, V>(P, k0, x, wv);
            double fv[NA][V];
#pragma unroll
            for (int a = 0; a < NA; ++a) ldv<double, V>(Fo + (size_t)a * Nvp + k0, fv[a]);
            double o[NA][V];
#pragma unroll
            for (int v = 0; v < V; ++v) {
                sn[v] = dot_rn<D>(x[v], An);
                double g0 = fv[0][v], g1 = NA == 2 ? fv[NA - 1][v] : 0.0;
                if (sn[v] < 0.0) eq_eval<D>(S.eq, x[v], g0, g1);
                o[0][v] = sn[v] * g0;
                if (NA == 2) o[NA - 1][v] = sn[v] * g1;
            }
#pragma unroll
            for (int a = 0; a < NA; ++a) stv<double, V>(Fo + (size_t)a * Nvp + k0, o[a]);
        }
    }
}

// One block per face, all nodes: setup, pass A, state, pass B.
template <int D, int NT, bool CACHE, int VF>
__global__ void __launch_bounds__(NT, 4) k_face(FaceP<D> P)
{
    constexpr int NW = D + 2;
    constexpr int NR = FaceNR<D>::v;
    __shared__ FaceSt S;
    __shared__ double sw[(NT / 32) * NR];
    __shared__ double red[NR];
    extern __shared__ __align__(16) unsigned char face_dsm[];
    double* fc = reinterpret_cast<double*>(face_dsm);     // [array][Nvp] foot values (CACHE)

    const int tid = threadIdx.x;
    const int f = P.order[blockIdx.x];
    if (tid == 0) face_setup<D>(P, f, S);
    __syncthreads();
    {
        double acc[NR];
        face_pass_a<D, NT, CACHE, VF>(P, S, fc, 0, P.Nv, acc, tid, f);
        block_sum_t<NR, NT>(acc, sw, red);
    }
    if (tid == 0) face_state<D>(P, S, red, P.AF + (size_t)f * NW);
    __syncthreads();
    double acc[NW];
    face_pass_b<D, NT, CACHE, VF>(P, S, fc, 0, P.Nv, acc, tid, f);
    if (S.kind == 0) {
        block_sum_t<NW, NT>(acc, sw, red);
        if (tid < NW) P.AF[(size_t)f * NW + tid] = red[tid];
    }
}

// ------------------------------------------------------------------ k_face_tab
// The FP64 face kernel where the tree's nodes have few different coordinates
// per axis.  A Maxwellian is a product over the axes, so pass B takes the
// interface equilibrium, xi . An and |c|^2 from tables of the axes' values, one
// entry per coordinate (xtab, at most half as many as nodes), built by the
// block once the face's state is known: an exponential and 16 further FP64
// operations per node become three products and four sums.  FP64 instructions
// per face and node 80 -> 48 (3D); per step 202 -> 128 us on the 32 x 32 cavity
// (298 nodes), 5.46 -> 3.46 ms on 1000 cells x 13824 nodes in 3D.
struct AxisEq {
    double E, c2, ca, xa;    // exp(-c^2 / 2RT) (axis 0: times wb pref), c^2, c alpha, xi An
};

template <int D, int NT>
__global__ void __launch_bounds__(NT) k_face_tab(FaceP<D> P, const double* __restrict__ xtab,
                                                 const unsigned short* __restrict__ tix, size_t xstride, int n0,
                                                 int n1, int nt)
{
    constexpr int NA = NArr<D>::v, NW = D + 2;
    constexpr int NR = FaceNR<D>::v;
    extern __shared__ __align__(16) unsigned char tab_dsm[];
    AxisEq* tab = reinterpret_cast<AxisEq*>(tab_dsm);
    __shared__ FaceSt S;
    __shared__ double sw[(NT / 32) * NR];
    __shared__ double red[NR];
    const int tid = threadIdx.x;
    const int f = P.order[blockIdx.x];
    if (tid == 0) face_setup<D>(P, f, S);
    __syncthreads();
    {
        double acc[NR];
        face_pass_a<D, NT, false, 2>(P, S, nullptr, 0, P.Nv, acc, tid, f);
        block_sum_t<NR, NT>(acc, sw, red);
    }
    if (tid == 0) face_state<D>(P, S, red, P.AF + (size_t)f * NW);
    __syncthreads();
    double acc[NW];
    if (S.kind != 0) {
        face_pass_b<D, NT, false, 2>(P, S, nullptr, 0, P.Nv, acc, tid, f);
        return;
    }
    for (int e = tid; e < nt; e += NT) {
        const int d = e < n0 ? 0 : e < n1 ? 1 : 2;
        const double x = xtab[e], c = x - S.eq.U[d], c2 = c * c;
        AxisEq q;
        q.E = ex(-c2 * S.eq.inv2RT);
        if (d == 0) q.E *= S.wb * S.eq.pref;
        q.c2 = c2;
        q.ca = c * S.eq.alpha[d];
        q.xa = dmul(x, S.An[d]);
        tab[e] = q;
    }
    __syncthreads();
    const double wa = S.wa, irt = S.eq.invRT, RTH = S.eq.RTH;
    const int Nvp = P.Nvp;
    double* Fo = P.FB + (size_t)f * NA * Nvp;            // foot values in, flux out
#pragma unroll
    for (int m = 0; m < NW; ++m) acc[m] = 0.0;
    for (int k0 = tid * 2; k0 < P.Nv; k0 += NT * 2) {
        double x[2][D], wv[2], fv[NA][2], o[NA][2];
        load_nodes<D, 2>(P, k0, x, wv);
        ushort2 ix[D];
#pragma unroll
        for (int d = 0; d < D; ++d) ix[d] = *reinterpret_cast<const ushort2*>(tix + d * xstride + k0);
#pragma unroll
        for (int a = 0; a < NA; ++a) ldv<double, 2>(Fo + (size_t)a * Nvp + k0, fv[a]);
#pragma unroll
        for (int v = 0; v < 2; ++v) {
            const AxisEq* q0 = tab + (v ? ix[0].y : ix[0].x);
            double E = q0->E, c2 = q0->c2, ca = q0->ca, sn = q0->xa;
            double x2 = x[v][0] * x[v][0];
#pragma unroll
            for (int d = 1; d < D; ++d) {
                const AxisEq* q = tab + (v ? ix[d].y : ix[d].x);
                E *= q->E;
                c2 += q->c2;
                ca += q->ca;
                sn = dadd(sn, q->xa);
                x2 += x[v][d] * x[v][d];
            }
            const double pG = wa * fv[0][v] + E * (1.0 + ca * (c2 * irt - (D + 2)));
            const double pH = NA == 2 ? wa * fv[NA - 1][v] + RTH * E * (1.0 + ca * (c2 * irt - D)) : 0.0;
            o[0][v] = sn * pG;
            const double q = wv[v] * o[0][v];
            acc[0] += q;
#pragma unroll
            for (int d = 0; d < D; ++d) acc[1 + d] += q * x[v][d];
            acc[D + 1] += q * x2;                          // twice the energy moment
            if (NA == 2) {
                o[NA - 1][v] = sn * pH;
                acc[D + 1] += wv[v] * o[NA - 1][v];
            }
        }
#pragma unroll
        for (int a = 0; a < NA; ++a) stv<double, 2>(Fo + (size_t)a * Nvp + k0, o[a]);
    }
    acc[D + 1] *= 0.5;
    block_sum_t<NW, NT>(acc, sw, red);
    if (tid < NW) P.AF[(size_t)f * NW + tid] = red[tid];
}

// ------------------------------------------------------------------ k_cell
// Per-cell parameters of the collision update, written by k_cell_state.
template <typename T>
struct CellPar {
    EqPar<T> eq;             // Shakhov(W~, q~) of the cell
    T upd[4];                // 1/dt, 1/tau~, 1/|V|, 1/(1/dt + 1/tau~)
    T Vn[3];                 // U(W~) in the element type: reference of the next raw moments
};

static_assert(sizeof(CellPar<double>) <= AVS_CELLPAR_BYTES, "CellPar buffer size");

template <int D, typename T>
struct CellP {
    int Nc, Nv, Nvp;
    size_t cstride;
    double dt, idt;
    double R, Pr, omega, mu_ref, T_ref;
    const T* __restrict__ fin;
    T* __restrict__ fout;
    const T* __restrict__ F;
    const double* __restrict__ AF;
    const double* __restrict__ Win;
    double* __restrict__ Wout;
    double* mom;             // [cell][NM] raw moments of f about U(W) (read by k_cell_state, rewritten by k_cell)
    CellPar<T>* par;         // [cell]
    const T* __restrict__ xi;
    const T* __restrict__ w;
    const int* __restrict__ slot;
    const unsigned char* __restrict__ nslot;
    const double* __restrict__ vol;
    int* err;
};

// Raw moments of the own f^n of cell i about its U(W^n) over nodes [kb, ke):
// per-thread partial sums in acc[NM].
template <int D, int NT, int VC>
__device__ __forceinline__ void cell_raw_moments(const CellP<D, double>& P, int i, int kb, int ke, double* acc)
{
    constexpr int NA = NArr<D>::v, NM = NMom<D>::v, NW = D + 2;
    constexpr int V = VC;
    double Vct[D];
#pragma unroll
    for (int d = 0; d < D; ++d) Vct[d] = P.Win[(size_t)i * NW + 1 + d] / P.Win[(size_t)i * NW];
    const double* fi = P.fin + (size_t)i * P.cstride;
#pragma unroll
    for (int m = 0; m < NM; ++m) acc[m] = 0.0;
    for (int k0 = kb + threadIdx.x * V; k0 < ke; k0 += NT * V) {
        double x[V][D], wv[V], f0[V], f1[V];
        load_nodes<D, V>(P, k0, x, wv);
        ldv<double, V>(fi + k0, f0);
        if (NA == 2) ldv<double, V>(fi + P.Nvp + k0, f1);
#pragma unroll
        for (int v = 0; v < V; ++v) {
            double xs[D];
#pragma unroll
            for (int d = 0; d < D; ++d) xs[d] = x[v][d] - Vct[d];
            raw_acc<D>(acc, xs, wv[v] * f0[v], NA == 2 ? wv[v] * f1[v] : 0.0);
        }
    }
}

// Raw moments of the own f^n of every cell about its U(W^n) (one block per
// cell); used when the previous step did not leave them (after init, set_f,
// set_W or an adaptation).
template <int D, int NT, int VC>
__global__ void __launch_bounds__(NT) k_raw_moments(CellP<D, double> P)
{
    constexpr int NM = NMom<D>::v;
    __shared__ double sw[(NT / 32) * NM];
    __shared__ double red[NM];
    const int i = blockIdx.x;
    double acc[NM];
    cell_raw_moments<D, NT, VC>(P, i, 0, P.Nv, acc);
    block_sum_t<NM, NT>(acc, sw, red);
    if (threadIdx.x < NM) P.mom[(size_t)i * NM + threadIdx.x] = red[threadIdx.x];
}

// Cell record of the FP32 kernels: out = (u0 f + u1 g~ + un N) u3.
__device__ __forceinline__ Cell32Par cell32_par(const EqPar<float>& e, float u0, float u1, float un, float u3,
                                                const float* V, float diag)
{
    Cell32Par z;
    for (int d = 0; d < 3; ++d) {
        z.U[d] = e.U[d];
        z.al[d] = e.alpha[d];
        z.V[d] = V[d];
    }
    z.k2 = e.k2;
    z.l2 = e.l2pref;
    z.u0 = u0;
    z.u1 = u1;
    z.un = un;
    z.u3 = u3;
    z.irt = e.invRT;
    z.RTH = e.RTH;
    z.diag = diag;
    z.pad[0] = z.pad[1] = 0.0f;
    return z;
}

// One thread per cell: lagged heat flux q~ from the raw moments of f^n (R3),
// W~ = W - dt/|V| sum_j sgn_j A F_j (R2), tau~ and the Shakhov parameters.
template <int D, typename T>
__global__ void k_cell_state(CellP<D, T> P)
{
    constexpr int NM = NMom<D>::v, NW = D + 2;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= P.Nc) return;
    const double* Wi = P.Win + (size_t)i * NW;
    double Vc[3] = {0.0, 0.0, 0.0}, m[NM];
    for (int d = 0; d < D; ++d) Vc[d] = (double)((T)Wi[1 + d] / (T)Wi[0]);
    for (int k = 0; k < NM; ++k) m[k] = P.mom[(size_t)i * NM + k];
    T rn, Un[3], RTn, qn[3];
    state_from_raw<D, T>(m, Vc, rn, Un, RTn, qn);
    const int ns = P.nslot[i];
    double Wt[5];
    // the FP32 form divides once by each of |V| and rho (an FP64 division is
    // about ten instructions of the scarce pipe)
    double iv, dtv;
    if constexpr (sizeof(T) == 4) {
        iv = 1.0 / P.vol[i];
        dtv = P.dt * iv;
    } else {
        dtv = P.dt / P.vol[i];
    }
    for (int c = 0; c < NW; ++c) {
        double sum = 0.0;
        for (int s = 0; s < ns; ++s) {
            const int sl = P.slot[i * AVS_MAXS + s];
            const double a = P.AF[(size_t)(sl >> 1) * NW + c];
            sum += (sl & 1) ? -a : a;
        }
        Wt[c] = Wi[c] - dtv * sum;
        P.Wout[(size_t)i * NW + c] = Wt[c];
    }
    CellPar<T> cp;
    for (int d = 0; d < 3; ++d) cp.Vn[d] = d < D ? (T)Wt[1 + d] / (T)Wt[0] : T(0);
    double rhod, Ud[3], RTd;
    if constexpr (sizeof(T) == 4) {
        rhod = Wt[0];
        const double ir = 1.0 / rhod;
        double m2 = 0.0;
        for (int d = 0; d < D; ++d) {
            Ud[d] = Wt[1 + d] * ir;
            m2 += Wt[1 + d] * Wt[1 + d];
        }
        RTd = (Wt[D + 1] - 0.5 * m2 * ir) * ir * (1.0 / 1.5);
    } else {
        prim<D>(Wt, rhod, Ud, RTd);
    }
    if (!(rhod > 0.0) || !(RTd > 0.0)) atomicOr(P.err, 1);
    const T rho = (T)rhod, RT = (T)RTd;
    T U[3];
    for (int d = 0; d < 3; ++d) U[d] = d < D ? (T)Ud[d] : T(0);
    const T tau = tau_vhs<T>(rho, RT, (T)P.R, (T)P.mu_ref, (T)P.T_ref, (T)P.omega);
    cp.eq = make_eq_a<D, T, T>(rho, U, RT, qn, (T)P.Pr);
    const T idt = (T)P.idt, itau = T(1) / tau;
    if constexpr (sizeof(T) == 4) {
        reinterpret_cast<Cell32Par*>(P.par)[i] =
            cell32_par(cp.eq, idt, itau, -(float)iv, 1.0f / (idt + itau), cp.Vn, 0.0f);
        return;
    }
    cp.upd[0] = idt;
    cp.upd[1] = itau;
    cp.upd[2] = (T)(1.0 / P.vol[i]);
    cp.upd[3] = T(1) / (idt + itau);
    P.par[i] = cp;
}

// Collision update of cell i over nodes [kb, ke): net flux N = sum_j sgn_j F_j
// per node and the update (diagonal of Eq. SGS_phi, R1); pad nodes are written
// as zero.  The raw moments of the new f about U(W~) are summed on the way
// (per-thread partials in acc[NM], same nodes per thread and order as
// cell_raw_moments).  fs, sg: the cell's face indices and signs; cp its
// collision parameters (shared memory).
template <int D, int NT, int VC>
__device__ __forceinline__ void cell_update(const CellP<D, double>& P, int i, int ns, const int* fs, const double* sg,
                                            const CellPar<double>& cp, int kb, int ke, double* acc)
{
    constexpr int NA = NArr<D>::v, NM = NMom<D>::v;
    constexpr int V = VC;
    const double* fi = P.fin + (size_t)i * P.cstride;
    double* fo = P.fout + (size_t)i * P.cstride;
    const double u0 = cp.upd[0], u1 = cp.upd[1], u2 = cp.upd[2], u3 = cp.upd[3];
    double Vnt[D];
#pragma unroll
    for (int d = 0; d < D; ++d) Vnt[d] = cp.Vn[d];
#pragma unroll
    for (int m = 0; m < NM; ++m) acc[m] = 0.0;
    for (int k0 = kb + threadIdx.x * V; k0 < ke; k0 += NT * V) {
        double x[V][D], wv[V];
        load_nodes<D, V>(P, k0, x, wv);
        double Nn[NA][V], fv[NA][V], out[NA][V];
#pragma unroll
        for (int a = 0; a < NA; ++a) {
            ldv_cg<double, V>(fi + (size_t)a * P.Nvp + k0, fv[a]);
#pragma unroll
            for (int v = 0; v < V; ++v) Nn[a][v] = 0.0;
        }
#pragma unroll
        for (int s = 0; s < AVS_MAXS; ++s) {
            if (s >= ns) break;
            const double* Fs = P.F + (size_t)fs[s] * NA * P.Nvp + k0;
            const double g = sg[s];
#pragma unroll
            for (int a = 0; a < NA; ++a) {
                double t[V];
                ldv_cg<double, V>(Fs + (size_t)a * P.Nvp, t);
#pragma unroll
                for (int v = 0; v < V; ++v) Nn[a][v] += g * t[v];
            }
        }
#pragma unroll
        for (int v = 0; v < V; ++v) {
            double gG, gH;
            eq_eval<D>(cp.eq, x[v], gG, gH);
            const bool real = k0 + v < P.Nv;
            out[0][v] = real ? (fv[0][v] * u0 + gG * u1 - Nn[0][v] * u2) * u3 : 0.0;
            if (NA == 2)
                out[NA - 1][v] = real ? (fv[NA - 1][v] * u0 + gH * u1 - Nn[NA - 1][v] * u2) * u3 : 0.0;
            double xs[D];
#pragma unroll
            for (int d = 0; d < D; ++d) xs[d] = x[v][d] - Vnt[d];
            raw_acc<D>(acc, xs, wv[v] * out[0][v], NA == 2 ? wv[v] * out[NA - 1][v] : 0.0);
        }
#pragma unroll
        for (int a = 0; a < NA; ++a) stv<double, V>(fo + (size_t)a * P.Nvp + k0, out[a]);
    }
}

// One block per cell, all nodes; the raw moments of f^{n+1} to P.mom.
template <int D, int NT, int VC>
__global__ void __launch_bounds__(NT, 4) k_cell(CellP<D, double> P)
{
    constexpr int NM = NMom<D>::v;
    __shared__ int fs[AVS_MAXS];
    __shared__ double sg[AVS_MAXS];
    __shared__ double sw[(NT / 32) * NM];
    __shared__ double red[NM];
    __shared__ CellPar<double> cp;

    const int tid = threadIdx.x;
    const int i = blockIdx.x;
    const int ns = P.nslot[i];
    if (tid < ns) {
        const int sl = P.slot[i * AVS_MAXS + tid];
        fs[tid] = sl >> 1;
        sg[tid] = (sl & 1) ? -1.0 : 1.0;
    }
    if (tid == 32 % NT) cp = P.par[i];
    __syncthreads();
    double acc[NM];
    cell_update<D, NT, VC>(P, i, ns, fs, sg, cp, 0, P.Nv, acc);
    block_sum_t<NM, NT>(acc, sw, red);
    if (tid < NM) P.mom[(size_t)i * NM + tid] = red[tid];
}

// k_cell in the FP64 form with the cell's equilibrium from tables of the axes'
// values, as k_face_tab (67 -> 39 FP64 instructions per cell and node in 3D; per
// step 61 -> 43 us and 1.63 -> 0.99 ms on the same cases).
// The carried raw moments are summed from c = xi - U(W~) as k_raw_moments forms
// it, in its node order.
struct AxisCell {
    double E, c, ca, pad;    // exp(-c^2 / 2RT) (axis 0: times pref), c, c alpha
};

template <int D, int NT>
__global__ void __launch_bounds__(NT) k_cell_tab(CellP<D, double> P, const double* __restrict__ xtab,
                                                 const unsigned short* __restrict__ tix, size_t xstride, int n0,
                                                 int n1, int nt)
{
    constexpr int NA = NArr<D>::v, NM = NMom<D>::v;
    extern __shared__ __align__(16) unsigned char tab_dsm[];
    AxisCell* tab = reinterpret_cast<AxisCell*>(tab_dsm);
    __shared__ int fs[AVS_MAXS];
    __shared__ double sg[AVS_MAXS];
    __shared__ double sw[(NT / 32) * NM];
    __shared__ double red[NM];
    const int tid = threadIdx.x;
    const int i = blockIdx.x;
    const int ns = P.nslot[i];
    const CellPar<double>& cp = P.par[i];
    if (tid < ns) {
        const int sl = P.slot[i * AVS_MAXS + tid];
        fs[tid] = sl >> 1;
        sg[tid] = (sl & 1) ? -1.0 : 1.0;
    }
    for (int e = tid; e < nt; e += NT) {
        const int d = e < n0 ? 0 : e < n1 ? 1 : 2;
        const double c = xtab[e] - cp.eq.U[d];
        AxisCell q;
        q.E = ex(-(c * c) * cp.eq.inv2RT);
        if (d == 0) q.E *= cp.eq.pref;
        q.c = c;
        q.ca = c * cp.eq.alpha[d];
        q.pad = 0.0;
        tab[e] = q;
    }
    __syncthreads();
    const double u0 = cp.upd[0], u1 = cp.upd[1], u2 = cp.upd[2], u3 = cp.upd[3], irt = cp.eq.invRT, RTH = cp.eq.RTH;
    const double* fi = P.fin + (size_t)i * P.cstride;
    double* fo = P.fout + (size_t)i * P.cstride;
    double acc[NM];
#pragma unroll
    for (int m = 0; m < NM; ++m) acc[m] = 0.0;
    for (int k0 = tid * 2; k0 < P.Nv; k0 += NT * 2) {
        double wv[2], Nn[NA][2], fv[NA][2], out[NA][2];
        ldv<double, 2>(P.w + k0, wv);
        ushort2 ix[D];
#pragma unroll
        for (int d = 0; d < D; ++d) ix[d] = *reinterpret_cast<const ushort2*>(tix + d * xstride + k0);
#pragma unroll
        for (int a = 0; a < NA; ++a) {
            ldv_cg<double, 2>(fi + (size_t)a * P.Nvp + k0, fv[a]);
            Nn[a][0] = Nn[a][1] = 0.0;
        }
#pragma unroll
        for (int s = 0; s < AVS_MAXS; ++s) {
            if (s >= ns) break;
            const double* Fs = P.F + (size_t)fs[s] * NA * P.Nvp + k0;
            const double g = sg[s];
#pragma unroll
            for (int a = 0; a < NA; ++a) {
                double t[2];
                ldv_cg<double, 2>(Fs + (size_t)a * P.Nvp, t);
                Nn[a][0] += g * t[0];
                Nn[a][1] += g * t[1];
            }
        }
#pragma unroll
        for (int v = 0; v < 2; ++v) {
            const AxisCell* q0 = tab + (v ? ix[0].y : ix[0].x);
            double E = q0->E, ca = q0->ca, c[D];
            c[0] = q0->c;
            double c2 = c[0] * c[0];
#pragma unroll
            for (int d = 1; d < D; ++d) {
                const AxisCell* q = tab + (v ? ix[d].y : ix[d].x);
                E *= q->E;
                ca += q->ca;
                c[d] = q->c;
                c2 += c[d] * c[d];
            }
            const double gG = E * (1.0 + ca * (c2 * irt - (D + 2)));
            const bool real = k0 + v < P.Nv;
            out[0][v] = real ? (fv[0][v] * u0 + gG * u1 - Nn[0][v] * u2) * u3 : 0.0;
            if (NA == 2) {
                const double gH = RTH * E * (1.0 + ca * (c2 * irt - D));
                out[NA - 1][v] = real ? (fv[NA - 1][v] * u0 + gH * u1 - Nn[NA - 1][v] * u2) * u3 : 0.0;
            }
            raw_acc<D>(acc, c, wv[v] * out[0][v], NA == 2 ? wv[v] * out[NA - 1][v] : 0.0);
        }
#pragma unroll
        for (int a = 0; a < NA; ++a) stv<double, 2>(fo + (size_t)a * P.Nvp + k0, out[a]);
    }
    block_sum_t<NM, NT>(acc, sw, red);
    if (tid < NM) P.mom[(size_t)i * NM + tid] = red[tid];
}

// geometry of the FP64 kernels (the FP32 ones read geo32)
template <typename T>
static CellGeo<T> cell_geo(const avs_ctx* c)
{
    CellGeo<T> geo;
    geo.nbr = c->nbr;
    geo.cg = (const T*)c->cg_d;
    geo.r = (const T*)c->r_d;
    geo.eps2 = (const T*)c->eps2_d;
    geo.ns = c->nslot;
    return geo;
}

// Limited gradients of every array of every cell into c->grad (allocated by the
// caller), FP64 form of the Rykov gas.
template <int D, int NA>
static void grad_t(avs_ctx* c, const void* fin)
{
    constexpr int VG = 4;
    const CellGeo<double> geo = cell_geo<double>(c);
    dim3 g(c->Nc, (c->Nv + 256 * VG - 1) / (256 * VG));
    if (D == 2 && c->max_ns <= 4)
        k_grad<D, double, VG, 4, NA><<<g, 256, 0, c->stream>>>(c->Nv, c->Nvp, c->cfg.limiter, (const double*)fin,
                                                               (double*)c->grad, geo);
    else
        k_grad<D, double, VG, AVS_MAXS, NA><<<g, 256, 0, c->stream>>>(c->Nv, c->Nvp, c->cfg.limiter, (const double*)fin,
                                                                      (double*)c->grad, geo);
    c->launches += 1;
}

// Foot values of the FP32 form into c->flux, either gas (the
// Rykov form takes the FP64 upwind choice).
template <int D, int NA, bool EXACT>
static void foot32_t(avs_ctx* c, const void* fin, double hd)
{
    constexpr int VG = 4;
    // 2D: 128 threads, or 64 where a row has no more quads (190 nodes, 12288
    // cells: 41 -> 25 us), with up to eight quads per thread (3.5k nodes, 12288
    // cells: 252 us, four 270; 12k nodes, 38400 cells: 2.48 ms, 2.56).  3D: 64
    // threads and up to four quads, as chunks of 1024 nodes let the rows of six
    // neighbours be reused from the caches (21k nodes, 36864 cells: 4.00 ms; 128
    // threads of up to eight 4.09, of up to four 4.24).  One block per cell and
    // chunk while that leaves 32 blocks per SM.  (All with the flushing reciprocal
    // in the limiter; with the division 259 us, 2.55 and 4.07 ms.)
    const int nquad = (c->Nv + VG - 1) / VG;
    const int nt = D == 3 || nquad <= 64 ? 64 : 128;
    const long long most = D == 3 ? 4 : 8;
    const int per = (int)std::max(1ll, std::min(most, (long long)c->Nc * nquad / nt / (32 * std::max(1, c->nsm))));
    const int ny = (nquad + nt * per - 1) / (nt * per);
    const int chunk = (nquad + ny - 1) / ny * VG;
    auto go = [&](auto ns) {
        k_foot_f2<D, decltype(ns)::value, NA, EXACT><<<dim3(c->Nc, ny), nt, 0, c->stream>>>(
            c->Nv, c->Nvp, chunk, c->cfg.limiter, (float)hd, (const float*)fin, (float*)c->flux, (const float4*)c->geo32,
            c->eps2_f, c->xi_s, c->xstride, c->xi_d, c->An_d);
    };
    c->launches += 1;
    if constexpr (D == 2)
        if (c->max_ns <= 4) return go(std::integral_constant<int, 4>{});
    go(std::integral_constant<int, AVS_MAXS>{});
}

void launch_foot32(avs_ctx* c, const void* fin, double hd)
{
    if (c->model == AVS_RYKOV) c->D == 2 ? foot32_t<2, 3, true>(c, fin, hd) : foot32_t<3, 2, true>(c, fin, hd);
    else c->D == 2 ? foot32_t<2, 2, false>(c, fin, hd) : foot32_t<3, 1, false>(c, fin, hd);
}

// Tables of the axes' coordinates pay where a face's or cell's nodes are at
// least twice the entries: an entry costs what a node without tables does, a
// node with them about half.
static bool axis_tables(const avs_ctx* c) { return c->tab_n > 0 && 2 * c->tab_n <= c->Nv; }

// Foot values of every face (k_foot) and the face stage of a step: per-node
// face flux in c->flux, area-weighted face flux of W in c->AFf (shared by
// the explicit and the implicit step).
template <int D, typename T>
static cudaError_t face_stage_t(avs_ctx* c, const void* fin, const double* Win, double dt)
{
    const int NA = NArr<D>::v;
    const cudaError_t ea = ensure_flux(c);
    if (ea != cudaSuccess) return ea;
    const double hd = 0.5 * dt;
    {
        if constexpr (sizeof(T) == 4) {
            launch_foot32(c, fin, hd);
        } else {
            const CellGeo<T> geo = cell_geo<T>(c);
            // two nodes per thread and iteration; 64 threads for short rows, up
            // to four iterations while that leaves 16 blocks per SM
            const int npair = (c->Nv + 1) / 2;
            const int nt = npair <= 64 ? 64 : 128;
            const int per = (int)std::max(1ll, std::min(4ll, (long long)c->Nc * npair / nt / (16 * std::max(1, c->nsm))));
            const int ny = (npair + nt * per - 1) / (nt * per);
            const int chunk = (npair + ny - 1) / ny * 2;
            auto go = [&](auto ns) {
                k_foot<D, decltype(ns)::value, NArr<D>::v><<<dim3(c->Nc, ny), nt, 0, c->stream>>>(
                    c->Nv, c->Nvp, chunk, c->cfg.limiter, hd, (const double*)fin, (double*)c->flux, geo,
                    c->An_d, c->xi_d, (const float4*)c->geo32, c->xi_s, c->xstride);
            };
            using Four = std::integral_constant<int, D == 2 ? 4 : AVS_MAXS>;      // 3D: six slots always
            if (c->max_ns <= 4) go(Four{});
            else go(std::integral_constant<int, AVS_MAXS>{});
            c->launches += 1;
        }
    }
    if constexpr (sizeof(T) == 4) {
        return launch_face32(c, Win, dt);
    } else {
        FaceP<D> P;
        P.Nv = c->Nv;
        P.Nvp = c->Nvp;
        P.cstride = (size_t)NA * c->Nvp;
        P.hd = hd;
        P.R = c->cfg.R;
        P.Pr = c->cfg.Pr;
        P.omega = c->cfg.omega;
        P.mu_ref = c->mu_ref;
        P.T_ref = c->cfg.T_ref;
        P.FB = (double*)c->flux;
        P.AF = c->AFf;
        P.Win = Win;
        P.xi = c->xi_d;
        P.w = c->w_d;
        P.order = c->forder;
        P.faceL = c->faceL;
        P.faceR = c->faceR;
        P.An = c->An_d;
        P.bc = c->bc;
        P.err = c->dev_err;
        constexpr int NT = 128;
        // foot values of pass A kept in shared memory for pass B when they fit in
        // the default dynamic allowance (48 KB); otherwise pass B re-reads the
        // face's row
        const size_t cache_bytes = (size_t)NA * c->Nvp * sizeof(T);
        constexpr int VF = 2;            // nodes per thread and iteration: 16-byte vectors
        // the default allowance covers static and dynamic shared memory together:
        // the block's own arrays (state, reductions: under 2 KB) come first
        constexpr size_t kStaticFace = 2048;
        static_assert(sizeof(FaceSt) + (NT / 32 + 1) * FaceNR<D>::v * sizeof(double) <= kStaticFace,
                      "static shared memory of the face block");
        if (axis_tables(c)) {
            const size_t smem = (size_t)c->tab_n * sizeof(AxisEq);
            if (smem > 40 * 1024) {      // the most of any context: as k_cell32
                const cudaError_t e = cudaFuncSetAttribute(k_face_tab<D, NT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                           (int)(AVS_TAB_MAX * sizeof(AxisEq)));
                if (e != cudaSuccess) return e;
            }
            k_face_tab<D, NT><<<c->Nf, NT, smem, c->stream>>>(P, c->xtab, c->tix, c->xstride, c->tab_end[0], c->tab_end[1],
                                                             c->tab_n);
        } else if (cache_bytes + kStaticFace <= 48 * 1024)
            k_face<D, NT, true, VF><<<c->Nf, NT, cache_bytes, c->stream>>>(P);
        else
            k_face<D, NT, false, VF><<<c->Nf, NT, 0, c->stream>>>(P);
        c->launches += 1;

        return cudaGetLastError();
    }
}

template <int D, typename T>
static cudaError_t launch_step_t(avs_ctx* c, const void* fin, void* fout, const double* Win, double* Wout,
                                 double dt)
{
    const bool f32 = sizeof(T) == 4;
    const int NA = NArr<D>::v;
    cudaError_t e = face_stage_t<D, T>(c, fin, Win, dt);
    if (e != cudaSuccess) return e;
    const T* xi = f32 ? (const T*)c->xi_f : (const T*)c->xi_d;
    const T* w = f32 ? (const T*)c->w_f : (const T*)c->w_d;
    constexpr int NT = 128;
    CellP<D, T> Q;
    Q.Nc = c->Nc;
    Q.Nv = c->Nv;
    Q.Nvp = c->Nvp;
    Q.cstride = (size_t)NA * c->Nvp;
    Q.dt = dt;
    Q.idt = 1.0 / dt;
    Q.R = c->cfg.R;
    Q.Pr = c->cfg.Pr;
    Q.omega = c->cfg.omega;
    Q.mu_ref = c->mu_ref;
    Q.T_ref = c->cfg.T_ref;
    Q.fin = (const T*)fin;
    Q.fout = (T*)fout;
    Q.F = (const T*)c->flux;
    Q.AF = c->AFf;
    Q.Win = Win;
    Q.Wout = Wout;
    Q.mom = c->cmom;
    Q.par = (CellPar<T>*)c->cpar;
    Q.xi = xi;
    Q.w = w;
    Q.slot = c->slot;
    Q.nslot = c->nslot;
    Q.vol = c->vol;
    Q.err = c->dev_err;
    if (!c->mom_valid) {
        if constexpr (sizeof(T) == 4) {
            e = launch_raw32(c, fin, Win);
            if (e != cudaSuccess) return e;
        } else {
            k_raw_moments<D, NT, VW<T>::v><<<c->Nc, NT, 0, c->stream>>>(Q);
            c->launches += 1;
        }
    }
    k_cell_state<D, T><<<(c->Nc + kCellNT - 1) / kCellNT, kCellNT, 0, c->stream>>>(Q);
    c->launches += 1;
    if constexpr (sizeof(T) == 4) {
        e = launch_cell32(c, fin, fout, false);
        if (e != cudaSuccess) return e;
    } else {
        // 16-byte vectors of nodes per thread; k_raw_moments takes the same
        // node mapping, so that its sums equal the carried ones bit for bit
        if (axis_tables(c)) {
            const size_t smem = (size_t)c->tab_n * sizeof(AxisCell);
            if (smem > 40 * 1024) {      // the most of any context: as k_cell32
                e = cudaFuncSetAttribute(k_cell_tab<D, NT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)(AVS_TAB_MAX * sizeof(AxisCell)));
                if (e != cudaSuccess) return e;
            }
            k_cell_tab<D, NT><<<c->Nc, NT, smem, c->stream>>>(Q, c->xtab, c->tix, c->xstride, c->tab_end[0],
                                                             c->tab_end[1], c->tab_n);
        } else {
            k_cell<D, NT, VW<T>::v><<<c->Nc, NT, 0, c->stream>>>(Q);
        }
        c->launches += 1;
    }
    c->mom_valid = 1;          // the raw moments of fout about U(Wout) are in cmom
    return cudaGetLastError();
}

// ================================================================== implicit step
// IUGKS (Sec. 2.3.1): after the face stage, the macroscopic Eq. (SGS_w) for
// dW = W~ - W^n and the microscopic Eq. (SGS_phi) for dphi are solved by
// symmetric Gauss-Seidel sweeps over a greedy cell colouring: the cells of one
// colour share no face, so a colour is updated in parallel with the values of
// the other colours as they stand, which is the sequential sweep in the order
// "colour 0, colour 1, ..." (forward) and back (backward).

// Euler flux of a conserved state W through the unit normal n (monatomic gas).
template <int D, typename A>
__device__ __forceinline__ void euler_flux_n(const A* W, const A* n, A* G)
{
    const A rho = W[0];
    A m2 = A(0), un = A(0);
#pragma unroll
    for (int d = 0; d < D; ++d) {
        m2 += W[1 + d] * W[1 + d];
        un += (W[1 + d] / rho) * n[d];
    }
    const A p = rho * ((W[D + 1] - A(0.5) * m2 / rho) / (A(1.5) * rho));
    G[0] = rho * un;
#pragma unroll
    for (int d = 0; d < D; ++d) G[1 + d] = W[1 + d] * un + p * n[d];
    G[D + 1] = (W[D + 1] + p) * un;
}

// Interior face slot of a cell, in sweep order: the slot's outward unit normal
// n, -A/2, A r/2 (r the face's spectral radius) and the Euler flux of the
// neighbour's W^n through n, so that a sweep only evaluates G(W~_j).
template <typename A>
struct alignas(16) ImpSlot {
    A n[3];
    A nhA;
    A hr;
    A Gn[5];
    int j;
};
static_assert(sizeof(ImpSlot<double>) <= AVS_IMPSLOT_BYTES, "slot record");

template <typename A>
struct ImpP {
    int Nc;
    double dt, R, mu_ref, T_ref, omega;
    const int* slot;
    const unsigned char* nslot;
    const int* faceL;
    const int* faceR;
    const double* An;
    const double* rL;
    const double* rR;
    const double* vol;
    const double* AF;
    const double* Wn;        // W^n [cell][NW]
    double* Wt;              // W~ [cell][NW] (the output W)
    A* dWa;                  // dW [cell][NW]
    A* Wta;                  // W~ rounded to A [cell][NW]; aliases Wt when A is double
    A* rhs;                  // [q][NW]  -sum sgn A F
    A* dg;                   // [q]      V/dt + 1/2 sum A r
    ImpSlot<A>* co;          // [q][MAXS] interior slots first
    unsigned char* nint;     // [q] interior slots
    const int* clist;        // cells by colour (q -> cell)
    int* err;
};

// Per cell, in sweep order q: diagonal V/dt + 1/2 sum A r over every slot,
// explicit residual -sum sgn A F, and the interior slot records.  r from the
// face's own orientation (L, R, n_LR), so both cells of a face use one value.
template <int D, typename A>
__global__ void k_imp_setup(ImpP<A> P)
{
    constexpr int NW = D + 2;
    const int q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= P.Nc) return;
    const int i = P.clist[q];
    const int ns = P.nslot[i];
    const double* Wi = P.Wn + (size_t)i * NW;
    for (int c = 0; c < NW; ++c) {
        double acc = 0.0;
        for (int s = 0; s < ns; ++s) {
            const int sl = P.slot[i * AVS_MAXS + s];
            const double a = P.AF[(size_t)(sl >> 1) * NW + c];
            acc += (sl & 1) ? -a : a;
        }
        P.rhs[(size_t)q * NW + c] = (A)(-acc);
        P.dWa[(size_t)i * NW + c] = A(0);
        P.Wt[(size_t)i * NW + c] = Wi[c];
        P.Wta[(size_t)i * NW + c] = (A)Wi[c];
    }
    double dg = P.vol[i] / P.dt;
    int nint = 0;
    for (int s = 0; s < ns; ++s) {
        const int sl = P.slot[i * AVS_MAXS + s];
        const int f = sl >> 1;
        const double sgn = (sl & 1) ? -1.0 : 1.0;
        const int L = P.faceL[f], R = P.faceR[f];
        const double* An = P.An + (size_t)f * D;
        double Aa = 0.0;
        for (int d = 0; d < D; ++d) Aa += An[d] * An[d];
        Aa = sqrt(Aa);
        double n[3] = {0, 0, 0}, dl = 0.0;
        for (int d = 0; d < D; ++d) n[d] = An[d] / Aa;
        for (int d = 0; d < D; ++d) {
            const double e = R >= 0 ? P.rL[(size_t)f * D + d] - P.rR[(size_t)f * D + d] : 2.0 * P.rL[(size_t)f * D + d];
            dl += e * e;
        }
        dl = sqrt(dl);
        // spectral radius |U.n| + a + 2 mu / (rho dl) from the mean primitive state
        double rl, Ul[3], RTl, rr, Ur[3], RTr;
        prim<D>(P.Wn + (size_t)L * NW, rl, Ul, RTl);
        prim<D>(P.Wn + (size_t)(R >= 0 ? R : L) * NW, rr, Ur, RTr);
        const double rho = 0.5 * (rl + rr), RT = 0.5 * (RTl + RTr);
        double un = 0.0;
        for (int d = 0; d < D; ++d) un += 0.5 * (Ul[d] + Ur[d]) * n[d];
        const double mu = P.mu_ref * pow(RT / P.R / P.T_ref, P.omega);
        const double r = Aa * (fabs(un) + sqrt(5.0 / 3.0 * RT) + 2.0 * mu / (rho * dl));
        dg += 0.5 * r;
        const int j = (sl & 1) ? L : R;
        if (j >= 0) {
            ImpSlot<A> sc;
            for (int d = 0; d < 3; ++d) sc.n[d] = d < D ? (A)(sgn * An[d] / Aa) : A(0);
            sc.nhA = (A)(-0.5 * Aa);
            sc.hr = (A)(0.5 * r);
            A Wj[NW];
            for (int c = 0; c < NW; ++c) Wj[c] = (A)P.Wn[(size_t)j * NW + c];
            euler_flux_n<D, A>(Wj, sc.n, sc.Gn);
            for (int c = NW; c < 5; ++c) sc.Gn[c] = A(0);
            sc.j = j;
            P.co[(size_t)q * AVS_MAXS + nint++] = sc;
        }
    }
    P.dg[q] = (A)dg;
    P.nint[q] = (unsigned char)nint;
}

// Self-test of the bounded grid barrier: `rounds` barriers, the last one
// waiting for `short_by` arrivals more than the grid has (none when 0), each
// passed barrier counted once per block in *passed.
__global__ void k_grid_barrier_check(unsigned* bar, int rounds, int short_by, int* err, int* passed)
{
    unsigned gen = 0;
    for (int r = 0; r < rounds; ++r) {
        const unsigned target = ++gen * gridDim.x + (r == rounds - 1 ? (unsigned)short_by : 0u);
        if (!grid_sync_bounded(bar, target, err)) return;
        if (threadIdx.x == 0) atomicAdd(passed, 1);
    }
}

cudaError_t launch_grid_barrier_check(avs_ctx* c, int blocks, int rounds, int short_by, int* passed_dev)
{
    cudaError_t e = cudaMemsetAsync(c->imp_bar, 0, sizeof(unsigned), c->stream);
    if (e != cudaSuccess) return e;
    unsigned* bar = c->imp_bar;
    int* err = c->dev_err;
    void* args[] = {&bar, &rounds, &short_by, &err, &passed_dev};
    e = cudaLaunchCooperativeKernel((const void*)k_grid_barrier_check, dim3(blocks), dim3(128), args, 0, c->stream);
    if (e == cudaSuccess) c->launches += 1;
    return e;
}

constexpr long long kWaitCycles = 2000000000ll;
// Self-test of a bounded mbarrier wait on a bulk copy: with `arrive`
// one 128-byte bulk copy completes the barrier and the copied bytes are
// compared with the source; without, no arrival ever comes and every thread's
// wait gives up after kWaitCycles, setting bit 4 of the error word.
__global__ void k_stage_wait_check(const float* __restrict__ src, int arrive, int* err, int* completed)
{
    __shared__ __align__(128) float buf[32];
    __shared__ __align__(8) unsigned long long bar;
    if (threadIdx.x == 0) {
        mbar_init(&bar, 1);
        mbar_init_fence();
    }
    __syncthreads();
    if (threadIdx.x == 0 && arrive) {
        mbar_arrive_expect_tx(&bar, 128u);
        bulk_g2s(buf, src, 128u, &bar);
    }
    const bool ok = mbar_wait_bounded(&bar, 0u, kWaitCycles);
    if (!ok) {
        if (threadIdx.x == 0) {
            atomicOr(err, 4);
            // a copy that was issued may still land: wait for it (bounded)
            if (arrive) mbar_wait_bounded(&bar, 0u, kWaitCycles);
        }
        return;
    }
    if (threadIdx.x == 0) {
        int same = 1;
        for (int j = 0; j < 32; ++j) same &= buf[j] == src[j];
        *completed = same;
    }
}

cudaError_t launch_stage_wait_check(avs_ctx* c, const float* src, bool arrive, int* completed_dev)
{
    k_stage_wait_check<<<1, 32, 0, c->stream>>>(src, arrive ? 1 : 0, c->dev_err, completed_dev);
    c->launches += 1;
    return cudaGetLastError();
}

// One cell of a macroscopic sweep: dW_i = (Res_i + 1/2 sum A r dW_j) / dg_i,
// Res_i = -sum sgn A F - 1/2 sum A (G(W~_j) - G(W^n_j)) over the interior faces.
// Arithmetic in A (FP32 in the mixed form, where dW is a small correction of
// the FP64 W^n); W~ = W^n + dW in FP64.  What no sweep changes is loaded by
// load() ahead of the grid barrier (FP32; in FP64 the slot records would not
// fit the registers and are read in update()), the neighbours' values after it,
// all before the arithmetic and past L1: other blocks wrote them.
template <int D, typename A, int NS>
struct ImpCell {
    static constexpr int NW = D + 2;
    static constexpr bool PRE = sizeof(A) == 4;
    int i, n, j[NS];
    A rhs[NW], dg;
    double Wn[NW];
    ImpSlot<A> s[PRE ? NS : 1];

    __device__ __forceinline__ void load(const ImpP<A>& P, int q)
    {
        i = P.clist[q];
        n = P.nint[q];
        dg = P.dg[q];
#pragma unroll
        for (int c = 0; c < NW; ++c) rhs[c] = P.rhs[(size_t)q * NW + c];
#pragma unroll
        for (int k = 0; k < NS; ++k) {
            if (k >= n) break;
            if constexpr (PRE) {
                s[k] = P.co[(size_t)q * AVS_MAXS + k];
                j[k] = s[k].j;
            } else {
                j[k] = P.co[(size_t)q * AVS_MAXS + k].j;
            }
        }
#pragma unroll
        for (int c = 0; c < NW; ++c) Wn[c] = P.Wn[(size_t)i * NW + c];
    }

    __device__ __forceinline__ void update(const ImpP<A>& P, int q)
    {
        A Wj[NS][NW], dWj[NS][NW];
#pragma unroll
        for (int k = 0; k < NS; ++k) {
            if (k >= n) break;
            ld_row<NW>(P.Wta + (size_t)j[k] * NW, Wj[k]);
            ld_row<NW>(P.dWa + (size_t)j[k] * NW, dWj[k]);
        }
#pragma unroll
        for (int k = 0; k < NS; ++k) {
            if (k >= n) break;
            if constexpr (!PRE) s[0] = P.co[(size_t)q * AVS_MAXS + k];
            const ImpSlot<A>& sc = s[PRE ? k : 0];
            A G[NW];
            euler_flux_n<D, A>(Wj[k], sc.n, G);
#pragma unroll
            for (int c = 0; c < NW; ++c) rhs[c] += sc.nhA * (G[c] - sc.Gn[c]) + sc.hr * dWj[k][c];
        }
        A d[NW], wt[NW];
#pragma unroll
        for (int c = 0; c < NW; ++c) {
            d[c] = rhs[c] / dg;
            wt[c] = (A)(Wn[c] + (double)d[c]);
        }
        st_row<NW>(P.dWa + (size_t)i * NW, d);
        st_row<NW>(P.Wta + (size_t)i * NW, wt);
    }
};

// The whole macroscopic solve in one cooperative launch: k_macro symmetric
// Gauss-Seidel iterations, each colour a grid-stride pass, a grid barrier
// between passes; the next pass's first cell is loaded while the barrier
// collects its arrivals.  A colour that follows itself (the turn of a symmetric
// sweep) is skipped: its neighbours have not changed, so the pass would
// rewrite the same values.  Bounded by latency (barrier, one trip to L2, the
// arithmetic of one cell per thread), so small blocks on many SMs: the 121
// passes of 6144 cells (cylinder) took 690 us with the loads face by face after
// the barrier, 368 us now.
template <int D, typename A, int NT, int NS>
__global__ void __launch_bounds__(NT) k_imp_macro(ImpP<A> P, int k_macro, int ncolor, const int* __restrict__ cstart,
                                                  unsigned* bar)
{
    constexpr int NW = D + 2;
    const unsigned nb = gridDim.x;
    unsigned gen = 0;
    const int q0 = blockIdx.x * NT + threadIdx.x, dq = nb * NT;
    ImpCell<D, A, NS> C;
    int col = 0, q = cstart[0] + q0, c1 = cstart[1];
    if (q < c1) C.load(P, q);
    for (int it = 0, r = 0;;) {                  // r: place in the symmetric sweep
        while (q < c1) {
            C.update(P, q);
            q += dq;
            if (q < c1) C.load(P, q);
        }
        int nx = col;
        while (nx == col && it < k_macro) {
            if (++r == 2 * ncolor) r = 0, ++it;
            nx = r < ncolor ? r : 2 * ncolor - 1 - r;
        }
        if (it >= k_macro) break;
        col = nx;
        grid_arrive(bar);
        q = cstart[col] + q0;
        c1 = cstart[col + 1];
        if (q < c1) C.load(P, q);
        if (!grid_wait(bar, ++gen * nb, P.err)) return;
    }
    if constexpr (sizeof(A) == 4) {              // W~ in FP64, by the thread that updated the cell
        for (col = 0; col < ncolor; ++col)
            for (q = cstart[col] + q0; q < cstart[col + 1]; q += dq) {
                const size_t o = (size_t)P.clist[q] * NW;
#pragma unroll
                for (int c = 0; c < NW; ++c) P.Wt[o + c] = P.Wn[o + c] + (double)__ldcg(P.dWa + o + c);
            }
    }
}

// Per cell: Shakhov state of W~ with the lagged heat flux of f^n (R3);
// upd[0] = V/dt + V/tau~, upd[1] = tau~, upd[2] = V.
template <int D, typename T>
__global__ void k_imp_state(CellP<D, T> P, const double* Wt)
{
    constexpr int NM = NMom<D>::v, NW = D + 2;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= P.Nc) return;
    const double* Wi = P.Win + (size_t)i * NW;
    double Vc[3] = {0.0, 0.0, 0.0}, m[NM];
    for (int d = 0; d < D; ++d) Vc[d] = (double)((T)Wi[1 + d] / (T)Wi[0]);
    for (int k = 0; k < NM; ++k) m[k] = P.mom[(size_t)i * NM + k];
    T rn, Un[3], RTn, qn[3];
    state_from_raw<D, T>(m, Vc, rn, Un, RTn, qn);
    double rhod, Ud[3], RTd;
    prim<D>(Wt + (size_t)i * NW, rhod, Ud, RTd);
    if (!(rhod > 0.0) || !(RTd > 0.0)) atomicOr(P.err, 1);
    const T rho = (T)rhod, RT = (T)RTd;
    T U[3];
    for (int d = 0; d < 3; ++d) U[d] = (T)Ud[d];
    CellPar<T> cp;
    const T tau = tau_vhs<T>(rho, RT, (T)P.R, (T)P.mu_ref, (T)P.T_ref, (T)P.omega);
    cp.eq = make_eq_a<D, T, T>(rho, U, RT, qn, (T)P.Pr);
    const T V = (T)P.vol[i];
    if constexpr (sizeof(T) == 4) {
        const float zero[3] = {0.0f, 0.0f, 0.0f};
        reinterpret_cast<Cell32Par*>(P.par)[i] =
            cell32_par(cp.eq, -V / tau, V / tau, -1.0f, 1.0f, zero, V / (float)P.dt + V / tau);
        return;
    }
    cp.upd[0] = V / (T)P.dt + V / tau;
    cp.upd[1] = tau;
    cp.upd[2] = V;
    cp.upd[3] = T(0);
    for (int d = 0; d < 3; ++d) cp.Vn[d] = T(0);
    P.par[i] = cp;
}

// Per cell and node: microscopic residual Res = V (g~ - phi^n) / tau~ - N,
// N the net flux of the cell's faces (written over the f^{n+1} buffer).  V
// consecutive nodes per thread as in k_cell; pad nodes get Res = 0.
template <int D, typename T, int NT, int V>
__global__ void __launch_bounds__(NT) k_imp_res(CellP<D, T> P)
{
    constexpr int NA = NArr<D>::v;
    __shared__ int fs[AVS_MAXS];
    __shared__ T sg[AVS_MAXS];
    __shared__ CellPar<T> cp;
    const int i = blockIdx.x, tid = threadIdx.x;
    const int ns = P.nslot[i];
    if (tid < ns) {
        const int sl = P.slot[i * AVS_MAXS + tid];
        fs[tid] = sl >> 1;
        sg[tid] = (sl & 1) ? T(-1) : T(1);
    }
    if (tid == 32 % NT) cp = P.par[i];
    __syncthreads();
    const T* fi = P.fin + (size_t)i * P.cstride;
    T* ro = P.fout + (size_t)i * P.cstride;
    const T Vc = cp.upd[2], tau = cp.upd[1];
    for (int k0 = tid * V; k0 < P.Nv; k0 += NT * V) {
        T x[V][D], wv[V];
        load_nodes<D, V>(P, k0, x, wv);
        T Nn[NA][V], fv[NA][V];
#pragma unroll
        for (int a = 0; a < NA; ++a) {
            ldv_cg<T, V>(fi + (size_t)a * P.Nvp + k0, fv[a]);
#pragma unroll
            for (int v = 0; v < V; ++v) Nn[a][v] = T(0);
        }
#pragma unroll
        for (int s = 0; s < AVS_MAXS; ++s) {
            if (s >= ns) break;
            const T* Fs = P.F + (size_t)fs[s] * NA * P.Nvp + k0;
            const T g = sg[s];
#pragma unroll
            for (int a = 0; a < NA; ++a) {
                T t[V];
                ldv_cg<T, V>(Fs + (size_t)a * P.Nvp, t);
#pragma unroll
                for (int v = 0; v < V; ++v) Nn[a][v] += g * t[v];
            }
        }
        T out[NA][V];
#pragma unroll
        for (int v = 0; v < V; ++v) {
            T gG, gH;
            eq_eval<D>(cp.eq, x[v], gG, gH);
            const bool real = k0 + v < P.Nv;
            out[0][v] = real ? Vc * (gG - fv[0][v]) / tau - Nn[0][v] : T(0);
            if (NA == 2) out[NA - 1][v] = real ? Vc * (gH - fv[NA - 1][v]) / tau - Nn[NA - 1][v] : T(0);
        }
#pragma unroll
        for (int a = 0; a < NA; ++a) stv<T, V>(ro + (size_t)a * P.Nvp + k0, out[a]);
    }
}

// One colour of a microscopic sweep: dphi_i = (Res_i - sum_{xi.n<0} (xi.n) dphi_j)
// / (V/dt + V/tau~ + sum_{xi.n>=0} xi.n), every node and array.  V consecutive
// nodes per thread (16-byte vectors); a neighbour's row is read only where one
// of the thread's nodes flows in from it.  Pad nodes get dphi = 0.
template <int D, typename T, int NT, int V>
__global__ void __launch_bounds__(NT) k_imp_micro(CellP<D, T> P, const T* __restrict__ res, T* dphi,
                                                  const T* __restrict__ An, const int* __restrict__ faceL,
                                                  const int* __restrict__ faceR, const int* __restrict__ clist, int c0)
{
    constexpr int NA = NArr<D>::v;
    __shared__ T sA[AVS_MAXS][D];
    __shared__ int snb[AVS_MAXS];
    const int i = clist[c0 + blockIdx.x];
    const int ns = P.nslot[i];
    const int tid = threadIdx.x;
    if (tid < ns) {
        const int sl = P.slot[i * AVS_MAXS + tid];
        const int f = sl >> 1;
#pragma unroll
        for (int d = 0; d < D; ++d) sA[tid][d] = (sl & 1) ? -An[(size_t)f * D + d] : An[(size_t)f * D + d];
        snb[tid] = (sl & 1) ? faceL[f] : faceR[f];
    }
    __syncthreads();
    const int k0 = (blockIdx.y * NT + tid) * V;
    if (k0 >= P.Nv) return;
    const T u0 = P.par[i].upd[0];
    T x[V][D], wv[V];
    load_nodes<D, V>(P, k0, x, wv);
    T sn[AVS_MAXS][V], dg[V];
#pragma unroll
    for (int v = 0; v < V; ++v) dg[v] = T(0);
#pragma unroll
    for (int s = 0; s < AVS_MAXS; ++s) {
        if (s >= ns) break;
        T a[D];
#pragma unroll
        for (int d = 0; d < D; ++d) a[d] = sA[s][d];
#pragma unroll
        for (int v = 0; v < V; ++v) {
            sn[s][v] = dot_rn<D>(x[v], a);
            if (sn[s][v] >= T(0)) dg[v] += sn[s][v];
        }
    }
#pragma unroll
    for (int v = 0; v < V; ++v) dg[v] = u0 + dg[v];
#pragma unroll
    for (int a = 0; a < NA; ++a) {
        T acc[V];
        ldv_cg<T, V>(res + ((size_t)i * NA + a) * P.Nvp + k0, acc);
#pragma unroll
        for (int s = 0; s < AVS_MAXS; ++s) {
            if (s >= ns) break;
            const int j = snb[s];
            bool in = false;
#pragma unroll
            for (int v = 0; v < V; ++v) in |= sn[s][v] < T(0);
            if (j < 0 || !in) continue;
            T t[V];
            ldv_cg<T, V>(dphi + ((size_t)j * NA + a) * P.Nvp + k0, t);
#pragma unroll
            for (int v = 0; v < V; ++v)
                if (sn[s][v] < T(0)) acc[v] -= sn[s][v] * t[v];
        }
        T o[V];
#pragma unroll
        for (int v = 0; v < V; ++v) o[v] = k0 + v < P.Nv ? acc[v] / dg[v] : T(0);
        stv<T, V>(dphi + ((size_t)i * NA + a) * P.Nvp + k0, o);
    }
}

// f^{n+1} = f^n + dphi (pad nodes zero)
template <typename T>
__global__ void k_imp_finish(int Nrows, int Nv, int Nvp, const T* __restrict__ fin, const T* __restrict__ dphi,
                             T* fout)
{
    const int r = blockIdx.x;
    for (int k = blockIdx.y * blockDim.x + threadIdx.x; k < Nvp; k += gridDim.y * blockDim.x)
        fout[(size_t)r * Nvp + k] = k < Nv ? fin[(size_t)r * Nvp + k] + dphi[(size_t)r * Nvp + k] : T(0);
    (void)Nrows;
}

template <int D, typename T>
static cudaError_t launch_step_implicit_t(avs_ctx* c, const void* fin, void* fout, const double* Win, double* Wout,
                                          double dt, int k_macro, int k_micro)
{
    const bool f32 = sizeof(T) == 4;
    const int NA = NArr<D>::v, NW = D + 2;
    cudaError_t e = face_stage_t<D, T>(c, fin, Win, dt);
    if (e != cudaSuccess) return e;
    using A = T;     // macroscopic sweep arithmetic: FP32 in the mixed form, FP64 in the FP64 form
    ImpP<A> I;
    I.Nc = c->Nc;
    I.dt = dt;
    I.R = c->cfg.R;
    I.mu_ref = c->mu_ref;
    I.T_ref = c->cfg.T_ref;
    I.omega = c->cfg.omega;
    I.slot = c->slot;
    I.nslot = c->nslot;
    I.faceL = c->faceL;
    I.faceR = c->faceR;
    I.An = c->An_d;
    I.rL = c->rL_d;
    I.rR = c->rR_d;
    I.vol = c->vol;
    I.AF = c->AFf;
    I.Wn = Win;
    I.Wt = Wout;
    I.dWa = (A*)c->imp_dW;
    I.Wta = f32 ? (A*)c->imp_Wta : (A*)Wout;
    I.rhs = (A*)c->imp_rhs0;
    I.dg = (A*)c->imp_diag;
    I.co = (ImpSlot<A>*)c->imp_co;
    I.nint = c->imp_nint;
    I.clist = c->clist;
    I.err = c->dev_err;
    const int cb = (c->Nc + kCellNT - 1) / kCellNT;
    k_imp_setup<D, A><<<cb, kCellNT, 0, c->stream>>>(I);
    c->launches += 1;
    const int nc = c->ncolor;
    if (k_macro > 0) {
        // one cooperative launch: every block resident, so the bounded grid
        // barriers between colour passes can complete
        constexpr int NTM = 64;
        int maxcol = 0;
        for (int k = 0; k < nc; ++k) maxcol = std::max(maxcol, c->cstart[k + 1] - c->cstart[k]);
        const void* kern = D == 2 && c->max_ns <= 4 ? (const void*)k_imp_macro<D, A, NTM, D == 2 ? 4 : AVS_MAXS>
                                                    : (const void*)k_imp_macro<D, A, NTM, AVS_MAXS>;
        int dev = 0, nsm = 0, occ = 0;
        e = cudaGetDevice(&dev);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
        if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, NTM, 0);
        if (e != cudaSuccess) return e;
        const int nblk = std::max(1, std::min(nsm * std::max(occ, 1), (maxcol + NTM - 1) / NTM));
        e = cudaMemsetAsync(c->imp_bar, 0, sizeof(unsigned), c->stream);
        if (e != cudaSuccess) return e;
        int km = k_macro, ncol = nc;
        const int* cs = c->cstart_d;
        unsigned* bar = c->imp_bar;
        void* args[] = {&I, &km, &ncol, &cs, &bar};
        e = cudaLaunchCooperativeKernel(kern, dim3(nblk), dim3(NTM), args, 0, c->stream);
        if (e != cudaSuccess) return e;
        c->launches += 1;
    }
    // microscopic system
    const T* xi = f32 ? (const T*)c->xi_f : (const T*)c->xi_d;
    const T* w = f32 ? (const T*)c->w_f : (const T*)c->w_d;
    CellP<D, T> Q;
    Q.Nc = c->Nc;
    Q.Nv = c->Nv;
    Q.Nvp = c->Nvp;
    Q.cstride = (size_t)NA * c->Nvp;
    Q.dt = dt;
    Q.idt = 1.0 / dt;
    Q.R = c->cfg.R;
    Q.Pr = c->cfg.Pr;
    Q.omega = c->cfg.omega;
    Q.mu_ref = c->mu_ref;
    Q.T_ref = c->cfg.T_ref;
    Q.fin = (const T*)fin;
    Q.fout = (T*)fout;
    Q.F = (const T*)c->flux;
    Q.AF = c->AFf;
    Q.Win = Win;
    Q.Wout = Wout;
    Q.mom = c->cmom;
    Q.par = (CellPar<T>*)c->cpar;
    Q.xi = xi;
    Q.w = w;
    Q.slot = c->slot;
    Q.nslot = c->nslot;
    Q.vol = c->vol;
    Q.err = c->dev_err;
    constexpr int NT = 128;
    if (!c->mom_valid) {
        if constexpr (sizeof(T) == 4) {
            e = launch_raw32(c, fin, Win);
            if (e != cudaSuccess) return e;
        } else {
            k_raw_moments<D, NT, VW<T>::v><<<c->Nc, NT, 0, c->stream>>>(Q);
            c->launches += 1;
        }
    }
    k_imp_state<D, T><<<cb, kCellNT, 0, c->stream>>>(Q, Wout);
    c->launches += 1;
    if constexpr (sizeof(T) == 4) {
        e = launch_cell32(c, fin, fout, true);
        if (e == cudaSuccess) e = launch_micro32(c, fin, fout, nullptr, k_micro);
        if (e != cudaSuccess) return e;
    } else {
        k_imp_res<D, T, NT, VW<T>::v><<<c->Nc, NT, 0, c->stream>>>(Q);
        c->launches += 1;
        T* dphi = (T*)c->flux;                // the face flux has been used: its buffer holds dphi
        e = cudaMemsetAsync(dphi, 0, (size_t)c->Nc * NA * c->Nvp * sizeof(T), c->stream);
        if (e != cudaSuccess) return e;
        constexpr int VM = VW<T>::v;
        const int nyb = (c->Nv + NT * VM - 1) / (NT * VM);
        int prev = -1;
        for (int it = 0; it < k_micro; ++it)
            for (int dir = 0; dir < 2; ++dir)
                for (int q = 0; q < nc; ++q) {
                    const int col = dir == 0 ? q : nc - 1 - q;
                    if (col == prev) continue;      // the turn of a symmetric sweep: same inputs, same values
                    prev = col;
                    const int c0 = c->cstart[col], c1 = c->cstart[col + 1];
                    if (c1 > c0) {
                        dim3 g(c1 - c0, nyb);
                        k_imp_micro<D, T, NT, VM><<<g, NT, 0, c->stream>>>(Q, (const T*)fout, dphi, c->An_d, c->faceL,
                                                                            c->faceR, c->clist, c0);
                        c->launches += 1;
                    }
                }
        dim3 gf(c->Nc * NA, (c->Nvp + 255) / 256 < 8 ? (c->Nvp + 255) / 256 : 8);
        k_imp_finish<T><<<gf, 256, 0, c->stream>>>(c->Nc * NA, c->Nv, c->Nvp, (const T*)fin, dphi, (T*)fout);
        c->launches += 1;
    }
    c->mom_valid = 0;          // the carried moments are of f^n
    (void)NW;
    return cudaGetLastError();
}

cudaError_t launch_step_implicit(avs_ctx* c, const void* fin, void* fout, const double* Win, double* Wout, double dt,
                                 int k_macro, int k_micro)
{
    if (c->D == 2)
        return c->mixed ? launch_step_implicit_t<2, float>(c, fin, fout, Win, Wout, dt, k_macro, k_micro)
                        : launch_step_implicit_t<2, double>(c, fin, fout, Win, Wout, dt, k_macro, k_micro);
    return c->mixed ? launch_step_implicit_t<3, float>(c, fin, fout, Win, Wout, dt, k_macro, k_micro)
                    : launch_step_implicit_t<3, double>(c, fin, fout, Win, Wout, dt, k_macro, k_micro);
}

void launch_grad_rykov(avs_ctx* c, const void* fin)
{
    c->D == 2 ? grad_t<2, 3>(c, fin) : grad_t<3, 2>(c, fin);
}

cudaError_t launch_face_stage(avs_ctx* c, const void* fin, const double* Win, double dt)
{
    if (c->D == 2)
        return c->mixed ? face_stage_t<2, float>(c, fin, Win, dt) : face_stage_t<2, double>(c, fin, Win, dt);
    return c->mixed ? face_stage_t<3, float>(c, fin, Win, dt) : face_stage_t<3, double>(c, fin, Win, dt);
}

cudaError_t launch_step(avs_ctx* c, const void* fin, void* fout, const double* Win, double* Wout, double dt)
{
    if (c->D == 2)
        return c->mixed ? launch_step_t<2, float>(c, fin, fout, Win, Wout, dt)
                        : launch_step_t<2, double>(c, fin, fout, Win, Wout, dt);
    return c->mixed ? launch_step_t<3, float>(c, fin, fout, Win, Wout, dt)
                    : launch_step_t<3, double>(c, fin, fout, Win, Wout, dt);
}

}  // namespace avs
