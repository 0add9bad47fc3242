// Face and cell kernels of the FP32 form, for either gas.
//
// k_foot_f2 (avs_step.cu) writes each face's foot values once.  Here
//   k_face32   reads a face's row of foot values twice: for the raw moments of
//              the interface state, then for the interface distribution
//              phi = wa phi_bar + wb g_ij; it writes the per-node flux
//              (xi . An) phi over the row and the face's flux of W;
//   k_cell32   sums the flux rows of the cell's faces, updates f and carries
//              the raw moments of the new f.
// The gas is a type G: D, its arrays NA (G, in 2D H, with rotation ROT also R),
// raw moments NM and conserved values NW; the interface state and the
// equilibria (face_eq, face_phi, cell_eq); EXACT: the upwind choice is the FP64
// one (see upwind_sure).  Shakhov's is in avs_step32.cu, Rykov's in avs_rykov.cu.
// Measured on GB300, five steps of the sphere (36864 cells, 21372 nodes) and ten
// of the cylinder (12288 cells, 3522 nodes), face and cell kernel: 24.0 + 15.1
// and 2.62 + 2.43 ms; one face or cell per block with rows staged by bulk copies
// or loaded directly, before: 31.3 + 21.2 and 4.20 + 2.91 ms.  The Rykov
// cylinder (12288 cells, 3216 nodes, ten steps): 3.59 + 3.39 ms with 4.01 for the
// foot values, against 10.3 + 4.7 and 3.5 for stored gradients that the face
// kernel read.
// Forming phi and its flux in the cell kernel instead, without storing them,
// spares the stores but takes 126 more FP32 operations per cell and node in 3D
// and was no gain (29.2 + 27.2 and 2.63 + 4.51 ms).
#pragma once

#include <algorithm>
#include <type_traits>

#include "avs_dev.cuh"
#include "avs_internal.h"
#include "avs_step32.h"

namespace avs {

namespace {

constexpr float kTwoLn2 = 1.3862943611198906f;     // 2 ln 2

// four nodes k..k+3 (k a multiple of 4) of a planar array as two lane pairs
__device__ __forceinline__ void ld4(const float* __restrict__ p, float2 (&o)[2])
{
    const float4 v = __ldg(reinterpret_cast<const float4*>(p));
    o[0] = lo2(v);
    o[1] = hi2(v);
}
// the same past L1 (rows that are read once, or were written by another kernel of the step)
__device__ __forceinline__ void ld4cg(const float* p, float2 (&o)[2])
{
    const float4 v = __ldcg(reinterpret_cast<const float4*>(p));
    o[0] = lo2(v);
    o[1] = hi2(v);
}

// 16-byte asynchronous copies global -> shared memory of the calling thread's
// own data: no other thread reads what it copies, so a wait for its own groups
// is all the synchronisation there is.  The ring starts on 128 bytes: from a
// base 16 bytes off a sector each warp's 512-byte copy took 16 shared-memory
// wavefronts instead of 4 and read its global sectors twice.
__device__ __forceinline__ void cp16(float* dst, const float* src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait()
{
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}
__device__ __forceinline__ void lds4(const float* p, float2 (&o)[2])
{
    const float4 v = *reinterpret_cast<const float4*>(p);
    o[0] = lo2(v);
    o[1] = hi2(v);
}

// xi . An of a node pair in the order k_foot_f2 takes for its upwind choice
template <int D>
__device__ __forceinline__ float2 dot2(const float2* x, const float* a)
{
    float2 s = mul2(x[0], bc2(a[0]));
#pragma unroll
    for (int d = 1; d < D; ++d) s = fma2(x[d], bc2(a[d]), s);
    return s;
}
// xi . An of the flux, every product and sum rounded: the heat flux of a gas near
// equilibrium, a small difference of large sums, follows the rounding of each
// node's flux
template <int D>
__device__ __forceinline__ float2 dot2r(const float2* x, const float* a)
{
    float2 s = mul2(x[0], bc2(a[0]));
#pragma unroll
    for (int d = 1; d < D; ++d) s = add2(s, mul2(x[d], bc2(a[d])));
    return s;
}

// raw moments of a node pair (values o of the gas's arrays: G, in 2D H, for a
// gas with rotation R) about V, y = xi - V
template <class G>
__device__ __forceinline__ void pair_moments(float2* m, const float2* y, float2 w, const float2* o)
{
    constexpr int D = G::D, N0 = NMom<D>::v;
    raw_acc2<D>(m, y, mul2(w, o[0]), D == 2 ? mul2(w, o[D == 2 ? 1 : 0]) : bc2(0.0f));
    if constexpr (G::ROT) {
        const float2 wr = mul2(w, o[G::NA - 1]);
        m[N0] = add2(m[N0], wr);
#pragma unroll
        for (int d = 0; d < D; ++d) m[N0 + 1 + d] = fma2(wr, y[d], m[N0 + 1 + d]);
    }
}

// flux moments of a node pair (values o of the per-node flux): mass, momentum,
// twice the energy without rotation, and the rotational energy
template <class G>
__device__ __forceinline__ void flux_moments(float2* m, const float2* x, float2 x2, float2 w, const float2* o)
{
    constexpr int D = G::D;
    const float2 q = mul2(w, o[0]);
    m[0] = add2(m[0], q);
#pragma unroll
    for (int d = 0; d < D; ++d) m[1 + d] = fma2(q, x[d], m[1 + d]);
    m[D + 1] = fma2(q, x2, m[D + 1]);
    if constexpr (D == 2) m[D + 1] = fma2(w, o[1], m[D + 1]);
    if constexpr (G::ROT) m[D + 2] = fma2(w, o[G::NA - 1], m[D + 2]);
}
template <class G>
__device__ __forceinline__ void flux_sums(const float2* m, float* v)
{
    constexpr int D = G::D;
#pragma unroll
    for (int q = 0; q < G::NW; ++q) v[q] = m[q].x + m[q].y;
    v[D + 1] *= 0.5f;
    if constexpr (G::ROT) v[D + 1] += v[D + 2];
}

// ---------------------------------------------------------------- reductions
// Per-thread floats v[N] of a group of NT threads (NT a multiple of 32, its
// warps consecutive) summed into out[N] (shared memory, FP64 across warps).
// sw: (NT / 32) * N floats.  gsync synchronises the group.
template <int N, int NT, typename Sync>
__device__ __forceinline__ void group_sum(float* v, int t, float* sw, double* out, Sync gsync)
{
    static_assert(N <= 32, "one value per lane at most");
    int idx = 0, cnt = N;
    WarpSum<float, N, 16>::run(v, idx, cnt);
    if constexpr (NT == 32) {
        if (cnt > 0) out[idx] = to_double(v[0]);
    } else {
        if (cnt > 0) sw[(t >> 5) * N + idx] = v[0];
        gsync();
        if (t < N) {
            double s = to_double(sw[t]);
#pragma unroll
            for (int w = 1; w < NT / 32; ++w) s += to_double(sw[w * N + t]);
            out[t] = s;
        }
    }
    gsync();
}

// The cell kernels' sums go in runs of kCellRun quads of a thread: FP32 over a
// thread's quads of a run (two terms a quad and lane) and over the warp, FP64 over
// the runs and the warps, so that an FP32 chain has at most 16 terms however long
// the row.  As one run, a cell of one warp took 334 terms a lane for 21372 nodes;
// with 1000 (64000 nodes, the first ones outweighing the rest) the lagged heat flux
// came out 1.36 times too large, now 1.005.  The runs cost 0.5 % of a step of the
// sphere (65.3 -> 65.6 ms for five; runs of 16 quads the same).
constexpr int kCellRun = 8;
// one run: lane pairs m, which are cleared, added to the warp's sums; a lane with
// cnt > 0 holds that of value idx
template <int N>
__device__ __forceinline__ void run_sum(float2* m, double& sum, int& idx, int& cnt)
{
    static_assert(N <= 32, "one value per lane at most");
    float v[N];
#pragma unroll
    for (int q = 0; q < N; ++q) {
        v[q] = m[q].x + m[q].y;
        m[q] = bc2(0.0f);
    }
    idx = 0;
    cnt = N;
    WarpSum<float, N, 16>::run(v, idx, cnt);
    sum += to_double(v[0]);
}
// the last run, and the sums of all runs and warps into out[N]; sw: (NT / 32) * N
// doubles.  one: there was no run before, so nothing is added (a branch of its own:
// an FP64 addition is 16 cycles of an SM's pipe, predicated off or not; 190 nodes,
// 12288 cells, 20 steps: 2.078 -> 2.055 ms).
template <int N, int NT, typename Sync>
__device__ __forceinline__ void run_sums(float2* m, double sum, bool one, int t, double* sw, double* out, Sync gsync)
{
    double* const o = NT == 32 ? out : sw + (t >> 5) * N;
    int idx, cnt;
    if (one) {
        double s = -0.0;                         // x + -0 is x: no instruction
        run_sum<N>(m, s, idx, cnt);
        if (cnt > 0) o[idx] = s;
    } else {
        run_sum<N>(m, sum, idx, cnt);
        if (cnt > 0) o[idx] = sum;
    }
    if constexpr (NT > 32) {
        gsync();
        if (t < N) {
            double s = sw[t];
#pragma unroll
            for (int w = 1; w < NT / 32; ++w) s += sw[w * N + t];
            out[t] = s;
        }
    }
    gsync();
}

template <int NT>
__device__ __forceinline__ void group_bar(int id)
{
    if constexpr (NT == 32) {
        __syncwarp();
    } else {
        asm volatile("bar.sync %0, %1;" ::"r"(id), "n"(NT) : "memory");
    }
}

// ------------------------------------------------------------------ k_face32
// A group of NT threads takes FPT interior faces (consecutive in the face
// order, so mostly faces of one cell) or one boundary face; a block holds HG
// groups that do not wait on one another.  Each thread takes node quads, with
// the rows, coordinates and weights of its next quads on their way into a ring
// of STG slots of its own in shared memory (cp.async); a thread reads only what
// it copied, so the loops have no barrier, and the copies of pass B are in
// flight during the state.  The coordinates and weights are loaded once for the
// FPT faces: at one face per load they were 32 of the 44 bytes that a face and
// node moved from L2 to the SM in the two passes.  The moment basis is formed
// once too, about the faces' common reference velocity, where their own (the mean
// of the two cells') lie close together: within (1/16 of the least internal
// energy)^(1/2), so that the mean is at most 0.16 sqrt(R T) from either and the
// central moments cancel no large terms.  Elsewhere (a shock, the first cells at a
// wall, faces far apart that follow each other in the order) each face has its own
// basis: with a stream at 24 sqrt(R T) beside gas at rest, numbered at random, the
// common one left an error of 9e-7 in the energy of the gas at rest after one step,
// its own 8e-9.  (Two loops and not a choice within one, which spilled.)
template <class G>
struct Face32P {
    int Nv, Nvp, Nfi, Nf;
    double hd;
    double R;
    typename G::Consts g;
    float* FB;               // [face][array][Nvp] foot values in, per-node flux out
    double* AF;              // [face][NW] area-weighted flux of W
    const double* Win;
    const float* xs;         // node coordinates by components [D][xstride]
    const float* w;
    size_t xstride;
    const int* order;        // interior faces, then boundary faces
    const int* faceL;
    const int* faceR;
    const float* An;
    const double* bc;
    const double* xid;       // FP64 coordinates and normals: G::EXACT
    const double* And;
    int* err;
};

template <class G, int FPT, int NT>
struct Face32S {
    static constexpr int NM = G::NM;
    double red[FPT * NM];
    float sw[(NT / 32) * FPT * NM];
    float V[FPT][3];
    float e[FPT];            // least translational energy of the face's cells, 3/2 R T
    float An[FPT][4];
    typename G::Eq eq[FPT];
};

template <class G, int FPT, int NT, int HG, int STG>
__global__ void __launch_bounds__(NT * HG, (NT * HG == 64 ? 8 : NT * HG == 128 ? (FPT > 2 ? 3 : 4) : 2)) k_face32(Face32P<G> P)
{
    constexpr int D = G::D, NA = G::NA, NM = G::NM, NW = G::NW, CH = 4 * NT;
    constexpr int NR = FPT * NA + D + 1;         // rows of a slot: foot values, coordinates, weights
    extern __shared__ __align__(128) float ring[];   // [slot][row][thread] of four nodes
    __shared__ Face32S<G, FPT, NT> SH[HG];
    const int half = threadIdx.x / NT, t = threadIdx.x % NT;
    Face32S<G, FPT, NT>& S = SH[half];
    auto gsync = [&]() { group_bar<NT>(1 + half); };
    const int ng = (P.Nfi + FPT - 1) / FPT;
    const int g = blockIdx.x * HG + half;
    const int Nv = P.Nv, Nvp = P.Nvp;
    const size_t rowlen = (size_t)NA * Nvp;
    if (g >= ng) {
        // ---------------- one boundary face: outgoing foot values, incoming Maxwellian
        const int b = P.Nfi + (g - ng);
        if (b >= P.Nf) return;
        const int f = P.order[b];
        const double* B = P.bc + (size_t)(-1 - P.faceR[f]) * 6;
        const bool wall = (int)B[0] == AVS_BC_WALL;
        const double Ub[3] = {B[2], B[3], B[4]};
        EqPar<float> eb = make_eq<D, float>(wall ? 1.0 : B[1], Ub, P.R * B[5], nullptr, 1.0);
        float An[D];
#pragma unroll
        for (int d = 0; d < D; ++d) An[d] = P.An[(size_t)f * D + d];
        float* row = P.FB + (size_t)f * rowlen;
        const float RTb = (float)(P.R * B[5]);   // H = R T G in 2D, R = R T G
        // a quad's coordinates, normal velocities and values: foot value out
        // (at sn >= 0, k_foot_f2's upwind choice), Maxwellian in
        auto quad = [&](int k, float2 (&X)[D][2], float2 (&sn)[2], bool (&up)[4], float2 (&v)[NA][2]) {
#pragma unroll
            for (int a = 0; a < NA; ++a) ld4cg(row + (size_t)a * Nvp + k, v[a]);
#pragma unroll
            for (int d = 0; d < D; ++d) ld4(P.xs + d * P.xstride + k, X[d]);
#pragma unroll
            for (int p = 0; p < 2; ++p) {
                float2 x[D];
#pragma unroll
                for (int d = 0; d < D; ++d) x[d] = X[d][p];
                sn[p] = dot2<D>(x, An);
                up[2 * p] = sn[p].x >= 0.0f;
                up[2 * p + 1] = sn[p].y >= 0.0f;
                float2 c = add2(x[0], bc2(-eb.U[0])), c2 = mul2(c, c);
#pragma unroll
                for (int d = 1; d < D; ++d) {
                    c = add2(x[d], bc2(-eb.U[d]));
                    c2 = fma2(c, c, c2);
                }
                const float2 e = fma2(c2, bc2(eb.k2), bc2(eb.l2pref));
                const float2 g = make_float2(ex2_approx(e.x), ex2_approx(e.y));
                if constexpr (G::EXACT) {
#pragma unroll
                    for (int z = 0; z < 2; ++z) {
                        float xz[D];
#pragma unroll
                        for (int d = 0; d < D; ++d) xz[d] = z ? x[d].y : x[d].x;
                        const int kn = k + 2 * p + z;
                        if (!upwind_sure<D>(xz, An, z ? sn[p].y : sn[p].x) && !upwind_zero<D>(xz, An) && kn < Nv)
                            up[2 * p + z] = upwind_exact<D>(P.xid + (size_t)kn * D, P.And + (size_t)f * D, false);
                    }
                }
#pragma unroll
                for (int a = 0; a < NA; ++a) {
                    const float2 ga = a == 0 ? g : mul2(bc2(RTb), g);
                    v[a][p] = make_float2(up[2 * p] ? v[a][p].x : ga.x, up[2 * p + 1] ? v[a][p].y : ga.y);
                }
            }
        };
        float2 m[2][NW];                         // moments out, moments in
#pragma unroll
        for (int q = 0; q < NW; ++q) m[0][q] = m[1][q] = bc2(0.0f);
        for (int k = t * 4; k < Nv; k += NT * 4) {
            float2 X[D][2], sn[2], v[NA][2], W2[2];
            bool up[4];
            quad(k, X, sn, up, v);
            ld4(P.w + k, W2);
#pragma unroll
            for (int p = 0; p < 2; ++p) {
                float2 x[D], o[NA], in[NA], x2 = mul2(X[0][p], X[0][p]);
#pragma unroll
                for (int d = 0; d < D; ++d) x[d] = X[d][p];
#pragma unroll
                for (int d = 1; d < D; ++d) x2 = fma2(x[d], x[d], x2);
#pragma unroll
                for (int a = 0; a < NA; ++a) {
                    const float2 q = mul2(sn[p], v[a][p]);
                    o[a] = make_float2(up[2 * p] ? q.x : 0.0f, up[2 * p + 1] ? q.y : 0.0f);
                    in[a] = make_float2(up[2 * p] ? 0.0f : q.x, up[2 * p + 1] ? 0.0f : q.y);
                }
                flux_moments<G>(m[0], x, x2, W2[p], o);
                flux_moments<G>(m[1], x, x2, W2[p], in);
            }
        }
        float acc[2 * NW];
        flux_sums<G>(m[0], acc);
        flux_sums<G>(m[1], acc + NW);
        group_sum<2 * NW, NT>(acc, t, S.sw, S.red, gsync);
        double rw = 1.0;
        if (wall) {
            const double Sin = -S.red[NW];       // incoming mass flux of the unit-density wall Maxwellian
            rw = Sin > 0.0 ? S.red[0] / Sin : 0.0;
            eb = make_eq<D, float>(rw, Ub, P.R * B[5], nullptr, 1.0);
        }
        if (t == 0)
            for (int q = 0; q < NW; ++q) P.AF[(size_t)f * NW + q] = S.red[q] + rw * S.red[NW + q];
        for (int k = t * 4; k < Nv; k += NT * 4) {
            float2 X[D][2], sn[2], v[NA][2];
            bool up[4];
            quad(k, X, sn, up, v);
#pragma unroll
            for (int a = 0; a < NA; ++a) {
                const float2 o0 = mul2(sn[0], v[a][0]), o1 = mul2(sn[1], v[a][1]);
                *reinterpret_cast<float4*>(row + (size_t)a * Nvp + k) = make_float4(o0.x, o0.y, o1.x, o1.y);
            }
        }
        return;
    }
    // ---------------- FPT interior faces (the last group repeats its last face)
    float* row[FPT];
#pragma unroll
    for (int j = 0; j < FPT; ++j) row[j] = P.FB + (size_t)P.order[min(g * FPT + j, P.Nfi - 1)] * rowlen;
    // the thread's quads k = 4 t, 4 t + CH, ..; numbers 0..nq-1 in pass A, nq..2nq-1 in pass B
    const int nq = (Nv - 4 * t + CH - 1) / CH, ntot = 2 * nq;
    auto node = [&](int q) { return (q < nq ? q : q - nq) * CH + t * 4; };
    float* const my = ring + (size_t)threadIdx.x * 4;
    constexpr int RS = NT * HG * 4;              // floats per row of a slot
    auto fetch = [&](int q, int slot) {
        if (q < ntot) {
            const int k = node(q);
            float* dst = my + (size_t)slot * NR * RS;
#pragma unroll
            for (int j = 0; j < FPT; ++j)
#pragma unroll
                for (int a = 0; a < NA; ++a) cp16(dst + (j * NA + a) * RS, row[j] + (size_t)a * Nvp + k);
#pragma unroll
            for (int d = 0; d < D; ++d) cp16(dst + (FPT * NA + d) * RS, P.xs + d * P.xstride + k);
            cp16(dst + (FPT * NA + D) * RS, P.w + k);
        }
        cp_commit();
    };
#pragma unroll
    for (int q = 0; q < STG - 1; ++q) fetch(q, q);
    if (t < FPT) {
        const int f = P.order[min(g * FPT + t, P.Nfi - 1)];
        const double *WL = P.Win + (size_t)P.faceL[f] * NW, *WR = P.Win + (size_t)P.faceR[f] * NW;
        const float rL = (float)WL[0], rR = (float)WR[0];
        float kL = 0.0f, kR = 0.0f;
#pragma unroll
        for (int d = 0; d < D; ++d) {
            const float uL = (float)WL[1 + d] / rL, uR = (float)WR[1 + d] / rR;
            S.An[t][d] = P.An[(size_t)f * D + d];
            S.V[t][d] = 0.5f * (uL + uR);
            kL = fmaf(0.5f * uL, uL, kL);
            kR = fmaf(0.5f * uR, uR, kR);
        }
        if constexpr (FPT > 1) {
            float eL = (float)WL[D + 1], eR = (float)WR[D + 1];
            if constexpr (G::ROT) {
                eL -= (float)WL[D + 2];
                eR -= (float)WR[D + 2];
            }
            S.e[t] = fminf(fdiv(eL, rL) - kL, fdiv(eR, rR) - kR);
        }
    }
    gsync();
    int slot = 0;
    // the thread's next quad: its copies are waited for, and the ones STG - 1
    // quads ahead are started into the slot read in the iteration before
    auto next = [&](int q, float2 (&X)[D][2], float2 (&W2)[2], float2 (&F)[FPT][NA][2]) {
        cp_wait<STG - 2>();
        const float* src = my + (size_t)slot * NR * RS;
#pragma unroll
        for (int j = 0; j < FPT; ++j)
#pragma unroll
            for (int a = 0; a < NA; ++a) lds4(src + (j * NA + a) * RS, F[j][a]);
#pragma unroll
        for (int d = 0; d < D; ++d) lds4(src + (FPT * NA + d) * RS, X[d]);
        lds4(src + (FPT * NA + D) * RS, W2);
        fetch(q + STG - 1, slot == 0 ? STG - 1 : slot - 1);
        slot = slot + 1 == STG ? 0 : slot + 1;
    };
    float V[D];                                  // reference velocity: of the group, or of its first face
    bool common = true;
#pragma unroll
    for (int d = 0; d < D; ++d) V[d] = S.V[0][d];
    if constexpr (FPT > 1) {
        static_assert(FPT == 2, "two faces per group at most");
        float dv = 0.0f;
#pragma unroll
        for (int d = 0; d < D; ++d) dv = fmaf(S.V[1][d] - V[d], S.V[1][d] - V[d], dv);
        common = dv <= 0.0625f * fminf(S.e[0], S.e[1]);
        if (common) {
#pragma unroll
            for (int d = 0; d < D; ++d) V[d] = 0.5f * (V[d] + S.V[1][d]);
        }
    }
    // ---------------- pass A: raw moments about V
    {
        float2 m[FPT][NM];
#pragma unroll
        for (int j = 0; j < FPT; ++j)
#pragma unroll
            for (int q = 0; q < NM; ++q) m[j][q] = bc2(0.0f);
        auto sums = [&](auto one) {              // one: the basis about V serves every face
            for (int q0 = 0; q0 < nq; ++q0) {    // pad nodes of the last quad carry w = 0
                float2 X[D][2], W2[2], F[FPT][NA][2];
                next(q0, X, W2, F);
#pragma unroll
                for (int p = 0; p < 2; ++p) {
                    // basis in the order of raw_acc: 1, y, y y (upper triangle), y s
                    constexpr int NG = 1 + D + D * (D + 1) / 2 + D;
                    float2 b[NG];
#pragma unroll
                    for (int j = 0; j < FPT; ++j) {
                        if (j == 0 || !decltype(one)::value) {
                            float2 y[D], wy[D];
#pragma unroll
                            for (int d = 0; d < D; ++d) {
                                y[d] = add2(X[d][p], bc2(-(j == 0 ? V[d] : S.V[j][d])));
                                wy[d] = mul2(W2[p], y[d]);
                            }
                            float2 s = mul2(y[0], y[0]);
#pragma unroll
                            for (int d = 1; d < D; ++d) s = fma2(y[d], y[d], s);
                            int q = 0;
                            b[q++] = W2[p];
#pragma unroll
                            for (int d = 0; d < D; ++d) b[q++] = wy[d];
#pragma unroll
                            for (int d = 0; d < D; ++d)
#pragma unroll
                                for (int e = d; e < D; ++e) b[q++] = mul2(wy[d], y[e]);
#pragma unroll
                            for (int d = 0; d < D; ++d) b[q++] = mul2(wy[d], s);
                        }
#pragma unroll
                        for (int z = 0; z < NG; ++z) m[j][z] = fma2(b[z], F[j][0][p], m[j][z]);
#pragma unroll
                        for (int a = 1; a < NA; ++a)
#pragma unroll
                            for (int z = 0; z <= D; ++z) {
                                const int mz = NG + (a - 1) * (D + 1) + z;
                                m[j][mz] = fma2(b[z], F[j][a][p], m[j][mz]);
                            }
                    }
                }
            }
        };
        if (FPT == 1 || common) sums(std::true_type{});
        else if constexpr (FPT > 1) sums(std::false_type{});
        if constexpr (FPT * NM <= 32) {
            float v[FPT * NM];
#pragma unroll
            for (int j = 0; j < FPT; ++j)
#pragma unroll
                for (int q = 0; q < NM; ++q) v[j * NM + q] = m[j][q].x + m[j][q].y;
            group_sum<FPT * NM, NT>(v, t, S.sw, S.red, gsync);
        } else {
#pragma unroll
            for (int j = 0; j < FPT; ++j) {
                float v[NM];
#pragma unroll
                for (int q = 0; q < NM; ++q) v[q] = m[j][q].x + m[j][q].y;
                group_sum<NM, NT>(v, t, S.sw, S.red + j * NM, gsync);
            }
        }
    }
    if (t < FPT) {
        const float* Vt = common ? V : S.V[t];
        const double Vd[3] = {(double)Vt[0], (double)Vt[1], D == 3 ? (double)Vt[D - 1] : 0.0};
        S.eq[t] = G::face_eq(P.g, P.hd, S.red + t * NM, Vd, P.err);
    }
    gsync();
    // ---------------- pass B: per-node flux and flux moments of phi_ij = wa phi_bar + wb g_ij
    {
        float2 m[FPT][NW];
        typename G::Eq e[FPT];
        float An[FPT][D];
#pragma unroll
        for (int j = 0; j < FPT; ++j) {
            e[j] = S.eq[j];
#pragma unroll
            for (int d = 0; d < D; ++d) An[j][d] = S.An[j][d];
#pragma unroll
            for (int q = 0; q < NW; ++q) m[j][q] = bc2(0.0f);
        }
        // a group past the end repeats its last face: the copies write the
        // same values, except that pass B overwrites its own input
        const int nf = min(FPT, P.Nfi - g * FPT);
        for (int q0 = nq; q0 < ntot; ++q0) {
            const int k = node(q0);
            {
                float2 X[D][2], W2[2], F[FPT][NA][2];
                next(q0, X, W2, F);
                float2 hx2[2];
#pragma unroll
                for (int p = 0; p < 2; ++p) {
                    hx2[p] = mul2(X[0][p], X[0][p]);
#pragma unroll
                    for (int d = 1; d < D; ++d) hx2[p] = fma2(X[d][p], X[d][p], hx2[p]);
                }
#pragma unroll
                for (int j = 0; j < FPT; ++j) {
                    float2 o[NA][2];
#pragma unroll
                    for (int p = 0; p < 2; ++p) {
                        float2 x[D];
#pragma unroll
                        for (int d = 0; d < D; ++d) x[d] = X[d][p];
                        const float2 sn = dot2r<D>(x, An[j]);
                        float2 F1[NA], o1[NA];
#pragma unroll
                        for (int a = 0; a < NA; ++a) F1[a] = F[j][a][p];
                        G::face_phi(e[j], x, F1, o1);
#pragma unroll
                        for (int a = 0; a < NA; ++a) o[a][p] = o1[a] = mul2(sn, o1[a]);
                        flux_moments<G>(m[j], x, hx2[p], W2[p], o1);
                    }
                    if (j < nf) {
#pragma unroll
                        for (int a = 0; a < NA; ++a)
                            *reinterpret_cast<float4*>(row[j] + (size_t)a * Nvp + k) =
                                make_float4(o[a][0].x, o[a][0].y, o[a][1].x, o[a][1].y);
                    }
                }
            }
        }
        float v[FPT * NW];
#pragma unroll
        for (int j = 0; j < FPT; ++j) flux_sums<G>(m[j], v + j * NW);
        group_sum<FPT * NW, NT>(v, t, S.sw, S.red, gsync);
        if (t < FPT * NW) {
            const int j = t / NW;
            if (j < nf) P.AF[(size_t)P.order[g * FPT + j] * NW + t % NW] = S.red[t];
        }
    }
}

// ------------------------------------------------------------------ k_cell32
// One block of NT threads per cell.  out = (u0 f + u1 g~ + un N) u3 per node, N the
// net flux of the cell's faces: the collision update (diagonal of Eq. SGS_phi)
// with 1/dt, 1/tau~, -1/|V| and 1 / (1/dt + 1/tau~), or the residual of the
// implicit step with -|V|/tau~, |V|/tau~, -1 and 1 (RES).  Each thread
// takes node quads, the rows of its next quads on their way into its own ring of
// STG slots in shared memory, as in k_face32.  The kernel moves one row of f in
// and out and the flux rows of the cell's faces (2D: four faces of two arrays,
// 3D: six faces).  RES = false also sums the raw moments of the new f about U(W~)
// (P.mom), in the node order that k_raw32 repeats, so that carried and
// recomputed moments are equal bit for bit.  (The update with
// u0 u3, u1 u3 and un u3 formed first takes two instructions less per value, no
// time, and rounds f differently: the heat flux of a gas near equilibrium, a
// small difference of large sums, moved by 2e-5 of itself.)
template <class G>
struct Cell32P {
    int Nc, Nv, Nvp;
    const float* fin;
    float* fout;
    const float* F;          // [face][array][Nvp] per-node flux
    const typename G::Par* par;
    const double* W;         // k_raw32: W of the reference velocity
    double* mom;
    const float* xs;
    const float* w;
    size_t xstride;
    const int* slot;
    const unsigned char* nslot;
    int* err;
};

template <class G, int NT, int STG, bool RES>
__global__ void __launch_bounds__(NT, NT == 32 ? 16 : 4) k_cell32(Cell32P<G> P, int nrow)
{
    constexpr int D = G::D, NA = G::NA, NM = G::NM, CH = 4 * NT, RS = 4 * NT;
    using Par = typename G::Par;
    extern __shared__ __align__(128) float ring[];   // [slot][row][thread]: coordinates, weights, f, fluxes
    __shared__ Par cp;
    __shared__ int fs[AVS_MAXS];
    __shared__ float sg[AVS_MAXS];
    __shared__ double sw[(NT / 32) * NM], red[NM];
    const int t = threadIdx.x;
    const int i = blockIdx.x;
    const int ns = P.nslot[i];
    const int Nv = P.Nv, Nvp = P.Nvp;
    const float* fi = P.fin + (size_t)i * NA * Nvp;
    float* fo = P.fout + (size_t)i * NA * Nvp;
    if (t < ns) {
        const int sl = P.slot[i * AVS_MAXS + t];
        fs[t] = sl >> 1;
        sg[t] = (sl & 1) ? -1.0f : 1.0f;
    }
    static_assert(sizeof(Par) / 4 <= 32, "copied by one warp");
    if (t < (int)(sizeof(Par) / 4)) reinterpret_cast<float*>(&cp)[t] = reinterpret_cast<const float*>(P.par + i)[t];
    group_bar<NT>(1);
    const int nq = (Nv - 4 * t + CH - 1) / CH;
    float* const my = ring + t * 4;
    auto fetch = [&](int q, int slot) {
        if (q < nq) {
            const int k = q * CH + t * 4;
            float* dst = my + (size_t)slot * nrow * RS;
#pragma unroll
            for (int d = 0; d < D; ++d) cp16(dst + d * RS, P.xs + d * P.xstride + k);
            if constexpr (!RES) cp16(dst + D * RS, P.w + k);
#pragma unroll
            for (int a = 0; a < NA; ++a) cp16(dst + (D + 1 + a) * RS, fi + (size_t)a * Nvp + k);
#pragma unroll
            for (int s = 0; s < AVS_MAXS; ++s) {
                if (s >= ns) break;
#pragma unroll
                for (int a = 0; a < NA; ++a)
                    cp16(dst + (D + 1 + NA * (1 + s) + a) * RS, P.F + ((size_t)fs[s] * NA + a) * Nvp + k);
            }
        }
        cp_commit();
    };
#pragma unroll
    for (int q = 0; q < STG - 1; ++q) fetch(q, q);
    float2 m[RES ? 1 : NM];
    double sum = 0.0;
    const int nall = (Nv + 3) / CH;              // quads that every thread has
    if constexpr (!RES) {
#pragma unroll
        for (int q = 0; q < NM; ++q) m[q] = bc2(0.0f);
    }
    int slot = 0;
    for (int q0 = 0; q0 < nq; q0 += kCellRun) {
        for (int q = q0; q < min(nq, q0 + kCellRun); ++q) {
            const int k = q * CH + t * 4;
            cp_wait<STG - 2>();
            const float* src = my + (size_t)slot * nrow * RS;
            float2 X[D][2], W2[2], f0[NA][2], N[NA][2], o[NA][2];
#pragma unroll
            for (int d = 0; d < D; ++d) lds4(src + d * RS, X[d]);
            if constexpr (!RES) lds4(src + D * RS, W2);
#pragma unroll
            for (int a = 0; a < NA; ++a) {
                lds4(src + (D + 1 + a) * RS, f0[a]);
                N[a][0] = N[a][1] = bc2(0.0f);
            }
#pragma unroll
            for (int s = 0; s < AVS_MAXS; ++s) {
                if (s >= ns) break;
                const float2 g = bc2(sg[s]);
#pragma unroll
                for (int a = 0; a < NA; ++a) {
                    float2 F[2];
                    lds4(src + (D + 1 + NA * (1 + s) + a) * RS, F);
#pragma unroll
                    for (int p = 0; p < 2; ++p) N[a][p] = fma2(g, F[p], N[a][p]);
                }
            }
            fetch(q + STG - 1, slot == 0 ? STG - 1 : slot - 1);
            slot = slot + 1 == STG ? 0 : slot + 1;
#pragma unroll
            for (int p = 0; p < 2; ++p) {
                float2 x[D], y[D], g[NA];
#pragma unroll
                for (int d = 0; d < D; ++d) x[d] = X[d][p];
                G::cell_eq(cp, x, g);
#pragma unroll
                for (int a = 0; a < NA; ++a)
                    o[a][p] = mul2(fma2(N[a][p], bc2(cp.un), fma2(f0[a][p], bc2(cp.u0), mul2(g[a], bc2(cp.u1)))), bc2(cp.u3));
                if (k + 4 > Nv) {                    // the last quad's pad nodes are stored as zero
                    const bool r0 = k + 2 * p < Nv, r1 = k + 2 * p + 1 < Nv;
#pragma unroll
                    for (int a = 0; a < NA; ++a) o[a][p] = make_float2(r0 ? o[a][p].x : 0.0f, r1 ? o[a][p].y : 0.0f);
                }
                if constexpr (!RES) {
                    float2 v[NA];
#pragma unroll
                    for (int a = 0; a < NA; ++a) v[a] = o[a][p];
#pragma unroll
                    for (int d = 0; d < D; ++d) y[d] = add2(x[d], bc2(-cp.V[d]));
                    pair_moments<G>(m, y, W2[p], v);
                }
            }
#pragma unroll
            for (int a = 0; a < NA; ++a)
                *reinterpret_cast<float4*>(fo + (size_t)a * Nvp + k) =
                    make_float4(o[a][0].x, o[a][0].y, o[a][1].x, o[a][1].y);
        }
        if constexpr (!RES)
            if (q0 + kCellRun <= nall) {
                int idx, cnt;
                run_sum<NM>(m, sum, idx, cnt);
            }
    }
    if constexpr (!RES) {
        run_sums<NM, NT>(m, sum, nall < kCellRun, t, sw, red, [] { group_bar<NT>(1); });
        if (t < NM) P.mom[(size_t)i * NM + t] = red[t];
    }
}

// Raw moments of the own f of every cell about its U(W) in k_cell32's node
// order; after anything but a step changed f or W.
template <class G, int NT>
__global__ void __launch_bounds__(NT) k_raw32(Cell32P<G> P)
{
    constexpr int D = G::D, NA = G::NA, NM = G::NM, NW = G::NW;
    __shared__ double sw[(NT / 32) * NM], red[NM];
    const int t = threadIdx.x, i = blockIdx.x;
    float V[D];
#pragma unroll
    for (int d = 0; d < D; ++d) V[d] = G::vref(P.W + (size_t)i * NW, d);
    const float* fi = P.fin + (size_t)i * NA * P.Nvp;
    float2 m[NM];
#pragma unroll
    for (int q = 0; q < NM; ++q) m[q] = bc2(0.0f);
    const int nq = (P.Nv - 4 * t + 4 * NT - 1) / (4 * NT), nall = (P.Nv + 3) / (4 * NT);
    double sum = 0.0;
    for (int q0 = 0; q0 < nq; q0 += kCellRun) {
        for (int q = q0; q < min(nq, q0 + kCellRun); ++q) {
            const int k = (q * NT + t) * 4;
            float2 X[D][2], W2[2], F[NA][2];
#pragma unroll
            for (int d = 0; d < D; ++d) ld4(P.xs + d * P.xstride + k, X[d]);
            ld4(P.w + k, W2);
#pragma unroll
            for (int a = 0; a < NA; ++a) ld4cg(fi + (size_t)a * P.Nvp + k, F[a]);
#pragma unroll
            for (int p = 0; p < 2; ++p) {
                float2 y[D], v[NA];
#pragma unroll
                for (int d = 0; d < D; ++d) y[d] = add2(X[d][p], bc2(-V[d]));
#pragma unroll
                for (int a = 0; a < NA; ++a) v[a] = F[a][p];
                pair_moments<G>(m, y, W2[p], v);
            }
        }
        if (q0 + kCellRun <= nall) {
            int idx, cnt;
            run_sum<NM>(m, sum, idx, cnt);
        }
    }
    run_sums<NM, NT>(m, sum, nall < kCellRun, t, sw, red, [] { group_bar<NT>(1); });
    if (t < NM) P.mom[(size_t)i * NM + t] = red[t];
}

// ------------------------------------------------------------------ launchers
template <class G>
cudaError_t face32_t(avs_ctx* c, const double* Win, double dt, const typename G::Consts& g)
{
    constexpr int D = G::D, NA = G::NA;
    Face32P<G> P;
    P.Nv = c->Nv;
    P.Nvp = c->Nvp;
    P.Nfi = c->Nfi;
    P.Nf = c->Nf;
    P.hd = 0.5 * dt;
    P.R = c->cfg.R;
    P.g = g;
    P.FB = (float*)c->flux;
    P.AF = c->AFf;
    P.Win = Win;
    P.xs = c->xi_s;
    P.w = c->w_f;
    P.xstride = c->xstride;
    P.order = c->iorder;
    P.faceL = c->faceL;
    P.faceR = c->faceR;
    P.An = c->An_f;
    P.bc = c->bc;
    P.xid = c->xi_d;
    P.And = c->An_d;
    P.err = c->dev_err;
    cudaError_t e = cudaSuccess;
    auto go = [&](auto fpt, auto nt, auto hg, auto stg) {
        constexpr int FPT = decltype(fpt)::value, NT = decltype(nt)::value, HG = decltype(hg)::value;
        constexpr int STG = decltype(stg)::value;
        constexpr size_t smem = (size_t)STG * (FPT * NA + D + 1) * NT * HG * 16;
        if (smem > 40 * 1024)
            e = cudaFuncSetAttribute(k_face32<G, FPT, NT, HG, STG>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)smem);
        if (e != cudaSuccess) return;
        const int groups = (c->Nfi + FPT - 1) / FPT + (c->Nf - c->Nfi);
        k_face32<G, FPT, NT, HG, STG><<<(groups + HG - 1) / HG, NT * HG, smem, c->stream>>>(P);
    };
    using std::integral_constant;
    using I1 = integral_constant<int, 1>;
    using I2 = integral_constant<int, 2>;
    using I4 = integral_constant<int, 4>;
    using N32 = integral_constant<int, 32>;
    using N64 = integral_constant<int, 64>;
    using N128 = integral_constant<int, 128>;
    using I3 = integral_constant<int, 3>;
    // Short rows (a few quads per lane): one warp per group, so that a group's
    // reductions and serial state hold no other warp.  Beyond, 64 threads, eight
    // groups per SM, so that some are in their loops while others wait for their
    // states (3D, 6783 cells x 2197 nodes, ten steps: 1.17 ms, 128 threads 1.53;
    // 2D, 12288 x 3522: 2.63 against 2.74); for rows over 48 KB 128 threads, whose
    // fewer rows in flight pass B still finds in L2 (2D, 12k nodes, four steps:
    // 10.9 against 12.8 ms; 3D, 21k, five steps: 24.0 against 24.2).  Two faces per
    // group where that leaves groups enough to fill the SMs (190 nodes, 24672
    // faces, 20 steps: 0.73 ms, one face 1.04 ms).  Slots of the ring: three, or
    // four in 3D and for long rows, again for L2 (12k nodes in 2D 10.9 against
    // 12.5 ms; 21k in 3D 24.0 against 25.7; 2D, 39 kB a row, 4.11 with four, 3.67
    // with three, in groups of 128).
    if (c->Nv <= 512 || (c->Nv <= 1024 && c->Nf >= 32 * c->nsm)) {
        if (c->Nf >= 16 * c->nsm) go(I2{}, N32{}, I4{}, I3{});
        else go(I1{}, N32{}, I4{}, I3{});
    } else if (c->Nf < 4 * c->nsm) {
        go(I1{}, N128{}, I1{}, I3{});
    } else if ((size_t)NA * c->Nvp * sizeof(float) > 49152) {
        go(I2{}, N128{}, I1{}, I4{});
    } else {
        go(I2{}, N64{}, I1{}, integral_constant<int, D == 3 ? 4 : 3>{});
    }
    if (e != cudaSuccess) return e;
    c->launches += 1;
    return cudaGetLastError();
}

template <class G>
Cell32P<G> cell_params(avs_ctx* c, const void* fin, void* fout, const double* W)
{
    Cell32P<G> P;
    P.Nc = c->Nc;
    P.Nv = c->Nv;
    P.Nvp = c->Nvp;
    P.fin = (const float*)fin;
    P.fout = (float*)fout;
    P.F = (const float*)c->flux;
    P.par = (const typename G::Par*)c->cpar;
    P.W = W;
    P.mom = c->cmom;
    P.xs = c->xi_s;
    P.w = c->w_f;
    P.xstride = c->xstride;
    P.slot = c->slot;
    P.nslot = c->nslot;
    P.err = c->dev_err;
    return P;
}

// one warp per cell where the cells fill the SMs with such blocks or the rows are short
inline bool warp_cells(const avs_ctx* c) { return c->Nv <= 256 || c->Nc >= 16 * c->nsm; }

template <class G, bool RES>
cudaError_t cell32_t(avs_ctx* c, const void* fin, void* fout)
{
    constexpr int D = G::D;
    const Cell32P<G> P = cell_params<G>(c, fin, fout, nullptr);
    const int nrow = D + 1 + G::NA * (1 + c->max_ns);
    auto go = [&](auto nt) -> cudaError_t {
        constexpr int NT = decltype(nt)::value, STG = 3;
        const size_t smem = (size_t)STG * nrow * NT * 16;
        // the limit is a property of the kernel, shared by every context: always
        // the most any mesh needs, never one mesh's own size, which another
        // thread's smaller one could replace before the launch
        constexpr size_t most = (size_t)STG * (D + 1 + G::NA * (1 + AVS_MAXS)) * NT * 16;
        if constexpr (most > 40 * 1024) {
            const cudaError_t e = cudaFuncSetAttribute(k_cell32<G, NT, STG, RES>,
                                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most);
            if (e != cudaSuccess) return e;
        }
        k_cell32<G, NT, STG, RES><<<c->Nc, NT, smem, c->stream>>>(P, nrow);
        return cudaGetLastError();
    };
    c->launches += 1;
    return warp_cells(c) ? go(std::integral_constant<int, 32>{}) : go(std::integral_constant<int, 128>{});
}

template <class G>
cudaError_t raw32_t(avs_ctx* c, const void* fin, const double* W)
{
    const Cell32P<G> P = cell_params<G>(c, fin, nullptr, W);
    if (warp_cells(c)) k_raw32<G, 32><<<c->Nc, 32, 0, c->stream>>>(P);
    else k_raw32<G, 128><<<c->Nc, 128, 0, c->stream>>>(P);
    c->launches += 1;
    return cudaGetLastError();
}

}  // namespace
}  // namespace avs
