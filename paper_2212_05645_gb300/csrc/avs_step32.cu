// FP32 form of the monatomic gas (Shakhov): its equilibria for the face and
// cell kernels, their launchers, and the microscopic sweep of both gases.
#include <vector>

#include "avs_step32.cuh"

namespace avs {

namespace {

// Equilibrium G and H at a node pair.
template <int D>
__device__ __forceinline__ void eq2(const float2* x, const float* U, const float* al, float k2, float l2, float irt,
                                    float RTH, float2& gG, float2& gH)
{
    float2 c[D];
#pragma unroll
    for (int d = 0; d < D; ++d) c[d] = add2(x[d], bc2(-U[d]));
    float2 c2 = mul2(c[0], c[0]), cq = mul2(c[0], bc2(al[0]));
#pragma unroll
    for (int d = 1; d < D; ++d) {
        c2 = fma2(c[d], c[d], c2);
        cq = fma2(c[d], bc2(al[d]), cq);
    }
    const float2 a = fma2(c2, bc2(k2), bc2(l2));
    const float2 e = make_float2(ex2_approx(a.x), ex2_approx(a.y));
    const float2 s = mul2(c2, bc2(irt));
    gG = mul2(e, fma2(cq, add2(s, bc2(-(float)(D + 2))), bc2(1.0f)));
    gH = D == 2 ? mul2(mul2(bc2(RTH), e), fma2(cq, add2(s, bc2(-(float)D)), bc2(1.0f))) : bc2(0.0f);
}
// the same with the prefactor wb within the exponent: e = 2^(l2 + k2 c^2) and
// the Shakhov factors, so that wb g^G = e pG and wb g^H = RTH e pH
template <int D>
__device__ __forceinline__ void eq2f(const float2* x, const float* U, const float* al, float k2, float l2, float2& e,
                                    float2& pG, float2& pH)
{
    float2 c[D];
#pragma unroll
    for (int d = 0; d < D; ++d) c[d] = add2(x[d], bc2(-U[d]));
    float2 c2 = mul2(c[0], c[0]), cq = mul2(c[0], bc2(al[0]));
#pragma unroll
    for (int d = 1; d < D; ++d) {
        c2 = fma2(c[d], c[d], c2);
        cq = fma2(c[d], bc2(al[d]), cq);
    }
    const float2 a = fma2(c2, bc2(k2), bc2(l2));
    e = make_float2(ex2_approx(a.x), ex2_approx(a.y));
    const float irt = -kTwoLn2 * k2;                 // 1 / RT
    const float2 s = fma2(c2, bc2(irt), bc2(-(float)(D + 2)));
    pG = fma2(cq, s, bc2(1.0f));
    pH = D == 2 ? fma2(cq, add2(s, bc2(2.0f)), bc2(1.0f)) : bc2(0.0f);
}

// Interface equilibrium: wb g^G = 2^(l2 + k2 |xi - U|^2) (1 + (c . al)(|c|^2/RT - D - 2))
// with log2 wb inside l2; RTH = (3 - D) R T; wa the weight of the foot value.
struct FaceEq {
    float U[3], k2;
    float al[3], l2;
    float wa, RTH;
};

template <int D_>
struct Shakhov {
    static constexpr int D = D_, NA = NArr<D>::v, NM = NMom<D>::v, NW = D + 2;
    static constexpr bool ROT = false, EXACT = false;
    struct Consts {
        double R, Pr, omega, mu_ref, T_ref;
    };
    using Eq = FaceEq;
    using Par = Cell32Par;

    // interface state (Eqs. 3, equ28, R4) from a face's raw moments about V
    static __device__ __forceinline__ FaceEq face_eq(const Consts& P, double hd, const double* red, const double* Vd, int* err)
    {
        float rho, U[3], RT, qb[3];
        state_from_raw<D, float>(red, Vd, rho, U, RT, qb);
        if (!(rho > 0.0f) || !(RT > 0.0f)) atomicOr(err, 1);
        const float T = fdiv(RT, (float)P.R);
        const float tau = fdiv((float)P.mu_ref * powa(fdiv(T, (float)P.T_ref), (float)P.omega), rho * RT);
        const float hh = (float)hd;
        const float qs = fdiv(tau, tau + hh * (float)P.Pr);
        float qf[3] = {0.0f, 0.0f, 0.0f};
        for (int d = 0; d < D; ++d) qf[d] = qs * qb[d];
        const EqPar<float> e = make_eq_a<D, float, float>(rho, U, RT, qf, (float)P.Pr);
        FaceEq q;
        for (int d = 0; d < 3; ++d) {
            q.U[d] = e.U[d];
            q.al[d] = e.alpha[d];
        }
        q.k2 = e.k2;
        q.l2 = e.l2pref + log2f(fdiv(hh, tau + hh));
        q.wa = fdiv(tau, tau + hh);
        q.RTH = e.RTH;
        return q;
    }
    // phi = wa phi_bar + wb g
    static __device__ __forceinline__ void face_phi(const FaceEq& e, const float2* x, const float2* F, float2* phi)
    {
        float2 ex, pG, pH;
        eq2f<D>(x, e.U, e.al, e.k2, e.l2, ex, pG, pH);
        phi[0] = fma2(ex, pG, mul2(bc2(e.wa), F[0]));
        if constexpr (NA == 2) phi[1] = fma2(mul2(bc2(e.RTH), ex), pH, mul2(bc2(e.wa), F[1]));
    }
    static __device__ __forceinline__ void cell_eq(const Par& c, const float2* x, float2* g)
    {
        float2 gH;
        eq2<D>(x, c.U, c.al, c.k2, c.l2, c.irt, c.RTH, g[0], gH);
        if constexpr (NA == 2) g[1] = gH;
    }
    static __device__ __forceinline__ float vref(const double* W, int d) { return (float)W[1 + d] / (float)W[0]; }
};

}  // namespace

cudaError_t launch_face32(avs_ctx* c, const double* Win, double dt)
{
    if (c->D == 2) return face32_t<Shakhov<2>>(c, Win, dt, {c->cfg.R, c->cfg.Pr, c->cfg.omega, c->mu_ref, c->cfg.T_ref});
    return face32_t<Shakhov<3>>(c, Win, dt, {c->cfg.R, c->cfg.Pr, c->cfg.omega, c->mu_ref, c->cfg.T_ref});
}

cudaError_t launch_cell32(avs_ctx* c, const void* fin, void* fout, bool residual)
{
    if (c->D == 2) return residual ? cell32_t<Shakhov<2>, true>(c, fin, fout) : cell32_t<Shakhov<2>, false>(c, fin, fout);
    return residual ? cell32_t<Shakhov<3>, true>(c, fin, fout) : cell32_t<Shakhov<3>, false>(c, fin, fout);
}

cudaError_t launch_raw32(avs_ctx* c, const void* fin, const double* W)
{
    return c->D == 2 ? raw32_t<Shakhov<2>>(c, fin, W) : raw32_t<Shakhov<3>>(c, fin, W);
}

// ------------------------------------------------------------------ k_micro32
// One colour of a microscopic sweep of the implicit step, FP32 form of either
// gas: dphi_i = (Res_i - sum_{xi.n<0} (xi.n) dphi_j) / (diag_i + sum_{xi.n>=0} xi.n)
// at every node of every array, by quads.  A neighbour's row is read only where
// one of the quad's nodes flows in from it, and only once its colour has been
// visited (`below`: colours that have; dphi is zero before), so dphi needs no
// clearing and the first pass reads no neighbour.  The last visit of a colour
// writes f^{n+1} = f^n + dphi over the residual (`finish`), and dphi itself only
// where another colour still follows (`keep`).  Against a pass for every step
// (clearing, sweeps of four-node threads, one addition at the end), per implicit
// step of the cylinder (12288 cells, 3522 nodes): 1.43 -> 0.60 ms.
template <int D, int NA>
struct Micro32P {
    int Nv, Nvp, chunk, c0, below;
    bool finish, keep;
    const float* fin;
    float* fout;             // the residual; f^{n+1} after the last visit
    float* dphi;
    const float4* geo;
    const Cell32Par* par;    // diag of the monatomic gas,
    const double* diag;      // or (par = nullptr) per cell
    const float* xs;
    size_t xstride;
    const int* nbr;
    const int* clist;
    const unsigned char* colour;
};

template <int D, int NS, int NA>
__global__ void __launch_bounds__(128, 8) k_micro32(Micro32P<D, NA> P)
{
    __shared__ float4 sA[NS];                    // outward normal, neighbour to read (-1: none)
    __shared__ float su;
    __shared__ int sn_;
    const int i = P.clist[P.c0 + blockIdx.x];
    const int t = threadIdx.x;
    if (t < NS) {
        const float4* r = P.geo + (size_t)i * (3 * AVS_MAXS) + 3 * t;
        const int j = P.nbr[i * AVS_MAXS + t], f = __float_as_int(r[1].w);
        float4 n = r[2];
        n.w = __int_as_float(f >= 0 && j >= 0 && P.colour[j] < P.below ? j : -1);
        sA[t] = n;
        const unsigned has = __ballot_sync((1u << NS) - 1u, f >= 0);
        if (t == 0) sn_ = __popc(has);
    } else if (t == 32) {
        su = P.par ? P.par[i].diag : (float)P.diag[i];
    }
    __syncthreads();
    const int ns = sn_;
    const float u = su;
    const int Nv = P.Nv, Nvp = P.Nvp;
    const size_t own = (size_t)i * NA * Nvp;
    const int kend = min(Nvp, (int)(blockIdx.y + 1) * P.chunk);
#pragma unroll 1
    for (int k = blockIdx.y * P.chunk + t * 4; k < kend; k += blockDim.x * 4) {
        float2 X[D][2], acc[NA][2], dg[2];
#pragma unroll
        for (int a = 0; a < NA; ++a) ld4cg(P.fout + own + (size_t)a * Nvp + k, acc[a]);
#pragma unroll
        for (int d = 0; d < D; ++d) ld4(P.xs + d * P.xstride + k, X[d]);
        dg[0] = dg[1] = bc2(0.0f);
#pragma unroll
        for (int s = 0; s < NS; ++s) {
            if (s >= ns) break;
            const float4 n4 = sA[s];
            const float An[3] = {n4.x, n4.y, n4.z};
            const int j = __float_as_int(n4.w);
            float2 in[2];
#pragma unroll
            for (int p = 0; p < 2; ++p) {
                float2 x[D];
#pragma unroll
                for (int d = 0; d < D; ++d) x[d] = X[d][p];
                const float2 sn = dot2<D>(x, An);
                dg[p] = add2(dg[p], make_float2(fmaxf(sn.x, 0.0f), fmaxf(sn.y, 0.0f)));
                in[p] = make_float2(fmaxf(-sn.x, 0.0f), fmaxf(-sn.y, 0.0f));
            }
            if (j < 0 || (in[0].x + in[0].y) + (in[1].x + in[1].y) == 0.0f) continue;
            const float* dj = P.dphi + (size_t)j * NA * Nvp + k;
#pragma unroll
            for (int a = 0; a < NA; ++a) {
                float2 v[2];
                ld4cg(dj + (size_t)a * Nvp, v);
#pragma unroll
                for (int p = 0; p < 2; ++p) {
                    // a node that flows out takes nothing, whatever the neighbour holds
                    const float2 w = make_float2(in[p].x > 0.0f ? v[p].x : 0.0f, in[p].y > 0.0f ? v[p].y : 0.0f);
                    acc[a][p] = fma2(in[p], w, acc[a][p]);
                }
            }
        }
        const float2 inv[2] = {make_float2(1.0f / (u + dg[0].x), 1.0f / (u + dg[0].y)),
                               make_float2(1.0f / (u + dg[1].x), 1.0f / (u + dg[1].y))};
#pragma unroll
        for (int a = 0; a < NA; ++a) {
            float2 o0 = mul2(acc[a][0], inv[0]), o1 = mul2(acc[a][1], inv[1]);
            if (k + 4 > Nv) {                    // pad nodes: zero
                if (k >= Nv) o0.x = 0.0f;
                if (k + 1 >= Nv) o0.y = 0.0f;
                if (k + 2 >= Nv) o1.x = 0.0f;
                o1.y = 0.0f;
            }
            if (P.keep)
                *reinterpret_cast<float4*>(P.dphi + own + (size_t)a * Nvp + k) = make_float4(o0.x, o0.y, o1.x, o1.y);
            if (P.finish) {
                float2 f[2];
                ld4cg(P.fin + own + (size_t)a * Nvp + k, f);
                f[0] = add2(f[0], o0);
                f[1] = add2(f[1], o1);
                *reinterpret_cast<float4*>(P.fout + own + (size_t)a * Nvp + k) =
                    make_float4(f[0].x, f[0].y, f[1].x, f[1].y);
            }
        }
    }
}

// k_micro symmetric Gauss-Seidel iterations over the colours, then f^{n+1}.  A
// colour that follows itself (the turn of a symmetric sweep) would write the
// same values and is skipped.
template <int D, int NA>
static cudaError_t micro32_t(avs_ctx* c, const void* fin, void* fout, const double* diag, int k_micro)
{
    std::vector<int> seq;
    for (int it = 0; it < k_micro; ++it)
        for (int dir = 0; dir < 2; ++dir)
            for (int q = 0; q < c->ncolor; ++q) {
                const int col = dir == 0 ? q : c->ncolor - 1 - q;
                if ((seq.empty() || col != seq.back()) && c->cstart[col + 1] > c->cstart[col]) seq.push_back(col);
            }
    if (seq.empty())
        return cudaMemcpyAsync(fout, fin, (size_t)c->Nc * NA * c->Nvp * sizeof(float), cudaMemcpyDeviceToDevice,
                               c->stream);
    std::vector<int> last(c->ncolor, -1);
    for (int p = 0; p < (int)seq.size(); ++p) last[seq[p]] = p;
    std::vector<char> seen(c->ncolor, 0);
    const int nquad = c->Nvp / 4;
    const int nt = nquad <= 64 ? 64 : 128;
    for (int p = 0; p < (int)seq.size(); ++p) {
        const int col = seq[p], cells = c->cstart[col + 1] - c->cstart[col];
        const int per = (int)std::max(1ll, std::min(4ll, (long long)cells * nquad / nt / (32 * std::max(1, c->nsm))));
        const int ny = (nquad + nt * per - 1) / (nt * per);
        Micro32P<D, NA> P;
        P.Nv = c->Nv;
        P.Nvp = c->Nvp;
        P.chunk = (nquad + ny - 1) / ny * 4;
        P.c0 = c->cstart[col];
        P.below = seen[col] ? c->ncolor : col;     // the first forward sweep visits the colours in order
        P.finish = last[col] == p;
        P.keep = p + 1 < (int)seq.size();
        P.fin = (const float*)fin;
        P.fout = (float*)fout;
        P.dphi = (float*)c->flux;                  // the face flux has been used
        P.geo = (const float4*)c->geo32;
        P.par = diag ? nullptr : (const Cell32Par*)c->cpar;
        P.diag = diag;
        P.xs = c->xi_s;
        P.xstride = c->xstride;
        P.nbr = c->nbr;
        P.clist = c->clist;
        P.colour = c->colour;
        seen[col] = 1;
        if (c->max_ns <= 4) k_micro32<D, D == 2 ? 4 : AVS_MAXS, NA><<<dim3(cells, ny), nt, 0, c->stream>>>(P);
        else k_micro32<D, AVS_MAXS, NA><<<dim3(cells, ny), nt, 0, c->stream>>>(P);
        c->launches += 1;
    }
    return cudaGetLastError();
}

cudaError_t launch_micro32(avs_ctx* c, const void* fin, void* fout, const double* diag, int k_micro)
{
    if (c->model == AVS_RYKOV)
        return c->D == 2 ? micro32_t<2, 3>(c, fin, fout, diag, k_micro) : micro32_t<3, 2>(c, fin, fout, diag, k_micro);
    return c->D == 2 ? micro32_t<2, 2>(c, fin, fout, diag, k_micro) : micro32_t<3, 1>(c, fin, fout, diag, k_micro);
}

}  // namespace avs
