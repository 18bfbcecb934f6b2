// Adjoint of S3-S5 (coherence -> EMI eigenvector -> referenced phase) with
// the SHP masks frozen: for L = sum_{p,i} w_{p,i} phihat_{p,i}, the gradient
// g(q) with dL = Re sum conj(g) dz over the SLC stack (the convention under
// which g = dL/dRe z + j dL/dIm z).  The coherence is recomputed here, not
// stored by the forward pass.
//
// Per output pixel p (an NP-lane group, lane r owning row r):
//   phihat_i = arg(v_i conj(v_ref)):  g_v,i = w_i j v_i / |v_i|^2 (i != ref),
//     g_v,ref = -(sum_{i != ref} w_i) j v_ref / |v_ref|^2; the common-phase
//     direction j v carries no gradient (the phases are gauge invariant).
//   v = unit eigenvector of A for the simple eigenvalue lambda (A = G^-1 o C,
//     or C itself on the EVD fallback):  dv = -(A - lambda I)^+ dA v, so with
//     u = (A - lambda I + c v v^H)^-1 (g_v - v v^H g_v)  (u orthogonal to v),
//     the gradient on A is GA = -u v^H.  c has the sign that makes the deflated
//     matrix definite, so that it is inverted without pivoting: positive where
//     lambda is the smallest eigenvalue, negative on the fallback, where it is
//     the largest.  (A single look has C - lambda I + c v v^H = 2 C - N I for
//     c = lambda, whose leading minor of order N / 2 vanishes.)
//   A = G^-1 o C:  GC += G^-1 o GA;  R = Re(conj(GA) o C);  GG = -G^-1 R G^-1;
//     G = (1-beta)|C| + beta I:  GC += (1-beta) GG o C/|C|  (off the diagonal,
//     which is constant).
//   C_ik = S_ik / sqrt(S_ii S_kk):  GS_ik = GC_ik / sqrt(S_ii S_kk) (i != k),
//     GS_ii = -(sum_k P_ik + sum_k P_ki) / (2 S_ii), P = Re(conj(GC) o C).
//   H_p = GS + GS^H  (Hermitian, stored as the packed upper triangle).
// Per input pixel q and date i (gather):  g_i(q) = sum over the output
//   pixels p whose window holds q with the mask bit set of (H_p z(q))_i.
#include <algorithm>
#include <cmath>
#include <type_traits>

#include "emi.cuh"

namespace plk {

namespace {

// Row of the coherence in shared memory, padded (see k_emi.cu).
template <int NP>
struct AdjRow {
    static constexpr bool kPadded = true;
    const cpx<float> *row;
    __device__ __forceinline__ cpx<float> operator()(int k) const { return row[k]; }
    __device__ __forceinline__ void all(cpx<float> (&c)[NP]) const {
        const uint4 *src = reinterpret_cast<const uint4 *>(row);
#pragma unroll
        for (int q = 0; q < NP / 2; ++q) {
            const uint4 v = src[q];
            memcpy(&c[2 * q], &v, 16);
        }
    }
};

// Two entries of a row, 16-byte aligned.
__device__ __forceinline__ void load_pair(const cpx<float> *src, cpx<float> (&c)[2]) {
    const float4 v = *reinterpret_cast<const float4 *>(src);
    c[0] = mk<float>(v.x, v.y);
    c[1] = mk<float>(v.z, v.w);
}
template <int NP>
__device__ __forceinline__ void store_row(float *dst, const float (&row)[NP]) {
#pragma unroll
    for (int k = 0; k < NP; k += 4)
        *reinterpret_cast<float4 *>(dst + k) = make_float4(row[k], row[k + 1], row[k + 2], row[k + 3]);
}

// Shared memory of one group (output pixel), in bytes from its base.  C holds
// NP padded rows and a zero row for the lanes past the last one (rows of 20,
// 24 and 28 entries run one pixel a warp); its pitch of NP + 2 entries puts the
// 16-byte chunks of 8 consecutive rows in different banks, and a row is also
// read as a broadcast.  Matrices of one value a lane are stored [k][r] (entry
// k of lane r's row), so a row's owner reads it without bank conflicts.
template <int NP>
struct AdjShared {
    static constexpr bool kPow2 = (NP & (NP - 1)) == 0;
    static constexpr int G = kPow2 ? 32 / NP : 1;
    static constexpr int kPitch = NP + 2;
    static constexpr int kLanes = kPow2 ? NP : 32;
    static constexpr int kMat = NP * NP * 4;  // one float matrix
    static constexpr int kBuf = (NP + 2 > kLanes ? NP + 2 : kLanes) * 8;
    static constexpr int oC = 0;
    static constexpr int oBuf = oC + (NP + 1) * kPitch * 8;
    static constexpr int oV = oBuf + kBuf;
    static constexpr int oRs = oV + kLanes * 8;
    static constexpr int oG = oRs + kLanes * 4;  // G^-1 [k][r], then [r][k]; k_adj_prep: the solve's G^-1 row slots
    static constexpr int oM = oG + 2 * kMat;     // k_adj_pixel: R [r][k], then T [k][r], then GG [r][k]
    static_assert(2 * kMat >= kLanes * (NP + 4) * 4, "the G^-1 row slots fit");
    static_assert(oG % 16 == 0 && kMat % 16 == 0, "16-byte loads");
    char *base;
    __device__ __forceinline__ cpx<float> *C() const { return reinterpret_cast<cpx<float> *>(base + oC); }
    __device__ __forceinline__ cpx<float> *buf() const { return reinterpret_cast<cpx<float> *>(base + oBuf); }
    __device__ __forceinline__ cpx<float> *v() const { return reinterpret_cast<cpx<float> *>(base + oV); }
    __device__ __forceinline__ float *rs() const { return reinterpret_cast<float *>(base + oRs); }
    __device__ __forceinline__ float *M() const { return reinterpret_cast<float *>(base + oM); }
    __device__ __forceinline__ float *g() const { return reinterpret_cast<float *>(base + oG); }
    __device__ __forceinline__ float *grow() const { return reinterpret_cast<float *>(base + oG + kMat); }
};

// Lane numbering of a group.
template <int NP>
struct AdjLane {
    int r, glane0, rr;  // row; first lane of the group; a row that exists (lanes past the last read it)
    unsigned gmask;
    __device__ __forceinline__ AdjLane(int lane) {
        constexpr bool kPow2 = (NP & (NP - 1)) == 0;
        const int grp = kPow2 ? lane / NP : 0;
        r = lane - grp * NP;
        rr = r < NP ? r : NP - 1;
        glane0 = grp * NP;
        gmask = (!kPow2 || NP == 32) ? 0xffffffffu : (((1u << NP) - 1u) << glane0);
    }
};

// C <- the padded Hermitian matrix of the packed triangle, unit diagonal: row i
// of the triangle is read by consecutive lanes and written as row and column i.
template <int NP>
__device__ __forceinline__ void adj_load(const AdjShared<NP> &sh, const float2 *Cpix, int r, int n) {
    constexpr int P = AdjShared<NP>::kPitch;
    cpx<float> *C = sh.C();
#pragma unroll 4
    for (int i = 0; i < NP; ++i) {
        if (r < i || r >= NP) continue;
        float2 c = make_float2(i == r ? 1.f : 0.f, 0.f);
        if (r < n && r > i) c = Cpix[packed_index(n, i, r)];
        C[i * P + r] = mk<float>(c.x, c.y);
        if (r > i) C[r * P + i] = mk<float>(c.x, -c.y);
    }
    if (r < NP) C[NP * P + r] = mk<float>(0.f, 0.f);
}

// |v|^2 with its one rounding order spelt out, so that both kernels weight the
// same gradient: where |C| is near singular an ulp of it moves H by 1e-4.
__device__ __forceinline__ float adj_norm2(cpx<float> v) { return __fmaf_rn(v.x, v.x, __fmul_rn(v.y, v.y)); }

// A prepared pixel (k_adj_prep): this lane's entry of the eigenvector and
// 1 / sqrt(S_rr) (0 where S_rr = 0), the eigenvalue, and the deflation's c:
// max(1, |lambda|), negative on the fallback.
struct AdjPixel {
    cpx<float> v;
    float rsr, lam, cdef;
    bool evd, live;
};
template <int NP>
__device__ __forceinline__ AdjPixel adj_read(const AdjShared<NP> &sh, int r, int n, const float2 *Cpix,
                                             const float *Sdp, const float2 *Hp) {
    AdjPixel S;
    S.live = r < n;
    S.v = S.live ? mk<float>(Sdp[r], Cpix[packed_index(n, r, r)].y) : mk<float>(0.f, 0.f);
    S.rsr = S.live ? Hp[r].x : 0.f;
    S.lam = Hp[1].y;
    S.evd = Hp[0].y != 0.f;
    S.cdef = S.evd ? -fmaxf(1.f, fabsf(S.lam)) : fmaxf(1.f, fabsf(S.lam));
    sh.v()[r] = S.v;
    sh.rs()[r] = S.rsr;
    return S;
}

// mrow: this lane's row of (A - lambda I + c v v^H)^-1 (c keeps the deflated
// matrix well scaled); G^-1 (1 on the EVD fallback) into sh.g(), where a lane
// reads its own row, and sh.grow(), where all lanes read one row.  G can be
// conditioned up to 1e6, and its computed inverse is then symmetric to 0.1 only,
// so the two are not interchangeable: the products keep the order G^-1 R, then
// (G^-1 R) G^-1, each over rows.
template <int NP>
__device__ __forceinline__ void adj_invert(const AdjPixel &S, cpx<float> (&mrow)[NP], const AdjShared<NP> &sh,
                                           const AdjLane<NP> &L, int n, float beta) {
    const int r = L.r;
    const AdjRow<NP> ld{sh.C() + (r < NP ? r : NP) * AdjShared<NP>::kPitch};
    ld.all(mrow);
    float gi[NP];
#pragma unroll
    for (int k = 0; k < NP; ++k) gi[k] = mag_t(norm2(mrow[k]));
    if (beta != 0.f) {
#pragma unroll
        for (int k = 0; k < NP; ++k) gi[k] = (1.f - beta) * gi[k] + ((k == r) ? beta : 0.f);
    }
    if (!S.evd) gj_invert<NP, float, float, true>(gi, reinterpret_cast<float *>(sh.buf()), r, n, L.gmask, 0.f);
    ld.all(mrow);
#pragma unroll
    for (int k = 0; k < NP; ++k) {
        if (S.evd) gi[k] = 1.f;
        if (r < NP) sh.g()[k * NP + r] = gi[k];
        // A's entry is rounded before the deflation is added (not contracted
        // with it): its gap can be small, and A is what lambda was formed with.
        mrow[k] = mk<float>(__fmul_rn(gi[k], mrow[k].x), __fmul_rn(gi[k], mrow[k].y));
        mrow[k] = mrow[k] + S.cdef * (S.v * conj(sh.v()[k]));
        if (k == r && S.live) mrow[k].x -= S.lam;
    }
    if (r < NP) store_row<NP>(sh.grow() + r * NP, gi);
    gj_invert<NP, float, cpx<float>, false>(mrow, sh.buf(), r, n, L.gmask, 0.f);
}

}  // namespace

// Diagonal sums S_ii = sum over the mask of |z_i(q)|^2, one thread per
// (output pixel, date).
__global__ void __launch_bounds__(256) k_adj_sdiag(const __grid_constant__ Planes z, int n, const Geom g,
                                                   const uint64_t *__restrict__ mask, float *__restrict__ Sd) {
    const long long nout = (long long)g.Ho * g.Wo;
    const long long total = nout * n;
    for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < total;
         t += (long long)gridDim.x * blockDim.x) {
        const int i = (int)(t / nout);
        const long long o = t - (long long)i * nout;
        const int oy = (int)(o / g.Wo), ox = (int)(o - (long long)oy * g.Wo);
        const int cy = oy * g.sy + g.sy / 2, cx = ox * g.sx + g.sx / 2;
        const uint64_t *mw = mask + o * g.nwords;
        float s = 0.f;
        int b = 0;
        for (int dy = -g.hy; dy <= g.hy; ++dy)
            for (int dx = -g.hx; dx <= g.hx; ++dx, ++b) {
                if (!((__ldg(mw + (b >> 6)) >> (b & 63)) & 1ull)) continue;
                const float2 v = __ldg(z.p[i] + (long long)(cy + dy) * g.W + (cx + dx));
                s += v.x * v.x + v.y * v.y;
            }
        Sd[o * n + i] = s;
    }
}

// The adjoint runs in two kernels: this one solves the pixel (the single-
// precision solve is what the adjoint differentiates), a second one forms what
// depends on the weights.  One kernel of both (110 to 190 KB of code, most of it
// the solve's) lost a third of its issue slots to instruction fetch.  Per output
// pixel, in place of what it has read: Sd: Re v;  C: Im v in the imaginary part
// of the diagonal;  H area: 1 / sqrt(S_kk) (0 where S_kk = 0, NaN where lambda is
// not finite) in its first n entries, whether the EVD fallback solved the pixel
// in the first imaginary part, lambda = v^H A v (the eigenvalue that the
// perturbation is about) in the second (n >= 2).  C's diagonal keeps its real
// part, whose NaN marks a pixel without data: a solve that gives no number is
// not one, and stays NaN.
constexpr int kAdjWarps = 2;

// CTAs an SM that registers are budgeted for: 16 warps at 128 a thread (8 or 7
// CTAs) for rows of up to 24 entries, 12 at 168 (6 or 5) beyond, the budgets of
// k_emi32, whose solve this is (at most 48 bytes of spills).
template <int NP>
struct AdjMinBlocks {
    static constexpr int value = NP > 24 ? 5 : (NP > 16 ? 7 : 8);
};

template <int NP>
__global__ void __launch_bounds__(kAdjWarps * 32, AdjMinBlocks<NP>::value)
    k_adj_prep(float2 *C, float *Sd, int n, long long npx, int ref, const EmiParams prm, float2 *__restrict__ Hout) {
    using Sh = AdjShared<NP>;
    constexpr int G = Sh::G, P = Sh::kPitch;
    __shared__ __align__(16) char smem[kAdjWarps * G * Sh::oM];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const AdjLane<NP> L(lane);
    const int r = L.r, grp = L.glane0 / NP;
    const unsigned gmask = L.gmask;
    const Sh sh{smem + (warp * G + grp) * Sh::oM};
    cpx<float> *cbuf = sh.buf();
    const AdjRow<NP> ld{sh.C() + (r < NP ? r : NP) * P};
    float *gslot = sh.g() + r * (NP + 4);
    const bool live = r < n;
    const long long nt = ntri(n);
    const long long step = (long long)gridDim.x * kAdjWarps * G;
    EmiParams q = prm;
    q.fp64_resolve = 0;

    for (long long base = ((long long)blockIdx.x * kAdjWarps + warp) * G; base < npx; base += step) {
        const long long p = base + grp;
        const bool valid = p < npx;
        float2 *Cpix = C + (valid ? p : 0) * nt;
        bool nan = false;
        if (valid && live) nan = isnan(Cpix[packed_index(n, r, r)].x);
        nan = __any_sync(gmask, nan);
        if (!valid || nan) continue;
        adj_load<NP>(sh, Cpix, r, n);
        __syncwarp(gmask);
        const PixelResult res =
            emi_solve<NP, float, AdjRow<NP>, true>(ld, r, n, ref, q, cbuf, gmask, L.glane0, false, gslot);
        const cpx<float> v = live ? res.v : mk<float>(0.f, 0.f);
        // A row: C, or G^-1 o C with the G^-1 row that the solve left in its slot
        cpx<float> m[NP];
        ld.all(m);
        if (!res.evd) {
#pragma unroll
            for (int q4 = 0; q4 < NP / 4; ++q4) {
                const float4 g4 = reinterpret_cast<const float4 *>(gslot)[q4];
                const float gg[4] = {g4.x, g4.y, g4.z, g4.w};
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const int k = q4 * 4 + e;
                    m[k] = mk<float>(gg[e] * m[k].x, gg[e] * m[k].y);
                }
            }
        }
        const cpx<float> av = group_matvec<NP, float>(m, v, cbuf, r, gmask);
        const float lam = group_sum<NP, float>(live ? (v.x * av.x + v.y * av.y) : 0.f, gmask);
        if (live) {
            const float sr = Sd[p * n + r];
            Sd[p * n + r] = v.x;
            const float rsr = !isfinite(lam) ? __int_as_float(0x7fc00000) : (sr > 0.f ? rsqrtf(sr) : 0.f);
            Hout[p * nt + r] = make_float2(rsr, r == 1 ? lam : (res.evd ? 1.f : 0.f));
            Cpix[packed_index(n, r, r)].y = v.y;
        }
        __syncwarp(gmask);
    }
}

// Per output pixel: H_p from the coherence C (packed), the diagonal sums and
// the phase weights w [n][npx].  Pixels without data get H_p = 0.  With
// K = GC + GC^H off the diagonal, H_rk = K_rk / sqrt(S_rr S_kk) and H_rr =
// -sum_k Re(conj(K_rk) C_rk) / S_rr; K_rk = -g_rk u_r conj(v_k) - g_kr v_r conj(u_k)
// + (1 - beta) (GG_rk + GG_kr) C_rk / |C_rk|.
// What bounds it is instruction issue and fetch: a pixel is two eliminations
// and two products of N x N matrices by one warp.  The products are loops over
// the rows (unrolled over both indices they are 576 to 1024 multiply-adds of
// straight-line code each, which every warp fetches for itself), in rows of 20
// to 32 entries in steps of 4.  301 x 403 pixels at stride 1, this and
// k_adj_prep: 2.55 ms at N = 20, 5.9 at N = 28 and 0.95 at N = 14; in one kernel,
// unrolled, in rows of 24 and 32 entries, 5.36, 12.4 and 1.38 ms.
template <int NP>
__global__ void __launch_bounds__(kAdjWarps * 32, AdjMinBlocks<NP>::value)
    k_adj_pixel(const float2 *__restrict__ C, const float *__restrict__ Sd, int n, long long npx, int ref,
                float beta, const float *__restrict__ w, float2 *Hout) {
    using Sh = AdjShared<NP>;
    constexpr int G = Sh::G, P = Sh::kPitch;
    constexpr int kBytes = Sh::oM + Sh::kMat;
    __shared__ __align__(16) char smem[kAdjWarps * G * kBytes];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const AdjLane<NP> L(lane);
    const int r = L.r, rr = L.rr, grp = L.glane0 / NP;
    const unsigned gmask = L.gmask;
    const Sh sh{smem + (warp * G + grp) * kBytes};
    const long long nt = ntri(n);
    const long long step = (long long)gridDim.x * kAdjWarps * G;

    for (long long base = ((long long)blockIdx.x * kAdjWarps + warp) * G; base < npx; base += step) {
        const long long p = base + grp;
        const bool valid = p < npx;
        const float2 *Cpix = C + (valid ? p : 0) * nt;
        const bool live = r < n;
        bool nan = false;
        if (valid && live) nan = isnan(__ldg(Cpix + packed_index(n, r, r)).x);
        nan = __any_sync(gmask, nan);
        if (!valid) continue;
        if (nan) {
            if (live)
                for (int k = r; k < n; ++k) Hout[p * nt + packed_index(n, r, k)] = make_float2(0.f, 0.f);
            continue;
        }
        adj_load<NP>(sh, Cpix, r, n);
        __syncwarp(gmask);
        float2 *Hp = Hout + p * nt;  // what k_adj_prep left; H at the end
        const AdjPixel S = adj_read<NP>(sh, r, n, Cpix, Sd + p * n, Hp);
        __syncwarp(gmask);
        cpx<float> u;
        {
            cpx<float> mrow[NP];
            adj_invert<NP>(S, mrow, sh, L, n, beta);
            // Gradient on v (gauge-free), projected orthogonal to v.
            const float wr = live ? __ldg(w + (long long)r * npx + p) : 0.f;
            const float wsum = group_sum<NP, float>(live && r != ref ? wr : 0.f, gmask);
            const float m2 = adj_norm2(S.v);
            const float coef = (r == ref) ? -wsum : wr;
            cpx<float> gv = (live && m2 > 0.f) ? (coef / m2) * mk<float>(-S.v.y, S.v.x) : mk<float>(0.f, 0.f);
            const cpx<float> t = conj(S.v) * gv;
            const float sx = group_sum<NP, float>(t.x, gmask), sy = group_sum<NP, float>(t.y, gmask);
            gv = gv - S.v * mk<float>(sx, sy);
            // u = (A - lambda I + c v v^H)^-1 g_v  (orthogonal to v)
            u = group_matvec<NP, float>(mrow, gv, sh.buf(), r, gmask);
        }
        cpx<float> *uall = sh.buf();
        const cpx<float> *Crow = sh.C() + rr * P, *vg = sh.v();
        const float *gcol = sh.g() + rr, *gtr = sh.grow() + rr;
        uall[r] = u;
        float GG[NP];
#pragma unroll
        for (int k = 0; k < NP; ++k) GG[k] = 0.f;
        if (!S.evd) {
            // R = Re(conj(GA) o C), GA = -u v^H (row r); GG = -G^-1 R G^-1.  The
            // products run over the rows of R and G^-1 in loops that are not
            // unrolled over the row index (short code), the left factor's
            // entry read from shared memory and the right factor's row as
            // broadcast 16-byte loads.
            float *R = sh.M(), *T = R;
            if (r < NP) {
                float rrow[NP];
#pragma unroll
                for (int k = 0; k < NP; k += 2) {
                    cpx<float> c[2], v[2];
                    load_pair(Crow + k, c);
                    load_pair(vg + k, v);
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        const cpx<float> ga = mk<float>(0.f, 0.f) - u * conj(v[e]);
                        rrow[k + e] = ga.x * c[e].x + ga.y * c[e].y;
                    }
                }
                store_row<NP>(R + rr * NP, rrow);
            }
            __syncwarp(gmask);
#pragma unroll 2
            for (int j = 0; j < n; ++j) {
                const float gj = gcol[j * NP];
                const float4 *row = reinterpret_cast<const float4 *>(R + j * NP);
#pragma unroll
                for (int q4 = 0; q4 < NP / 4; ++q4) {
                    const float4 x = row[q4];
                    GG[q4 * 4 + 0] += gj * x.x;
                    GG[q4 * 4 + 1] += gj * x.y;
                    GG[q4 * 4 + 2] += gj * x.z;
                    GG[q4 * 4 + 3] += gj * x.w;
                }
            }
            __syncwarp(gmask);
            if (r < NP) {
#pragma unroll
                for (int k = 0; k < NP; ++k) T[k * NP + rr] = GG[k];
            }
            __syncwarp(gmask);  // lanes past the last row read its column
#pragma unroll
            for (int k = 0; k < NP; ++k) GG[k] = 0.f;
#pragma unroll 2
            for (int j = 0; j < n; ++j) {
                const float tj = T[j * NP + rr];
                const float4 *row = reinterpret_cast<const float4 *>(sh.grow() + j * NP);
#pragma unroll
                for (int q4 = 0; q4 < NP / 4; ++q4) {
                    const float4 x = row[q4];
                    GG[q4 * 4 + 0] -= tj * x.x;
                    GG[q4 * 4 + 1] -= tj * x.y;
                    GG[q4 * 4 + 2] -= tj * x.z;
                    GG[q4 * 4 + 3] -= tj * x.w;
                }
            }
            // GG + GG^T: the transpose through the same buffer
            __syncwarp(gmask);
            if (r < NP) store_row<NP>(R + rr * NP, GG);
            __syncwarp(gmask);
#pragma unroll
            for (int k = 0; k < NP; ++k) GG[k] = (1.f - beta) * (GG[k] + R[k * NP + rr]);
        }
        __syncwarp(gmask);
        // Row r of K, its diagonal, and H, written as the columns of the packed
        // upper triangle's rows: lane k writes H_ik = conj(H_ki) for i <= k, a
        // run of consecutive addresses across the lanes.
        cpx<float> h[NP];
        float diag = 0.f;
#pragma unroll
        for (int k2 = 0; k2 < NP; k2 += 2) {
            cpx<float> cc[2], vv[2], uu[2];
            load_pair(Crow + k2, cc);
            load_pair(vg + k2, vv);
            load_pair(uall + k2, uu);
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const int k = k2 + e;
                const cpx<float> c = cc[e];
                const cpx<float> t = gcol[k * NP] * (u * conj(vv[e])) + gtr[k * NP] * (S.v * conj(uu[e]));
                const float m2 = norm2(c);
                const float a = m2 > 0.f ? rsqrtf(m2) * GG[k] : 0.f;
                h[k] = k == r ? mk<float>(0.f, 0.f) : mk<float>(a * c.x - t.x, a * c.y - t.y);
                diag += h[k].x * c.x + h[k].y * c.y;
            }
        }
        if (live) {
#pragma unroll
            for (int k = 0; k < NP; ++k) {
                const float s = S.rsr * sh.rs()[k];
                if (k < r) Hp[packed_index(n, k, r)] = make_float2(s * h[k].x, -s * h[k].y);
                if (k == r) Hp[packed_index(n, k, r)] = make_float2(-S.rsr * S.rsr * diag, 0.f);
            }
        }
        __syncwarp(gmask);
    }
}

// First-order phase uncertainty: white circular noise of variance sigma2 on
// every SLC sample, E|n|^2 = sigma2, propagated through the linked phases.
// With g(q) = H_p z(q) the gradient of phihat_i(p) over the pixel's masked
// window, Var phihat_i = (sigma2 / 2) sum_q |g(q)|^2 = (sigma2 / 2) tr(H^H H S),
// S = sum_q m(q) z(q) z(q)^H = D C D, D = diag(sqrt(S_kk)), and H = D^-1 K D^-1
// (K as in k_adj_pixel, K_rr = -sum_k Re(conj(K_rk) C_rk)), so
//     Var phihat_i = (sigma2 / 2) sum_r (1 / S_rr) k_r C k_r^H,   k_r row r of K.
// Both inverses and u of every date are formed once a pixel; a date costs the
// two products of GG, the row k_r, and its quadratic form over one triangle of
// C (Hermitian: half the products of k_r C).
// W warps share a pixel (G pixels) and take two dates a pass; a pass reads each
// row of G^-1 and C once for both, as broadcast 16-byte loads in loops that are
// not unrolled over the row index (short code).
// With the products unrolled, the solve in the same kernel and H S formed whole,
// 201 x 301 pixels at stride 1 and N = 20 took 17.5 ms, k_adj_prep and this 7.5;
// 101 x 301 pixels at N = 28 38.9 and 9.6 ms, 201 x 301 at N = 12 2.42 and 1.73 ms.
// (X G^-1, X = C diag(v), formed once a pixel would serve every date and save a
// fifth, but where G is conditioned to 1e6 its order of products moves the
// result by 1e-4.)
template <int NP>
struct UncCfg {
    static constexpr int W = 2;
    using Sh = AdjShared<NP>;
    static constexpr int oU = Sh::oM;             // u [date][r]
    static constexpr int oK = oU + 2 * Sh::kMat;  // per warp, two dates: R [r][k] and T [k][r], then rows k_r [NP][NP + 1]
    static constexpr int kKPitch = NP + 1;             // odd: a lane reads its own row 8 bytes at a time
    static constexpr int kK = NP * kKPitch * 8;        // one date's rows
    static constexpr int kBytes = oK + W * 2 * kK;     // of one group
    static_assert(2 * Sh::kMat <= kK && kK % 16 == 0, "the products fit the row buffers");
    static constexpr int kSmem = Sh::G * kBytes;
    // CTAs an SM that registers are budgeted for, no more than shared memory
    // holds (13, 7, 9, 6, 4 and 3 at rows of 8 to 32 entries): 128 registers a
    // thread at 7, 168 at 5, all 255 at 4 and 3; none spills.
    static constexpr int kMinBlocks = NP > 28 ? 3 : (NP > 24 ? 4 : (NP > 20 ? 5 : 7));
};

template <int NP>
__global__ void __launch_bounds__(UncCfg<NP>::W * 32, UncCfg<NP>::kMinBlocks)
    k_adj_uncert(const float2 *__restrict__ C, const float *__restrict__ Sd, const float2 *__restrict__ Hin, int n,
                 long long npx, int ref, float beta, float sigma2, float *__restrict__ sd_out) {
    using Cfg = UncCfg<NP>;
    using Sh = AdjShared<NP>;
    constexpr int G = Sh::G, P = Sh::kPitch, W = Cfg::W;
    extern __shared__ __align__(16) char unc_smem[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const AdjLane<NP> L(lane);
    const int r = L.r, rr = L.rr, grp = L.glane0 / NP;
    const unsigned gmask = L.gmask;
    char *gbase = unc_smem + grp * Cfg::kBytes;
    const Sh sh{gbase};
    cpx<float> *U = reinterpret_cast<cpx<float> *>(gbase + Cfg::oU);
    cpx<float> *K[2];
    float *R[2], *T[2];
#pragma unroll
    for (int d = 0; d < 2; ++d) {
        K[d] = reinterpret_cast<cpx<float> *>(gbase + Cfg::oK + (warp * 2 + d) * Cfg::kK);
        R[d] = reinterpret_cast<float *>(K[d]);
        T[d] = R[d] + NP * NP;
    }
    const cpx<float> *Crow = sh.C() + rr * P, *vg = sh.v();
    const float *gcol = sh.g() + rr, *gtr = sh.grow() + rr;
    const long long nt = ntri(n);
    const long long step = (long long)gridDim.x * G;
    const float qnan = __int_as_float(0x7fc00000);
    const bool live = r < n;

    for (long long base = (long long)blockIdx.x * G; base < npx; base += step) {
        const long long p = base + grp;
        const bool valid = p < npx;
        const float2 *Cpix = C + (valid ? p : 0) * nt;
        bool nan = false;
        if (valid && live) nan = isnan(__ldg(Cpix + packed_index(n, r, r)).x);
        nan = __any_sync(gmask, nan);
        const bool solve = valid && !nan;
        if (warp == 0 && valid) {
            if (live && (nan || r == ref)) sd_out[(long long)r * npx + p] = nan ? qnan : 0.f;
            if (solve) {
                adj_load<NP>(sh, Cpix, r, n);
                const AdjPixel S = adj_read<NP>(sh, r, n, Cpix, Sd + p * n, Hin + p * nt);
                __syncwarp(gmask);
                {
                    cpx<float> mrow[NP];
                    adj_invert<NP>(S, mrow, sh, L, n, beta);
                    // u of every date: the gradient on v (gauge-free) of the
                    // weight 1, projected orthogonal to v
                    const float m2 = adj_norm2(S.v);
#pragma unroll 1
                    for (int i = 0; i < n; ++i) {
                        const float coef = i == ref ? 0.f : (r == ref ? -1.f : (r == i ? 1.f : 0.f));
                        cpx<float> gv =
                            (live && m2 > 0.f) ? (coef / m2) * mk<float>(-S.v.y, S.v.x) : mk<float>(0.f, 0.f);
                        const cpx<float> t = conj(S.v) * gv;
                        const float sx = group_sum<NP, float>(t.x, gmask), sy = group_sum<NP, float>(t.y, gmask);
                        gv = gv - S.v * mk<float>(sx, sy);
                        const cpx<float> u = group_matvec<NP, float>(mrow, gv, sh.buf(), r, gmask);
                        if (r < NP) U[i * NP + r] = u;
                    }
                }
            }
        }
        __syncthreads();
        if (solve) {
            const bool evd = __ldg(&Hin[p * nt].y) != 0.f;
            const float rsr = sh.rs()[r];
            const cpx<float> vr = vg[r];
            for (int i0 = 2 * warp; i0 < n; i0 += 2 * W) {
                const int i1 = i0 + 1 < n ? i0 + 1 : i0;
                const cpx<float> *U0 = U + i0 * NP, *U1 = U + i1 * NP;
                float A0[NP], A1[NP];
#pragma unroll
                for (int k = 0; k < NP; ++k) A0[k] = A1[k] = 0.f;
                const cpx<float> ur0 = U0[rr], ur1 = U1[rr];
                if (!evd) {
                    // GG = -G^-1 R G^-1 (see k_adj_pixel), both dates
                    if (r < NP) {
#pragma unroll
                        for (int k2 = 0; k2 < NP; k2 += 4) {
                            float q0[4], q1[4];
#pragma unroll
                            for (int e = 0; e < 4; ++e) {
                                const cpx<float> c = Crow[k2 + e], vk = vg[k2 + e];
                                const cpx<float> h0 = mk<float>(0.f, 0.f) - ur0 * conj(vk);
                                const cpx<float> h1 = mk<float>(0.f, 0.f) - ur1 * conj(vk);
                                q0[e] = h0.x * c.x + h0.y * c.y;
                                q1[e] = h1.x * c.x + h1.y * c.y;
                            }
                            *reinterpret_cast<float4 *>(R[0] + r * NP + k2) = make_float4(q0[0], q0[1], q0[2], q0[3]);
                            *reinterpret_cast<float4 *>(R[1] + r * NP + k2) = make_float4(q1[0], q1[1], q1[2], q1[3]);
                        }
                    }
                    __syncwarp(gmask);
#pragma unroll 2
                    for (int j = 0; j < n; ++j) {
                        const float g = gcol[j * NP];
                        const float4 *r0 = reinterpret_cast<const float4 *>(R[0] + j * NP);
                        const float4 *r1 = reinterpret_cast<const float4 *>(R[1] + j * NP);
#pragma unroll
                        for (int k = 0; k < NP; k += 4) {
                            const float4 x = r0[k / 4], y = r1[k / 4];
                            A0[k] += g * x.x;
                            A0[k + 1] += g * x.y;
                            A0[k + 2] += g * x.z;
                            A0[k + 3] += g * x.w;
                            A1[k] += g * y.x;
                            A1[k + 1] += g * y.y;
                            A1[k + 2] += g * y.z;
                            A1[k + 3] += g * y.w;
                        }
                    }
                    if (r < NP) {
#pragma unroll
                        for (int k = 0; k < NP; ++k) {
                            T[0][k * NP + r] = A0[k];
                            T[1][k * NP + r] = A1[k];
                        }
                    }
                    __syncwarp(gmask);  // lanes past the last row read its column
#pragma unroll
                    for (int k = 0; k < NP; ++k) A0[k] = A1[k] = 0.f;
#pragma unroll 2
                    for (int j = 0; j < n; ++j) {
                        const float t0 = T[0][j * NP + rr], t1 = T[1][j * NP + rr];
                        const float4 *row = reinterpret_cast<const float4 *>(sh.grow() + j * NP);
#pragma unroll
                        for (int k = 0; k < NP; k += 4) {
                            const float4 x = row[k / 4];
                            A0[k] -= t0 * x.x;
                            A0[k + 1] -= t0 * x.y;
                            A0[k + 2] -= t0 * x.z;
                            A0[k + 3] -= t0 * x.w;
                            A1[k] -= t1 * x.x;
                            A1[k + 1] -= t1 * x.y;
                            A1[k + 2] -= t1 * x.z;
                            A1[k + 3] -= t1 * x.w;
                        }
                    }
                    // GG + GG^T through the row buffers
                    __syncwarp(gmask);
                    if (r < NP) {
                        store_row<NP>(R[0] + r * NP, A0);
                        store_row<NP>(R[1] + r * NP, A1);
                    }
                    __syncwarp(gmask);
#pragma unroll
                    for (int k = 0; k < NP; ++k) {
                        A0[k] += R[0][k * NP + rr];
                        A1[k] += R[1][k * NP + rr];
                    }
                    __syncwarp(gmask);
                }
                // Rows k_r of both dates into this lane's row buffers.
                float diag0 = 0.f, diag1 = 0.f;
                cpx<float> *k0 = K[0] + rr * Cfg::kKPitch, *k1 = K[1] + rr * Cfg::kKPitch;
#pragma unroll
                for (int k2 = 0; k2 < NP; k2 += 2) {
                    cpx<float> cc[2], vv[2], w0[2], w1[2];
                    load_pair(Crow + k2, cc);
                    load_pair(vg + k2, vv);
                    load_pair(U0 + k2, w0);
                    load_pair(U1 + k2, w1);
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        const int k = k2 + e;
                        const cpx<float> c = cc[e];
                        const float m2 = norm2(c), g = gcol[k * NP], gt = gtr[k * NP];
                        const float im = m2 > 0.f ? (1.f - beta) * rsqrtf(m2) : 0.f;
                        const cpx<float> t0 = g * (ur0 * conj(vv[e])) + gt * (vr * conj(w0[e]));
                        const cpx<float> t1 = g * (ur1 * conj(vv[e])) + gt * (vr * conj(w1[e]));
                        const float a0 = im * A0[k], a1 = im * A1[k];
                        cpx<float> h0 = mk<float>(a0 * c.x - t0.x, a0 * c.y - t0.y);
                        cpx<float> h1 = mk<float>(a1 * c.x - t1.x, a1 * c.y - t1.y);
                        // nothing from or to a date without power (S_kk = 0)
                        if (k == r || !(sh.rs()[k] > 0.f)) h0 = h1 = mk<float>(0.f, 0.f);
                        diag0 += h0.x * c.x + h0.y * c.y;
                        diag1 += h1.x * c.x + h1.y * c.y;
                        if (r < NP) {
                            k0[k] = h0;
                            k1[k] = h1;
                        }
                    }
                }
                if (r < NP) {
                    k0[r] = mk<float>(-diag0, 0.f);
                    k1[r] = mk<float>(-diag1, 0.f);
                }
                __syncwarp(gmask);  // lanes past the last row read its K row
                // k C k^H = Re sum_m conj(k_m) sum_l w_lm k_l C_lm over blocks of
                // columns m: weight 1 inside the diagonal block (both orders
                // of a pair appear), 2 below it (one order).
                float q0 = 0.f, q1 = 0.f;
#pragma unroll
                for (int mb = 0; mb < NP; mb += 8) {
                    constexpr int kB = 8;
                    const int width = NP - mb < kB ? NP - mb : kB;
                    if (mb >= n) break;
                    cpx<float> s0[kB], s1[kB];
#pragma unroll
                    for (int e = 0; e < kB; ++e) s0[e] = s1[e] = mk<float>(0.f, 0.f);
#pragma unroll 1
                    for (int l = mb; l < n; ++l) {
                        const float wl = l < mb + kB ? 1.f : 2.f;
                        const cpx<float> a0 = wl * k0[l], a1 = wl * k1[l];
                        const float4 *row = reinterpret_cast<const float4 *>(sh.C() + l * P + mb);
#pragma unroll
                        for (int e = 0; e < kB; e += 2) {
                            if (e < width) {
                                const float4 t = row[e / 2];
                                const cpx<float> ca = mk<float>(t.x, t.y), cb = mk<float>(t.z, t.w);
                                s0[e] = cfma(a0, ca, s0[e]);
                                s0[e + 1] = cfma(a0, cb, s0[e + 1]);
                                s1[e] = cfma(a1, ca, s1[e]);
                                s1[e + 1] = cfma(a1, cb, s1[e + 1]);
                            }
                        }
                    }
#pragma unroll
                    for (int e = 0; e < kB; ++e) {
                        if (e < width) {
                            const cpx<float> a0 = k0[mb + e], a1 = k1[mb + e];
                            q0 += a0.x * s0[e].x + a0.y * s0[e].y;
                            q1 += a1.x * s1[e].x + a1.y * s1[e].y;
                        }
                    }
                }
                const float s2 = live ? rsr * rsr : 0.f;
                const float tr0 = group_sum<NP, float>(s2 != 0.f ? s2 * q0 : 0.f, gmask);
                const float tr1 = group_sum<NP, float>(s2 != 0.f ? s2 * q1 : 0.f, gmask);
                if (r == 0) {
                    // a sum rounded below 0 counts as 0, one that is not a number stays so
                    const float var0 = 0.5f * sigma2 * tr0, var1 = 0.5f * sigma2 * tr1;
                    if (i0 != ref) sd_out[(long long)i0 * npx + p] = sqrtf(var0 < 0.f ? 0.f : var0);
                    if (i1 != i0 && i1 != ref) sd_out[(long long)i1 * npx + p] = sqrtf(var1 < 0.f ? 0.f : var1);
                }
                __syncwarp(gmask);  // the row buffers are free for the next pass
            }
        }
        __syncthreads();
    }
}

// Per (input pixel q, date i): g_i(q) = sum over the output pixels p whose
// window holds q, with q's mask bit set, of sum_k H_p,ik z_k(q).  NT >= n.
// The date index runs fastest across threads: a warp covers one or two
// pixels, so its loads of H_p rows fall on one or two packed matrices and the
// loads of z(q) are broadcasts.
template <int NT>
__global__ void __launch_bounds__(256) k_adj_gather(const __grid_constant__ Planes z, int n, const Geom g,
                                                    const uint64_t *__restrict__ mask,
                                                    const float2 *__restrict__ H, float2 *__restrict__ grad) {
    const long long npix = (long long)g.H * g.W;
    const long long total = npix * n;
    const long long nt = ntri(n);
    for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < total;
         t += (long long)gridDim.x * blockDim.x) {
        const long long qi = t / n;
        const int i = (int)(t - qi * n);
        const int qy = (int)(qi / g.W), qx = (int)(qi - (long long)qy * g.W);
        cpx<float> zq[NT];
#pragma unroll
        for (int k = 0; k < NT; ++k) {
            const float2 v = k < n ? __ldg(z.p[k] + qi) : make_float2(0.f, 0.f);
            zq[k] = mk<float>(v.x, v.y);
        }
        // output rows/columns whose window centre lies within hy/hx of q
        const int oy_lo = max(0, (qy - g.hy - g.sy / 2 + g.sy - 1) / g.sy);
        const int oy_hi = min(g.Ho - 1, (qy + g.hy - g.sy / 2) >= 0 ? (qy + g.hy - g.sy / 2) / g.sy : -1);
        const int ox_lo = max(0, (qx - g.hx - g.sx / 2 + g.sx - 1) / g.sx);
        const int ox_hi = min(g.Wo - 1, (qx + g.hx - g.sx / 2) >= 0 ? (qx + g.hx - g.sx / 2) / g.sx : -1);
        cpx<float> acc = mk<float>(0.f, 0.f);
        for (int oy = oy_lo; oy <= oy_hi; ++oy) {
            const int dy = qy - (oy * g.sy + g.sy / 2);
            if (dy < -g.hy || dy > g.hy) continue;
            for (int ox = ox_lo; ox <= ox_hi; ++ox) {
                const int dx = qx - (ox * g.sx + g.sx / 2);
                if (dx < -g.hx || dx > g.hx) continue;
                const long long o = (long long)oy * g.Wo + ox;
                const int b = (dy + g.hy) * g.wx + (dx + g.hx);
                if (!((__ldg(mask + o * g.nwords + (b >> 6)) >> (b & 63)) & 1ull)) continue;
                const float2 *Hp = H + o * nt;
#pragma unroll
                for (int k = 0; k < NT; ++k) {
                    if (k >= n) break;
                    // H_ik from the packed upper triangle (H Hermitian)
                    const float2 h = __ldg(Hp + (i <= k ? packed_index(n, i, k) : packed_index(n, k, i)));
                    const cpx<float> hik = i <= k ? mk<float>(h.x, h.y) : mk<float>(h.x, -h.y);
                    acc = cfma(hik, zq[k], acc);
                }
            }
        }
        grad[(long long)i * npix + qi] = make_float2(acc.x, acc.y);
    }
}

// Gradient of L with respect to real per-sample window weights (the SHP mask
// read as weights w_b in S = sum_b w_b z(q_b) z(q_b)^H, evaluated at w = mask):
// dL/dw_b = Re sum_jk conj(GS_jk) z_j conj(z_k) = (1/2) z^H H_p z, z = z(q_b);
// 0 for window samples outside the image and for pixels without data (H_p = 0).
// One thread per (output pixel, window sample), samples fastest: a warp spans
// one or two pixels, so its loads of H_p are broadcasts.  NT >= n.
template <int NT>
__global__ void __launch_bounds__(256) k_adj_wgrad(const __grid_constant__ Planes z, int n, const Geom g,
                                                   const float2 *__restrict__ H, float *__restrict__ dw) {
    const long long npx = (long long)g.Ho * g.Wo;
    const int nb = g.wy * g.wx;
    const long long total = npx * nb;
    const long long nt = ntri(n);
    for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < total;
         t += (long long)gridDim.x * blockDim.x) {
        const long long o = t / nb;
        const int b = (int)(t - o * nb);
        const int oy = (int)(o / g.Wo), ox = (int)(o - (long long)oy * g.Wo);
        const int by = b / g.wx, bx = b - by * g.wx;
        const int y = oy * g.sy + g.sy / 2 - g.hy + by, x = ox * g.sx + g.sx / 2 - g.hx + bx;
        float acc = 0.f;
        if (y >= 0 && y < g.H && x >= 0 && x < g.W) {
            const long long qi = (long long)y * g.W + x;
            cpx<float> zq[NT];
#pragma unroll
            for (int k = 0; k < NT; ++k) {
                const float2 v = k < n ? __ldg(z.p[k] + qi) : make_float2(0.f, 0.f);
                zq[k] = mk<float>(v.x, v.y);
            }
            // z^H H z = sum_j H_jj |z_j|^2 + 2 Re sum_{j<k} conj(z_j) H_jk z_k
            const float2 *Hp = H + o * nt;
#pragma unroll
            for (int j = 0; j < NT; ++j) {
                if (j >= n) break;
                const float2 *row = Hp + packed_index(n, j, j);
                const float2 hd = __ldg(row);
                cpx<float> s = mk<float>(0.f, 0.f);
#pragma unroll
                for (int k = j + 1; k < NT; ++k) {
                    if (k >= n) break;
                    const float2 h = __ldg(row + (k - j));
                    s = cfma(mk<float>(h.x, h.y), zq[k], s);
                }
                acc += hd.x * norm2(zq[j]) + 2.f * (zq[j].x * s.x + zq[j].y * s.y);
            }
        }
        dw[t] = 0.5f * acc;
    }
}

// Tiled scatter of the same sum: a CTA owns a TY x TX tile of output pixels and
// holds the z of the input region that their windows cover, and accumulators
// of it, in shared memory, date-major.  A warp owns RB dates (rows of every
// H_p) of its team's share of the tile and takes those pixels in turn: its RB
// rows of H_p go to a buffer of its own (the next pixel's are in flight
// meanwhile), its lanes are the looks of the window, two a lane, and every pair
// of entries of an H row, read as one broadcast, serves 16 multiply-adds.  Each
// team has an accumulator, where only the owner adds to a date's, a lane at its
// own looks, so nothing is atomic and no warp waits for another within a tile.
// The teams' sums are then added into the gradient (tiles overlap by the window
// halo: 8-byte global reductions, whose order, and so the last bits of the
// result, may vary from run to run).  Few dates need several teams to fill an
// SM, many dates are warps enough (scatter_plan).  Issue bounds it: 55 of a
// 5 x 11 window's 64 lane slots work; rejected looks cost as accepted ones.
struct AdjTile {
    int TY, TX, RY, RX, L, teams;
};

constexpr int kScatterMaxWarps = 8, kScatterBudget = 220 * 1024;

template <int RB>
__global__ void __launch_bounds__(kScatterMaxWarps * 32) k_adj_scatter(
    const __grid_constant__ Planes z, int n, const Geom g, const uint64_t *__restrict__ mask,
    const float2 *__restrict__ H, float2 *__restrict__ grad, const AdjTile t, long long ntiles, int tilesY) {
    extern __shared__ __align__(16) float2 sm[];
    const int npr = t.RY * t.RX, pitch = (n + 1) & ~1;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nwarps = blockDim.x >> 5;
    const int team = warp % t.teams, i0 = warp / t.teams * RB;
    float2 *hbuf = sm + (size_t)warp * 2 * RB * pitch;                       // [2][RB][pitch]
    float2 *zreg = sm + (size_t)nwarps * 2 * RB * pitch;                     // [n][npr]
    float2 *accs = zreg + (size_t)npr * n;                                   // [teams][n][npr]
    float2 *acc = accs + (size_t)team * npr * n;                             // this team's
    int *lkoff = reinterpret_cast<int *>(accs + (size_t)t.teams * npr * n);  // [L]
    const long long nt = ntri(n), npix = (long long)g.H * g.W;
    for (int l = threadIdx.x; l < t.L; l += blockDim.x) lkoff[l] = (l / g.wx) * t.RX + (l % g.wx);
    // This lane's share of the warp's rows: where each entry lies in the packed
    // triangle (the conjugate below the diagonal) and in the buffer; -1: none.
    int src[RB], dst[RB];
    unsigned low = 0;
#pragma unroll
    for (int m = 0; m < RB; ++m) {
        const int e = lane + 32 * m, jr = e / n, k = e - jr * n, i = i0 + jr;
        const bool in = jr < RB && i < n;
        src[m] = in ? (i <= k ? packed_index(n, i, k) : packed_index(n, k, i)) : -1;
        dst[m] = jr * pitch + k;
        if (in && i > k) low |= 1u << m;
    }
    // rows past the last date stay zero
    for (int e = lane; e < 2 * RB * pitch; e += 32) hbuf[e] = make_float2(0.f, 0.f);
    for (long long tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        const int ty0 = (int)(tile % tilesY) * t.TY, tx0 = (int)(tile / tilesY) * t.TX;
        const int y0 = ty0 * g.sy + g.sy / 2 - g.hy, x0 = tx0 * g.sx + g.sx / 2 - g.hx;
        __syncthreads();  // previous tile done with the buffers (and the look table written)
        for (int pr = threadIdx.x; pr < npr; pr += blockDim.x) {
            const int y = y0 + pr / t.RX, x = x0 + pr % t.RX;
            const bool in = y >= 0 && y < g.H && x >= 0 && x < g.W;
            const long long at = in ? (long long)y * g.W + x : 0;
#pragma unroll 8
            for (int d = 0; d < n; ++d) zreg[d * npr + pr] = in ? __ldg(z.p[d] + at) : make_float2(0.f, 0.f);
        }
        for (int e = threadIdx.x; e < t.teams * n * npr; e += blockDim.x) accs[e] = make_float2(0.f, 0.f);
        __syncthreads();
        const int ny = min(t.TY, g.Ho - ty0), nx = min(t.TX, g.Wo - tx0), npx = ny * nx;
        float2 h[RB];
        auto fetch = [&](int s) {
            const int tx = s / ny, ty = s - tx * ny;
            const float2 *Hp = H + ((long long)(ty0 + ty) * g.Wo + tx0 + tx) * nt;
#pragma unroll
            for (int m = 0; m < RB; ++m) h[m] = src[m] >= 0 ? __ldg(Hp + src[m]) : make_float2(0.f, 0.f);
        };
        auto put = [&](int slot) {
#pragma unroll
            for (int m = 0; m < RB; ++m)
                if (src[m] >= 0)
                    hbuf[slot * RB * pitch + dst[m]] = make_float2(h[m].x, (low >> m) & 1u ? -h[m].y : h[m].y);
        };
        if (team < npx) {
            fetch(team);
            put(0);
        }
        int slot = 0;
        for (int s = team; s < npx; s += t.teams, slot ^= 1) {
            __syncwarp();
            if (s + t.teams < npx) fetch(s + t.teams);
            const float2 *hb = hbuf + slot * RB * pitch;
            const int tx = s / ny, ty = s - tx * ny;
            const uint64_t *mw = mask + ((long long)(ty0 + ty) * g.Wo + tx0 + tx) * g.nwords;
            const int corner = ty * g.sy * t.RX + tx * g.sx;
            for (int w0 = 0; w0 < t.L; w0 += 64) {
                const uint64_t bits = __ldg(mw + (w0 >> 6));
                const int l0 = w0 + lane, l1 = l0 + 32;
                const bool on0 = l0 < t.L && ((bits >> lane) & 1ull), on1 = l1 < t.L && ((bits >> (lane + 32)) & 1ull);
                const int q0 = corner + (on0 ? lkoff[l0] : 0), q1 = corner + (on1 ? lkoff[l1] : 0);
                cpx<float> a0[RB], a1[RB];
#pragma unroll
                for (int j = 0; j < RB; ++j) a0[j] = a1[j] = mk<float>(0.f, 0.f);
                const float2 *z0 = zreg + q0, *z1 = zreg + q1;
#pragma unroll 2
                for (int k = 0; k + 1 < n; k += 2, z0 += 2 * npr, z1 += 2 * npr) {
                    const float2 u0 = z0[0], v0 = z0[npr], u1 = z1[0], v1 = z1[npr];
#pragma unroll
                    for (int j = 0; j < RB; ++j) {
                        const float4 hh = *reinterpret_cast<const float4 *>(hb + j * pitch + k);
                        const cpx<float> ha = mk<float>(hh.x, hh.y), hc = mk<float>(hh.z, hh.w);
                        a0[j] = cfma(ha, mk<float>(u0.x, u0.y), a0[j]);
                        a1[j] = cfma(ha, mk<float>(u1.x, u1.y), a1[j]);
                        a0[j] = cfma(hc, mk<float>(v0.x, v0.y), a0[j]);
                        a1[j] = cfma(hc, mk<float>(v1.x, v1.y), a1[j]);
                    }
                }
                if (n & 1) {
                    const float2 u0 = z0[0], u1 = z1[0];
#pragma unroll
                    for (int j = 0; j < RB; ++j) {
                        const float2 hh = hb[j * pitch + n - 1];
                        a0[j] = cfma(mk<float>(hh.x, hh.y), mk<float>(u0.x, u0.y), a0[j]);
                        a1[j] = cfma(mk<float>(hh.x, hh.y), mk<float>(u1.x, u1.y), a1[j]);
                    }
                }
#pragma unroll
                for (int j = 0; j < RB; ++j) {
                    if (i0 + j >= n) break;
                    float2 *row = acc + (size_t)(i0 + j) * npr;
                    if (on0) {
                        const float2 v = row[q0];
                        row[q0] = make_float2(v.x + a0[j].x, v.y + a0[j].y);
                    }
                    if (on1) {
                        const float2 v = row[q1];
                        row[q1] = make_float2(v.x + a1[j].x, v.y + a1[j].y);
                    }
                }
                __syncwarp();  // the next looks (or pixel) add to these sums from other lanes
            }
            if (s + t.teams < npx) put(slot ^ 1);
        }
        __syncthreads();
        for (int pr = threadIdx.x; pr < npr; pr += blockDim.x) {
            const int y = y0 + pr / t.RX, x = x0 + pr % t.RX;
            if (y < 0 || y >= g.H || x < 0 || x >= g.W) continue;
            float2 *out = grad + (long long)y * g.W + x;
#pragma unroll 4
            for (int d = 0; d < n; ++d) {
                float2 v = accs[d * npr + pr];
                for (int m = 1; m < t.teams; ++m) {
                    const float2 u = accs[(m * n + d) * npr + pr];
                    v = make_float2(v.x + u.x, v.y + u.y);
                }
                if (v.x != 0.f || v.y != 0.f) atomicAdd(out + (long long)d * npix, v);
            }
        }
    }
}

// Shared memory of the scatter: the warps' H rows, z and the teams' accumulators
// over the region, the look table.
static size_t scatter_smem(int n, const AdjTile &t, int warps, int rb) {
    return (size_t)warps * 2 * rb * ((n + 1) & ~1) * sizeof(float2) +
           (size_t)t.RY * t.RX * n * (1 + t.teams) * sizeof(float2) + (size_t)t.L * sizeof(int);
}

// Tile for the scatter: the most output pixels whose region fits the budget
// (TY = 0: none does).
static AdjTile adj_tile(int n, const Geom &g, size_t budget, int warps, int rb, int teams) {
    AdjTile best{0, 0, 0, 0, g.wy * g.wx, teams};
    const AdjTile empty{0, 0, 0, 0, g.wy * g.wx, teams};
    const size_t fixed = scatter_smem(n, empty, warps, rb);
    if (fixed >= budget) return best;
    const int region = (int)((budget - fixed) / ((size_t)n * (1 + teams) * sizeof(float2)));
    for (int TY = 1; TY <= std::min(32, g.Ho); ++TY) {
        const int RY = (TY - 1) * g.sy + g.wy, RXmax = region / RY;
        if (RXmax < g.wx) break;
        const int TX = std::min({64, g.Wo, (RXmax - g.wx) / g.sx + 1}), RX = (TX - 1) * g.sx + g.wx;
        if (TY * TX > best.TY * best.TX || (TY * TX == best.TY * best.TX && RY * RX < best.RY * best.RX))
            best = AdjTile{TY, TX, RY, RX, g.wy * g.wx, teams};
    }
    return best;
}

// Teams and tile of the scatter (TY = 0: no tile fits).  More teams and more
// CTAs an SM put more warps in flight; both shrink the tile, and a small tile
// spends its time on the region (z in, accumulators cleared and added out).
// The estimate, in cycles of an SM: a warp takes 1000 + 160 n for 64 looks of a
// pixel, side by side up to 14 warps an SM, and a region sample costs 0.8 a
// date and buffer.  Fitted to 136 combinations of 2 to 32 dates, windows of
// 3 x 3 to 31 x 31, strides and image sizes: the choice is within 10% of the
// fastest one tried in 121 of them, within 20% in 129.  160 x 240 pixels at
// stride 1, one team a CTA and this: 13 x 25 windows at N = 4 5.50 and 0.16 ms, at
// N = 8 2.31 and 0.35, 19 x 39 at N = 4 6.18 and 0.45, 3 x 3 at N = 2 0.33 and 0.05 ms.
static AdjTile scatter_plan(int n, const Geom &g, int rb) {
    const int groups = (n + rb - 1) / rb, words = (g.wy * g.wx + 63) / 64, sms = device_sm_count();
    AdjTile best{};
    double best_cost = 0.0;
    for (int teams : {1, 2, 3, 4, 6, 8})
        for (int ctas : {1, 2, 3, 4, 6, 12}) {
            const int warps = teams * groups;
            if (warps > kScatterMaxWarps || warps * ctas > 24) continue;
            const AdjTile t = adj_tile(n, g, kScatterBudget / ctas, warps, rb, teams);
            if (t.TY == 0) continue;
            const double tiles =
                (double)((g.Ho + t.TY - 1) / t.TY) * ((g.Wo + t.TX - 1) / t.TX) / sms;  // an SM
            const double side = std::min((double)ctas, std::ceil(tiles));               // of them at a time
            const double looks = (double)((t.TY * t.TX + teams - 1) / teams) * words * (1000.0 + 160.0 * n);
            const double cost = std::max(1.0, tiles / ctas) *
                                (looks * std::max(1.0, warps * side / 14.0) +
                                 0.8 * n * (2 + teams) * t.RY * t.RX * side);
            if (best.TY == 0 || cost < best_cost) {
                best = t;
                best_cost = cost;
            }
        }
    return best;
}

template <int RB>
static cudaError_t run_scatter(const Planes &z, int n, const Geom &g, const uint64_t *mask, const float2 *H,
                               float2 *grad, const AdjTile &t, cudaStream_t s) {
    const int warps = t.teams * ((n + RB - 1) / RB);
    const size_t smem = scatter_smem(n, t, warps, RB);
    cudaError_t e = cudaFuncSetAttribute(k_adj_scatter<RB>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         kScatterBudget);
    if (e != cudaSuccess) return e;
    const int tilesY = (g.Ho + t.TY - 1) / t.TY;
    const long long ntiles = (long long)tilesY * ((g.Wo + t.TX - 1) / t.TX);
    const long long grid = std::min<long long>(ntiles, (long long)device_sm_count() * 16);
    k_adj_scatter<RB><<<(unsigned)grid, warps * 32, smem, s>>>(z, n, g, mask, H, grad, t, ntiles, tilesY);
    return cudaGetLastError();
}

static int adj_grid(long long work) {
    long long blocks = (work + 255) / 256;
    const long long cap = (long long)device_sm_count() * 8;
    return (int)std::max<long long>(1, std::min(blocks, cap));
}

// Launches of the two-kernel adjoint: the preparation (parts of C, Sd and the H
// area overwritten), then H, or the standard deviations.
template <int NP>
static int adj_blocks(long long npx) {
    constexpr int G = AdjShared<NP>::G;
    const long long blocks = ((npx + G - 1) / G + kAdjWarps - 1) / kAdjWarps;
    return (int)std::max<long long>(1, std::min(blocks, (long long)device_sm_count() * 16));
}

template <int NP>
static cudaError_t run_adj_pixel(float2 *C, float *Sd, int n, long long npx, int ref, const EmiParams &prm,
                                 const float *w, float2 *H, cudaStream_t s) {
    k_adj_prep<NP><<<adj_blocks<NP>(npx), kAdjWarps * 32, 0, s>>>(C, Sd, n, npx, ref, prm, H);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_adj_pixel<NP><<<adj_blocks<NP>(npx), kAdjWarps * 32, 0, s>>>(C, Sd, n, npx, ref, prm.beta, w, H);
    return cudaGetLastError();
}

template <int NP>
static cudaError_t run_adj_uncert(float2 *C, float *Sd, float2 *H, int n, long long npx, int ref,
                                  const EmiParams &prm, float sigma2, float *out, cudaStream_t s) {
    using Cfg = UncCfg<NP>;
    constexpr int G = AdjShared<NP>::G;
    cudaError_t e = cudaFuncSetAttribute(k_adj_uncert<NP>, cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg::kSmem);
    if (e != cudaSuccess) return e;
    k_adj_prep<NP><<<adj_blocks<NP>(npx), kAdjWarps * 32, 0, s>>>(C, Sd, n, npx, ref, prm, H);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    const long long cap = (long long)device_sm_count() * 32;
    const long long blocks = std::max<long long>(1, std::min((npx + G - 1) / G, cap));
    k_adj_uncert<NP><<<(unsigned)blocks, Cfg::W * 32, Cfg::kSmem, s>>>(C, Sd, H, n, npx, ref, prm.beta, sigma2, out);
    return cudaGetLastError();
}

// f(row length) for the rows of n dates (emi_row_length).
template <class F>
static cudaError_t with_row_length(int n, const F &f) {
    switch (emi_row_length(n)) {
        case 8: return f(std::integral_constant<int, 8>());
        case 16: return f(std::integral_constant<int, 16>());
        case 20: return f(std::integral_constant<int, 20>());
        case 24: return f(std::integral_constant<int, 24>());
        case 28: return f(std::integral_constant<int, 28>());
        default: return f(std::integral_constant<int, 32>());
    }
}

// Workspace layout: C [npx][ntri], H [npx][ntri], Sd [npx][n] (256-byte aligned parts).
size_t adjoint_workspace_bytes(int n, const Geom &g) {
    const long long npx = (long long)g.Ho * g.Wo;
    auto a256 = [](size_t v) { return (v + 255) & ~(size_t)255; };
    return 2 * a256((size_t)npx * ntri(n) * sizeof(float2)) + a256((size_t)npx * n * sizeof(float));
}

// Recomputed coherence, diagonal sums and H_p of every output pixel into the
// workspace; *Hout points at H.  npx > 0.
static cudaError_t adjoint_h(const Planes &z, int n, const Geom &g, const uint64_t *mask, int ref,
                             const EmiParams &prm, const float *dphase, void *workspace, cudaStream_t s, Prof *prof,
                             float2 **Hout) {
    const long long npx = (long long)g.Ho * g.Wo;
    auto a256 = [](size_t v) { return (v + 255) & ~(size_t)255; };
    char *ws = static_cast<char *>(workspace);
    float2 *C = reinterpret_cast<float2 *>(ws);
    float2 *H = reinterpret_cast<float2 *>(ws + a256((size_t)npx * ntri(n) * sizeof(float2)));
    float *Sd = reinterpret_cast<float *>(ws + 2 * a256((size_t)npx * ntri(n) * sizeof(float2)));
    *Hout = H;
    if (prof) prof->begin("adjoint_covariance", s);
    cudaError_t e = launch_covariance(z, n, g, mask, C, s);  // recomputed, not stored by the forward pass
    if (prof) prof->end(s);
    if (e != cudaSuccess) return e;
    if (prof) prof->begin("adjoint_pixel", s);
    k_adj_sdiag<<<adj_grid(npx * n), 256, 0, s>>>(z, n, g, mask, Sd);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    e = with_row_length(
        n, [&](auto np) { return run_adj_pixel<decltype(np)::value>(C, Sd, n, npx, ref, prm, dphase, H, s); });
    if (prof) prof->end(s);
    return e;
}

cudaError_t launch_adjoint(const Planes &z, int n, const Geom &g, const uint64_t *mask, int ref,
                           const EmiParams &prm, const float *dphase, void *workspace, float2 *grad,
                           cudaStream_t s, Prof *prof) {
    const long long npx = (long long)g.Ho * g.Wo, npix = (long long)g.H * g.W;
    if (npx == 0) return cudaMemsetAsync(grad, 0, (size_t)npix * n * sizeof(float2), s);
    float2 *H = nullptr;
    cudaError_t e = adjoint_h(z, n, g, mask, ref, prm, dphase, workspace, s, prof, &H);
    if (e != cudaSuccess) return e;
    if (prof) prof->begin("adjoint_gather", s);
    // rows a warp: the fewest padded rows, then the most (reuse of z)
    int rb = 4;
    for (int c = 5; c <= 6; ++c)
        if ((n + c - 1) / c * c <= (n + rb - 1) / rb * rb) rb = c;
    const AdjTile t = scatter_plan(n, g, rb);
    if (t.TY > 0) {
        // tiled scatter (H read once)
        e = cudaMemsetAsync(grad, 0, (size_t)npix * n * sizeof(float2), s);
        if (e == cudaSuccess)
            e = rb == 4   ? run_scatter<4>(z, n, g, mask, H, grad, t, s)
                : rb == 5 ? run_scatter<5>(z, n, g, mask, H, grad, t, s)
                          : run_scatter<6>(z, n, g, mask, H, grad, t, s);
        if (e != cudaSuccess) return e;
    } else {
        // window too large for a shared-memory region: per-element gather
        const int grid = adj_grid(npix * n);
        if (n <= 8) k_adj_gather<8><<<grid, 256, 0, s>>>(z, n, g, mask, H, grad);
        else if (n <= 16) k_adj_gather<16><<<grid, 256, 0, s>>>(z, n, g, mask, H, grad);
        else k_adj_gather<32><<<grid, 256, 0, s>>>(z, n, g, mask, H, grad);
    }
    e = cudaGetLastError();
    if (prof) prof->end(s);
    return e;
}

// Gradient of L = sum(dphase * phase) with respect to the window weights
// [Ho][Wo][wy*wx] (k_adj_wgrad) over the workspace of the adjoint.
cudaError_t launch_weight_gradient(const Planes &z, int n, const Geom &g, const uint64_t *mask, int ref,
                                   const EmiParams &prm, const float *dphase, void *workspace, float *dw,
                                   cudaStream_t s) {
    const long long npx = (long long)g.Ho * g.Wo;
    if (npx == 0) return cudaSuccess;
    float2 *H = nullptr;
    cudaError_t e = adjoint_h(z, n, g, mask, ref, prm, dphase, workspace, s, nullptr, &H);
    if (e != cudaSuccess) return e;
    const int grid = adj_grid(npx * g.wy * g.wx);
    if (n <= 8) k_adj_wgrad<8><<<grid, 256, 0, s>>>(z, n, g, H, dw);
    else if (n <= 16) k_adj_wgrad<16><<<grid, 256, 0, s>>>(z, n, g, H, dw);
    else k_adj_wgrad<32><<<grid, 256, 0, s>>>(z, n, g, H, dw);
    return cudaGetLastError();
}

// First-order phase standard deviations (k_adj_uncert) over the workspace of
// the adjoint: the coherence and the diagonal sums are recomputed there.
cudaError_t launch_phase_uncertainty(const Planes &z, int n, const Geom &g, const uint64_t *mask, int ref,
                                     const EmiParams &prm, float sigma2, void *workspace, float *sd,
                                     cudaStream_t s) {
    const long long npx = (long long)g.Ho * g.Wo;
    if (npx == 0) return cudaSuccess;
    auto a256 = [](size_t v) { return (v + 255) & ~(size_t)255; };
    char *ws = static_cast<char *>(workspace);
    float2 *C = reinterpret_cast<float2 *>(ws);
    float *Sd = reinterpret_cast<float *>(ws + 2 * a256((size_t)npx * ntri(n) * sizeof(float2)));
    cudaError_t e = launch_covariance(z, n, g, mask, C, s);
    if (e != cudaSuccess) return e;
    k_adj_sdiag<<<adj_grid(npx * n), 256, 0, s>>>(z, n, g, mask, Sd);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    float2 *H = reinterpret_cast<float2 *>(ws + a256((size_t)npx * ntri(n) * sizeof(float2)));
    return with_row_length(
        n, [&](auto np) { return run_adj_uncert<decltype(np)::value>(C, Sd, H, n, npx, ref, prm, sigma2, sd, s); });
}

}  // namespace plk
