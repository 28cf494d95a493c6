// Track fit along fixed hit lists: one thread per track, state and covariance in
// registers for the whole hit list (Sec. 1: Kalman-filter fitting), and the
// backward fit, the same filter through the hits in reverse order.
#include <cuda_runtime.h>

#include <type_traits>

#include "mkf_internal.h"

namespace {

using namespace mkf;

struct FitArgs {
    Geom G;
    const float *X, *Y, *Z;
    const int32_t *hit_layer;
    int32_t n_hits;
    const int32_t *hit_idx;
    int32_t max_hits, n;
    const float *seed_par, *seed_cov;
    float inflate;  // backward fit: factor on the starting covariance
    float *sm_par, *sm_cov;  // smoother: [max_hits][6][n], [max_hits][21][n]
    float *out_par, *out_cov, *chi2;
    int32_t *ndf;
    uint32_t *status;
    mkf_fault *fault;
};

__device__ __forceinline__ void record_fault(mkf_fault *f, int code, int where) {
    if (atomicCAS(&f->code, 0, code) == 0) f->where = where;
}

// The helix traversed the other way: the same curve with the momentum turned
// around, p -> (x, y, z, -q/pT, phi + pi, pi - theta) with pi as a float pair
// (phi and theta are pairs too),
// and C -> F C F with F = diag(1, 1, 1, -1, 1, -1) (the covariances between
// {q/pT, theta} and the other parameters change sign).
__device__ __forceinline__ void reverse_state(float p[6], Lo &lo, float C[21]) {
    constexpr float kPiHi = 3.14159274101257324219f;  // float(pi)
    constexpr float kPiLo = -8.74227765734758e-8f;    // pi - float(pi)
    p[3] = -p[3];
    df_add(p[4], lo.phi, kPiHi);
    df_add(p[4], lo.phi, kPiLo);
    df_wrap_pi(p[4], lo.phi);
    float th = kPiHi, thl = kPiLo;
    df_add(th, thl, -p[5]);
    df_add(th, thl, -lo.th);
    p[5] = th;
    lo.th = thl;
#pragma unroll
    for (int i = 0; i < 6; ++i)
#pragma unroll
        for (int j = 0; j <= i; ++j)
            if ((i == 3 || i == 5) != (j == 3 || j == 5)) C[sym(i, j)] = -C[sym(i, j)];
}

// Move the state onto layer Ld (the helix or, for kPhys = 2, Runge-Kutta steps
// in the parameterised field, kCols: see propagate_field); false if the layer is
// not reached.
template <int kPhys, int kCols, class Cov>
__device__ __forceinline__ bool move_to(const Geom &G, const LayerDesc &Ld, float p[6], Lo &lo, Cov C) {
    float sphi, cphi;
    sincos_pair(p[4], lo.phi, sphi, cphi);
    const float cot = cot_pair(p[5], lo.th);
    const float kbl = kPhys == 2 ? G.kb * bz_factor(G.alpha, p[0], p[1], p[2]) : G.kb;
    float s;
    if (!path_to_layer(Ld, kbl, p, lo, sphi, cphi, cot, s)) return false;
    if (kPhys == 2)
        propagate_field<kCols>(Ld, G.kb, G.alpha, p, lo, C, sphi, cphi, -p[3] * kbl, s);
    else
        propagate_transport(Ld, G.kb, p, lo, C, sphi, cphi, cot, s);
    return true;
}

// Kalman update with the hit (xh, yh, zh) on layer Ld; false if the residual
// covariance is not positive definite.
__device__ __forceinline__ bool update_with(const LayerDesc &Ld, float xh, float yh, float zh, float p[6], Lo &lo,
                                            float C[21], float &dchi2) {
    const Frame f = frame_of(p);
    Innov I;
    if (!innovation(Ld.kind, Ld.su2, Ld.sv2, f, C, I)) return false;
    float u, v;
    const float zr = Ld.kind == 0 ? zh : sqrtf(fmaf(xh, xh, yh * yh));
    residual(Ld.kind, Ld.rz, p, lo, f, xh, yh, zr, u, v);
    dchi2 = chi2_of(I, u, v);
    kf_apply_joseph(I, u, v, p, lo, C);
    return true;
}

// The same with the covariance as a square root (the seed hits).
template <int K>
__device__ __forceinline__ bool update_with(const LayerDesc &Ld, float xh, float yh, float zh, float p[6], Lo &lo,
                                            SqrtCov<K> *Q, float &dchi2) {
    const Frame f = frame_of(p);
    float u, v;
    const float zr = Ld.kind == 0 ? zh : sqrtf(fmaf(xh, xh, yh * yh));
    residual(Ld.kind, Ld.rz, p, lo, f, xh, yh, zr, u, v);
    dchi2 = sqrt_update(Ld.kind, Ld.su2, Ld.sv2, f, u, v, p, lo, Q);
    return true;
}

// One row of a track's hit list: the hit (-1: none) with its layer and position.
struct HitRow {
    int h, l;
    float x, y, z;
};

// A track's hits row by row (kBackward: from the last row), each copied into
// shared memory while the row before it is processed, its index loaded one row
// earlier still: the gathers (four of them behind an index load, 700 cycles
// each from L2) then cost the filter no wait, and no registers (prefetched into
// registers they spilled and gained nothing).  The kernel of one event of 1000
// tracks went from 20.5 to 17.3 us (a call takes 23 as before: the host's part
// is longer); for 10^6 tracks see fit_kernel.  Every thread waits for its own
// copies only.  An index outside [0, n_hits) is a device
// fault and taken as no hit.
constexpr int kFitThreads = 128;

template <bool kBackward, bool kAhead>
struct HitFeed {
    const FitArgs &A;
    const int t;
    int kk = 0;       // rows handed out
    int h0, h1 = -1;  // the next row's hit (its copy is under way) and the one after
    __device__ __forceinline__ int row(int i) const { return kBackward ? A.max_hits - 1 - i : i; }
    __device__ __forceinline__ int index(int i) const {
        return i < A.max_hits ? A.hit_idx[(int64_t)row(i) * A.n + t] : -1;
    }
    __device__ __forceinline__ int checked(int h) const {
        if (h < A.n_hits) return h < 0 ? -1 : h;
        record_fault(A.fault, kFaultBadHitIndex, t);
        return -1;
    }
#ifdef __CUDACC__
    float (*buf)[4][kFitThreads];
    __device__ __forceinline__ void copy(int i, int h) {
        if (h >= 0) {
            const void *src[4] = {A.X + h, A.Y + h, A.Z + h, A.hit_layer + h};
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const unsigned dst = static_cast<unsigned>(__cvta_generic_to_shared(&buf[i & 1][c][threadIdx.x]));
                asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst), "l"(src[c]));
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    }
    __device__ __forceinline__ HitFeed(const FitArgs &A_, int t_, float (*buf_)[4][kFitThreads])
        : A(A_), t(t_), buf(buf_) {
        if (!kAhead) return;
        h0 = checked(index(0));
        h1 = index(1);
        copy(0, h0);
    }
#else
    HitFeed(const FitArgs &A_, int t_, float (*)[4][kFitThreads]) : A(A_), t(t_) {}
#endif
    // the next row; false after the last one
    __device__ __forceinline__ bool next(HitRow &r) {
        if (kk >= A.max_hits) return false;
#ifdef __CUDACC__
        if constexpr (kAhead) {
            r.h = h0;
            h0 = checked(h1);
            copy(kk + 1, h0);
            h1 = index(kk + 2);
            asm volatile("cp.async.wait_group 1;" ::: "memory");
            const float (*b)[kFitThreads] = buf[kk & 1];
            if (r.h >= 0) {
                r.x = b[0][threadIdx.x];
                r.y = b[1][threadIdx.x];
                r.z = b[2][threadIdx.x];
                r.l = __float_as_int(b[3][threadIdx.x]);
            }
            ++kk;
            return true;
        }
#endif
        r.h = index(kk++);
        if (kAhead) r.h = checked(r.h);
        else if (r.h >= A.n_hits) r.h = -1;
#ifndef __CUDACC__
        if (kAhead && r.h >= 0) {
            r.l = A.hit_layer[r.h];
            r.x = A.X[r.h];
            r.y = A.Y[r.h];
            r.z = A.Z[r.h];
        }
#endif
        return true;
    }
    // the row handed out last
    __device__ __forceinline__ int k() const { return row(kk - 1); }
};

// The first three hits of a track's list (false: it has fewer); reports the
// invalid indices on the way.
__device__ __forceinline__ bool first_three(const FitArgs &A, int t, int first[3]) {
    int nfirst = 0;
    // the first three rows at once: nearly always the three hits
    int h[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) h[k] = k < A.max_hits ? A.hit_idx[(int64_t)k * A.n + t] : -1;
    for (int k = 0; k < A.max_hits && nfirst < 3; ++k) {
        const int hk = k == 0 ? h[0] : k == 1 ? h[1] : k == 2 ? h[2] : A.hit_idx[(int64_t)k * A.n + t];
        if (hk >= A.n_hits) record_fault(A.fault, kFaultBadHitIndex, t);
        if (hk < 0 || hk >= A.n_hits) continue;
        if (nfirst == 0) first[0] = hk;
        else if (nfirst == 1) first[1] = hk;
        else first[2] = hk;
        ++nfirst;
    }
    return nfirst >= 3;
}

// Blocks of 128 tracks per SM that fit_kernel is compiled for, by physics variant
// (see there), and the choice for a call: more blocks on an SM mean spilled
// registers but fewer waves, and where the last wave is nearly empty that decides.
// A wave of 4, 5 and 6 blocks costs about 16, 18 (backward) and 23 (a full wave,
// material, forward / backward: 86 / 77, - / 91, 121 / 115 us); over many waves
// they come out alike and the variants without spills are taken.  With the
// fewest blocks only, calls just above one wave took as long as two: 110 000
// tracks of 24 rows with material 146 / 131 us, now 121 / 116 (6 blocks); 90 000
// tracks 135 / 121 us, now 106 / 89 (6 / 5 blocks); uniform field, 110 000 tracks
// of 12 rows 54, now 46.  Forward with material 5 blocks are never the best by
// more than 3 %.
constexpr int fit_blocks(int phys) { return phys == 0 ? 5 : phys == 1 ? 4 : 3; }

inline int fit_blocks_for(int phys, bool backward, int blocks, int sms) {
    int best = fit_blocks(phys);
    if (phys == 2) return best;
    auto waves = [&](int k) { return (blocks - 1) / (sms * k) + 1; };
    auto cost = [&](int k) { return static_cast<int64_t>(waves(k)) * (k == 4 ? 16 : k == 5 ? (backward ? 18 : 20) : 23); };
    if (phys == 1 && backward && cost(5) < cost(4)) best = 5;
    if (waves(6) <= (backward ? 1 : 3) && cost(6) < cost(best)) best = 6;
    return best;
}

// kBackward: hits in reverse order from the given state at the last hit, turned
// around and inflated; the result at the first hit is turned back.  kPhys: 0
// uniform field without material; 1 material effects compiled in (selected
// when any layer has material); 2 the parameterised field (Runge-Kutta
// propagation) with the material effects.
// Bound: issue and instruction fetch (the uniform-field fit: 72 % of issue slots,
// the hit code is there twice).  kBlocks per SM, measured with the row feed:
// uniform field 6 / 5 / 4: 334 / 322 / 333 us for 10^6 tracks of 10 hits (at 5
// nothing spills; 336 us before the feed, at 6); material, out and back, 6 / 5 /
// 4 / 3: 384 / 332 / 311 / 342 us for 144 000 tracks of 16 hits (367 us before,
// at 6, where the square root of nine columns spilled 420 bytes a thread);
// parameterised field 4 / 3 / 2: 547 / 497 / 512 us for 10^5 tracks of 10 hits.
// Which one a call gets: fit_blocks_for.  kCols: see propagate_field.  At 6 the rows are loaded where they are
// used: the feed's registers spill (material, forward, 110 000 tracks: 13 % slower).
template <bool kBackward, int kPhys, int kBlocks = fit_blocks(kPhys), int kCols = 1>
__global__ void __launch_bounds__(128, kBlocks) fit_kernel(const __grid_constant__ FitArgs A) {
    constexpr bool kMaterial = kPhys >= 1, kParamField = kPhys == 2;
    constexpr bool kAhead = kBlocks < 6;
    constexpr int kSq = kMaterial ? 9 : 5;  // square-root columns through the seed hits
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= A.n) return;
#ifdef __CUDACC__
    __shared__ float shared[kAhead ? 2 : 1][4][kAhead ? kFitThreads : 1];
    float (*const buf)[4][kFitThreads] = reinterpret_cast<float (*)[4][kFitThreads]>(shared);
#else
    float (*const buf)[4][kFitThreads] = nullptr;
#endif
    const Geom &G = A.G;
    float p[6], C[21];
    SqrtCov<kSq> Q;
    Lo lo{0.f, 0.f, 0.f, 0.f, 0.f};
    uint32_t st = 0;
    float chi2 = 0.f;
    int used = 0;

    int first[3] = {-1, -1, -1};
    bool ok = first_three(A, t, first);
    if (ok) {
        int l0 = A.hit_layer[first[0]];
        if (l0 < 0 || l0 >= G.n_layers) {
            record_fault(A.fault, kFaultBadLayer, first[0]);
            ok = false;
        } else if (A.seed_par) {
#pragma unroll
            for (int i = 0; i < 6; ++i) p[i] = A.seed_par[(int64_t)i * A.n + t];
#pragma unroll
            for (int k = 0; k < 21; ++k) C[k] = A.seed_cov[(int64_t)k * A.n + t];
            if (kBackward) {
                reverse_state(p, lo, C);
#pragma unroll
                for (int k = 0; k < 21; ++k) C[k] *= A.inflate;
            }
        } else {
            float h1[3], h2[3], h3[3], eta;
            h1[0] = A.X[first[0]]; h1[1] = A.Y[first[0]]; h1[2] = A.Z[first[0]];
            h2[0] = A.X[first[1]]; h2[1] = A.Y[first[1]]; h2[2] = A.Z[first[1]];
            h3[0] = A.X[first[2]]; h3[1] = A.Y[first[2]]; h3[2] = A.Z[first[2]];
            // the parameterised field at the middle hit sets the curvature scale
            const float kbs = kParamField ? G.kb * bz_factor(G.alpha, h2[0], h2[1], h2[2]) : G.kb;
            ok = seed_state(G.L[l0], kbs, h1, h2, h3, p, Q, eta);
        }
    }
    if (!ok) st |= MKF_ST_BADSEED;
    if (!ok || !kAhead) {  // (else the feed reports them)
        // the list's invalid indices are reported all the same
        for (int k = 0; k < A.max_hits; ++k)
            if (A.hit_idx[(int64_t)k * A.n + t] >= A.n_hits) record_fault(A.fault, kFaultBadHitIndex, t);
    }

    if (ok) {
        bool firsthit = true;
        // one hit: onto its layer (after the first), material, update; Cx is
        // the covariance (float[21]) or, through the seed hits, its square root
        auto hit = [&](auto Cx, const HitRow &r) {
            const int l = kAhead ? r.l : A.hit_layer[r.h];
            if (l < 0 || l >= G.n_layers) {
                record_fault(A.fault, kFaultBadLayer, r.h);
                return;
            }
            const LayerDesc &Ld = G.L[l];
            if (!firsthit) {
                if (!move_to<kPhys, kCols>(G, Ld, p, lo, Cx)) {
                    st |= MKF_ST_UNREACHABLE;
                    return;
                }
                if (!kBackward && kMaterial) {
                    float mx0, mk;
                    material_at(G, Ld, p, mx0, mk);
                    add_scattering(Ld.kind, mx0, p, Cx);
                    apply_eloss(Ld.kind, mx0, mk, p, Cx, 1.f);
                }
            }
            firsthit = false;
            float dchi2;
            if (update_with(Ld, kAhead ? r.x : A.X[r.h], kAhead ? r.y : A.Y[r.h], kAhead ? r.z : A.Z[r.h], p, lo, Cx,
                            dchi2)) {
                chi2 += dchi2;
                ++used;
            } else {
                st |= MKF_ST_BADS;
            }
            // reversed in time a layer's material follows its hit (at every hit,
            // the last one included): the energy lost there is gained back, then
            // the scattering noise is added
            if (kBackward && kMaterial) {
                float mx0, mk;
                material_at(G, Ld, p, mx0, mk);
                apply_eloss(Ld.kind, mx0, mk, p, Cx, -1.f);
                add_scattering(Ld.kind, mx0, p, Cx);
            }
        };
        HitFeed<kBackward, kAhead> feed(A, t, buf);
        HitRow r;
        if constexpr (!kBackward) {
            if (!A.seed_par) {  // from the seed prior: the seed hits with the square root
                while (used < 3 && feed.next(r))
                    if (r.h >= 0) hit(&Q, r);
                sqrt_to_cov(Q, C);
            }
        }
        while (feed.next(r))
            if (r.h >= 0) hit(C, r);
        if (kBackward) reverse_state(p, lo, C);
        if (!finite_state(p) || !isfinite(chi2)) st |= MKF_ST_NONFINITE;
    }
    const float nanv = __int_as_float(0x7fc00000);
    p[0] += lo.x;
    p[1] += lo.y;
    p[2] += lo.z;
    p[4] += lo.phi;
    p[5] += lo.th;
#pragma unroll
    for (int i = 0; i < 6; ++i) A.out_par[(int64_t)i * A.n + t] = ok ? p[i] : nanv;
#pragma unroll
    for (int k = 0; k < 21; ++k) A.out_cov[(int64_t)k * A.n + t] = ok ? C[k] : nanv;
    A.chi2[t] = chi2;
    A.ndf[t] = 2 * used - (G.kb != 0.f ? 5 : 4);
    A.status[t] = st;
}

// ---------------------------------------------------------------------------
// Smoother: the state at every hit from all of the track's hits (two filters).

// Weighted mean of two independent estimates (pf, Cf), (pb, Cb) of the state on
// a surface, in its five free parameters P p: (u, z, q/pT, phi, theta) on a
// cylinder (u along the surface, perpendicular to the radius at pf), (x, y,
// q/pT, phi, theta) on a disk.  The mean is symmetric in the two; the one with
// the smaller q/pT variance is taken as base (a): with d = P (po - pa) (phi
// wrapped), S = P (Ca + Co) P^T, X = S^-1 P Ca (Cholesky of S scaled to unit
// diagonal) and K = X^T: ps = pa + K d, and Cs in the Joseph form
// (I - K P) Ca (I - K P)^T + K (P Co P^T) K^T, a sum of two positive terms
// instead of the FP32 difference Ca - K P Ca, which cancels where one estimate
// is much sharper than the other.  The mean lies on the surface (radius or
// z = rz): a move along the tangent at pa is put back on it, and the position
// block of Cs is projected onto the tangent plane there.  False if S is not
// positive definite.
__device__ __forceinline__ bool combine5(int kind, float rz, const float pf_[6], const float Cf_[21],
                                         const float pb_[6], const float Cb_[21], float ps[6], float Cs[21]) {
    const bool swap = Cb_[9] < Cf_[9];
    // base (pf, Cf) and other (pb, Cb), by selects: a pointer that chooses
    // between two arrays would put both in local memory
    float pf[6], pb[6], Cf[21], Cb[21];
#pragma unroll
    for (int i = 0; i < 6; ++i) {
        pf[i] = swap ? pb_[i] : pf_[i];
        pb[i] = swap ? pf_[i] : pb_[i];
    }
#pragma unroll
    for (int i = 0; i < 21; ++i) {
        Cf[i] = swap ? Cb_[i] : Cf_[i];
        Cb[i] = swap ? Cf_[i] : Cb_[i];
    }
    float c = 1.f, sn = 0.f;
    if (kind == 0) {
        const float ir = 1.f / sqrtf(fmaf(pf[0], pf[0], pf[1] * pf[1]));
        c = pf[0] * ir;
        sn = pf[1] * ir;
    }
    // P v for a 6-vector v
    auto proj = [&](const float v[6], float o[5]) {
        if (kind == 0) {
            o[0] = fmaf(c, v[1], -sn * v[0]);
            o[1] = v[2];
        } else {
            o[0] = v[0];
            o[1] = v[1];
        }
        o[2] = v[3];
        o[3] = v[4];
        o[4] = v[5];
    };
    float dp[6], d[5];
#pragma unroll
    for (int i = 0; i < 6; ++i) dp[i] = pb[i] - pf[i];
    dp[4] = wrap_pi(dp[4]);
    proj(dp, d);
    // PC = P Cf (5 x 6), PS = P (Cf + Cb) (5 x 6)
    float PC[5][6], PS[5][6];
#pragma unroll
    for (int j = 0; j < 6; ++j) {
        float cf[6], cs[6];
#pragma unroll
        for (int i = 0; i < 6; ++i) {
            cf[i] = Cf[sym(i, j)];
            cs[i] = cf[i] + Cb[sym(i, j)];
        }
        float o[5], q[5];
        proj(cf, o);
        proj(cs, q);
#pragma unroll
        for (int a = 0; a < 5; ++a) {
            PC[a][j] = o[a];
            PS[a][j] = q[a];
        }
    }
    // S = PS P^T, scaled to unit diagonal
    float S[5][5], sc[5];
#pragma unroll
    for (int a = 0; a < 5; ++a) {
        float row[5];
        proj(PS[a], row);
#pragma unroll
        for (int b = 0; b < 5; ++b) S[a][b] = row[b];
    }
#pragma unroll
    for (int a = 0; a < 5; ++a) {
        if (!(S[a][a] > 0.f)) return false;
        sc[a] = 1.f / sqrtf(S[a][a]);
    }
    // Cholesky of the scaled S (lower triangle in place)
    float L[5][5];
#pragma unroll
    for (int a = 0; a < 5; ++a)
#pragma unroll
        for (int b = 0; b <= a; ++b) {
            float v = S[a][b] * sc[a] * sc[b];
#pragma unroll
            for (int m = 0; m < b; ++m) v = fmaf(-L[a][m], L[b][m], v);
            if (a == b) {
                if (!(v > 0.f)) return false;
                L[a][a] = sqrtf(v);
            } else {
                L[a][b] = v / L[b][b];
            }
        }
    // X = S^-1 PC column by column (and S^-1 d), through the scaling
    float X[5][6], y[5];
#pragma unroll
    for (int j = 0; j < 7; ++j) {
        float r[5];
#pragma unroll
        for (int a = 0; a < 5; ++a) r[a] = (j < 6 ? PC[a][j] : d[a]) * sc[a];
#pragma unroll
        for (int a = 0; a < 5; ++a) {
            float v = r[a];
#pragma unroll
            for (int m = 0; m < a; ++m) v = fmaf(-L[a][m], r[m], v);
            r[a] = v / L[a][a];
        }
#pragma unroll
        for (int a = 4; a >= 0; --a) {
            float v = r[a];
#pragma unroll
            for (int m = a + 1; m < 5; ++m) v = fmaf(-L[m][a], r[m], v);
            r[a] = v / L[a][a];
        }
#pragma unroll
        for (int a = 0; a < 5; ++a) {
            if (j < 6)
                X[a][j] = r[a] * sc[a];
            else
                y[a] = r[a] * sc[a];
        }
    }
    // ps = pf + Cf P^T S^-1 d = pf + PC^T y
#pragma unroll
    for (int i = 0; i < 6; ++i) {
        float v = pf[i];
#pragma unroll
        for (int a = 0; a < 5; ++a) v = fmaf(PC[a][i], y[a], v);
        ps[i] = v;
    }
    ps[4] = wrap_pi(ps[4]);
    if (kind == 0) {
        const float f = rz / sqrtf(fmaf(ps[0], ps[0], ps[1] * ps[1]));
        ps[0] *= f;
        ps[1] *= f;
    } else {
        ps[2] = rz;
    }
    // Joseph form with K[i][a] = X[a][i]: A = I - K P
    float Am[6][6];
#pragma unroll
    for (int i = 0; i < 6; ++i) {
        float e[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        e[i] = 1.f;
        float kp[6];
        if (kind == 0) {
            kp[0] = -sn * X[0][i];
            kp[1] = c * X[0][i];
            kp[2] = X[1][i];
        } else {
            kp[0] = X[0][i];
            kp[1] = X[1][i];
            kp[2] = 0.f;
        }
        kp[3] = X[2][i];
        kp[4] = X[3][i];
        kp[5] = X[4][i];
#pragma unroll
        for (int j = 0; j < 6; ++j) Am[i][j] = e[j] - kp[j];
    }
    // R = P Co P^T = P (Cf + Cb) P^T - P Cf P^T would cancel: from Co directly
    float R[5][5];
#pragma unroll
    for (int j = 0; j < 6; ++j) {
        float cb[6];
#pragma unroll
        for (int i = 0; i < 6; ++i) cb[i] = Cb[sym(i, j)];
        float o[5];
        proj(cb, o);
#pragma unroll
        for (int a = 0; a < 5; ++a) PS[a][j] = o[a];  // reuse: P Co
    }
#pragma unroll
    for (int a = 0; a < 5; ++a) {
        float row[5];
        proj(PS[a], row);
#pragma unroll
        for (int b = 0; b < 5; ++b) R[a][b] = row[b];
    }
    // M = A Ca, KR = K R
    float M[6][6], KR[6][5];
#pragma unroll
    for (int i = 0; i < 6; ++i) {
#pragma unroll
        for (int j = 0; j < 6; ++j) {
            float v = 0.f;
#pragma unroll
            for (int m = 0; m < 6; ++m) v = fmaf(Am[i][m], Cf[sym(m, j)], v);
            M[i][j] = v;
        }
#pragma unroll
        for (int b = 0; b < 5; ++b) {
            float v = 0.f;
#pragma unroll
            for (int a = 0; a < 5; ++a) v = fmaf(X[a][i], R[a][b], v);
            KR[i][b] = v;
        }
    }
#pragma unroll
    for (int i = 0; i < 6; ++i)
#pragma unroll
        for (int j = 0; j <= i; ++j) {
            float v = 0.f;
#pragma unroll
            for (int m = 0; m < 6; ++m) v = fmaf(M[i][m], Am[j][m], v);
#pragma unroll
            for (int b = 0; b < 5; ++b) v = fmaf(KR[i][b], X[b][j], v);
            Cs[sym(i, j)] = v;
        }
    // no variance along the surface normal n at ps: Cs -> (I - n n^T) Cs (I - n n^T)
    float nv[3] = {0.f, 0.f, 1.f};
    if (kind == 0) {
        const float ir = 1.f / sqrtf(fmaf(ps[0], ps[0], ps[1] * ps[1]));
        nv[0] = ps[0] * ir, nv[1] = ps[1] * ir, nv[2] = 0.f;
    }
    float Q[6][6];
#pragma unroll
    for (int j = 0; j < 6; ++j) {
        float col[6];
#pragma unroll
        for (int i = 0; i < 6; ++i) col[i] = Cs[sym(i, j)];
        const float v = fmaf(nv[0], col[0], fmaf(nv[1], col[1], nv[2] * col[2]));
#pragma unroll
        for (int i = 0; i < 3; ++i) col[i] = fmaf(-nv[i], v, col[i]);
#pragma unroll
        for (int i = 0; i < 6; ++i) Q[i][j] = col[i];
    }
#pragma unroll
    for (int i = 0; i < 6; ++i) {
        const float v = fmaf(nv[0], Q[i][0], fmaf(nv[1], Q[i][1], nv[2] * Q[i][2]));
#pragma unroll
        for (int j = 0; j < 3; ++j) Q[i][j] = fmaf(-nv[j], v, Q[i][j]);
    }
#pragma unroll
    for (int i = 0; i < 6; ++i)
#pragma unroll
        for (int j = 0; j <= i; ++j) Cs[sym(i, j)] = Q[i][j];
    return true;
}

// One thread per track: the forward filter writes its state after each hit
// into that hit's output row; the backward filter then starts from the state at
// the last hit (turned around, covariance times inflate), predicts each earlier
// hit from the later ones, replaces the row by the weighted mean of the two
// (combine5) and is updated with the hit, its material applied in reverse.  The
// last hit's row keeps the forward state.
// Bound: issue and the local memory of what does not fit in registers.  Blocks
// per SM 5 / 4 / 3 / 2: 602 / 273 / 211 / 229 us for 10^5 tracks of 9 hits (12
// rows); 334 us with every row set to NaN first, the two estimates of the mean
// chosen through pointers (both then lay in local memory) and 4 blocks.
template <int kPhys>
__global__ void __launch_bounds__(128, 3) smooth_kernel(const __grid_constant__ FitArgs A) {
    constexpr bool kMaterial = kPhys >= 1, kParamField = kPhys == 2;
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= A.n) return;
    const Geom &G = A.G;
    const float nanv = __int_as_float(0x7fc00000);
    const int64_t n = A.n;
#ifdef __CUDACC__
    __shared__ float buf[2][4][kFitThreads];
#else
    float (*const buf)[4][kFitThreads] = nullptr;
#endif
    auto no_state = [&](int k) {
#pragma unroll
        for (int i = 0; i < 6; ++i) A.sm_par[((int64_t)k * 6 + i) * n + t] = nanv;
#pragma unroll
        for (int i = 0; i < 21; ++i) A.sm_cov[((int64_t)k * 21 + i) * n + t] = nanv;
    };
    constexpr int kSq = kMaterial ? 9 : 5;  // square-root columns through the seed hits
    float p[6], C[21];
    SqrtCov<kSq> Q;
    Lo lo{0.f, 0.f, 0.f, 0.f, 0.f};
    uint32_t st = 0;
    float chi2 = 0.f;
    int used = 0;
    int first[3] = {-1, -1, -1};
    bool ok = first_three(A, t, first);
    if (ok) {
        const int l0 = A.hit_layer[first[0]];
        if (l0 < 0 || l0 >= G.n_layers) {
            record_fault(A.fault, kFaultBadLayer, first[0]);
            ok = false;
        } else if (A.seed_par) {
#pragma unroll
            for (int i = 0; i < 6; ++i) p[i] = A.seed_par[(int64_t)i * n + t];
#pragma unroll
            for (int k = 0; k < 21; ++k) C[k] = A.seed_cov[(int64_t)k * n + t];
        } else {
            float h1[3], h2[3], h3[3], eta;
            h1[0] = A.X[first[0]]; h1[1] = A.Y[first[0]]; h1[2] = A.Z[first[0]];
            h2[0] = A.X[first[1]]; h2[1] = A.Y[first[1]]; h2[2] = A.Z[first[1]];
            h3[0] = A.X[first[2]]; h3[1] = A.Y[first[2]]; h3[2] = A.Z[first[2]];
            const float kbs = kParamField ? G.kb * bz_factor(G.alpha, h2[0], h2[1], h2[2]) : G.kb;
            ok = seed_state(G.L[l0], kbs, h1, h2, h3, p, Q, eta);
        }
    }
    if (!ok) {
        st |= MKF_ST_BADSEED;
        // no states; the list's invalid indices are reported all the same
        for (int k = 0; k < A.max_hits; ++k) {
            if (A.hit_idx[(int64_t)k * n + t] >= A.n_hits) record_fault(A.fault, kFaultBadHitIndex, t);
            no_state(k);
        }
    }

    // forward filter, its state after each hit kept in the hit's row (a row
    // without one is set to NaN here, not all rows first: a pass less over the output)
    int lastk = -1;
    unsigned long long have = 0;  // rows with a forward state
    if (ok) {
        bool firsthit = true;
        // one hit; Cx is the covariance (float[21]) or, through the seed hits,
        // its square root
        auto fwd = [&](auto Cx, int k, const HitRow &r) {
            if (r.l < 0 || r.l >= G.n_layers) {
                record_fault(A.fault, kFaultBadLayer, r.h);
                return;
            }
            const LayerDesc &Ld = G.L[r.l];
            if (!firsthit) {
                if (!move_to<kPhys, 1>(G, Ld, p, lo, Cx)) {
                    st |= MKF_ST_UNREACHABLE;
                    return;
                }
                if (kMaterial) {
                    float mx0, mk;
                    material_at(G, Ld, p, mx0, mk);
                    add_scattering(Ld.kind, mx0, p, Cx);
                    apply_eloss(Ld.kind, mx0, mk, p, Cx, 1.f);
                }
            }
            firsthit = false;
            float dchi2;
            if (update_with(Ld, r.x, r.y, r.z, p, lo, Cx, dchi2)) {
                chi2 += dchi2;
                ++used;
                const float pw[6] = {p[0] + lo.x, p[1] + lo.y, p[2] + lo.z, p[3], p[4] + lo.phi, p[5] + lo.th};
#pragma unroll
                for (int i = 0; i < 6; ++i) A.sm_par[((int64_t)k * 6 + i) * n + t] = pw[i];
                float Cw[21];
                if constexpr (std::is_same_v<decltype(Cx), float *>) {
#pragma unroll
                    for (int i = 0; i < 21; ++i) Cw[i] = Cx[i];
                } else {
                    sqrt_to_cov(*Cx, Cw);
                }
#pragma unroll
                for (int i = 0; i < 21; ++i) A.sm_cov[((int64_t)k * 21 + i) * n + t] = Cw[i];
                lastk = k;
                have |= 1ull << k;
            } else {
                st |= MKF_ST_BADS;
            }
        };
        HitFeed<false, true> feed(A, t, buf);
        HitRow r;
        auto row = [&](auto Cx) {
            const int k = feed.k();
            if (r.h >= 0) fwd(Cx, k, r);
            if (!((have >> k) & 1ull)) no_state(k);
        };
        if (!A.seed_par) {  // from the seed prior: the seed hits with the square root
            while (used < 3 && feed.next(r)) row(&Q);
            sqrt_to_cov(Q, C);
        }
        while (feed.next(r)) row(C);
    }

    // backward filter and the weighted means
    if (lastk >= 0 && finite_state(p) && isfinite(chi2)) {
#pragma unroll
        for (int i = 0; i < 6; ++i) p[i] = A.sm_par[((int64_t)lastk * 6 + i) * n + t];
#pragma unroll
        for (int i = 0; i < 21; ++i) C[i] = A.sm_cov[((int64_t)lastk * 21 + i) * n + t] * A.inflate;
        lo = Lo{0.f, 0.f, 0.f, 0.f, 0.f};
        reverse_state(p, lo, C);
        for (int k = lastk; k >= 0; --k) {
            const int h = A.hit_idx[(int64_t)k * n + t];
            if (h < 0 || h >= A.n_hits) continue;
            const int l = A.hit_layer[h];
            if (l < 0 || l >= G.n_layers) continue;
            const LayerDesc &Ld = G.L[l];
            if (k < lastk) {
                if (!move_to<kPhys, 1>(G, Ld, p, lo, C)) {
                    st |= MKF_ST_UNREACHABLE;
                    continue;
                }
                float pf[6], Cf[21];
                bool had = (have >> k) & 1ull;  // the forward filter has a state here
                if (had) {
#pragma unroll
                    for (int i = 0; i < 6; ++i) pf[i] = A.sm_par[((int64_t)k * 6 + i) * n + t];
#pragma unroll
                    for (int i = 0; i < 21; ++i) Cf[i] = A.sm_cov[((int64_t)k * 21 + i) * n + t];
                    had = Cf[0] == Cf[0];
                }
                if (had) {
                    float pb[6] = {p[0] + lo.x, p[1] + lo.y, p[2] + lo.z, p[3], p[4], p[5]}, Cb[21];
                    Lo lb{0.f, 0.f, 0.f, lo.phi, lo.th};
#pragma unroll
                    for (int i = 0; i < 21; ++i) Cb[i] = C[i];
                    reverse_state(pb, lb, Cb);
                    pb[4] += lb.phi;
                    pb[5] += lb.th;
                    float ps[6], Cs[21];
                    const bool good = combine5(Ld.kind, Ld.rz, pf, Cf, pb, Cb, ps, Cs);
                    if (!good) st |= MKF_ST_BADS;
#pragma unroll
                    for (int i = 0; i < 6; ++i) A.sm_par[((int64_t)k * 6 + i) * n + t] = good ? ps[i] : nanv;
#pragma unroll
                    for (int i = 0; i < 21; ++i) A.sm_cov[((int64_t)k * 21 + i) * n + t] = good ? Cs[i] : nanv;
                }
            }
            float dchi2;
            if (!update_with(Ld, A.X[h], A.Y[h], A.Z[h], p, lo, C, dchi2)) st |= MKF_ST_BADS;
            if (kMaterial) {
                float mx0, mk;
                material_at(G, Ld, p, mx0, mk);
                apply_eloss(Ld.kind, mx0, mk, p, C, -1.f);
                add_scattering(Ld.kind, mx0, p, C);
            }
        }
    }
    if (!isfinite(chi2)) st |= MKF_ST_NONFINITE;
    A.chi2[t] = chi2;
    A.ndf[t] = 2 * used - (G.kb != 0.f ? 5 : 4);
    A.status[t] = st;
}

}  // namespace

// mode: 0 forward fit, 1 backward fit, 2 smoother (out_par / out_cov are then
// the per-hit arrays [max_hits][6][n] / [max_hits][21][n]).
static mkf_status launch_fit(mkf_ctx *ctx, const float *xyz, const int32_t *hit_layer, int32_t n_hits,
                             const int32_t *hit_idx, int32_t max_hits, int32_t n, const float *seed_par,
                             const float *seed_cov, float inflate, int mode, float *out_par, float *out_cov,
                             float *chi2, int32_t *ndf, uint32_t *status) {
    const bool backward = mode == 1;
    if (!ctx) return MKF_ERR_ARG;
    if (!ctx->has_geom) return MKF_ERR_GEOMETRY;
    if (n < 0 || n_hits < 0 || max_hits < 1) return MKF_ERR_ARG;
    if (max_hits > MKF_MAX_LAYERS) return MKF_ERR_CAPACITY;
    if (n_hits > MKF_MAX_HITS) return MKF_ERR_CAPACITY;
    if ((seed_par == nullptr) != (seed_cov == nullptr)) return MKF_ERR_ARG;
    if (mode != 0 && !(inflate >= 1.f && inflate < 3.0e38f)) return MKF_ERR_ARG;
    if (n == 0) return MKF_OK;
    if (!xyz || !hit_layer || !hit_idx || !out_par || !out_cov || !chi2 || !ndf || !status) return MKF_ERR_ARG;
    if (backward && !seed_par) return MKF_ERR_ARG;
    DeviceGuard g(ctx->device);
    if (!g.ok) return MKF_ERR_CUDA;
    FitArgs A;
    A.G = ctx->geom;
    A.X = xyz;
    A.Y = xyz + n_hits;
    A.Z = xyz + 2 * (int64_t)n_hits;
    A.hit_layer = hit_layer;
    A.n_hits = n_hits;
    A.hit_idx = hit_idx;
    A.max_hits = max_hits;
    A.n = n;
    A.seed_par = seed_par;
    A.seed_cov = seed_cov;
    A.inflate = inflate;
    A.out_par = mode == 2 ? nullptr : out_par;
    A.out_cov = mode == 2 ? nullptr : out_cov;
    A.sm_par = mode == 2 ? out_par : nullptr;
    A.sm_cov = mode == 2 ? out_cov : nullptr;
    A.chi2 = chi2;
    A.ndf = ndf;
    A.status = status;
    A.fault = ctx->fault;
    const int threads = kFitThreads;
    const int blocks = (n + threads - 1) / threads;
    if (mode == 2) {
        switch (mkf_phys_variant(ctx->geom)) {
            case 0: smooth_kernel<0><<<blocks, threads, 0, ctx->stream>>>(A); break;
            case 1: smooth_kernel<1><<<blocks, threads, 0, ctx->stream>>>(A); break;
            default: smooth_kernel<2><<<blocks, threads, 0, ctx->stream>>>(A); break;
        }
        MKF_CUDA_TRY(cudaGetLastError());
        return MKF_OK;
    }
    const int phys = mkf_phys_variant(ctx->geom);
    const int per_sm = fit_blocks_for(phys, backward, blocks, ctx->num_sms);
    typedef void (*FitFn)(FitArgs);
    FitFn fn;
    switch ((phys == 2 ? 6 : phys * 3 + per_sm - 4) + (backward ? 7 : 0)) {
        case 1: fn = fit_kernel<false, 0, 5>; break;
        case 2: fn = fit_kernel<false, 0, 6>; break;
        case 3: fn = fit_kernel<false, 1, 4>; break;
        case 5: fn = fit_kernel<false, 1, 6>; break;
        case 6:
            // forward in the field, up to a wave: two columns of a move at a time (1000
            // tracks 161 -> 155 us, 38 000 241 -> 237; 100 000 500 -> 506; backward the
            // other way round: 151 -> 155 us for 1000)
            fn = blocks <= fit_blocks(2) * ctx->num_sms ? fit_kernel<false, 2, fit_blocks(2), 2> : fit_kernel<false, 2>;
            break;
        case 8: fn = fit_kernel<true, 0, 5>; break;
        case 9: fn = fit_kernel<true, 0, 6>; break;
        case 10: fn = fit_kernel<true, 1, 4>; break;
        case 11: fn = fit_kernel<true, 1, 5>; break;
        case 12: fn = fit_kernel<true, 1, 6>; break;
        default: fn = fit_kernel<true, 2>; break;
    }
    fn<<<blocks, threads, 0, ctx->stream>>>(A);
    MKF_CUDA_TRY(cudaGetLastError());
    return MKF_OK;
}

extern "C" mkf_status mkf_fit(mkf_ctx *ctx, const float *xyz, const int32_t *hit_layer, int32_t n_hits,
                              const int32_t *hit_idx, int32_t max_hits, int32_t n, const float *seed_par,
                              const float *seed_cov, float *out_par, float *out_cov, float *chi2, int32_t *ndf,
                              uint32_t *status) {
    return launch_fit(ctx, xyz, hit_layer, n_hits, hit_idx, max_hits, n, seed_par, seed_cov, 1.f, 0, out_par,
                      out_cov, chi2, ndf, status);
}

extern "C" mkf_status mkf_fit_backward(mkf_ctx *ctx, const float *xyz, const int32_t *hit_layer, int32_t n_hits,
                                       const int32_t *hit_idx, int32_t max_hits, int32_t n, const float *last_par,
                                       const float *last_cov, float inflate, float *out_par, float *out_cov,
                                       float *chi2, int32_t *ndf, uint32_t *status) {
    return launch_fit(ctx, xyz, hit_layer, n_hits, hit_idx, max_hits, n, last_par, last_cov, inflate, 1, out_par,
                      out_cov, chi2, ndf, status);
}

extern "C" mkf_status mkf_fit_smooth(mkf_ctx *ctx, const float *xyz, const int32_t *hit_layer, int32_t n_hits,
                                     const int32_t *hit_idx, int32_t max_hits, int32_t n, const float *seed_par,
                                     const float *seed_cov, float inflate, float *sm_par, float *sm_cov, float *chi2,
                                     int32_t *ndf, uint32_t *status) {
    return launch_fit(ctx, xyz, hit_layer, n_hits, hit_idx, max_hits, n, seed_par, seed_cov, inflate, 2, sm_par,
                      sm_cov, chi2, ndf, status);
}
