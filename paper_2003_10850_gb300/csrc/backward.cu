// backward.cu -- adjoint of the density and force passes (sph_backward).
//
// Given seeds abar_i = dL/da_i and rhobar_i = dL/drho_i for all particles,
// returns dL/dx, dL/du and dL/dm through the whole forward chain:
//   h_i(x)        implicit: N_i(h_i, x) = N_t (number-weighted, mass-free)
//   rho_i, D_i    = sum_j m_j {W, dW/dh}(r_ij, h_i)
//   Omega_i       = 1 / (1 + h_i D_i / (3 rho_i))
//   a_i           = sum_j m_j G_ij (x_j - x_i),
//   G_ij          = A_i F(r,h_i) + A_j F(r,h_j) + Pi_ij (F(r,h_i)+F(r,h_j))/2,
//   A = Omega (gamma-1) u / rho, c = sqrt(gamma (gamma-1) u), F = W_r / r.
// Reverse mode runs as three gathers over each particle's symmetric pair set
// (j != k, r_kj < max(h_k, h_j)), so every particle collects its own adjoint
// without atomics (deterministic):
//   pass 0  force adjoint: x, m (explicit), and the adjoints of h, A, c, rho;
//           per particle it then folds A, c into u, Omega, rho and the Omega
//           adjoint into h, D, rho;
//   pass 1  density adjoint: x and m through rho and D, h through D, and the
//           implicit-h multiplier lambda_k = hbar_k / (dN_k/dh_k);
//   pass 2  implicit h: x through N, weighted by lambda.
// The pair sets come from the neighbour lists and extra partners that an
// all-active density call recorded (k_bw_list), when they are the ones of this
// state; particles the lists cannot serve, or all of them, walk the hierarchy
// (k_backward). FP32 pair terms with compensated sums. The paper has no
// gradients; this is the build's extension of its hot path.
#include <algorithm>

#include "wpp.cuh"

namespace sph {

constexpr int kBwThreads = 128;
constexpr int kBwStack = 96;

// w, w', w'' of the cubic spline (branch-free, as spline()).
__device__ __forceinline__ void spline2(float q, float& w, float& dw, float& ddw) {
    const float a = fmaxf(1.f - q, 0.f), b = fmaxf(0.5f - q, 0.f);
    const float a2 = a * a, b2 = b * b;
    w = 2.f * a2 * a - 8.f * b2 * b;
    dw = 24.f * b2 - 6.f * a2;
    ddw = 12.f * a - 48.f * b;
}

__device__ __forceinline__ bool bw_node_near(uint4 c, float4 e, uint4 X, float sf, float R) {
    const float dx = (float)(int)(c.x - X.x) * sf, dy = (float)(int)(c.y - X.y) * sf,
                dz = (float)(int)(c.z - X.z) * sf;
    const float gx = fmaxf(fabsf(dx) - e.x, 0.f), gy = fmaxf(fabsf(dy) - e.y, 0.f),
                gz = fmaxf(fabsf(dz) - e.z, 0.f);
    const float Rt = R * (1.f + 3.0517578125e-05f) + 2.384185791015625e-07f * (fabsf(dx) + fabsf(dy) + fabsf(dz)) +
                     4.f * sf;
    return gx * gx + gy * gy + gz * gz < Rt * Rt;
}

struct BwArgs {
    const BoxDesc* boxes;
    int n_boxes;
    int n;
    const uint4* posm;
    const float4* posf;
    const uint4* node_c;
    const float4* node_e;
    const float4* fvel;     // v, h
    const float4* fthermo;  // rho, A, c, 1/h
    const float4* ga;       // abar (xyz), rhobar seed (w)
    const float* u;         // sorted u
    const float* omega;     // sorted Omega
    float4* xbar;           // accumulated dL/dx (xyz)
    float* mbar;
    float* ubar;
    float* hbar;
    float4* rd;             // total rhobar, Dbar, mass, 1/h
    float* lam;
    float alpha, gamma;
    // neighbour lists (nbr NULL: every particle walks)
    const float4* fvm;      // v, m
    const int32_t* nbr;
    const int32_t* nbr_off;
    const int32_t* nbr_n;
    const int32_t* ext;
    const uint32_t* ext_n;
    const uint4* list_xh;   // integer position, h bits
    const uint32_t* list_ep;
    unsigned* list_st;
    int32_t* fb_list;
};

// Sorted copies of the seeds, u and Omega. With lists (list_xh given): note
// in *changed whether any particle's position or h differs from the one its
// list was made with; the lists then serve nobody.
__global__ void k_bw_prep(int n, const int32_t* __restrict__ perm, const float* __restrict__ g_acc,
                          const float* __restrict__ g_rho, const float* __restrict__ u,
                          const float* __restrict__ omega, float4* __restrict__ ga, float* __restrict__ us,
                          float* __restrict__ oms, const float* __restrict__ h, const uint4* __restrict__ posm,
                          const uint4* __restrict__ list_xh, unsigned* changed) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= n) return;
    const int o = perm[p];
    if (list_xh) {
        const uint4 X = posm[p], Y = list_xh[p];
        if (X.x != Y.x || X.y != Y.y || X.z != Y.z || !(h[o] == __uint_as_float(Y.w))) atomicOr(changed, 1u);
    }
    ga[p] = make_float4(g_acc[3 * (size_t)o], g_acc[3 * (size_t)o + 1], g_acc[3 * (size_t)o + 2],
                        g_rho ? g_rho[o] : 0.f);
    us[p] = u[o];
    oms[p] = omega[o];
}

__global__ void k_bw_scatter(int n, const int32_t* __restrict__ perm, const float4* __restrict__ xbar,
                             const float* __restrict__ ubar, const float* __restrict__ mbar,
                             float* __restrict__ g_pos, float* __restrict__ g_u, float* __restrict__ g_mass) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= n) return;
    const int o = perm[p];
    const float4 x = xbar[p];
    g_pos[3 * (size_t)o] = x.x;
    g_pos[3 * (size_t)o + 1] = x.y;
    g_pos[3 * (size_t)o + 2] = x.z;
    g_u[o] = ubar[p];
    g_mass[o] = mbar[p];
}

// The particle's own constants.
struct BwI {
    float vx, vy, vz;
    float h, hinv, rho, A, c, n4, m;   // n4 = (8/pi) h^-4
    float4 g;                          // pass 0: abar, rhobar seed
    float2 rd;                         // pass 1: rhobar, Dbar
    float lam;                         // pass 2
};
// A partner's.
struct BwJ {
    float h, hinv, m;
    float4 v, t, g;   // pass 0: (v, -), (rho, A, c, -), abar
    float2 rd;        // pass 1
    float lam;        // pass 2
};
struct BwSum {
    float x = 0.f, y = 0.f, z = 0.f, m = 0.f, h = 0.f, A = 0.f, c = 0.f, r = 0.f, dN = 0.f;
};

template <int PASS>
__device__ __forceinline__ BwI bw_own(const BwArgs& a, int k, uint4 X) {
    const float kN = 2.5464790894703255f;  // 8/pi
    const float4 v = a.fvel[k], t = a.fthermo[k];
    BwI I;
    I.vx = v.x; I.vy = v.y; I.vz = v.z;
    I.h = v.w; I.hinv = t.w; I.rho = t.x; I.A = t.y; I.c = t.z;
    I.n4 = kN * t.w * t.w * t.w * t.w;
    I.m = __uint_as_float(X.w);
    I.g = make_float4(0.f, 0.f, 0.f, 0.f);
    I.rd = make_float2(0.f, 0.f);
    I.lam = 0.f;
    if (PASS == 0) I.g = a.ga[k];
    if (PASS == 1) {
        const float4 q = a.rd[k];
        I.rd = make_float2(q.x, q.y);
    }
    if (PASS == 2) I.lam = a.lam[k];
    return I;
}

// One pair's terms, d = x_j - x_k, r2 = |d|^2 > 0, added to P.
template <int PASS>
__device__ __forceinline__ void bw_pair(const BwI& K, const BwJ& J, float alpha, float dx, float dy, float dz, float r2,
                                        BwSum& P) {
    const float kN = 2.5464790894703255f;  // 8/pi
    const float rinv = rsqrtf(r2), r = r2 * rinv;
    const float ux = dx * rinv, uy = dy * rinv, uz = dz * rinv;   // d-hat; e_kj = -d-hat
    const float qk = r * K.hinv, qj = r * J.hinv;
    float wk, dwk, ddwk, wj, dwj, ddwj;
    spline2(qk, wk, dwk, ddwk);
    spline2(qj, wj, dwj, ddwj);
    if (PASS == 0) {
        const float rhoj = J.t.x, Aj = J.t.y, cj = J.t.z;
        const float nj4 = kN * J.hinv * J.hinv * J.hinv * J.hinv;
        const float Fk = K.n4 * dwk * rinv, Fj = nj4 * dwj * rinv;
        const float Fbar = 0.5f * (Fk + Fj);
        // F_r = (8/pi) h^-4 (w''/(h r) - w'/r^2), F_h = -(8/pi) h^-5 (4w' + q w'')/r
        const float Frk = K.n4 * (ddwk * K.hinv * rinv - dwk * rinv * rinv);
        const float Frj = nj4 * (ddwj * J.hinv * rinv - dwj * rinv * rinv);
        const float Fhk = -K.n4 * K.hinv * (4.f * dwk + qk * ddwk) * rinv;
        const float vx = K.vx - J.v.x, vy = K.vy - J.v.y, vz = K.vz - J.v.z;   // v_kj
        const float w = -(vx * ux + vy * uy + vz * uz);                        // v_kj . r_kj / r
        const float rbar = 0.5f * (K.rho + rhoj);
        const float vsig = K.c + cj - 3.f * w;
        const bool visc = w < 0.f;
        const float PI = visc ? -0.5f * alpha * vsig * w / rbar : 0.f;
        const float PIw = visc ? -0.5f * alpha * (vsig - 3.f * w) / rbar : 0.f;
        const float PIc = visc ? -0.5f * alpha * w / rbar : 0.f;
        const float PIr = visc ? -0.5f * PI / rbar : 0.f;
        const float G = K.A * Fk + Aj * Fj + PI * Fbar;
        const float Gr = (K.A + 0.5f * PI) * Frk + (Aj + 0.5f * PI) * Frj;
        const float Gw = Fbar * PIw;
        const float s1 = K.g.x * dx + K.g.y * dy + K.g.z * dz;      // abar_k . d
        const float s2 = -(J.g.x * dx + J.g.y * dy + J.g.z * dz);   // abar_j . (x_k - x_j)
        const float S = J.m * s1 + K.m * s2;
        const float cw = S * Gw * rinv;
        P.x += G * (K.m * J.g.x - J.m * K.g.x) - S * Gr * ux + cw * (vx + w * ux);
        P.y += G * (K.m * J.g.y - J.m * K.g.y) - S * Gr * uy + cw * (vy + w * uy);
        P.z += G * (K.m * J.g.z - J.m * K.g.z) - S * Gr * uz + cw * (vz + w * uz);
        P.h += S * (K.A + 0.5f * PI) * Fhk;
        P.A += S * Fk;
        P.c += S * Fbar * PIc;
        P.r += S * Fbar * PIr;
        P.m += G * s2;
    } else if (PASS == 1) {
        const float nj4 = kN * J.hinv * J.hinv * J.hinv * J.hinv;
        // W_r = (8/pi) h^-4 w', W_hr = -(8/pi) h^-5 (4w' + q w''), W = (8/pi) h^-3 w,
        // W_h = -(8/pi) h^-4 (3w + q w'), W_hh = (8/pi) h^-5 (12w + 8q w' + q^2 w'')
        const float Wrk = K.n4 * dwk, Wrj = nj4 * dwj;
        const float Whrk = -K.n4 * K.hinv * (4.f * dwk + qk * ddwk);
        const float Whrj = -nj4 * J.hinv * (4.f * dwj + qj * ddwj);
        const float coef = K.rd.x * J.m * Wrk + J.rd.x * K.m * Wrj + K.rd.y * J.m * Whrk + J.rd.y * K.m * Whrj;
        P.x -= coef * ux;   // e_kj = -d-hat
        P.y -= coef * uy;
        P.z -= coef * uz;
        P.m += J.rd.x * (nj4 * J.h * wj) + J.rd.y * (-nj4 * (3.f * wj + qj * dwj));
        P.h += J.m * K.n4 * K.hinv * (12.f * wk + 8.f * qk * dwk + qk * qk * ddwk);
        P.dN += qk * dwk;
    } else {
        const float coef = -(32.f / 3.f) * (K.lam * dwk * K.hinv + J.lam * dwj * J.hinv);
        P.x -= coef * ux;   // e_kj = -d-hat
        P.y -= coef * uy;
        P.z -= coef * uz;
    }
}

// The particle's outputs of the pass from its pair sums.
template <int PASS>
__device__ __forceinline__ void bw_finish(const BwArgs& a, int k, const BwI& K, const BwSum& S) {
    const float gam = a.gamma;
    if (PASS == 0) {
        const float om = a.omega[k], uk = a.u[k];
        const float ubar = S.A * om * (gam - 1.f) / K.rho + (K.c > 0.f ? S.c * gam * (gam - 1.f) / (2.f * K.c) : 0.f);
        const float Ombar = S.A * (gam - 1.f) * uk / K.rho;
        const float D = 3.f * K.rho * (1.f / om - 1.f) * K.hinv;         // d rho / d h from Omega
        const float Bbar = -Ombar * om * om;
        const float rhobar = S.r - S.A * K.A / K.rho + K.g.w - Bbar * K.h * D / (3.f * K.rho * K.rho);
        const float hbar = S.h + Bbar * D / (3.f * K.rho) + rhobar * D;
        a.xbar[k] = make_float4(S.x, S.y, S.z, 0.f);
        a.mbar[k] = S.m;
        a.ubar[k] = ubar;
        a.hbar[k] = hbar;
        a.rd[k] = make_float4(rhobar, Bbar * K.h / (3.f * K.rho), K.m, K.hinv);
    } else if (PASS == 1) {
        // self terms of rho_k and D_k: W(0,h) = (8/pi) h^-3, W_h(0,h) = -3 (8/pi) h^-4,
        // W_hh(0,h) = 12 (8/pi) h^-5
        const float mbar = S.m + K.rd.x * K.n4 * K.h - 3.f * K.rd.y * K.n4;
        const float hbar = a.hbar[k] + K.rd.y * (S.h + 12.f * K.m * K.n4 * K.hinv);
        const float dNdh = -(32.f / 3.f) * K.hinv * S.dN;
        const float4 x0 = a.xbar[k];
        a.xbar[k] = make_float4(x0.x + S.x, x0.y + S.y, x0.z + S.z, 0.f);
        a.mbar[k] += mbar;
        a.lam[k] = dNdh != 0.f ? hbar / dNdh : 0.f;
    } else {
        const float4 x0 = a.xbar[k];
        a.xbar[k] = make_float4(x0.x + S.x, x0.y + S.y, x0.z + S.z, 0.f);
    }
}

// Pairs from the recorded lists: four particles per warp, eight lanes each, as
// the list force. Each lane adds its pairs with Kahan compensation, the octet's
// sums are folded error-free. Bound by the gathers of its partners' records
// (64 bytes a pair in pass 0, 32 and 20 in the others), issued for the next
// pair while this one's terms are formed. At 262k clustered particles: walking
// one particle per thread 4.4 + 3.3 + 3.0 ms, from the lists 0.54 + 0.28 + 0.25 ms.
// Particles the lists cannot serve go to fb_list (pass 0) for k_backward.
template <int PASS>
__global__ void __launch_bounds__(kBwThreads, PASS == 0 ? 4 : 6) k_bw_list(BwArgs a) {
    if (!wpp_lists_valid(a.list_st)) return;
    const unsigned gen = a.list_st[kListGen];
    const unsigned lane = lane_id();
    const int slot = (int)(lane >> 3), sub = (int)(lane & 7u);
    const int warps = gridDim.x * (kBwThreads / 32);
    for (int t0 = (blockIdx.x * (kBwThreads / 32) + (int)(threadIdx.x >> 5)) * 4; t0 < a.n; t0 += warps * 4) {
        int k = t0 + slot;
        int cn = 0, ec = 0;
        bool live = k < a.n;
        if (live) {
            cn = a.nbr_n[k];
            const unsigned e = a.ext_n[k];
            ec = (int)e;
            if (cn < 0 || e > (unsigned)kExtCap || a.list_ep[k] != gen) {
                if (PASS == 0 && sub == 0) a.fb_list[atomicAdd(&a.list_st[3], 1u)] = k;
                live = false;
            }
        }
        if (!live) k = 0;
        const float sf = a.boxes[a.n_boxes == 1 ? 0 : wpp_box(a.boxes, a.n_boxes, k)].sf;
        const uint4 Xk = a.posm[k];
        const BwI K = bw_own<PASS>(a, k, Xk);
        const int tot = live ? cn + ec : 0;
        const int32_t* ln = a.nbr + (live ? a.nbr_off[k] : 0);
        const int32_t* le = a.ext + (size_t)k * kExtCap;
        auto partner = [&](int i) { return i < cn ? ln[i] : le[i - cn]; };
        uint4 Xn = make_uint4(0u, 0u, 0u, 0u);
        BwJ Jn = {};
        auto fetch = [&](int q) {
            Xn = __ldg(a.list_xh + q);
            if (PASS == 0) {
                Jn.v = __ldg(a.fvm + q);
                Jn.t = __ldg(a.fthermo + q);
                Jn.g = __ldg(a.ga + q);
            } else if (PASS == 1) {
                Jn.t = a.rd[q];
            } else {
                Jn.hinv = __ldg(&a.fthermo[q].w);
                Jn.lam = a.lam[q];
            }
        };
        BwSum S, C;
        if (sub < tot) fetch(partner(sub));
        int qn = sub + 8 < tot ? partner(sub + 8) : 0;
        for (int i = sub; i < tot; i += 8) {
            const uint4 X = Xn;
            BwJ J = Jn;
            if (i + 8 < tot) fetch(qn);
            if (i + 16 < tot) qn = partner(i + 16);
            J.h = __uint_as_float(X.w);
            if (PASS == 0) {
                J.hinv = J.t.w;
                J.m = J.v.w;
            } else if (PASS == 1) {
                J.rd = make_float2(J.t.x, J.t.y);
                J.m = J.t.z;
                J.hinv = J.t.w;
            }
            const float dx = (float)(int)(X.x - Xk.x) * sf, dy = (float)(int)(X.y - Xk.y) * sf,
                        dz = (float)(int)(X.z - Xk.z) * sf;
            const float r2 = dx * dx + dy * dy + dz * dz;
            if (r2 > 0.f) {
                BwSum P;
                bw_pair<PASS>(K, J, a.alpha, dx, dy, dz, r2, P);
                kahan_add(S.x, C.x, P.x);
                kahan_add(S.y, C.y, P.y);
                kahan_add(S.z, C.z, P.z);
                if (PASS <= 1) {
                    kahan_add(S.m, C.m, P.m);
                    kahan_add(S.h, C.h, P.h);
                }
                if (PASS == 0) {
                    kahan_add(S.A, C.A, P.A);
                    kahan_add(S.c, C.c, P.c);
                    kahan_add(S.r, C.r, P.r);
                }
                if (PASS == 1) kahan_add(S.dN, C.dN, P.dN);
            }
        }
        __syncwarp();
        const int o0 = (int)(lane & 24u);   // the octet's first lane; sum c of a fold is in lane o0 + 2c
        const float f = wpp_fold4_oct(S.x - C.x, S.y - C.y, S.z - C.z, S.m - C.m);
        S.x = __shfl_sync(0xffffffffu, f, o0);
        S.y = __shfl_sync(0xffffffffu, f, o0 + 2);
        S.z = __shfl_sync(0xffffffffu, f, o0 + 4);
        S.m = __shfl_sync(0xffffffffu, f, o0 + 6);
        if (PASS <= 1) {
            const float e = PASS == 0 ? wpp_fold4_oct(S.h - C.h, S.A - C.A, S.c - C.c, S.r - C.r)
                                      : wpp_fold4_oct(S.h - C.h, S.dN - C.dN, 0.f, 0.f);
            S.h = __shfl_sync(0xffffffffu, e, o0);
            const float e1 = __shfl_sync(0xffffffffu, e, o0 + 2);
            if (PASS == 0) {
                S.A = e1;
                S.c = __shfl_sync(0xffffffffu, e, o0 + 4);
                S.r = __shfl_sync(0xffffffffu, e, o0 + 6);
            } else {
                S.dN = e1;
            }
        }
        if (live && sub == 0) bw_finish<PASS>(a, k, K, S);
    }
}

// The walk, one particle per thread: every particle, or those of fb_list when
// the lists serve the others.
template <int PASS>
__global__ void __launch_bounds__(kBwThreads) k_backward(BwArgs a) {
    const bool lists = a.nbr != nullptr && wpp_lists_valid(a.list_st);
    const int nk = lists ? (int)a.list_st[3] : a.n;
    for (int t0 = blockIdx.x * blockDim.x + threadIdx.x; t0 < nk; t0 += gridDim.x * blockDim.x) {
        const int k = lists ? a.fb_list[t0] : t0;
        const BoxDesc& B = a.boxes[a.n_boxes == 1 ? 0 : wpp_box(a.boxes, a.n_boxes, k)];
        const double s = ldexp(B.L, -32);
        const float sf = (float)s;
        const uint4 Xk = a.posm[k];
        const BwI K = bw_own<PASS>(a, k, Xk);
        BwSum S, C;   // Kahan per leaf

        int stack[kBwStack];
        int sp = 0;
        stack[sp++] = B.nlev == 1 ? 0 : (B.nlev - 1) << 27;
        for (;;) {
            int lt = -1;
            while (sp > 0) {
                const int enc = stack[--sp];
                const int lev = enc >> 27, t = enc & ((1 << 27) - 1);
                if (lev == 0) { lt = t; break; }
                const int cl = lev - 1;
                const int c0 = t * kFan, c1 = min(c0 + kFan, B.lvl_n[cl]);
                const int base = B.lvl_off[cl];
                for (int c = c0; c < c1; ++c) {
                    const float4 e = a.node_e[base + c];
                    if (bw_node_near(a.node_c[base + c], e, Xk, sf, fmaxf(K.h, e.w))) stack[sp++] = (cl << 27) | c;
                }
            }
            if (lt < 0) break;
            const int nd = B.lvl_off[0] + lt;
            const uint4 C0 = a.node_c[nd];
            const float4 E = a.node_e[nd];
            const long long q0 = B.off + (long long)lt * kLeaf, q1 = min(q0 + kLeaf, B.off + B.n);
            const bool wide = 2.f * (E.x + E.y + E.z) + fmaxf(K.h, E.w) >= 0.45f * (float)B.L;
            const float ox = (float)(int)(C0.x - Xk.x) * sf, oy = (float)(int)(C0.y - Xk.y) * sf,
                        oz = (float)(int)(C0.z - Xk.z) * sf;
            BwSum P;
            for (long long q = q0; q < q1; ++q) {
                if (q == k) continue;
                float dx, dy, dz;   // d = x_j - x_k
                BwJ J;
                if (!wide) {
                    const float4 f = a.posf[q];
                    dx = ox + f.x; dy = oy + f.y; dz = oz + f.z; J.m = f.w;
                } else {
                    const uint4 Xj = a.posm[q];
                    dx = (float)(int)(Xj.x - Xk.x) * sf; dy = (float)(int)(Xj.y - Xk.y) * sf;
                    dz = (float)(int)(Xj.z - Xk.z) * sf; J.m = __uint_as_float(Xj.w);
                }
                const float r2 = dx * dx + dy * dy + dz * dz;
                J.v = a.fvel[q];
                J.h = J.v.w;
                const float hm = fmaxf(K.h, J.h);
                if (!(r2 < hm * hm) || r2 <= 0.f) continue;
                J.hinv = 1.f / J.h;
                if (PASS == 0) {
                    J.t = a.fthermo[q];
                    J.g = a.ga[q];
                } else if (PASS == 1) {
                    const float4 rd = a.rd[q];
                    J.rd = make_float2(rd.x, rd.y);
                } else {
                    J.lam = a.lam[q];
                }
                bw_pair<PASS>(K, J, a.alpha, dx, dy, dz, r2, P);
            }
            kahan_add(S.x, C.x, P.x);
            kahan_add(S.y, C.y, P.y);
            kahan_add(S.z, C.z, P.z);
            if (PASS <= 1) {
                kahan_add(S.m, C.m, P.m);
                kahan_add(S.h, C.h, P.h);
            }
            if (PASS == 0) {
                kahan_add(S.A, C.A, P.A);
                kahan_add(S.c, C.c, P.c);
                kahan_add(S.r, C.r, P.r);
            }
            if (PASS == 1) kahan_add(S.dN, C.dN, P.dN);
        }
        S.x -= C.x; S.y -= C.y; S.z -= C.z; S.m -= C.m; S.h -= C.h;
        S.A -= C.A; S.c -= C.c; S.r -= C.r; S.dN -= C.dN;
        bw_finish<PASS>(a, k, K, S);
    }
}

cudaError_t run_backward(sph_ctx* ctx, sph_grid* g, const BackwardLaunch& b, cudaStream_t s) {
    const int n = (int)g->n;
    if (!g->bw_ga) {
        const Part parts[] = {{&g->bw_ga, sizeof(float4) * n}, {&g->bw_xbar, sizeof(float4) * n},
                              {&g->bw_rd, sizeof(float4) * n}, {&g->bw_f, sizeof(float) * 6 * (size_t)n}};
        const cudaError_t e = carve(&g->bw_arena, parts);
        if (e) return e;
    }
    grid_refresh_hmax(g, b.h, s);
    force_pack(g, b.vel, b.u, b.h, b.rho, b.omega, (float)b.gamma, s);
    ++ctx->launches;
    float* us = g->bw_f;
    float* oms = g->bw_f + n;
    float* mbar = g->bw_f + 2 * (size_t)n;
    float* ubar = g->bw_f + 3 * (size_t)n;
    float* hbar = g->bw_f + 4 * (size_t)n;
    float* lam = g->bw_f + 5 * (size_t)n;
    const int pb = (n + 255) / 256;
    const bool lists = g->nbr != nullptr && g->lists_rec;
    if (lists) {
        const cudaError_t e = cudaMemsetAsync(g->list_st + 2, 0, 2 * sizeof(unsigned), s);
        if (e) return e;
    }
    k_bw_prep<<<pb, 256, 0, s>>>(n, g->perm, b.g_acc, b.g_rho, b.u, b.omega, g->bw_ga, us, oms, b.h, g->posm,
                                 lists ? g->list_xh : nullptr, lists ? g->list_st + 2 : nullptr);
    ++ctx->launches;
    BwArgs a;
    a.boxes = g->boxes;
    a.n_boxes = g->n_boxes;
    a.n = n;
    a.posm = g->posm;
    a.posf = g->posf;
    a.node_c = g->node_c;
    a.node_e = g->node_e;
    a.fvel = g->fvel;
    a.fthermo = g->fthermo;
    a.ga = g->bw_ga;
    a.u = us;
    a.omega = oms;
    a.xbar = g->bw_xbar;
    a.mbar = mbar;
    a.ubar = ubar;
    a.hbar = hbar;
    a.rd = g->bw_rd;
    a.lam = lam;
    a.alpha = (float)b.alpha;
    a.gamma = (float)b.gamma;
    a.fvm = g->fvm;
    a.nbr = lists ? g->nbr : nullptr;
    a.nbr_off = g->nbr_off;
    a.nbr_n = g->nbr_n;
    a.ext = g->ext;
    a.ext_n = g->ext_n;
    a.list_xh = g->list_xh;
    a.list_ep = g->list_ep;
    a.list_st = g->list_st;
    a.fb_list = g->fb_list;
    const long long want = (n + kBwThreads - 1) / kBwThreads;
    const int blocks = (int)std::max<long long>(1, std::min<long long>(want, (long long)ctx->sm_count * 16));
    const int lb = (int)std::max<long long>(1, std::min<long long>((n + 15) / 16, (long long)ctx->sm_count * 16));
    if (lists) k_bw_list<0><<<lb, kBwThreads, 0, s>>>(a);
    k_backward<0><<<blocks, kBwThreads, 0, s>>>(a);
    if (lists) k_bw_list<1><<<lb, kBwThreads, 0, s>>>(a);
    k_backward<1><<<blocks, kBwThreads, 0, s>>>(a);
    if (lists) k_bw_list<2><<<lb, kBwThreads, 0, s>>>(a);
    k_backward<2><<<blocks, kBwThreads, 0, s>>>(a);
    if (lists) ctx->launches += 3;
    k_bw_scatter<<<pb, 256, 0, s>>>(n, g->perm, g->bw_xbar, ubar, mbar, b.g_pos, b.g_u, b.g_mass);
    ctx->launches += 4;
    return cudaGetLastError();
}

}  // namespace sph
