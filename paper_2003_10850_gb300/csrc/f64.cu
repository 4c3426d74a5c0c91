// f64.cu -- SPH_FP64: the plain method in double (pair arithmetic and sums in
// FP64 on exact integer separations).
//
// One warp per active particle. The FP64 pipe is narrow on this part, so a warp
// spends an FP64 instruction only on true pairs, 32 at a time: the walk and the
// candidate test are FP32 with a margin that covers their rounding (whatever
// they let through is settled by the exact predicate), and what passes is
// compacted into a list in shared memory first.
//  - density: the pairs within 1.04 h are kept, with their distance, across the
//    h iterations; each iteration is a few multiplications per pair. A particle
//    whose list overflows works it off as it fills, once per iteration.
//  - force: each particle's A, c, 1/h and predicate bound are formed once per
//    call (k_f64_pack), not once per pair.
// Sums: at most eight terms of a lane plainly, everything above that (further terms,
// the lanes) with the rounding errors carried along, in the density pass once per
// particle. It is 5 % of the two passes' time; errors in units of 2^-53 of the sum of
// the magnitudes (55 to 100 pairs, simulated): 0.4, with a plain fold 0.8, with Kahan's
// sum over plain sums of leaves 0.6.
// One particle per thread, every candidate tested and every square root and
// division taken in FP64 in the pair loop, took 2.9 + 3.1 ms (density + force)
// for 32,768 lattice particles; this form takes 0.73 + 0.58 ms.
#include "wpp.cuh"

namespace sph {

constexpr int kF64Near = 128;                 // list entries per warp
constexpr float kF64Margin = 1.f + 1.9073486328125e-06f;   // 2^-19: FP32 squared distances are off by less than 2^-21

struct F64Smem {
    WppSmem w;
    double r[kF64Near];                       // distance (box units)
    unsigned long long d2[kF64Near];          // exact squared distance (integer units); prepare() makes it a double
    float m[kF64Near];
    int j[kF64Near];
};
static_assert(kWppWarps * sizeof(F64Smem) <= 48 * 1024, "static shared memory");

// a + b rounded, with the rounding error in e: the larger exponent first (compared as
// integers), then three FP64 additions.
__device__ __forceinline__ double f64_two_sum(double a, double b, double& e) {
    const bool sw = (__double2hiint(a) & 0x7fffffff) < (__double2hiint(b) & 0x7fffffff);
    const double l = sw ? b : a, r = sw ? a : b, t = __dadd_rn(l, r);
    e = __dsub_rn(r, __dsub_rn(t, l));
    return t;
}

// Sums of two per-lane values over the warp, in every lane.
__device__ __forceinline__ void f64_fold2(double& x, double& y) {
    const bool lo16 = lane_id() < 16u;
    double s = (lo16 ? x : y) + __shfl_xor_sync(0xffffffffu, lo16 ? y : x, 16);
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    x = __shfl_sync(0xffffffffu, s, 0);
    y = __shfl_sync(0xffffffffu, s, 16);
}

// Sums of four per-lane values over the warp, in every lane, the additions' errors
// carried along and added at the end: four times the additions of a plain fold, so the
// density kernel takes it once per particle, not once per evaluation.
__device__ __forceinline__ void f64_fold4(double& x, double& y, double& z, double& u) {
    const bool lo16 = lane_id() < 16u, lo8 = (lane_id() & 8u) == 0u;
    double ea, eb, e;
    const double a = f64_two_sum(lo16 ? x : z, __shfl_xor_sync(0xffffffffu, lo16 ? z : x, 16), ea);
    const double b = f64_two_sum(lo16 ? y : u, __shfl_xor_sync(0xffffffffu, lo16 ? u : y, 16), eb);
    double s = f64_two_sum(lo8 ? a : b, __shfl_xor_sync(0xffffffffu, lo8 ? b : a, 8), e);
    double c = __dadd_rn(__dadd_rn(lo8 ? ea : eb, __shfl_xor_sync(0xffffffffu, lo8 ? eb : ea, 8)), e);
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) {
        const double c2 = __shfl_xor_sync(0xffffffffu, c, o);
        s = f64_two_sum(s, __shfl_xor_sync(0xffffffffu, s, o), e);
        c = __dadd_rn(__dadd_rn(c, c2), e);
    }
    s = __dadd_rn(s, c);
    x = __shfl_sync(0xffffffffu, s, 0);
    y = __shfl_sync(0xffffffffu, s, 8);
    z = __shfl_sync(0xffffffffu, s, 16);
    u = __shfl_sync(0xffffffffu, s, 24);
}

// Four per-lane sums, taken up part by part: a part of a few terms is a plain sum (as
// a leaf's is on the other paths), the parts are added with Kahan's compensation.
struct F64Sum4 {
    double x = 0.0, y = 0.0, z = 0.0, u = 0.0, cx = 0.0, cy = 0.0, cz = 0.0, cu = 0.0;
    __device__ __forceinline__ void add(double& px, double& py, double& pz, double& pu) {
        kahan_add(x, cx, px);
        kahan_add(y, cy, py);
        kahan_add(z, cz, pz);
        kahan_add(u, cu, pu);
        px = py = pz = pu = 0.0;
    }
    __device__ __forceinline__ void fold(double& px, double& py, double& pz, double& pu) const {
        px = x; py = y; pz = z; pu = u;
        double dx = cx, dy = cy, dz = cz, du = cu;
        f64_fold4(px, py, pz, pu);
        f64_fold4(dx, dy, dz, du);
        px -= dx; py -= dy; pz -= dz; pu -= du;
    }
};

// The candidates of the walk's leaf list, 32 per step: cand(q, X, valid).
template <class Cand>
__device__ __forceinline__ void f64_leaves(F64Smem& sm, const uint4* __restrict__ posm, int off, int pend, int& nlf,
                                           Cand&& cand) {
    const unsigned lane = lane_id();
    for (int base = 0; base < nlf; base += 4) {
        const int li = base + (int)(lane >> 3);
        const int q = li < nlf ? off + (sm.w.lid[li] & 0x7fffffff) * kLeaf + (int)(lane & 7u) : pend;
        const bool ok = q < pend;
        cand(q, posm[ok ? q : off], ok);
    }
    nlf = 0;
    __syncwarp();
}

__device__ __forceinline__ float f64_d2f(uint4 X, uint4 Xi) {
    const float fx = (float)(int)(X.x - Xi.x), fy = (float)(int)(X.y - Xi.y), fz = (float)(int)(X.z - Xi.z);
    return fx * fx + fy * fy + fz * fz;
}

template <bool HASH>
__global__ void __launch_bounds__(kWppThreads) k_density_f64(WppArgs a) {
    __shared__ F64Smem smem[kWppWarps];
    F64Smem& sm = smem[threadIdx.x >> 5];
    const unsigned lane = lane_id();
    const unsigned lt = (1u << lane) - 1u;
    const int cnt = (int)*a.count_ptr, warps = gridDim.x * kWppWarps;
    unsigned long long c_pairs = 0, c_evals = 0, c_tests = 0;
    unsigned c_status = 0;
    for (int t = blockIdx.x * kWppWarps + (int)(threadIdx.x >> 5); t < cnt; t += warps) {
        const int p = a.act[t];
        const BoxDesc& B = a.boxes[a.n_boxes == 1 ? 0 : wpp_box(a.boxes, a.n_boxes, p)];
        const int off = (int)B.off, pend = (int)(B.off + B.n);
        const double s = ldexp(B.L, -32);
        const uint4 Xi = a.posm[p];
        const int oi = a.perm[p];
        float h = a.h[oi];
        if (a.guess_h || !(h > 0.f) || !isfinite(h)) h = wpp_guess_h(B, a.node_lo, a.node_hi, p, s, a.n_target);
        const double cap = 0.5 * B.L * (1.0 - 1e-9);
        double blo = 0.0, bhi = INFINITY;
        float dold = INFINITY, Rw = 0.f;
        unsigned st = 0;
        bool direct = false;   // the list overflowed: every evaluation sweeps again
        int nnear = 0;
        double Sw, Sdw, Smw, Smdw;   // per-lane sums: at most five terms of a list
        F64Sum4 Q;                   // of the lists already worked off (direct)
        int nn;
        unsigned long long hs;
        // distances of the list's entries
        auto prepare = [&]() {
            __syncwarp();
            for (int k = (int)lane; k < nnear; k += 32) {
                const double d = __ull2double_rn(sm.d2[k]);
                sm.d2[k] = (unsigned long long)__double_as_longlong(d);
                sm.r[k] = sqrt(d) * s;
            }
            __syncwarp();
        };
        // the list's pairs within h, added to the per-lane sums
        auto accumulate = [&](double hinv, double HH) {
            for (int k = (int)lane; k < nnear; k += 32) {
                if (!(__longlong_as_double((long long)sm.d2[k]) < HH)) continue;
                const double q = sm.r[k] * hinv, m = (double)sm.m[k];
                double w, dw;
                spline<double>(q, w, dw);
                const double qdw = q * dw;
                Sw += w;
                Sdw += qdw;
                Smw += m * w;
                Smdw += m * qdw;
                ++nn;
                if (HASH) hs += splitmix64((unsigned long long)a.perm[sm.j[k]]);
            }
        };
        // the other particles within R into the list; a full list is worked off
        // (direct) or reported
        auto sweep = [&](float R, double hinv, double HH) {
            const float T = R * B.Hs, T2 = T * T * kF64Margin;
            bool over = false;
            int nlf = 0;
            bool complete = true;
            nnear = 0;
            auto scan = [&]() {
                f64_leaves(sm, a.posm, off, pend, nlf, [&](int q, uint4 X, bool ok) {
                    if (nnear > kF64Near - 32) {
                        if (direct) {
                            prepare();
                            accumulate(hinv, HH);
                            Q.add(Sw, Sdw, Smw, Smdw);
                            __syncwarp();
                            nnear = 0;
                        } else {
                            over = true;
                        }
                    }
                    if (over) return;
                    c_tests += ok ? 1u : 0u;
                    const bool pass = ok && q != p && f64_d2f(X, Xi) < T2;
                    const unsigned b = __ballot_sync(0xffffffffu, pass);
                    if (pass) {
                        const int k = nnear + __popc(b & lt);
                        sm.d2[k] = exact_d2(X, Xi);
                        sm.m[k] = __uint_as_float(X.w);
                        if (HASH) sm.j[k] = q;
                    }
                    nnear += __popc(b);
                });
            };
            wpp_walk(sm.w, B, a.node_c, a.node_e, Xi, B.sf, nlf, complete, [&](float4) { return R; }, scan);
            scan();
            prepare();
            return !over;
        };
        for (int it = 0;; ++it) {
            const double hd = (double)h, hinv = 1.0 / hd;
            const double HH = wpp_hh(h, B);
            Sw = lane == 0 ? 1.0 : 0.0;   // the particle itself: w(0) = 1, q w'(0) = 0
            Smw = lane == 0 ? (double)__uint_as_float(Xi.w) : 0.0;
            Sdw = Smdw = 0.0;
            nn = 0;
            hs = 0;
            if (!direct && !(h <= Rw)) {
                Rw = a.fixed_h ? h : h * a.walk_r;
                direct = !sweep(Rw, hinv, HH);
            }
            if (direct) {
                Q = F64Sum4();
                sweep(h, hinv, HH);
            }
            accumulate(hinv, HH);
            __syncwarp();
            if (direct) Q.add(Sw, Sdw, Smw, Smdw);
            // what moves h takes a plain fold: its rounding, below 2^-49 of N, is 2^-27 of
            // what the smallest step of h (FP32) changes; the outputs' sums are folded below
            double fw = direct ? Q.x - Q.cx : Sw, fdw = direct ? Q.y - Q.cy : Sdw;
            f64_fold2(fw, fdw);
            ++c_evals;
            const double f = (32.0 / 3.0) * fw - a.n_target;
            if (a.fixed_h || fabs(f) <= a.n_tol) break;
            if (it >= a.max_iter) {
                st |= ST_NOT_CONVERGED;
                break;
            }
            const float N = (float)((32.0 / 3.0) * fw), dN = -(32.f / 3.f) * (float)fdw / h;
            if (!h_update(h, f, N, dN, (float)a.n_target, cap, blo, bhi, dold, st)) break;
        }
        if (direct) Q.fold(Sw, Sdw, Smw, Smdw);
        else f64_fold4(Sw, Sdw, Smw, Smdw);
        nn = warp_sum(nn);
        if (HASH) hs = warp_sum(hs);
        if (lane == 0) {
            const double hd = (double)h;
            a.h[oi] = h;
            a.rho[oi] = (float)(8.0 / (3.141592653589793 * hd * hd * hd) * Smw);
            a.omega[oi] = (float)(Smdw != 0.0 ? -3.0 * Smw / Smdw : 1.0);
            a.n_ngb[oi] = nn;
            a.flags[oi] = (uint8_t)st;
            if (HASH) a.hash[oi] = hs;
            c_pairs += (unsigned long long)nn;
            c_status |= st;
        }
        __syncwarp();
    }
    c_tests = warp_sum(c_tests);
    if (lane == 0) {
        atomicAdd(&a.ctr->density_pairs, c_pairs);
        atomicAdd(&a.ctr->density_evals, c_evals);
        atomicAdd(&a.ctr->pair_tests, c_tests);
        if (c_status) atomicOr(&a.ctr->status, c_status);
    }
}

// Per particle, in FP64: (A, c) and (1/h, (h 2^32/L)^2).
__global__ void k_f64_pack(int n, const int32_t* __restrict__ perm, const BoxDesc* __restrict__ boxes, int nb,
                           const float* __restrict__ u, const float* __restrict__ h, const float* __restrict__ rho,
                           const float* __restrict__ omega, double gam, double2* __restrict__ ac,
                           double2* __restrict__ hh) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= n) return;
    const int o = perm[p];
    const BoxDesc& B = boxes[nb == 1 ? 0 : wpp_box(boxes, nb, p)];
    const double r = (double)rho[o], P = (gam - 1.0) * r * (double)u[o];
    ac[p] = make_double2((double)omega[o] * P / (r * r), sqrt(gam * P / r));
    hh[p] = make_double2(1.0 / (double)h[o], wpp_hh(h[o], B));
}

template <bool HASH>
__global__ void __launch_bounds__(kWppThreads) k_force_f64(WppArgs a, const double2* __restrict__ ac,
                                                           const double2* __restrict__ hh, double alpha) {
    __shared__ F64Smem smem[kWppWarps];
    F64Smem& sm = smem[threadIdx.x >> 5];
    const unsigned lane = lane_id();
    const unsigned lt = (1u << lane) - 1u;
    const double kNorm = 8.0 / 3.141592653589793;
    const int cnt = (int)*a.count_ptr, warps = gridDim.x * kWppWarps;
    unsigned long long c_pairs = 0, c_tests = 0;
    for (int t = blockIdx.x * kWppWarps + (int)(threadIdx.x >> 5); t < cnt; t += warps) {
        const int p = a.act[t];
        const BoxDesc& B = a.boxes[a.n_boxes == 1 ? 0 : wpp_box(a.boxes, a.n_boxes, p)];
        const int off = (int)B.off, pend = (int)(B.off + B.n);
        const double s = ldexp(B.L, -32);
        const uint4 Xi = a.posm[p];
        const float4 vi = a.fvel[p];
        const double rhoi = (double)a.fthermo[p].x, Ai = ac[p].x, ci = ac[p].y, hinvi = hh[p].x, HHi = hh[p].y;
        const double normi = kNorm * hinvi * hinvi * hinvi * hinvi;
        const float Ti = vi.w * B.Hs, Ti2 = Ti * Ti * kF64Margin;
        double Sx = 0.0, Sy = 0.0, Sz = 0.0, Su = 0.0, vsmax = 0.0;   // sums: at most eight terms
        F64Sum4 Q;   // of the earlier ones
        int np = 0, nh = 0, nev = 0;
        unsigned long long hs = 0;
        // the pair terms of buffered partners, one per lane
        auto eval = [&](int k) {
            if ((int)lane >= k) return;
            const int q = sm.j[lane];
            const uint4 X = a.posm[q];
            const double2 hj = hh[q];
            const double D2 = __ull2double_rn(exact_d2(Xi, X));
            if (!(D2 < HHi || D2 < hj.y)) return;
            ++np;
            if (HASH) hs += splitmix64((unsigned long long)a.perm[q]);
            const double2 aj = ac[q];
            const double dx = (double)(int)(X.x - Xi.x) * s, dy = (double)(int)(X.y - Xi.y) * s,
                         dz = (double)(int)(X.z - Xi.z) * s;   // d = x_j - x_i
            const double r2 = dx * dx + dy * dy + dz * dz;
            if (r2 <= 0.0) {   // coincident: no direction, no force
                vsmax = fmax(vsmax, ci + aj.y);
                return;
            }
            const float4 vj = a.fvel[q];
            const double rhoj = (double)a.fthermo[q].x, mj = (double)__uint_as_float(X.w);
            const double rinv = rsqrt(r2), r = r2 * rinv;
            double w_, dwi, dwj;
            spline<double>(r * hinvi, w_, dwi);
            spline<double>(r * hj.x, w_, dwj);
            const double hj2 = hj.x * hj.x;
            const double Fi = normi * dwi * rinv, Fj = kNorm * hj2 * hj2 * dwj * rinv;
            // r_ij = x_i - x_j = -d ; v_ij = v_i - v_j
            const double vr = -(((double)vi.x - (double)vj.x) * dx + ((double)vi.y - (double)vj.y) * dy +
                                ((double)vi.z - (double)vj.z) * dz);
            const double wij = vr * rinv;
            const double vs = ci + aj.y - 3.0 * wij;
            vsmax = fmax(vsmax, vs);
            const double PI = wij < 0.0 ? -alpha * vs * wij / (rhoi + rhoj) : 0.0;
            const double Fbar = 0.5 * (Fi + Fj);
            const double coef = mj * (Ai * Fi + aj.x * Fj + PI * Fbar);
            Sx += coef * dx;   // -coef * r_ij
            Sy += coef * dy;
            Sz += coef * dz;
            Su += mj * vr * (Ai * Fi + 0.5 * PI * Fbar);
        };
        int nlf = 0;
        bool complete = true;
        auto scan = [&]() {
            f64_leaves(sm, a.posm, off, pend, nlf, [&](int q, uint4 X, bool ok) {
                c_tests += ok ? 1u : 0u;
                bool pass = ok && q != p;
                if (pass) {
                    const float Tj = a.fvel[q].w * B.Hs;
                    pass = f64_d2f(X, Xi) < fmaxf(Ti2, Tj * Tj * kF64Margin);
                }
                const unsigned b = __ballot_sync(0xffffffffu, pass);
                if (pass) sm.j[nh + __popc(b & lt)] = q;
                nh += __popc(b);
                __syncwarp();
                if (nh >= 32) {
                    eval(32);
                    if ((++nev & 7) == 0) Q.add(Sx, Sy, Sz, Su);
                    nh -= 32;
                    const int v = (int)lane < nh ? sm.j[lane + 32] : 0;
                    __syncwarp();
                    if ((int)lane < nh) sm.j[lane] = v;
                    __syncwarp();
                }
            });
        };
        wpp_walk(sm.w, B, a.node_c, a.node_e, Xi, B.sf, nlf, complete, [&](float4 e) { return fmaxf(vi.w, e.w); }, scan);
        scan();
        eval(nh);
        __syncwarp();
        if (nev >= 8) {
            Q.add(Sx, Sy, Sz, Su);
            Q.fold(Sx, Sy, Sz, Su);
        } else {
            f64_fold4(Sx, Sy, Sz, Su);
        }
        vsmax = warp_max(vsmax);
        np = warp_sum(np);
        if (HASH) hs = warp_sum(hs);
        if (lane == 0) {
            const int oi = a.perm[p];
            a.acc[3 * (size_t)oi] = (float)Sx;
            a.acc[3 * (size_t)oi + 1] = (float)Sy;
            a.acc[3 * (size_t)oi + 2] = (float)Sz;
            a.dudt[oi] = (float)Su;
            a.vsig[oi] = (float)vsmax;
            if (HASH) a.hash[oi] = hs;
            c_pairs += (unsigned long long)np;
        }
    }
    c_tests = warp_sum(c_tests);
    if (lane == 0) {
        atomicAdd(&a.ctr->force_pairs, c_pairs);
        atomicAdd(&a.ctr->pair_tests, c_tests);
    }
}

static int f64_blocks(sph_ctx* ctx, int bps, int64_t n_active) {
    const long long want = (n_active + kWppWarps - 1) / kWppWarps;
    return (int)std::max<long long>(1, std::min<long long>(want, (long long)ctx->sm_count * (bps > 0 ? bps : 16)));
}

cudaError_t launch_density_f64(sph_ctx* ctx, const DensityLaunch& a, int64_t n_active, cudaStream_t s) {
    WppArgs c = wpp_common(ctx, a.g, nullptr);
    c.h = a.h;
    c.rho = a.rho;
    c.omega = a.omega;
    c.n_ngb = a.n_ngb;
    c.flags = a.flags;
    c.hash = a.hash;
    c.n_target = a.n_target;
    c.n_tol = a.n_tol;
    c.max_iter = a.max_iter;
    c.guess_h = a.guess_h;
    c.fixed_h = a.fixed_h;
    c.walk_r = a.walk_radius > 0.0 ? (float)a.walk_radius : kWppWalkR;
    WppSpan sp;
    cudaError_t e = span_begin(ctx, a.time_kernels, 0, s, sp);
    if (e) return e;
    const int blocks = f64_blocks(ctx, a.blocks_per_sm, n_active);
    a.hash ? k_density_f64<true><<<blocks, kWppThreads, 0, s>>>(c) : k_density_f64<false><<<blocks, kWppThreads, 0, s>>>(c);
    ++ctx->launches;
    if ((e = span_end(ctx, sp, s))) return e;
    return cudaGetLastError();
}

cudaError_t launch_force_f64(sph_ctx* ctx, const ForceLaunch& a, int64_t n_active, cudaStream_t s) {
    const sph_grid* g = a.g;
    const int n = (int)g->n;
    force_pack(g, a.vel, a.u, a.h, a.rho, a.omega, (float)a.gamma, s);
    // the records of the FP32 paths that this call does not read hold the FP64 ones
    double2* ac = reinterpret_cast<double2*>(g->fposh);
    double2* hh = reinterpret_cast<double2*>(g->fvm);
    k_f64_pack<<<(n + 255) / 256, 256, 0, s>>>(n, g->perm, g->boxes, g->n_boxes, a.u, a.h, a.rho, a.omega, a.gamma, ac,
                                               hh);
    ctx->launches += 2;
    WppArgs c = wpp_common(ctx, g, nullptr);
    c.fvel = g->fvel;
    c.fthermo = g->fthermo;
    c.acc = a.acc;
    c.dudt = a.dudt;
    c.vsig = a.vsig;
    c.hash = a.hash;
    WppSpan sp;
    cudaError_t e = span_begin(ctx, a.time_kernels, 1, s, sp);
    if (e) return e;
    const int blocks = f64_blocks(ctx, a.blocks_per_sm, n_active);
    a.hash ? k_force_f64<true><<<blocks, kWppThreads, 0, s>>>(c, ac, hh, a.alpha)
           : k_force_f64<false><<<blocks, kWppThreads, 0, s>>>(c, ac, hh, a.alpha);
    ++ctx->launches;
    if ((e = span_end(ctx, sp, s))) return e;
    return cudaGetLastError();
}

}  // namespace sph
