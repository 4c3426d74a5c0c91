// gravity.cu -- short-range gravity of the TreePM split by a Barnes-Hut walk.
//
// The paper's code computes short-range gravity by Barnes-Hut: particles
// interact with distant tree nodes as point masses chosen by an opening
// criterion, and the interactions happen inside the walk (Sec. 1, Sec. 3).
// Long-range gravity (the particle mesh) is not part of this pass.
//
// The tree is the grid's hierarchy (a leaf is 8 consecutive Morton-sorted
// particles, a node 8 consecutive nodes of the level below). Its node boxes are
// exact integer boxes, and the rule of the walk is one of exact integer arithmetic
// on coarse coordinates (integer coordinates >> 8); FP32 tests with a margin decide
// where they are sure of its outcome, the rule itself elsewhere, with no FP64 on the
// per-node or per-pair path:
//   D2 = sum_a G_a^2, G_a the periodic gap between X_i and the box on axis a;
//   F2 = sum_a F_a^2, F_a the periodic distance to the far side, rounded up;
//   L2 = l^2, l the box's largest side;  RCi = ceil((r_cut 2^24 / L)^2);
//   P = rint(theta^2 2^16).
// The root is always opened; a child of an opened node is skipped if
// D2 >= RCi, taken as its monopole if P > 0, D2 > 0, F2 < RCi, L2 <= D2 and
// 2^16 L2 <= P D2, and opened otherwise (a leaf: its particles one by one,
// each if its coarse distance is below RCi). D2 < RCi <= 2^44 and P <= 2^16
// keep the products below 2^60.
//
// A warp walks for a group of up to M active particles (its members) of one
// aligned run of 64 sorted particles, 32/M lanes serving each member:
// - a step pops up to four opened nodes, one child per lane; with four or more
//   members the children beyond every member's cutoff go (by the members' box, in
//   FP32 with a margin) and the others wait until there are 32;
// - 32 children, one per lane, are tested against every member, in FP32 where that
//   settles the exact rule and by the rule itself elsewhere (see grav_decide); a
//   child that some member opens is
//   pushed with its member mask, and a member that accepts a node or opens a leaf
//   puts it on its own list;
// - a full list is worked off by the lanes of its member: accepted nodes, and the
//   particles of opened leaves, each inside the cutoff by an FP32 test of the
//   separation that the pair term needs anyway (the exact test in a thin band).
// The pair term is
//   a_i += G m_j K(r) (x_j - x_i),  K(r) = M(r/h_s) g(r) / r^3,
// M the spline softening's mass fraction, g(r) = erfc(r/2r_s) + r/(r_s sqrt(pi))
// exp(-r^2/4r_s^2) the short-range factor (erfc to 1.5e-7, see grav_K).
#include <cmath>

#include "wpp.cuh"

namespace sph {

constexpr int kGravStack = 256;   // see the bound below
constexpr int kGravLeaves = 128;  // opened leaves waiting per member; a step adds <= 32
constexpr int kGravNodes = 64;    // accepted nodes waiting per member; a step adds <= 32

// Stack bound: the 32 children tested after pop-4 steps from sp <= 96 push <= 32, and
// the <= 31 still waiting then go before the next pop: sp <= 155. In the pop-1
// regime the children of a node are tested at once (<= 8 pushed), so the stack grows
// by at most 7 per level of depth-first descent: sp <= 155 + 7 kMaxLev < kGravStack.

struct GravBox {
    unsigned long long RCi;
    float rcu;               // 256 sqrt(RCi): the cutoff in integer units
    float r2_in, r2_out;     // squared separation (box units): surely inside below, surely outside above
    float pad;
};
static_assert(sizeof(GravBox) == kGravBoxBytes, "the grid's per-box gravity store");

struct GravArgs {
    const BoxDesc* boxes;
    int n_boxes;
    const int32_t* act;
    const uint32_t* count_ptr;
    unsigned* queue;
    const uint4* posm;
    const int32_t* perm;
    const uint4* node_lo;
    const uint4* node_hi;
    const uint4* node_c;
    const float4* node_m;   // centre of mass - node centre (box units), mass
    const GravBox* gbox;    // per box: the cutoff
    float* acc;
    int32_t* n_nodes;
    int32_t* n_pairs;
    Counters* ctr;
    float G;
    unsigned long long P;    // rint(theta^2 2^16)
    float inv_theta;         // 256 / sqrt(P) (P = 0: unused)
    float hs, inv_hs;        // softening radius (0: none)
    float inv2rs;            // 1 / (2 r_s); r_s <= 0: 0
};

// Mass and centre of mass relative to the node centre of a node whose children
// c0..c1 are in (q: moments, cc: centres), in order.
template <class Q, class C>
__device__ __forceinline__ float4 grav_join(int c0, int c1, uint4 c, float sf, Q&& q_, C&& cc_) {
    float M = 0.f, sx = 0.f, sy = 0.f, sz = 0.f;
    for (int k = c0; k < c1; ++k) {
        const float4 q = q_(k);
        const uint4 cc = cc_(k);
        M += q.w;
        sx = fmaf(q.w, fmaf((float)(int)(cc.x - c.x), sf, q.x), sx);
        sy = fmaf(q.w, fmaf((float)(int)(cc.y - c.y), sf, q.y), sy);
        sz = fmaf(q.w, fmaf((float)(int)(cc.z - c.z), sf, q.z), sz);
    }
    const float s = M > 0.f ? 1.f / M : 0.f;
    return make_float4(sx * s, sy * s, sz * s, M);
}

// Moments of levels 0 to 3, a block per kTreeT leaves (as the bounds, see grid.cu).
__global__ void __launch_bounds__(kTreeT) k_grav_low(const uint4* __restrict__ posm, const BoxDesc* __restrict__ boxes,
                                                     const uint4* __restrict__ nc, float4* __restrict__ nm) {
    __shared__ float4 sq[kTreeT];
    __shared__ uint4 sc[kTreeT];
    const BoxDesc& B = boxes[blockIdx.y];
    const int tid = threadIdx.x, t = blockIdx.x * kTreeT + tid;
    if (blockIdx.x * kTreeT >= B.lvl_n[0]) return;
    const float sf = B.sf;
    float4 q = make_float4(0.f, 0.f, 0.f, 0.f);
    uint4 c = make_uint4(0u, 0u, 0u, 0u);
    if (t < B.lvl_n[0]) {
        const long long p0 = B.off + (long long)t * kLeaf, p1 = min(p0 + kLeaf, B.off + B.n);
        const int nd = B.lvl_off[0] + t;
        c = nc[nd];
        float M = 0.f, sx = 0.f, sy = 0.f, sz = 0.f;
        for (long long p = p0; p < p1; ++p) {
            const uint4 x = posm[p];
            const float m = __uint_as_float(x.w);
            M += m;
            sx = fmaf(m, (float)(int)(x.x - c.x), sx);
            sy = fmaf(m, (float)(int)(x.y - c.y), sy);
            sz = fmaf(m, (float)(int)(x.z - c.z), sz);
        }
        const float s = M > 0.f ? sf / M : 0.f;
        q = make_float4(sx * s, sy * s, sz * s, M);
        nm[nd] = q;
    }
    sq[tid] = q;
    sc[tid] = c;
    int w = kTreeT;
#pragma unroll
    for (int lev = 1; lev < kTreeLow; ++lev) {
        w /= kFan;
        __syncthreads();
        const int tt = blockIdx.x * w + tid;
        const bool live = tid < w && lev < B.nlev && tt < B.lvl_n[lev];
        if (live) {
            const int c0 = tid * kFan, c1 = c0 + min(kFan, B.lvl_n[lev - 1] - tt * kFan);
            c = nc[B.lvl_off[lev] + tt];
            q = grav_join(c0, c1, c, sf, [&](int k) { return sq[k]; }, [&](int k) { return sc[k]; });
            nm[B.lvl_off[lev] + tt] = q;
        }
        __syncthreads();
        if (live) {
            sq[tid] = q;
            sc[tid] = c;
        }
    }
}

// The levels above, a block per box.
__global__ void __launch_bounds__(kTreeTopT) k_grav_top(const BoxDesc* __restrict__ boxes,
                                                        const uint4* __restrict__ nc, float4* nm) {
    const BoxDesc& B = boxes[blockIdx.x];
    for (int lev = kTreeLow; lev < B.nlev; ++lev) {
        const int below = B.lvl_off[lev - 1];
        for (int t = threadIdx.x; t < B.lvl_n[lev]; t += kTreeTopT) {
            const int nd = B.lvl_off[lev] + t;
            nm[nd] = grav_join(t * kFan, min(t * kFan + kFan, B.lvl_n[lev - 1]), nc[nd], B.sf,
                               [&](int k) { return nm[below + k]; }, [&](int k) { return nc[below + k]; });
        }
        __syncthreads();
    }
}

// The cutoff of each box: RCi = ceil((r_cut 2^24 / L)^2) (FP64, then exact), its
// radius in integer units, and the FP32 bounds of the particle test on the
// squared separation in box units. A coarse distance is between the true one
// less 256 sqrt(3) units and the true one, so below 256 sqrt(RCi) a particle is
// inside and 444 units beyond it is outside; 2^-19 covers the FP32 rounding of
// the squared separation. Box sizes whose squares leave the FP32 range take the
// exact test always.
__global__ void k_grav_box_rc(const BoxDesc* __restrict__ boxes, int nb, double r_cut, GravBox* __restrict__ gb) {
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= nb) return;
    const double rcu = r_cut / boxes[b].L * 16777216.0;
    GravBox g;
    g.RCi = (unsigned long long)ceil(rcu * rcu);
    const double rc = 256.0 * sqrt((double)g.RCi), s = boxes[b].L * 2.3283064365386962890625e-10;
    const double lo = rc * s * rc * s * (1.0 - 1.9073486328125e-06), hi = (rc + 448.0) * s * (rc + 448.0) * s *
                                                                         (1.0 + 1.9073486328125e-06);
    const bool ok = lo > 1e-30 && hi < 1e30;
    g.rcu = (float)rc;
    g.r2_in = ok ? (float)lo : -1.f;
    g.r2_out = ok ? (float)hi : INFINITY;
    g.pad = 0.f;
    gb[b] = g;
}

// 2^x, a subnormal result as zero (an exponential that small adds nothing).
__device__ __forceinline__ float grav_ex2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// Mass fraction of the cubic spline (support 1) inside q < 1.
__device__ __forceinline__ float grav_soft(float q) {
    const float q2 = q * q, q3 = q2 * q;
    return q <= 0.5f ? q3 * fmaf(q2, fmaf(32.f, q, -192.f / 5.f), 32.f / 3.f)
                     : fmaf(q3, fmaf(q, fmaf(q, fmaf(-32.f / 3.f, q, 192.f / 5.f), -48.f), 64.f / 3.f), -1.f / 15.f);
}

// M(q) g(r) / r^3 of two pairs, r^2 = r2 > 0.
// The split factor g = erfc(x) + (2/sqrt(pi)) x e^{-x^2}, x = r / (2 r_s), takes
// erfc from Abramowitz & Stegun 7.1.26 (Hastings' rational approximation,
// |error| <= 1.5e-7): erfc(x) = t (a1 + t (a2 + t (a3 + t (a4 + t a5)))) e^{-x^2},
// t = 1 / (1 + p x), so that both terms share one exponential.
// 1/r^3 goes in as 1/r^2, then 1/r: r^3 is subnormal for pairs closer than 2.3e-13
// (box units; any box smaller than 1e-3 has some), where the softened term is not.
__device__ __forceinline__ float2 grav_K(const GravArgs& a, float2 r2) {
    const float2 rinv = make_float2(rsqrt_ftz(r2.x), rsqrt_ftz(r2.y)), r = mul2(r2, rinv);
    float2 K = both(1.f);
    if (r.x < a.hs) K.x = grav_soft(r.x * a.inv_hs);
    if (r.y < a.hs) K.y = grav_soft(r.y * a.inv_hs);
    if (a.inv2rs > 0.f) {
        const float2 x = mul2(r, both(a.inv2rs));
        const float2 y = fma2(both(0.3275911f), x, both(1.f));
        const float2 t = make_float2(rcp_ftz(y.x), rcp_ftz(y.y));
        float2 e = fma2(t, both(1.061405429f), both(-1.453152027f));
        e = fma2(t, e, both(1.421413741f));
        e = fma2(t, e, both(-0.284496736f));
        e = fma2(t, e, both(0.254829592f));
        e = fma2(both(1.1283791671f), x, mul2(t, e));   // 2 / sqrt(pi)
        const float2 z = mul2(mul2(x, x), both(-1.4426950409f));   // log2 e
        K = mul2(K, mul2(make_float2(grav_ex2(z.x), grav_ex2(z.y)), e));
    }
    return mul2(mul2(K, rcp2_ftz(r2)), rinv);
}

// One axis of the exact coarse box geometry: squared gap, squared far-side
// distance (rounded up) and coarse side.
__device__ __forceinline__ void grav_axis(unsigned x, unsigned lo, unsigned hi, unsigned long long& D2,
                                          unsigned long long& F2, unsigned& l) {
    unsigned gap = 0u, far;
    if (x < lo || x > hi) {
        const unsigned g1 = lo - x, g2 = x - hi;   // both ways round the periodic axis
        gap = min(g1, g2);
        far = gap + (hi - lo);
    } else {
        far = max(x - lo, hi - x);
    }
    const unsigned g = gap >> 8, f = (unsigned)(((unsigned long long)far + 255ull) >> 8);
    D2 += (unsigned long long)g * g;
    F2 += (unsigned long long)f * f;
    l = max(l, (hi - lo) >> 8);
}

// Exact coarse geometry of a node box seen from X: D2 (gap), F2 (far side,
// rounded up), L2 (largest side squared), per the rules above.
__device__ __forceinline__ void grav_box(uint4 X, uint4 lo, uint4 hi, unsigned long long& D2,
                                         unsigned long long& F2, unsigned long long& L2) {
    D2 = F2 = 0ull;
    unsigned l = 0u;
    grav_axis(X.x, lo.x, hi.x, D2, F2, l);
    grav_axis(X.y, lo.y, hi.y, D2, F2, l);
    grav_axis(X.z, lo.z, hi.z, D2, F2, l);
    L2 = (unsigned long long)l * l;
}

// The monopole rule of the walk (see the top of the file).
__device__ __forceinline__ bool grav_accept(unsigned long long P, unsigned long long D2, unsigned long long F2,
                                            unsigned long long L2, unsigned long long RCi) {
    return P > 0ull && D2 > 0ull && F2 < RCi && L2 <= D2 && (L2 << 16) <= P * D2;
}

// A node as the FP32 decision sees it, in integer units: centre and half
// extents, and the squared bounds that settle the rule for any member.
// With d the periodic offset of a member from the centre, the gap on an axis is
// max(|d| - e, 0) and the far side |d| + e. Against the rule's coarse D and F
// the FP32 norms are off by at most 2^-22 of themselves (the conversions), 2^-20
// of the extents (through the differences), and 256 sqrt(3) + 4 units (the
// coarse shift and the centre's half unit); the side is off by 256 units. `tol`
// holds the extents' part and the units, the factor m the relative part.
struct GravNode {
    uint4 lo, hi;
    unsigned cx, cy, cz;
    float ex, ey, ez;
    float out2, in2;    // D or F surely beyond the cutoff above out2, surely inside below in2
    float acc2, opn2;   // D surely >= l / theta above acc2, surely < l / theta below opn2
};

__device__ __forceinline__ void grav_node(GravNode& N, float rcu, float inv_theta) {
    const unsigned sx = N.hi.x - N.lo.x, sy = N.hi.y - N.lo.y, sz = N.hi.z - N.lo.z;
    N.cx = N.lo.x + (sx >> 1);
    N.cy = N.lo.y + (sy >> 1);
    N.cz = N.lo.z + (sz >> 1);
    N.ex = 0.5f * (float)sx;
    N.ey = 0.5f * (float)sy;
    N.ez = 0.5f * (float)sz;
    const float m = 1.9073486328125e-06f;   // 2^-19
    const float e = fmaxf(N.ex, fmaxf(N.ey, N.ez)), tol = fmaf(m, e, 512.f);
    const float T = 2.f * e * inv_theta, Tl = (2.f * e - 256.f) * inv_theta;
    const float o = rcu + tol, i = fmaxf(rcu - tol, 0.f), ah = T + tol, al = fmaxf(Tl - tol, 0.f);
    N.out2 = o * o * (1.f + m);
    N.in2 = i * i * (1.f - m);
    N.acc2 = ah * ah * (1.f + m);
    N.opn2 = al * al * (1.f - m);
}

constexpr int kGravSkip = 0, kGravTake = 1, kGravOpen = 2;

// The rule for one member: FP32 where it is sure, the exact rule otherwise.
__device__ __forceinline__ int grav_decide(const GravNode& N, uint4 X, unsigned long long RCi, unsigned long long P) {
    const float dx = fabsf((float)(int)(N.cx - X.x)), dy = fabsf((float)(int)(N.cy - X.y)),
                dz = fabsf((float)(int)(N.cz - X.z));
    const float gx = fmaxf(dx - N.ex, 0.f), gy = fmaxf(dy - N.ey, 0.f), gz = fmaxf(dz - N.ez, 0.f);
    const float fx = dx + N.ex, fy = dy + N.ey, fz = dz + N.ez;
    const float D2f = fmaf(gx, gx, fmaf(gy, gy, gz * gz)), F2f = fmaf(fx, fx, fmaf(fy, fy, fz * fz));
    if (D2f > N.out2) return kGravSkip;
    if (D2f < N.in2) {
        if (P == 0ull || F2f > N.out2 || D2f < N.opn2) return kGravOpen;
        if (F2f < N.in2 && D2f > N.acc2) return kGravTake;
    }
    unsigned long long D2, F2, L2;
    grav_box(X, N.lo, N.hi, D2, F2, L2);
    return D2 >= RCi ? kGravSkip : grav_accept(P, D2, F2, L2, RCi) ? kGravTake : kGravOpen;
}

// Error-free (TwoSum) fold of a per-lane sum over aligned runs of W lanes; every
// lane of a run ends with the total, rounded once.
template <int W>
__device__ __forceinline__ float grav_fold(float s) {
    float c = 0.f;
#pragma unroll
    for (int o = 1; o < W; o <<= 1) {
        const float s2 = __shfl_xor_sync(0xffffffffu, s, o), c2 = __shfl_xor_sync(0xffffffffu, c, o);
        const float t = __fadd_rn(s, s2);
        const float bp = __fsub_rn(t, s);
        const float e = __fadd_rn(__fsub_rn(s, __fsub_rn(t, bp)), __fsub_rn(s2, bp));
        s = t;
        c = __fsub_rn(__fadd_rn(c, c2), e);
    }
    return __fsub_rn(s, c);
}

template <int M>
struct GravSmem {
    int stk[kGravStack];
    unsigned char stm[kGravStack];   // member mask of each stacked node
    uint4 mX[M];                     // member integer positions
    int lf[M][kGravLeaves];          // opened leaves (first particle)
    int nd[M][kGravNodes];           // accepted nodes (global index)
    int qe[M >= 4 ? 64 : 1];         // children waiting for the members' tests (level, index)
    unsigned char qm[M >= 4 ? 64 : 1];
};

template <int M>
__global__ void __launch_bounds__(kWppThreads, 5) k_gravity(GravArgs a) {
    __shared__ GravSmem<M> smem[kWppWarps];
    GravSmem<M>& sm = smem[threadIdx.x >> 5];
    constexpr int W = 32 / M;   // lanes per member
    const unsigned lane = lane_id();
    const unsigned lt = (1u << lane) - 1u;
    const int cnt = (int)*a.count_ptr;
    const int mm = (int)lane / W, sub = (int)lane % W;   // list work: lane (member, part)
    unsigned long long c_nodes = 0, c_pairs = 0;
    for (;;) {
        int t0 = 0;
        if (lane == 0) t0 = (int)atomicAdd(a.queue, (unsigned)M);
        t0 = __shfl_sync(0xffffffffu, t0, 0);
        if (t0 >= cnt) break;
        const int t1 = min(t0 + M, cnt);
        for (int t = t0; t < t1;) {
            const WppGroup G = wpp_group(a.boxes, a.n_boxes, a.act, t, t1, 6);
            t += G.n;
            const BoxDesc& B = a.boxes[G.box];
            const float sf = B.sf;
            const GravBox gb = a.gbox[G.box];
            const int off = (int)B.off, pend = (int)(B.off + B.n);
            uint4 Xl = make_uint4(0u, 0u, 0u, 0u);
            if (G.p >= 0) Xl = a.posm[G.p];
            if ((int)lane < M) sm.mX[lane] = Xl;
            const uint4 Xm = make_uint4(__shfl_sync(0xffffffffu, Xl.x, mm), __shfl_sync(0xffffffffu, Xl.y, mm),
                                        __shfl_sync(0xffffffffu, Xl.z, mm), 0u);
            const int pmm = __shfl_sync(0xffffffffu, G.p, mm);
            float2 ax = both(0.f), ay = ax, az = ax;   // this list's sums
            float Sx = 0.f, Sy = 0.f, Sz = 0.f, Cx = 0.f, Cy = 0.f, Cz = 0.f;   // the lists' (Kahan)
            int nn = 0, np = 0;
            int nl[M], na[M];   // list lengths (warp-uniform)
#pragma unroll
            for (int m = 0; m < M; ++m) nl[m] = na[m] = 0;
            int sp = 0;
            const int top = B.nlev - 1;
            if (lane == 0) {
                sm.stk[0] = (int)((unsigned)top << 28);
                sm.stm[0] = (unsigned char)((1u << G.n) - 1u);
            }
            if (top == 0) {   // a single leaf: opened whatever the rule says
                if ((int)lane < M) sm.lf[lane][0] = off;
#pragma unroll
                for (int m = 0; m < M; ++m) nl[m] = m < G.n ? 1 : 0;
            } else {
                sp = 1;
            }
            __syncwarp();
            // two interactions; ok false: none
            auto add = [&](float2 ex, float2 ey, float2 ez, float2 r2, float2 m, bool ok0, bool ok1) {
                ok0 = ok0 && r2.x > 0.f;   // coincident: no force
                ok1 = ok1 && r2.y > 0.f;
                if (!ok0 && !ok1) return;
                m = mul2(both(a.G), make_float2(ok0 ? m.x : 0.f, ok1 ? m.y : 0.f));
                const float2 f = mul2(m, grav_K(a, make_float2(ok0 ? r2.x : 1.f, ok1 ? r2.y : 1.f)));
                ax = fma2(f, ex, ax);
                ay = fma2(f, ey, ay);
                az = fma2(f, ez, az);
            };
            // a particle that passed neither FP32 bound: the exact test
            auto inside = [&](uint4 X) {
                const unsigned gx = (unsigned)abs((int)(X.x - Xm.x)) >> 8, gy = (unsigned)abs((int)(X.y - Xm.y)) >> 8,
                               gz = (unsigned)abs((int)(X.z - Xm.z)) >> 8;
                return (unsigned long long)gx * gx + (unsigned long long)gy * gy + (unsigned long long)gz * gz < gb.RCi;
            };
            auto total = [&]() {
                kahan_add(Sx, Cx, ax.x + ax.y);
                kahan_add(Sy, Cy, ay.x + ay.y);
                kahan_add(Sz, Cz, az.x + az.y);
                ax = ay = az = both(0.f);
            };
            // the members' box: centre, half extents (integer units, rounded up)
            uint4 Gc = make_uint4(0u, 0u, 0u, 0u);
            float gex = 0.f, gey = 0.f, gez = 0.f;
            bool gok = false;
            if (M >= 4) {
                const unsigned X0x = __shfl_sync(0xffffffffu, Xl.x, 0), X0y = __shfl_sync(0xffffffffu, Xl.y, 0),
                               X0z = __shfl_sync(0xffffffffu, Xl.z, 0);
                const bool mv = G.p >= 0;
                const int dx = mv ? (int)(Xl.x - X0x) : 0, dy = mv ? (int)(Xl.y - X0y) : 0, dz = mv ? (int)(Xl.z - X0z) : 0;
                const int lx = warp_min(dx), ly = warp_min(dy), lz = warp_min(dz);
                const long long sx = (long long)warp_max(dx) - lx, sy = (long long)warp_max(dy) - ly,
                                sz = (long long)warp_max(dz) - lz;
                gok = sx < (1ll << 30) && sy < (1ll << 30) && sz < (1ll << 30);
                Gc = make_uint4(X0x + (unsigned)(lx + (int)(sx >> 1)), X0y + (unsigned)(ly + (int)(sy >> 1)),
                                X0z + (unsigned)(lz + (int)(sz >> 1)), 0u);
                const float up = 1.f + 3.814697265625e-06f;   // 2^-18: also the rounding of offsets this size
                gex = fmaf((float)sx, 0.5f * up, 4.f);
                gey = fmaf((float)sy, 0.5f * up, 4.f);
                gez = fmaf((float)sz, 0.5f * up, 4.f);
            }
            int nq = 0;   // children waiting
            bool done = sp == 0;
            for (;;) {
                int ml = 0, mn = 0;
#pragma unroll
                for (int m = 0; m < M; ++m) {
                    ml = max(ml, nl[m]);
                    mn = max(mn, na[m]);
                }
                if (done ? ml > 0 : ml > kGravLeaves - 32) {
                    // the particles of the opened leaves, two per lane and step, the
                    // next step's positions loaded ahead
                    int k = 0;
#pragma unroll
                    for (int m = 0; m < M; ++m) {
                        k = mm == m ? nl[m] : k;
                        nl[m] = 0;
                    }
                    const int* lf = sm.lf[mm];
                    k *= kLeaf;
                    // (the last leaf may reach past the box: those reads stay in the padded store)
                    auto fetch = [&](int j, uint4& X) {
                        const int q = j < k ? lf[j >> 3] + (j & 7) : pend;
                        X = a.posm[j < k ? q : off];
                        return q < pend;
                    };
                    uint4 n0, n1;
                    bool v0 = fetch(sub, n0), v1 = fetch(sub + W, n1);
                    for (int j = sub; j < k; j += 2 * W) {
                        const uint4 X0 = n0, X1 = n1;
                        bool i0 = v0, i1 = v1;
                        v0 = fetch(j + 2 * W, n0);
                        v1 = fetch(j + 3 * W, n1);
                        const float2 s2 = both(sf);
                        const float2 ex = mul2(make_float2((float)(int)(X0.x - Xm.x), (float)(int)(X1.x - Xm.x)), s2),
                                     ey = mul2(make_float2((float)(int)(X0.y - Xm.y), (float)(int)(X1.y - Xm.y)), s2),
                                     ez = mul2(make_float2((float)(int)(X0.z - Xm.z), (float)(int)(X1.z - Xm.z)), s2);
                        const float2 r2 = fma2(ez, ez, fma2(ey, ey, mul2(ex, ex)));
                        i0 = i0 && !(r2.x > gb.r2_out);
                        i1 = i1 && !(r2.y > gb.r2_out);
                        if (i0 && !(r2.x < gb.r2_in)) i0 = inside(X0);
                        if (i1 && !(r2.y < gb.r2_in)) i1 = inside(X1);
                        np += (i0 ? 1 : 0) + (i1 ? 1 : 0);
                        add(ex, ey, ez, r2, make_float2(__uint_as_float(X0.w), __uint_as_float(X1.w)), i0, i1);
                    }
                    total();
                    __syncwarp();
                }
                if (done ? mn > 0 : mn > kGravNodes - 32) {
                    int k = 0;
#pragma unroll
                    for (int m = 0; m < M; ++m) {
                        k = mm == m ? na[m] : k;
                        na[m] = 0;
                    }
                    nn += k;
                    const int* nd = sm.nd[mm];
                    for (int j = sub; j < k; j += 2 * W) {
                        const bool two = j + W < k;
                        const int i0 = nd[j], i1 = nd[two ? j + W : j];
                        const uint4 C0 = a.node_c[i0], C1 = a.node_c[i1];
                        const float4 q0 = a.node_m[i0], q1 = a.node_m[i1];
                        const float2 s2 = both(sf);
                        const float2 ex = fma2(make_float2((float)(int)(C0.x - Xm.x), (float)(int)(C1.x - Xm.x)), s2,
                                               make_float2(q0.x, q1.x)),
                                     ey = fma2(make_float2((float)(int)(C0.y - Xm.y), (float)(int)(C1.y - Xm.y)), s2,
                                               make_float2(q0.y, q1.y)),
                                     ez = fma2(make_float2((float)(int)(C0.z - Xm.z), (float)(int)(C1.z - Xm.z)), s2,
                                               make_float2(q0.z, q1.z));
                        add(ex, ey, ez, fma2(ez, ez, fma2(ey, ey, mul2(ex, ex))), make_float2(q0.w, q1.w), true, two);
                    }
                    total();
                    __syncwarp();
                }
                if (done) break;
                int lev, child, id;
                unsigned mask;
                GravNode N;
                // the children of up to four opened nodes, one per lane
                auto pop = [&]() {
                    const int npop = sp <= 96 ? min(4, sp) : 1;
                    const int slot = (int)(lane >> 3);
                    lev = child = -1;
                    mask = 0u;
                    if (slot < npop) {
                        const unsigned en = (unsigned)sm.stk[sp - 1 - slot];
                        const int k = (int)(en >> 28), c = (int)(en & 0x0fffffffu) * kFan + (int)(lane & 7u);
                        if (c < B.lvl_n[k - 1]) {
                            lev = k - 1;
                            child = c;
                            mask = sm.stm[sp - 1 - slot];
                        }
                    }
                    __syncwarp();
                    sp -= npop;
                };
                auto load = [&]() {
                    id = B.lvl_off[max(lev, 0)] + max(child, 0);
                    N.lo = a.node_lo[id];
                    N.hi = a.node_hi[id];
                    grav_node(N, gb.rcu, a.inv_theta);
                };
                if (M >= 4) {
                    while (sp > 0 && nq < 32 && (sp <= 96 || nq == 0)) {
                        pop();
                        load();
                        // a member is no farther from the centre than the half extents
                        const float gx = fmaxf(fabsf((float)(int)(N.cx - Gc.x)) - N.ex - gex, 0.f),
                                    gy = fmaxf(fabsf((float)(int)(N.cy - Gc.y)) - N.ey - gey, 0.f),
                                    gz = fmaxf(fabsf((float)(int)(N.cz - Gc.z)) - N.ez - gez, 0.f);
                        const bool keep = child >= 0 && !(gok && fmaf(gx, gx, fmaf(gy, gy, gz * gz)) > N.out2);
                        const unsigned bk = __ballot_sync(0xffffffffu, keep);
                        if (keep) {
                            const int o = nq + __popc(bk & lt);
                            sm.qe[o] = (int)(((unsigned)lev << 28) | (unsigned)child);
                            sm.qm[o] = (unsigned char)mask;
                        }
                        nq += __popc(bk);
                        __syncwarp();
                    }
                    const int k = min(nq, 32);
                    nq -= k;
                    lev = child = -1;
                    mask = 0u;
                    if ((int)lane < k) {
                        const unsigned en = (unsigned)sm.qe[nq + (int)lane];
                        lev = (int)(en >> 28);
                        child = (int)(en & 0x0fffffffu);
                        mask = sm.qm[nq + (int)lane];
                    }
                    __syncwarp();
                } else {
                    pop();
                }
                load();
                unsigned om = 0u;   // members that open the child
#pragma unroll
                for (int m = 0; m < M; ++m) {
                    int v = kGravSkip;
                    if ((mask >> m) & 1u) v = grav_decide(N, sm.mX[m], gb.RCi, a.P);
                    if (v == kGravOpen) om |= 1u << m;
                    const unsigned bl = __ballot_sync(0xffffffffu, v == kGravOpen && lev == 0),
                                   bn = __ballot_sync(0xffffffffu, v == kGravTake);
                    if (v == kGravOpen && lev == 0) sm.lf[m][nl[m] + __popc(bl & lt)] = off + child * kLeaf;
                    if (v == kGravTake) sm.nd[m][na[m] + __popc(bn & lt)] = id;
                    nl[m] += __popc(bl);
                    na[m] += __popc(bn);
                }
                const bool push = om != 0u && lev > 0;
                const unsigned bp = __ballot_sync(0xffffffffu, push);
                if (push) {
                    const int o = sp + __popc(bp & lt);
                    sm.stk[o] = (int)(((unsigned)lev << 28) | (unsigned)child);
                    sm.stm[o] = (unsigned char)om;
                }
                sp += __popc(bp);
                done = sp == 0 && nq == 0;
                __syncwarp();
            }
            // per member: fold its lanes' sums, write its outputs
            Sx = grav_fold<W>(Sx - Cx);
            Sy = grav_fold<W>(Sy - Cy);
            Sz = grav_fold<W>(Sz - Cz);
#pragma unroll
            for (int o = 1; o < W; o <<= 1) np += __shfl_xor_sync(0xffffffffu, np, o);
            if (mm < G.n && sub == 0) {
                np -= gb.RCi > 0ull ? 1 : 0;   // itself: in its own leaf, always opened, at distance 0
                const int oi = a.perm[pmm];
                a.acc[3 * (size_t)oi] = Sx;
                a.acc[3 * (size_t)oi + 1] = Sy;
                a.acc[3 * (size_t)oi + 2] = Sz;
                if (a.n_nodes) a.n_nodes[oi] = nn;
                if (a.n_pairs) a.n_pairs[oi] = np;
                c_nodes += (unsigned long long)nn;
                c_pairs += (unsigned long long)np;
            }
            __syncwarp();
        }
    }
    c_nodes = warp_sum(c_nodes);
    c_pairs = warp_sum(c_pairs);
    if (lane == 0 && (c_nodes | c_pairs)) {
        atomicAdd(&a.ctr->grav_nodes, c_nodes);
        atomicAdd(&a.ctr->grav_pairs, c_pairs);
    }
}

template <int M>
static void grav_run(sph_ctx* ctx, const GravArgs& a, int64_t n_active, cudaStream_t s) {
    const long long want = (n_active + M * kWppWarps - 1) / (M * kWppWarps);
    const int blocks = (int)std::max<long long>(1, std::min<long long>((long long)ctx->sm_count * 8, want));
    k_gravity<M><<<blocks, kWppThreads, 0, s>>>(a);
}

cudaError_t launch_gravity(sph_ctx* ctx, const GravityLaunch& L, int64_t n_active, cudaStream_t s) {
    sph_grid* g = const_cast<sph_grid*>(L.g);
    const int nb = g->n_boxes;
    k_grav_low<<<dim3((g->max_leaves + kTreeT - 1) / kTreeT, nb), kTreeT, 0, s>>>(g->posm, g->boxes, g->node_c,
                                                                              g->node_m);
    ++ctx->launches;
    if (g->max_lev > kTreeLow) {
        k_grav_top<<<nb, kTreeTopT, 0, s>>>(g->boxes, g->node_c, g->node_m);
        ++ctx->launches;
    }
    GravBox* gbox = reinterpret_cast<GravBox*>(g->grav_box);
    k_grav_box_rc<<<(nb + 127) / 128, 128, 0, s>>>(g->boxes, nb, L.r_cut, gbox);
    ++ctx->launches;
    GravArgs a = {};
    a.boxes = g->boxes;
    a.n_boxes = nb;
    a.act = g->act;
    a.count_ptr = g->act_n;
    a.queue = ctx->queue + 4;
    a.posm = g->posm;
    a.perm = g->perm;
    a.node_lo = g->node_lo;
    a.node_hi = g->node_hi;
    a.node_c = g->node_c;
    a.node_m = g->node_m;
    a.gbox = gbox;
    a.acc = L.acc;
    a.n_nodes = L.n_nodes;
    a.n_pairs = L.n_pairs;
    a.ctr = ctx->counters;
    a.G = (float)L.G;
    a.P = (unsigned long long)std::rint(L.theta * L.theta * 65536.0);
    a.inv_theta = a.P ? (float)(256.0 / std::sqrt((double)a.P)) : 0.f;
    a.hs = (float)L.h_soft;
    a.inv_hs = L.h_soft > 0.0 ? (float)(1.0 / L.h_soft) : 0.f;
    a.inv2rs = L.r_split > 0.0 ? (float)(0.5 / L.r_split) : 0.f;
    // Members per walk: more of them share the node loads and tests, but a group
    // of 8 takes 8 times as long, so a set must be large enough to fill the GPU
    // with groups several times over, and dense enough that groups are full.
    // Measured (clustered, theta 0.5), us for 1/2/4/8 members: 9,000 of 30,000 active
    // 139/170/209/430; all of 30,000 280/253/267/320; of 60,000 559/493/478/531;
    // of 500,000 5255/4514/4108/4078; of 1M 12700/11200/10440/10100; 100,000 of 1M
    // 1588/1484/1524/1956; 25,000 of 500,000 396/407/467/904.
    const long long sm = ctx->sm_count, na = n_active, n = g->n;
    if (na >= 3000 * sm && na * 2 >= n) grav_run<8>(ctx, a, na, s);
    else if (na >= 320 * sm && na * 4 >= n) grav_run<4>(ctx, a, na, s);
    else if (na >= 176 * sm && na * 16 >= n) grav_run<2>(ctx, a, na, s);
    else grav_run<1>(ctx, a, na, s);
    ++ctx->launches;
    return cudaGetLastError();
}

}  // namespace sph
