// steady.cu -- cell labelling as its own entry point, and the batched steady
// morphogen solve: the D2Q5 relaxation of Sec. 6.1 with u = 0 on a static
// tissue, iterated until the residual r = max|phi^{n+1} - phi^n| /
// max|phi^{n+1}| (checked every `check_every` steps) reaches `tol`.
//
// B tissues of the same lattice size run side by side and each stops on its
// own, on exactly the step count at which it converged.  A tissue that fits
// in the registers of one thread-block cluster (16 CTAs of 4,096 nodes) is
// relaxed there from the first step to the last in one launch
// (steady_cluster: one 256^2 tissue 8.8 -> 2.1 ms, 96 of them 128.9 -> 26.3
// ms).  Larger ones take one launch per step (grid.z = tissue): the residual
// kernel writes phi of the state it checked to the output, and the decision
// kernel freezes a converged tissue (its update kernels return at once from
// then on).
#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstring>
#include <string>
#include <vector>

#include "lbib_internal.cuh"

namespace lbib {

// ---------------------------------------------------------------- labels
__global__ void labels_to_ids(uint32_t* packed, uint8_t* src, int64_t n) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const uint32_t v = packed[i];
    if (src) src[i] = (v == kOutside) ? 0 : (uint8_t)(v & 0xFu);
    packed[i] = (v == kOutside) ? 0u : (v >> 4) + 1u;
}

// ---------------------------------------------------------------- steady D2Q5
struct SteadyArgs {
    const float* gsrc;
    float* gdst;
    const uint8_t* src;   // batch * N source flags (bit 0)
    const float* omegaD;  // per tissue 1/tau_D
    const float* decay;   // per tissue
    const float* srate;   // per tissue
    const int* active;    // per tissue
    float* phi_prev;      // batch * N: phi^{n} stored by flagged updates
    int nx, ny;
    int64_t pitch, plane, tstride;  // tstride: elements per tissue (5 planes)
    int store_prev;
};

// one D2Q5 update of every active tissue: pull, phi, reaction, BGK with u = 0
__global__ void __launch_bounds__(256) steady_update(SteadyArgs a) {
    const int b = blockIdx.z;
    if (!a.active[b]) return;
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y;
    if (x >= a.nx) return;
    const int xm = (x == 0) ? a.nx - 1 : x - 1;
    const int xp = (x == a.nx - 1) ? 0 : x + 1;
    const int ym = (y == 0) ? a.ny - 1 : y - 1;
    const int yp = (y == a.ny - 1) ? 0 : y + 1;
    const int64_t P = a.plane;
    const float* G = a.gsrc + (int64_t)b * a.tstride;
    const int64_t r0 = (int64_t)y * a.pitch, node = r0 + x;
    float g[5];
    g[0] = __ldg(G + node);
    g[1] = __ldg(G + 1 * P + r0 + xm);
    g[2] = __ldg(G + 2 * P + (int64_t)ym * a.pitch + x);
    g[3] = __ldg(G + 3 * P + r0 + xp);
    g[4] = __ldg(G + 4 * P + (int64_t)yp * a.pitch + x);
    const uint8_t s = a.src[(int64_t)b * a.nx * a.ny + (int64_t)y * a.nx + x];
    const float phi = ((g[0] + g[1]) + (g[2] + g[3])) + g[4];
    const float R = ((s & 1u) ? a.srate[b] : 0.f) - a.decay[b] * phi;
    const float om = a.omegaD[b];
    float* O = a.gdst + (int64_t)b * a.tstride;
    // weights that sum to one exactly in FP32 (1 - 4 w1 is exact): the
    // update creates no mass from their rounding
    constexpr float w1 = (float)(1.0 / 6.0);
    constexpr float w0 = 1.0f - 4.0f * w1;
#pragma unroll
    for (int q = 0; q < 5; ++q) {
        const float w = q == 0 ? w0 : w1;
        O[q * P + node] = g[q] + om * (phi * w - g[q]) + w * R;
    }
    if (a.store_prev) a.phi_prev[(int64_t)b * a.nx * a.ny + (int64_t)y * a.nx + x] = phi;
}

// phi of the current state, residual against the stored previous phi
__global__ void __launch_bounds__(256) steady_residual(const float* G0, int64_t pitch,
                                                       int64_t plane, int64_t tstride, int nx,
                                                       int ny, const int* active,
                                                       const float* phi_prev, float* phi_out,
                                                       unsigned* dmax, unsigned* pmax) {
    const int b = blockIdx.z;
    if (!active[b]) return;
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y;
    float d = 0.f, pm = 0.f;
    if (x < nx) {
        const int xm = (x == 0) ? nx - 1 : x - 1;
        const int xp = (x == nx - 1) ? 0 : x + 1;
        const int ym = (y == 0) ? ny - 1 : y - 1;
        const int yp = (y == ny - 1) ? 0 : y + 1;
        const float* G = G0 + (int64_t)b * tstride;
        const int64_t r0 = (int64_t)y * pitch;
        const float phi = ((G[r0 + x] + G[plane + r0 + xm]) +
                           (G[2 * plane + (int64_t)ym * pitch + x] + G[3 * plane + r0 + xp])) +
                          G[4 * plane + (int64_t)yp * pitch + x];
        const int64_t o = (int64_t)b * nx * ny + (int64_t)y * nx + x;
        d = fabsf(phi - phi_prev[o]);
        pm = fabsf(phi);
        // a non-finite value counts as +inf (fmaxf would drop a NaN), so the
        // tissue's residual becomes inf / inf = NaN and never passes the test
        if (!isfinite(d)) d = INFINITY;
        if (!isfinite(pm)) pm = INFINITY;
        phi_out[o] = phi;
    }
#pragma unroll
    for (int k = 16; k > 0; k >>= 1) {
        d = fmaxf(d, __shfl_xor_sync(0xffffffffu, d, k));
        pm = fmaxf(pm, __shfl_xor_sync(0xffffffffu, pm, k));
    }
    // non-negative floats order like their bit patterns
    if ((threadIdx.x & 31) == 0) {
        atomicMax(dmax + b, __float_as_uint(d));
        atomicMax(pmax + b, __float_as_uint(pm));
    }
}

// Warm-start fallback: a tissue started from a prediction goes back to the
// cold start (g = 0) when its residual is not finite, or when after this many
// checks it is not below the residual of its first check (the prediction has
// not brought the relaxation closer); its step count runs on.
constexpr int kFallbackChecks = 64;

struct SteadyState {
    int* active;
    int* warm;        // still watched: on the warm start, fewer than kFallbackChecks checks
    int* grow;        // checks so far (warm only)
    int* fellback;    // the warm start was abandoned
    int* reset;       // restart from g = 0 after this check
    float* prevr;     // residual of the first check
};

// per tissue: r = dmax / pmax; freeze converged tissues, reset the maxima,
// abandon failing warm starts
__global__ void steady_decide(int batch, int64_t n, double tol, SteadyState S, unsigned* dmax,
                              unsigned* pmax, long long* steps, double* resid, int* n_active) {
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= batch) return;
    S.reset[b] = 0;
    if (!S.active[b]) return;
    const float d = __uint_as_float(dmax[b]), p = __uint_as_float(pmax[b]);
    const double r = p > 0.f ? (double)d / (double)p : (d > 0.f ? INFINITY : 0.0);
    resid[b] = r;
    steps[b] = n;
    dmax[b] = 0u;
    pmax[b] = 0u;
    if (S.warm[b]) {
        const bool finite = isfinite(r);
        const int c = ++S.grow[b];
        if (c == 1) S.prevr[b] = (float)r;
        if (!finite || (c >= kFallbackChecks && !(r < (double)S.prevr[b]))) {
            S.warm[b] = 0;
            S.fellback[b] = 1;
            S.reset[b] = 1;
            resid[b] = INFINITY;
            return;
        }
        if (c >= kFallbackChecks) S.warm[b] = 0;  // the prediction has helped: stop watching
    }
    if (r <= tol) {
        S.active[b] = 0;
        atomicSub(n_active, 1);
    }
}

// ---------------------------------------------------------------- on-chip solve
// The whole relaxation of a tissue on one thread-block cluster.  A launch per
// step moves 40 bytes per node and step through the caches and waits for a
// launch each time; here a tissue's populations stay in registers for all its
// steps: what bounds a step is the shared memory's bandwidth (about 5 of the
// 128-byte accesses per 32 nodes) and the latency of one round of publish,
// barrier and dependent operations (0.45 us).  A cluster of C CTAs divides the rows into strips of V rows; a thread
// owns one column of one strip as V/2 pairs of rows, each pair one packed FP32
// value per population, and a step is
//   publish   g1 and g3 of every node (they move in x) to the CTA's shared
//             memory, g2 of a strip's top row and g4 of its bottom row (they
//             leave the strip in y) to the strip above / below, in the next
//             CTA's shared memory where that strip lives there;
//   sync      one CTA barrier; the values for another CTA travel as
//             asynchronous remote stores that complete on that CTA's mbarrier,
//             and only the threads that need them wait, after their strip's
//             inner rows;
//   collide   the operations of steady_update on both rows of a pair at once
//             (the packed instructions round each half as the scalar ones
//             do), so a solve takes the same steps to the same bits.
// The shared arrays alternate between two copies, so one CTA barrier per step
// is enough.  The residual check reduces over the cluster through distributed
// shared memory and every CTA takes the same decision, so converged tissues
// leave, and failing warm starts restart, without the host.
constexpr int kSteadyClusterMax = 16;  // CTAs of a cluster (above 8: non-portable)

// shared memory per thread: g1, g3 in two copies, the sources and phi of the
// step before a check for V nodes; the strip's incoming g2 and g4 in two copies
constexpr int steady_cluster_smem(int V, int threads) { return threads * 4 * (6 * V + 4); }

struct SteadyClusterArgs {
    float* g;                 // the populations between launches
    const float* phi0;        // first launch: the warm start (NULL: zero)
    const uint8_t* src;
    const float* omegaD;
    const float* decay;
    const float* srate;
    float* phi_out;
    SteadyState S;
    long long* steps;
    double* resid;
    int* n_active;
    int* lost;                // a wait ran out
    double tol;
    int64_t pitch, plane, tstride;
    long long n0;             // steps taken before this launch
    int n_steps;              // steps of this launch
    int phase;                // n0 % check_every
    int nx, ny, check_every, strips, strips_per_cta, first;
};

__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
}
__device__ __forceinline__ uint32_t smem_addr(const void* p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}
// the address of this CTA's shared variable in the cluster's CTA `rank`
__device__ __forceinline__ uint32_t cluster_addr(const void* p, uint32_t rank) {
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(smem_addr(p)), "r"(rank));
    return r;
}
__device__ __forceinline__ void st_cluster(uint32_t addr, float v) {
    asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(addr), "f"(v) : "memory");
}
// the same, asynchronous, counted by the mbarrier at `bar` of the target CTA
__device__ __forceinline__ void st_cluster_async(uint32_t addr, float v, uint32_t bar) {
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];" ::"r"(
                     addr),
                 "r"(__float_as_uint(v)), "r"(bar)
                 : "memory");
}
// wait for a phase of an mbarrier of this CTA, for about a second at most
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity) {
    unsigned long long t0 = 0;
    for (int spin = 0;; ++spin) {
        uint32_t ok;
        asm volatile(
            "{\n.reg .pred p;\n"
            "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n"
            "selp.u32 %0, 1, 0, p;\n}"
            : "=r"(ok)
            : "r"(bar), "r"(parity)
            : "memory");
        if (ok) return true;
        if ((spin & 63) == 63) {
            unsigned long long t;
            asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
            if (!t0) t0 = t;
            if (t - t0 > 1000000000ull) return false;
        }
    }
}

// phi of the pulled populations of two rows, in the order of steady_update
__device__ __forceinline__ float2 steady_phi(float2 p0, float2 p1, float2 p2, float2 p3,
                                             float2 p4) {
    return __fadd2_rn(__fadd2_rn(__fadd2_rn(p0, p1), __fadd2_rn(p2, p3)), p4);
}
__device__ __forceinline__ float2 pair2(float v) { return make_float2(v, v); }

// NT: threads per CTA at most (the stride of the shared arrays); FULL: every
// strip holds V rows (ny a multiple of V)
template <int V, int NT, bool FULL>
__global__ void __launch_bounds__(NT, 1) steady_cluster(SteadyClusterArgs a) {
    constexpr int P = V / 2;  // pairs of rows
    static_assert(V % 2 == 0 && P >= 2, "at least two pairs");
    extern __shared__ __align__(16) unsigned char steady_smem[];
    __shared__ float wd[32], wp[32];
    __shared__ float red[2][kSteadyClusterMax];
    // the watch of a warm start: still watched, checks so far, first residual
    __shared__ int warm, grow, verdict;
    __shared__ float prevr;
    __shared__ __align__(8) unsigned long long mbar[2];  // one per copy
    uint32_t C, rank;
    asm("mov.u32 %0, %%cluster_nctaid.x;" : "=r"(C));
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
    const int b = blockIdx.x / C;
    if (!a.S.active[b]) return;  // the whole cluster
    const int tid = threadIdx.x;
    float2* const sh1 = reinterpret_cast<float2*>(steady_smem);  // [2][P][NT]
    float2* const sh3 = sh1 + 2 * P * NT;                        // [2][P][NT]
    float2* const prev = sh3 + 2 * P * NT;                       // [P][NT]
    float2* const rate = prev + P * NT;                          // [P][NT]
    float* const up = reinterpret_cast<float*>(rate + P * NT);   // [2][NT] g2 from below
    float* const dn = up + 2 * NT;                               // [2][NT] g4 from above

    // this thread's column x of strip s (CTA-local ls); threads without a
    // strip only take part in the barriers
    const int ls = tid / a.nx, x = tid - ls * a.nx;
    const int s = (int)rank * a.strips_per_cta + ls;
    const bool on = ls < a.strips_per_cta && s < a.strips;
    const int y0 = s * V;
    const int nv = !on ? 0 : (FULL ? V : min(V, a.ny - y0));
    const int tm = on ? ls * a.nx + (x == 0 ? a.nx - 1 : x - 1) : 0;
    const int tp = on ? ls * a.nx + (x == a.nx - 1 ? 0 : x + 1) : 0;
    // where the strip's outgoing g2 and g4 go (the strips above and below,
    // periodic), first copy; the second copy lies NT floats further on
    uint32_t far_up = 0, far_dn = 0, bar_up = 0, bar_dn = 0;  // in another CTA (0: not)
    int near_up = tid, near_dn = tid;
    if (on) {
        const int su = s + 1 == a.strips ? 0 : s + 1, sd = s == 0 ? a.strips - 1 : s - 1;
        const uint32_t ru = su / a.strips_per_cta, rd = sd / a.strips_per_cta;
        near_up = (su % a.strips_per_cta) * a.nx + x;
        near_dn = (sd % a.strips_per_cta) * a.nx + x;
        if (ru != rank) far_up = cluster_addr(up + near_up, ru);
        if (rd != rank) far_dn = cluster_addr(dn + near_dn, rd);
        bar_up = cluster_addr(mbar, ru);
        bar_dn = cluster_addr(mbar, rd);
    }
    const uint32_t bar0 = smem_addr(mbar);
    if (tid == 0) {
        for (int i = 0; i < 2; ++i)
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar0 + 8 * i) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        warm = a.S.warm[b];
        grow = a.S.grow[b];
        prevr = a.S.prevr[b];
    }
    const bool first_thread = rank == 0 && tid == 0;
    bool done = false, lost = false;
    uint32_t phases = 0u;  // the parity each mbarrier completes next (bits 0, 1)

    constexpr float w1 = (float)(1.0 / 6.0);
    constexpr float w0 = 1.0f - 4.0f * w1;
    // t = g - phi w rounds to minus (phi w - g), so g - om t is g + om (phi w - g)
    const float2 nom = pair2(-a.omegaD[b]), ndec = pair2(-a.decay[b]);

    float2 g0[P], g1[P], g2[P], g3[P], g4[P];
    float* const G = a.g + (int64_t)b * a.tstride;
    const int64_t N = (int64_t)a.nx * a.ny;
    {
        const float srate = a.srate[b];
        float* const rf = reinterpret_cast<float*>(rate);
#pragma unroll
        for (int j = 0; j < V; ++j) {
            float v[5] = {0.f, 0.f, 0.f, 0.f, 0.f}, r = 0.f;
            if (j < nv) {
                const int64_t o = (int64_t)b * N + (int64_t)(y0 + j) * a.nx + x;
                if (a.src[o] & 1u) r = srate;
                if (a.first) {
                    const float p = a.phi0 ? a.phi0[o] : 0.f;
#pragma unroll
                    for (int q = 0; q < 5; ++q) v[q] = (q == 0 ? w0 : w1) * p;
                } else {
                    const float* q0 = G + (int64_t)(y0 + j) * a.pitch + x;
#pragma unroll
                    for (int q = 0; q < 5; ++q) v[q] = q0[q * a.plane];
                }
            }
            rf[2 * ((j / 2) * NT + tid) + j % 2] = r;
            if (j % 2 == 0) {
                g0[j / 2].x = v[0], g1[j / 2].x = v[1], g2[j / 2].x = v[2], g3[j / 2].x = v[3];
                g4[j / 2].x = v[4];
            } else {
                g0[j / 2].y = v[0], g1[j / 2].y = v[1], g2[j / 2].y = v[2], g3[j / 2].y = v[3];
                g4[j / 2].y = v[4];
            }
        }
    }
    // every CTA of the cluster runs, its mbarriers ready, before a remote store
    cluster_sync();

    int n = 0, phase = a.phase, par = 0;
    bool checked = true;  // the check at n0 (if any) ended the launch before
    for (;;) {
        float2* const c1 = sh1 + par * P * NT;
        float2* const c3 = sh3 + par * P * NT;
        if (on) {
            float top = g2[P - 1].y;
#pragma unroll
            for (int i = 0; i < P; ++i) {
                c1[i * NT + tid] = g1[i];
                c3[i * NT + tid] = g3[i];
                if (!FULL) {
                    if (2 * i == nv - 1) top = g2[i].x;
                    if (2 * i + 1 == nv - 1) top = g2[i].y;
                }
            }
            if (far_up)
                st_cluster_async(far_up + 4 * par * NT, top, bar_up + 8 * par);
            else
                up[par * NT + near_up] = top;
            if (far_dn)
                st_cluster_async(far_dn + 4 * par * NT, g4[0].x, bar_dn + 8 * par);
            else
                dn[par * NT + near_dn] = g4[0].x;
        }
        if (tid == 0 && C > 1)  // one row of g2 and one of g4 from other CTAs
            asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar0 + 8 * par),
                         "r"(8 * a.nx)
                         : "memory");
        __syncthreads();
        // the threads whose strip borders on another CTA
        auto neighbours = [&] {
            if ((far_up | far_dn) && !lost) {
                lost = !mbar_wait(bar0 + 8 * par, (phases >> par) & 1u);
                if (lost) atomicExch(a.lost, 1);
            }
            phases ^= 1u << par;
        };
        const float* const cu = up + par * NT;
        const float* const cd = dn + par * NT;
        // the populations arriving in pair i from below and above, `below` and
        // `above` the rows next to the pair
        auto from_above = [&](int i, float above, float in4) {
            float2 v = make_float2(g4[i].y, above);
            if (!FULL) {
                if (2 * i == nv - 1) v.x = in4;
                if (2 * i + 1 == nv - 1) v.y = in4;
            }
            return v;
        };

        const bool check = !checked && phase == 0;
        if (check || n == a.n_steps) {
            // phi of the current state: the residual, or the last output
            neighbours();
            float dmax = 0.f, pmax = 0.f;
            if (on) {
                const float in2 = cu[tid], in4 = cd[tid];
#pragma unroll
                for (int i = 0; i < P; ++i) {
                    const float2 p2 = make_float2(i > 0 ? g2[i > 0 ? i - 1 : 0].y : in2, g2[i].x);
                    const float2 p4 =
                        from_above(i, i + 1 < P ? g4[i + 1 < P ? i + 1 : i].x : in4, in4);
                    const float2 phi =
                        steady_phi(g0[i], c1[i * NT + tm], p2, c3[i * NT + tp], p4);
                    const float2 was = prev[i * NT + tid];
                    // a non-finite value counts as +inf (see steady_residual)
                    auto count = [&](float ph, float old) {
                        float d = fabsf(ph - old), m = fabsf(ph);
                        if (!isfinite(d)) d = INFINITY;
                        if (!isfinite(m)) m = INFINITY;
                        dmax = fmaxf(dmax, d);
                        pmax = fmaxf(pmax, m);
                    };
                    if (FULL || 2 * i < nv) count(phi.x, was.x);
                    if (FULL || 2 * i + 1 < nv) count(phi.y, was.y);
                    prev[i * NT + tid] = phi;
                }
            }
            bool restart = false;
            if (check) {
                // non-negative floats order like their bit patterns
                dmax = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(dmax)));
                pmax = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(pmax)));
                if ((tid & 31) == 0) {
                    wd[tid >> 5] = dmax;
                    wp[tid >> 5] = pmax;
                }
                __syncthreads();
                if (tid < 32) {
                    const int nw = blockDim.x / 32;
                    dmax = __uint_as_float(__reduce_max_sync(
                        0xffffffffu, tid < nw ? __float_as_uint(wd[tid]) : 0u));
                    pmax = __uint_as_float(__reduce_max_sync(
                        0xffffffffu, tid < nw ? __float_as_uint(wp[tid]) : 0u));
                    if (tid < (int)C) {
                        st_cluster(cluster_addr(&red[0][rank], tid), dmax);
                        st_cluster(cluster_addr(&red[1][rank], tid), pmax);
                    }
                }
                cluster_sync();
                // one thread per CTA takes the decision (FP64 is slow), the
                // same in each
                if (tid == 0) {
                    float d = 0.f, p = 0.f;
                    for (uint32_t r = 0; r < C; ++r) {
                        d = fmaxf(d, red[0][r]);
                        p = fmaxf(p, red[1][r]);
                    }
                    const double r = p > 0.f ? (double)d / (double)p : (d > 0.f ? INFINITY : 0.0);
                    bool again = false;
                    if (warm) {
                        if (++grow == 1) prevr = (float)r;
                        again = !isfinite(r) || (grow >= kFallbackChecks && !(r < (double)prevr));
                        // abandoned, or the prediction has helped: stop watching
                        if (again || grow >= kFallbackChecks) warm = 0;
                    }
                    verdict = again ? 2 : (r <= a.tol ? 1 : 0);
                    if (rank == 0) {
                        a.resid[b] = again ? INFINITY : r;
                        a.steps[b] = a.n0 + n;
                        if (again) a.S.fellback[b] = 1;
                    }
                }
                __syncthreads();
                restart = verdict == 2;
                done = verdict == 1;
            }
            if (restart) {  // the cold start: from the zero state
#pragma unroll
                for (int i = 0; i < P; ++i) g0[i] = g1[i] = g2[i] = g3[i] = g4[i] = pair2(0.f);
            }
            if (done || n == a.n_steps) break;
            if (restart) {
                checked = true;
                par ^= 1;
                continue;
            }
        }
        const bool keep = phase + 1 == a.check_every;  // phi for the check that follows
        auto collide = [&](int i, float2 p2, float2 p4) {
            const float2 p0 = g0[i], p1 = c1[i * NT + tm], p3 = c3[i * NT + tp];
            const float2 phi = steady_phi(p0, p1, p2, p3, p4);
            if (keep) prev[i * NT + tid] = phi;
            const float2 R = __ffma2_rn(ndec, phi, rate[i * NT + tid]);
            auto bgk = [&](float2 g, float w) {
                return __ffma2_rn(pair2(w), R,
                                  __ffma2_rn(nom, __ffma2_rn(phi, pair2(-w), g), g));
            };
            g0[i] = bgk(p0, w0);
            g1[i] = bgk(p1, w1);
            g2[i] = bgk(p2, w1);
            g3[i] = bgk(p3, w1);
            g4[i] = bgk(p4, w1);
        };
        if (FULL) {
            // inner pairs first (they need nothing from other strips), then
            // the last and the first
            const float above0 = g4[1].x, below_last = g2[P - 2].y;
            if (on) {
                float below = g2[0].y;
#pragma unroll
                for (int i = 1; i < P - 1; ++i) {
                    const float next = g2[i].y;
                    collide(i, make_float2(below, g2[i].x), make_float2(g4[i].y, g4[i + 1].x));
                    below = next;
                }
            }
            if (!check) neighbours();
            if (on) {
                collide(P - 1, make_float2(below_last, g2[P - 1].x),
                        make_float2(g4[P - 1].y, cd[tid]));
                collide(0, make_float2(cu[tid], g2[0].x), make_float2(g4[0].y, above0));
            }
        } else {
            if (!check) neighbours();
            if (on) {
                const float in4 = cd[tid];
                float below = cu[tid];
#pragma unroll
                for (int i = 0; i < P; ++i) {
                    const float next = g2[i].y;
                    collide(i, make_float2(below, g2[i].x),
                            from_above(i, i + 1 < P ? g4[i + 1 < P ? i + 1 : i].x : in4, in4));
                    below = next;
                }
            }
        }
        ++n;
        phase = keep ? 0 : phase + 1;
        checked = false;
        par ^= 1;
    }
    if (on) {
        const float* const pf = reinterpret_cast<const float*>(prev);
#pragma unroll
        for (int j = 0; j < V; ++j) {
            if (j < nv) {
                a.phi_out[(int64_t)b * N + (int64_t)(y0 + j) * a.nx + x] =
                    pf[2 * ((j / 2) * NT + tid) + j % 2];
                if (!done) {
                    float* q0 = G + (int64_t)(y0 + j) * a.pitch + x;
                    q0[0] = j % 2 ? g0[j / 2].y : g0[j / 2].x;
                    q0[a.plane] = j % 2 ? g1[j / 2].y : g1[j / 2].x;
                    q0[2 * a.plane] = j % 2 ? g2[j / 2].y : g2[j / 2].x;
                    q0[3 * a.plane] = j % 2 ? g3[j / 2].y : g3[j / 2].x;
                    q0[4 * a.plane] = j % 2 ? g4[j / 2].y : g4[j / 2].x;
                }
            }
        }
    }
    // no CTA leaves while another may still store to it
    cluster_sync();
    if (first_thread) {
        a.S.warm[b] = warm;
        a.S.grow[b] = grow;
        a.S.prevr[b] = prevr;
        if (done) {
            a.S.active[b] = 0;
            atomicSub(a.n_active, 1);
        }
    }
}

// the cold start for the tissues that abandoned their warm start
__global__ void steady_reset(int nx, int64_t pitch, int64_t plane, int64_t tstride,
                             const int* reset, float* g) {
    const int b = blockIdx.z;
    if (!reset[b]) return;
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y;
    if (x >= nx) return;
    float* G = g + (int64_t)b * tstride;
    for (int q = 0; q < 5; ++q) G[q * plane + (int64_t)y * pitch + x] = 0.f;
}

__global__ void steady_init(int batch, int nx, int ny, int64_t pitch, int64_t plane,
                            int64_t tstride, const float* phi0, float* g) {
    const int b = blockIdx.z;
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y;
    if (x >= nx) return;
    const float v = phi0 ? phi0[(int64_t)b * nx * ny + (int64_t)y * nx + x] : 0.f;
    float* G = g + (int64_t)b * tstride;
    constexpr float w1 = (float)(1.0 / 6.0);
    constexpr float w0 = 1.0f - 4.0f * w1;
    for (int q = 0; q < 5; ++q) G[q * plane + (int64_t)y * pitch + x] = (q == 0 ? w0 : w1) * v;
}

// How a batch runs on clusters: a form of the kernel, CTAs per cluster, strips
// per CTA.  cluster = 0: a tissue does not fit in one cluster and goes through
// steady_update.
struct SteadyPlan {
    int form = 0, cluster = 0, threads = 0, strips = 0, per_cta = 0;
    double cost = 0.0;
};

// The forms: rows per strip and threads per CTA at most.  Both hold 4,096
// nodes per CTA at most (5 registers of state per node); with the same nodes
// on an SM the taller strips publish less (256^2 on 16 CTAs: 0.96 us per step
// against 1.15), and the shorter ones spread a small tissue over more CTAs
// (256 x 64 on 16 CTAs of 256 threads: 0.58 us).
struct SteadyForm {
    int rows, threads;
};
constexpr SteadyForm kSteadyForms[2] = {{4, 1024}, {8, 512}};

template <int FORM, bool FULL>
static cudaError_t launch_steady_cluster(const SteadyPlan& p, int batch, const SteadyClusterArgs& a,
                                         cudaStream_t st, int* max_clusters) {
    constexpr int V = kSteadyForms[FORM].rows, NT = kSteadyForms[FORM].threads;
    auto kern = steady_cluster<V, NT, FULL>;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)p.cluster * (unsigned)batch);
    cfg.blockDim = dim3((unsigned)p.threads);
    cfg.dynamicSmemBytes = steady_cluster_smem(V, NT);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)p.cluster;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (!max_clusters) return cudaLaunchKernelEx(&cfg, kern, a);
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         steady_cluster_smem(V, NT));
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveClusters(max_clusters, kern, &cfg);
    return e;
}

static cudaError_t launch_steady_plan(const SteadyPlan& p, int batch, const SteadyClusterArgs& a,
                                      cudaStream_t st, int* max_clusters) {
    const bool full = a.ny % kSteadyForms[p.form].rows == 0;
    if (p.form == 0)
        return full ? launch_steady_cluster<0, true>(p, batch, a, st, max_clusters)
                    : launch_steady_cluster<0, false>(p, batch, a, st, max_clusters);
    return full ? launch_steady_cluster<1, true>(p, batch, a, st, max_clusters)
                : launch_steady_cluster<1, false>(p, batch, a, st, max_clusters);
}

// Clusters of C = 2^log2c CTAs that the current device holds at once (one CTA
// per SM whatever its threads), 0 where such a cluster cannot be launched.
// Asked of the driver once per device (a query costs about 10 us), which also
// sets the kernel's attributes there.
static int steady_clusters_resident(int form, bool full, int log2c) {
    constexpr int kDevices = 64;
    static std::atomic<int> known[kDevices][2][2][5];  // the answer + 1; 0: not asked yet
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev >= kDevices) return 0;
    std::atomic<int>& k = known[dev][form][full ? 1 : 0][log2c];
    int v = k.load();
    if (v == 0) {
        SteadyPlan p;
        p.form = form;
        p.cluster = 1 << log2c;
        p.threads = kSteadyForms[form].threads;
        SteadyClusterArgs a = {};
        a.ny = full ? kSteadyForms[form].rows : 1;
        int n = 0;
        if (launch_steady_plan(p, 1, a, nullptr, &n) != cudaSuccess) {
            cudaGetLastError();
            n = 0;
        }
        v = n + 1;
        k.store(v);
    }
    return v - 1;
}

// The plan with the least estimated time of a step: the rounds of clusters
// that are resident at once, times 0.45 us (the barrier and the dependent
// operations of a step) plus 0.5 us for 4,096 nodes on an SM, as measured.
static SteadyPlan steady_plan(int nx, int ny, int batch) {
    SteadyPlan best;
    for (int form = 0; form < 2; ++form) {
        const int V = kSteadyForms[form].rows;
        for (int l = 0; (1 << l) <= kSteadyClusterMax; ++l) {
            const int C = 1 << l;
            SteadyPlan p;
            p.form = form;
            p.cluster = C;
            p.strips = (ny + V - 1) / V;
            p.per_cta = (p.strips + C - 1) / C;
            if ((p.strips + p.per_cta - 1) / p.per_cta != C) continue;  // a CTA without rows
            if ((int64_t)nx * p.per_cta > kSteadyForms[form].threads) continue;
            p.threads = (nx * p.per_cta + 31) / 32 * 32;
            const int resident = steady_clusters_resident(form, ny % V == 0, l);
            if (resident < 1) continue;
            p.cost = std::ceil((double)batch / resident) *
                     (0.45 + 0.5 * (double)p.threads * V / 4096.0);
            if (!best.cluster || p.cost < best.cost) best = p;
        }
    }
    return best;
}

struct SteadyLayout {
    int64_t pitch, plane, tstride;
    uint64_t g[2], phi_prev, coef, active, dmax, pmax, steps, resid, nact, total;
    uint64_t warm, grow, fellback, reset, prevr, lost;
};

static SteadyLayout steady_layout(int nx, int ny, int batch) {
    SteadyLayout L;
    L.pitch = (nx + 31) / 32 * 32;
    L.plane = L.pitch * ny;
    L.tstride = 5 * L.plane;
    uint64_t o = 0;
    auto take = [&](uint64_t bytes) {
        uint64_t at = o;
        o = (o + bytes + 255) / 256 * 256;
        return at;
    };
    const uint64_t B = (uint64_t)batch, N = (uint64_t)nx * ny;
    L.g[0] = take(B * L.tstride * 4);
    L.g[1] = take(B * L.tstride * 4);
    L.phi_prev = take(B * N * 4);
    L.coef = take(B * 3 * 4);
    L.dmax = take(B * 4);
    L.pmax = take(B * 4);
    L.warm = take(B * 4);
    L.grow = take(B * 4);
    L.reset = take(B * 4);
    L.prevr = take(B * 4);
    // what the host reads, side by side
    L.steps = take(B * 8);
    L.resid = take(B * 8);
    L.fellback = take(B * 4);
    L.active = take(B * 4);
    L.nact = take(4);
    L.lost = take(4);
    L.total = o;
    return L;
}

// the state of every tissue before the first step
__global__ void steady_setup(int batch, int watched, SteadyState S, unsigned* dmax, unsigned* pmax,
                             long long* steps, double* resid, int* n_active, int* lost) {
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b == 0) {
        *n_active = batch;
        *lost = 0;
    }
    if (b >= batch) return;
    S.active[b] = 1;
    S.warm[b] = watched;  // a warm start is watched for the fallback; a cold start is not
    S.grow[b] = 0;
    S.fellback[b] = 0;
    S.reset[b] = 0;
    S.prevr[b] = 0.f;
    dmax[b] = pmax[b] = 0u;
    steps[b] = 0;
    resid[b] = INFINITY;
}

// One launch per step over every active tissue: lattices too large for a
// cluster's registers.  *n_out: the steps taken.
static cudaError_t steady_by_launches(int nx, int ny, int batch, const uint8_t* d_src,
                                      const float* d_phi0, double tol, int64_t max_steps,
                                      int check_every, float* d_phi_out, const SteadyLayout& L,
                                      char* ws, SteadyState S, long long* steps, double* resid,
                                      int* nact, unsigned* dmax, unsigned* pmax,
                                      cudaStream_t st, int64_t* n_out) {
    float* g[2] = {reinterpret_cast<float*>(ws + L.g[0]), reinterpret_cast<float*>(ws + L.g[1])};
    float* cf = reinterpret_cast<float*>(ws + L.coef);
    int* active = S.active;
    const dim3 blk(128), grd((nx + 127) / 128, ny, batch);
    cudaError_t e = cudaSuccess;
    {
        steady_init<<<grd, blk, 0, st>>>(batch, nx, ny, L.pitch, L.plane, L.tstride, d_phi0, g[0]);
        e = cudaGetLastError();
    }
    SteadyArgs a;
    a.src = d_src;
    a.omegaD = cf;
    a.decay = cf + batch;
    a.srate = cf + 2 * batch;
    a.active = active;
    a.phi_prev = reinterpret_cast<float*>(ws + L.phi_prev);
    a.nx = nx;
    a.ny = ny;
    a.pitch = L.pitch;
    a.plane = L.plane;
    a.tstride = L.tstride;
    int cur = 0;
    int64_t& n = *n_out;
    n = 0;
    const int64_t host_every = (int64_t)check_every * 8;
    while (e == cudaSuccess && n < max_steps) {
        const int64_t chunk_end = std::min(max_steps, n + host_every);
        for (; n < chunk_end && e == cudaSuccess;) {
            a.gsrc = g[cur];
            a.gdst = g[1 - cur];
            a.store_prev = ((n + 1) % check_every) == 0;
            steady_update<<<grd, blk, 0, st>>>(a);
            e = cudaGetLastError();
            cur = 1 - cur;
            ++n;
            if (e == cudaSuccess && n % check_every == 0) {
                steady_residual<<<grd, blk, 0, st>>>(g[cur], L.pitch, L.plane, L.tstride, nx,
                                                     ny, active, a.phi_prev, d_phi_out, dmax,
                                                     pmax);
                e = cudaGetLastError();
                if (e == cudaSuccess) {
                    steady_decide<<<(batch + 127) / 128, 128, 0, st>>>(
                        batch, n, tol, S, dmax, pmax, steps, resid, nact);
                    e = cudaGetLastError();
                }
                if (e == cudaSuccess && d_phi0) {
                    steady_reset<<<grd, blk, 0, st>>>(nx, L.pitch, L.plane, L.tstride, S.reset,
                                                      g[cur]);
                    e = cudaGetLastError();
                }
            }
        }
        int left = 0;
        if (e == cudaSuccess) e = cudaMemcpyAsync(&left, nact, 4, cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
        if (e == cudaSuccess && left == 0) break;
    }
    // tissues that ran out of steps: phi of their final state (residual of the
    // last check is kept); the residual kernel also writes phi_out
    if (e == cudaSuccess && n % check_every != 0) {
        // the last partial chunk left phi_prev stale: recompute phi only
        steady_residual<<<grd, blk, 0, st>>>(g[cur], L.pitch, L.plane, L.tstride, nx, ny, active,
                                             a.phi_prev, d_phi_out, dmax, pmax);
        e = cudaGetLastError();
    }
    return e;
}

}  // namespace lbib

using namespace lbib;

extern "C" {

int lbib_label_cells(int32_t nx, int32_t ny, int32_t bc_y, int32_t n_cells,
                     const int32_t* d_cell_off, const double* d_xy, const uint8_t* d_src_flag,
                     int32_t* d_id, uint8_t* d_src, void* cuda_stream) {
    NvtxRange nvtx_range("lbib_label_cells");
    if (nx < 8 || ny < 8 || bc_y < 0 || bc_y > 1 || n_cells < 0 || !d_id)
        return set_thread_error(LBIB_E_PARAM, "lbib_label_cells: invalid arguments");
    if (n_cells > 0 && (!d_cell_off || !d_xy || !d_src_flag))
        return set_thread_error(LBIB_E_PARAM, "lbib_label_cells: missing cell arrays");
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    const int64_t N = (int64_t)nx * ny;
    cudaError_t e = cudaMemsetAsync(d_id, 0xFF, N * 4, st);
    if (e == cudaSuccess && n_cells > 0) {
        IBArgs a;
        std::memset(&a, 0, sizeof(a));
        a.xy = const_cast<double2*>(reinterpret_cast<const double2*>(d_xy));
        a.off = d_cell_off;
        a.srcf = d_src_flag;
        a.id = reinterpret_cast<uint32_t*>(d_id);
        a.nx = nx;
        a.ny = ny;
        a.bc_y = bc_y;
        a.n_cells = n_cells;
        a.pitch = nx;
        a.plane = (int64_t)nx * ny;
        a.do_move = 0;
        a.do_prep = 1;
        a.do_mask = 1;
        a.do_force = 0;
        // packed labels (cell << 4 | bits, the lower cell index wins) ...
        a.do_ids = 1;
        e = launch_ib(LBIB_FP32, a, kMaxVertsPerCell, st);
        // ... then every containing cell ORs its source bits into the low bits
        if (e == cudaSuccess) {
            a.do_ids = 0;
            a.id = nullptr;
            a.src = d_id;
            a.src_words = 1;
            e = launch_ib(LBIB_FP32, a, kMaxVertsPerCell, st);
        }
    }
    if (e == cudaSuccess) {
        labels_to_ids<<<(unsigned)((N + 255) / 256), 256, 0, st>>>(
            reinterpret_cast<uint32_t*>(d_id), d_src, N);
        e = cudaGetLastError();
    }
    if (e != cudaSuccess)
        return set_thread_error(LBIB_E_CUDA, std::string("lbib_label_cells: ") +
                                                 cudaGetErrorString(e));
    return LBIB_OK;
}

int lbib_steady_workspace_size(int32_t nx, int32_t ny, int32_t batch, uint64_t* bytes_out) {
    if (nx < 8 || ny < 8 || batch < 1 || batch > 65535 || !bytes_out)
        return set_thread_error(LBIB_E_PARAM, "lbib_steady_workspace_size: invalid arguments");
    *bytes_out = steady_layout(nx, ny, batch).total;
    return LBIB_OK;
}

int lbib_steady_solve(int32_t nx, int32_t ny, int32_t batch, const uint8_t* d_src,
                      const double* D, const double* decay, const double* src_rate,
                      const float* d_phi0, double tol, int64_t max_steps, int32_t check_every,
                      float* d_phi_out, int64_t* steps_out, double* resid_out,
                      int32_t* fallback_out, void* d_workspace, uint64_t ws_bytes,
                      void* cuda_stream) {
    NvtxRange nvtx_range("lbib_steady_solve");
    if (nx < 8 || ny < 8 || batch < 1 || batch > 65535 || !d_src || !D || !decay ||
        !src_rate || !d_phi_out || !steps_out || !resid_out || check_every < 1 ||
        max_steps < 0 || !(tol >= 0.0))
        return set_thread_error(LBIB_E_PARAM, "lbib_steady_solve: invalid arguments");
    const SteadyLayout L = steady_layout(nx, ny, batch);
    if (!d_workspace || ws_bytes < L.total ||
        reinterpret_cast<uintptr_t>(d_workspace) % 256)
        return set_thread_error(LBIB_E_WORKSPACE, "lbib_steady_solve: workspace too small or misaligned");
    std::vector<float> coef((size_t)3 * batch);
    for (int b = 0; b < batch; ++b) {
        if (!(D[b] > 0.0) || !(decay[b] >= 0.0))
            return set_thread_error(LBIB_E_PARAM, "lbib_steady_solve: need D > 0, decay >= 0");
        coef[b] = (float)(1.0 / (3.0 * D[b] + 0.5));
        coef[batch + b] = (float)decay[b];
        coef[2 * batch + b] = (float)src_rate[b];
    }
    char* ws = static_cast<char*>(d_workspace);
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    float* cf = reinterpret_cast<float*>(ws + L.coef);
    unsigned* dmax = reinterpret_cast<unsigned*>(ws + L.dmax);
    unsigned* pmax = reinterpret_cast<unsigned*>(ws + L.pmax);
    long long* steps = reinterpret_cast<long long*>(ws + L.steps);
    double* resid = reinterpret_cast<double*>(ws + L.resid);
    int* nact = reinterpret_cast<int*>(ws + L.nact);
    int* lost = reinterpret_cast<int*>(ws + L.lost);
    SteadyState S;
    S.active = reinterpret_cast<int*>(ws + L.active);
    S.warm = reinterpret_cast<int*>(ws + L.warm);
    S.grow = reinterpret_cast<int*>(ws + L.grow);
    S.fellback = reinterpret_cast<int*>(ws + L.fellback);
    S.reset = reinterpret_cast<int*>(ws + L.reset);
    S.prevr = reinterpret_cast<float*>(ws + L.prevr);
    cudaError_t e = cudaMemcpyAsync(cf, coef.data(), coef.size() * 4, cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) {
        steady_setup<<<(batch + 127) / 128, 128, 0, st>>>(batch, d_phi0 ? 1 : 0, S, dmax, pmax,
                                                          steps, resid, nact, lost);
        e = cudaGetLastError();
    }
    // the results of every tissue, and how many are left, in one copy
    std::vector<char> host(L.lost + 4 - L.steps);
    const auto fetch = [&] {
        cudaError_t f = cudaMemcpyAsync(host.data(), ws + L.steps, host.size(),
                                        cudaMemcpyDeviceToHost, st);
        return f == cudaSuccess ? cudaStreamSynchronize(st) : f;
    };
    const auto host_int = [&](uint64_t at) {
        int v;
        std::memcpy(&v, host.data() + (at - L.steps), 4);
        return v;
    };
    const SteadyPlan plan = steady_plan(nx, ny, batch);
    int64_t n = 0;
    if (plan.cluster) {
        SteadyClusterArgs ca = {};
        ca.g = reinterpret_cast<float*>(ws + L.g[0]);
        ca.phi0 = d_phi0;
        ca.src = d_src;
        ca.omegaD = cf;
        ca.decay = cf + batch;
        ca.srate = cf + 2 * batch;
        ca.phi_out = d_phi_out;
        ca.S = S;
        ca.steps = steps;
        ca.resid = resid;
        ca.n_active = nact;
        ca.lost = lost;
        ca.tol = tol;
        ca.pitch = L.pitch;
        ca.plane = L.plane;
        ca.tstride = L.tstride;
        ca.nx = nx;
        ca.ny = ny;
        ca.check_every = check_every;
        ca.strips = plan.strips;
        ca.strips_per_cta = plan.per_cta;
        // a launch is bounded (8 ms for a 256^2 tissue); converged tissues
        // end theirs early
        constexpr int64_t kSteps = 8192;
        do {
            ca.first = n == 0;
            ca.n0 = n;
            ca.phase = (int)(n % check_every);
            ca.n_steps = (int)std::min(max_steps - n, kSteps);
            if (e == cudaSuccess && ca.n_steps > 0)
                e = launch_steady_plan(plan, batch, ca, st, nullptr);
            n += ca.n_steps;
            if (e == cudaSuccess) e = fetch();
            if (e == cudaSuccess && host_int(L.lost))
                return set_thread_error(LBIB_E_TIMEOUT, "lbib_steady_solve: a wait between the "
                                                        "CTAs of a cluster ran out");
        } while (e == cudaSuccess && n < max_steps && host_int(L.nact) > 0);
    } else {
        if (e == cudaSuccess)
            e = steady_by_launches(nx, ny, batch, d_src, d_phi0, tol, max_steps, check_every,
                                   d_phi_out, L, ws, S, steps, resid, nact, dmax, pmax, st, &n);
        if (e == cudaSuccess) e = fetch();
    }
    if (e != cudaSuccess)
        return set_thread_error(LBIB_E_CUDA, std::string("lbib_steady_solve: ") +
                                                 cudaGetErrorString(e));
    for (int b = 0; b < batch; ++b) {
        long long sb;
        std::memcpy(&sb, host.data() + (size_t)8 * b, 8);
        steps_out[b] = host_int(L.active + (uint64_t)4 * b) ? n : sb;
        std::memcpy(resid_out + b, host.data() + (L.resid - L.steps) + (size_t)8 * b, 8);
        if (fallback_out) fallback_out[b] = host_int(L.fellback + (uint64_t)4 * b);
    }
    return LBIB_OK;
}

}  // extern "C"
