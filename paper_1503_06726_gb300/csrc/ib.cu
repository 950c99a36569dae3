// ib.cu -- immersed-boundary side of the coupled step, one CTA per cell.
//
// A cell's vertices live in shared memory for the whole CTA, so the chain
//   interpolate u^n at X^n -> X^{n+1} = X^n + U^n      (Eq. conversion2, Fig. 1)
//   label the lattice nodes inside the new polygon      (Fig. 2, domainID)
//   vertex forces from springs, pressure, tension       (Sec. 3.2.3)
//   spread the forces to the 4x4 kernel support        (Eq. forcedistribution)
// runs in one launch between two lattice updates; no grid-wide sync is needed
// because every step only needs the cell's own vertices.
//
// Kernel of Eq. 1Dkernel: delta1D(r) = (1 + cos(pi r / 2)) / 4 for |r| <= 2,
// the 2-D kernel is delta1D(dx) delta1D(dy) over nodes floor(X)-1 .. floor(X)+2.
//
// Labelling: a node is inside a polygon by the crossing-number rule, half-open
// in y: edge a->b crosses row y when (y_a <= y) != (y_b <= y) and counts when
// x < x_a + (y - y_a)(x_b - x_a)/(y_b - y_a).  The CTA evaluates that crossing
// abscissa once per (edge, row) -- a scanline -- and keeps, per row, the
// integer thresholds ceil(x_c): a node at integer x is inside iff an odd
// number of thresholds exceed it.  This is the same predicate node by node,
// evaluated with explicitly rounded FP64 operations (no contraction), so the
// labels are exact.  Overlapping cells: the lowest cell index wins (atomicMin
// on the packed label cell << 4 | source bits).
#include <climits>
#include <type_traits>

#include "ib_cell.cuh"
#include "ib_cell_half.cuh"

namespace lbib {

// The FP64 kernel.  GB300 issues one FP64 instruction of a warp every 16
// cycles, so a cell costs its FP64 instructions (and, with few cells, their
// latency in a chain): what each needs is done once and side by side.  The
// spring of an edge serves both its vertices; the kernel weights of a vertex
// (a sincospi per axis) serve the spreading and, kept in a.vw, the next
// move; springs, the two axes' weights and the scanline crossings are tasks
// of different warps at the same time; and the sixteen stencil nodes of a
// vertex are shared by four lanes, a row each.  One 64-vertex cell on 64^2:
// 21.5 -> 14.1 us; 570 cells: 37.4 -> 30.3 us.
struct IBShared64 {
    double2* sx;   // positions
    double2* spr;  // spring force of the edge to the next vertex
    double* wt;    // the kernel weights, 4 in x then 4 in y, each maxv long
    int2* sb;      // floor(X)
    int4* wbox;    // each warp's bounding box
    int* rowcnt;   // kMaxRows
    int* thr;      // kMaxRows * kMaxCross
    int* s_flag;   // a scanline row overflowed
};
constexpr int kIBSmem64Fixed = 8 * 16 + ((kMaxRows + kMaxRows * kMaxCross + 1) * 4 + 15) / 16 * 16;
constexpr int kIBSmem64PerVertex = 16 + 16 + 8 * 8 + 8;

// |v| < 1e9 (not a NaN) by the bits, off the FP64 pipe
__device__ __forceinline__ bool within_1e9(double v) {
    return (__double2hiint(v) & 0x7fffffff) < 0x41cdcd65;
}

__global__ void __launch_bounds__(kIBThreads) ib_cell_kernel_f64(IBArgs a, int maxv) {
    extern __shared__ __align__(16) unsigned char ib_smem64[];
    IBShared64 S;
    S.wbox = reinterpret_cast<int4*>(ib_smem64);
    S.rowcnt = reinterpret_cast<int*>(S.wbox + 8);
    S.thr = S.rowcnt + kMaxRows;
    S.s_flag = S.thr + kMaxRows * kMaxCross;
    S.sx = reinterpret_cast<double2*>(ib_smem64 + kIBSmem64Fixed);
    S.spr = S.sx + maxv;
    S.wt = reinterpret_cast<double*>(S.spr + maxv);
    S.sb = reinterpret_cast<int2*>(S.wt + 8 * maxv);
    double2* const sx = S.sx;

    const int c = blockIdx.x;
    const int v0 = __ldcg(a.off + c);
    const int n = __ldcg(a.off + c + 1) - v0;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    constexpr int NT = kIBThreads, NW = NT / 32;
    // the shared arrays hold maxv vertices and a polygon needs three; callers
    // that pass device offsets unchecked (the allocation-free step) get the
    // geometry flag instead of an access past sx
    const bool vok = LBIB_CHK_INDEX(a.diag, kSiteIbVertex, v0, (int64_t)__ldcg(a.off + a.n_cells)) &&
                     LBIB_CHK_INDEX(a.diag, kSiteIbVertex, (int64_t)v0 + n - 1,
                                    (int64_t)__ldcg(a.off + a.n_cells));
    if (n > maxv || n < 3 || !vok) {
        griddep_wait();
        griddep_launch_dependents();
        if (tid == 0) raise_flag(a.diag, kDiagGeometry);
        return;
    }
    // the cell is labelled when the caller wants the packed labels or the cell
    // has source bits to deposit
    const bool may_label =
        a.do_prep && a.do_mask && (a.do_ids || (a.src && (__ldcg(a.srcf + c) & 0xF)));
    if (tid < kMaxRows) S.rowcnt[tid] = 0;
    if (tid == 0) *S.s_flag = 0;
    // four lanes per vertex; the vertex's state was written by the IB launch
    // two launches back (see griddep_wait)
    const int j = tid & 3;
    double2 X0 = make_double2(0.0, 0.0), wxa, wxb;
    double wy0 = 0.0;
    int2 b0 = make_int2(0, 0);
    wxa = wxb = X0;
    auto weights = [&](int t, double2* lo, double2* hi, double* y, int2* b, double2 X) {
        if (a.vw) {
            const double* w = a.vw + (int64_t)8 * (v0 + t);
            *lo = __ldcg(reinterpret_cast<const double2*>(w));
            *hi = __ldcg(reinterpret_cast<const double2*>(w) + 1);
            *y = __ldcg(w + 4 + j);
            *b = __ldcg(a.vbase + v0 + t);
        } else {
            double wx[4], wy[4];
            int bx, by;
            axis_weights<double>(X.x, &bx, wx);
            axis_weights<double>(X.y, &by, wy);
            *lo = make_double2(wx[0], wx[1]);
            *hi = make_double2(wx[2], wx[3]);
            *y = j == 0 ? wy[0] : (j == 1 ? wy[1] : (j == 2 ? wy[2] : wy[3]));
            *b = make_int2(bx + 1, by + 1);
        }
    };
    if ((tid >> 2) < n) {
        X0 = __ldcg(a.xy + v0 + (tid >> 2));
        if (a.do_move) weights(tid >> 2, &wxa, &wxb, &wy0, &b0, X0);
    }
    griddep_wait();
    griddep_launch_dependents();
    const int pitch = (int)a.pitch;  // a plane holds fewer than 2^31 nodes

    // ---- (1) interpolate u^n at X^n and move (or just load); integer bounding box
    int ilo = INT_MAX, ihi = INT_MIN, jlo = INT_MAX, jhi = INT_MIN;
    bool finite_x = true;
    for (int base = 0; base < n; base += NT / 4) {
        const int t = base + (tid >> 2);
        const bool in = t < n;
        double2 X = X0;
        double Ux = 0.0, Uy = 0.0;  // this lane's row
        if (in) {
            double2 lo = wxa, hi = wxb;
            double y = wy0;
            int2 b = b0;
            if (base) {
                X = a.xy[v0 + t];
                if (a.do_move) weights(t, &lo, &hi, &y, &b, X);
            }
            if (a.do_move) {
                const int x0 = wrap_near(b.x - 1, a.nx);
                int J = b.y - 1 + j;
                if (!a.bc_y) J = wrap_near(J, a.ny);
                if ((unsigned)J < (unsigned)a.ny) {  // else outside a walled lattice
                    const double2* row = static_cast<const double2*>(a.u) + J * pitch;
                    double2 v[4];
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        v[i] = u_ld(a, row + (x0 + i >= a.nx ? x0 + i - a.nx : x0 + i));
                    Ux = y * fma(hi.y, v[3].x, fma(hi.x, v[2].x, fma(lo.y, v[1].x, lo.x * v[0].x)));
                    Uy = y * fma(hi.y, v[3].y, fma(hi.x, v[2].y, fma(lo.y, v[1].y, lo.x * v[0].y)));
                }
            }
        }
        if (a.do_move) {
            // the four rows of a vertex: the even lanes sum x, the odd ones y
            const bool odd = j & 1;
            const double other = __shfl_xor_sync(0xffffffffu, odd ? Ux : Uy, 1);
            double U = (odd ? Uy : Ux) + other;
            U += __shfl_xor_sync(0xffffffffu, U, 2);
            U += odd ? X.y : X.x;
            X.x = U;
            X.y = __shfl_xor_sync(0xffffffffu, U, 1);  // (used by the even lanes)
        }
        if (in && j == 0) {
            if (a.do_move) a.xy[v0 + t] = X;
            sx[t] = X;
            finite_x = finite_x && within_1e9(X.x) && within_1e9(X.y);
            ilo = min(ilo, __double2int_rd(X.x));
            ihi = max(ihi, __double2int_ru(X.x));
            jlo = min(jlo, __double2int_rd(X.y));
            jhi = max(jhi, __double2int_ru(X.y));
        }
    }
    if (!a.do_prep) return;
    ilo = __reduce_min_sync(0xffffffffu, ilo);
    ihi = __reduce_max_sync(0xffffffffu, ihi);
    jlo = __reduce_min_sync(0xffffffffu, jlo);
    jhi = __reduce_max_sync(0xffffffffu, jhi);
    finite_x = __all_sync(0xffffffffu, finite_x);
    // the warps' boxes side by side, a non-finite one as the whole range
    if (lane == 0) S.wbox[warp] = make_int4(ilo, finite_x ? ihi : INT_MAX, jlo, jhi);
    __syncthreads();
#pragma unroll
    for (int w = 0; w < NW; ++w) {
        const int4 o = S.wbox[w];
        ilo = min(ilo, o.x);
        ihi = max(ihi, o.y);
        jlo = min(jlo, o.z);
        jhi = max(jhi, o.w);
    }
    if (a.msrc_out && warp == NW - 1) {  // the cell's mass source (Sec. 3.2.3)
        const double a_c = cell_area_warp(sx, n, lane);
        if (lane == 0) static_cast<double*>(a.msrc_out)[c] = mass_source(a, c, a_c);
    }
    const int I0 = ilo, I1 = ihi, J0 = jlo, J1 = jhi;
    // Labels need a finite box no wider than the lattice; otherwise the
    // geometry has blown up: flag it and leave the labels empty so that every
    // loop below stays bounded by the lattice size.
    const bool geom_ok = ihi != INT_MAX && (I1 - I0) <= a.nx && (J1 - J0) <= a.ny;
    if (a.do_mask && !geom_ok && tid == 0) raise_flag(a.diag, kDiagGeometry);
    const bool labels = may_label && geom_ok;
    const int rows = J1 - J0 + 1, cols = I1 - I0 + 1;
    const bool scan = labels && rows <= kMaxRows;

    // ---- (2) per vertex or edge: the spring of the edge, the weights of the
    // two axes, the scanline crossings of the edge, whole warps of each
    const int n32 = (n + 31) & ~31;
    for (int e = tid; e < (scan ? 4 : 3) * n32; e += NT) {
        const int kind = e / n32, t = e - kind * n32;
        if (t >= n) continue;
        if (kind == 0) {
            if (!a.do_force) continue;
            double2 F;
            spring<double>(sx[t], sx[t == n - 1 ? 0 : t + 1], a.L0[v0 + t], a.k[v0 + t], &F.x,
                           &F.y);
            S.spr[t] = F;
        } else if (kind < 3) {
            if (!a.do_force) continue;
            const int axis = kind - 1;
            int base;
            double w[4];
            axis_weights<double>(axis ? sx[t].y : sx[t].x, &base, w);
#pragma unroll
            for (int i = 0; i < 4; ++i) S.wt[(4 * axis + i) * maxv + t] = w[i];
            reinterpret_cast<int*>(S.sb + t)[axis] = base + 1;
            if (a.vw) {
                double2* o = reinterpret_cast<double2*>(a.vw + (int64_t)8 * (v0 + t) + 4 * axis);
                o[0] = make_double2(w[0], w[1]);
                o[1] = make_double2(w[2], w[3]);
                reinterpret_cast<int*>(a.vbase + v0 + t)[axis] = base + 1;
            }
        } else {
            // the edge's rows J with (y_a <= J) != (y_b <= J), exactly, and on
            // each the threshold ceil(x_c): in FP32 where that decides it, else
            // by the FP64 formula (as in ib_cell_f32)
            const double2 A = sx[t], B = sx[(t == n - 1) ? 0 : t + 1];
            int2 ba, bb;
            float2 fa, fb;
            base_frac(A.x, &ba.x, &fa.x);
            base_frac(A.y, &ba.y, &fa.y);
            base_frac(B.x, &bb.x, &fb.x);
            base_frac(B.y, &bb.y, &fb.y);
            // (a fraction that rounds to one in FP32 is still above zero)
            const int cya = __double2int_ru(A.y), cyb = __double2int_ru(B.y);
            const int jl = min(cya, cyb), jh = max(cya, cyb) - 1;
            const float2 d = edge_vec(ba, fa, bb, fb);
            const float ratio = fabsf(d.x) / fabsf(d.y);
            for (int J = jl; J <= jh; ++J) {
                const float pr = (float)(J - ba.y) - fa.y;
                const float xr = fa.x + (pr * d.x) / d.y;
                const float E = 9.5367431640625e-07f * (4.f + 4.f * ratio + fabsf(d.x) + fabsf(xr));
                const float clo = ceilf(xr - E), chi = ceilf(xr + E);
                int ti;
                if (clo == chi) {
                    ti = ba.x + (int)clo;
                } else {
                    const double tc = ceil(crossing_x(A, B, (double)J));
                    ti = tc < (double)I0 ? I0 : (tc > (double)(I1 + 1) ? I1 + 1 : (int)tc);
                }
                ti = ti < I0 ? I0 : (ti > I1 + 1 ? I1 + 1 : ti);
                const int slot = atomicAdd(&S.rowcnt[J - J0], 1);
                if (slot < kMaxCross)
                    S.thr[(J - J0) * kMaxCross + slot] = ti;
                else
                    *S.s_flag = 1;
            }
        }
    }
    __syncthreads();

    // ---- (3) vertex forces and spreading, four lanes per vertex
    if (a.do_force) {
        double2* force = static_cast<double2*>(a.force);
        const double hp = 0.5 * a.pres[c];
        const double ten = a.tension;
        for (int e = tid; e < 4 * n; e += NT) {
            const int t = e >> 2;
            const unsigned quad = 0xfu << (lane & 28);  // the vertex's four lanes
            const int tp = (t == 0) ? n - 1 : t - 1;
            const int tn = (t == n - 1) ? 0 : t + 1;
            const double2 X = sx[t], Xp = sx[tp], Xn = sx[tn];
            // the even lanes form the x component (springs, and the pressure
            // p dA/dX of a CCW polygon), the odd ones y
            const double2 s0 = S.spr[t], s1 = S.spr[tp];
            const bool odd = j & 1;
            const double F1 = fma(hp, odd ? Xp.x - Xn.x : Xn.y - Xp.y,
                                  (odd ? s0.y : s0.x) - (odd ? s1.y : s1.x));
            const double F2 = __shfl_xor_sync(quad, F1, 1);
            double Fx = odd ? F2 : F1, Fy = odd ? F1 : F2;
            if (ten != 0.0) {  // Eq. membraneforce
                const double ux_ = Xp.x - X.x, uy_ = Xp.y - X.y;
                const double vx_ = Xn.x - X.x, vy_ = Xn.y - X.y;
                const double la = sqrt(ux_ * ux_ + uy_ * uy_), lb = sqrt(vx_ * vx_ + vy_ * vy_);
                Fx += ten * (ux_ / la + vx_ / lb);
                Fy += ten * (uy_ / la + vy_ / lb);
            }
            if (a.jpartner) {  // Eq. celljunctionforce (a launch without the move)
                const double2 J = junction_force64(a, X, a.jpartner[v0 + t]);
                Fx += J.x;
                Fy += J.y;
            }
            if (a.write_vforce && j == 0) a.vforce[v0 + t] = make_double2(Fx, Fy);
            const int2 b = S.sb[t];
            const int x0 = wrap_near(b.x - 1, a.nx);
            int J = b.y - 1 + j;
            if (a.bc_y) {
                if (J < 0 || J >= a.ny) {
                    raise_flag(a.diag, kDiagWallStencil);
                    continue;
                }
            } else {
                J = wrap_near(J, a.ny);
            }
            const double y = S.wt[(4 + j) * maxv + t];
            const double Fxw = Fx * y, Fyw = Fy * y;
            int ix[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                ix[i] = x0 + i >= a.nx ? x0 + i - a.nx : x0 + i;
                const double w = S.wt[i * maxv + t];
                spread_add(a, force + (J * pitch + ix[i]), Fxw * w, Fyw * w);
            }
            mark_row(a, a.fmask, (int64_t)J * pitch, ix);
        }
    }
    if (!labels) return;  // uniform over the CTA
    fill_labels_body(a, c, n, sx, S.rowcnt, S.thr, scan && *S.s_flag == 0, I0, J0, rows, cols, tid,
                     NT);
}

// FP32 path: dynamic shared memory sized for the largest cell, NT threads
template <int NT>
__device__ __forceinline__ void ib_f32_body(const IBArgs& a, int maxv) {
    extern __shared__ __align__(16) unsigned char ib_smem[];
    const IBShared32 S = ib_shared32_view(ib_smem, maxv);
    ib_cell_f32<NT, true, NT == 256>(a, blockIdx.x, S, threadIdx.x, 0);
}

// the 128- and 256-thread kernels at the registers the compiler chooses
template <int NT>
__global__ void __launch_bounds__(NT) ib_cell_kernel_f32(IBArgs a, int maxv) {
    ib_f32_body<NT>(a, maxv);
}

// the 64-thread kernel (many small cells): 12 CTAs per SM leave it the 80
// registers that hold a vertex's velocity rows at once (9,801 cells: 79 us;
// 81 at 14 or 16 CTAs, 82 at 10, 123 at 20, where the rows spill)
__global__ void __launch_bounds__(64, 12) ib_cell_kernel_f32_64(IBArgs a, int maxv) {
    ib_f32_body<64>(a, maxv);
}

// FP16 storage: the same kernels over ib_cell_half
template <int NT>
__device__ __forceinline__ void ib_half_body(const IBArgs& a, int maxv) {
    extern __shared__ __align__(16) unsigned char ib_smem[];
    const IBSharedHalf S = ib_shared_half_view(ib_smem, maxv);
    ib_cell_half<NT>(a, blockIdx.x, S, threadIdx.x, 0);
}
template <int NT>
__global__ void __launch_bounds__(NT) ib_cell_kernel_half(IBArgs a, int maxv) {
    ib_half_body<NT>(a, maxv);
}
__global__ void __launch_bounds__(64, 18) ib_cell_kernel_half_64(IBArgs a, int maxv) {
    ib_half_body<64>(a, maxv);
}

cudaError_t launch_ib(int precision, const IBArgs& a, int maxv_cell, cudaStream_t s, bool pdl) {
    if (a.n_cells <= 0) return cudaSuccess;
    int maxv = maxv_cell < 3 ? 3 : (maxv_cell > kMaxVertsPerCell ? kMaxVertsPerCell : maxv_cell);
    maxv = (maxv + 7) / 8 * 8;
    if (precision == LBIB_FP64) {
        const size_t bytes = kIBSmem64Fixed + (size_t)maxv * kIBSmem64PerVertex;
        if (bytes > 48 * 1024) {  // cells of more than 420 vertices
            const cudaError_t e = cudaFuncSetAttribute(
                ib_cell_kernel_f64, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
            if (e != cudaSuccess) return e;
        }
        return launch_kernel(ib_cell_kernel_f64, dim3(a.n_cells), dim3(kIBThreads), bytes, s, pdl,
                             a, maxv);
    }
    // small, numerous cells: 128-thread CTAs and shared memory sized to the
    // largest cell let many more CTAs be resident per SM
    if (precision == LBIB_FP16) {
        const size_t half = kIBSmemHalfFixed + (size_t)maxv * kIBSmemHalfPerVertex;
        if (maxv <= 64 && a.n_cells >= 2048)
            return launch_kernel(ib_cell_kernel_half_64, dim3(a.n_cells), dim3(64), half, s, pdl,
                                 a, maxv);
        if (maxv <= 128 && a.n_cells >= 2048)
            return launch_kernel(ib_cell_kernel_half<128>, dim3(a.n_cells), dim3(128), half, s,
                                 pdl, a, maxv);
        return launch_kernel(ib_cell_kernel_half<256>, dim3(a.n_cells), dim3(256), half, s, pdl,
                             a, maxv);
    }
    const size_t smem = kIBSmemFixed + (size_t)maxv * kIBSmemPerVertex;
    if (maxv <= 64 && a.n_cells >= 2048)
        return launch_kernel(ib_cell_kernel_f32_64, dim3(a.n_cells), dim3(64), smem, s, pdl, a,
                             maxv);
    if (maxv <= 128 && a.n_cells >= 2048)
        return launch_kernel(ib_cell_kernel_f32<128>, dim3(a.n_cells), dim3(128), smem, s, pdl, a,
                             maxv);
    return launch_kernel(ib_cell_kernel_f32<256>, dim3(a.n_cells), dim3(256), smem, s, pdl, a,
                         maxv);
}

// Per-cell shoelace area relative to the first vertex, FP64 (computeAreas).
__global__ void areas_kernel(const double2* xy, const int32_t* off, int n_cells, double* area) {
    const int c = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (c >= n_cells) return;
    const int v0 = off[c], n = off[c + 1] - v0;
    const double2 P0 = xy[v0];
    double s = 0.0;
    for (int t = lane; t < n; t += 32) {
        double2 A = xy[v0 + t], B = xy[v0 + ((t == n - 1) ? 0 : t + 1)];
        double xl = A.x - P0.x, yl = A.y - P0.y, xm = B.x - P0.x, ym = B.y - P0.y;
        s += xl * ym - xm * yl;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) area[c] = 0.5 * s;
}

cudaError_t launch_areas(const double2* xy, const int32_t* off, int n_cells, double* area,
                         cudaStream_t s) {
    if (n_cells <= 0) return cudaSuccess;
    areas_kernel<<<(n_cells + 3) / 4, 128, 0, s>>>(xy, off, n_cells, area);
    return cudaGetLastError();
}

}  // namespace lbib
