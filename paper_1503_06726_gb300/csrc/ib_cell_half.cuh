// ib_cell_half.cuh -- the immersed-boundary work of one cell for FP16 storage.
//
// The populations of FP16 storage are rounded to 11 bits every step, so the
// order in which the force reductions of neighbouring cells land, which
// changes the last bit of a force now and then, is felt in the trajectory
// (vertex positions at 1e-8 after 300 steps; FP32 storage 1e-11).  The kernel
// of ib_cell.cuh lands them in another order (its CTAs are shorter and fewer
// to an SM) and took the positions of an FP16 run after 600 steps 2.1e-8
// from those of this one, whose own runs differ by 1.5e-8; it is 1.1 times
// as fast per step there (3,339 cells: 34 us against 47).  Runs in FP16 keep
// this kernel and with it the spread they had.
#pragma once

#include "ib_cell.cuh"

namespace lbib {

// shared memory of one cell, as pointers into the CTA's shared memory; the
// vertex arrays hold `maxv` entries
struct IBSharedHalf {
    double2* sx;  // FP64 positions (exact fallbacks)
    int2* sb;     // floor(X)
    float2* sf;   // X - floor(X)
    int* rowcnt;  // kMaxRows
    int* thr;     // kMaxRows * kMaxCross
    int* sbox;    // 4
    int* s_flag;  // 1
    // the cell's force-mask words (kMaskTable keys and bits): the spreading
    // ORs its group bits here and the CTA then ORs each distinct word into
    // the mask once
    uint32_t* mkey;
    uint32_t* mval;
    int maxv;
};

constexpr int kMaskTableLog2 = 8;
constexpr int kMaskTable = 1 << kMaskTableLog2;
constexpr uint32_t kMaskEmpty = 0xFFFFFFFFu;

constexpr int kIBSmemHalfFixed =
    ((kMaxRows + kMaxRows * kMaxCross + 4 + 1 + 2 * kMaskTable) * 4 + 15) / 16 * 16;
constexpr int kIBSmemHalfPerVertex = 16 + 8 + 8;

__device__ __forceinline__ IBSharedHalf ib_shared_half_view(unsigned char* base, int maxv) {
    IBSharedHalf v;
    int* fixed = reinterpret_cast<int*>(base);
    v.rowcnt = fixed;
    v.thr = fixed + kMaxRows;
    v.sbox = v.thr + kMaxRows * kMaxCross;
    v.s_flag = v.sbox + 4;
    v.mkey = reinterpret_cast<uint32_t*>(v.s_flag + 1);
    v.mval = v.mkey + kMaskTable;
    v.sx = reinterpret_cast<double2*>(base + kIBSmemHalfFixed);
    v.sb = reinterpret_cast<int2*>(v.sx + maxv);
    v.sf = reinterpret_cast<float2*>(v.sb + maxv);
    v.maxv = maxv;
    return v;
}

// OR `bits` into mask word `wd` through the CTA's table of the cell's words
// (open addressing in shared memory; the word goes to the mask once, at the
// flush after the spreading); a full table falls back to the global atomic.
__device__ __forceinline__ void mask_or_table(const IBArgs& a, uint32_t* mask, int64_t wd,
                                              uint32_t bits, uint32_t* mkey, uint32_t* mval) {
    if (!LBIB_CHK_INDEX(a.diag, kSiteMask, wd, mask_words(a.plane))) return;
    const uint32_t k = (uint32_t)wd;
    uint32_t h = (k * 2654435761u) >> (32 - kMaskTableLog2);
#pragma unroll 1
    for (int probe = 0; probe < 16; ++probe) {
        const uint32_t old = atomicCAS(mkey + h, kMaskEmpty, k);
        if (old == kMaskEmpty || old == k) {
            atomicOr(mval + h, bits);
            return;
        }
        h = (h + 1) & (uint32_t)(kMaskTable - 1);
    }
    atomicOr(mask + wd, bits);
}

// mark_row through the table
__device__ __forceinline__ void mark_row_table(const IBArgs& a, uint32_t* mask, int64_t rowbase,
                                               const int ix[4], uint32_t* mkey, uint32_t* mval) {
    if (!mask) return;
    int64_t wd = -1;
    uint32_t bits = 0u;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int64_t g = (rowbase + ix[i]) >> 2;
        if ((g >> 5) != wd) {
            if (bits) mask_or_table(a, mask, wd, bits, mkey, mval);
            wd = g >> 5;
            bits = 0u;
        }
        bits |= 1u << (g & 31);
    }
    mask_or_table(a, mask, wd, bits, mkey, mval);
}

// spring force on the first vertex of an edge with vector d (FP32)
__device__ __forceinline__ float2 spring32_force(float2 d, float L0, float kk) {
    const float len2 = d.x * d.x + d.y * d.y;
    const float len = sqrtf(len2);
    const float sc = kk * ((len2 - L0 * L0) / (len + L0)) / len;
    return make_float2(sc * d.x, sc * d.y);
}

// The work of one cell by the NT threads of a CTA.  The force-mask bits go
// through the cell's table of mask words (NT <= 128), or straight to the mask
// (the 256-thread kernel of few large cells).
template <int NT>
static __device__ void ib_cell_half(const IBArgs& a, int c, const IBSharedHalf& S, int tid,
                                    int bar) {
    constexpr bool GRIDDEP = true, INLINE_FILL = NT == 256, OPTS = true, MASK_TABLE = NT <= 128;
    static_assert(NT % 64 == 0, "CTA size");
    constexpr int kIBThreads = NT;
    double2* sx = S.sx;
    int2* sb = S.sb;
    float2* sf = S.sf;
    int* rowcnt = S.rowcnt;
    int* thr = S.thr;
    int* sbox = S.sbox;
    int& s_flag = *S.s_flag;
    cell_sync<NT>(bar);

    const int v0 = __ldcg(a.off + c);
    const int n = __ldcg(a.off + c + 1) - v0;
    const int lane = tid & 31;
    // the checking build: the cell's vertices inside the vertex arrays
    const bool vok = LBIB_CHK_INDEX(a.diag, kSiteIbVertex, v0, (int64_t)__ldcg(a.off + a.n_cells)) &&
                     LBIB_CHK_INDEX(a.diag, kSiteIbVertex, (int64_t)v0 + n - 1,
                                    (int64_t)__ldcg(a.off + a.n_cells));
    if (n > S.maxv || n < 3 || !vok) {  // cannot happen for callers that size maxv from the cells
        if (GRIDDEP) {
            griddep_wait();
            griddep_launch_dependents();
        }
        if (tid == 0) raise_flag(a.diag, kDiagGeometry);
        return;
    }

    for (int r = tid; r < kMaxRows; r += NT) rowcnt[r] = 0;
    if (MASK_TABLE) {
        for (int i = tid; i < kMaskTable; i += NT) {
            S.mkey[i] = kMaskEmpty;
            S.mval[i] = 0u;
        }
    }
    if (tid == 0) {
        sbox[0] = INT_MAX; sbox[1] = INT_MIN; sbox[2] = INT_MAX; sbox[3] = INT_MIN;
        s_flag = 0;
    }

    // spring data of the vertices this thread will handle in phase 2, loaded
    // now so that phase 2 waits on no load: vertex tid (every thread: the whole
    // CTA computes forces when the cell is not labelled) and vertex tid + half
    // (the first half, which alone computes forces while the second half
    // scans the rows of a labelled cell)
    constexpr int half = kIBThreads / 2;
    float pL0[2] = {0.f, 0.f}, pk[2] = {0.f, 0.f}, pL0p[2] = {0.f, 0.f}, pkp[2] = {0.f, 0.f};
    float ppres = 0.f;
    if (a.do_prep && a.do_force) {
        ppres = (float)__ldcg(a.pres + c);
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const int t = tid + r * half;
            if (t < n && (r == 0 || tid < half)) {
                const int tp = (t == 0) ? n - 1 : t - 1;
                pL0[r] = (float)__ldcg(a.L0 + v0 + t);
                pk[r] = (float)__ldcg(a.k + v0 + t);
                pL0p[r] = (float)__ldcg(a.L0 + v0 + tp);
                pkp[r] = (float)__ldcg(a.k + v0 + tp);
            }
        }
    }
    // the vertex state of this thread's first vertex
    double2 X0 = make_double2(0.0, 0.0);
    int2 b0 = make_int2(0, 0);
    float2 f0 = make_float2(0.f, 0.f);
    if (tid < n) {
        X0 = __ldcg(a.xy + v0 + tid);
        if (a.do_move && a.vbase) {
            b0 = __ldcg(a.vbase + v0 + tid);
            f0 = __ldcg(a.vfrac + v0 + tid);
        }
    }
    if (GRIDDEP) {
        griddep_wait();
        griddep_launch_dependents();
    }

    // ---- (1) interpolate u^n at X^n and move; (base, frac) of the new X
    int ilo = INT_MAX, ihi = INT_MIN, jlo = INT_MAX, jhi = INT_MIN;
    bool finite = true;
    for (int t = tid; t < n; t += kIBThreads) {
        double2 X = (t == tid) ? X0 : a.xy[v0 + t];
        int2 b;
        float2 f;
        if (a.do_move) {
            if (a.vbase) {
                b = (t == tid) ? b0 : a.vbase[v0 + t];
                f = (t == tid) ? f0 : a.vfrac[v0 + t];
            } else {
                base_frac(X.x, &b.x, &f.x);
                base_frac(X.y, &b.y, &f.y);
            }
            float wx[4], wy[4];
            weights_from_frac(f.x, wx);
            weights_from_frac(f.y, wy);
            const float2* u = static_cast<const float2*>(a.u);
            float Ux = 0.f, Uy = 0.f;
            int ix[4];
            ix[0] = wrapi(b.x - 1, a.nx);
#pragma unroll
            for (int i = 1; i < 4; ++i) ix[i] = (ix[i - 1] + 1 == a.nx) ? 0 : ix[i - 1] + 1;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                int J = b.y - 1 + j;
                if (a.bc_y) {
                    if (J < 0 || J >= a.ny) continue;
                } else {
                    J = wrapi(J, a.ny);
                }
                const float2* row = u + (int64_t)J * a.pitch;
                // the four nodes of the row, 16 bytes per load where aligned
                float2 v[4];
                if (ix[3] == ix[0] + 3) {
                    const float2* r0 = row + ix[0];
                    if ((ix[0] & 1) == 0) {
                        const float4 p0 = u_ld4(a, r0);
                        const float4 p1 = u_ld4(a, r0 + 2);
                        v[0] = make_float2(p0.x, p0.y);
                        v[1] = make_float2(p0.z, p0.w);
                        v[2] = make_float2(p1.x, p1.y);
                        v[3] = make_float2(p1.z, p1.w);
                    } else {
                        const float4 p1 = u_ld4(a, r0 + 1);
                        v[0] = u_ld(a, r0);
                        v[1] = make_float2(p1.x, p1.y);
                        v[2] = make_float2(p1.z, p1.w);
                        v[3] = u_ld(a, r0 + 3);
                    }
                } else {
#pragma unroll
                    for (int i = 0; i < 4; ++i) v[i] = u_ld(a, row + ix[i]);
                }
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const float w = wx[i] * wy[j];
                    Ux += v[i].x * w;
                    Uy += v[i].y * w;
                }
            }
            X.x += (double)Ux;
            X.y += (double)Uy;
            a.xy[v0 + t] = X;
        }
        base_frac(X.x, &b.x, &f.x);
        base_frac(X.y, &b.y, &f.y);
        sx[t] = X;
        sb[t] = b;
        sf[t] = f;
        if (a.do_prep && a.vbase) {
            a.vbase[v0 + t] = b;
            a.vfrac[v0 + t] = f;
        }
        finite = finite && isfinite(f.x) && isfinite(f.y) && b.x > -1000000000 &&
                 b.x < 1000000000 && b.y > -1000000000 && b.y < 1000000000;
        const int cyv = b.y + (f.y > 0.f ? 1 : 0);  // ceil(y), exact
        ilo = min(ilo, b.x);
        ihi = max(ihi, b.x);
        jlo = min(jlo, cyv);
        jhi = max(jhi, cyv);
    }
    if (!a.do_prep) return;
    ilo = __reduce_min_sync(0xffffffffu, ilo);
    ihi = __reduce_max_sync(0xffffffffu, ihi);
    jlo = __reduce_min_sync(0xffffffffu, jlo);
    jhi = __reduce_max_sync(0xffffffffu, jhi);
    finite = __all_sync(0xffffffffu, finite);
    cell_sync<NT>(bar);
    if (lane == 0) {
        atomicMin(&sbox[0], ilo);
        atomicMax(&sbox[1], ihi);
        atomicMin(&sbox[2], jlo);
        atomicMax(&sbox[3], jhi);
        if (!finite) s_flag = 2;
    }
    cell_sync<NT>(bar);
    if (OPTS && a.msrc_out && tid < 32) {
        // mass source of the cell (Sec. 3.2.3): S_c = rate + alpha (A0 - A_c),
        // A_c the shoelace area of the moved polygon about its first vertex
        const double a_c = cell_area_warp(sx, n, lane);
        if (lane == 0) static_cast<float*>(a.msrc_out)[c] = (float)mass_source(a, c, a_c);
    }
    // columns: floor(x) over the vertices, widened by one on each side (the
    // fractions are FP32); rows: every J with min ceil(y) <= J < max ceil(y),
    // exactly the rows some edge crosses
    const int I0 = sbox[0] - 1, I1 = sbox[1] + 1, J0 = sbox[2], J1 = sbox[3] - 1;
    // a box no wider than the lattice keeps the wrapped indices of the fill
    // within one period; anything wider means the geometry has blown up
    const bool geom_ok = s_flag == 0 && (I1 - I0) < a.nx && (J1 - J0) <= a.ny;
    if (a.do_mask && !geom_ok && tid == 0) raise_flag(a.diag, kDiagGeometry);
    // the cell is labelled when the caller wants the packed labels or the cell
    // has source bits to deposit
    const bool labels =
        a.do_mask && geom_ok && J1 >= J0 && (a.do_ids || (a.src && (a.srcf[c] & 0xF)));
    const int rows = J1 - J0 + 1, cols = I1 - I0 + 1;
    const bool scan = labels && rows <= kMaxRows;

    if (tid < half || !scan) {  // forces: the first half, or all threads without a scan
        if (a.do_force) {
            float2* force = static_cast<float2*>(a.force);
            const float p = ppres;
            const float ten = (float)a.tension;
            const int stride = scan ? half : kIBThreads;
            for (int t = tid, r = 0; t < n; t += stride, ++r) {
                const int tp = (t == 0) ? n - 1 : t - 1;
                const int tn = (t == n - 1) ? 0 : t + 1;
                const int2 b = sb[t];
                const float2 f = sf[t];
                const float2 dn = edge_vec(b, f, sb[tn], sf[tn]);   // X_{t+1} - X_t
                const float2 dp = edge_vec(sb[tp], sf[tp], b, f);   // X_t - X_{t-1}
                // prefetched for the first two vertices of this thread
                const bool pre1 = r == 1 && stride == half;  // tid + half, prefetched
                const float L0t = r == 0 ? pL0[0] : (pre1 ? pL0[1] : (float)a.L0[v0 + t]);
                const float kt = r == 0 ? pk[0] : (pre1 ? pk[1] : (float)a.k[v0 + t]);
                const float L0p = r == 0 ? pL0p[0] : (pre1 ? pL0p[1] : (float)a.L0[v0 + tp]);
                const float kp = r == 0 ? pkp[0] : (pre1 ? pkp[1] : (float)a.k[v0 + tp]);
                const float2 s0 = spring32_force(dn, L0t, kt);
                const float2 s1 = spring32_force(dp, L0p, kp);
                float Fx = s0.x - s1.x, Fy = s0.y - s1.y;
                // pressure p dA/dX: (p/2)(y_{t+1} - y_{t-1}, x_{t-1} - x_{t+1})
                Fx += 0.5f * p * (dn.y + dp.y);
                Fy -= 0.5f * p * (dn.x + dp.x);
                if (ten != 0.f) {  // Eq. membraneforce
                    const float ln = sqrtf(dn.x * dn.x + dn.y * dn.y);
                    const float lp = sqrtf(dp.x * dp.x + dp.y * dp.y);
                    Fx += ten * (dn.x / ln - dp.x / lp);
                    Fy += ten * (dn.y / ln - dp.y / lp);
                }
                if (OPTS && a.jpartner) {  // Eq. celljunctionforce (a launch without the move)
                    const float2 J = junction_force32(a, sx[t], a.jpartner[v0 + t]);
                    Fx += J.x;
                    Fy += J.y;
                }
                if (a.write_vforce) a.vforce[v0 + t] = make_double2((double)Fx, (double)Fy);

                float wx[4], wy[4];
                weights_from_frac(f.x, wx);
                weights_from_frac(f.y, wy);
                int ix[4];
                ix[0] = wrapi(b.x - 1, a.nx);
#pragma unroll
                for (int i = 1; i < 4; ++i) ix[i] = (ix[i - 1] + 1 == a.nx) ? 0 : ix[i - 1] + 1;
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    int J = b.y - 1 + j;
                    if (a.bc_y) {
                        if (J < 0 || J >= a.ny) {
                            raise_flag(a.diag, kDiagWallStencil);
                            continue;
                        }
                    } else {
                        J = wrapi(J, a.ny);
                    }
                    float2* row = force + (int64_t)J * a.pitch;
                    float cx4[4], cy4[4];
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const float w = wx[i] * wy[j];
                        cx4[i] = Fx * w;
                        cy4[i] = Fy * w;
                    }
                    // the four nodes of the row: two 16-byte reductions when
                    // the row starts on an even node, 8 + 16 + 8 bytes when it
                    // starts on an odd one, one per node across the periodic seam
                    if (ix[3] == ix[0] + 3) {
                        float2* r0 = row + ix[0];
                        if ((ix[0] & 1) == 0) {
                            force_red2(a, r0, cx4[0], cy4[0], cx4[1], cy4[1]);
                            force_red2(a, r0 + 2, cx4[2], cy4[2], cx4[3], cy4[3]);
                        } else {
                            force_red1(a, r0, cx4[0], cy4[0]);
                            force_red2(a, r0 + 1, cx4[1], cy4[1], cx4[2], cy4[2]);
                            force_red1(a, r0 + 3, cx4[3], cy4[3]);
                        }
                    } else {
#pragma unroll
                        for (int i = 0; i < 4; ++i) spread_add(a, &row[ix[i]], cx4[i], cy4[i]);
                    }
                    if (MASK_TABLE)
                        mark_row_table(a, a.fmask, (int64_t)J * a.pitch, ix, S.mkey, S.mval);
                    else
                        mark_row(a, a.fmask, (int64_t)J * a.pitch, ix);
                }
            }
        }
    } else if (scan) {
        for (int e = tid - half; e < n; e += half) {
            const int eb = (e == n - 1) ? 0 : e + 1;
            const int2 ba = sb[e], bb = sb[eb];
            const float2 fa = sf[e], fb = sf[eb];
            const int cya = ba.y + (fa.y > 0.f ? 1 : 0), cyb = bb.y + (fb.y > 0.f ? 1 : 0);
            if (cya == cyb) continue;
            // rows J with (y_a <= J) != (y_b <= J): min(cy) <= J < max(cy)
            const int jl = min(cya, cyb), jh = max(cya, cyb) - 1;
            const float2 d = edge_vec(ba, fa, bb, fb);
            const float ratio = fabsf(d.x) / fabsf(d.y);
            for (int J = jl; J <= jh; ++J) {
                // x_c - base_a.x = frac_a.x + (J - y_a)(x_b - x_a)/(y_b - y_a)
                const float pr = (float)(J - ba.y) - fa.y;
                const float xr = fa.x + (pr * d.x) / d.y;
                const float E = 9.5367431640625e-07f * (4.f + 4.f * ratio + fabsf(d.x) + fabsf(xr));
                const float clo = ceilf(xr - E), chi = ceilf(xr + E);
                int ti;
                if (clo == chi) {
                    ti = ba.x + (int)clo;
                } else {
                    const double tc = ceil(crossing_x(sx[e], sx[eb], (double)J));
                    ti = tc < (double)I0 ? I0 : (tc > (double)(I1 + 1) ? I1 + 1 : (int)tc);
                }
                ti = ti < I0 ? I0 : (ti > I1 + 1 ? I1 + 1 : ti);
                const int slot = atomicAdd(&rowcnt[J - J0], 1);
                if (slot < kMaxCross)
                    thr[(J - J0) * kMaxCross + slot] = ti;
                else
                    s_flag = 1;
            }
        }
    }
    // every distinct force-mask word of the cell into the mask, once
    if (MASK_TABLE && a.do_force && a.fmask) {
        cell_sync<NT>(bar);
        for (int i = tid; i < kMaskTable; i += NT) {
            const uint32_t k = S.mkey[i];
            if (k != kMaskEmpty) atomicOr(a.fmask + k, S.mval[i]);
        }
    }
    if (!labels) return;  // uniform over the CTA
    cell_sync<NT>(bar);
    if (INLINE_FILL)
        fill_labels_body(a, c, n, sx, rowcnt, thr, scan && s_flag == 0, I0, J0, rows, cols, tid,
                         NT);
    else
        fill_labels_call(a, c, n, sx, rowcnt, thr, scan && s_flag == 0, I0, J0, rows, cols, tid,
                         NT);
}

}  // namespace lbib
