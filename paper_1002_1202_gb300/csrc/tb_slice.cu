// Column slices: whole outer steps of a few columns of a small system inside
// one thread-block cluster (sm_103a).
//
// The columns of a panel are independent of one another -- inner solve, outer
// recurrence, shifts, convergence and seed switching of a column never read
// another column -- so a slice of NC columns can run any number of outer steps
// with no grid-wide step at all.  On small systems that is what bounds the
// panel kernels: a Chebyshev step of 64-500 atoms took 15-20 us (a chain of 17
// dependent gathers in a few CTAs, ~60 launches per outer step), an FP64 CG
// iteration 50-70 us.
//
// Here a cluster of CL CTAs owns a slice.  The vector that the products gather
// (d_k of the Chebyshev step, the split u' of the double-float products, r of
// the FP64 CG) is kept whole in the shared memory of every CTA of the cluster;
// each CTA computes its share of the rows and stores the new rows into all CL
// copies (distributed shared memory), one cluster barrier per step.  Rows of S
// and H are read from L1 / L2 in the order the warp consumes them.
//
// Layout of a system's rows (SliceDev, built once per handle).  Orbitals are
// taken in groups of four rows: an sp atom, or four s atoms with much the same
// neighbours.  An item of a group is one column of S that meets it: the
// column's row index x and the four coefficients.  The items with x % 4 == a go
// to stream a of the group, so the four lanes of a group always read four
// different bank groups of the gathered vector, whatever its columns are; two
// groups (eight streams) form an octet, whose items are interleaved step by
// step: one step of an octet is one 128-byte line of coefficients.  Stream a's
// lane ends with row a of the group by a reduce-scatter over the four streams.
// Item 0 of every stream is the column of the group's own row a (the diagonal).
#include "tb_internal.h"
#include "tb_device.cuh"

#include <cooperative_groups.h>

#include <algorithm>
#include <cstdlib>
#include <mutex>
#include <vector>

namespace cg = cooperative_groups;

namespace tb {

namespace {

constexpr int SL_T = 512;    // threads per CTA, at most
constexpr int SL_CL = 8;     // CTAs per cluster, at most
constexpr int SL_SPARE = 2;  // refinement rounds beyond the planned ones (residual with FP64 products)

template <int NC>
struct SliceShared {
    double red[2][SL_CL][2 * NC];          // reductions: per-CTA sums, two buffers
    unsigned long long best[SL_CL][NC];    // largest residual among a CTA's shifts (bits)
    int bestk[SL_CL][NC];                  // and the lowest shift that has it
    int nun[SL_CL][NC];                    // unconverged shifts of a CTA's share
    ColState cs[NC];
    double scale[NC], unscale[NC], b2[NC], tsum[NC];
    double alpha[NC], beta[NC], gprev[NC];
    double nu[NC], inv_nu[NC], Bn[NC], rhat[NC];
    unsigned long long lbest[NC];
    int lbestk[NC], lnun[NC];
    int skip[NC], want[NC];
    int open, bad, wanted, active;
};

// double-float sum of two partial sums
__device__ __forceinline__ void df_add2(float2& hi, float2& lo, float2 h, float2 l) {
    const float2 t = __fadd2_rn(hi, h);
    const float2 bp = __fadd2_rn(t, neg2(hi));
    const float2 err = __fadd2_rn(__fadd2_rn(hi, neg2(__fadd2_rn(t, neg2(bp)))), __fadd2_rn(h, neg2(bp)));
    hi = t;
    lo = __fadd2_rn(lo, __fadd2_rn(l, err));
}

__device__ __forceinline__ float2 shfl2(float2 v, int d) {
    return make_float2(__shfl_xor_sync(0xffffffffu, v.x, d), __shfl_xor_sync(0xffffffffu, v.y, d));
}

// CPL columns of one orbital row, as a lane holds them
template <int CPL>
struct Cols {
    double v[CPL];
};
template <int CPL>
__device__ __forceinline__ Cols<CPL> ldcols(const double* p) {
    Cols<CPL> r;
    if (CPL == 2) {
        const double2 q = *reinterpret_cast<const double2*>(p);
        r.v[0] = q.x;
        r.v[CPL - 1] = q.y;
    } else {
        r.v[0] = *p;
    }
    return r;
}
template <int CPL>
__device__ __forceinline__ void stcols(double* p, const Cols<CPL>& r) {
    if (CPL == 2) *reinterpret_cast<double2*>(p) = make_double2(r.v[0], r.v[CPL - 1]);
    else *p = r.v[0];
}

// One lane's element: a row (of the slice order) and its CPL columns.
struct Elem {
    bool on;      // a lane of the CTA's share
    int oct, s8;  // octet and stream
    int row, q;   // slice row, lane within the row
    int slot;     // padded orbital slot (-1: a filling row, always zero)
};

template <bool MIXED, int NC>
struct Slice {
    static constexpr int CPL = MIXED ? 2 : 1;   // columns per lane
    static constexpr int LPS = NC / CPL;        // lanes per row
    using Sh = SliceShared<NC>;
    const SliceDev& ss;
    const DevSystem& s;
    const PanelDev& p;
    const SliceArgs& a;
    Sh& sh;
    double* part;     // [2 * CPL][T] reduction scratch (full mode: coefficients)
    double* dfun;     // [NC][M]
    float* omega;
    unsigned char* vec;   // the gathered vector(s), the same in every CTA
    unsigned char* own;   // per-element values of this CTA
    int CL, rank, c0, tid, T, nel, nel_pad, par;

    __device__ Slice(const SliceDev& ss_, const DevSystem& s_, const PanelDev& p_, const SliceArgs& a_, Sh& sh_)
        : ss(ss_), s(s_), p(p_), a(a_), sh(sh_) {}

    __device__ void barrier() {
        if (CL == 1) __syncthreads();
        else cg::this_cluster().sync();
    }
    // v into the same place of every CTA's copy
    template <class V>
    __device__ __forceinline__ void bcast(V* dst, V v) {
        if (CL == 1) {
            *dst = v;
        } else {
            for (int r = 0; r < CL; ++r) *cg::this_cluster().map_shared_rank(dst, r) = v;
        }
    }
    __device__ __forceinline__ Elem elem(int e0) const {
        Elem e;
        const int el = e0 + tid;
        e.on = el < nel;
        const int lr = el / LPS;
        e.q = el % LPS;
        e.s8 = lr & 7;
        e.oct = (lr >> 3) * CL + rank;
        e.row = e.oct * 8 + e.s8;
        e.slot = e.on ? __ldg(ss.row_slot + e.row) : -1;
        return e;
    }
    __device__ __forceinline__ double* at(double2* base, const Elem& e) const {
        return reinterpret_cast<double*>(base) + (size_t)e.slot * p.P + c0 + e.q * CPL;
    }

    // Sums over all rows of the slice of NQ values per column; out[qn] valid
    // in threads tid < NC (column tid) of every CTA, the same in all of them.
    // Fixed order: threads' values, warps' trees, ranks.
    template <int NQ>
    __device__ void sum(const double (&v)[NQ][CPL], double (&out)[NQ]) {
#pragma unroll
        for (int n = 0; n < NQ; ++n)
#pragma unroll
            for (int j = 0; j < CPL; ++j) part[(n * CPL + j) * T + tid] = v[n][j];
        __syncthreads();
        const int lane = tid & 31, nw = T >> 5;
        for (int val = tid >> 5; val < NQ * NC; val += nw) {
            const int n = val / NC, c = val % NC, q = c / CPL, j = c % CPL;
            const double* src = part + (n * CPL + j) * T + q;
            double acc = 0.0;
            for (int i = lane; i < T / LPS; i += 32) acc += src[i * LPS];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
            if (lane == 0) bcast(&sh.red[par][rank][val], acc);
        }
        barrier();
        if (tid < NC) {
#pragma unroll
            for (int n = 0; n < NQ; ++n) {
                double acc = 0.0;
                for (int r = 0; r < CL; ++r) acc += sh.red[par][r][n * NC + tid];
                out[n] = acc;
            }
        }
        par ^= 1;
    }

    // ---- products ----------------------------------------------------------
    // item loop of one stream: f(item offset, row of the gathered vector)
    template <class F>
    __device__ __forceinline__ void items(const Elem& e, bool diag, F&& f) const {
        const int i0 = __ldg(ss.oct_ptr + e.oct), n = __ldg(ss.oct_ptr + e.oct + 1) - i0;
        const int base = i0 * 8 + e.s8;
        if (diag) f(base, e.row);
        const ushort4* ix = ss.idx + (size_t)__ldg(ss.idx_ptr + e.oct) * 8 + e.s8;
        int k = 1;
#pragma unroll 2
        for (; k + 4 <= n; k += 4, ix += 8) {
            const ushort4 id = __ldg(ix);
            const int b = base + 8 * k;
            f(b, id.x);
            f(b + 8, id.y);
            f(b + 16, id.z);
            f(b + 24, id.w);
        }
        if (k < n) {
            const ushort4 id = __ldg(ix);
            const int b = base + 8 * k;
            f(b, id.x);
            if (k + 1 < n) f(b + 8, id.y);
            if (k + 2 < n) f(b + 16, id.z);
        }
    }
    // the four streams' partial sums of rows 0..3 -> row (stream) of each lane
    __device__ __forceinline__ static float2 scatter4(const float2 (&acc)[4], int st) {
        const bool up = st & 2, odd = st & 1;
        float2 k0 = up ? acc[2] : acc[0], k1 = up ? acc[3] : acc[1];
        const float2 s0 = shfl2(up ? acc[0] : acc[2], 2 * LPS), s1 = shfl2(up ? acc[1] : acc[3], 2 * LPS);
        k0 = __fadd2_rn(k0, s0);
        k1 = __fadd2_rn(k1, s1);
        const float2 t = shfl2(odd ? k0 : k1, LPS);
        return __fadd2_rn(odd ? k1 : k0, t);
    }
    __device__ __forceinline__ float2 spmv32(const Elem& e, const float2* cur, bool diag) const {
        float2 acc[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) acc[i] = make_float2(0.f, 0.f);
        if (e.on) {
            const float2* xq = cur + e.q;
            items(e, diag, [&](int it, int x) {
                const float4 c = __ldg(ss.Shi + it);
                const float2 v = xq[x * LPS];
                acc[0] = __ffma2_rn(make_float2(c.x, c.x), v, acc[0]);
                acc[1] = __ffma2_rn(make_float2(c.y, c.y), v, acc[1]);
                acc[2] = __ffma2_rn(make_float2(c.z, c.z), v, acc[2]);
                acc[3] = __ffma2_rn(make_float2(c.w, c.w), v, acc[3]);
            });
        }
        __syncwarp();
        return scatter4(acc, e.s8 & 3);
    }
    // double-float product with (Mh, Ml) of the split vector (xh, xl)
    __device__ __forceinline__ double2 spmv_df(const Elem& e, const float4* Mh, const float4* Ml, const float2* xh,
                                               const float2* xl) const {
        float2 hi[4], lo[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) hi[i] = lo[i] = make_float2(0.f, 0.f);
        if (e.on) {
            items(e, true, [&](int it, int x) {
                const float4 ch = __ldg(Mh + it), cl = __ldg(Ml + it);
                const float2 vh = xh[x * LPS + e.q], vl = xl[x * LPS + e.q];
                df_mac2(hi[0], lo[0], ch.x, cl.x, vh, vl);
                df_mac2(hi[1], lo[1], ch.y, cl.y, vh, vl);
                df_mac2(hi[2], lo[2], ch.z, cl.z, vh, vl);
                df_mac2(hi[3], lo[3], ch.w, cl.w, vh, vl);
            });
        }
        __syncwarp();
        const int st = e.s8 & 3;
        const bool up = st & 2, odd = st & 1;
        float2 h0 = up ? hi[2] : hi[0], l0 = up ? lo[2] : lo[0], h1 = up ? hi[3] : hi[1], l1 = up ? lo[3] : lo[1];
        const float2 a0 = shfl2(up ? hi[0] : hi[2], 2 * LPS), b0 = shfl2(up ? lo[0] : lo[2], 2 * LPS);
        const float2 a1 = shfl2(up ? hi[1] : hi[3], 2 * LPS), b1 = shfl2(up ? lo[1] : lo[3], 2 * LPS);
        df_add2(h0, l0, a0, b0);
        df_add2(h1, l1, a1, b1);
        const float2 at_ = shfl2(odd ? h0 : h1, LPS), bt = shfl2(odd ? l0 : l1, LPS);
        float2 h = odd ? h1 : h0, l = odd ? l1 : l0;
        df_add2(h, l, at_, bt);
        return make_double2((double)h.x + (double)l.x, (double)h.y + (double)l.y);
    }
    __device__ __forceinline__ Cols<CPL> spmv64(const Elem& e, const double2* M, const double* x_) const {
        double acc[4][CPL];
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < CPL; ++j) acc[i][j] = 0.0;
        if (e.on) {
            const double* xq = x_ + e.q * CPL;
            items(e, true, [&](int it, int x) {
                const double2 c01 = __ldg(M + 2 * (size_t)it), c23 = __ldg(M + 2 * (size_t)it + 1);
                const Cols<CPL> v = ldcols<CPL>(xq + x * NC);
#pragma unroll
                for (int j = 0; j < CPL; ++j) {
                    acc[0][j] += c01.x * v.v[j];
                    acc[1][j] += c01.y * v.v[j];
                    acc[2][j] += c23.x * v.v[j];
                    acc[3][j] += c23.y * v.v[j];
                }
            });
        }
        __syncwarp();
        const int st = e.s8 & 3;
        const bool up = st & 2, odd = st & 1;
        Cols<CPL> r;
#pragma unroll
        for (int j = 0; j < CPL; ++j) {
            double k0 = up ? acc[2][j] : acc[0][j], k1 = up ? acc[3][j] : acc[1][j];
            k0 += __shfl_xor_sync(0xffffffffu, up ? acc[0][j] : acc[2][j], 2 * LPS);
            k1 += __shfl_xor_sync(0xffffffffu, up ? acc[1][j] : acc[3][j], 2 * LPS);
            const double t = __shfl_xor_sync(0xffffffffu, odd ? k0 : k1, LPS);
            r.v[j] = (odd ? k1 : k0) + t;
        }
        return r;
    }

    // ---- the current u' as the products of the outer step take it ------------
    // mixed: split into vec[0] (hi) and vec[1] (lo); FP64: as it is
    __device__ void publish_x() {
        for (int e0 = 0; e0 < nel_pad; e0 += T) {
            const Elem e = elem(e0);
            if (!e.on) continue;
            Cols<CPL> x{};
            if (e.slot >= 0) x = ldcols<CPL>(at(p.Rp, e));
            if (MIXED) {
                const float4 f = df_split(make_double2(x.v[0], x.v[CPL - 1]));
                float2* xa = reinterpret_cast<float2*>(vec);
                float2* xb = xa + (size_t)ss.nrows * LPS;
                bcast(xa + (size_t)e.row * LPS + e.q, make_float2(f.x, f.y));
                bcast(xb + (size_t)e.row * LPS + e.q, make_float2(f.z, f.w));
            } else {
                bcast(reinterpret_cast<double*>(vec) + (size_t)e.row * NC + e.q, x.v[0]);
            }
        }
    }

    // column threads: right-hand side norm of the next inner solve
    __device__ void set_rhs(double b2) {
        ColState& c = sh.cs[tid];
        if (c.active) c.rnorm = sqrt(b2);
        sh.b2[tid] = b2;
        sh.skip[tid] = (!c.active || b2 == 0.0) ? 1 : 0;
        sh.unscale[tid] = sh.skip[tid] ? 0.0 : sqrt(b2);
        sh.scale[tid] = sh.skip[tid] ? 0.0 : 1.0 / sh.unscale[tid];
    }

    // ---- inner solve S u' = u, mixed: FP32 Chebyshev corrections inside FP64
    // refinement, as mixed_inner of the panel path (same scaling, plan and
    // convergence test).  Leaves u' in Rp and published, its residual in Rin,
    // t = u^T u' in tsum.  False: not converged (the caller falls back).
    __device__ bool inner_mixed(int& steps) {
        float2* xa = reinterpret_cast<float2*>(vec);
        float2* xb = xa + (size_t)ss.nrows * LPS;
        float2* fb = reinterpret_cast<float2*>(own);
        const bool skip_diag = ss.unit_diag != 0;
        for (int round = 0;; ++round) {
            const int n = round >= a.R - 1 ? a.n_last : a.n;
            steps += n;
            const bool fp64 = round >= a.R;
            for (int e0 = 0; e0 < nel_pad; e0 += T) {
                const Elem e = elem(e0);
                if (!e.on) continue;
                float2 f = make_float2(0.f, 0.f);
                if (e.slot >= 0) {
                    const Cols<CPL> v = ldcols<CPL>(at(round == 0 ? p.Rcur : p.Rin, e));
                    f = make_float2((float)(v.v[0] * sh.scale[2 * e.q]), (float)(v.v[CPL - 1] * sh.scale[2 * e.q + 1]));
                }
                fb[e0 + tid] = f;
                const float2 d1 = make_float2(a.gamma * f.x, a.gamma * f.y);
                bcast(xa + (size_t)e.row * LPS + e.q, d1);
                if (n == 1 && e.slot >= 0) add_correction(e, d1, round);
            }
            barrier();
            for (int k = 1; k < n; ++k) {
                const float2* cur = (k & 1) ? xa : xb;
                float2* io = (k & 1) ? xb : xa;
                const float om = omega[k];
                for (int e0 = 0; e0 < nel_pad; e0 += T) {
                    if (e0 + (tid & ~31) >= nel_pad) break;
                    const Elem e = elem(e0);
                    float2 y = spmv32(e, cur, !skip_diag);
                    if (!e.on) continue;
                    const size_t w = (size_t)e.row * LPS + e.q;
                    const float2 dc = cur[w], f = fb[e0 + tid];
                    const float2 dp = k == 1 ? make_float2(0.f, 0.f) : io[w];
                    if (skip_diag) {
                        y.x += dc.x;
                        y.y += dc.y;
                    }
                    float2 dn = make_float2(dp.x + om * (a.gamma * (f.x - y.x) + dc.x - dp.x),
                                            dp.y + om * (a.gamma * (f.y - y.y) + dc.y - dp.y));
                    if (e.slot < 0) dn = make_float2(0.f, 0.f);
                    if (k == n - 1) {
                        if (e.slot >= 0) add_correction(e, dn, round);
                    } else {
                        bcast(io + w, dn);
                    }
                }
                barrier();
            }
            double v[2][CPL] = {};
            if (!fp64) {
                publish_x();
                barrier();
                for (int e0 = 0; e0 < nel_pad; e0 += T) {
                    if (e0 + (tid & ~31) >= nel_pad) break;
                    const Elem e = elem(e0);
                    const double2 y = spmv_df(e, ss.Shi, ss.Slo, xa, xb);
                    if (e.slot >= 0) residual(e, y.x, y.y, v);
                }
            } else {
                double* xd = reinterpret_cast<double*>(vec);
                for (int e0 = 0; e0 < nel_pad; e0 += T) {
                    const Elem e = elem(e0);
                    if (!e.on) continue;
                    Cols<CPL> x{};
                    if (e.slot >= 0) x = ldcols<CPL>(at(p.Rp, e));
                    bcast(reinterpret_cast<double2*>(xd + (size_t)e.row * NC + 2 * e.q), make_double2(x.v[0], x.v[CPL - 1]));
                }
                barrier();
                for (int e0 = 0; e0 < nel_pad; e0 += T) {
                    if (e0 + (tid & ~31) >= nel_pad) break;
                    const Elem e = elem(e0);
                    const Cols<CPL> y = spmv64(e, ss.S64, xd);
                    if (e.slot >= 0) residual(e, y.v[0], y.v[CPL - 1], v);
                }
            }
            double out[2];
            sum<2>(v, out);
            if (tid == 0) sh.open = sh.bad = 0;
            __syncthreads();
            if (tid < NC) {
                sh.tsum[tid] = out[1];
                if (!sh.skip[tid]) {
                    const double r2 = out[0];
                    if (!isfinite(r2)) {
                        atomicExch(&sh.bad, 1);
                    } else {
                        if (r2 <= a.inner_tol * a.inner_tol * sh.b2[tid] || r2 == 0.0) sh.skip[tid] = 1;
                        sh.unscale[tid] = sh.skip[tid] ? 0.0 : sqrt(r2);
                        sh.scale[tid] = sh.skip[tid] ? 0.0 : 1.0 / sh.unscale[tid];
                    }
                }
                if (!sh.skip[tid]) atomicAdd(&sh.open, 1);
            }
            __syncthreads();
            if (sh.bad) return false;
            if (sh.open == 0) {
                if (fp64) {
                    publish_x();
                    barrier();
                }
                return true;
            }
            if (round + 1 >= a.R + SL_SPARE) return false;
        }
    }
    // u' += d * ||res|| (a non-finite correction is dropped, as in k_refine_add)
    __device__ __forceinline__ void add_correction(const Elem& e, float2 d, int round) {
        Cols<CPL> x{};
        double* px = at(p.Rp, e);
        if (round > 0) x = ldcols<CPL>(px);
        if (isfinite(d.x)) x.v[0] += (double)d.x * sh.unscale[2 * e.q];
        if (isfinite(d.y)) x.v[CPL - 1] += (double)d.y * sh.unscale[2 * e.q + 1];
        stcols<CPL>(px, x);
    }
    __device__ __forceinline__ void residual(const Elem& e, double y0, double y1, double (&v)[2][CPL]) {
        const Cols<CPL> u = ldcols<CPL>(at(p.Rcur, e)), x = ldcols<CPL>(at(p.Rp, e));
        Cols<CPL> r;
        r.v[0] = u.v[0] - y0;
        if (CPL == 2) r.v[CPL - 1] = u.v[CPL - 1] - y1;
        stcols<CPL>(at(p.Rin, e), r);
#pragma unroll
        for (int j = 0; j < CPL; ++j) {
            v[0][j] += r.v[j] * r.v[j];
            v[1][j] += u.v[j] * x.v[j];
        }
    }

    // ---- inner solve in FP64: Chronopoulos-Gear CG, as k_inner_spmv and
    // k_inner_update (one column per lane)
    __device__ bool inner_fp64(int& steps) {
        double* rv = reinterpret_cast<double*>(vec);
        double* pv = reinterpret_cast<double*>(own);
        double* sv = pv + nel_pad;
        double* xv = sv + nel_pad;
        double* wv = xv + nel_pad;
        for (int e0 = 0; e0 < nel_pad; e0 += T) {
            const Elem e = elem(e0);
            if (!e.on) continue;
            bcast(rv + (size_t)e.row * NC + e.q, e.slot >= 0 ? *at(p.Rcur, e) : 0.0);
            pv[e0 + tid] = sv[e0 + tid] = xv[e0 + tid] = 0.0;
        }
        barrier();
        int it = 0;
        for (;; ++it) {
            double v[2][CPL] = {};
            for (int e0 = 0; e0 < nel_pad; e0 += T) {
                if (e0 + (tid & ~31) >= nel_pad) break;
                const Elem e = elem(e0);
                const Cols<CPL> w = spmv64(e, ss.S64, rv);
                if (!e.on) continue;
                const double r = rv[(size_t)e.row * NC + e.q];
                wv[e0 + tid] = w.v[0];
                if (e.slot >= 0) {
                    v[0][0] += r * r;
                    v[1][0] += w.v[0] * r;
                }
            }
            double out[2];
            sum<2>(v, out);
            if (tid == 0) sh.open = sh.bad = 0;
            __syncthreads();
            if (tid < NC) {
                const double gam = out[0], del = out[1];
                if (!sh.skip[tid]) {
                    if (gam <= a.inner_tol * a.inner_tol * sh.b2[tid]) {
                        sh.skip[tid] = 1;
                    } else {
                        const double beta = it == 0 ? 0.0 : gam / sh.gprev[tid];
                        const double den = del - (it == 0 ? 0.0 : beta * gam / sh.alpha[tid]);
                        if (!(den > 0.0)) {
                            atomicExch(&sh.bad, 1);
                        } else {
                            sh.alpha[tid] = gam / den;
                            sh.beta[tid] = beta;
                            sh.gprev[tid] = gam;
                            atomicAdd(&sh.open, 1);
                        }
                    }
                }
            }
            __syncthreads();
            if (sh.bad) return false;
            if (sh.open == 0) break;
            if (it + 1 >= a.inner_max) return false;
            for (int e0 = 0; e0 < nel_pad; e0 += T) {
                const Elem e = elem(e0);
                if (!e.on || sh.skip[e.q]) continue;
                const int i = e0 + tid;
                const double al = sh.alpha[e.q], be = sh.beta[e.q];
                const size_t w = (size_t)e.row * NC + e.q;
                const double r = rv[w];
                const double pn = r + be * pv[i], sn = wv[i] + be * sv[i];
                pv[i] = pn;
                sv[i] = sn;
                xv[i] += al * pn;
                bcast(rv + w, r - al * sn);
            }
            barrier();
        }
        steps += it;
        double v[1][CPL] = {};
        for (int e0 = 0; e0 < nel_pad; e0 += T) {
            const Elem e = elem(e0);
            if (!e.on) continue;
            const size_t w = (size_t)e.row * NC + e.q;
            const double x = xv[e0 + tid];
            if (e.slot >= 0) {
                *at(p.Rin, e) = rv[w];
                *at(p.Rp, e) = x;
                v[0][0] += *at(p.Rcur, e) * x;
            }
            bcast(rv + w, x);   // the products of the outer step gather u'
        }
        double out[1];
        sum<1>(v, out);
        if (tid < NC) sh.tsum[tid] = out[0];
        __syncthreads();
        return true;
    }
    __device__ bool inner(int& steps) {
        if (MIXED) return inner_mixed(steps);
        return inner_fp64(steps);
    }

    // ---- functionals of u' (written by every CTA of the cluster: read at L2)
    __device__ void functionals() {
        const double* Rp = reinterpret_cast<const double*>(p.Rp);
        if (p.proj == PROJ_ROWS) {
            for (int i = tid; i < NC * p.M; i += T) {
                const int c = i / p.M, m = i % p.M;
                if (m < sh.cs[c].nfun) dfun[i] = __ldcg(Rp + (size_t)p.frow[(size_t)(c0 + c) * p.M + m] * p.P + c0 + c);
            }
        } else if (p.proj == PROJ_SROW) {
            const int lane = tid & 31;
            for (int c = tid >> 5; c < NC; c += T >> 5) {
                double acc = 0.0;
                if (sh.cs[c].row >= 0) {
                    const int row = sh.cs[c].row, I = row >> 2, ra = row & 3;
                    const int b0 = s.brow[I], nbl = s.brow[I + 1] - b0;
                    for (int i = lane; i < 4 * nbl; i += 32) {
                        const int b = b0 + i / 4, be = i % 4;
                        acc += s.S[16 * (size_t)b + 4 * ra + be] *
                               __ldcg(Rp + (size_t)(4 * s.bcol[b] + be) * p.P + c0 + c);
                    }
                }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
                if (lane == 0) dfun[c] = acc;
            }
        }
    }

    __device__ void krange(int& k0, int& kl) const {
        const int per = (p.K + CL - 1) / CL;
        k0 = min(p.K, rank * per);
        kl = min(p.K, k0 + per) - k0;
    }

    // ---- shift state of u'_0 (k_shift_init, k_full_init)
    __device__ void shift_init() {
        if (tid < NC) {
            ColState& c = sh.cs[tid];
            const double nu = sqrt(sh.tsum[tid]);
            c.t = c.t_new = sh.tsum[tid];
            c.nu = nu;
            c.inv_nu = nu > 0.0 ? 1.0 / nu : 0.0;
            c.n_unconv = p.K;
        }
        functionals();
        __syncthreads();
        int k0, kl;
        krange(k0, kl);
        for (int i = tid; i < NC * kl; i += T) {
            const int c = i / kl, k = k0 + i % kl;
            if (!sh.cs[c].active) continue;
            const size_t o = (size_t)(c0 + c) * p.K + k;
            p.zeta[o] = cmk(sh.cs[c].nu, 0.0);
            p.pinv[o] = cmk(0.0, 0.0);
            p.conv_iter[o] = -1;
            if (p.deriv) p.dzeta[o] = p.dpinv[o] = cmk(0.0, 0.0);
        }
        if (p.proj != PROJ_NONE) {
            for (int i = tid; i < NC * kl * p.M; i += T) {
                const int c = i / (kl * p.M), k = k0 + (i / p.M) % kl, m = i % p.M;
                if (!sh.cs[c].active || m >= sh.cs[c].nfun) continue;
                const size_t o = ((size_t)(c0 + c) * p.K + k) * p.M + m;
                p.t[o] = cmk(0.0, 0.0);
                p.u[o] = cmk(dfun[c * p.M + m] * sh.cs[c].inv_nu, 0.0);
                if (p.deriv) p.dt[o] = p.du[o] = cmk(0.0, 0.0);
            }
        } else {
            for (int e0 = 0; e0 < nel_pad; e0 += T) {
                const Elem e = elem(e0);
                if (e.slot < 0) continue;
                const Cols<CPL> x = ldcols<CPL>(at(p.Rp, e));
                for (int k = 0; k < p.K; ++k) {
                    const size_t o = ((size_t)k * p.npad + e.slot) * p.P + c0 + e.q * CPL;
#pragma unroll
                    for (int j = 0; j < CPL; ++j) {
                        p.X[o + j] = cmk(0.0, 0.0);
                        p.Pk[o + j] = cmk(x.v[j] * sh.cs[e.q * CPL + j].inv_nu, 0.0);
                    }
                }
            }
        }
        barrier();   // the shifts' state is read by other CTAs (seed), and written again by its own
    }

    // ---- a5 + a6 for the slice's columns (k_shift_step, k_full_update); the
    // shifts of every column are split over the CTAs of the cluster
    __device__ void shift_step() {
        if (tid < NC) {
            const ColState& c = sh.cs[tid];
            const double tn = sh.tsum[tid];
            const double nu = sqrt(tn);
            sh.nu[tid] = nu;
            sh.inv_nu[tid] = nu > 0.0 ? 1.0 / nu : 0.0;
            sh.Bn[tid] = c.s * nu;
            sh.rhat[tid] = nu > 0.0 ? c.rnorm * sh.inv_nu[tid] : 0.0;
            sh.lnun[tid] = 0;
            sh.lbest[tid] = 0ull;
            sh.lbestk[tid] = p.K;
        }
        functionals();
        __syncthreads();
        int k0, kl;
        krange(k0, kl);
        const bool inl = p.proj != PROJ_NONE && p.M == 1 && !p.deriv;
        for (int i = tid; i < NC * kl; i += T) {
            const int c = i / kl, k = k0 + i % kl;
            const ColState& cs = sh.cs[c];
            const size_t o = (size_t)(c0 + c) * p.K + k;
            if (!cs.active || p.conv_iter[o] >= 0) {
                if (!inl) p.ak[o] = cmk(0.0, 0.0);
                continue;
            }
            const double2 pinv = p.pinv[o], zeta = p.zeta[o];
            const ShiftCoef f = shift_coef(p.z[k], cs.sigma, cs.asig, cs.B, sh.Bn[c], pinv, zeta);
            const double res = sqrt(f.zeta.x * f.zeta.x + f.zeta.y * f.zeta.y) * sh.rhat[c];
            p.pinv[o] = f.inv;
            p.zeta[o] = f.zeta;
            if (p.deriv) {
                const double2 dp = p.dpinv[o], dz = p.dzeta[o];
                const double B2 = cs.B * cs.B;
                const double2 dD = cmk(1.0 - B2 * dp.x, -B2 * dp.y);
                const double2 i2 = cmul(f.inv, f.inv), id = cmul(i2, dD);
                const double2 dinv = cmk(-id.x, -id.y);
                const double2 dal = cadd(cmul(zeta, dinv), cmul(dz, f.inv));
                a.dak[o] = dal;
                a.dbk[o] = cmk(sh.Bn[c] * dinv.x, sh.Bn[c] * dinv.y);
                p.dpinv[o] = dinv;
                p.dzeta[o] = cmk(sh.Bn[c] * dal.x, sh.Bn[c] * dal.y);
            }
            if (inl) {
                const double2 u = p.u[o], un = cmul(f.l, u);
                p.t[o] = cadd(p.t[o], cmul(f.al, u));
                p.u[o] = cmk(dfun[c] * sh.inv_nu[c] + un.x, un.y);
            } else {
                p.ak[o] = f.al;
                p.bk[o] = f.l;
            }
            if (res <= p.tol) p.conv_iter[o] = cs.iters + 1;
            else atomicAdd(&sh.lnun[c], 1);
        }
        __syncthreads();
        if (p.proj != PROJ_NONE && !inl) {
            const int M = p.M;
            for (int i = tid; i < NC * kl * M; i += T) {
                const int c = i / (kl * M), k = k0 + (i / M) % kl, m = i % M;
                const ColState& cs = sh.cs[c];
                if (!cs.active || m >= cs.nfun) continue;
                const size_t ok = (size_t)(c0 + c) * p.K + k, o = ok * M + m;
                const double2 al = p.ak[ok];
                if (al.x == 0.0 && al.y == 0.0) continue;
                const double2 l = p.bk[ok], u = p.u[o], un = cmul(l, u);
                if (p.deriv) {
                    const double2 du = p.du[o];
                    p.dt[o] = cadd(p.dt[o], cadd(cmul(a.dak[ok], u), cmul(al, du)));
                    p.du[o] = cadd(cmul(a.dbk[ok], u), cmul(l, du));
                }
                p.t[o] = cadd(p.t[o], cmul(al, u));
                p.u[o] = cmk(dfun[c * M + m] * sh.inv_nu[c] + un.x, un.y);
            }
        }
        if (tid < NC) bcast(&sh.nun[rank][tid], sh.lnun[tid]);
        if (tid == 0) sh.wanted = sh.active = 0;
        barrier();
        // which columns switch their seed (decided alike in every CTA)
        if (tid < NC) {
            const ColState& c = sh.cs[tid];
            int n = 0;
            for (int r = 0; r < CL; ++r) n += sh.nun[r][tid];
            sh.want[tid] = 0;
            if (c.active) {
                sh.lnun[tid] = n;
                const bool forced = p.force_switch_every > 0 && (c.iters + 1) % p.force_switch_every == 0;
                if (n > 0 && p.switching &&
                    (forced || __ldcg(p.conv_iter + (size_t)(c0 + tid) * p.K + c.seed) >= 0)) {
                    sh.want[tid] = 1;
                    sh.wanted = 1;
                }
            }
        }
        __syncthreads();
        if (sh.wanted) {
            // the unconverged shift of the largest residual, ties to the lowest
            for (int pass = 0; pass < 2; ++pass) {
                for (int i = tid; i < NC * kl; i += T) {
                    const int c = i / kl, k = k0 + i % kl;
                    if (!sh.want[c]) continue;
                    const size_t o = (size_t)(c0 + c) * p.K + k;
                    if (p.conv_iter[o] >= 0) continue;
                    const double2 z = p.zeta[o];
                    const double res = sqrt(z.x * z.x + z.y * z.y) * sh.rhat[c];
                    if (!(res >= 0.0)) continue;
                    const unsigned long long bits = (unsigned long long)__double_as_longlong(res);
                    if (pass == 0) atomicMax(&sh.lbest[c], bits);
                    else if (bits == sh.lbest[c]) atomicMin(&sh.lbestk[c], k);
                }
                __syncthreads();
            }
            if (tid < NC) {
                bcast(&sh.best[rank][tid], sh.lbest[tid]);
                bcast(&sh.bestk[rank][tid], sh.lbestk[tid]);
            }
            barrier();
        }
        if (tid < NC && sh.cs[tid].active) {
            ColState& c = sh.cs[tid];
            c.iters += 1;
            c.n_unconv = sh.lnun[tid];
            if (c.n_unconv == 0) c.active = 0;
            c.t = c.t_new = sh.tsum[tid];
            c.nu_prev = c.nu;
            c.nu = sh.nu[tid];
            c.inv_nu = sh.inv_nu[tid];
            c.B = sh.Bn[tid];
            if (sh.want[tid]) {
                unsigned long long bb = 0ull;
                int bk = p.K;
                for (int r = 0; r < CL; ++r)
                    if (sh.bestk[r][tid] < p.K && (bk == p.K || sh.best[r][tid] > bb)) {
                        bb = sh.best[r][tid];
                        bk = sh.bestk[r][tid];
                    }
                if (bk < p.K && bk != c.seed) {
                    c.seed = bk;
                    c.sigma = p.z[bk].x;
                    c.switches += 1;
                }
            }
            c.sinv = __ldcg(p.pinv + (size_t)(c0 + tid) * p.K + c.seed);
            if (c.active) atomicAdd(&sh.active, 1);
        }
        __syncthreads();
        if (p.proj == PROJ_NONE) full_update();
    }

    // x^k += alpha^k q^k, q^k = u'_{n+1} / nu_{n+1} + l^k q^k on the own rows;
    // the coefficients, written by every CTA, staged in chunks of shifts
    __device__ void full_update() {
        double2* co = reinterpret_cast<double2*>(part);     // [KC][NC][2]
        const int KC = (2 * CPL * T / 2) / (2 * NC);
        for (int kb = 0; kb < p.K; kb += KC) {
            const int kn = min(KC, p.K - kb);
            __syncthreads();
            for (int i = tid; i < kn * NC; i += T) {
                const int c = i % NC, k = kb + i / NC;
                const size_t o = (size_t)(c0 + c) * p.K + k;
                co[2 * i] = __ldcg(p.ak + o);
                co[2 * i + 1] = __ldcg(p.bk + o);
            }
            __syncthreads();
            for (int e0 = 0; e0 < nel_pad; e0 += T) {
                const Elem e = elem(e0);
                if (e.slot < 0) continue;
                const Cols<CPL> x = ldcols<CPL>(at(p.Rp, e));
#pragma unroll
                for (int j = 0; j < CPL; ++j) {
                    const int c = e.q * CPL + j;
                    const double xn = x.v[j] * sh.cs[c].inv_nu;
                    const size_t o0 = (size_t)e.slot * p.P + c0 + c, st = (size_t)p.npad * p.P;
#pragma unroll 4
                    for (int k = 0; k < kn; ++k) {
                        const double2 al = co[2 * (k * NC + c)];
                        if (al.x == 0.0 && al.y == 0.0) continue;
                        const double2 l = co[2 * (k * NC + c) + 1];
                        const size_t o = o0 + (size_t)(kb + k) * st;
                        const double2 q = p.Pk[o], qn = cmul(l, q);
                        p.X[o] = cadd(p.X[o], cmul(al, q));
                        p.Pk[o] = cmk(xn + qn.x, qn.y);
                    }
                }
            }
        }
        __syncthreads();
    }

    // ---- one outer step up to u_{n+1} (k_outer_spmm, k_outer_update)
    __device__ void outer(int& err) {
        double v[1][CPL] = {};
        for (int e0 = 0; e0 < nel_pad; e0 += T) {
            if (e0 + (tid & ~31) >= nel_pad) break;
            const Elem e = elem(e0);
            Cols<CPL> h;
            if (MIXED) {
                const float2* xa = reinterpret_cast<const float2*>(vec);
                const double2 y = spmv_df(e, ss.Hhi, ss.Hlo, xa, xa + (size_t)ss.nrows * LPS);
                h.v[0] = y.x;
                if (CPL == 2) h.v[CPL - 1] = y.y;
            } else {
                h = spmv64(e, ss.H64, reinterpret_cast<const double*>(vec));
            }
            if (e.slot < 0) continue;
            const Cols<CPL> u = ldcols<CPL>(at(p.Rcur, e)), r = ldcols<CPL>(at(p.Rin, e)), x = ldcols<CPL>(at(p.Rp, e));
            Cols<CPL> w;
#pragma unroll
            for (int j = 0; j < CPL; ++j) {
                w.v[j] = h.v[j] - sh.cs[e.q * CPL + j].sigma * (u.v[j] - r.v[j]);
                v[0][j] += x.v[j] * w.v[j];
            }
            stcols<CPL>(at(p.W, e), w);
        }
        double out[1];
        sum<1>(v, out);
        if (tid < NC && sh.cs[tid].active) {
            ColState& c = sh.cs[tid];
            if (!lanczos_step_scalars(c, out[0], p.z[c.seed])) sh.bad = 2;
        }
        __syncthreads();
        if (sh.bad == 2) err = 1;
        double w2[1][CPL] = {};
        for (int e0 = 0; e0 < nel_pad; e0 += T) {
            const Elem e = elem(e0);
            if (e.slot < 0) continue;
            const Cols<CPL> u = ldcols<CPL>(at(p.Rcur, e)), um = ldcols<CPL>(at(p.Rprev, e)), w = ldcols<CPL>(at(p.W, e));
            Cols<CPL> un = u, uo = um;
#pragma unroll
            for (int j = 0; j < CPL; ++j) {
                const ColState& c = sh.cs[e.q * CPL + j];
                if (c.active) {
                    un.v[j] = c.g * (w.v[j] - c.asig * u.v[j]) - c.f * um.v[j];
                    uo.v[j] = u.v[j];
                }
                w2[0][j] += un.v[j] * un.v[j];
            }
            stcols<CPL>(at(p.Rprev, e), uo);
            stcols<CPL>(at(p.Rcur, e), un);
        }
        sum<1>(w2, out);
        if (tid < NC) set_rhs(out[0]);
        __syncthreads();
    }
};

template <bool MIXED, int NC>
__global__ void __launch_bounds__(SL_T, 1) k_slice(SliceDev ss, DevSystem s, PanelDev p, SliceArgs a) {
    extern __shared__ __align__(16) unsigned char smem[];
    using S = Slice<MIXED, NC>;
    typename S::Sh& sh = *reinterpret_cast<typename S::Sh*>(smem);
    S sl(ss, s, p, a, sh);
    sl.CL = a.cl;
    sl.rank = blockIdx.x % a.cl;
    sl.c0 = (int)(blockIdx.x / a.cl) * NC;
    sl.tid = threadIdx.x;
    sl.T = blockDim.x;
    sl.par = 0;
    const int noct_l = sl.rank < ss.noct ? (ss.noct - sl.rank + a.cl - 1) / a.cl : 0;
    sl.nel = noct_l * 8 * S::LPS;
    sl.nel_pad = (sl.nel + 31) & ~31;
    unsigned char* q = smem + ((sizeof(typename S::Sh) + 15) & ~(size_t)15);
    sl.part = reinterpret_cast<double*>(q);
    q += sizeof(double) * 2 * S::CPL * sl.T;
    sl.dfun = reinterpret_cast<double*>(q);
    q += ((sizeof(double) * NC * (size_t)(p.M > 0 ? p.M : 1)) + 15) & ~(size_t)15;
    sl.omega = reinterpret_cast<float*>(q);
    q += ((sizeof(float) * (size_t)(MIXED ? a.n : 0)) + 15) & ~(size_t)15;
    sl.vec = q;
    q += sizeof(double) * NC * (size_t)ss.nrows;   // mixed: two FP32 copies; FP64: one
    sl.own = q;
    const int tid = threadIdx.x;
    for (int i = tid; i < NC; i += sl.T) sh.cs[i] = p.col[sl.c0 + i];
    if (MIXED)
        for (int i = tid; i < a.n; i += sl.T) sl.omega[i] = a.omega[i];
    if (tid == 0) sh.open = sh.bad = sh.wanted = sh.active = 0;
    __syncthreads();
    if (tid < NC && sh.cs[tid].active) atomicAdd(&sh.active, 1);
    __syncthreads();
    if (sh.active == 0) return;    // the same in every CTA of the cluster
    sl.barrier();                  // every CTA runs before its shared memory is written
    int steps = 0, err = 0;
    bool ok = true;
    if (a.start) {
        double v[1][S::CPL] = {};
        for (int e0 = 0; e0 < sl.nel_pad; e0 += sl.T) {
            const Elem e = sl.elem(e0);
            if (e.slot < 0) continue;
            const Cols<S::CPL> u = ldcols<S::CPL>(sl.at(p.Rcur, e));
#pragma unroll
            for (int j = 0; j < S::CPL; ++j) v[0][j] += u.v[j] * u.v[j];
        }
        double out[1];
        sl.template sum<1>(v, out);
        if (tid < NC) sl.set_rhs(out[0]);
        __syncthreads();
        ok = sl.inner(steps);
        if (ok) sl.shift_init();
    } else {
        sl.publish_x();
        sl.barrier();
    }
    for (int n = 0; ok && n < a.nsteps; ++n) {
        sl.outer(err);
        ok = sl.inner(steps);
        if (!ok) break;
        sl.shift_step();
        if (sh.active == 0) break;
    }
    sl.barrier();   // no CTA ends while another may still store into its shared memory
    if (sl.rank == 0) {
        if (tid < NC) p.col[sl.c0 + tid] = sh.cs[tid];
        if (tid == 0) {
            if (sh.active) atomicAdd(&p.flags[2], sh.active);
            if (err) atomicOr(&p.flags[0], ERR_BREAKDOWN);
            if (!ok) atomicOr(&p.flags[0], ERR_INNER);
            atomicMax(&p.flags[3], steps);
        }
    }
}

template <bool MIXED, int NC>
size_t slice_smem(const SliceDev& ss, const PanelDev& p, int n_omega, int cl, int T) {
    constexpr int LPS = NC / (MIXED ? 2 : 1);
    const size_t noct_l = (ss.noct + cl - 1) / cl;
    const size_t nel_pad = (noct_l * 8 * LPS + 31) & ~(size_t)31;
    size_t b = (sizeof(SliceShared<NC>) + 15) & ~(size_t)15;
    b += sizeof(double) * 2 * (MIXED ? 2 : 1) * T;
    b += (sizeof(double) * NC * (size_t)(p.M > 0 ? p.M : 1) + 15) & ~(size_t)15;
    b += (sizeof(float) * (size_t)(MIXED ? n_omega : 0) + 15) & ~(size_t)15;
    b += sizeof(double) * NC * (size_t)ss.nrows;
    b += MIXED ? sizeof(float2) * nel_pad : sizeof(double) * 4 * nel_pad;
    return b;
}

constexpr size_t SL_SMEM = 220 * 1024;

template <bool MIXED, int NC>
bool slice_launch(const SliceDev& ss, const DevSystem& s, const PanelDev& p, const SliceArgs& a, int ncols,
                  cudaStream_t st) {
    constexpr int LPS = NC / (MIXED ? 2 : 1);
    const int noct_l = (ss.noct + a.cl - 1) / a.cl;
    const int T = std::min(SL_T, (noct_l * 8 * LPS + 31) / 32 * 32);
    const size_t sm = slice_smem<MIXED, NC>(ss, p, a.n, a.cl, T);
    static std::mutex mu;
    static size_t cur = 0;
    {
        std::lock_guard<std::mutex> lk(mu);
        if (sm > cur) {
            if (cudaFuncSetAttribute(k_slice<MIXED, NC>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm) !=
                cudaSuccess) {
                cudaGetLastError();
                return false;
            }
            cur = sm;
        }
    }
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)((ncols + NC - 1) / NC * a.cl));
    cfg.blockDim = dim3((unsigned)T);
    cfg.dynamicSmemBytes = sm;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)a.cl;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    void* mark = launch_mark_begin(K_SLICE, st);
    const cudaError_t e = cudaLaunchKernelEx(&cfg, k_slice<MIXED, NC>, ss, s, p, a);
    launch_mark_end(mark);
    if (e != cudaSuccess) cudaGetLastError();
    return e == cudaSuccess;
}

size_t slice_smem_for(bool mixed, int nc, const SliceDev& ss, const PanelDev& p, int n, int cl) {
    if (mixed) {
        if (nc == 2) return slice_smem<true, 2>(ss, p, n, cl, SL_T);
        if (nc == 4) return slice_smem<true, 4>(ss, p, n, cl, SL_T);
        return slice_smem<true, 8>(ss, p, n, cl, SL_T);
    }
    if (nc == 1) return slice_smem<false, 1>(ss, p, n, cl, SL_T);
    if (nc == 2) return slice_smem<false, 2>(ss, p, n, cl, SL_T);
    return slice_smem<false, 4>(ss, p, n, cl, SL_T);
}

// values of the items from the 4x4 blocks (src: offset in the block array, -1: zero)
__global__ void k_slice_fill(const double* __restrict__ M, const int* __restrict__ src, long long n,
                             double* __restrict__ m64, float* __restrict__ hi, float* __restrict__ lo) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const int o = src[i];
        const double v = o >= 0 ? M[o] : 0.0;
        const float h = (float)v;
        m64[i] = v;
        hi[i] = h;
        lo[i] = (float)(v - (double)h);
    }
}

}  // namespace

void launch_slice_fill(const double* M, const int* src, long long n, double* m64, float* hi, float* lo, cudaStream_t st) {
    void* mark = launch_mark_begin(K_OTHER, st);
    const long long g = std::min<long long>((n + THREADS - 1) / THREADS, 1216);
    k_slice_fill<<<(unsigned)std::max<long long>(g, 1), THREADS, 0, st>>>(M, src, n, m64, hi, lo);
    launch_mark_end(mark);
}

// Columns per slice and CTAs per cluster for ncols columns on `sms` SMs:
// the fewest columns whose slices fit the SMs at once (a slice's FP64 vector
// work and its gathers grow with its columns), then as many CTAs per slice as
// the SMs and the rows allow (at least two octets of rows per warp).  False:
// the system's rows do not fit.
bool slice_choose(const SliceDev& ss, const PanelDev& p, int n_omega, int ncols, int sms, SliceArgs& a) {
    // TB_SLICE_NC, TB_SLICE_CL: columns per slice and CTAs per cluster by hand
    const char* nc_env = std::getenv("TB_SLICE_NC");
    const char* cl_env = std::getenv("TB_SLICE_CL");
    const int env_nc = nc_env ? std::atoi(nc_env) : 0, env_cl = cl_env ? std::atoi(cl_env) : 0;
    const bool mixed = p.mixed != 0;
    int nc = mixed ? 2 : 1;
    const int top = mixed ? 8 : 4;
    while (nc < top && (ncols + nc - 1) / nc > sms) nc *= 2;
    if (env_nc == 1 || env_nc == 2 || env_nc == 4 || env_nc == 8) nc = std::max(mixed ? 2 : 1, std::min(top, env_nc));
    for (; nc >= (mixed ? 2 : 1); nc /= 2) {
        if (nc > p.P) continue;
        const int slices = (ncols + nc - 1) / nc;
        int cl = std::max(1, std::min({SL_CL, sms / std::max(slices, 1), ss.noct / 2}));
        if (env_cl > 0) cl = std::min({env_cl, SL_CL, ss.noct});
        if (slice_smem_for(mixed, nc, ss, p, n_omega, cl) <= SL_SMEM) {
            a.nc = nc;
            a.cl = cl;
            return true;
        }
    }
    return false;
}

bool launch_slice(const SliceDev& ss, const DevSystem& s, const PanelDev& p, const SliceArgs& a, int ncols,
                  cudaStream_t st) {
    if (p.mixed) {
        if (a.nc == 2) return slice_launch<true, 2>(ss, s, p, a, ncols, st);
        if (a.nc == 4) return slice_launch<true, 4>(ss, s, p, a, ncols, st);
        return slice_launch<true, 8>(ss, s, p, a, ncols, st);
    }
    if (a.nc == 1) return slice_launch<false, 1>(ss, s, p, a, ncols, st);
    if (a.nc == 2) return slice_launch<false, 2>(ss, s, p, a, ncols, st);
    return slice_launch<false, 4>(ss, s, p, a, ncols, st);
}

// Host: groups, octets and items of one system (see the head of the file).
// brow, bcol: its block rows (first block b0 of the handle's arrays), columns
// local to the system; orb: orbitals per atom.
void slice_layout(int n, const int32_t* orb, const int64_t* brow, const int32_t* bcol, int32_t col0, SliceHost& out) {
    struct Group {
        int atom[4];
        int rows;      // rows of the group (4: sp atom or four s atoms)
        bool sp;
        int size;
    };
    std::vector<Group> groups;
    std::vector<char> used(n, 0);
    std::vector<int> mark(n, -1);
    for (int i = 0; i < n; ++i) {
        if (used[i]) continue;
        used[i] = 1;
        Group g{};
        if (orb[i] == 4) {
            g.sp = true;
            g.rows = 4;
            for (int a = 0; a < 4; ++a) g.atom[a] = i;
        } else {
            // the s atoms among i's neighbours that share most of its neighbours
            g.sp = false;
            g.rows = 1;
            g.atom[0] = i;
            for (int64_t b = brow[i]; b < brow[i + 1]; ++b) mark[bcol[b] - col0] = i;
            std::vector<std::pair<int, int>> cand;
            for (int64_t b = brow[i]; b < brow[i + 1]; ++b) {
                const int j = bcol[b] - col0;
                if (used[j] || orb[j] != 1) continue;
                int common = 0;
                for (int64_t d = brow[j]; d < brow[j + 1]; ++d) common += mark[bcol[d] - col0] == i;
                cand.push_back({-common, j});
            }
            std::sort(cand.begin(), cand.end());
            for (size_t k = 0; k < cand.size() && g.rows < 4; ++k) {
                g.atom[g.rows++] = cand[k].second;
                used[cand[k].second] = 1;
            }
        }
        groups.push_back(g);
    }
    // longest groups first, so that the octets of a warp have about the same length
    std::fill(mark.begin(), mark.end(), -1);
    for (size_t k = 0; k < groups.size(); ++k) {
        Group& g = groups[k];
        g.size = 0;
        for (int a = 0; a < (g.sp ? 1 : g.rows); ++a)
            for (int64_t b = brow[g.atom[a]]; b < brow[g.atom[a] + 1]; ++b) {
                const int j = bcol[b] - col0;
                if (mark[j] == (int)k) continue;
                mark[j] = (int)k;
                g.size += orb[j];
            }
    }
    std::stable_sort(groups.begin(), groups.end(), [](const Group& x, const Group& y) { return x.size > y.size; });
    const int ng = (int)groups.size(), noct = (ng + 1) / 2;
    out.noct = noct;
    out.nrows = 8 * noct;
    out.row_slot.assign(out.nrows, -1);
    std::vector<int> row_of((size_t)4 * n, -1);
    for (int k = 0; k < ng; ++k)
        for (int a = 0; a < groups[k].rows; ++a) {
            const int slot = groups[k].sp ? 4 * groups[k].atom[0] + a : 4 * groups[k].atom[a];
            out.row_slot[4 * k + a] = slot;
            row_of[slot] = 4 * k + a;
        }
    struct Item {
        int x;
        int src[4];
    };
    std::vector<std::vector<Item>> st((size_t)8 * noct);
    std::vector<int> pos(out.nrows, -1);
    for (int k = 0; k < ng; ++k) {
        const Group& g = groups[k];
        std::vector<Item> list;
        for (int a = 0; a < (g.sp ? 1 : g.rows); ++a)
            for (int64_t b = brow[g.atom[a]]; b < brow[g.atom[a] + 1]; ++b) {
                const int j = bcol[b] - col0;
                for (int e = 0; e < orb[j]; ++e) {
                    const int x = row_of[4 * j + e];
                    if (pos[x] < 0) {
                        pos[x] = (int)list.size();
                        list.push_back({x, {-1, -1, -1, -1}});
                    }
                    Item& it = list[pos[x]];
                    if (g.sp)
                        for (int r = 0; r < 4; ++r) it.src[r] = (int)(16 * b + 4 * r + e);
                    else it.src[a] = (int)(16 * b + e);
                }
            }
        for (int a = 0; a < 4; ++a) st[4 * k + a].push_back({4 * k + a, {-1, -1, -1, -1}});   // item 0: the own row
        for (const Item& it : list) {
            pos[it.x] = -1;
            if (it.x / 4 == k) st[it.x].front() = it;
            else st[4 * k + (it.x & 3)].push_back(it);
        }
    }
    out.oct_ptr.assign(noct + 1, 0);
    out.idx_ptr.assign(noct + 1, 0);
    for (int o = 0; o < noct; ++o) {
        size_t len = 1;
        for (int q = 0; q < 8; ++q) len = std::max(len, st[8 * o + q].size());
        out.oct_ptr[o + 1] = out.oct_ptr[o] + (int)len;
        out.idx_ptr[o + 1] = out.idx_ptr[o] + (int)((len - 1 + 3) / 4);
    }
    out.src.assign((size_t)out.oct_ptr[noct] * 8 * 4, -1);
    out.idx.assign((size_t)out.idx_ptr[noct] * 8 * 4, 0);
    for (int o = 0; o < noct; ++o)
        for (int q = 0; q < 8; ++q) {
            const std::vector<Item>& v = st[8 * o + q];
            const int len = out.oct_ptr[o + 1] - out.oct_ptr[o];
            for (int k = 0; k < len; ++k) {
                const bool have = k < (int)v.size();
                if (have)
                    for (int r = 0; r < 4; ++r)
                        out.src[4 * ((size_t)(out.oct_ptr[o] + k) * 8 + q) + r] = v[k].src[r];
                if (k > 0)
                    out.idx[4 * ((size_t)(out.idx_ptr[o] + (k - 1) / 4) * 8 + q) + (k - 1) % 4] =
                        (unsigned short)(have ? v[k].x : 8 * o + q);
            }
        }
}

}  // namespace tb
