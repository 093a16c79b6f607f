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
// Here a cluster of CL CTAs owns a slice.  The rows are split over its CTAs;
// each keeps, in shared memory, its own rows of the vector that the products
// gather (d_k of the Chebyshev step, the split u' of the double-float products,
// r of the FP64 CG) and a copy of the other CTAs' rows that its products meet
// (the halo; on small systems simply all of them).  A CTA stores every new row
// also into the copies that need it (distributed shared memory), one cluster
// barrier per step.  The coefficients of S that the inner solve reads every
// step stay in shared memory when they fit; otherwise every warp copies the
// next rows' coefficients ahead (cp.async) while it works on the present ones.
//
// Layout of a system's rows for clusters of CL CTAs (SliceDev, built on first
// use and kept in the handle).  Orbitals are taken in groups of four rows: an
// sp atom, or four s atoms with much the same neighbours.  An item of a group
// is one column of S that meets it: the column's place x among the CTA's rows
// and the four coefficients.  The items with x % 4 == a go to stream a of the
// group, so the four lanes of a group always read four different bank groups
// of the gathered vector, whatever its columns are; two groups (eight streams)
// form an octet, whose items are interleaved step by step: one step of an
// octet is one 128-byte line of coefficients.  Stream a's lane ends with row a
// of the group by a reduce-scatter over the four streams.  Item 0 of every
// stream is the column of the group's own row a (the diagonal).
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
constexpr int SL_CL = 16;    // CTAs per cluster, at most
constexpr int SL_RL = 18;    // steps of a stream whose coefficients a lane keeps in registers, at most
constexpr int SL_SPARE = 2;  // refinement rounds beyond the planned ones (residual with FP64 products)

template <int NC>
struct SliceShared {
    double red[2][SL_CL][2 * NC];          // reductions: per-CTA sums, two buffers
    unsigned long long best[SL_CL][NC];    // largest residual among a CTA's shifts (bits)
    int bestk[SL_CL][NC];                  // and the lowest shift that has it
    int nun[SL_CL][NC];                    // unconverged shifts of a CTA's share
    ColState cs[NC];
    double scale[NC], unscale[NC], b2[NC], tsum[NC];
    double alpha[NC], beta[NC], ainv[2][NC], gprev[2][NC];   // FP64 CG: alpha, beta, 1 / alpha, 1 / gamma
    double nu[NC], inv_nu[NC], Bn[NC], rhat[NC];
    unsigned long long lbest[NC];
    int lbestk[NC], lnun[NC];
    int skip[NC], want[NC];
    int open, bad, wanted, active;
    int bstep;             // step of the block of steps whose coefficients are stored
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

// CPL columns of one orbital row, as a lane holds them: FP64 and FP32, moved in
// 16-byte pieces
template <int CPL>
struct Cols {
    double v[CPL];
};
template <int CPL>
__device__ __forceinline__ Cols<CPL> ldcols(const double* p) {
    Cols<CPL> r;
    if (CPL == 1) {
        r.v[0] = *p;
    } else {
#pragma unroll
        for (int j = 0; j < CPL; j += 2) {
            const double2 q = *reinterpret_cast<const double2*>(p + j);
            r.v[j] = q.x;
            r.v[(j + 1) % CPL] = q.y;
        }
    }
    return r;
}
template <int CPL>
__device__ __forceinline__ void stcols(double* p, const Cols<CPL>& r) {
    if (CPL == 1) {
        *p = r.v[0];
    } else {
#pragma unroll
        for (int j = 0; j < CPL; j += 2)
            *reinterpret_cast<double2*>(p + j) = make_double2(r.v[j], r.v[(j + 1) % CPL]);
    }
}
template <int CPL>
struct alignas(4 * CPL) ColsF {
    float v[CPL];
};

// One lane's element: a row (of the slice order) and its CPL columns.
struct Elem {
    bool on;      // a lane of the CTA's share
    int oct, s8;  // octet of the CTA and stream
    int row, q;   // the CTA's row, lane within the row
    int slot;     // padded orbital slot (-1: a filling row, always zero)
};

// Where things lie in a CTA's dynamic shared memory (byte offsets)
struct SliceMem {
    size_t part, dfun, omega, tab, vec, own, sbuf, total;
};
__host__ __device__ __forceinline__ size_t up16(size_t v) { return (v + 15) & ~(size_t)15; }
template <bool MIXED, int NC, int CPL>
__host__ __device__ __forceinline__ SliceMem slice_mem(const SliceDev& ss, int M, int n_omega, int resident, int obytes,
                                                       int T) {
    constexpr int LPS = NC / CPL;
    const size_t nel_pad = ((size_t)ss.max_oct * 8 * LPS + 31) & ~(size_t)31;
    SliceMem m;
    m.part = up16(sizeof(SliceShared<NC>));
    m.dfun = m.part + up16(sizeof(double) * CPL * T);
    m.omega = m.dfun + up16(sizeof(double) * NC * (size_t)(M > 0 ? M : 1));
    m.tab = m.omega + up16((MIXED ? sizeof(float) : sizeof(double)) * (size_t)n_omega);
    m.vec = m.tab + up16(sizeof(int) * (size_t)(4 * ss.max_oct + 3 + ss.max_dest));
    m.own = m.vec + (MIXED ? 1 : 2) * sizeof(double) * NC * (size_t)ss.nloc;   // two vectors, FP32 or FP64
    m.sbuf = m.own + (MIXED ? sizeof(float) * CPL * nel_pad : sizeof(double) * 4 * nel_pad);
    m.total = m.sbuf;
    if (resident == 2) return m;                                // S in registers
    if (resident) m.total += (size_t)ss.max_steps * (MIXED ? 128 : 256) + (size_t)ss.max_bat * 64;
    else if (MIXED) m.total += (size_t)(T / 32) * 2 * (4 / LPS > 0 ? 4 / LPS : 1) * obytes;
    return m;
}

template <bool MIXED, int NC, int CPL, bool REG>
struct Slice {   // CPL: columns per lane
    static constexpr int LPS = NC / CPL;        // lanes per row
    static constexpr int NP = CPL > 1 ? CPL / 2 : 1;            // pairs of them
    using Sh = SliceShared<NC>;
    using VF = ColsF<CPL>;
    const SliceDev& ss;
    const DevSystem& s;
    const PanelDev& p;
    const SliceArgs& a;
    Sh& sh;
    double* part;     // [CPL][T] reduction scratch
    double* dfun;     // [NC][M]
    float* omega;
    unsigned char* vec;   // the gathered vector(s): own rows, then the halo
    unsigned char* own;   // per-element values of this CTA
    int* optr;            // [octets + 1] first step of the CTA's octets
    int* iptr;            // [octets + 1] first index batch
    int* dptr;            // [groups + 1] destinations of a group's rows
    int* dest;            // rank << 16 | group there
    unsigned char* sbuf;  // coefficients and indices: all octets, or two buffers per warp
    int CL, rank, c0, tid, T, nel, nel_pad, par;
    int oct0, step0, bat0;   // the CTA's first octet, its first step and index batch
    int nloc;                // rows of the gathered vector
    int nsteps_all;          // steps of all octets of the CTA
    int phase;               // ring: parity of the buffer that holds the present pass

    __device__ Slice(const SliceDev& ss_, const DevSystem& s_, const PanelDev& p_, const SliceArgs& a_, Sh& sh_)
        : ss(ss_), s(s_), p(p_), a(a_), sh(sh_) {}

    __device__ void barrier() {
        if (CL == 1) __syncthreads();
        else cg::this_cluster().sync();
    }
    // v into element i of row `row`'s entry of buf, here and in every copy of
    // the row (buf: [rows][n])
    template <class V>
    __device__ __forceinline__ void bcast(V* buf, int row, int n, int i, V v) {
        buf[(size_t)row * n + i] = v;
        const int g = row >> 2;
        for (int d = dptr[g]; d < dptr[g + 1]; ++d) {
            const int e = dest[d];
            V* to = buf + ((size_t)(e & 0xffff) * 4 + (row & 3)) * n + i;
            *cg::this_cluster().map_shared_rank(to, e >> 16) = v;
        }
    }
    __device__ __forceinline__ Elem elem(int e0) const {
        Elem e;
        const int el = e0 + tid;
        e.on = el < nel;
        e.row = el / LPS;
        e.q = el % LPS;
        e.s8 = e.row & 7;
        e.oct = e.row >> 3;
        e.slot = e.on ? __ldg(ss.row_slot + oct0 * 8 + e.row) : -1;
        return e;
    }
    __device__ __forceinline__ double* at(double2* base, const Elem& e) const {
        return reinterpret_cast<double*>(base) + (size_t)e.slot * p.P + c0 + e.q * CPL;
    }

    // column thread tid: v into this CTA's entry of arr[rank][column] of every CTA
    template <class V>
    __device__ __forceinline__ void share(V (&arr)[SL_CL][NC], V v) {
        if (CL == 1) arr[0][tid] = v;
        else
            for (int r = 0; r < CL; ++r) *cg::this_cluster().map_shared_rank(&arr[rank][tid], r) = v;
    }

    // Sums over all rows of the slice of NQ values per column; out[qn] valid
    // in threads tid < NC (column tid) of every CTA, the same in all of them.
    // Fixed order: threads' values, warps' trees, ranks.
    template <int NQ>
    __device__ void sum(const double (&v)[NQ][CPL], double (&out)[NQ]) {
        const int lane = tid & 31, nw = T >> 5;
#pragma unroll
        for (int n = 0; n < NQ; ++n) {
            if (n > 0) __syncthreads();
#pragma unroll
            for (int j = 0; j < CPL; ++j) part[j * T + tid] = v[n][j];
            __syncthreads();
            for (int c = tid >> 5; c < NC; c += nw) {
                const int q = c / CPL, j = c % CPL;
                const double* src = part + j * T + q;
                // four chains: an FP64 operation here takes ~70 cycles to its result
                double acc = 0.0, c1 = 0.0, c2 = 0.0, c3 = 0.0;
                const int ne = T / LPS;
                for (int i = lane; i < ne; i += 128) {
                    acc += src[i * LPS];
                    if (i + 32 < ne) c1 += src[(i + 32) * LPS];
                    if (i + 64 < ne) c2 += src[(i + 64) * LPS];
                    if (i + 96 < ne) c3 += src[(i + 96) * LPS];
                }
                acc = (acc + c1) + (c2 + c3);
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
                if (lane == 0) {
                    if (CL == 1) sh.red[par][0][n * NC + c] = acc;
                    else
                        for (int r = 0; r < CL; ++r)
                            *cg::this_cluster().map_shared_rank(&sh.red[par][rank][n * NC + c], r) = acc;
                }
            }
        }
        barrier();
        if (tid < NC) {
#pragma unroll
            for (int n = 0; n < NQ; ++n) {
                double acc[4] = {0.0, 0.0, 0.0, 0.0};
                for (int r = 0; r < CL; r += 4)
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        if (r + j < CL) acc[j] += sh.red[par][r + j][n * NC + tid];
                out[n] = (acc[0] + acc[1]) + (acc[2] + acc[3]);
            }
        }
        par ^= 1;
    }

    // ---- products ----------------------------------------------------------
    // item loop of one stream: f(step, row of the gathered vector); ix: the
    // octet's index batches of this stream
    template <class F>
    __device__ __forceinline__ static void items(int row, int n, const ushort4* ix, bool diag, F&& f) {
        if (diag) f(0, row);
        int k = 1;
#pragma unroll 2
        for (; k + 4 <= n; k += 4, ix += 8) {
            const ushort4 id = *ix;
            f(k, id.x);
            f(k + 1, id.y);
            f(k + 2, id.z);
            f(k + 3, id.w);
        }
        if (k < n) {
            const ushort4 id = *ix;
            f(k, id.x);
            if (k + 1 < n) f(k + 1, id.y);
            if (k + 2 < n) f(k + 2, id.z);
        }
    }
    __device__ __forceinline__ int len(const Elem& e) const { return optr[e.oct + 1] - optr[e.oct]; }
    // first item of the element's stream in the coefficient arrays
    __device__ __forceinline__ size_t item0(const Elem& e) const { return (size_t)(step0 + optr[e.oct]) * 8 + e.s8; }
    __device__ __forceinline__ const ushort4* batches(const Elem& e) const {
        return ss.idx + (size_t)(bat0 + iptr[e.oct]) * 8 + e.s8;
    }

    // ---- S in shared memory ----------------------------------------------
    // Resident: coefficients of all octets of the CTA, then their indices.
    // FP64: the two halves of a step's coefficients in separate lines.
    __device__ __forceinline__ static void cp16(void* dst, const void* src) {
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                         static_cast<uint32_t>(__cvta_generic_to_shared(dst))),
                     "l"(src));
    }
    __device__ __forceinline__ static void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
    __device__ __forceinline__ static void cp_wait() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }
    static constexpr int LINE = MIXED ? 128 : 256;   // bytes of one step of an octet
    __device__ void load_resident(int noct) {
        const int steps = optr[noct], nb = iptr[noct];
        if (MIXED) {
            const float4* src = ss.Shi + (size_t)step0 * 8;
            for (int i = tid; i < steps * 8; i += T) cp16(sbuf + 16 * (size_t)i, src + i);
        } else {
            const double2* src = ss.S64 + (size_t)step0 * 16;
            for (int i = tid; i < steps * 16; i += T) {
                const int k = i >> 4, s8 = (i >> 1) & 7, h = i & 1;
                cp16(sbuf + 16 * ((size_t)(2 * k + h) * 8 + s8), src + i);
            }
        }
        const ushort4* si = ss.idx + (size_t)bat0 * 8;
        unsigned char* di = sbuf + (size_t)steps * LINE;
        for (int i = tid; i < nb * 4; i += T) cp16(di + 16 * (size_t)i, si + 2 * i);
        cp_commit();
        cp_wait();
        __syncthreads();
    }
    // Ring: a warp's octets of the pass that starts at element e0 into its
    // buffer `b` (octet j of the warp at stride a.obytes: lines, then indices)
    static constexpr int WO = 4 / LPS > 0 ? 4 / LPS : 1;   // octets of a warp
    __device__ __forceinline__ unsigned char* ring(int b) const {
        return sbuf + ((size_t)(tid >> 5) * 2 + b) * (WO * (size_t)a.obytes);
    }
    __device__ __forceinline__ void ring_load(int e0, int b) {
        unsigned char* dst = ring(b);
        const int lane = tid & 31, o0 = (e0 + (tid & ~31)) / LPS >> 3, no = nel / LPS >> 3;
#pragma unroll
        for (int j = 0; j < WO; ++j) {
            const int o = o0 + j;
            if (o >= no) break;
            const int n8 = (optr[o + 1] - optr[o]) * 8, nb = iptr[o + 1] - iptr[o];
            const float4* src = ss.Shi + (size_t)(step0 + optr[o]) * 8;
            const ushort4* si = ss.idx + (size_t)(bat0 + iptr[o]) * 8;
            unsigned char* d = dst + (size_t)j * a.obytes;
            for (int i = lane; i < n8; i += 32) cp16(d + 16 * i, src + i);
            for (int i = lane; i < nb * 4; i += 32) cp16(d + (size_t)a.ibase + 16 * i, si + 2 * i);
        }
        cp_commit();
    }
    // Where the first REMOTE copies of an element's row lie (shared::cluster
    // addresses in xa; xb at the same distance in every CTA), worked out once a
    // round: 13 columns of 144 atoms, four CTAs per slice, 36.9 -> 34.8 ms per
    // call; with S in shared memory and one element per thread too, a
    // charge-self-consistent call of 48 water molecules 42.6 -> 40.9 ms (the row
    // itself kept across steps: 40.5, but a batch of boxes 26.0 -> 26.5); FP64,
    // one column of 64 atoms 36.2 -> 34.6, 48 of 216 atoms 107.3 -> 105.9.  With
    // four columns per lane the registers are full (512 atoms: 109.0 -> 110.0
    // ms), and every copy is looked up at its store.
    static constexpr int REMOTE = CPL <= 2 ? 3 : 0;
    struct Copies {
        unsigned at[REMOTE + 1];
        unsigned to_b;
        int n, first;
    };
    template <class V>
    __device__ __forceinline__ Copies copies(const Elem& e, V* xa, V* xb) {
        Copies c;
        c.n = c.first = 0;
        c.to_b = (unsigned)(reinterpret_cast<unsigned char*>(xb) - reinterpret_cast<unsigned char*>(xa));
        if (e.on) {
            c.first = dptr[e.row >> 2];
            c.n = dptr[(e.row >> 2) + 1] - c.first;
        }
#pragma unroll
        for (int i = 0; i < REMOTE; ++i) {
            c.at[i] = 0;
            if (i < c.n) {
                const int d = dest[c.first + i];
                const uint32_t here = static_cast<uint32_t>(
                    __cvta_generic_to_shared(xa + ((size_t)(d & 0xffff) * 4 + (e.row & 3)) * LPS + e.q));
                asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(c.at[i]) : "r"(here), "r"(d >> 16));
            }
        }
        return c;
    }
    __device__ __forceinline__ static void st_remote(unsigned at, double v) {
        asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(at), "d"(v) : "memory");
    }
    __device__ __forceinline__ static void st_remote(unsigned at, const VF& v) {
        asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(at), "f"(v.v[0]), "f"(v.v[CPL - 1]) : "memory");
    }
    // bcast(to, ...) of a row whose copies are known; to: xa, or xb (b)
    template <class V>
    __device__ __forceinline__ void publish(const Elem& e, const Copies& c, V* to, bool b, const V& v) {
        if constexpr (REMOTE == 0) {
            bcast(to, e.row, LPS, e.q, v);
        } else {
            to[(size_t)e.row * LPS + e.q] = v;
            const unsigned off = b ? c.to_b : 0u;
#pragma unroll
            for (int i = 0; i < REMOTE; ++i)
                if (i < c.n) st_remote(c.at[i] + off, v);
            for (int i = REMOTE; i < c.n; ++i) {
                const int d = dest[c.first + i];
                *cg::this_cluster().map_shared_rank(to + ((size_t)(d & 0xffff) * 4 + (e.row & 3)) * LPS + e.q, d >> 16) = v;
            }
        }
    }
    // FP32 product with S; cf, ix: the stream's coefficients and indices in
    // shared memory.  Scalar FMAs: a packed one needs its coefficient twice in a
    // register pair, which costs as many moves as it saves.  The four streams'
    // partial sums of rows 0..3 become row (stream) of each lane.
    __device__ __forceinline__ VF spmv32(const Elem& e, const float* cur, bool diag, const float4* cf,
                                         const ushort4* ix) const {
        float acc[4][CPL];
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < CPL; ++j) acc[i][j] = 0.f;
        if (e.on) {
            const float* xq = cur + e.q * CPL;
            items(e.row, len(e), ix, diag, [&](int k, int x) {
                const float4 c = cf[k * 8];
                const VF v = *reinterpret_cast<const VF*>(xq + x * NC);
#pragma unroll
                for (int j = 0; j < CPL; ++j) {
                    acc[0][j] = fmaf(c.x, v.v[j], acc[0][j]);
                    acc[1][j] = fmaf(c.y, v.v[j], acc[1][j]);
                    acc[2][j] = fmaf(c.z, v.v[j], acc[2][j]);
                    acc[3][j] = fmaf(c.w, v.v[j], acc[3][j]);
                }
            });
        }
        __syncwarp();
        const int st = e.s8 & 3;
        const bool up = st & 2, odd = st & 1;
        VF r;
#pragma unroll
        for (int j = 0; j < CPL; ++j) {
            float k0 = up ? acc[2][j] : acc[0][j], k1 = up ? acc[3][j] : acc[1][j];
            k0 += __shfl_xor_sync(0xffffffffu, up ? acc[0][j] : acc[2][j], 2 * LPS);
            k1 += __shfl_xor_sync(0xffffffffu, up ? acc[1][j] : acc[3][j], 2 * LPS);
            const float t = __shfl_xor_sync(0xffffffffu, odd ? k0 : k1, LPS);
            r.v[j] = (odd ? k1 : k0) + t;
        }
        return r;
    }
    // double-float product with (Mh, Ml) of the split vector (xh, xl)
    __device__ __forceinline__ Cols<CPL> spmv_df(const Elem& e, const float4* Mh, const float4* Ml, const float* xh,
                                                 const float* xl) const {
        float2 hi[4][NP], lo[4][NP];
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < NP; ++j) hi[i][j] = lo[i][j] = make_float2(0.f, 0.f);
        if (e.on) {
            const float4 *mh = Mh + item0(e), *ml = Ml + item0(e);
            items(e.row, len(e), batches(e), true, [&](int k, int x) {
                const float4 ch = __ldg(mh + 8 * k), cl = __ldg(ml + 8 * k);
                const VF vh = *reinterpret_cast<const VF*>(xh + x * NC + e.q * CPL);
                const VF vl = *reinterpret_cast<const VF*>(xl + x * NC + e.q * CPL);
#pragma unroll
                for (int j = 0; j < NP; ++j) {
                    const float2 h = make_float2(vh.v[2 * j], vh.v[(2 * j + 1) % CPL]);
                    const float2 l = make_float2(vl.v[2 * j], vl.v[(2 * j + 1) % CPL]);
                    df_mac2(hi[0][j], lo[0][j], ch.x, cl.x, h, l);
                    df_mac2(hi[1][j], lo[1][j], ch.y, cl.y, h, l);
                    df_mac2(hi[2][j], lo[2][j], ch.z, cl.z, h, l);
                    df_mac2(hi[3][j], lo[3][j], ch.w, cl.w, h, l);
                }
            });
        }
        __syncwarp();
        const int st = e.s8 & 3;
        const bool up = st & 2, odd = st & 1;
        Cols<CPL> r;
#pragma unroll
        for (int j = 0; j < NP; ++j) {
            float2 h0 = up ? hi[2][j] : hi[0][j], l0 = up ? lo[2][j] : lo[0][j];
            float2 h1 = up ? hi[3][j] : hi[1][j], l1 = up ? lo[3][j] : lo[1][j];
            const float2 a0 = shfl2(up ? hi[0][j] : hi[2][j], 2 * LPS), b0 = shfl2(up ? lo[0][j] : lo[2][j], 2 * LPS);
            const float2 a1 = shfl2(up ? hi[1][j] : hi[3][j], 2 * LPS), b1 = shfl2(up ? lo[1][j] : lo[3][j], 2 * LPS);
            df_add2(h0, l0, a0, b0);
            df_add2(h1, l1, a1, b1);
            const float2 a2 = shfl2(odd ? h0 : h1, LPS), b2 = shfl2(odd ? l0 : l1, LPS);
            float2 h = odd ? h1 : h0, l = odd ? l1 : l0;
            df_add2(h, l, a2, b2);
            r.v[2 * j] = (double)h.x + (double)l.x;
            r.v[(2 * j + 1) % CPL] = (double)h.y + (double)l.y;
        }
        return r;
    }
    // FP64 product; M: the coefficients in global memory (mc == nullptr), or
    // mc, ix: the stream's in shared memory
    __device__ __forceinline__ Cols<CPL> spmv64(const Elem& e, const double2* M, const double* x_,
                                                const double2* mc = nullptr, const ushort4* ix = nullptr) const {
        double acc[4][CPL];
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < CPL; ++j) acc[i][j] = 0.0;
        if (e.on) {
            const double* xq = x_ + e.q * CPL;
            auto mac = [&](const double2 c01, const double2 c23, int x) {
                const Cols<CPL> v = ldcols<CPL>(xq + x * NC);
#pragma unroll
                for (int j = 0; j < CPL; ++j) {
                    acc[0][j] += c01.x * v.v[j];
                    acc[1][j] += c01.y * v.v[j];
                    acc[2][j] += c23.x * v.v[j];
                    acc[3][j] += c23.y * v.v[j];
                }
            };
            if (mc) {
                items(e.row, len(e), ix, true, [&](int k, int x) { mac(mc[16 * k], mc[16 * k + 8], x); });
            } else {
                const double2* m = M + 2 * item0(e);
                items(e.row, len(e), batches(e), true,
                      [&](int k, int x) { mac(__ldg(m + 16 * k), __ldg(m + 16 * k + 1), x); });
            }
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
                VF h, l;
#pragma unroll
                for (int j = 0; j < CPL; ++j) {
                    h.v[j] = (float)x.v[j];
                    l.v[j] = (float)(x.v[j] - (double)h.v[j]);
                }
                VF* xa = reinterpret_cast<VF*>(vec);
                bcast(xa, e.row, LPS, e.q, h);
                bcast(xa + (size_t)nloc * LPS, e.row, LPS, e.q, l);
            } else {
                bcast(reinterpret_cast<double*>(vec), e.row, NC, e.q, x.v[0]);
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
        VF* xa = reinterpret_cast<VF*>(vec);
        VF* xb = xa + (size_t)nloc * LPS;
        VF* fb = reinterpret_cast<VF*>(own);
        const bool skip_diag = ss.unit_diag != 0;
        for (int round = 0;; ++round) {
            const int n = round >= a.R - 1 ? a.n_last : a.n;
            steps += n;
            const bool fp64 = round >= a.R;
            for (int e0 = 0; e0 < nel_pad; e0 += T) {
                const Elem e = elem(e0);
                if (!e.on) continue;
                VF f = {}, d1;
                if (e.slot >= 0) {
                    const Cols<CPL> v = ldcols<CPL>(at(round == 0 ? p.Rcur : p.Rin, e));
#pragma unroll
                    for (int j = 0; j < CPL; ++j) f.v[j] = (float)(v.v[j] * sh.scale[e.q * CPL + j]);
                }
                fb[e0 + tid] = f;
#pragma unroll
                for (int j = 0; j < CPL; ++j) d1.v[j] = a.gamma * f.v[j];
                bcast(xa, e.row, LPS, e.q, d1);
                if (n == 1 && e.slot >= 0) add_correction(e, d1, round);
            }
            barrier();
            if (REG) chebyshev_reg(n, round, xa, xb, fb);
            // one element per thread: its row's copies are the same in every step
            const bool single = !REG && nel_pad <= T;
            const Copies cp = copies(elem(0), xa, xb);
            for (int k = 1; !REG && k < n; ++k) {
                const VF* cur = (k & 1) ? xa : xb;
                VF* io = (k & 1) ? xb : xa;
                const float om = omega[k];
                for (int e0 = 0; e0 < nel_pad; e0 += T) {
                    if (e0 + (tid & ~31) >= nel_pad) break;
                    const Elem e = elem(e0);
                    const unsigned char* sb;
                    const ushort4* ix;
                    if (a.resident) {
                        sb = sbuf + (size_t)(e.on ? optr[e.oct] : 0) * LINE;
                        ix = reinterpret_cast<const ushort4*>(sbuf + (size_t)nsteps_all * LINE) +
                             (size_t)(e.on ? iptr[e.oct] : 0) * 8;
                    } else {
                        // this pass is in the buffer of the present phase (copied
                        // during the pass before); the next one goes to the other
                        cp_wait();
                        __syncwarp();
                        int nx = e0 + T;
                        if (nx + (tid & ~31) >= nel_pad) nx = 0;
                        ring_load(nx, phase ^ 1);
                        sb = ring(phase) + (size_t)((tid & 31) / LPS >> 3) * a.obytes;
                        ix = reinterpret_cast<const ushort4*>(sb + a.ibase);
                        phase ^= 1;
                    }
                    const VF y = spmv32(e, reinterpret_cast<const float*>(cur), !skip_diag,
                                        reinterpret_cast<const float4*>(sb) + e.s8, ix + e.s8);
                    if (!e.on) continue;
                    const size_t w = (size_t)e.row * LPS + e.q;
                    const VF dc = cur[w], f = fb[e0 + tid];
                    VF dp = {}, dn;
                    if (k > 1) dp = io[w];
#pragma unroll
                    for (int j = 0; j < CPL; ++j) {
                        const float yj = skip_diag ? y.v[j] + dc.v[j] : y.v[j];
                        dn.v[j] = e.slot < 0 ? 0.f
                                             : dp.v[j] + om * (a.gamma * (f.v[j] - yj) + dc.v[j] - dp.v[j]);
                    }
                    if (k == n - 1) {
                        if (e.slot >= 0) add_correction(e, dn, round);
                    } else {
                        if (single) publish(e, cp, io, (k & 1) != 0, dn);
                        else bcast(io, e.row, LPS, e.q, dn);
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
                    const Cols<CPL> y = spmv_df(e, ss.Shi, ss.Slo, reinterpret_cast<const float*>(xa),
                                                reinterpret_cast<const float*>(xb));
                    if (e.slot >= 0) residual(e, y, v);
                }
            } else {
                double* xd = reinterpret_cast<double*>(vec);
                for (int e0 = 0; e0 < nel_pad; e0 += T) {
                    const Elem e = elem(e0);
                    if (!e.on) continue;
                    Cols<CPL> x{};
                    if (e.slot >= 0) x = ldcols<CPL>(at(p.Rp, e));
                    bcast(reinterpret_cast<Cols<CPL>*>(xd), e.row, LPS, e.q, x);
                }
                barrier();
                for (int e0 = 0; e0 < nel_pad; e0 += T) {
                    if (e0 + (tid & ~31) >= nel_pad) break;
                    const Elem e = elem(e0);
                    const Cols<CPL> y = spmv64(e, ss.S64, xd);
                    if (e.slot >= 0) residual(e, y, v);
                }
            }
            // t = u^T u' is summed with the residual of a round that may be the last
            double out[2] = {0.0, 0.0};
            if (round >= a.R - 1) {
                sum<2>(v, out);
            } else {
                double w[1][CPL], o1[1];
#pragma unroll
                for (int j = 0; j < CPL; ++j) w[0][j] = v[0][j];
                sum<1>(w, o1);
                out[0] = o1[0];
            }
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
                if (round < a.R - 1) {   // converged before the planned rounds: t is still to be summed
                    double w[1][CPL], o1[1];
#pragma unroll
                    for (int j = 0; j < CPL; ++j) w[0][j] = v[1][j];
                    sum<1>(w, o1);
                    if (tid < NC) sh.tsum[tid] = o1[0];
                    __syncthreads();
                }
                if (fp64) {
                    publish_x();
                    barrier();
                }
                return true;
            }
            if (round + 1 >= a.R + SL_SPARE) return false;
        }
    }
    // The steps of a round with one element per thread: the coefficients and
    // places of its stream, f, d_k and d_{k-1} of its own row stay in registers;
    // only the gathered rows are read from shared memory (half its traffic, and
    // with the coefficients there it is what bounds the step).
    __device__ __forceinline__ void chebyshev_reg(int n, int round, VF* xa, VF* xb, const VF* fb) {
        const Elem e = elem(0);
        float4 sr[SL_RL];
        unsigned xi[(SL_RL + 1) / 2];
        {
            const int ln = e.on ? len(e) : 0;
            const float4* src = ss.Shi + (e.on ? item0(e) : 0);
            const ushort4* ix = ss.idx + (e.on ? (size_t)(bat0 + iptr[e.oct]) * 8 + e.s8 : 0);
            const unsigned short own_row = (unsigned short)(e.on ? e.row : 0);
#pragma unroll
            for (int k = 0; k < SL_RL; ++k) sr[k] = k < ln ? __ldg(src + 8 * k) : make_float4(0.f, 0.f, 0.f, 0.f);
            unsigned short id[SL_RL + 3];
            id[0] = own_row;
#pragma unroll
            for (int b = 0; b < (SL_RL + 2) / 4; ++b) {
                ushort4 q = make_ushort4(own_row, own_row, own_row, own_row);
                if (4 * b + 1 < ln) q = __ldg(ix + 8 * b);
                id[4 * b + 1] = q.x;
                id[4 * b + 2] = q.y;
                id[4 * b + 3] = q.z;
                if (4 * b + 4 < SL_RL + 3) id[4 * b + 4] = q.w;
            }
#pragma unroll
            for (int k = 0; k < SL_RL; k += 2) xi[k / 2] = id[k] | ((unsigned)id[k + 1] << 16);
        }
        const bool skip_diag = ss.unit_diag != 0;
        VF f = {}, dk, dp = {};
        if (e.on) f = fb[tid];
#pragma unroll
        for (int j = 0; j < CPL; ++j) dk.v[j] = a.gamma * f.v[j];
        const int st = e.s8 & 3;
        const bool up = st & 2, odd = st & 1;
        const Copies cp = copies(e, xa, xb);
        for (int k = 1; k < n; ++k) {
            const float* xq = reinterpret_cast<const float*>((k & 1) ? xa : xb) + e.q * CPL;
            float acc[4][CPL];
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < CPL; ++j) acc[i][j] = 0.f;
#pragma unroll
            for (int i = 0; i < SL_RL; ++i) {
                if (i == 0 && skip_diag) continue;
                if (i == SL_RL - 1 && ss.max_len < SL_RL) continue;
                const unsigned x = (i & 1) ? xi[i / 2] >> 16 : xi[i / 2] & 0xffffu;
                const VF v = *reinterpret_cast<const VF*>(xq + x * NC);
#pragma unroll
                for (int j = 0; j < CPL; ++j) {
                    acc[0][j] = fmaf(sr[i].x, v.v[j], acc[0][j]);
                    acc[1][j] = fmaf(sr[i].y, v.v[j], acc[1][j]);
                    acc[2][j] = fmaf(sr[i].z, v.v[j], acc[2][j]);
                    acc[3][j] = fmaf(sr[i].w, v.v[j], acc[3][j]);
                }
            }
            VF dn;
            const float om = omega[k];
#pragma unroll
            for (int j = 0; j < CPL; ++j) {
                float k0 = up ? acc[2][j] : acc[0][j], k1 = up ? acc[3][j] : acc[1][j];
                k0 += __shfl_xor_sync(0xffffffffu, up ? acc[0][j] : acc[2][j], 2 * LPS);
                k1 += __shfl_xor_sync(0xffffffffu, up ? acc[1][j] : acc[3][j], 2 * LPS);
                const float t = __shfl_xor_sync(0xffffffffu, odd ? k0 : k1, LPS);
                float y = (odd ? k1 : k0) + t;
                if (skip_diag) y += dk.v[j];
                dn.v[j] = e.slot < 0 ? 0.f : dp.v[j] + om * (a.gamma * (f.v[j] - y) + dk.v[j] - dp.v[j]);
            }
            dp = dk;
            dk = dn;
            if (k < n - 1 && e.on) publish(e, cp, (k & 1) ? xb : xa, (k & 1) != 0, dn);
            barrier();
        }
        if (n > 1 && e.slot >= 0) add_correction(e, dk, round);
    }

    // u' += d * ||res|| (a non-finite correction is dropped, as in k_refine_add)
    __device__ __forceinline__ void add_correction(const Elem& e, const VF& d, int round) {
        Cols<CPL> x{};
        double* px = at(p.Rp, e);
        if (round > 0) x = ldcols<CPL>(px);
#pragma unroll
        for (int j = 0; j < CPL; ++j)
            if (isfinite(d.v[j])) x.v[j] += (double)d.v[j] * sh.unscale[e.q * CPL + j];
        stcols<CPL>(px, x);
    }
    __device__ __forceinline__ void residual(const Elem& e, const Cols<CPL>& y, double (&v)[2][CPL]) {
        const Cols<CPL> u = ldcols<CPL>(at(p.Rcur, e)), x = ldcols<CPL>(at(p.Rp, e));
        Cols<CPL> r;
#pragma unroll
        for (int j = 0; j < CPL; ++j) {
            r.v[j] = u.v[j] - y.v[j];
            v[0][j] += r.v[j] * r.v[j];
            v[1][j] += u.v[j] * x.v[j];
        }
        stcols<CPL>(at(p.Rin, e), r);
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
            bcast(rv, e.row, NC, e.q, e.slot >= 0 ? *at(p.Rcur, e) : 0.0);
            pv[e0 + tid] = sv[e0 + tid] = xv[e0 + tid] = 0.0;
        }
        barrier();
        int it = 0;
        for (;; ++it) {
            double v[2][CPL] = {};
            for (int e0 = 0; e0 < nel_pad; e0 += T) {
                if (e0 + (tid & ~31) >= nel_pad) break;
                const Elem e = elem(e0);
                const double w = product_S(e, rv);
                if (!e.on) continue;
                const double r = rv[(size_t)e.row * NC + e.q];
                wv[e0 + tid] = w;
                if (e.slot >= 0) {
                    v[0][0] += r * r;
                    v[1][0] += w * r;
                }
            }
            double out[2];
            sum<2>(v, out);
            if (tid == 0) sh.open = sh.bad = 0;
            __syncthreads();
            // beta = gam / gam_prev and den = del - beta gam / alpha_prev with the
            // reciprocals of the iteration before; an FP64 division takes ~800
            // cycles, so three lanes of a column form alpha, 1 / alpha and 1 / gam
            // in one
            if (tid < NC) {
                sh.tsum[tid] = out[0];
                sh.rhat[tid] = out[1];
            }
            __syncthreads();
            if (tid < 3 * NC) {
                const int role = tid / NC, c = tid % NC;
                const double gam = sh.tsum[c], del = sh.rhat[c];
                const bool done = sh.skip[c] || gam <= a.inner_tol * a.inner_tol * sh.b2[c];
                const double beta = it == 0 ? 0.0 : gam * sh.gprev[it & 1][c];
                const double den = it == 0 ? del : del - beta * gam * sh.ainv[it & 1][c];
                const double q = (role == 0 ? gam : role == 1 ? den : 1.0) / (role == 0 ? den : gam);
                if (!done) {
                    if (role == 0) {
                        if (!(den > 0.0)) {
                            atomicExch(&sh.bad, 1);
                        } else {
                            sh.alpha[c] = q;
                            sh.beta[c] = beta;
                            atomicAdd(&sh.open, 1);
                        }
                    } else if (role == 1) {
                        sh.ainv[(it + 1) & 1][c] = q;
                    } else {
                        sh.gprev[(it + 1) & 1][c] = q;
                    }
                }
                __syncwarp((1u << (3 * NC)) - 1u);
                if (role == 0 && done) sh.skip[c] = 1;
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
                bcast(rv, e.row, NC, e.q, r - al * sn);
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
            bcast(rv, e.row, NC, e.q, x);   // the products of the outer step gather u'
        }
        double out[1];
        sum<1>(v, out);
        if (tid < NC) sh.tsum[tid] = out[0];
        __syncthreads();
        return true;
    }
    // ---- inner solve in FP64 by Chebyshev steps for the spectrum of S (the
    // recurrence of the mixed path's corrections, all of it in FP64): no inner
    // products, so a step is a product and a barrier where a CG iteration has two
    // reductions, ~2000 cycles of scalars and a second barrier.  The residual
    // u - S u' at its end decides; a column above inner_tol takes further rounds
    // on its residual (a.n_last steps each).
    __device__ bool inner_cheb64(int& steps) {
        double* xa = reinterpret_cast<double*>(vec);
        double* xb = xa + (size_t)nloc * NC;
        double* fb = reinterpret_cast<double*>(own);
        double* xs = fb + nel_pad;
        const double* om = reinterpret_cast<const double*>(omega);
        for (int round = 0;; ++round) {
            const int n = round == 0 ? a.n : a.n_last;
            steps += n;
            for (int e0 = 0; e0 < nel_pad; e0 += T) {
                const Elem e = elem(e0);
                if (!e.on) continue;
                const double f = e.slot >= 0 && !sh.skip[e.q] ? *at(round == 0 ? p.Rcur : p.Rin, e) : 0.0;
                fb[e0 + tid] = f;
                if (round == 0) xs[e0 + tid] = 0.0;
                bcast(xa, e.row, NC, e.q, a.gamma64 * f);
                if (n == 1) xs[e0 + tid] += a.gamma64 * f;
            }
            barrier();
            const bool single = nel_pad <= T;
            const Copies cp = copies(elem(0), xa, xb);
            for (int k = 1; k < n; ++k) {
                const double* cur = (k & 1) ? xa : xb;
                double* io = (k & 1) ? xb : xa;
                const double w = om[k];
                for (int e0 = 0; e0 < nel_pad; e0 += T) {
                    if (e0 + (tid & ~31) >= nel_pad) break;
                    const Elem e = elem(e0);
                    const double y = product_S(e, cur);
                    if (!e.on) continue;
                    const size_t i = (size_t)e.row * NC + e.q;
                    const double dc = cur[i], dp = k == 1 ? 0.0 : io[i];
                    const double dn = e.slot < 0 ? 0.0 : dp + w * (a.gamma64 * (fb[e0 + tid] - y) + dc - dp);
                    if (k == n - 1) xs[e0 + tid] += dn;
                    else if (single) publish(e, cp, io, (k & 1) != 0, dn);
                    else bcast(io, e.row, NC, e.q, dn);
                }
                barrier();
            }
            // u' published, then its residual and t = u^T u'
            for (int e0 = 0; e0 < nel_pad; e0 += T) {
                const Elem e = elem(e0);
                if (e.on) bcast(xa, e.row, NC, e.q, xs[e0 + tid]);
            }
            barrier();
            double v[2][CPL] = {};
            for (int e0 = 0; e0 < nel_pad; e0 += T) {
                if (e0 + (tid & ~31) >= nel_pad) break;
                const Elem e = elem(e0);
                const double y = product_S(e, xa);
                if (e.slot < 0) continue;
                const double u = *at(p.Rcur, e), x = xs[e0 + tid], r = u - y;
                *at(p.Rin, e) = r;
                *at(p.Rp, e) = x;
                v[0][0] += r * r;
                v[1][0] += u * x;
            }
            double out[2];
            sum<2>(v, out);
            if (tid == 0) sh.open = sh.bad = 0;
            __syncthreads();
            if (tid < NC) {
                sh.tsum[tid] = out[1];
                if (!isfinite(out[0])) atomicExch(&sh.bad, 1);
                if (out[0] <= a.inner_tol * a.inner_tol * sh.b2[tid]) sh.skip[tid] = 1;
                if (!sh.skip[tid]) atomicAdd(&sh.open, 1);
            }
            __syncthreads();
            if (sh.bad) return false;
            if (sh.open == 0) return true;
            if (round >= SL_SPARE + 1) return false;
        }
    }
    // one row of S x with the coefficients where they are
    __device__ __forceinline__ double product_S(const Elem& e, const double* x) const {
        const double2* mc = nullptr;
        const ushort4* ix = nullptr;
        if (a.resident && e.on) {
            mc = reinterpret_cast<const double2*>(sbuf + (size_t)optr[e.oct] * LINE) + e.s8;
            ix = reinterpret_cast<const ushort4*>(sbuf + (size_t)nsteps_all * LINE) + (size_t)iptr[e.oct] * 8 + e.s8;
        }
        return spmv64(e, ss.S64, x, mc, ix).v[0];
    }
    __device__ bool inner(int& steps) {
        if (MIXED) return inner_mixed(steps);
        return a.n > 0 ? inner_cheb64(steps) : inner_fp64(steps);
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
        if (a.blk.D) {
            if (tid < NC) sh.inv_nu[tid] = sh.cs[tid].inv_nu;
            __syncthreads();
            keep_vectors(0);
        } else {
            for (int i = tid; i < NC * kl; i += T) {
                const int c = i / kl, k = k0 + i % kl;
                if (!sh.cs[c].active) continue;
                const size_t o = (size_t)(c0 + c) * p.K + k;
                p.t[o] = cmk(0.0, 0.0);
                p.u[o] = cmk(dfun[c] * sh.cs[c].inv_nu, 0.0);
            }
        }
        barrier();   // the shifts' state is read by other CTAs (seed), and written again by its own
    }

    // ---- block mode: v_i = u'_n / nu_n of the block's step i (projected rows or
    // whole vector) into the block's store
    __device__ void keep_vectors(int i) {
        if (p.proj == PROJ_ROWS) {
            if (rank == 0)
                for (int x = tid; x < NC * p.M; x += T) {
                    const int c = x / p.M, m = x % p.M;
                    if (sh.cs[c].active && m < sh.cs[c].nfun)
                        a.blk.D[((size_t)i * p.P + c0 + c) * a.blk.rows + m] = dfun[x] * sh.inv_nu[c];
                }
        } else {
            for (int e0 = 0; e0 < nel_pad; e0 += T) {
                const Elem e = elem(e0);
                if (e.slot < 0) continue;
                const Cols<CPL> x = ldcols<CPL>(at(p.Rp, e));
#pragma unroll
                for (int j = 0; j < CPL; ++j)
                    a.blk.D[((size_t)i * p.P + c0 + e.q * CPL + j) * a.blk.rows + e.slot] =
                        x.v[j] * sh.inv_nu[e.q * CPL + j];
            }
        }
    }

    // ---- a5 + a6 for the slice's columns (k_shift_step); the shifts of every
    // column are split over the CTAs of the cluster.  One projected functional is
    // updated at once; more of them, their z-derivatives and full solutions are
    // sums of real vectors with complex coefficients, which the step only stores
    // (block mode, k_block_*)
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
        const bool inl = a.blk.D == nullptr;
        const int bi = sh.bstep;      // step of the block
        for (int i = tid; i < NC * kl; i += T) {
            const int c = i / kl, k = k0 + i % kl;
            const ColState& cs = sh.cs[c];
            const size_t o = (size_t)(c0 + c) * p.K + k;
            if (!cs.active || p.conv_iter[o] >= 0) continue;
            const size_t ob = (size_t)bi * p.P * p.K + o;
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
                a.blk.dA[ob] = dal;
                a.blk.dL[ob] = cmk(sh.Bn[c] * dinv.x, sh.Bn[c] * dinv.y);
                p.dpinv[o] = dinv;
                p.dzeta[o] = cmk(sh.Bn[c] * dal.x, sh.Bn[c] * dal.y);
            }
            if (inl) {
                const double2 u = p.u[o], un = cmul(f.l, u);
                p.t[o] = cadd(p.t[o], cmul(f.al, u));
                p.u[o] = cmk(dfun[c] * sh.inv_nu[c] + un.x, un.y);
            } else {
                a.blk.A[ob] = f.al;
                a.blk.L[ob] = f.l;
            }
            if (res <= p.tol) p.conv_iter[o] = cs.iters + 1;
            else atomicAdd(&sh.lnun[c], 1);
        }
        __syncthreads();
        if (!inl) keep_vectors(bi + 1);
        if (tid < NC) share(sh.nun, sh.lnun[tid]);
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
                share(sh.best, sh.lbest[tid]);
                share(sh.bestk, sh.lbestk[tid]);
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
        if (tid == 0) ++sh.bstep;
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
                const float* xa = reinterpret_cast<const float*>(vec);
                h = spmv_df(e, ss.Hhi, ss.Hlo, xa, xa + (size_t)nloc * NC);
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

template <bool MIXED, int NC, int CPL, bool REG>
__global__ void __launch_bounds__(SL_T, 1) k_slice(SliceDev ss, DevSystem s, PanelDev p, SliceArgs a) {
    extern __shared__ __align__(32) unsigned char smem[];
    using S = Slice<MIXED, NC, CPL, REG>;
    typename S::Sh& sh = *reinterpret_cast<typename S::Sh*>(smem);
    S sl(ss, s, p, a, sh);
    sl.CL = a.cl;
    sl.rank = blockIdx.x % a.cl;
    sl.c0 = (int)(blockIdx.x / a.cl) * NC;
    sl.tid = threadIdx.x;
    sl.T = blockDim.x;
    sl.par = 0;
    sl.oct0 = __ldg(ss.rank_oct + sl.rank);
    const int noct_l = __ldg(ss.rank_oct + sl.rank + 1) - sl.oct0;
    sl.nel = noct_l * 8 * S::LPS;
    sl.nel_pad = (sl.nel + 31) & ~31;
    sl.nloc = ss.nloc;
    sl.phase = 0;
    const SliceMem mem = slice_mem<MIXED, NC, CPL>(ss, p.M, a.n, a.resident, a.obytes, sl.T);
    sl.part = reinterpret_cast<double*>(smem + mem.part);
    sl.dfun = reinterpret_cast<double*>(smem + mem.dfun);
    sl.omega = reinterpret_cast<float*>(smem + mem.omega);
    sl.vec = smem + mem.vec;
    sl.own = smem + mem.own;
    sl.optr = reinterpret_cast<int*>(smem + mem.tab);
    sl.iptr = sl.optr + ss.max_oct + 1;
    sl.dptr = sl.iptr + ss.max_oct + 1;
    sl.dest = sl.dptr + 2 * ss.max_oct + 1;
    sl.sbuf = smem + mem.sbuf;
    sl.step0 = __ldg(ss.oct_ptr + sl.oct0);
    sl.bat0 = __ldg(ss.idx_ptr + sl.oct0);
    const int d0 = __ldg(ss.dest_ptr + 2 * sl.oct0);
    for (int i = threadIdx.x; i <= noct_l; i += sl.T) {
        sl.optr[i] = __ldg(ss.oct_ptr + sl.oct0 + i) - sl.step0;
        sl.iptr[i] = __ldg(ss.idx_ptr + sl.oct0 + i) - sl.bat0;
    }
    for (int i = threadIdx.x; i <= 2 * noct_l; i += sl.T) sl.dptr[i] = __ldg(ss.dest_ptr + 2 * sl.oct0 + i) - d0;
    const int nd = __ldg(ss.dest_ptr + 2 * (sl.oct0 + noct_l)) - d0;
    for (int i = threadIdx.x; i < nd; i += sl.T) sl.dest[i] = __ldg(ss.dest + d0 + i);
    sl.nsteps_all = __ldg(ss.oct_ptr + sl.oct0 + noct_l) - sl.step0;
    const int tid = threadIdx.x;
    for (int i = tid; i < NC; i += sl.T) sh.cs[i] = p.col[sl.c0 + i];
    for (int i = tid; i < a.n; i += sl.T) {
        if (MIXED) sl.omega[i] = a.omega[i];
        else reinterpret_cast<double*>(sl.omega)[i] = a.omega64[i];
    }
    if (tid == 0) {
        sh.open = sh.bad = sh.wanted = sh.active = 0;
        sh.bstep = a.blk.step;
    }
    __syncthreads();
    if (tid < NC && sh.cs[tid].active) atomicAdd(&sh.active, 1);
    __syncthreads();
    if (sh.active == 0) return;    // the same in every CTA of the cluster
    if (REG) {}
    else if (a.resident) sl.load_resident(noct_l);
    else if (MIXED && (tid & ~31) < sl.nel_pad) sl.ring_load(0, 0);
    sl.barrier();                  // every CTA runs before its shared memory is written
    int steps = 0, err = 0;
    bool ok = true;
    if (a.start) {
        double v[1][CPL] = {};
        for (int e0 = 0; e0 < sl.nel_pad; e0 += sl.T) {
            const Elem e = sl.elem(e0);
            if (e.slot < 0) continue;
            const Cols<CPL> u = ldcols<CPL>(sl.at(p.Rcur, e));
#pragma unroll
            for (int j = 0; j < CPL; ++j) v[0][j] += u.v[j] * u.v[j];
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
    S::cp_wait();
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

constexpr size_t SL_SMEM = 226 * 1024;   // shared memory of a CTA, at most

template <bool MIXED, int NC, int CPL>
size_t slice_smem(const SliceDev& ss, const PanelDev& p, const SliceArgs& a, int T) {
    return slice_mem<MIXED, NC, CPL>(ss, p.M, a.n, a.resident, a.obytes, T).total;
}

// One instance of the kernel: fits (fills the launch's shape) and launches.
template <bool MIXED, int NC, int CPL, bool REG>
struct Instance {
    static constexpr int LPS = NC / CPL;

    static bool fit(const SliceDev& ss, const PanelDev& p, SliceArgs& a) {
        a.nc = NC;
        a.cl = ss.cl;
        a.obytes = ss.max_len * 128 + ((ss.max_len + 2) / 4) * 64;
        a.ibase = ss.max_len * 128;
        const int rows = (ss.max_oct * 8 * LPS + 31) / 32 * 32;
        if (REG) {
            // S in the lanes' registers: one element per thread, short streams
            a.resident = 2;
            a.threads = rows;
            return rows <= SL_T && ss.max_len <= SL_RL && slice_smem<MIXED, NC, CPL>(ss, p, a, rows) <= SL_SMEM;
        }
        // S resident in shared memory with as many threads as the rows need,
        // else the ring (mixed) or S from global memory (FP64); fewer threads
        // when the ring is too large
        const int full = std::min(SL_T, rows);
        a.resident = 1;
        a.threads = full;
        if (slice_smem<MIXED, NC, CPL>(ss, p, a, full) <= SL_SMEM) return true;
        a.resident = 0;
        for (a.threads = full; a.threads >= 128; a.threads -= 32)
            if (slice_smem<MIXED, NC, CPL>(ss, p, a, a.threads) <= SL_SMEM) return true;
        return false;
    }

    // shared-memory limit raised (never lowered), clusters of 16 allowed, on the
    // current device (both are per device)
    static bool prepare(size_t sm) {
        static std::mutex mu;
        static size_t limit[64] = {0};
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) {
            cudaGetLastError();
            return false;
        }
        std::lock_guard<std::mutex> lk(mu);
        size_t& cur = limit[dev];
        if (sm <= cur) return true;
        const auto k = k_slice<MIXED, NC, CPL, REG>;
        if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm) != cudaSuccess ||
            cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) {
            cudaGetLastError();
            return false;
        }
        cur = sm;
        return true;
    }

    static void config(cudaLaunchConfig_t& cfg, cudaLaunchAttribute& at, int clusters, int cl, int threads, size_t sm) {
        cfg = cudaLaunchConfig_t{};
        cfg.gridDim = dim3((unsigned)(clusters * cl));
        cfg.blockDim = dim3((unsigned)threads);
        cfg.dynamicSmemBytes = sm;
        at.id = cudaLaunchAttributeClusterDimension;
        at.val.clusterDim.x = (unsigned)cl;
        at.val.clusterDim.y = 1;
        at.val.clusterDim.z = 1;
        cfg.attrs = &at;
        cfg.numAttrs = 1;
    }

    // clusters of this shape that the device holds at once
    static int clusters(int cl, int threads, size_t sm) {
        if (sm > SL_SMEM || !prepare(sm)) return 0;
        cudaLaunchConfig_t cfg;
        cudaLaunchAttribute at[1];
        config(cfg, at[0], 1, cl, threads, sm);
        int n = 0;
        if (cudaOccupancyMaxActiveClusters(&n, k_slice<MIXED, NC, CPL, REG>, &cfg) != cudaSuccess) {
            cudaGetLastError();
            return 0;
        }
        return n;
    }

    static bool launch(const SliceDev& ss, const DevSystem& s, const PanelDev& p, const SliceArgs& a, int ncols,
                       cudaStream_t st) {
        const size_t sm = slice_smem<MIXED, NC, CPL>(ss, p, a, a.threads);
        if (!prepare(sm)) return false;
        cudaLaunchConfig_t cfg;
        cudaLaunchAttribute at[1];
        config(cfg, at[0], (ncols + NC - 1) / NC, a.cl, a.threads, sm);
        cfg.stream = st;
        void* mark = launch_mark_begin(K_SLICE, st);
        const cudaError_t e = cudaLaunchKernelEx(&cfg, k_slice<MIXED, NC, CPL, REG>, ss, s, p, a);
        launch_mark_end(mark);
        if (e != cudaSuccess) cudaGetLastError();
        return e == cudaSuccess;
    }
};

// f<Instance>() for the instance of (precision, columns, registers)
template <class F>
bool with_instance(bool mixed, int nc, bool reg, F&& f) {
    if (mixed && reg) {
        if (nc == 2) return f(Instance<true, 2, 2, true>());
        if (nc == 4) return f(Instance<true, 4, 4, true>());
        if (nc == 8) return f(Instance<true, 8, 4, true>());
    } else if (mixed) {
        if (nc == 2) return f(Instance<true, 2, 2, false>());
        if (nc == 4) return f(Instance<true, 4, 2, false>());
        if (nc == 8) return f(Instance<true, 8, 2, false>());
    } else if (!reg) {
        if (nc == 1) return f(Instance<false, 1, 1, false>());
        if (nc == 2) return f(Instance<false, 2, 1, false>());
        if (nc == 4) return f(Instance<false, 4, 1, false>());
    }
    return false;
}

// values of the items from the 4x4 blocks of the system (src: offset in M, -1: zero)
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

// ---- block mode -----------------------------------------------------------
// The iterates of shift k after the steps 0 .. m-1 of a block, from the state
// q_0 before it, the step coefficients alpha_i, l_i and the real vectors v_i:
//     x += sum_i alpha_i q_i,   q_{i+1} = v_{i+1} + l_i q_i
//        = C_0 q_0 + sum_{i=1}^{m-1} C_i v_i,      C_m = 0, C_i = alpha_i + l_i C_{i+1},
//     q_m = E_0 q_0 + sum_{i=1}^{m} E_i v_i,        E_m = 1, E_i = l_i E_{i+1}.
// A real vector times a complex coefficient costs 2 FP64 FMAs per element and
// step instead of the 8 of the complex updates (4 instead of ~28 with the
// z-derivatives), and x, q are read and written once per block, not per step.
// FP64 arithmetic bounds both (1.7 FMA per cycle and SM on this part): 64 atoms,
// all 256 columns, 68 rows, 64 shifts with z-derivatives: 31.6 ms per call with
// updates every step, 20.4 with blocks.  In the first block q_0 = v_0.

// (alpha, l) -> (C, E) in place, one thread per (column, shift); a shift's
// steps end at its convergence
__global__ void k_block_coef(PanelDev p, SliceBlock b, int nsteps, int n0) {
    const int o = blockIdx.x * blockDim.x + threadIdx.x;
    if (o >= p.P * p.K) return;
    const int c = o / p.K;
    const size_t st = (size_t)p.P * p.K;
    const int conv = p.conv_iter[o], it = p.col[c].iters;
    int m = (conv >= 0 ? min(conv, it) : it) - n0;
    m = max(0, min(m, nsteps));
    b.count[o] = m;
    double2 C = cmk(0.0, 0.0), E = cmk(1.0, 0.0), dC = C, dE = C;
    for (int i = m - 1; i >= 0; --i) {
        const double2 al = b.A[i * st + o], l = b.L[i * st + o];
        if (p.deriv) {
            const double2 da = b.dA[i * st + o], dl = b.dL[i * st + o];
            dC = cadd(cadd(da, cmul(dl, C)), cmul(l, dC));
            dE = cadd(cmul(dl, E), cmul(l, dE));
            b.dA[i * st + o] = dC;
            b.dL[i * st + o] = dE;
        }
        C = cadd(al, cmul(l, C));
        E = cmul(l, E);
        b.A[i * st + o] = C;
        b.L[i * st + o] = E;
    }
}

// x (and q when the solve goes on) of rows [128 per CTA] and BK shifts of one
// column.  first: x = 0 and q_0 = v_0.
template <int BK, bool DERIV, bool WITHQ>
__global__ void __launch_bounds__(128) k_block_apply(PanelDev p, SliceBlock b, int first) {
    __shared__ double2 co[32][BK * (DERIV ? 2 : 1) * (WITHQ ? 2 : 1)];
    const int c = blockIdx.z, kb = blockIdx.y * BK, r = blockIdx.x * 128 + threadIdx.x;
    const int K = p.K;
    const bool full = p.proj == PROJ_NONE;
    if (p.col[c].nfun == 0 && !full) return;
    const bool on = r < (full ? p.npad : p.col[c].nfun);
    const size_t st = (size_t)p.P * K;
    constexpr int NV = (DERIV ? 2 : 1) * (WITHQ ? 2 : 1);   // C, [dC], [E, [dE]]
    int top = 0, cnt[BK];
#pragma unroll
    for (int j = 0; j < BK; ++j) {
        cnt[j] = kb + j < K ? b.count[(size_t)c * K + kb + j] : 0;
        top = max(top, cnt[j]);
    }
    double2 acc[BK][NV];
#pragma unroll
    for (int j = 0; j < BK; ++j)
#pragma unroll
        for (int v = 0; v < NV; ++v) acc[j][v] = cmk(0.0, 0.0);
    for (int i0 = 0; i0 < top; i0 += 32) {
        __syncthreads();
        for (int x = threadIdx.x; x < 32 * BK; x += 128) {
            const int i = i0 + x / BK, j = x % BK;
            // cnt[] is indexed statically only: read the count again
            const int n = kb + j < K ? b.count[(size_t)c * K + kb + j] : 0;
            const size_t o = i * st + (size_t)c * K + kb + j;
            const bool have = i < n;
            const double2 z = cmk(0.0, 0.0);
            co[x / BK][j * NV] = have ? b.A[o] : z;
            if (DERIV) co[x / BK][j * NV + 1] = have ? b.dA[o] : z;
            if (WITHQ) {
                co[x / BK][j * NV + (DERIV ? 2 : 1)] = have ? b.L[o] : z;
                if (DERIV) co[x / BK][j * NV + 3] = have ? b.dL[o] : z;
            }
        }
        __syncthreads();
        const int ie = min(32, top - i0);
        if (on)
            for (int i = i0 == 0 && !first ? 1 : 0; i < ie; ++i) {
                const double d = b.D[((size_t)(i0 + i) * p.P + c) * b.rows + r];
#pragma unroll
                for (int j = 0; j < BK; ++j)
#pragma unroll
                    for (int v = 0; v < NV; ++v) {
                        const double2 f = co[i][j * NV + v];
                        acc[j][v].x += f.x * d;
                        acc[j][v].y += f.y * d;
                    }
            }
    }
    if (!on) return;
#pragma unroll
    for (int j = 0; j < BK; ++j) {
        const int k = kb + j;
        if (k >= K) break;
        const size_t o = full ? ((size_t)k * p.npad + r) * p.XP + c : ((size_t)c * K + k) * p.M + r;
        double2* X = full ? p.X : p.t;
        double2* Q = full ? p.Pk : p.u;
        double2 x = acc[j][0], dx = DERIV ? acc[j][1 % NV] : cmk(0.0, 0.0);
        double2 q = cmk(0.0, 0.0), dq = q;
        if (WITHQ) {
            q = acc[j][(DERIV ? 2 : 1) % NV];
            if (DERIV) dq = acc[j][3 % NV];
        }
        if (cnt[j] > 0) {
            if (!first) {
                // the state before the block
                const size_t ob = (size_t)c * K + k;
                const double2 q0 = Q[o], C0 = b.A[ob];
                x = cadd(cadd(X[o], x), cmul(C0, q0));
                if (DERIV) dx = cadd(cadd(p.dt[o], dx), cadd(cmul(b.dA[ob], q0), cmul(C0, p.du[o])));
                if (WITHQ) {
                    const double2 E0 = b.L[ob];
                    if (DERIV) dq = cadd(dq, cadd(cmul(b.dL[ob], q0), cmul(E0, p.du[o])));
                    q = cadd(q, cmul(E0, q0));
                }
            }
            X[o] = x;
            if (DERIV) p.dt[o] = dx;
            if (WITHQ) {
                q.x += b.D[((size_t)cnt[j] * p.P + c) * b.rows + r];   // E_m = 1
                Q[o] = q;
                if (DERIV) p.du[o] = dq;
            }
        } else if (first) {
            X[o] = cmk(0.0, 0.0);
            if (DERIV) p.dt[o] = cmk(0.0, 0.0);
        }
    }
}

}  // namespace

// Ends a block of nsteps steps that began at outer step n0: the coefficients
// into their block form and the sums into x (and q when the solve goes on).
void launch_block_flush(const PanelDev& p, const SliceBlock& b, int nsteps, int n0, bool goes_on, cudaStream_t st) {
    void* mark = launch_mark_begin(K_FULL_UPDATE, st);
    k_block_coef<<<(p.P * p.K + 63) / 64, 64, 0, st>>>(p, b, nsteps, n0);
    launch_mark_end(mark);
    mark = launch_mark_begin(K_FULL_UPDATE, st);
    const int rows = p.proj == PROJ_NONE ? p.npad : p.M;
    constexpr int BK = 4;
    const dim3 g((rows + 127) / 128, (p.K + BK - 1) / BK, p.proj == PROJ_NONE ? p.XP : p.P);
    const int first = n0 == 0 ? 1 : 0;
    if (p.deriv && goes_on) k_block_apply<BK, true, true><<<g, 128, 0, st>>>(p, b, first);
    else if (p.deriv) k_block_apply<BK, true, false><<<g, 128, 0, st>>>(p, b, first);
    else if (goes_on) k_block_apply<BK, false, true><<<g, 128, 0, st>>>(p, b, first);
    else k_block_apply<BK, false, false><<<g, 128, 0, st>>>(p, b, first);
    launch_mark_end(mark);
}

void launch_slice_fill(const double* M, const int* src, long long n, double* m64, float* hi, float* lo, cudaStream_t st) {
    void* mark = launch_mark_begin(K_OTHER, st);
    const long long g = std::min<long long>((n + THREADS - 1) / THREADS, 1216);
    k_slice_fill<<<(unsigned)std::max<long long>(g, 1), THREADS, 0, st>>>(M, src, n, m64, hi, lo);
    launch_mark_end(mark);
}

// Whether slices of nc columns (reg: with S in registers) run on this layout;
// fills the launch's shape.
bool slice_fit(const SliceDev& ss, const PanelDev& p, int nc, bool reg, SliceArgs& a) {
    if (nc > p.P) return false;
    return with_instance(p.mixed != 0, nc, reg, [&](auto inst) { return inst.fit(ss, p, a); });
}

// Clusters of cl CTAs of `threads` threads and `smem` bytes that the device holds at once.
int slice_clusters(bool mixed, int nc, bool reg, int cl, int threads, size_t smem) {
    int n = 0;
    with_instance(mixed, nc, reg, [&](auto inst) {
        n = inst.clusters(cl, threads, smem);
        return true;
    });
    return n;
}

bool launch_slice(const SliceDev& ss, const DevSystem& s, const PanelDev& p, const SliceArgs& a, int ncols,
                  cudaStream_t st) {
    return with_instance(p.mixed != 0, a.nc, a.resident == 2,
                         [&](auto inst) { return inst.launch(ss, s, p, a, ncols, st); });
}

// Host: groups, octets and items of one system for clusters of cl CTAs (see
// the head of the file).  brow, bcol: its block rows, columns local to col0;
// orb: orbitals per atom.  The coefficients' offsets count from the system's
// first block, brow[0].
void slice_layout(int n, const int32_t* orb, const int64_t* brow, const int32_t* bcol, int32_t col0, int cl,
                  SliceHost& out) {
    struct Group {
        int atom[4];
        int rows;      // rows of the group (4: sp atom or four s atoms)
        bool sp;
        int size;      // columns that meet it
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
    std::fill(mark.begin(), mark.end(), -1);
    int64_t total = 0;
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
        total += g.size;
    }
    // consecutive groups (the caller's atom order) to the CTAs: by number, in
    // pairs, where all have about the same size (a group more than its share is a
    // warp more, and no longer one element per thread: 512 atoms on four CTAs, an
    // input on which the split by work gave one CTA 129 of 512 groups, 144.8 ->
    // 109.5 ms), else by their work; in a CTA the longest first, so that a warp's
    // octets have about one length; a CTA's odd group is paired with a filling one
    const int ng = (int)groups.size();
    int largest = 0;
    for (const Group& g : groups) largest = std::max(largest, g.size);
    const bool even = 16 * (int64_t)largest * ng <= 17 * total;
    out.rank_oct.assign(cl + 1, 0);
    std::vector<int> order;   // groups in row order, -1: filling
    int64_t acc = 0;
    for (int r = 0, k = 0; r < cl; ++r) {
        const int k0 = k;
        if (even) k = std::min(ng, (int)(2 * ((int64_t)((ng + 1) / 2) * (r + 1) / cl)));
        else
            while (k < ng && (r == cl - 1 || acc + groups[k].size / 2 <= total * (r + 1) / cl)) acc += groups[k++].size;
        const size_t o0 = order.size();
        for (int q = k0; q < k; ++q) order.push_back(q);
        std::stable_sort(order.begin() + o0, order.end(),
                         [&](int x, int y) { return groups[x].size > groups[y].size; });
        if (order.size() & 1) order.push_back(-1);
        out.rank_oct[r + 1] = (int)(order.size() / 2);
    }
    const int noct = (int)(order.size() / 2);
    out.noct = noct;
    out.cl = cl;
    out.nrows = 8 * noct;
    out.row_slot.assign(out.nrows, -1);
    std::vector<int> place((size_t)4 * n, -1);   // row of a padded slot
    std::vector<int> rank_of(2 * (size_t)noct, 0);
    for (int r = 0; r < cl; ++r)
        for (int g = 2 * out.rank_oct[r]; g < 2 * out.rank_oct[r + 1]; ++g) rank_of[g] = r;
    for (int g = 0; g < 2 * noct; ++g) {
        if (order[g] < 0) continue;
        const Group& G = groups[order[g]];
        for (int a = 0; a < G.rows; ++a) {
            const int slot = G.sp ? 4 * G.atom[0] + a : 4 * G.atom[a];
            out.row_slot[4 * g + a] = slot;
            place[slot] = 4 * g + a;
        }
    }
    // halo: the groups of other CTAs that a CTA's products meet, each with its
    // place after the CTA's own rows, and per group the CTAs that keep a copy
    std::vector<std::vector<int>> to(2 * (size_t)noct);   // rank << 16 | group there
    std::vector<int> local(2 * (size_t)noct, -1);         // of the present rank
    struct Item {
        int x;
        int src[4];
    };
    std::vector<std::vector<Item>> st((size_t)8 * noct);
    std::vector<int> pos(out.nrows, -1);
    out.nloc = 0;
    for (int r = 0; r < cl; ++r) {
        const int g0 = 2 * out.rank_oct[r], g1 = 2 * out.rank_oct[r + 1];
        std::vector<int> halo;
        int nl = g1 - g0;
        for (int g = g0; g < g1; ++g) {
            if (order[g] < 0) continue;
            const Group& G = groups[order[g]];
            for (int a = 0; a < (G.sp ? 1 : G.rows); ++a)
                for (int64_t b = brow[G.atom[a]]; b < brow[G.atom[a] + 1]; ++b) {
                    const int h = place[4 * (bcol[b] - col0)] >> 2;
                    if (rank_of[h] == r || local[h] >= 0) continue;
                    local[h] = nl++;
                    halo.push_back(h);
                }
        }
        for (int h : halo) to[h].push_back(r << 16 | local[h]);
        out.nloc = std::max(out.nloc, 4 * nl);
        for (int g = g0; g < g1; ++g) {
            for (int a = 0; a < 4; ++a) st[4 * g + a].push_back({4 * (g - g0) + a, {-1, -1, -1, -1}});   // item 0: the own row
            if (order[g] < 0) continue;
            const Group& G = groups[order[g]];
            std::vector<Item> list;
            std::vector<int> seen;
            for (int a = 0; a < (G.sp ? 1 : G.rows); ++a)
                for (int64_t b = brow[G.atom[a]]; b < brow[G.atom[a] + 1]; ++b) {
                    const int j = bcol[b] - col0;
                    for (int e = 0; e < orb[j]; ++e) {
                        const int row = place[4 * j + e];
                        if (pos[row] < 0) {
                            pos[row] = (int)list.size();
                            seen.push_back(row);
                            list.push_back({row, {-1, -1, -1, -1}});
                        }
                        Item& it = list[pos[row]];
                        if (G.sp)
                            for (int q = 0; q < 4; ++q) it.src[q] = (int)(16 * (b - brow[0]) + 4 * q + e);
                        else it.src[a] = (int)(16 * (b - brow[0]) + e);
                    }
                }
            for (int row : seen) pos[row] = -1;
            for (Item& it : list) {
                const int h = it.x >> 2, e = it.x & 3;
                const bool own = h == g;
                it.x = 4 * (rank_of[h] == r ? h - g0 : local[h]) + e;
                if (own) st[4 * g + e].front() = it;
                else st[4 * g + e].push_back(it);
            }
        }
        for (int h : halo) local[h] = -1;
    }
    // order of the second group's items: at each step of the octet a place of
    // the other parity than the first group's, so that rows of 16 bytes (four
    // columns) of the two groups lie in different banks where that is possible
    for (int o = 0; o < noct; ++o)
        for (int a = 0; a < 4; ++a) {
            const std::vector<Item>& A = st[8 * o + a];
            std::vector<Item>& B = st[8 * o + 4 + a];
            std::vector<Item> half[2];
            for (size_t k = B.size(); k-- > 1;) half[(B[k].x >> 2) & 1].push_back(B[k]);
            for (size_t k = 1; k < B.size(); ++k) {
                int want = k < A.size() ? 1 - ((A[k].x >> 2) & 1) : 0;
                if (half[want].empty()) want = 1 - want;
                B[k] = half[want].back();
                half[want].pop_back();
            }
        }
    out.dest_ptr.assign(2 * (size_t)noct + 1, 0);
    out.dest.clear();
    for (int g = 0; g < 2 * noct; ++g) {
        out.dest.insert(out.dest.end(), to[g].begin(), to[g].end());
        out.dest_ptr[g + 1] = (int)out.dest.size();
    }
    out.oct_ptr.assign(noct + 1, 0);
    out.idx_ptr.assign(noct + 1, 0);
    out.max_len = 1;
    // The octets that a warp works on (four, two or one) get one length where
    // that adds at most a sixteenth to their steps: lanes that end apart run the
    // item loop's remainders one after another, and an FP64 instruction takes a
    // warp ~75 cycles of its unit.  On silicon with a few neighbours beyond the
    // cutoff, where lengths are 17 and 15 or 16: FP64, one column of 64 atoms
    // 44.4 -> 35.7 ms, 48 of 216 atoms 105.9 -> 94.7; mixed, 13 of 144 atoms 34.9
    // -> 33.6.  Water's lengths lie further apart (at one length everywhere, a
    // charge-self-consistent call of 48 molecules took 44.3 instead of 42.0 ms).
    for (int r = 0; r < cl; ++r)
        for (int w = out.rank_oct[r]; w < out.rank_oct[r + 1]; w += 4) {
            const int w1 = std::min(w + 4, out.rank_oct[r + 1]);
            size_t len[4] = {1, 1, 1, 1}, most = 1, sum = 0;
            for (int o = w; o < w1; ++o) {
                for (int q = 0; q < 8; ++q) len[o - w] = std::max(len[o - w], st[8 * o + q].size());
                most = std::max(most, len[o - w]);
                sum += len[o - w];
            }
            const bool one = 16 * most * (w1 - w) <= 17 * sum;
            out.max_len = std::max(out.max_len, (int)most);
            for (int o = w; o < w1; ++o) {
                const int n = (int)(one ? most : len[o - w]);
                out.oct_ptr[o + 1] = out.oct_ptr[o] + n;
                out.idx_ptr[o + 1] = out.idx_ptr[o] + (n - 1 + 3) / 4;
            }
        }
    out.max_oct = out.max_steps = out.max_bat = out.max_dest = 0;
    for (int r = 0; r < cl; ++r) {
        const int a = out.rank_oct[r], b = out.rank_oct[r + 1];
        out.max_oct = std::max(out.max_oct, b - a);
        out.max_steps = std::max(out.max_steps, out.oct_ptr[b] - out.oct_ptr[a]);
        out.max_bat = std::max(out.max_bat, out.idx_ptr[b] - out.idx_ptr[a]);
        out.max_dest = std::max(out.max_dest, out.dest_ptr[2 * b] - out.dest_ptr[2 * a]);
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
                        (unsigned short)(have ? v[k].x : v[0].x);
            }
            // the last batch's unused places: the own row as well (never read)
            for (int k = len; (k - 1) % 4 != 0; ++k)
                out.idx[4 * ((size_t)(out.idx_ptr[o] + (k - 1) / 4) * 8 + q) + (k - 1) % 4] = (unsigned short)v[0].x;
        }
}

}  // namespace tb
