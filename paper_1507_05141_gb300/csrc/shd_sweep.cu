// Stage a4 in single precision with the linear integrator (Sec. 2 eq:shdom,
// Sec. 2.1 eq:time): the plane sweep with a column of rows per thread, on one
// CTA a plane or a thread-block cluster, its schedules and their timed choice.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <type_traits>
#include <vector>

#include "shd_internal.cuh"

namespace cg = cooperative_groups;

namespace shd {

// asynchronous copy of 16 bytes from global to shared memory
__device__ __forceinline__ void cp_async16(void *smem, const void *gmem)
{
    const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(sa), "l"(gmem));
}

// -------------------------------------------------------------------------
// a4, single precision, linear integrator: columns of rows in registers.
// A CTA (or, with a cluster of C CTAs, each CTA of it) sweeps a block of
// rows of every plane.  A thread owns R consecutive rows of one column of
// the block, in upwind order, and keeps their state of the previous plane
// (I, S~, chi~) in registers.  Per plane it publishes that state once in
// shared memory (vectors of its rows) and reads back only what other threads
// own: the rows of the neighbouring upwind column, and the halo row before
// its first row in both columns (thread t's own column one row block back is
// thread t - n2).  Per node that is one store and 1 + 2/R loads of a state
// instead of one store and four loads (104 B of shared traffic an update in
// a node-a-thread layout, about 60 at R = 4).  (I, S~) travel as packed
// pairs; each lane rounds as the scalar form does.
//
// The inputs of plane s+1 (I^n, eta, chi) stream into a two-stage
// shared-memory ring while plane s is computed: 16-byte cp.async copies; a
// plane that does not start on a 16-byte boundary is copied as its aligned
// cover and read from its offset.  With the chi0 table (chi0L, aligned
// planes) chi comes from chi_lab only for the 4-node pieces that hold a
// moving node.  Two exchange buffers alternate, so one block barrier per
// plane suffices: it makes plane s-1's state and the copies of plane s
// visible, and every read of the buffer plane s overwrites is done by then.
// Issue slots bound it as much as memory: the ring and exchange strides are
// compile-time (NS threads), so that every shared access is a thread
// constant plus an immediate, and the plane loop is unrolled over the two
// parities (97 instructions an update in the node-a-thread layout, 66 here).
// NS = 0 takes the strides at run time (rows that do not divide the threads,
// at the least shared memory).  64^3, 16 groups, 512 ordinates: 8.08 ms a
// sweep before, 5.9 now, 5.5 TB/s of DRAM traffic, 0.81 of the copy rate.
//
// In a cluster the halo row of a CTA's first row block is the last row of
// the upwind CTA, which sends it: each thread of its last row block writes
// 16 bytes into one of four halo slots of the downwind CTA by st.async,
// counted on that CTA's mbarrier, and only the first row block's warps there
// wait for it.  A slot is handed back by a remote arrive two planes later,
// so the CTAs of a cluster run as a pipeline a plane or so apart and no
// plane pays a cluster barrier, its release fence and its wait (128^3, 3
// groups: 15.5 ms a sweep with a barrier a plane, 14.4 now, with chi at rest
// from the table; the two CTAs an SM need 106.6 KB each, so the exchange
// holds no separate halo rows).
// Waits are bounded: on timeout the thread raises *err and runs on.
//
// The arithmetic of a node does not depend on R, V, the threads or the
// cluster, so every schedule gives the same bits.
// -------------------------------------------------------------------------
// reals by which p lies past the 16-byte boundary below it (p 4-byte aligned)
__device__ __forceinline__ int shift16(const float *p)
{
    return (int)((reinterpret_cast<unsigned long long>(p) >> 2) & 3ull);
}

// One exchange buffer of `ns` threads (ns a multiple of 4): the (I, S~) of a
// thread's R rows as float4 row pairs (and a float2 for an odd last row),
// then the chi~ as float4 / float2 / float.
template <int R>
struct ColExchange {
    static constexpr int kReals = 3 * R;  // per thread
    float *b;
    int ns;
    __device__ __forceinline__ void put(int t, const float2 (&v)[R], const float (&c)[R]) const
    {
#pragma unroll
        for (int g = 0; g < R / 2; ++g)
            reinterpret_cast<float4 *>(b + 4 * g * ns)[t] = make_float4(v[2 * g].x, v[2 * g].y, v[2 * g + 1].x, v[2 * g + 1].y);
        if constexpr (R & 1) reinterpret_cast<float2 *>(b + 2 * (R - 1) * ns)[t] = v[R - 1];
        float *bc = b + 2 * R * ns;
#pragma unroll
        for (int g = 0; g < R / 4; ++g)
            reinterpret_cast<float4 *>(bc + 4 * g * ns)[t] = make_float4(c[4 * g], c[4 * g + 1], c[4 * g + 2], c[4 * g + 3]);
        constexpr int q = R / 4 * 4;
        if constexpr (R & 2) reinterpret_cast<float2 *>(bc + q * ns)[t] = make_float2(c[q], c[q + 1]);
        if constexpr (R & 1) bc[(R - 1) * ns + t] = c[R - 1];
    }
    __device__ __forceinline__ void get(int t, float2 (&v)[R], float (&c)[R]) const
    {
#pragma unroll
        for (int g = 0; g < R / 2; ++g) {
            const float4 x = reinterpret_cast<const float4 *>(b + 4 * g * ns)[t];
            v[2 * g] = make_float2(x.x, x.y);
            v[2 * g + 1] = make_float2(x.z, x.w);
        }
        if constexpr (R & 1) v[R - 1] = reinterpret_cast<const float2 *>(b + 2 * (R - 1) * ns)[t];
        const float *bc = b + 2 * R * ns;
#pragma unroll
        for (int g = 0; g < R / 4; ++g) {
            const float4 x = reinterpret_cast<const float4 *>(bc + 4 * g * ns)[t];
            c[4 * g] = x.x; c[4 * g + 1] = x.y; c[4 * g + 2] = x.z; c[4 * g + 3] = x.w;
        }
        constexpr int q = R / 4 * 4;
        if constexpr (R & 2) {
            const float2 x = reinterpret_cast<const float2 *>(bc + q * ns)[t];
            c[q] = x.x; c[q + 1] = x.y;
        }
        if constexpr (R & 1) c[R - 1] = bc[(R - 1) * ns + t];
    }
    // thread t's last row
    __device__ __forceinline__ float2 last_is(int t) const
    {
        if constexpr (R & 1) return reinterpret_cast<const float2 *>(b + 2 * (R - 1) * ns)[t];
        else return reinterpret_cast<const float2 *>(b + 2 * (R - 2) * ns)[2 * t + 1];
    }
    __device__ __forceinline__ float last_c(int t) const
    {
        const float *bc = b + 2 * R * ns;
        if constexpr (R & 1) return bc[(R - 1) * ns + t];
        else if constexpr (R & 2) return bc[(R - 2) * ns + 2 * t + 1];
        else return bc[(R - 4) * ns + 4 * t + 3];
    }
};

// ---- the cluster's halo channel --------------------------------------------
// (Waits acquire at cluster scope: a slot's data are another CTA's.  A hand-back
// publishes nothing, it only follows this CTA's reads of the slot, done at the
// block barrier before it; a cluster-scope release there would also wait for the
// plane's global stores: 128^3, 3 groups, 14.4 ms a sweep, 15.2 with it.)
constexpr int kHaloShift = 2;  // log2 of the slots: 4, or 2 where the planes' columns leave no room for them
constexpr long long kHaloWaitLimit = 1LL << 22;  // mbarrier polls before giving up (about a second)

__device__ __forceinline__ uint32_t remote_addr(uint32_t local, int rank)
{
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;\n" : "=r"(r) : "r"(local), "r"(rank));
    return r;
}
__device__ __forceinline__ bool halo_try(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile("{\n .reg .pred p;\n mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n"
                 " selp.u32 %0, 1, 0, p;\n}\n"
                 : "=r"(ok)
                 : "r"(bar), "r"(parity)
                 : "memory");
    return ok != 0;
}
__device__ __forceinline__ void halo_wait(uint32_t bar, uint32_t parity, bool &dead, int *err)
{
    if (dead) return;
    for (long long i = 0; i < kHaloWaitLimit; ++i)
        if (halo_try(bar, parity)) return;
    dead = true;
    atomicExch(err, 1);
}

// One (ordinate, group) pair.  V: column passes of a plane with more columns
// than threads (thread t also plays threads t + blockDim.x, ...).  NS: the
// exchange's threads at compile time (0: ns_rt), the ring then NS R + 8 reals
// an array (else ps_rt); hs_rt: the halo slots' columns, hsh_rt: log2 of their
// number (NS: kHaloShift).  tune_col >= 0
// (schedule timing only): into column tune_col of a scratch intensity [.][Nc].
// MEM: A lies in shared memory and is read again for every plane (a batch's
// descriptor: its pointers would not fit the registers, where a launch of its
// own has them as constant operands).
struct SweepArrays {
    float *I;
    const float *eta, *chi, *chi0L;
    const unsigned long long *mbits;
};
template <class Q>
__device__ __forceinline__ Q array_of(const Q &p)
{
    return *const_cast<const volatile Q *>(&p);
}

template <int R, int V, int NS, bool CL, bool FLAT, bool MEM>
__device__ __forceinline__ void sweep_pair_rays(const Prob<float> &P, const SweepArrays &A, int npc, int nwin, int pair,
                                               long long tune_col, int ps_rt, int ns_rt, int hs_rt, int hsh_rt, bool wide,
                                               int *err, unsigned char *smem_raw)
{
    const int k = pair / P.G;
    const int g = pair - k * P.G;
    const Ordinate &o = P.ord[k];
    const int dims[3] = {P.nx, P.ny, P.nz};
    const int od = o.d, s1 = o.s1, s2 = o.s2;
    const bool fwd = o.sd > 0;
    const int nd = dims[od], n1 = dims[o.e1], n2 = dims[o.e2];
    const int plane = n1 * n2;
    const int tid = threadIdx.x, nthr = blockDim.x;
    const int ns = NS ? NS : ns_rt, pstride = NS ? NS * R + 8 : ps_rt;
    const int xsize = ns * ColExchange<R>::kReals;
    float *const ring = reinterpret_cast<float *>(smem_raw);  // [2][3][pstride]
    float *const xbuf = ring + 6 * pstride;                   // [2][xsize]
    // cluster: halo slots [slots][hs] float4, then full and free barriers
    const int hsh = NS ? kHaloShift : hsh_rt, slots = 1 << hsh;
    float4 *const halo = reinterpret_cast<float4 *>(xbuf + 2 * xsize);
    uint64_t *const hbar = reinterpret_cast<uint64_t *>(halo + slots * hs_rt);
    // this CTA's rows
    int row0 = 0, nrows = n1, up = -1, down = -1;
    if constexpr (CL) {
        cg::cluster_group cl = cg::this_cluster();
        const int C = (int)cl.num_blocks(), crank = (int)cl.block_rank();
        // ceil(n1 / C), rounded up so every CTA's block starts on a 16-byte boundary
        int rows_cta = (n1 + C - 1) / C;
        const int q4 = (n2 & 3) == 0 ? 1 : ((n2 & 1) == 0 ? 2 : 4);
        rows_cta = (rows_cta + q4 - 1) / q4 * q4;
        row0 = crank * rows_cta;
        nrows = row0 >= n1 ? 0 : (n1 - row0 < rows_cta ? n1 - row0 : rows_cta);
        const int used = (n1 + rows_cta - 1) / rows_cta;  // CTAs that have rows
        if (s1 != 0 && nrows > 0) {
            up = crank - s1;
            down = crank + s1;
            if (up < 0 || up >= used) up = -1;
            if (down < 0 || down >= used) down = -1;
        }
        if (tid == 0) {
            for (int i = 0; i < 2 * slots; ++i)
                asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"((uint32_t)__cvta_generic_to_shared(hbar + i))
                             : "memory");
            asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
            if (up >= 0)
                for (int i = 0; i < slots; ++i)
                    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(
                                     (uint32_t)__cvta_generic_to_shared(hbar + i)),
                                 "r"(16 * n2)
                                 : "memory");
        }
        asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;\n" ::: "memory");
    }
    const int nloc = nrows * n2, j0 = row0 * n2;
    const long long base = ((long long)k * P.G + g) * P.Nc;
    const bool table = A.chi0L != nullptr;
    auto I_of = [&, I = MEM ? nullptr : (tune_col >= 0 ? A.I + (tune_col * P.Nc - base) : A.I)]() -> float * {
        if constexpr (MEM) return array_of(A.I);
        else return I;
    };
    auto eta_of = [&, e = MEM ? nullptr : A.eta]() -> const float * {
        if constexpr (MEM) return array_of(A.eta);
        else return e;
    };
    auto chi_of = [&, e = MEM ? nullptr : A.chi]() -> const float * {
        if constexpr (MEM) return array_of(A.chi);
        else return e;
    };
    const long long c0off = ((long long)od * P.G + g) * P.Nc;
    auto chi0_of = [&, e = MEM || !table ? nullptr : A.chi0L + c0off]() -> const float * {
        if constexpr (MEM) return array_of(A.chi0L) + c0off;
        else return e;
    };
    const size_t mb0 = (size_t)od * nwin * npc;
    auto bits_of = [&, e = MEM || !table ? nullptr : A.mbits + mb0]() -> const unsigned long long * {
        if constexpr (MEM) return array_of(A.mbits) + mb0;
        else return e;
    };
    const float fr1 = (float)o.fr1, fr2 = (float)o.fr2, hs = (float)o.s * 0.5f, kap = P.kappa;
    const float w00 = (1.f - fr1) * (1.f - fr2), w10 = fr1 * (1.f - fr2), w01 = (1.f - fr1) * fr2, w11 = fr1 * fr2;
    const float bc_iso = P.bc_mode == SHD_BC_ISO ? P.bc[g] : 0.f;
    const bool bc_full = P.bc_mode == SHD_BC_FULL;

    // thread t (pass v: t + v nthr) owns rows rb R .. rb R + nv - 1, in upwind
    // order, of column i2: offset off + q dr in the CTA's block of the plane
    // (rows past nv, computed but never stored, repeat the last one's inputs)
    const int nb = (nrows + R - 1) / R, nact = nb * n2;
    const bool exact = nb * R == nrows;  // every thread has R rows
    const int dr = s1 >= 0 ? n2 : -n2;
    int off[V][R], slot_n[V], slot_h[V], nv[V];
    unsigned face[V];
    bool act[V], first_rb[V], last_rb[V];
#pragma unroll
    for (int v = 0; v < V; ++v) {
        const int t = tid + v * nthr;
        act[v] = t < nact;
        const int rb = act[v] ? t / n2 : 0, i2 = act[v] ? t - rb * n2 : 0;
        nv[v] = act[v] ? (nrows - rb * R < R ? nrows - rb * R : R) : 0;
        const int off0 = (s1 >= 0 ? rb * R : nrows - 1 - rb * R) * n2 + i2;
#pragma unroll
        for (int q = 0; q < R; ++q) off[v][q] = off0 + (q < nv[v] || nv[v] == 0 ? (nv[v] == 0 ? 0 : q) : nv[v] - 1) * dr;
        const bool edge2 = s2 != 0 && i2 == (s2 > 0 ? 0 : n2 - 1);
        face[v] = edge2 ? ~0u : ((s1 != 0 && rb == 0 && up < 0) ? 1u : 0u);
        // the neighbouring column's thread (this one on the inflow edge: not used there)
        slot_n[v] = edge2 ? t : t - s2;
        // the thread before this one in its column (itself on the first rows)
        slot_h[v] = rb > 0 ? -n2 : 0;
        first_rb[v] = CL && act[v] && rb == 0 && up >= 0;
        last_rb[v] = CL && act[v] && rb == nb - 1 && down >= 0;
    }
    bool dead = false;  // a halo wait ran out
    // the moving-node bits of this thread's chi pieces (at most MP pieces of
    // 4 nodes) for the current 64-plane window, reloaded when it changes
    constexpr int MP = (R * V + 3) / 4;
    unsigned long long mw[MP];
    int mwin = -1;

    auto issue = [&](int step, float *r) {
        if (step < nd && nrows > 0) {
            const int id = fwd ? step : nd - 1 - step;
            const long long pb = base + (long long)id * plane + j0;
            const float *I = I_of(), *eta = eta_of(), *chi = chi_of();
            if (!table) {
                const int aI = shift16(I + pb), aE = shift16(eta + pb), aC = shift16(chi + pb);
                const float *gI = I + pb - aI, *gE = eta + pb - aE, *gC = chi + pb - aC;
                const int nI = (aI + nloc + 3) >> 2, nE = (aE + nloc + 3) >> 2, nC = (aC + nloc + 3) >> 2;
                for (int q = tid; q < nI; q += nthr) cp_async16(&r[q * 4], gI + q * 4);
                for (int q = tid; q < nE; q += nthr) cp_async16(&r[pstride + q * 4], gE + q * 4);
                for (int q = tid; q < nC; q += nthr) cp_async16(&r[2 * pstride + q * 4], gC + q * 4);
            } else {
                const int np = nloc / 4;  // 16-byte pieces per array (aligned planes)
                if ((id >> 6) != mwin) {
                    mwin = id >> 6;
                    const unsigned long long *mb = bits_of();
#pragma unroll
                    for (int i = 0; i < MP; ++i) {
                        const int q = tid + i * nthr;
                        mw[i] = q < np ? mb[(size_t)mwin * npc + (j0 >> 2) + q] : 0ull;
                    }
                }
                const float *c0 = chi0_of() + (long long)id * plane + j0;
#pragma unroll
                for (int i = 0; i < MP; ++i) {
                    const int q = tid + i * nthr;
                    if (q >= np) break;
                    cp_async16(&r[q * 4], &I[pb + q * 4]);
                    cp_async16(&r[pstride + q * 4], &eta[pb + q * 4]);
                    const float *src = ((mw[i] >> (id & 63)) & 1ull) ? chi + pb + q * 4 : c0 + q * 4;
                    cp_async16(&r[2 * pstride + q * 4], src);
                }
            }
        }
        asm volatile("cp.async.commit_group;\n" ::);
    };

    float2 a[V][R];  // (I, S~) of the thread's rows on the previous plane
    float ac[V][R];  // chi~
#pragma unroll
    for (int v = 0; v < V; ++v)
#pragma unroll
        for (int q = 0; q < R; ++q) {
            a[v][q] = make_float2(0.f, 0.f);
            ac[v][q] = 0.f;
        }

    // plane `step` of parity PAR
    auto plane_of = [&](int step, auto par_c, auto first_c) {
        constexpr int PAR = decltype(par_c)::value;
        constexpr bool first = decltype(first_c)::value;
        asm volatile("cp.async.wait_group 0;\n" ::);
        __syncthreads();
        issue(step + 1, ring + (1 - PAR) * 3 * pstride);
        const int id = fwd ? step : nd - 1 - step;
        const long long pb = base + (long long)id * plane + j0;
        // the three arrays share the plane's offset in its aligned cover (when
        // timing, the scratch intensity's may differ: any finite value serves)
        const float *rI = ring + PAR * 3 * pstride + (table ? 0 : shift16(eta_of() + pb));
        const float *rE = rI + pstride, *rC = rI + 2 * pstride;
        const ColExchange<R> xp{xbuf + (1 - PAR) * xsize, ns}, xn{xbuf + PAR * xsize, ns};
        if constexpr (CL) {
            // the reads of halo slot step - 2 are done: hand it back
            if (up >= 0 && tid == 0 && step >= 2) {
                const int h = (step - 2) & (slots - 1);
                if (step - 2 + slots <= nd - 2) {
                    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(
                                     (uint32_t)__cvta_generic_to_shared(hbar + h)),
                                 "r"(16 * n2)
                                 : "memory");
                    asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];\n" ::"r"(
                                     remote_addr((uint32_t)__cvta_generic_to_shared(hbar + slots + h), up))
                                 : "memory");
                }
            }
        }
#pragma unroll
        for (int v = 0; v < V; ++v) {
            if (!act[v]) break;
            const int t = tid + v * nthr;
            float2 u[R];
            float x[R], st[R], ct[R];
            if constexpr (!first) {
                float2 bn[R];
                float bc[R];
                xp.get(slot_n[v], bn, bc);
                float2 ha = make_float2(0.f, 0.f), hb = ha;
                float hac = 0.f, hbc = 0.f;
                if constexpr (!FLAT) {
                    if (CL && first_rb[v]) {
                        const int h = (step - 1) & (slots - 1);
                        halo_wait((uint32_t)__cvta_generic_to_shared(hbar + h),
                                  (uint32_t)(((step - 1) >> hsh) & 1), dead, err);
                        const float4 A = halo[h * hs_rt + t], B = halo[h * hs_rt + slot_n[v]];
                        ha = make_float2(A.x, A.y);
                        hac = A.z;
                        hb = make_float2(B.x, B.y);
                        hbc = B.z;
                    } else {
                        ha = xp.last_is(t + slot_h[v]);
                        hb = xp.last_is(slot_n[v] + slot_h[v]);
                        hac = xp.last_c(t + slot_h[v]);
                        hbc = xp.last_c(slot_n[v] + slot_h[v]);
                    }
                }
#pragma unroll
                for (int q = 0; q < R; ++q) {
                    // the row one step upwind in this column and the neighbouring one
                    constexpr int back = FLAT ? 0 : 1;
                    const bool own = FLAT || q > 0;
                    const int p = q >= back ? q - back : 0;
                    const float2 a1 = own ? a[v][p] : ha, b1 = own ? bn[p] : hb;
                    const float c1 = own ? ac[v][p] : hac, d1 = own ? bc[p] : hbc;
                    float2 r = __fmul2_rn(make_float2(w00, w00), a[v][q]);
                    r = __ffma2_rn(make_float2(w10, w10), a1, r);
                    r = __ffma2_rn(make_float2(w01, w01), bn[q], r);
                    u[q] = __ffma2_rn(make_float2(w11, w11), b1, r);
                    x[q] = fmaf(w11, d1, fmaf(w01, bc[q], fmaf(w10, c1, w00 * ac[v][q])));
                }
            }
#pragma unroll
            for (int q = 0; q < R; ++q) {
                const float In = rI[off[v][q]];
                ct[q] = rC[off[v][q]] + kap;
                st[q] = ct[q] > 0.f ? fmaf(kap, In, rE[off[v][q]]) * hw_rcp(ct[q]) : 0.f;
            }
            if constexpr (first) {
#pragma unroll
                for (int q = 0; q < R; ++q) u[q].x = bc_iso;
            } else {
                float xm = 1e30f, xM = 0.f;
#pragma unroll
                for (int q = 0; q < R; ++q) {
                    x[q] = hs * (x[q] + ct[q]);
                    xm = fminf(xm, x[q]);
                    xM = fmaxf(xM, x[q]);
                }
                if (xm >= 0.5f && xM <= kTauPlain) {
                    // every row above the weights' series (a time step's
                    // kappa s is at least 2 at c dt = half a node spacing) and
                    // within the plain exponential
#pragma unroll
                    for (int q = 0; q < R; ++q) {
                        const float e = hw_exp2(-x[q] * kLog2eF);
                        const float a0 = (1.f - e) * hw_rcp(x[q]);
                        u[q].x = fmaf(u[q].y, a0 - e, fmaf(st[q], 1.f - a0, u[q].x * e));
                    }
                } else {
#pragma unroll
                    for (int q = 0; q < R; ++q) {
                        float e, wp, wu;
                        if (wide) sc_weights<float>(x[q], e, wp, wu);
                        else sc_weights_narrow_x2(x[q], e, wp, wu);
                        u[q].x = fmaf(u[q].y, wu, fmaf(st[q], wp, u[q].x * e));
                    }
                }
                if (face[v]) {
#pragma unroll
                    for (int q = 0; q < R; ++q)
                        if ((face[v] >> q) & 1u) u[q].x = bc_iso;
                }
            }
            if (bc_full) {
#pragma unroll
                for (int q = 0; q < R; ++q)
                    if (q < nv[v] && (first || ((face[v] >> q) & 1u))) u[q].x = P.bc[pb + off[v][q]];
            }
#pragma unroll
            for (int q = 0; q < R; ++q) {
                a[v][q] = make_float2(u[q].x, st[q]);
                ac[v][q] = ct[q];
            }
            xn.put(t, a[v], ac[v]);
            if (CL && last_rb[v]) {
                float2 hv = a[v][R - 1];
                float hc = ac[v][R - 1];
                if (!exact) {
#pragma unroll
                    for (int q = 0; q < R - 1; ++q)
                        if (q == nv[v] - 1) {
                            hv = a[v][q];
                            hc = ac[v][q];
                        }
                }
                if (step <= nd - 2) {
                    const int h = step & (slots - 1);
                    if (step >= slots)
                        halo_wait((uint32_t)__cvta_generic_to_shared(hbar + slots + h),
                                  (uint32_t)(((step >> hsh) - 1) & 1), dead, err);
                    asm volatile(
                        "st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];\n" ::"r"(
                            remote_addr((uint32_t)__cvta_generic_to_shared(halo + h * hs_rt + t - (nb - 1) * n2), down)),
                        "r"(__float_as_uint(hv.x)), "r"(__float_as_uint(hv.y)), "r"(__float_as_uint(hc)), "r"(0u),
                        "r"(remote_addr((uint32_t)__cvta_generic_to_shared(hbar + h), down))
                        : "memory");
                }
            }
            float *const ig = I_of() + pb;
            if (exact) {
#pragma unroll
                for (int q = 0; q < R; ++q) ig[off[v][q]] = u[q].x;
            } else {
#pragma unroll
                for (int q = 0; q < R; ++q)
                    if (q < nv[v]) ig[off[v][q]] = u[q].x;
            }
        }
    };

    using I0c = std::integral_constant<int, 0>;
    using I1c = std::integral_constant<int, 1>;
    if (!CL || nrows > 0) {
        issue(0, ring);
        plane_of(0, I0c{}, std::true_type{});
        for (int step = 1; step < nd; step += 2) {
            plane_of(step, I1c{}, std::false_type{});
            if (step + 1 < nd) plane_of(step + 1, I0c{}, std::false_type{});
        }
        asm volatile("cp.async.wait_group 0;\n" ::);
    }
    if constexpr (CL)  // the peers' arrivals at this CTA's barriers have landed
        asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;\n" ::: "memory");
}

// FLAT: the ray has no component along the rows; another row's state, though
// its weight is 0, must not enter then (it may be infinite).  Code of its own:
// as a branch in the loop it cost every ray 1.5 to 4 % of the sweep.
template <int R, int V, int NS, bool CL, bool MEM = false>
__device__ __forceinline__ void sweep_pair_col(const Prob<float> &P, const SweepArrays &A, int npc, int nwin, int pair,
                                               long long tune_col, int ps_rt, int ns_rt, int hs_rt, int hsh_rt, bool wide,
                                               int *err, unsigned char *smem_raw)
{
    if (P.ord[pair / P.G].s1 == 0)
        sweep_pair_rays<R, V, NS, CL, true, MEM>(P, A, npc, nwin, pair, tune_col, ps_rt, ns_rt, hs_rt, hsh_rt, wide, err,
                                                 smem_raw);
    else
        sweep_pair_rays<R, V, NS, CL, false, MEM>(P, A, npc, nwin, pair, tune_col, ps_rt, ns_rt, hs_rt, hsh_rt, wide, err,
                                                  smem_raw);
}

// One CTA a plane.  NT bounds the threads (the launch takes as many as the
// planes' columns need); two CTAs an SM at 512, four at 256, 64 registers a
// thread; R above 4 takes half as many and more registers.
constexpr int col_min_ctas(int NT, int R)
{
    return NT >= 768 ? 1 : (R > 4 ? 512 / NT : 1024 / NT);
}

template <int R, int V, int NT, int NS>
__global__ void __launch_bounds__(NT, col_min_ctas(NT, R)) k_sweep_col(Prob<float> P, float *__restrict__ I,
                                                   const float *__restrict__ eta, const float *__restrict__ chi,
                                                   const float *__restrict__ chi0L,
                                                   const unsigned long long *__restrict__ mbits, int npc, int nwin,
                                                   int pstride, int ns, int hs, int hsh, int wide, int *err, int first,
                                                   int tune_stride)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    // CTA b sweeps pair first + b; with tune_stride > 0 (schedule timing only)
    // pair (first + b) * tune_stride, its intensity in that column of a scratch
    // array I [.][Nc]
    const int idx = first + (int)blockIdx.x, pair = tune_stride > 0 ? idx * tune_stride : idx;
    sweep_pair_col<R, V, NS, false>(P, SweepArrays{I, eta, chi, chi0L, mbits}, npc, nwin, pair,
                                                 tune_stride > 0 ? (long long)idx : -1, pstride, ns, hs, hsh,
                                                 wide != 0, err, smem_raw);
}

// The plane split over a cluster of C CTAs.
template <int R, int V, int NT, int NS>
__global__ void __launch_bounds__(NT, col_min_ctas(NT, R)) k_sweep_cl(Prob<float> P, float *__restrict__ I,
                                                   const float *__restrict__ eta, const float *__restrict__ chi,
                                                   const float *__restrict__ chi0L,
                                                   const unsigned long long *__restrict__ mbits, int npc, int nwin,
                                                   int pstride, int ns, int hs, int hsh, int wide, int *err, int first,
                                                   int tune_stride)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int idx = first + (int)blockIdx.x / (int)cg::this_cluster().num_blocks();
    const int pair = tune_stride > 0 ? idx * tune_stride : idx;
    sweep_pair_col<R, V, NS, true>(P, SweepArrays{I, eta, chi, chi0L, mbits}, npc, nwin, pair,
                                                tune_stride > 0 ? (long long)idx : -1, pstride, ns, hs, hsh, wide != 0,
                                                err, smem_raw);
}

// The plane sweeps of a batch of problems in one persistent launch: CTAs
// walk the work list of every problem's (ordinate, group) pairs (problem p
// owns items [item0, item0 + N G)), each item as k_sweep_col sweeps it, with
// the problem's own fields and arrays.  One launch per class of problems
// that share the kernel's variant.
template <int R, int NT, int NS>
__global__ void __launch_bounds__(NT, col_min_ctas(NT, R)) k_sweep_batch(const SweepBatchProb *__restrict__ bp, int nprob,
                                                         long long nitems)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ SweepArrays A;
    for (long long it = blockIdx.x; it < nitems; it += gridDim.x) {
        int lo = 0, hi = nprob - 1;  // the last problem whose first item is <= it
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (bp[mid].item0 <= it) lo = mid;
            else hi = mid - 1;
        }
        const SweepBatchProb &b = bp[lo];
        __syncthreads();  // the previous item's reads of the shared buffers are done
        if (threadIdx.x == 0) A = SweepArrays{b.I, b.eta, b.chi, b.chi0L, b.mbits};
        __syncthreads();
        sweep_pair_col<R, 1, NS, false, true>(b.P, A, b.npc, b.nwin, (int)(it - b.item0), -1, b.pstride, b.ns, 0, 0,
                                              b.wide != 0, nullptr, smem_raw);
    }
}

// ---- schedules ---------------------------------------------------------------
// A schedule (C, NT) splits every plane over a cluster of C CTAs of up to NT
// threads (C = 1: one CTA a plane, k_sweep_col).  A kernel holds R rows of V
// columns a thread: R is the least for which the columns of the planes fit NT
// threads (n2 ceil(rows / R) of them); planes with more columns than threads
// take V = 4 columns of one row.  The launch takes only the threads the largest
// plane needs.  One launch sweeps every class of ordinates; where the largest
// class's planes need a kernel with its strides at run time (many rows a
// thread above all, which leave the small planes of an elongated grid to a few
// threads' serial work), classes that need another R or V have launches of
// their own (8 x 584 x 28, 4 groups, L = 3, 4 CTAs: 2.38 ms a sweep, 8.75 in one
// launch, 3.08 for the node-a-thread kernel; 8 x 160 x 100: 0.76, 4.43, 1.80).
struct SweepPart {
    int k0 = 0, k1 = 0;  // ordinates
    int R = 0, V = 0, cap = 0, nthr = 0;
    bool rt = false;  // strides at run time
    int pstride = 0, ns = 0, hs = 0, hsh = 0;
    size_t smem = 0;
};
struct SweepSched {
    int C = 0, NT = 0, nparts = 0;
    SweepPart part[3];
};

// rows of a plane per CTA of a C-CTA cluster (the kernel's own rule)
static int sweep_rows_per_cta(int n1, int n2, int C)
{
    int R = (n1 + C - 1) / C;
    const int q4 = (n2 & 3) == 0 ? 1 : ((n2 & 1) == 0 ? 2 : 4);
    return (R + q4 - 1) / q4 * q4;
}

// f(n1, n2, first ordinate, end) for the plane (rows, columns) of each ordinate
// class present in `classes` (bits: z, y, x, their order)
constexpr int kAllClasses = 7;
template <class F>
static void each_plane(const shd_ctx *c, int classes, F f)
{
    const int dims[3] = {c->nx, c->ny, c->nz};
    const int from[3] = {0, c->nZ, c->nA}, to[3] = {c->nZ, c->nA, c->N};
    for (int i = 0; i < 3; ++i)
        if (((classes >> i) & 1) && to[i] > from[i])
            f(dims[c->h_ord[from[i]].e1], dims[c->h_ord[from[i]].e2], from[i], to[i]);
}

// Nodes per CTA of the largest of the classes' planes under a C-CTA split.
static int sweep_nloc_max(const shd_ctx *c, int C, int classes = kAllClasses)
{
    int m = 0;
    each_plane(c, classes, [&](int n1, int n2, int, int) {
        const int R = C == 1 ? n1 : sweep_rows_per_cta(n1, n2, C);
        m = std::max(m, (R < n1 ? R : n1) * n2);
    });
    return m;
}

// Threads that R rows a thread need, the largest plane's.
static int sweep_threads(const shd_ctx *c, int C, int classes, int R)
{
    int m = 0;
    each_plane(c, classes, [&](int n1, int n2, int, int) {
        const int rows = C == 1 ? n1 : std::min(sweep_rows_per_cta(n1, n2, C), n1);
        m = std::max(m, (rows + R - 1) / R * n2);
    });
    return m;
}

// columns of the widest plane
static int sweep_columns(const shd_ctx *c, int classes)
{
    int m = 0;
    each_plane(c, classes, [&](int, int n2, int, int) { m = std::max(m, n2); });
    return m;
}

// The launch of schedule (C, NT) for the classes: R, V, the kernel's thread
// bound, the buffers.  Strides at compile time for R <= 4 where they fit, else
// at run time; two halo slots only where four leave no plan (planes of some 600
// columns and more).  Not built: one row a thread in a cluster (blocks of at
// most NT nodes run two rows on half the threads) and eight rows below 1024
// threads.
static bool sweep_plan(const shd_ctx *c, int C, int NT, int classes, SweepPart &pt)
{
    const size_t limit = 227 * 1024;
    const int ps = ((sweep_nloc_max(c, C, classes) + 3) & ~3) + (C == 1 ? 4 : 0);
    static const int Rs[7] = {1, 2, 3, 4, 6, 8, 1}, Vs[7] = {1, 1, 1, 1, 1, 1, 4};
    pt.hs = C > 1 ? sweep_columns(c, classes) : 0;
    for (pt.hsh = kHaloShift; pt.hsh >= (C > 1 ? 1 : kHaloShift); --pt.hsh)
        for (int i = 0; i < 7; ++i) {
            const int R = Rs[i], V = Vs[i];
            if ((R == 8 && NT != 1024) || (R == 1 && V == 1 && C > 1)) continue;
            const int slots = sweep_threads(c, C, classes, R);
            if (slots > NT * V) continue;
            const int nthr = ((slots + V - 1) / V + 31) & ~31;
            // one CTA a plane of 513 to 768 threads: the kernel bounded by 768,
            // with 85 registers a thread instead of 64
            const int cap = C == 1 && NT == 1024 && V == 1 && R <= 6 && nthr > 512 && nthr <= 768 ? 768 : NT;
            for (int rt = R > 4 || V > 1 || pt.hsh != kHaloShift; rt < (R > 2 || V > 1 ? 2 : 1); ++rt) {
                pt.ns = rt ? (slots + 3) & ~3 : cap * V;
                pt.pstride = rt ? ps : cap * V * R + 8;
                pt.smem = sizeof(float) * (6 * (size_t)pt.pstride + 2 * (size_t)pt.ns * 3 * R) +
                          (C > 1 ? ((size_t)1 << pt.hsh) * (16 * (size_t)pt.hs + 16) : 0);
                if (pt.pstride < ps || pt.smem > limit) continue;
                pt.R = R;
                pt.V = V;
                pt.rt = rt != 0;
                pt.nthr = nthr;
                pt.cap = cap;
                pt.k0 = c->N;
                pt.k1 = 0;
                each_plane(c, classes, [&](int, int, int k0, int k1) {
                    pt.k0 = std::min(pt.k0, k0);
                    pt.k1 = std::max(pt.k1, k1);
                });
                return true;
            }
        }
    return false;
}

// The launches of (C, NT); false where a plane finds no plan (none of the
// schedules sweep_sched_make accepts).
static bool sweep_parts(const shd_ctx *c, SweepSched &sc)
{
    SweepPart all;
    if (!sweep_plan(c, sc.C, sc.NT, kAllClasses, all)) return false;
    sc.part[0] = all;
    sc.nparts = 1;
    if (!all.rt) return true;
    int mask[3], n = 0;  // runs of classes of one R and V
    SweepPart pt, last;
    for (int i = 0; i < 3; ++i) {
        bool present = false;
        each_plane(c, 1 << i, [&](int, int, int, int) { present = true; });
        if (!present || !sweep_plan(c, sc.C, sc.NT, 1 << i, pt)) continue;
        if (n > 0 && pt.R == last.R && pt.V == last.V) mask[n - 1] |= 1 << i;
        else mask[n++] = 1 << i;
        last = pt;
    }
    for (int i = 0; i < n; ++i)
        if (!sweep_plan(c, sc.C, sc.NT, mask[i], sc.part[i])) {
            sc.part[0] = all;
            return true;
        }
    sc.nparts = n;
    return true;
}

using SweepKernel = void (*)(Prob<float>, float *, const float *, const float *, const float *,
                             const unsigned long long *, int, int, int, int, int, int, int, int *, int, int);

template <int R, int V, int NT, int NS, bool CL>
static SweepKernel sweep_kernel_of()
{
    if constexpr (CL) return k_sweep_cl<R, V, NT, NS>;
    else return k_sweep_col<R, V, NT, NS>;
}

template <int NT, bool CL>
static SweepKernel sweep_kernel_ns(int R)
{
    switch (R) {
        case 1: if constexpr (!CL) return sweep_kernel_of<1, 1, NT, NT, CL>(); break;
        case 2: return sweep_kernel_of<2, 1, NT, NT, CL>();
        case 3: return sweep_kernel_of<3, 1, NT, NT, CL>();
        case 4: return sweep_kernel_of<4, 1, NT, NT, CL>();
    }
    return nullptr;
}

template <bool CL>
static SweepKernel sweep_kernel(const SweepPart &sc)
{
    if (sc.rt) {  // one instantiation for every thread count up to 1024 (64 registers)
        if (sc.V == 4) return sc.R == 1 ? sweep_kernel_of<1, 4, 1024, 0, CL>() : nullptr;
        switch (sc.R) {
            case 3: return sweep_kernel_of<3, 1, 1024, 0, CL>();
            case 4: return sweep_kernel_of<4, 1, 1024, 0, CL>();
            case 6: return sc.nthr <= 512 ? sweep_kernel_of<6, 1, 512, 0, CL>() : sweep_kernel_of<6, 1, 1024, 0, CL>();
            case 8: return sweep_kernel_of<8, 1, 1024, 0, CL>();
        }
        return nullptr;
    }
    switch (sc.cap) {
        case 256: return sweep_kernel_ns<256, CL>(sc.R);
        case 384: if constexpr (CL) return sweep_kernel_ns<384, CL>(sc.R); break;
        case 512: return sweep_kernel_ns<512, CL>(sc.R);
        case 768: return sweep_kernel_ns<768, CL>(sc.R);
        case 1024: return sweep_kernel_ns<1024, CL>(sc.R);
    }
    return nullptr;
}

// Run schedule sc over every (ordinate, group) pair or, when timing, over the
// first n of every tune_stride-th into a scratch intensity.
static cudaError_t run_sweep_sched(const shd_ctx *ctx, const SweepSched &sc, float *I, const float *eta,
                                   const float *chi, cudaStream_t st, bool bits, bool wide, int n, int tune_stride)
{
    Prob<float> P = make_prob<float>(ctx);
    const float *c0L = bits ? (const float *)ctx->d_chi0L : nullptr;
    const unsigned long long *mb = bits ? ctx->d_mbits : nullptr;
    for (int i = 0; i < sc.nparts; ++i) {
        const SweepPart &pt = sc.part[i];
        int first = pt.k0 * ctx->G, end = pt.k1 * ctx->G;
        if (tune_stride > 0) {
            first = (first + tune_stride - 1) / tune_stride;
            end = std::min(n, (end + tune_stride - 1) / tune_stride);
        }
        if (end <= first) continue;
        SweepKernel kern = sc.C > 1 ? sweep_kernel<true>(pt) : sweep_kernel<false>(pt);
        if (!kern) return cudaErrorInvalidConfiguration;
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)pt.smem);
        if (e != cudaSuccess) return e;
        // the whole unified L1 as shared memory, so that the CTAs the register
        // budget allows also fit there
        e = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
        if (e != cudaSuccess) return e;
        if (sc.C > 8) {  // 16-CTA clusters are beyond the portable size: opted in per kernel
            e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
            if (e != cudaSuccess) return e;
        }
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)((end - first) * sc.C));
        cfg.blockDim = dim3((unsigned)pt.nthr);
        cfg.dynamicSmemBytes = pt.smem;
        cfg.stream = st;
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = (unsigned)sc.C;
        at[0].val.clusterDim.y = 1;
        at[0].val.clusterDim.z = 1;
        cfg.attrs = at;
        cfg.numAttrs = sc.C > 1 ? 1 : 0;
        e = cudaLaunchKernelEx(&cfg, kern, P, I, eta, chi, c0L, mb, ctx->mbits_npc, ctx->mbits_nwin, pt.pstride, pt.ns,
                               pt.hs, pt.hsh, wide ? 1 : 0, ctx->d_tc_err, first, tune_stride);
        note_launch();
        if (e != cudaSuccess) return e;
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    return cudaSuccess;
}

// The schedule (C, NT) is one of this problem's: planes of at most 4 NT nodes
// a CTA, more than half the threads busy.  false otherwise.
static bool sweep_sched_make(const shd_ctx *c, int C, int NT, SweepSched &sc)
{
    sc = SweepSched();
    const size_t limit = 227 * 1024;
    const int nl = sweep_nloc_max(c, C);
    if (C == 1) {  // any grid: unaligned planes are copied as their aligned cover
        if (NT != 1024 && NT != 512 && NT != 256) return false;
        if (nl > 4 * NT) return false;
        // smaller CTAs only where they keep more than half their threads busy
        // and share the SM (at 56 B a node)
        if (NT < 1024 && (nl <= NT / 2 || (1024 / NT) * 56 * ((size_t)((nl + 3) & ~3) + 4) > limit)) return false;
    } else {
        if (C != 2 && C != 4 && C != 8 && C != 16) return false;
        if (!sweep_planes_aligned(c)) return false;  // a CTA's rows start on 16-byte boundaries
        if (NT != 256 && NT != 384 && NT != 512 && NT != 768 && NT != 1024) return false;
        if ((NT == 384 || NT == 768) ? (nl <= 2 * NT || nl > 3 * NT) : nl > 4 * NT) return false;
        if (nl <= NT / 2) return false;  // half the threads or more would idle
        if (56 * (size_t)((nl + 3) & ~3) > limit) return false;
    }
    sc.C = C;
    sc.NT = NT;
    return sweep_parts(c, sc);  // (every schedule of these bounds has its plans)
}

// Every schedule that fits, one CTA a plane first.
static std::vector<SweepSched> sweep_candidates(const shd_ctx *c, size_t most = 64)
{
    std::vector<SweepSched> v;
    SweepSched sc;
    for (int NT : {1024, 512, 256})
        if (v.size() < most && sweep_sched_make(c, 1, NT, sc)) v.push_back(sc);
    for (int C : {2, 4, 8, 16})
        for (int NT : {256, 384, 512, 768, 1024})
            if (v.size() < most && sweep_sched_make(c, C, NT, sc)) v.push_back(sc);
    return v;
}

// some schedule of this file sweeps the problem (the forced one, if forced)
bool sweep_has_schedule(const shd_ctx *c)
{
    SweepSched sc;
    if (c->sweep_force_C > 0) return sweep_sched_make(c, c->sweep_force_C, c->sweep_force_NT, sc);
    return !sweep_candidates(c, 1).empty();
}

// The FP32 sweep's schedule: forced, chosen earlier, or chosen now by timing
// each candidate (one warm-up and three timed launches over every
// tune_stride-th pair, intensity in a scratch array) when the stream is not
// being captured; under capture without a choice, the first candidate.
static bool sweep_schedule(const shd_ctx *cc, cudaStream_t st, const float *eta, const float *chi, bool bits,
                           bool wide, SweepSched &out)
{
    shd_ctx *c = const_cast<shd_ctx *>(cc);  // the choice is a cache of the context
    if (c->sweep_force_C > 0) return sweep_sched_make(c, c->sweep_force_C, c->sweep_force_NT, out);
    if (c->sweep_C > 0 && sweep_sched_make(c, c->sweep_C, c->sweep_NT, out)) return true;
    std::vector<SweepSched> cand = sweep_candidates(c);
    if (cand.empty()) return false;
    out = cand[0];
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(st, &cs) != cudaSuccess || cs != cudaStreamCaptureStatusNone) return true;
    c->sweep_ntune = 0;
    if (cand.size() > 1) {
        int sms = 0;
        if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, c->device) != cudaSuccess || sms <= 0)
            sms = 148;
        const int npairs = c->N * c->G;
        const int n = npairs < 4 * sms ? npairs : 4 * sms;
        const int stride = npairs / n;
        float *scratch = nullptr;
        // (+16 bytes: the aligned cover of an unaligned last plane)
        if (cudaMalloc(&scratch, sizeof(float) * (size_t)n * c->Nc + 16) != cudaSuccess) {
            cudaGetLastError();
            return true;  // no room to time them: the first candidate
        }
        cudaMemsetAsync(scratch, 0, sizeof(float) * (size_t)n * c->Nc, st);
        cudaEvent_t e0, e1;
        cudaEventCreate(&e0);
        cudaEventCreate(&e1);
        float best = 1e30f;
        for (const SweepSched &sc : cand) {
            float ms = 1e30f;
            if (run_sweep_sched(c, sc, scratch, eta, chi, st, bits, wide, n, stride) == cudaSuccess) {
                cudaEventRecord(e0, st);
                bool ok = true;
                for (int r = 0; r < 3 && ok; ++r)
                    ok = run_sweep_sched(c, sc, scratch, eta, chi, st, bits, wide, n, stride) == cudaSuccess;
                cudaEventRecord(e1, st);
                if (ok && cudaEventSynchronize(e1) == cudaSuccess) {
                    cudaEventElapsedTime(&ms, e0, e1);
                    ms /= 3.f;
                }
            }
            cudaGetLastError();  // a candidate that cannot launch here is skipped
            if (c->sweep_ntune < 16) {
                c->sweep_tune[c->sweep_ntune][0] = (float)sc.C;
                c->sweep_tune[c->sweep_ntune][1] = (float)sc.NT;
                c->sweep_tune[c->sweep_ntune][2] = ms;
                c->sweep_ntune++;
            }
            if (ms < best) {
                best = ms;
                out = sc;
            }
        }
        cudaEventDestroy(e0);
        cudaEventDestroy(e1);
        cudaFree(scratch);
    }
    c->sweep_C = out.C;
    c->sweep_NT = out.NT;
    return true;
}

// ---- the batch's sweep ----------------------------------------------------------
// A batch's launch sweeps the problems that the one-CTA schedule of 1024
// threads sweeps, with the variant that their own launch of it takes
// (k_sweep_col's R and thread bound; one variant an R with strides at run time
// was slower than the node-a-thread kernel before it: four 48^3 jets, 12
// groups, 20.8 ms a step then, 23.0 with it, 18.8 now).  Variants of more than
// two rows under the 64 registers of 1024 threads spill without a launch's
// constant operands (three 64^3 jets 23.6 ms, 19.3 in launches of their own,
// 22.5 before; 52^3 19.3, 15.8, 17.9): those problems sweep on their own.
static bool sweep_batch_plan(const shd_ctx *c, SweepPart &pt)
{
    SweepSched sc;
    if (!sweep_sched_make(c, 1, 1024, sc) || sc.nparts != 1) return false;
    pt = sc.part[0];
    return pt.V == 1 && !pt.rt && (pt.R <= 2 || pt.cap == 768);
}

size_t sweep_batch_smem(const shd_ctx *c)
{
    SweepPart pt;
    return sweep_batch_plan(c, pt) ? pt.smem : 0;
}

// the descriptor of problem c as its own sweep launch would see it
void sweep_batch_fill(const shd_ctx *c, SweepBatchProb &d, long long item0)
{
    d.P = make_prob<float>(c);
    d.I = (float *)c->d_I;
    d.eta = (const float *)c->d_eta;
    d.chi = (const float *)c->d_chi;
    const bool bits = sweep_uses_chi0L<float>(c);
    d.chi0L = bits ? (const float *)c->d_chi0L : nullptr;
    d.mbits = bits ? c->d_mbits : nullptr;
    d.npc = c->mbits_npc;
    d.nwin = c->mbits_nwin;
    d.wide = sweep_tau_bounded(c) ? 0 : 1;
    SweepPart pt;
    sweep_batch_plan(c, pt);
    d.pstride = pt.pstride;
    d.ns = pt.ns;
    d.item0 = item0;
}

int sweep_batch_class(const shd_ctx *c)
{
    if (c->precision == SHD_FP64 || c->integrator != SHD_SC_LINEAR) return 0;
    SweepPart pt;
    if (!sweep_batch_plan(c, pt)) return 0;
    if (c->sweep_force_C > 0 && !(c->sweep_force_C == 1 && c->sweep_force_NT == 1024)) return 0;
    if (c->sweep_force_C <= 0 && c->sweep_C > 0 && !(c->sweep_C == 1 && c->sweep_NT == 1024)) {
        // another schedule won the problem's timing: it joins only if the
        // 1024-thread one-CTA sweep (the batch's) timed within 3 % of that
        float pp = -1.f, best = 1e30f;
        for (int k = 0; k < c->sweep_ntune; ++k) {
            if (c->sweep_tune[k][0] == 1.f && c->sweep_tune[k][1] == 1024.f) pp = c->sweep_tune[k][2];
            best = fminf(best, c->sweep_tune[k][2]);
        }
        if (!(pp > 0.f && pp <= 1.03f * best)) return 0;
    }
    return pt.R * 8 + pt.cap / 256;
}

cudaError_t launch_sweep_batch(int cls, const SweepBatchProb *d_probs, int nprob, long long nitems, size_t smem,
                               int device, cudaStream_t st)
{
    if (nprob <= 0 || nitems <= 0) return cudaSuccess;
    using KB = void (*)(const SweepBatchProb *, int, long long);
    KB kern = nullptr;
    int NT = 1024;
    switch (cls) {
        case 1 * 8 + 3: kern = k_sweep_batch<1, 768, 768>, NT = 768; break;
        case 1 * 8 + 4: kern = k_sweep_batch<1, 1024, 1024>; break;
        case 2 * 8 + 3: kern = k_sweep_batch<2, 768, 768>, NT = 768; break;
        case 2 * 8 + 4: kern = k_sweep_batch<2, 1024, 1024>; break;
        case 3 * 8 + 3: kern = k_sweep_batch<3, 768, 768>, NT = 768; break;
        case 4 * 8 + 3: kern = k_sweep_batch<4, 768, 768>, NT = 768; break;
        default: return cudaErrorInvalidConfiguration;
    }
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    int nsm = 0, per = 0;
    if (cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, device) != cudaSuccess || nsm <= 0) nsm = 148;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kern, NT, smem) != cudaSuccess || per < 1) per = 1;
    long long grid = (long long)nsm * per;  // persistent: every CTA that fits at once
    if (grid > nitems) grid = nitems;
    kern<<<(unsigned)grid, NT, smem, st>>>(d_probs, nprob, nitems);
    note_launch();
    return cudaGetLastError();
}

// (C, NT) is a schedule of the FP32 plane sweep for this problem
bool sweep_schedule_valid(const shd_ctx *c, int C, int NT)
{
    SweepSched sc;
    return c->precision != SHD_FP64 && sweep_sched_make(c, C, NT, sc);
}


// The FP32 sweep on its schedule; *ran false where none fits (the caller's
// generic sweep then runs).  bits: chi at rest comes from the chi0 table.
cudaError_t launch_sweep_f(const shd_ctx *ctx, float *I, const float *eta, const float *chi, cudaStream_t st,
                           bool bits, bool *ran)
{
    const bool wide = !sweep_tau_bounded(ctx);
    SweepSched sc;
    *ran = sweep_schedule(ctx, st, eta, chi, bits, wide, sc);
    if (!*ran) return cudaSuccess;
    return run_sweep_sched(ctx, sc, I, eta, chi, st, bits, wide, ctx->N * ctx->G, 0);
}

}  // namespace shd
