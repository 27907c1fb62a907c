// Stages a1 (project) and a3 (sh2lab) as node-tiled contractions on CUDA
// cores, plus the Lorentz remaps of moving nodes (Sec. 2.2).
//
// A node tile is an 8 x 8 brick in (x, y) at one z.  In every sweep layout
// (see shd_internal.cuh) such a brick is 8 contiguous runs of 8 nodes, so the
// tile of one (ordinate, group) is read or written as eight 32-byte runs.
//
//   a1  I_lm(c,g)  = sum_k W_k Y_p(n_k) I0(c,k,g)          (Sec. 2.3 SH)
//       moments    = sum_k W_k {1, n_i, n_i n_j}/(4 pi) I(c,k,g)
//     as one contraction per (tile, g): [64 nodes x N] x [N x (NLM + 10)].
//     For a moving node I0 is the comoving intensity from k_remap_to_comoving
//     (in the scratch buffer); its moments still use the laboratory I.
//   a3  S0(c,k,g)  = sum_p Y_p(n_k) S_p(c,g)   per (tile, g): [64 x NLM] x [NLM x N];
//     a node at rest writes eta = chi0 S0, chi = chi0 directly; a moving node
//     writes S0 to the scratch buffer and k_remap_to_lab does the transform.
//
// The remaps (one CTA per moving node, its G x N values in shared memory)
// are shared by every precision.  In single precision they read each
// (node, ordinate)'s boosted stencil and Doppler ratio from the tables that
// k_remap_tables builds once per flow field, and with group centres equally
// spaced in log energy they replace the bracket search by a constant shift.
#include <cuda_runtime.h>

#include <algorithm>
#include <type_traits>

#include "shd_internal.cuh"

namespace shd {

__device__ inline int tile_row(int d, int q)
{
    // element q of a run-ordered brick -> row r = (iy - y0)*8 + (ix - x0);
    // runs follow x for the z- and y-dominant layouts and y for the x-dominant one
    return d == 0 ? ((q & 7) << 3) | (q >> 3) : q;
}

// -------------------------------------------------------------------------
// FP64.  GB300's FP64 pipe takes about 1.6 FMAs a clock and SM, so both
// contractions are bound by it with one warp in flight already: what matters
// is that no product is formed twice or for padding, and that the work lies
// evenly over the SMs.  A thread owns one node (row of an 8 x 8 brick, 64
// threads a CTA) x four columns, operands straight from global memory with
// eight ordinates in flight; a CTA per (brick, group, slice of columns), the
// slices small enough that a 16^3 problem fills the GPU.
// 16^3, one group, 128 ordinates: a1 107 -> 42 us, a3 47 -> 21 us
// (a 64 x 32-column tile on 64 of the 152 SMs before, with the moving
// bricks' harmonics formed twice).
//
// a1: column slices 0 .. nsh - 1 hold four harmonics each, from the
// laboratory intensity at rest and the comoving (node-major) one of moving
// nodes; the rest four laboratory moments each (one holds J alone, nmom = 1).
// A CTA takes slice sl0 + blockIdx.x mod nsl: all of them (sl0 = 0), or the
// three of the moments.
// -------------------------------------------------------------------------
__global__ void __launch_bounds__(64) k_project_f64(Prob<double> P, const double *__restrict__ I,
                                                    const double *__restrict__ I0, double *__restrict__ Ip,
                                                    double *__restrict__ mom, int nmom, int nZ, int nA, int nsl, int sl0)
{
    constexpr int U = 8;
    const int NLM = P.NLM, N = P.N, G = P.G, NB = P.NB;
    const int nsh = (NLM + 3) >> 2;
    const long long item = blockIdx.x / nsl;
    const int sl = sl0 + (int)(blockIdx.x - item * nsl);
    const int g = (int)(item / P.ntiles);
    const TileInfo ti = P.tiles[item - g * P.ntiles];
    const bool harm = sl < nsh;
    const int col0 = harm ? 4 * sl : NLM + 4 * (sl - nsh), cend = harm ? NLM : NLM + nmom;
    const int r = threadIdx.x, x = ti.x0 + (r & 7), y = ti.y0 + (r >> 3);
    const bool in = x < P.nx && y < P.ny;
    const int xx = in ? x : P.nx - 1, yy = in ? y : P.ny - 1;
    const long long c = ((long long)ti.z * P.ny + yy) * P.nx + xx;
    const int m = harm && in ? P.midx[c] : -1;
    // ordinate k's value at base[k * step + the class's offset]
    const double *base = m >= 0 ? I0 + ((long long)m * G + g) * N : I + (long long)g * P.Nc;
    const long long step = m >= 0 ? 1 : (long long)G * P.Nc;
    const long long oz = m >= 0 ? 0 : c, oy = m >= 0 ? 0 : ((long long)yy * P.nz + ti.z) * P.nx + xx;
    const long long ox = m >= 0 ? 0 : ((long long)xx * P.nz + ti.z) * P.ny + yy;
    int cc[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) cc[j] = col0 + j < cend ? col0 + j : cend - 1;
    double acc[4] = {0.0, 0.0, 0.0, 0.0};
    double a[U], an[U];  // a batch of ordinates, and the next one in flight
    auto load = [&](int k0, double (&v)[U]) {
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int k = k0 + u < N ? k0 + u : N - 1;
            v[u] = base[k * step + (k < nZ ? oz : (k < nA ? oy : ox))];
        }
    };
    load(0, a);
    for (int k0 = 0; k0 < N; k0 += U) {
        if (k0 + U < N) load(k0 + U, an);
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (k0 + u >= N) break;
            const double *b = P.Bproj + (size_t)(k0 + u) * NB;
#pragma unroll
            for (int j = 0; j < 4; ++j) acc[j] += a[u] * b[cc[j]];
        }
#pragma unroll
        for (int u = 0; u < U; ++u) a[u] = an[u];
    }
    if (!in) return;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int col = col0 + j;
        if (col >= cend) break;
        if (harm) Ip[(c * G + g) * NLM + col] = acc[j];
        else mom[(c * G + g) * 10 + (col - NLM)] = acc[j];
    }
}

// a3: a CTA of 128 threads per (brick, group, slice of eight ordinates): a
// thread's node x four ordinates, the brick's S staged in shared memory.  A
// node at rest writes eta = chi0 S0, chi = chi0; a moving node's S0 goes
// node-major for its remap.
__global__ void __launch_bounds__(128) k_sh2lab_f64(Prob<double> P, const double *__restrict__ Sp,
                                                    double *__restrict__ eta, double *__restrict__ chi,
                                                    double *__restrict__ S0, int nsl)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    double *As = reinterpret_cast<double *>(smem_raw);  // [NLM][65]
    const int NLM = P.NLM, N = P.N, G = P.G;
    const long long item = blockIdx.x / nsl;
    const int sl = (int)(blockIdx.x - item * nsl);
    const int g = (int)(item / P.ntiles);
    const TileInfo ti = P.tiles[item - g * P.ntiles];
    for (int e = threadIdx.x; e < 64 * NLM; e += 128) {
        const int q = e / NLM, p = e - q * NLM, x = ti.x0 + (q & 7), y = ti.y0 + (q >> 3);
        As[p * 65 + q] = x < P.nx && y < P.ny ? Sp[((((long long)ti.z * P.ny + y) * P.nx + x) * G + g) * NLM + p] : 0.0;
    }
    __syncthreads();
    const int r = threadIdx.x & 63, k0 = sl * 8 + 4 * (threadIdx.x >> 6);
    const double *Y[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) Y[j] = P.Y + (size_t)(k0 + j < N ? k0 + j : N - 1) * NLM;
    double acc[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll 4
    for (int p = 0; p < NLM; ++p) {
        const double a = As[p * 65 + r];
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[j] += a * Y[j][p];
    }
    const int x = ti.x0 + (r & 7), y = ti.y0 + (r >> 3);
    if (x >= P.nx || y >= P.ny) return;
    const long long c = ((long long)ti.z * P.ny + y) * P.nx + x;
    const double ch = P.chi0[c * G + g];
    const int m = P.midx[c];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int k = k0 + j;
        if (k >= N) break;
        if (m >= 0) {
            S0[((long long)m * G + g) * N + k] = acc[j];
        } else {
            const long long o = ((long long)k * G + g) * P.Nc + perm_offset(P.ord[k].d, x, y, ti.z, P.nx, P.ny, P.nz);
            eta[o] = ch * acc[j];
            chi[o] = ch;
        }
    }
}

// -------------------------------------------------------------------------
// Single precision.  Both contractions are bound by the FP32 FMA rate (about
// 65 TFLOP/s reachable; 2 x 65.5 kflop per node and group at L = 7), so the
// tiles are chosen for FMAs per shared-memory load: 16 x TN (a1) and 4 x 16
// (a3) register tiles, 80 and 64 FMAs per 9 and 5 loads at L = 7, operands
// streamed by 16-byte cp.async (a1) or resident (a3).  48^3, 16 groups, 512
// ordinates: a1 4.5 and a3 6.5 ms a call (23.2 and 11.9 ms for the 4 x 5 and
// 8 x 4 tiles, with 4-byte copies and index arithmetic an element, that
// these replaced).
// -------------------------------------------------------------------------
__device__ inline void cp_async4(void *smem, const void *gmem, bool on)
{
    const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;\n" ::"r"(s), "l"(gmem), "r"(on ? 4 : 0));
}
__device__ inline void cp_async16(void *smem, const void *gmem, bool on)
{
    const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(s), "l"(gmem), "r"(on ? 16 : 0));
}
__device__ inline void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::); }
template <int N>
__device__ inline void cp_async_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N)); }

// a1: [128 rows x N] x [N x 16 TN] per CTA of 128 threads = 8 row groups of 16
// rows x 16 column groups (columns tc + 16 j).  ROWS = 0: the rows are two
// bricks of the tile list (consecutive tiles) in one energy group, their
// laboratory intensity in run order (VEC: rows of the grid are 16-byte
// multiples, one copy per half run); moments of every node and I_lm of nodes
// at rest are stored, and the laboratory intensity of moving nodes goes
// node-major into nmo for their remap (from the tile in shared memory: a
// separate transpose pass over the bricks took 1.2 ms a call).  The x-class
// ordinates' runs go along y: their rows are read transposed.  ROWS = 1: 128
// (moving node, group) rows of the node-major comoving intensity, I_lm of
// moving nodes.
constexpr int kPKC = 16, kPStages = 3, kPRow = 132;

template <int TN, int ROWS, bool VEC>
__global__ void __launch_bounds__(128, TN <= 5 ? 3 : 2) k_project_f32(Prob<float> P, const float *__restrict__ I,
                                                                      float *__restrict__ Ip,
                                                                      float *__restrict__ mom,
                                                                      float *__restrict__ nmo, int nA, long long ntp)
{
    constexpr int KC = kPKC, NBC = 16 * TN;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float *As = reinterpret_cast<float *>(smem_raw);  // [kPStages][KC][kPRow]
    float *Bs = As + kPStages * KC * kPRow;            // [kPStages][KC][NBC]
    const int tid = threadIdx.x, tr = tid >> 4, tc = tid & 15;
    const int G = P.G, N = P.N, NLM = P.NLM, nx = P.nx, ny = P.ny, nz = P.nz;
    const int nchunk = (N + KC - 1) / KC;
    // laboratory rows: tile pair fastest, so that CTAs in flight read
    // neighbouring runs
    const int g0 = ROWS ? 0 : (int)(blockIdx.x / ntp);
    const long long t0 = ROWS ? 0 : 2 * (blockIdx.x - g0 * ntp);
    const long long row0 = ROWS ? (long long)blockIdx.x * 128 : 0, nrows = P.nmoving * G;
    // this thread's piece of every ordinate's tile (VEC: a half run; else a
    // node): offsets in the z-, y- and x-class layouts
    long long oz = 0, oy = 0, ox = 0;
    bool inz = false, inx = false;
    if constexpr (!ROWS) {
        const int b = VEC ? (tid & 31) >> 4 : tid >> 6, j = VEC ? (tid >> 1) & 7 : (tid >> 3) & 7;
        const int i = VEC ? 4 * (tid & 1) : tid & 7;
        if (t0 + b < P.ntiles) {
            const TileInfo ti = P.tiles[t0 + b];
            const int x = ti.x0 + i, y = ti.y0 + j, xt = ti.x0 + j, yt = ti.y0 + i;
            inz = x < nx && y < ny;
            inx = xt < nx && yt < ny;
            oz = ((long long)ti.z * ny + y) * nx + x;
            oy = ((long long)y * nz + ti.z) * nx + x;
            ox = ((long long)xt * nz + ti.z) * ny + yt;
        }
    }
    // the node-major row of tile row `tid` when its node moves
    float *nrow = nullptr;
    if constexpr (!ROWS) {
        const long long t = t0 + (tid >> 6);
        if (t < P.ntiles) {
            const TileInfo ti = P.tiles[t];
            const int x = ti.x0 + (tid & 7), y = ti.y0 + ((tid >> 3) & 7);
            if ((ti.flags & 1) && x < nx && y < ny) {
                const int m = P.midx[((long long)ti.z * ny + y) * nx + x];
                if (m >= 0) nrow = nmo + ((long long)m * G + g0) * N;
            }
        }
    }
    const float *Ig = I + (ROWS ? 0 : (long long)g0 * P.Nc);
    const long long kstride = (long long)G * P.Nc;
    const bool rvec = (N & 3) == 0;
    float4 pre[4];  // ROWS: the next chunk's pieces
    auto load_rows = [&](int ch) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int r = (i & 1) * 64 + (tid >> 1), k = ch * KC + 8 * (i >> 1) + 4 * (tid & 1);
            pre[i] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (row0 + r >= nrows || k >= N) continue;
            const float *src = I + (row0 + r) * N + k;
            if (rvec) {
                pre[i] = *reinterpret_cast<const float4 *>(src);
            } else {
                pre[i].x = src[0];
                if (k + 1 < N) pre[i].y = src[1];
                if (k + 2 < N) pre[i].z = src[2];
                if (k + 3 < N) pre[i].w = src[3];
            }
        }
    };
    auto put_rows = [&](int ch) {
        float *A = As + (ch % kPStages) * KC * kPRow;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int r = (i & 1) * 64 + (tid >> 1), kk = 8 * (i >> 1) + 4 * (tid & 1);
            A[kk * kPRow + r] = pre[i].x;
            A[(kk + 1) * kPRow + r] = pre[i].y;
            A[(kk + 2) * kPRow + r] = pre[i].z;
            A[(kk + 3) * kPRow + r] = pre[i].w;
        }
    };
    auto issue = [&](int ch) {
        if (ch < nchunk) {
            const int st = ch % kPStages;
            float *B = Bs + st * KC * NBC;
            for (int e = tid; e < KC * NBC / 4; e += 128) {
                const int kk = e / (NBC / 4), c4 = e - kk * (NBC / 4), k = ch * KC + kk;
                cp_async16(B + kk * NBC + 4 * c4, P.Bproj + (size_t)(k < N ? k : 0) * P.NB + 4 * c4, k < N);
            }
            if constexpr (!ROWS) {
                float *A = As + st * KC * kPRow;
#pragma unroll
                for (int i = 0; i < (VEC ? 4 : 16); ++i) {
                    const int kk = VEC ? (tid >> 5) + 4 * i : i, k = ch * KC + kk;
                    const bool xc = k >= nA;
                    const long long o = xc ? ox : (P.ord[k < N ? k : 0].d == 2 ? oz : oy);
                    const bool on = k < N && (xc ? inx : inz);
                    const float *src = on ? Ig + k * kstride + o : I;
                    if constexpr (VEC) cp_async16(A + kk * kPRow + 4 * (tid & 31), src, on);
                    else cp_async4(A + kk * kPRow + tid, src, on);
                }
            }
        }
        cp_async_commit();
    };

    float acc[16][TN];
#pragma unroll
    for (int i = 0; i < 16; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) acc[i][j] = 0.f;
    if constexpr (ROWS != 0) {
        load_rows(0);
        put_rows(0);
        load_rows(1);
    }
    issue(0);
    issue(1);
    for (int ch = 0; ch < nchunk; ++ch) {
        cp_async_wait<1>();
        __syncthreads();  // chunk ch is visible; chunk ch - 1's readers are done
        issue(ch + 2);
        if constexpr (ROWS != 0) {
            put_rows(ch + 1);
            load_rows(ch + 2);
        }
        const float *A = As + (ch % kPStages) * KC * kPRow, *B = Bs + (ch % kPStages) * KC * NBC + tc;
        const int kv = ROWS ? KC : (nA - ch * KC < KC ? (nA - ch * KC > 0 ? nA - ch * KC : 0) : KC);
        if (!ROWS && nrow) {
            const float *An = A + tid, *At = A + (tid & 64) + ((tid & 7) << 3) + ((tid >> 3) & 7);
            float *dst = nrow + ch * KC;
#pragma unroll
            for (int q = 0; q < KC; q += 4) {
                float v[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) v[e] = (q + e < kv ? An : At)[(q + e) * kPRow];
                if (rvec) {
                    if (ch * KC + q < N) *reinterpret_cast<float4 *>(dst + q) = make_float4(v[0], v[1], v[2], v[3]);
                } else {
#pragma unroll
                    for (int e = 0; e < 4; ++e)
                        if (ch * KC + q + e < N) dst[q + e] = v[e];
                }
            }
        }
#pragma unroll 2
        for (int kk = 0; kk < kv; ++kk) {
            float a[16], b[TN];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const float4 v = *reinterpret_cast<const float4 *>(A + kk * kPRow + tr * 16 + 4 * q);
                a[4 * q] = v.x; a[4 * q + 1] = v.y; a[4 * q + 2] = v.z; a[4 * q + 3] = v.w;
            }
#pragma unroll
            for (int j = 0; j < TN; ++j) b[j] = B[kk * NBC + 16 * j];
#pragma unroll
            for (int i = 0; i < 16; ++i)
#pragma unroll
                for (int j = 0; j < TN; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
        }
        if constexpr (!ROWS) {
#pragma unroll 2
            for (int kk = kv; kk < KC; ++kk) {
                float a[16], b[TN];
                const float *At = A + kk * kPRow + (tr >> 2) * 64 + 2 * (tr & 3);
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const float2 v = *reinterpret_cast<const float2 *>(At + 8 * i);
                    a[i] = v.x;
                    a[8 + i] = v.y;
                }
#pragma unroll
                for (int j = 0; j < TN; ++j) b[j] = B[kk * NBC + 16 * j];
#pragma unroll
                for (int i = 0; i < 16; ++i)
#pragma unroll
                    for (int j = 0; j < TN; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
            }
        }
    }
    cp_async_wait<0>();
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        long long cg;
        bool sh = true;
        if constexpr (ROWS != 0) {
            const long long row = row0 + tr * 16 + i;
            if (row >= nrows) break;
            const long long m = row / G;
            cg = P.moving[m] * G + (row - m * G);
        } else {
            const long long t = t0 + (tr >> 2);
            if (t >= P.ntiles) break;
            const TileInfo ti = P.tiles[t];
            const int x = ti.x0 + (i & 7), y = ti.y0 + 2 * (tr & 3) + (i >> 3);
            if (x >= nx || y >= ny) continue;
            const long long c = ((long long)ti.z * ny + y) * nx + x;
            cg = c * G + g0;
            sh = P.mflag[c] == 0;
        }
#pragma unroll
        for (int j = 0; j < TN; ++j) {
            const int col = tc + 16 * j;
            if (col < NLM) {
                if (sh) Ip[cg * NLM + col] = acc[i][j];
            } else if (!ROWS && col < NLM + 10) {
                mom[cg * 10 + (col - NLM)] = acc[i][j];
            }
        }
    }
}

// a3: [64 nodes x NLM] x [NLM x ordinates] per (brick, group).  A CTA is
// persistent over the (brick, group) items for one slice of the ordinates,
// at most kSGroups groups of 16 of one kind (z- and y-class, or x-class),
// with that slice of Y^T resident in shared memory; three CTAs share an SM,
// so one's stores and barriers overlap another's FMAs (one CTA for all
// ordinates spent 40 % of its time at its barriers).  A thread computes four
// nodes of a run (along x; for x-class slices along y, S staged transposed) x
// the 16 ordinates of a group: 16 threads a group, lanes pairwise completing
// 32-byte runs.  S is staged as it lies, rows of harmonics, by cp.async one
// item ahead; 16-byte pieces are swizzled by the row so that a thread's four
// harmonics of a node are one conflict-free 16-byte load.  ROWS = 1 covers
// the bricks that hold a moving node and stores those nodes' comoving S0
// node-major for their remap (k_nodes_to_brick brings the result back; read
// here instead, it cost this kernel 3.8 ms for the pass's 2.2); ROWS = 0
// stores eta of nodes at rest, and chi where it is not the kept chi0
// (chi_all), or in a run of four that holds a moving node.
constexpr int kSGroups = 9, kSThreads = 160;

// slices of the z- and y-class groups (nA ordinates), of the x-class groups,
// and groups a slice
struct SliceShape {
    int nsA, nsX, gA, gX;
};
__host__ __device__ inline SliceShape sh2lab_f32_slices(int nA, int N)
{
    SliceShape h;
    const int a = (nA + 15) / 16, x = (N - nA + 15) / 16;
    h.nsA = (a + kSGroups - 1) / kSGroups;
    h.nsX = (x + kSGroups - 1) / kSGroups;
    h.gA = h.nsA ? (a + h.nsA - 1) / h.nsA : 0;
    h.gX = h.nsX ? (x + h.nsX - 1) / h.nsX : 0;
    return h;
}

template <int ROWS>
__global__ void __launch_bounds__(kSThreads, 3) k_sh2lab_f32(Prob<float> P, const float *__restrict__ Sp,
                                                             float *__restrict__ eta, float *__restrict__ chi,
                                                             float *__restrict__ S0, int nZ, int nA, int chi_all)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int NLM = P.NLM, N = P.N, G = P.G, nx = P.nx, ny = P.ny, nz = P.nz;
    const SliceShape sh = sh2lab_f32_slices(nA, N);
    const int nsl = sh.nsA + sh.nsX, sl = (int)(blockIdx.x % nsl);
    const bool xc = sl >= sh.nsA;
    const int gs = xc ? sh.gX : sh.gA, NS = gs * 16;
    const int kb = xc ? nA + (sl - sh.nsA) * NS : sl * NS;                          // the slice's first ordinate
    const int kend = xc ? N : (kb + NS < nA ? kb + NS : nA);                        // and its end
    const int smax = (sh.gA > sh.gX ? sh.gA : sh.gX) * 16;
    float *Bs = reinterpret_cast<float *>(smem_raw);  // [NLM][NS]
    const int NP = (NLM + 3) & ~3, pitch = (NLM + 31) & ~31;
    float *As = Bs + (size_t)NP * smax;                // [2 items][64][pitch]
    float *chir = As + (size_t)2 * 64 * pitch;         // [2][64], rows of the brick in staged order
    int *mrow = reinterpret_cast<int *>(chir + 128);   // [2][64]: moving index, -1 at rest, -2 outside
    const int tid = threadIdx.x, nthr = blockDim.x;
    for (int e = tid; e < NP * NS; e += nthr) {
        const int q = e / NP, p = e - q * NP;
        Bs[p * NS + q] = kb + q < kend && p < NLM ? P.Y[(size_t)(kb + q) * NLM + p] : 0.f;
    }
    for (int e = tid; e < 2 * 64 * pitch; e += nthr) As[e] = 0.f;  // rows outside the grid and the padding stay zero
    __syncthreads();
    const int nt = (int)(ROWS ? P.nmtiles : P.ntiles);
    const long long items = (long long)nt * G;
    // node of staged row r: z- and y-class along x, x-class along y
    auto row_xy = [&](const TileInfo &ti, int r, int &x, int &y) {
        x = ti.x0 + (xc ? r >> 3 : r & 7);
        y = ti.y0 + (xc ? r & 7 : r >> 3);
        return x < nx && y < ny;
    };
    // 16-byte piece c of row r
    auto piece = [](int r, int c) { return (c & ~7) | ((c ^ (r >> 2)) & 7); };
    // items in order of (group, tile): w = g nt + t
    struct Item {
        TileInfo ti;
        int g;
    };
    auto item_of = [&](long long w) {
        Item it;
        it.g = (int)(w / nt);
        const int t = (int)(w - (long long)it.g * nt);
        it.ti = P.tiles[ROWS ? P.mtiles[t] : t];
        return it;
    };
    float pch = 0.f;
    int pm = -2;
    auto load_item = [&](const Item &it, int b) {
        float *A = As + b * 64 * pitch;
        int x, y;
        if ((NLM & 3) == 0) {
            const int np = NLM >> 2;
            for (int e = tid; e < 64 * np; e += nthr) {
                const int r = e / np, c = e - r * np;
                const bool on = row_xy(it.ti, r, x, y);
                const float *src = on ? Sp + ((((long long)it.ti.z * ny + y) * nx + x) * G + it.g) * NLM + 4 * c : Sp;
                cp_async16(A + r * pitch + 4 * piece(r, c), src, on);
            }
        } else {
            for (int e = tid; e < 64 * NLM; e += nthr) {
                const int r = e / NLM, p = e - r * NLM;
                const bool on = row_xy(it.ti, r, x, y);
                const float *src = on ? Sp + ((((long long)it.ti.z * ny + y) * nx + x) * G + it.g) * NLM + p : Sp;
                cp_async4(A + r * pitch + 4 * piece(r, p >> 2) + (p & 3), src, on);
            }
        }
        cp_async_commit();
        pm = -2;
        if (tid < 64 && row_xy(it.ti, tid, x, y)) {
            const long long c = ((long long)it.ti.z * ny + y) * nx + x;
            pch = P.chi0[c * G + it.g];
            pm = P.midx[c];
        }
    };
    auto put_item = [&](int b) {
        cp_async_wait<0>();
        if (tid < 64) {
            chir[b * 64 + tid] = pch;
            mrow[b * 64 + tid] = pm;
        }
    };
    const int j = (tid >> 1) & 7, h4 = 4 * (tid & 1), r0 = j * 8 + h4;  // staged rows r0 .. r0 + 3
    const bool rows16 = (nx & 3) == 0 && (ny & 3) == 0;                 // runs of four nodes are 16-byte aligned
    const bool kvec = (N & 3) == 0;
    const long long w0 = blockIdx.x / nsl, ws = gridDim.x / nsl;
    Item cur, nxt;
    if (w0 < items) {
        cur = item_of(w0);
        load_item(cur, 0);
        put_item(0);
    }
    int buf = 0;
    for (long long w = w0; w < items; w += ws, buf ^= 1) {
        __syncthreads();  // this item's S is in place; the other buffer's readers are done
        const bool more = w + ws < items;
        if (more) {
            nxt = item_of(w + ws);
            load_item(nxt, buf ^ 1);
        }
        const int gr = tid >> 4;
        if (gr < gs && kb + gr * 16 < kend) {
            const float *A = As + (buf * 64 + r0) * pitch;
            const float *B = Bs + gr * 16;
            float acc[4][16];
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int q = 0; q < 16; ++q) acc[i][q] = 0.f;
            for (int c = 0; c < NP / 4; ++c) {
                float a[4][4];  // [node][harmonic]
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const float4 v = *reinterpret_cast<const float4 *>(A + i * pitch + 4 * piece(r0, c));
                    a[i][0] = v.x; a[i][1] = v.y; a[i][2] = v.z; a[i][3] = v.w;
                }
#pragma unroll
                for (int pp = 0; pp < 4; ++pp)
#pragma unroll
                    for (int q4 = 0; q4 < 4; ++q4) {
                        const float4 b = *reinterpret_cast<const float4 *>(B + (4 * c + pp) * NS + 4 * q4);
                        const float bv[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
                        for (int i = 0; i < 4; ++i)
#pragma unroll
                            for (int q = 0; q < 4; ++q)
                                acc[i][4 * q4 + q] = fmaf(a[i][pp], bv[q], acc[i][4 * q4 + q]);
                    }
            }
            const int k0 = kb + gr * 16, kn = kend - k0 < 16 ? kend - k0 : 16;
            float ch[4];
            int m[4];
            bool rest = true, moves = false;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                ch[i] = chir[buf * 64 + r0 + i];
                m[i] = mrow[buf * 64 + r0 + i];
                rest = rest && m[i] == -1;
                moves = moves || m[i] >= 0;
            }
            const bool vec = kvec && kn == 16 && (k0 & 3) == 0;
            if constexpr (ROWS != 0) {
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    if (m[i] < 0) continue;
                    float *dst = S0 + ((long long)m[i] * G + cur.g) * N + k0;
                    if (vec) {
#pragma unroll
                        for (int q4 = 0; q4 < 4; ++q4)
                            reinterpret_cast<float4 *>(dst)[q4] =
                                make_float4(acc[i][4 * q4], acc[i][4 * q4 + 1], acc[i][4 * q4 + 2], acc[i][4 * q4 + 3]);
                    } else {
#pragma unroll
                        for (int q = 0; q < 16; ++q)
                            if (q < kn) dst[q] = acc[i][q];
                    }
                }
            } else {
                const bool wchi = chi_all || moves;
                const int x = cur.ti.x0 + (xc ? j : h4), y = cur.ti.y0 + (xc ? h4 : j);
                const long long oz = ((long long)cur.ti.z * ny + y) * nx + x, oy = ((long long)y * nz + cur.ti.z) * nx + x;
                const long long ox = ((long long)x * nz + cur.ti.z) * ny + y;
                const long long kst = (long long)G * P.Nc;
                const long long og = (long long)k0 * kst + (long long)cur.g * P.Nc;
#pragma unroll
                for (int q = 0; q < 16; ++q) {
                    if (q >= kn) break;
                    const long long o = og + q * kst + (xc ? ox : (k0 + q < nZ ? oz : oy));
                    if (rest && rows16) {
                        *reinterpret_cast<float4 *>(eta + o) =
                            make_float4(ch[0] * acc[0][q], ch[1] * acc[1][q], ch[2] * acc[2][q], ch[3] * acc[3][q]);
                        if (wchi) *reinterpret_cast<float4 *>(chi + o) = make_float4(ch[0], ch[1], ch[2], ch[3]);
                    } else {
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            if (m[i] != -1) continue;
                            eta[o + i] = ch[i] * acc[i][q];
                            if (wchi) chi[o + i] = ch[i];
                        }
                    }
                }
            }
        }
        if (more) {
            put_item(buf ^ 1);
            cur = nxt;
        }
    }
}

// -------------------------------------------------------------------------
// Moving nodes.  Their per-node Lorentz remaps need all (ordinate, group)
// values of one node at once, so they work on a node-major scratch
// [m][g][k] (m = index in the moving list).  Brick transposes move data
// between the sweep layout and that scratch through shared memory, both
// sides coalesced: a brick is read / written as 32-byte runs per (k, g) and
// the scratch as contiguous runs of ordinates per (m, g).
// -------------------------------------------------------------------------

// sweep layout -> node-major scratch for the moving nodes of the bricks in
// the moving-tile list; one CTA per (brick, group)
template <class T>
__global__ void __launch_bounds__(256) k_brick_to_nodes(Prob<T> P, const T *__restrict__ src, T *__restrict__ dst)
{
    constexpr int R = 64, KC = 32;
    __shared__ T S[KC][R + 1];
    __shared__ int mrow[R];
    const int tile = P.mtiles[blockIdx.x / P.G];
    const int g = blockIdx.x - (blockIdx.x / P.G) * P.G;
    const TileInfo ti = P.tiles[tile];
    const int tid = threadIdx.x;
    for (int r = tid; r < R; r += 256) {
        int ix = ti.x0 + (r & 7), iy = ti.y0 + (r >> 3);
        mrow[r] = (ix < P.nx && iy < P.ny) ? P.midx[((long long)ti.z * P.ny + iy) * P.nx + ix] : -1;
    }
    __syncthreads();
    for (int k0 = 0; k0 < P.N; k0 += KC) {
        for (int e = tid; e < KC * R; e += 256) {
            int kk = e >> 6, q = e & 63, k = k0 + kk;
            if (k >= P.N) continue;
            int d = P.ord[k].d;
            int r = tile_row(d, q);
            if (mrow[r] < 0) continue;
            int ix = ti.x0 + (r & 7), iy = ti.y0 + (r >> 3);
            S[kk][r] = src[((long long)k * P.G + g) * P.Nc + perm_offset(d, ix, iy, ti.z, P.nx, P.ny, P.nz)];
        }
        __syncthreads();
        for (int e = tid; e < R * KC; e += 256) {
            int r = e / KC, kk = e - r * KC, k = k0 + kk;
            int m = mrow[r];
            if (m >= 0 && k < P.N) dst[((long long)m * P.G + g) * P.N + k] = S[kk][r];
        }
        __syncthreads();
    }
}

// node-major scratch (two arrays) -> sweep layout, moving nodes only
template <class T>
__global__ void __launch_bounds__(256) k_nodes_to_brick(Prob<T> P, const T *__restrict__ srcA,
                                                        const T *__restrict__ srcB, T *__restrict__ dstA,
                                                        T *__restrict__ dstB)
{
    constexpr int R = 64, KC = 32;
    __shared__ T SA[KC][R + 1];
    __shared__ T SB[KC][R + 1];
    __shared__ int mrow[R];
    const int tile = P.mtiles[blockIdx.x / P.G];
    const int g = blockIdx.x - (blockIdx.x / P.G) * P.G;
    const TileInfo ti = P.tiles[tile];
    const int tid = threadIdx.x;
    for (int r = tid; r < R; r += 256) {
        int ix = ti.x0 + (r & 7), iy = ti.y0 + (r >> 3);
        mrow[r] = (ix < P.nx && iy < P.ny) ? P.midx[((long long)ti.z * P.ny + iy) * P.nx + ix] : -1;
    }
    __syncthreads();
    for (int k0 = 0; k0 < P.N; k0 += KC) {
        for (int e = tid; e < R * KC; e += 256) {
            int r = e / KC, kk = e - r * KC, k = k0 + kk;
            int m = mrow[r];
            if (m >= 0 && k < P.N) {
                long long o = ((long long)m * P.G + g) * P.N + k;
                SA[kk][r] = srcA[o];
                SB[kk][r] = srcB[o];
            }
        }
        __syncthreads();
        for (int e = tid; e < KC * R; e += 256) {
            int kk = e >> 6, q = e & 63, k = k0 + kk;
            if (k >= P.N) continue;
            int d = P.ord[k].d;
            int r = tile_row(d, q);
            if (mrow[r] < 0) continue;
            int ix = ti.x0 + (r & 7), iy = ti.y0 + (r >> 3);
            long long a = ((long long)k * P.G + g) * P.Nc + perm_offset(d, ix, iy, ti.z, P.nx, P.ny, P.nz);
            dstA[a] = SA[kk][r];
            dstB[a] = SB[kk][r];
        }
        __syncthreads();
    }
}

// Shared tables of the remap kernels: mu[nmu], lc[G], linv[G] (working
// precision) and mesh2int[N], staged once per CTA after the node's values.
template <class T>
struct RemapTables {
    T *mu, *lc, *linv;
    int *m2i;
};

template <class T>
__device__ inline RemapTables<T> remap_tables(const Prob<T> &P, unsigned char *base)
{
    RemapTables<T> t;
    t.mu = reinterpret_cast<T *>(base);
    t.lc = t.mu + P.nmu;
    t.linv = t.lc + P.G;
    t.m2i = reinterpret_cast<int *>(t.linv + P.G);
    for (int i = threadIdx.x; i < P.nmu; i += blockDim.x) t.mu[i] = P.mu[i];
    for (int i = threadIdx.x; i < P.G; i += blockDim.x) {
        t.lc[i] = P.lc[i];
        t.linv[i] = P.linv[i];
    }
    for (int i = threadIdx.x; i < P.N; i += blockDim.x) t.m2i[i] = P.mesh2int[i];
    return t;
}

// The node's G x N values (node-major, internal ordinate order) into shared
// memory, vectorised when the rows allow it.
template <class T>
__device__ inline void stage_node(T *dst, const T *src, int n)
{
    constexpr int V = 16 / sizeof(T);
    if ((reinterpret_cast<uintptr_t>(src) & 15) == 0 && (reinterpret_cast<uintptr_t>(dst) & 15) == 0 && n % V == 0) {
        // every 16-byte piece of the node in flight at once: one memory round
        // trip per CTA (the caller's barrier publishes the copies)
        const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
        for (int i = threadIdx.x; i < n / V; i += blockDim.x)
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d + 16u * (uint32_t)i),
                         "l"(src + (size_t)i * V)
                         : "memory");
        asm volatile("cp.async.wait_all;\n" ::: "memory");
    } else {
        // B loads in flight per thread before their stores
        constexpr int B = sizeof(T) == 4 ? 8 : 4;
        const int nt = blockDim.x;
        int i = threadIdx.x;
        for (; i + (B - 1) * nt < n; i += B * nt) {
            T v[B];
#pragma unroll
            for (int j = 0; j < B; ++j) v[j] = src[i + j * nt];
#pragma unroll
            for (int j = 0; j < B; ++j) dst[i + j * nt] = v[j];
        }
        for (; i < n; i += nt) dst[i] = src[i];
    }
}

// Ring averages at the two poles (mesh rings 0 and nmu - 1, summed in mesh
// order) for every group.
// One warp per (group, ring) pair: the lanes take the ring's ordinates in
// strides of 32 and a butterfly adds their partial sums.
template <class T>
__device__ inline void pole_averages(const Prob<T> &P, const T *sv, const int *m2i, T *spole)
{
    const int lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    for (int i = threadIdx.x >> 5; i < 2 * P.G; i += nw) {
        const int g = i >> 1, rr = i & 1;
        const T *F = sv + (size_t)g * P.N;
        const int base = rr ? (P.nmu - 1) * P.nphi : 0;
        T s = 0;
        for (int j = lane; j < P.nphi; j += 32) s += F[m2i[base + j]];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (lane == 0) spole[i] = s / T(P.nphi);
    }
}

// Bilinear stencil of direction n over the (mu, phi) mesh (from the shared mu
// table), with its four ordinates given as internal indices.
template <class T>
__device__ inline Stencil<T> stencil_internal(const Prob<T> &P, const RemapTables<T> &t, const T n[3])
{
    Stencil<T> s = make_stencil<T>(t.mu, P.nmu, P.nphi, n);
#pragma unroll
    for (int i = 0; i < 4; ++i) s.k[i] = t.m2i[s.k[i]];
    return s;
}

// Stencil values of one direction per group, with the last two evaluations
// kept: consecutive output groups usually bracket neighbouring input groups.
template <class T>
struct GroupCache {
    int g0 = -1, g1 = -1;
    T v0 = 0, v1 = 0;
    __device__ inline T get(const Stencil<T> &st, const T *sv, const T *spole, int N, int g)
    {
        if (g == g1) return v1;
        if (g == g0) return v0;
        const T v = eval_stencil<T>(st, sv + (size_t)g * N, spole + 2 * g);
        g0 = g1; v0 = v1;
        g1 = g; v1 = v;
        return v;
    }
};

// Remap table entries: the stencil placement packed as mode | a << 2 | b << 12
// in the first word (a < 1024 rings, b < 2^20 phi bins), then t, tp and the
// Doppler ratio.
__device__ inline float4 table_entry(const StencilParams<float> &p, float ratio)
{
    return make_float4(__int_as_float(p.mode | (p.a << 2) | (p.b << 12)), p.t, p.tp, ratio);
}

// FP64 entries: the placement, the ratio q and what follows from it
struct RemapEntry64 {
    double t, tp, q, lq, iq3;
    int code, pad;
};

__device__ inline RemapEntry64 table_entry64(const StencilParams<double> &p, double q)
{
    RemapEntry64 e;
    e.t = p.t;
    e.tp = p.tp;
    e.q = q;
    e.lq = log(q);
    e.iq3 = 1.0 / (q * q * q);
    e.code = p.mode | (p.a << 2) | (p.b << 12);
    e.pad = 0;
    return e;
}

__device__ inline Stencil<double> table_stencil64(const RemapEntry64 &e, int nphi, const int *m2i)
{
    StencilParams<double> p;
    p.mode = e.code & 3;
    p.a = (e.code >> 2) & 1023;
    p.b = e.code >> 12;
    p.t = e.t;
    p.tp = e.tp;
    Stencil<double> s = stencil_from_params<double>(p, nphi);
#pragma unroll
    for (int i = 0; i < 4; ++i) s.k[i] = m2i[s.k[i]];
    return s;
}

template <class T>
__device__ inline Stencil<T> table_stencil(const float4 &e, int nphi, const int *m2i)
{
    const int code = __float_as_int(e.x);
    StencilParams<T> p;
    p.mode = code & 3;
    p.a = (code >> 2) & 1023;
    p.b = code >> 12;
    p.t = (T)e.y;
    p.tp = (T)e.z;
    Stencil<T> s = stencil_from_params<T>(p, nphi);
#pragma unroll
    for (int i = 0; i < 4; ++i) s.k[i] = m2i[s.k[i]];
    return s;
}

// One thread per (moving node m, internal ordinate k): the Lorentz boosts of
// n_k (Sec. 2.2) and the stencils of the boosted directions, as the remap
// kernels would compute them: tc for the comoving remap (n_k taken to the
// laboratory, nu/nu0), tl for the laboratory remap (n_k taken to the
// comoving frame, nu0/nu).  They depend only on the flow and the angles.
// rc, rl: the output groups whose looked-up energy (centre x the ratio) lies
// within the outer group edges, [lo, hi) packed as lo | hi << 8, decided in
// FP64 from the FP64 flow and directions.  Beyond the edges the remapped
// intensity is zero (Sec. 2.2), a jump that a single-precision ratio would
// place a rounding away from where the FP64 definition puts it.
// Within this distance of an outer edge (in group spacings, or in log
// energy for unequal groups) a single-precision lookup defers to the table's
// FP64 range: its own rounding stays below 1e-6 there.
constexpr float kEdgeTol = 1e-5f;

__device__ inline unsigned short group_range(const Prob<float> &P, double r)
{
    const int G = P.G;
    int lo = 0, hi = G;
    while (lo < G && P.centre[lo] * r < P.edges[0]) ++lo;
    while (hi > lo && P.centre[hi - 1] * r > P.edges[G]) --hi;
    return (unsigned short)(lo | (hi << 8));
}

__global__ void __launch_bounds__(256) k_remap_tables(Prob<float> P, float4 *__restrict__ tc, float4 *__restrict__ tl,
                                                      unsigned short *__restrict__ rc, unsigned short *__restrict__ rl,
                                                      const double *__restrict__ u64, const double *__restrict__ dirs64)
{
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= P.nmoving * P.N) return;
    const long long m = i / P.N;
    const int k = (int)(i - m * P.N);
    const long long c = P.moving[m];
    const float u[3] = {P.u[3 * c], P.u[3 * c + 1], P.u[3 * c + 2]};
    const float nk[3] = {P.dirs[3 * k], P.dirs[3 * k + 1], P.dirs[3 * k + 2]};
    float nb[3];
    const float q = boost_any<float>(u, nk, nb, -1.f, P.fp64_boost);
    tc[i] = table_entry(stencil_params<float>(P.mu, P.nmu, P.nphi, nb), q);
    const float D = boost_any<float>(u, nk, nb, 1.f, P.fp64_boost);
    tl[i] = table_entry(stencil_params<float>(P.mu, P.nmu, P.nphi, nb), D);
    const double ud[3] = {u64[3 * c], u64[3 * c + 1], u64[3 * c + 2]};
    const double nd[3] = {dirs64[3 * k], dirs64[3 * k + 1], dirs64[3 * k + 2]};
    double od[3];
    rc[i] = group_range(P, boost_dir<double>(ud, nd, od, -1.0));
    rl[i] = group_range(P, boost_dir<double>(ud, nd, od, 1.0));
}

// The FP64 tables: the values the FP64 remaps would compute in place (two
// square roots, ten divisions, an arctangent and a logarithm a (node,
// ordinate) and remap on the narrow FP64 pipe, every step): 23 x 21 x 18
// nodes, 8 groups, 128 ordinates 1.23 -> 0.94 ms comoving, 1.90 -> 1.23 ms
// laboratory (there with chi0's log ratios taken once a node).
__global__ void __launch_bounds__(256) k_remap_tables64(Prob<double> P, RemapEntry64 *__restrict__ tc,
                                                        RemapEntry64 *__restrict__ tl)
{
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= P.nmoving * P.N) return;
    const long long m = i / P.N;
    const int k = (int)(i - m * P.N);
    const long long c = P.moving[m];
    const double u[3] = {P.u[3 * c], P.u[3 * c + 1], P.u[3 * c + 2]};
    const double nk[3] = {P.dirs[3 * k], P.dirs[3 * k + 1], P.dirs[3 * k + 2]};
    double nb[3];
    const double q = boost_dir<double>(u, nk, nb, -1.0);
    tc[i] = table_entry64(stencil_params<double>(P.mu, P.nmu, P.nphi, nb), q);
    const double D = boost_dir<double>(u, nk, nb, 1.0);
    tl[i] = table_entry64(stencil_params<double>(P.mu, P.nmu, P.nphi, nb), D);
}

// Energy offset x = l / (log spacing) of equally spaced log centres, split
// into its whole part s and fraction t.
template <class T>
struct UniformShift {
    T x, t;
    int s;
};

template <class T>
__device__ inline UniformShift<T> uniform_shift(const Prob<T> &P, T l)
{
    UniformShift<T> u;
    u.x = l * P.lgidl;
    const T f = dfloor<T>(u.x);
    const T lim = T(P.G + 1);  // shifts beyond the group range act alike
    u.s = (int)dclamp<T>(f, -lim, lim);
    u.t = u.x - f;
    return u;
}

// A stencil flattened for the group loop: shared-memory offsets and weights
// of the four ordinates plus the pole term, whose weight is 0 when the
// direction lies between the outer rings (the pole slot read is then finite).
template <class T>
struct FlatStencil {
    int o0, o1, o2, o3, po;
    T w0, w1, w2, w3, wp;
    // V(g) from the group-major values sv[g][N] and pole averages spole[g][2]
    __device__ inline T eval(const T *sv, const T *spole, int N, int g) const
    {
        const T *F = sv + g * N;
        T v = w0 * F[o0] + w1 * F[o1] + w2 * F[o2] + w3 * F[o3];
        return v + wp * spole[2 * g + po];
    }
};

template <class T>
__device__ inline FlatStencil<T> flat_stencil(const Stencil<T> &s)
{
    FlatStencil<T> f;
    f.o0 = s.k[0]; f.o1 = s.k[1]; f.o2 = s.k[2]; f.o3 = s.k[3];
    f.w0 = s.w[0]; f.w1 = s.w[1]; f.w2 = s.w[2]; f.w3 = s.w[3];
    f.po = s.pole_ring > 0 ? 1 : 0;
    f.wp = s.pole_ring >= 0 ? s.wpole : T(0);
    return f;
}

// lower group of an inner bracket, kept in [0, G-2]
__device__ inline int clamp_group(int ga, int G) { return ga < 0 ? 0 : (ga > G - 2 ? G - 2 : ga); }

// chi0 between centres ga and ga+1: geometric from the node's log-ratio
// table where both are positive, linear otherwise (FP64: the natural
// logarithm, so that the value is freq_mix's)
template <class T>
__device__ inline T chi_mix(const T *schi, const T *slr, int ga, T t)
{
    const T a = schi[ga], b = schi[ga + 1];
    if constexpr (sizeof(T) == 8) {
        if (a > T(0) && b > T(0)) return a * exp(t * slr[ga]);
    }
    if (a > T(0) && b > T(0)) return freq_mix_lr<T>(a, slr[ga], t);
    return (T(1) - t) * a + t * b;
}

// laboratory I (node-major) -> comoving I0 (node-major), one CTA per moving
// node: I0(k0, g0) = (ebar_g0/eps)^3 I_lab(n, eps), n = boost of n_k0 to the
// laboratory, eps = ebar_g0 (Gamma + u.n_k0)   (Sec. 2.2)
// TAB: the boosts and stencils come from the per-flow table (FP32 only);
// otherwise they are computed in place.  Two instantiations, so that the
// table path carries none of the computed path's FP64 boost code, which the
// compiler would otherwise evaluate alongside it.
template <class T, int TAB>
__global__ void __launch_bounds__(256, sizeof(T) == 8 ? 3 : 4) k_remap_to_comoving(Prob<T> P, const T *__restrict__ In, T *__restrict__ I0,
                                                           const float4 *__restrict__ tab,
                                                           const unsigned short *__restrict__ rng)
{
    constexpr bool F32 = sizeof(T) == 4;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int G = P.G, N = P.N;
    T *sI = reinterpret_cast<T *>(smem_raw);  // [G][N] internal order
    T *spole = sI + (size_t)G * N;            // [G][2]
    const long long m = blockIdx.x;
    const long long c = P.moving[m];
    // the first two table entries of this thread, in flight during the staging
    float4 epre[2] = {};
    if constexpr (TAB && F32) {
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const int kk = threadIdx.x + i * blockDim.x;
            if (kk < N) epre[i] = tab[m * N + kk];
        }
    }
    stage_node<T>(sI, In + m * G * N, G * N);
    const RemapTables<T> tb = remap_tables<T>(P, reinterpret_cast<unsigned char *>(spole + 2 * G));
    __syncthreads();
    pole_averages<T>(P, sI, tb.m2i, spole);
    __syncthreads();
    const T u[3] = {P.u[3 * c], P.u[3 * c + 1], P.u[3 * c + 2]};
    T *dst = I0 + m * G * N;
    int iter = 0;
    for (int k0 = threadIdx.x; k0 < N; k0 += blockDim.x, ++iter) {
        T q;  // nu/nu0
        Stencil<T> st;
        // output groups [glo, ghi) look up energies within the outer edges
        // (the table's FP64 decision; in place, the working precision's)
        // (read only for a lookup within kEdgeTol of an edge, where the
        // single-precision test could differ from the FP64 one)
        int glo = -1, ghi = -1;
        auto range = [&]() {
            if (glo < 0) {
                const unsigned r = rng[m * N + k0];
                glo = (int)(r & 255u);
                ghi = (int)(r >> 8);
            }
        };
        T iq3, lq;
        if constexpr (TAB && F32) {
            const float4 e = iter == 0 ? epre[0] : (iter == 1 ? epre[1] : tab[m * N + k0]);
            q = (T)e.w;
            st = table_stencil<T>(e, P.nphi, tb.m2i);
        } else if constexpr (TAB) {
            const RemapEntry64 e = reinterpret_cast<const RemapEntry64 *>(tab)[m * N + k0];
            q = e.q;
            lq = e.lq;
            iq3 = e.iq3;
            st = table_stencil64(e, P.nphi, tb.m2i);
        } else {
            T n0[3] = {P.dirs[3 * k0], P.dirs[3 * k0 + 1], P.dirs[3 * k0 + 2]};
            T n[3];
            q = boost_any<T>(u, n0, n, T(-1), P.fp64_boost);
            st = stencil_internal<T>(P, tb, n);
        }
        if constexpr (!TAB || F32) {
            iq3 = T(1) / (q * q * q);
            lq = dlog<T>(q);
        }
        GroupCache<T> cache;
        if (sizeof(T) == 4 && P.lgu) {
            // equally spaced log centres: energy lc[g0] + lq sits at g0 + x
            // group spacings from lc[0], x = s + t with s whole, so output
            // group g0 lies between input groups g0 + s and g0 + s + 1 at the
            // same fraction t for every g0.  Output groups below [gm0, gm1)
            // fall at or below the first centre, those above it at or beyond
            // the last.
            const FlatStencil<T> fs = flat_stencil<T>(st);
            const UniformShift<T> us = uniform_shift<T>(P, lq);
            const int gm0 = min(max(-us.s, 0), G), gm1 = max(min(G - 1 - us.s, G), gm0);
            T *out = dst + k0;
            if (gm0 > 0) {
                const T v0 = fs.eval(sI, spole, N, 0);
                for (int g0 = 0; g0 < gm0; ++g0, out += N) {
                    const T dx = T(g0) + us.x - P.lgx0;
                    bool in = dx >= T(0);
                    if (TAB && dabs<T>(dx) < T(kEdgeTol)) {
                        range();
                        in = g0 >= glo;
                    }
                    *out = (in ? v0 : T(0)) * iq3;
                }
            }
            if (gm1 > gm0) {
                int ga = gm0 + us.s, g0 = gm0;
                T va = fs.eval(sI, spole, N, ga);
                for (; g0 + 1 < gm1; g0 += 2, ga += 2, out += 2 * N) {
                    const T vb = fs.eval(sI, spole, N, ga + 1);
                    const T vc = fs.eval(sI, spole, N, ga + 2);
                    out[0] = freq_mix<T>(va, vb, us.t) * iq3;
                    out[N] = freq_mix<T>(vb, vc, us.t) * iq3;
                    va = vc;
                }
                if (g0 < gm1) {
                    *out = freq_mix<T>(va, fs.eval(sI, spole, N, ga + 1), us.t) * iq3;
                    out += N;
                }
            }
            if (gm1 < G) {
                const T v1 = fs.eval(sI, spole, N, G - 1);
                for (int g0 = gm1; g0 < G; ++g0, out += N) {
                    const T dx = T(g0) + us.x - P.lgx1;
                    bool in = dx <= T(0);
                    if (TAB && dabs<T>(dx) < T(kEdgeTol)) {
                        range();
                        in = g0 < ghi;
                    }
                    *out = (in ? v1 : T(0)) * iq3;
                }
            }
            continue;
        }
        int hint = 0;
        for (int g0 = 0; g0 < G; ++g0) {
            const T le = tb.lc[g0] + lq;
            FreqBracket<T> fb = freq_bracket<T>(tb.lc, tb.linv, P.le0, P.leG, G, le, hint);
            if (TAB && F32 && (dabs<T>(le - P.le0) < T(kEdgeTol) || dabs<T>(le - P.leG) < T(kEdgeTol))) {
                range();  // inside or beyond the edges as the table decided
                if (g0 < glo || g0 >= ghi) fb.mode = 0;
                else if (fb.mode == 0) fb.mode = 1;  // the nearest outer group (fb.ga)
            }
            T v = 0;
            if (fb.mode == 1) {
                v = cache.get(st, sI, spole, N, fb.ga);
            } else if (fb.mode == 2) {
                T fa = cache.get(st, sI, spole, N, fb.ga);
                T fbv = cache.get(st, sI, spole, N, fb.ga + 1);
                v = freq_mix<T>(fa, fbv, fb.t);
            }
            dst[(size_t)g0 * N + k0] = v * iq3;
        }
    }
}

// comoving S0 (node-major) -> laboratory eta, chi (node-major):
// D = Gamma - u.n_k, n0 = comoving direction, eps0 = ebar_g D,
// S_lab = S0(n0, eps0)/D^3, chi_lab = chi0(eps0) D, eta_lab = chi_lab S_lab
template <class T, int TAB>
__global__ void __launch_bounds__(256, sizeof(T) == 8 ? 3 : 4) k_remap_to_lab(Prob<T> P, const T *__restrict__ S0, T *__restrict__ eta_n,
                                                      T *__restrict__ chi_n, const float4 *__restrict__ tab,
                                                      const unsigned short *__restrict__ rng)
{
    constexpr bool F32 = sizeof(T) == 4;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int G = P.G, N = P.N;
    T *sS = reinterpret_cast<T *>(smem_raw);  // [G][N] internal order
    T *spole = sS + (size_t)G * N;            // [G][2]
    T *schi = spole + 2 * G;                  // [G]
    T *slr = schi + G;                        // [G] log2 (FP64: log) of chi0[g+1]/chi0[g] where both > 0
    const long long m = blockIdx.x;
    const long long c = P.moving[m];
    stage_node<T>(sS, S0 + m * G * N, G * N);
    for (int g = threadIdx.x; g < G; g += blockDim.x) schi[g] = P.chi0[c * G + g];
    const RemapTables<T> tb = remap_tables<T>(P, reinterpret_cast<unsigned char *>(slr + G));
    __syncthreads();
    pole_averages<T>(P, sS, tb.m2i, spole);
    for (int g = threadIdx.x; g + 1 < G; g += blockDim.x) {
        const T a = schi[g], b = schi[g + 1];
        if constexpr (F32) slr[g] = (a > T(0) && b > T(0)) ? T(log2f(float(b / a))) : T(0);
        else slr[g] = (a > T(0) && b > T(0)) ? log(b / a) : T(0);
    }
    __syncthreads();
    const T u[3] = {P.u[3 * c], P.u[3 * c + 1], P.u[3 * c + 2]};
    T *de = eta_n + m * G * N, *dc = chi_n + m * G * N;
    for (int k = threadIdx.x; k < N; k += blockDim.x) {
        T D;  // nu0/nu
        Stencil<T> st;
        // output groups [glo, ghi) look up source energies within the outer
        // edges (the table's FP64 decision; in place, the working precision's)
        // (read only for a lookup within kEdgeTol of an edge, as above)
        int glo = -1, ghi = -1;
        auto range = [&]() {
            if (glo < 0) {
                const unsigned r = rng[m * N + k];
                glo = (int)(r & 255u);
                ghi = (int)(r >> 8);
            }
        };
        T iD3, lD;
        if constexpr (TAB && F32) {
            const float4 e = tab[m * N + k];
            D = (T)e.w;
            st = table_stencil<T>(e, P.nphi, tb.m2i);
        } else if constexpr (TAB) {
            const RemapEntry64 e = reinterpret_cast<const RemapEntry64 *>(tab)[m * N + k];
            D = e.q;
            lD = e.lq;
            iD3 = e.iq3;
            st = table_stencil64(e, P.nphi, tb.m2i);
        } else {
            T n[3] = {P.dirs[3 * k], P.dirs[3 * k + 1], P.dirs[3 * k + 2]};
            T n0[3];
            D = boost_any<T>(u, n, n0, T(1), P.fp64_boost);
            st = stencil_internal<T>(P, tb, n0);
        }
        if constexpr (!TAB || F32) {
            iD3 = T(1) / (D * D * D);
            lD = dlog<T>(D);
        }
        GroupCache<T> cache;
        if (sizeof(T) == 4 && P.lgu) {
            // equally spaced log centres: the constant shift s and fraction t
            // of the comoving remap above; below [gm0, gm1) chi0 is the first
            // group's, above it the last group's
            const FlatStencil<T> fs = flat_stencil<T>(st);
            const UniformShift<T> us = uniform_shift<T>(P, lD);
            const int gm0 = min(max(-us.s, 0), G), gm1 = max(min(G - 1 - us.s, G), gm0);
            T *oe = de + k, *oc = dc + k;
            if (gm0 > 0) {
                const T v0 = fs.eval(sS, spole, N, 0);
                const T chl = schi[0] * D;
                for (int g = 0; g < gm0; ++g, oe += N, oc += N) {
                    const T dx = T(g) + us.x - P.lgx0;
                    bool in = dx >= T(0);
                    if (TAB && dabs<T>(dx) < T(kEdgeTol)) {
                        range();
                        in = g >= glo;
                    }
                    *oc = chl;
                    *oe = chl * (in ? v0 : T(0)) * iD3;
                }
            }
            if (gm1 > gm0) {
                int ga = gm0 + us.s, g = gm0;
                T va = fs.eval(sS, spole, N, ga);
                // one output group: between ga and ga + 1, with V(ga + 1) = vb
                auto emit = [&](int a, T v0, T v1, T *pe, T *pc) {
                    const T c0 = schi[a], c1 = schi[a + 1];
                    const T sv = freq_mix<T>(v0, v1, us.t);
                    const T ch = (c0 > T(0) && c1 > T(0)) ? freq_mix_lr<T>(c0, slr[a], us.t)
                                                          : (T(1) - us.t) * c0 + us.t * c1;
                    const T chl = ch * D;
                    *pc = chl;
                    *pe = chl * sv * iD3;
                };
                for (; g + 1 < gm1; g += 2, ga += 2, oe += 2 * N, oc += 2 * N) {
                    const T vb = fs.eval(sS, spole, N, ga + 1);
                    const T vc = fs.eval(sS, spole, N, ga + 2);
                    emit(ga, va, vb, oe, oc);
                    emit(ga + 1, vb, vc, oe + N, oc + N);
                    va = vc;
                }
                if (g < gm1) {
                    emit(ga, va, fs.eval(sS, spole, N, ga + 1), oe, oc);
                    oe += N;
                    oc += N;
                }
            }
            if (gm1 < G) {
                const T v1 = fs.eval(sS, spole, N, G - 1);
                const T chl = schi[G - 1] * D;
                for (int g = gm1; g < G; ++g, oe += N, oc += N) {
                    const T dx = T(g) + us.x - P.lgx1;
                    bool in = dx <= T(0);
                    if (TAB && dabs<T>(dx) < T(kEdgeTol)) {
                        range();
                        in = g < ghi;
                    }
                    *oc = chl;
                    *oe = chl * (in ? v1 : T(0)) * iD3;
                }
            }
            continue;
        }
        int hint = 0;
        for (int g = 0; g < G; ++g) {
            const T le = tb.lc[g] + lD;
            FreqBracket<T> fb = freq_bracket<T>(tb.lc, tb.linv, P.le0, P.leG, G, le, hint);
            if (TAB && F32 && (dabs<T>(le - P.le0) < T(kEdgeTol) || dabs<T>(le - P.leG) < T(kEdgeTol))) {
                range();  // inside or beyond the edges as the table decided
                if (g < glo || g >= ghi) fb.mode = 0;
                else if (fb.mode == 0) fb.mode = 1;  // the nearest outer group (fb.ga)
            }
            T s = 0, ch;
            if (fb.mode == 0) {
                ch = schi[fb.ga];
            } else if (fb.mode == 1) {
                s = cache.get(st, sS, spole, N, fb.ga);
                ch = schi[fb.ga];
            } else {
                T fa = cache.get(st, sS, spole, N, fb.ga);
                T fbv = cache.get(st, sS, spole, N, fb.ga + 1);
                s = freq_mix<T>(fa, fbv, fb.t);
                ch = chi_mix<T>(schi, slr, fb.ga, fb.t);
            }
            T chl = ch * D;
            dc[(size_t)g * N + k] = chl;
            de[(size_t)g * N + k] = chl * s * iD3;
        }
    }
}

// -------------------------------------------------------------------------
// launchers
// -------------------------------------------------------------------------
size_t remap_smem_bytes(const shd_ctx *c)
{
    // values [G][N], poles [G][2], chi0 [G], chi0 log ratios [G], tables mu,
    // lc, linv, mesh2int
    return (size_t)c->esize * ((size_t)c->G * c->N + 4 * c->G + c->nmu + 2 * c->G) + sizeof(int) * (size_t)c->N + 16;
}

// -------------------------------------------------------------------------
// Moments alone, single precision: J, H, K of the laboratory intensity are ten
// sums over the ordinates, so a caller who reads them needs neither the
// comoving remap nor the harmonics of a1 (which also rounds them through BF16
// pieces in MIXED).  One read of I bounds it.  A CTA of 512 threads takes 16 x
// 16 (x, y) nodes of one z and group: 128 threads hold two nodes x ten sums in
// registers (20 FMAs and three broadcast 16-byte loads of coefficients per 8
// bytes of I; four nodes a thread cost the registers that keep loads in
// flight), and four such thread groups share the ordinates, eight loads in
// flight a thread.  The z- and y-class layouts run along x, the x-class one
// along y, so the threads change to nodes along y for it, and the partial sums
// meet in shared memory in a fixed order.  Rows of an odd number of nodes
// (PAIR = false) take 4-byte loads, a thread's nodes eight rows apart.  The
// summation chains are N / 6 and N / 12 products long.
// 64^3, 16 groups, 512 ordinates: 1.84 ms (4.7 TB/s, 0.69 of the copy rate)
// against 5.78 for a1 with a widening pass; with four nodes a thread 4.8.
// -------------------------------------------------------------------------
constexpr int kMomPitch = 16 * 17 + 1;  // the words of a sum: a row of 16 nodes every 17
constexpr int kMomChunk = 1024;         // ordinates whose coefficients are held at once

template <bool PAIR, class TO>
__global__ void __launch_bounds__(512, 2) k_moments_f32(Prob<float> P, const float *__restrict__ I, TO *__restrict__ mom,
                                                        int nZ, long long items)
{
    constexpr int U = 8;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float4 *cf = reinterpret_cast<float4 *>(smem_raw);    // [min(N, kMomChunk)][3]
    const int nk = P.N < kMomChunk ? P.N : kMomChunk;
    float *red = reinterpret_cast<float *>(cf + 3 * nk);  // [4][10][kMomPitch]
    const int tid = threadIdx.x, kg = tid >> 7, t = tid & 127;
    float *slab = red + kg * 10 * kMomPitch;
    const int ntx = (P.nx + 15) >> 4, nty = (P.ny + 15) >> 4;
    const long long step = (long long)P.G * P.Nc;
    // the thread's nodes within the tile: (f, s) and (f + 1, s) or (f, s + 8),
    // f along the layout's fast axis
    const int f = PAIR ? 2 * (t & 7) : (t & 15), s = PAIR ? t >> 3 : t >> 4;

    auto coefficients = [&](int k0, int n) {
        for (int e = tid; e < 12 * n; e += 512) {
            const int k = e / 12, q = e - 12 * k;
            reinterpret_cast<float *>(cf)[e] = q < 10 ? P.Bproj[(size_t)(k0 + k) * P.NB + P.NLM + q] : 0.0f;
        }
    };
    if (P.N <= kMomChunk) coefficients(0, P.N);

    for (long long item = blockIdx.x; item < items; item += gridDim.x) {
        const int tx = (int)(item % ntx);
        const long long r1 = item / ntx, r2 = r1 / nty;
        const int ty = (int)(r1 - r2 * nty), z = (int)(r2 % P.nz), g = (int)(r2 / P.nz);
        const int x0 = 16 * tx, y0 = 16 * ty;
        const float *Ig = I + (long long)g * P.Nc;

        float acc[2][10];
        auto take = [&](float a, float b, const float4 *c) {
            const float4 c0 = c[0], c1 = c[1], c2 = c[2];
            acc[0][0] += a * c0.x; acc[1][0] += b * c0.x;
            acc[0][1] += a * c0.y; acc[1][1] += b * c0.y;
            acc[0][2] += a * c0.z; acc[1][2] += b * c0.z;
            acc[0][3] += a * c0.w; acc[1][3] += b * c0.w;
            acc[0][4] += a * c1.x; acc[1][4] += b * c1.x;
            acc[0][5] += a * c1.y; acc[1][5] += b * c1.y;
            acc[0][6] += a * c1.z; acc[1][6] += b * c1.z;
            acc[0][7] += a * c1.w; acc[1][7] += b * c1.w;
            acc[0][8] += a * c2.x; acc[1][8] += b * c2.x;
            acc[0][9] += a * c2.y; acc[1][9] += b * c2.y;
        };
        // ordinates [ka, kb) of one layout, the nodes at o0 and o1 (o0 + 1 with PAIR)
        auto add = [&](int ka, int kb, int k0, long long o0, long long o1) {
            const float *p = Ig + (long long)ka * step;
            const float4 *c = cf + 3 * (ka - k0);
            int n = kb - ka;
            auto at = [&](const float *q) {
                if constexpr (PAIR) return __ldcs(reinterpret_cast<const float2 *>(q + o0));
                else return make_float2(__ldg(q + o0), __ldg(q + o1));
            };
            for (; n >= U; n -= U, c += 3 * U) {
                float2 v[U];
#pragma unroll
                for (int u = 0; u < U; ++u, p += step) v[u] = at(p);
#pragma unroll
                for (int u = 0; u < U; ++u) take(v[u].x, v[u].y, c + 3 * u);
            }
            if (n > 0) {
                float2 v[U];
#pragma unroll
                for (int u = 0; u < U; ++u, p += step) v[u] = u < n ? at(p) : make_float2(0.0f, 0.0f);
#pragma unroll
                for (int u = 0; u < U; ++u)
                    if (u < n) take(v[u].x, v[u].y, c + 3 * u);
            }
        };
        auto clear = [&]() {
#pragma unroll
            for (int q = 0; q < 10; ++q) acc[0][q] = acc[1][q] = 0.0f;
        };
        // a node outside the grid reads the tile's first one; its sums are not stored
        auto offset = [&](int ff, int ss, int d) -> long long {
            int x = x0 + (d == 0 ? ss : ff), y = y0 + (d == 0 ? ff : ss);
            if (x >= P.nx || y >= P.ny) { x = x0; y = y0; }
            return perm_offset(d, x, y, z, P.nx, P.ny, P.nz);
        };
        const int f1 = PAIR ? f + 1 : f, s1 = PAIR ? s : s + 8;
        for (int k0 = 0; k0 < P.N; k0 += kMomChunk) {
            const int k1 = P.N - k0 < kMomChunk ? P.N : k0 + kMomChunk;
            __syncthreads();  // the previous tile's sums are read (and the first tile's coefficients are there)
            if (P.N > kMomChunk) {
                coefficients(k0, k1 - k0);
                __syncthreads();
            }
            // z and y classes: along x
            clear();
            {
                const int kb = P.nA < k1 ? P.nA : k1, n = kb - k0;
                if (n > 0) {
                    const int a = k0 + n * kg / 4, b = k0 + n * (kg + 1) / 4;
                    const int bz = b < nZ ? b : nZ, ay = a > nZ ? a : nZ;
                    if (a < bz) add(a, bz, k0, offset(f, s, 2), offset(f1, s1, 2));
                    if (ay < b) add(ay, b, k0, offset(f, s, 1), offset(f1, s1, 1));
                }
            }
#pragma unroll
            for (int q = 0; q < 10; ++q) {
                float *d = slab + q * kMomPitch;
                float &d0 = d[17 * s + f], &d1 = d[17 * s1 + f1];
                d0 = k0 == 0 ? acc[0][q] : d0 + acc[0][q];
                d1 = k0 == 0 ? acc[1][q] : d1 + acc[1][q];
            }
            // x class: along y
            clear();
            {
                const int ka = P.nA > k0 ? P.nA : k0, n = k1 - ka;
                const int a = ka + n * kg / 4, b = ka + n * (kg + 1) / 4;
                if (n > 0 && a < b) add(a, b, k0, offset(f, s, 0), offset(f1, s1, 0));
            }
            __syncthreads();
#pragma unroll
            for (int q = 0; q < 10; ++q) {
                float *d = slab + q * kMomPitch;
                d[17 * f + s] += acc[0][q];
                d[17 * f1 + s1] += acc[1][q];
            }
        }
        __syncthreads();
        for (int e = tid; e < 2560; e += 512) {
            const int n = e / 10, q = e - 10 * n, x = x0 + (n & 15), y = y0 + (n >> 4);
            if (x < P.nx && y < P.ny) {
                const float *d = red + q * kMomPitch + 17 * (n >> 4) + (n & 15);
                const float v = (d[0] + d[10 * kMomPitch]) + (d[20 * kMomPitch] + d[30 * kMomPitch]);
                mom[((((long long)z * P.ny + y) * P.nx + x) * P.G + g) * 10 + q] = (TO)v;
            }
        }
    }
}

static int num_sms(const shd_ctx *ctx)
{
    int n = 0;
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, ctx->device) != cudaSuccess || n <= 0) n = 148;
    return n;
}

// rows of the grid along x and y are 16-byte multiples
static bool rows_aligned(const shd_ctx *c) { return c->nx % 4 == 0 && c->ny % 4 == 0; }

template <int TN, int ROWS, bool VEC>
static cudaError_t launch_project_f32_k(const shd_ctx *ctx, const float *I, float *Ip, float *mom, float *nmo,
                                        cudaStream_t st)
{
    const Prob<float> P = make_prob<float>(ctx);
    const int sm = (int)sizeof(float) * kPStages * kPKC * (kPRow + 16 * TN);
    auto kern = k_project_f32<TN, ROWS, VEC>;
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, sm);
    if (e != cudaSuccess) return e;
    const long long ntp = (ctx->ntiles + 1) / 2;
    const long long grid = ROWS ? (ctx->nmoving * ctx->G + 127) / 128 : ntp * ctx->G;
    kern<<<(unsigned)grid, 128, sm, st>>>(P, I, Ip, mom, nmo, ctx->nA, ntp);
    note_launch();
    return cudaGetLastError();
}

template <int ROWS, bool VEC>
static cudaError_t launch_project_f32_tn(const shd_ctx *ctx, int tn, const float *I, float *Ip, float *mom,
                                         float *nmo, cudaStream_t st)
{
    switch (tn) {
        case 1: return launch_project_f32_k<1, ROWS, VEC>(ctx, I, Ip, mom, nmo, st);
        case 2: return launch_project_f32_k<2, ROWS, VEC>(ctx, I, Ip, mom, nmo, st);
        case 3: return launch_project_f32_k<3, ROWS, VEC>(ctx, I, Ip, mom, nmo, st);
        case 4: return launch_project_f32_k<4, ROWS, VEC>(ctx, I, Ip, mom, nmo, st);
        case 5: return launch_project_f32_k<5, ROWS, VEC>(ctx, I, Ip, mom, nmo, st);
        case 6: return launch_project_f32_k<6, ROWS, VEC>(ctx, I, Ip, mom, nmo, st);
        case 7: return launch_project_f32_k<7, ROWS, VEC>(ctx, I, Ip, mom, nmo, st);
        default: return cudaErrorInvalidConfiguration;
    }
}

// the laboratory rows' columns [W Y | moments] and the moving rows' copy, then
// the comoving remap and the moving rows' W Y
static cudaError_t launch_project_f32(const shd_ctx *ctx, const float *I, float *Ip, float *mom, float *nm0,
                                      float *nm1, cudaStream_t st)
{
    const int tn = ctx->NB / 16;
    cudaError_t e = rows_aligned(ctx) ? launch_project_f32_tn<0, true>(ctx, tn, I, Ip, mom, nm0, st)
                                      : launch_project_f32_tn<0, false>(ctx, tn, I, Ip, mom, nm0, st);
    if (e != cudaSuccess || ctx->nmoving == 0) return e;
    if ((e = launch_remap_to_comoving_f(ctx, nm0, nm1, st)) != cudaSuccess) return e;
    return launch_project_f32_tn<1, true>(ctx, (ctx->NLM + 15) / 16, nm1, Ip, mom, nullptr, st);
}

static size_t sh2lab_f32_smem_bytes(const shd_ctx *c)
{
    const SliceShape h = sh2lab_f32_slices(c->nA, c->N);
    return sizeof(float) * ((size_t)((c->NLM + 3) & ~3) * 16 * std::max(h.gA, h.gX) +
                            (size_t)2 * 64 * ((c->NLM + 31) & ~31) + 256);
}

// FP32's a3 keeps chi_lab at rest (as the mixed segment transform does); its
// slices fit every order (124 KB at L = 9)
bool sh2lab_f32_usable(const shd_ctx *c) { return c->precision == SHD_FP32; }

template <int ROWS>
static cudaError_t launch_sh2lab_f32_k(const shd_ctx *ctx, const float *Sp, float *eta, float *chi, float *S0,
                                       cudaStream_t st, bool full_chi)
{
    const Prob<float> P = make_prob<float>(ctx);
    const size_t sm = sh2lab_f32_smem_bytes(ctx);
    auto kern = k_sh2lab_f32<ROWS>;
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    const long long items = (ROWS ? ctx->nmtiles : ctx->ntiles) * ctx->G;
    const SliceShape h = sh2lab_f32_slices(ctx->nA, ctx->N);
    const int nsl = h.nsA + h.nsX;
    const int nthr = std::max(64, (16 * std::max(h.gA, h.gX) + 31) & ~31);
    int per = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kern, nthr, sm) != cudaSuccess || per < 1) per = 1;
    // every slice over as many CTAs
    const long long ctas = std::min<long long>(items, std::max(1, num_sms(ctx) * per / nsl));
    const long long grid = ctas * nsl;
    kern<<<(unsigned)grid, nthr, sm, st>>>(P, Sp, eta, chi, S0, ctx->nZ, ctx->nA, full_chi ? 1 : 0);
    note_launch();
    return cudaGetLastError();
}

// eta and chi of nodes at rest, S0 of moving nodes
static cudaError_t launch_sh2lab_f32(const shd_ctx *ctx, const float *Sp, float *eta, float *chi, float *S0,
                                     cudaStream_t st, bool full_chi)
{
    const cudaError_t e = launch_sh2lab_f32_k<0>(ctx, Sp, eta, chi, nullptr, st, full_chi);
    if (e != cudaSuccess || ctx->nmoving == 0) return e;
    return launch_sh2lab_f32_k<1>(ctx, Sp, nullptr, nullptr, S0, st, false);
}

template <class T>
static cudaError_t run_remap_to_comoving(const shd_ctx *ctx, const T *nm0, T *nm1, cudaStream_t st)
{
    Prob<T> P = make_prob<T>(ctx);
    size_t sm = remap_smem_bytes(ctx);
    const float4 *tab = ctx->rtab_valid ? (const float4 *)ctx->d_rtab[0] : nullptr;
    auto kern = tab ? k_remap_to_comoving<T, 1> : k_remap_to_comoving<T, 0>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    kern<<<(unsigned)ctx->nmoving, 256, sm, st>>>(P, nm0, nm1, tab, tab ? ctx->d_rrng[0] : nullptr);
    note_launch();
    return cudaGetLastError();
}

template <class T>
static cudaError_t run_remap_to_lab(const shd_ctx *ctx, const T *nm0, T *nm1, T *nm2, cudaStream_t st)
{
    Prob<T> P = make_prob<T>(ctx);
    size_t sr = remap_smem_bytes(ctx);
    const float4 *tab = ctx->rtab_valid ? (const float4 *)ctx->d_rtab[1] : nullptr;
    auto kern = tab ? k_remap_to_lab<T, 1> : k_remap_to_lab<T, 0>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sr);
    if (e != cudaSuccess) return e;
    kern<<<(unsigned)ctx->nmoving, 256, sr, st>>>(P, nm0, nm1, nm2, tab, tab ? ctx->d_rrng[1] : nullptr);
    note_launch();
    return cudaGetLastError();
}

cudaError_t launch_remap_tables_f(const shd_ctx *ctx, float4 *tc, float4 *tl, unsigned short *rc, unsigned short *rl,
                                  const double *u64, const double *dirs64, cudaStream_t st)
{
    Prob<float> P = make_prob<float>(ctx);
    const long long n = ctx->nmoving * ctx->N;
    if (n == 0) return cudaSuccess;
    k_remap_tables<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(P, tc, tl, rc, rl, u64, dirs64);
    note_launch();
    return cudaGetLastError();
}

cudaError_t launch_remap_tables_d(const shd_ctx *ctx, void *tc, void *tl, cudaStream_t st)
{
    const long long n = ctx->nmoving * ctx->N;
    if (n == 0) return cudaSuccess;
    k_remap_tables64<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(make_prob<double>(ctx), (RemapEntry64 *)tc, (RemapEntry64 *)tl);
    note_launch();
    return cudaGetLastError();
}
size_t remap_entry64_bytes() { return sizeof(RemapEntry64); }

cudaError_t launch_remap_to_comoving_f(const shd_ctx *ctx, const float *nm0, float *nm1, cudaStream_t st)
{
    return run_remap_to_comoving<float>(ctx, nm0, nm1, st);
}
cudaError_t launch_remap_to_lab_f(const shd_ctx *ctx, const float *nm0, float *nm1, float *nm2, cudaStream_t st)
{
    return run_remap_to_lab<float>(ctx, nm0, nm1, nm2, st);
}

// Moving nodes first: brick transpose of I into nm0, comoving remap into
// nm1; then the projection contraction (reading nm1 for moving rows).  Of the
// moments J is stored, all that a step's sums read (kernels that compute the
// others beside it may store them); launch_moments gives all ten.
template <class T>
cudaError_t launch_project_nm(const shd_ctx *ctx, const T *I, T *Ip, T *mom, T *nm0, T *nm1, cudaStream_t st)
{
    Prob<T> P = make_prob<T>(ctx);
    cudaError_t e;
    if constexpr (sizeof(T) == 4) {
        // the segment kernels write the moving rows node-major themselves
        if (seg_usable(ctx)) return launch_project_seg(ctx, I, Ip, mom, nm0, nm1, st);
        if (!tc_usable(ctx)) return launch_project_f32(ctx, I, Ip, mom, nm0, nm1, st);
    }
    if (ctx->nmoving > 0) {
        k_brick_to_nodes<T><<<(unsigned)(ctx->nmtiles * ctx->G), 256, 0, st>>>(P, I, nm0);
        note_launch();
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        if ((e = run_remap_to_comoving<T>(ctx, nm0, nm1, st)) != cudaSuccess) return e;
    }
    if constexpr (sizeof(T) == 4) {
        return launch_project_tc(ctx, I, Ip, mom, nm1, st);
    } else {
        const int nsl = (ctx->NLM + 3) / 4 + 1;  // four harmonics a slice, and J's
        k_project_f64<<<(unsigned)(ctx->ntiles * ctx->G * nsl), 64, 0, st>>>(P, I, nm1, Ip, mom, 1, ctx->nZ,
                                                                              ctx->nA, nsl, 0);
        note_launch();
        return cudaGetLastError();
    }
}

template <class T>
cudaError_t launch_project(const shd_ctx *ctx, const T *I, T *Ip, T *mom, cudaStream_t st)
{
    return launch_project_nm<T>(ctx, I, Ip, mom, (T *)ctx->d_nm[0], (T *)ctx->d_nm[1], st);
}

template <bool PAIR, class TO>
static cudaError_t launch_moments_f32(const shd_ctx *ctx, const float *I, TO *mom, cudaStream_t st)
{
    const Prob<float> P = make_prob<float>(ctx);
    const int sm = (int)(48 * (size_t)std::min(ctx->N, kMomChunk) + sizeof(float) * 40 * kMomPitch);
    auto kern = k_moments_f32<PAIR, TO>;
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, sm);
    if (e != cudaSuccess) return e;
    const long long items = (long long)((ctx->nx + 15) / 16) * ((ctx->ny + 15) / 16) * ctx->nz * ctx->G;
    int per = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kern, 512, sm) != cudaSuccess || per < 1) per = 1;
    kern<<<(unsigned)std::min<long long>(items, (long long)num_sms(ctx) * per), 512, sm, st>>>(P, I, mom, ctx->nZ, items);
    note_launch();
    return cudaGetLastError();
}

// The laboratory moments [c][g][10] alone, in working precision (TO = T) or
// widened exactly.  FP64 runs a1's moment slices (the same sums, bit for bit).
template <class T, class TO>
cudaError_t launch_moments(const shd_ctx *ctx, const T *I, TO *mom, cudaStream_t st)
{
    if constexpr (sizeof(T) == 8) {
        k_project_f64<<<(unsigned)(ctx->ntiles * ctx->G * 3), 64, 0, st>>>(make_prob<double>(ctx), I, nullptr, nullptr, mom, 10,
                                                                            ctx->nZ, ctx->nA, 3, (ctx->NLM + 3) / 4);
        note_launch();
        return cudaGetLastError();
    } else {
        // rows of pairs of nodes in every layout
        return ctx->nx % 2 == 0 && ctx->ny % 2 == 0 ? launch_moments_f32<true>(ctx, I, mom, st)
                                                    : launch_moments_f32<false>(ctx, I, mom, st);
    }
}

// The contraction writes S0 of moving rows to nm0; their laboratory eta, chi
// go to nm1, nm2 and are transposed into the sweep layout.
template <class T>
cudaError_t launch_sh2lab(const shd_ctx *ctx, const T *Sp, T *eta, T *chi, cudaStream_t st, bool full_chi)
{
    Prob<T> P = make_prob<T>(ctx);
    cudaError_t e = cudaSuccess;
    T *nm0 = (T *)ctx->d_nm[0], *nm1 = (T *)ctx->d_nm[1], *nm2 = (T *)ctx->d_nm[2];
    if constexpr (sizeof(T) == 4) {
        // the segment kernels run the remap and write the moving rows themselves
        if (seg_usable(ctx)) return launch_sh2lab_seg(ctx, Sp, eta, chi, nm0, nm1, nm2, st, full_chi);
        e = tc_usable(ctx) ? launch_sh2lab_tc(ctx, Sp, eta, chi, nm0, st)
                           : launch_sh2lab_f32(ctx, Sp, eta, chi, nm0, st, full_chi || !sh2lab_f32_usable(ctx));
        if (e != cudaSuccess) return e;
    } else {
        const int nsl = (ctx->N + 7) / 8;
        const size_t sm = sizeof(double) * 65 * (size_t)ctx->NLM;
        e = cudaFuncSetAttribute(k_sh2lab_f64, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
        if (e != cudaSuccess) return e;
        k_sh2lab_f64<<<(unsigned)(ctx->ntiles * ctx->G * nsl), 128, sm, st>>>(P, Sp, eta, chi, nm0, nsl);
        note_launch();
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    if (ctx->nmoving > 0) {
        if ((e = run_remap_to_lab<T>(ctx, nm0, nm1, nm2, st)) != cudaSuccess) return e;
        k_nodes_to_brick<T><<<(unsigned)(ctx->nmtiles * ctx->G), 256, 0, st>>>(P, nm1, nm2, eta, chi);
        note_launch();
        e = cudaGetLastError();
    }
    return e;
}

// Stage a1 with the moving nodes' node-major intermediates (laboratory I and
// comoving I0: 2 * nmoving * G * N reals) in caller-provided `scratch`
// instead of the context's buffers.
template <class T>
cudaError_t launch_project_scratch(const shd_ctx *ctx, const T *I, T *Ip, T *mom, T *scratch, cudaStream_t st)
{
    T *nm0 = scratch, *nm1 = scratch + (size_t)ctx->nmoving * ctx->G * ctx->N;
    return launch_project_nm<T>(ctx, I, Ip, mom, nm0, nm1, st);
}

template cudaError_t launch_project_scratch<double>(const shd_ctx *, const double *, double *, double *, double *,
                                                    cudaStream_t);
template cudaError_t launch_project_scratch<float>(const shd_ctx *, const float *, float *, float *, float *,
                                                   cudaStream_t);

template cudaError_t launch_moments<double, double>(const shd_ctx *, const double *, double *, cudaStream_t);
template cudaError_t launch_moments<float, double>(const shd_ctx *, const float *, double *, cudaStream_t);
template cudaError_t launch_moments<float, float>(const shd_ctx *, const float *, float *, cudaStream_t);
template cudaError_t launch_project<double>(const shd_ctx *, const double *, double *, double *, cudaStream_t);
template cudaError_t launch_project<float>(const shd_ctx *, const float *, float *, float *, cudaStream_t);
template cudaError_t launch_sh2lab<double>(const shd_ctx *, const double *, double *, double *, cudaStream_t, bool);
template cudaError_t launch_sh2lab<float>(const shd_ctx *, const float *, float *, float *, cudaStream_t, bool);

}  // namespace shd
