// Triangular solves of a few right-hand sides with the joined LU operators.
//
// A refinement or a time step solves for one to four columns per box: a
// product of a unit then reads its operator once (4 bytes an entry, 2 MB a box
// and direction at n = 1000) for at most four multiply-adds, so the sweep is a
// stream over the FP32 operators F and B, bound by HBM.  The tensor-core form
// pads the columns to 64, gathers them into packed operands first and took 43 us
// + 8 us (gather) for the first unit of 64 boxes at n = 1000, one column, where
// the stream needs 20 at 6.8 TB/s.
//
// Each launch applies one unit: a CTA stages the unit's block of pivot rows (at
// most 1024 x 4 values) in shared memory, and every warp takes four rows of the
// operator at a time, 16 bytes a lane, so that a warp has up to 16 loads in
// flight.  Source and result are different buffers (the columns of M at the
// ends, two compact [row][column] buffers between), so no rows are saved and no
// order among the CTAs matters; rows outside the unit are copied along.
// Products are FP32 multiply-adds of the FP32 operators.
#include <algorithm>

#include "hps_internal.h"

namespace hps {

namespace {

constexpr int SW_PARTS = 8, SW_WARPS = 8, SW_RW = 4, SW_ROWS = SW_WARPS * SW_RW * 2;

struct SweepArgs {
    const float* A[SW_PARTS];   // operator of each step of the unit (row 0 of its part)
    int off[SW_PARTS];          // its first row, counted from the unit's (forward) or the matrix's (backward)
    int rows[SW_PARTS];         // its rows
    int K[SW_PARTS];            // its columns
    int nparts, NB, wp;         // wp: columns of the unit
    long long sA;
    int n, k;                   // the unit's first row
    bool fwd;
    const int* perm;            // forward: old row (from k) at each row
    long long sP;
    const float* in;
    long long ldi, si;
    float* out;
    long long ldo, so;
    int N;
    const int* skip;
};

template <int NC>
__global__ void __launch_bounds__(32 * SW_WARPS)
k_sweep(const SweepArgs a)
{
    extern __shared__ float G[];   // [wp][NC]
    const int box = blockIdx.y;
    if (a.skip && a.skip[box]) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const float* in = a.in + box * a.si;
    float* out = a.out + box * a.so;
    const int* pb = a.fwd ? a.perm + box * a.sP : nullptr;
    const int r_first = blockIdx.x * SW_ROWS;                       // rows of the matrix
    const int lo = a.fwd ? a.k : 0, hi = a.fwd ? a.n : a.k + a.wp;   // rows that the unit changes
    if (r_first < hi && r_first + SW_ROWS > lo) {
        for (int i = threadIdx.x; i < a.wp * NC; i += blockDim.x) {
            const int j = i / NC, c = i - j * NC;
            G[i] = c < a.N ? in[(long long)(a.k + (pb ? pb[j] : j)) * a.ldi + c] : 0.0f;
        }
    }
    __syncthreads();
#pragma unroll 1
    for (int h = 0; h < 2; ++h) {
        const int r0 = r_first + (h * SW_WARPS + warp) * SW_RW;
        if (r0 >= a.n) break;
        float acc[SW_RW][NC];
#pragma unroll
        for (int q = 0; q < SW_RW; ++q)
#pragma unroll
            for (int c = 0; c < NC; ++c) acc[q][c] = 0.0f;
        if (r0 < hi && r0 + SW_RW > lo) {
            int kb = 0;
            for (int p = 0; p < a.nparts; ++p) {
                const float* A = a.A[p] + box * a.sA;
                const int K = a.K[p];
                for (int kk = 4 * lane; kk < K; kk += 128) {
                    float v[SW_RW][4];
#pragma unroll
                    for (int q = 0; q < SW_RW; ++q) {
                        const int r = r0 + q - (a.fwd ? a.k : 0) - a.off[p];
                        const bool on = r >= 0 && r < a.rows[p] && r0 + q < hi;
                        const float* Ar = A + (long long)r * a.NB + kk;
                        if (kk + 4 <= K) {
                            const float4 t = on ? __ldcs(reinterpret_cast<const float4*>(Ar)) : make_float4(0.f, 0.f, 0.f, 0.f);
                            v[q][0] = t.x; v[q][1] = t.y; v[q][2] = t.z; v[q][3] = t.w;
                        } else {
#pragma unroll
                            for (int u = 0; u < 4; ++u) v[q][u] = on && kk + u < K ? Ar[u] : 0.0f;
                        }
                    }
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        if (kk + u >= K) break;
                        const float* g = G + (kb + kk + u) * NC;
#pragma unroll
                        for (int c = 0; c < NC; ++c) {
                            const float gc = g[c];
#pragma unroll
                            for (int q = 0; q < SW_RW; ++q) acc[q][c] = fmaf(v[q][u], gc, acc[q][c]);
                        }
                    }
                }
                kb += K;
            }
#pragma unroll
            for (int q = 0; q < SW_RW; ++q)
#pragma unroll
                for (int c = 0; c < NC; ++c)
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) acc[q][c] += __shfl_xor_sync(0xffffffffu, acc[q][c], o);
        }
        // lane q NC + c writes entry (r0 + q, c)
        float mine = 0.0f;
#pragma unroll
        for (int q = 0; q < SW_RW; ++q)
#pragma unroll
            for (int c = 0; c < NC; ++c)
                if (lane == q * NC + c) mine = acc[q][c];
        const int q = lane / NC, c = lane - q * NC, r = r0 + q;
        if (q < SW_RW && c < a.N && r < a.n) {
            float src;
            if (r < lo || r >= hi) src = in[(long long)r * a.ldi + c];          // not of this unit
            else if (a.fwd) src = r < a.k + a.wp ? 0.0f : in[(long long)(a.k + pb[r - a.k]) * a.ldi + c];
            else src = r < a.k ? in[(long long)r * a.ldi + c] : 0.0f;
            out[(long long)r * a.ldo + c] = src - mine;
        }
    }
}

void launch_sweep(const SweepArgs& a, int nbox, cudaStream_t st)
{
    const dim3 grd((unsigned)((a.n + SW_ROWS - 1) / SW_ROWS), (unsigned)nbox);
    auto go = [&](auto kern, int nc) { kern<<<grd, 32 * SW_WARPS, (size_t)a.wp * nc * sizeof(float), st>>>(a); };
    const int cls = a.skip ? KC_UPDATE_TC_REFINE : KC_UPDATE_TC;
    prof_begin(cls, st);
    if (a.N == 1) go(k_sweep<1>, 1);
    else if (a.N == 2) go(k_sweep<2>, 2);
    else go(k_sweep<4>, 4);
    double el = 0.0;
    for (int p = 0; p < a.nparts; ++p) el += (double)a.rows[p] * a.K[p];
    prof_end(cls, st, 2.0 * nbox * el * a.N, (double)nbox * el * 4.0);
}

}  // namespace

bool narrow_solve(const Plan& P, Work<float>& w, int nbox, int c0, int nc, const int* skip, cudaStream_t st)
{
    // Four columns is the line: solves with stored factors take, streamed against
    // tensor-core, 536 : 1044 us for one column, 657 : 1087 for four and 1276 :
    // 1118 for eight (64 boxes at p = 12), 2973 : 5800, 4352 : 5937 and 9677 : 6209
    // (128 boxes at p = 16): eight columns' accumulators and their reads of the
    // staged block outgrow the stream.
    if (!P.tc || nc > 4 || P.unit_max > SW_PARTS) return false;
    const auto units = lu_units(P);
    const int U = (int)units.size(), total = 2 * U;
    if ((size_t)P.n * nc * sizeof(float) > P.bW) return false;   // the compact buffers are W and W2
    for (int t = 0; t < total; ++t) {
        const bool fwd = t < U;
        const auto [s, len] = units[fwd ? t : total - 1 - t];
        SweepArgs a{};
        a.nparts = len;
        a.NB = P.NB;
        a.n = P.n;
        a.k = P.k0[s];
        a.fwd = fwd;
        a.sA = fwd ? w.sF : w.sB;
        for (int i = 0; i < len; ++i) {
            const int q = s + i;
            a.A[i] = fwd ? w.F + P.fw_off[q] : w.B + P.bw_off[q];
            a.off[i] = fwd ? P.k0[q] - a.k : 0;
            a.rows[i] = fwd ? P.n - P.k0[q] : P.k0[q] + P.nbs[q];
            a.K[i] = P.nbs[q];
            a.wp += P.nbs[q];
        }
        a.perm = w.perm + P.perm_off[s];
        a.sP = w.sP;
        float* Y[2] = {w.W, w.W2};
        a.in = t == 0 ? w.M + c0 : Y[(t - 1) & 1];
        a.ldi = t == 0 ? P.ldm : nc;
        a.si = t == 0 ? w.sM : w.sG;
        a.out = t == total - 1 ? w.M + c0 : Y[t & 1];
        a.ldo = t == total - 1 ? P.ldm : nc;
        a.so = t == total - 1 ? w.sM : w.sG;
        a.N = nc;
        a.skip = skip;
        launch_sweep(a, nbox, st);
    }
    return true;
}

}  // namespace hps
