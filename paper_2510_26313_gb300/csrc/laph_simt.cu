// FP32 CUDA-core path of the block contraction (K-h).
//
// The contraction is a complex matrix product over K = 3V (site, colour):
//   C[row][col] = sum_{x,c} A[row](x,c) * Psi[col](x,c)
// with A = conj(phi_i) for a meson row i, A = (phi_i x phi_j) (the diquark,
// eps_cab phi_i^a phi_j^b) for a pair row (i<j), and Psi[(k,p)] = ph_p(x) phi_k.
// Then M[p][i][k] = C[i][(k,p)] and B[p][i,j,k] = C[(i,j)][(k,p)] for k > j.
//
// One block computes a 64-row x 64-column tile of one timeslice; the tile
// table skips tiles that lie wholly below the k > j triangle.  Per chunk of
// 16 sites the block forms the A and Psi operands in shared memory and every
// thread accumulates a 4x4 complex micro-tile in FP32.  Every chunk_sites
// sites (rounded up to 16) the FP32 partial sums are added in FP64 into the
// output, which each element's owner thread alone reads and writes (first
// chunk stores).
//
// Bound by FP32 issue.  A warp owns 32 rows x 16 columns; a lane reads two
// consecutive rows (columns) with one 16-byte load, and the lanes of a load
// read 8 (4) such pairs side by side, so that no load conflicts: four loads
// per 64 multiply-adds.  A warp leaves out the 8-column groups that none of its
// rows needs (k <= j everywhere), which the tile table's 64 x 64 steps cannot:
// at N=32 and 7 momenta the tiles hold 1.86 times the needed products, the
// groups 1.12 times.  The groups left out are spread over the four schedulers.
// Two operand buffers, one barrier per chunk: while some warps form the next
// chunk others multiply this one.  Two blocks per SM.  L=24, T=48, N=32, 7
// momenta: 26.5 -> 23.8 ms.  (Packed fma.rn.f32x2 on operands stored
// in the doubled form they need: 28.3 ms.  Three blocks per SM: 26 ms.)
#include "laph_internal.cuh"

namespace laph {

namespace {
constexpr int KS = 16;               // sites per shared-memory chunk
constexpr int KC = 3 * KS;           // complex K entries per chunk
constexpr int DRAIN = 16;            // a drain interval is a multiple of this many sites
constexpr int PITCH = SIMT_TR + 2;   // float2 per K entry, 16-byte aligned rows
constexpr int NTHREADS = 256;
constexpr int NPT = SIMT_TR * KS / NTHREADS;   // rows (and columns) of a site formed per thread
static_assert(SIMT_TR == 64 && SIMT_TC == 64 && NPT == 4, "thread mapping assumes 64x64 tiles");

// One chunk's multiply-adds of a lane: rows 2 lr + {0, 1} + 16 m, columns
// 2 lc + {0, 1} + 8 n, column groups n >= N0 (As, Bs point at the lane's first).
template <int N0>
__device__ __forceinline__ void mac(float2 (&acc)[4][4], const float2 *__restrict__ As, const float2 *__restrict__ Bs)
{
#pragma unroll 2
    for (int kk = 0; kk < KC; kk++) {
        float2 a[4], b[4];
#pragma unroll
        for (int m = 0; m < 2; m++) {
            const float4 t = *reinterpret_cast<const float4 *>(As + kk * PITCH + 16 * m);
            a[2 * m] = make_float2(t.x, t.y);
            a[2 * m + 1] = make_float2(t.z, t.w);
        }
#pragma unroll
        for (int n = N0; n < 2; n++) {
            const float4 t = *reinterpret_cast<const float4 *>(Bs + kk * PITCH + 8 * n);
            b[2 * n] = make_float2(t.x, t.y);
            b[2 * n + 1] = make_float2(t.z, t.w);
        }
#pragma unroll
        for (int m = 0; m < 4; m++)
#pragma unroll
            for (int n = 2 * N0; n < 4; n++) {
                acc[m][n].x = fmaf(a[m].x, b[n].x, acc[m][n].x);
                acc[m][n].x = fmaf(-a[m].y, b[n].y, acc[m][n].x);
                acc[m][n].y = fmaf(a[m].x, b[n].y, acc[m][n].y);
                acc[m][n].y = fmaf(a[m].y, b[n].x, acc[m][n].y);
            }
    }
}
}  // namespace

__global__ void __launch_bounds__(NTHREADS, 2)
simt_kernel(const InstDev *__restrict__ insts, const TileDev *__restrict__ tiles, int chunk_sites)
{
    extern __shared__ __align__(16) float2 sm[];   // two buffers of [A: KC][PITCH], [Psi: KC][PITCH]

    const TileDev tile = tiles[blockIdx.x];
    const InstDev &I = insts[tile.inst];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const long long V = I.V;
    const int N = I.N, P = I.P;
    const float2 *__restrict__ phit = I.phi + (long long)tile.t * N * V * 3, *__restrict__ phase = I.phase;

    // ---- operand-production mapping: site s, rows/cols tid/KS + 32*m
    const int s = tid % KS;
    // vectors of this thread's rows and columns (as element offsets / V): rows and columns past the tile's end are
    // formed from vector 0 and never read back; aj < 0 marks a meson row
    int ai[NPT], aj[NPT], bk[NPT], bp[NPT];
#pragma unroll
    for (int m = 0; m < NPT; m++) {
        const int r = tid / KS + (NTHREADS / KS) * m;
        const int g = tile.row0 + r;
        ai[m] = bk[m] = bp[m] = 0;
        aj[m] = -1;
        if (g < I.mes_rows)
            ai[m] = g;
        else if (g < I.rows)
            pair_of(g - I.mes_rows, ai[m], aj[m]);
        const int col = tile.col0 + r;
        if (col < I.cols) {
            bk[m] = col / P;
            bp[m] = col - bk[m] * P;
        }
    }
    const long long Vs = I.Vs;

    // ---- accumulation mapping (see mac)
    // Warps w and w + 4 share a scheduler: they get
    // column groups two apart, turned from block to block, so that the
    // groups left out (the leading ones) are spread over the schedulers.
    const int wr = (warp >> 2) * 32, wc = ((warp + 2 * (warp >> 2) + blockIdx.x) & 3) * 16;
    const int r0 = wr + 2 * (lane >> 2), c0 = wc + 2 * (lane & 3);
    // first column group the warp's rows need (2: none)
    int n0 = 0;
    {
        const int gw = tile.row0 + wr, cw = tile.col0 + wc;
        if (gw >= I.rows || cw >= I.cols) {
            n0 = 2;
        } else if (gw >= I.mes_rows) {
            int i, j;
            pair_of(gw - I.mes_rows, i, j);   // the smallest j of the warp's rows
            while (n0 < 2 && (cw + 8 * n0 + 7) / P <= j) n0++;
        }
    }
    float2 acc[4][4];
#pragma unroll
    for (int m = 0; m < 4; m++)
#pragma unroll
        for (int n = 0; n < 4; n++) acc[m][n] = make_float2(0.f, 0.f);

    // chunk ch of the operands into buffer buf
    auto form = [&](long long ch, int buf) {
        float2 *As = sm + buf * 2 * KC * PITCH;
        const long long x = ch * KS + s;
#pragma unroll
        for (int m = 0; m < NPT; m++) {
            float2 *pa = As + 3 * s * PITCH + tid / KS + (NTHREADS / KS) * m, *pb = pa + KC * PITCH;
            if (x >= V) {   // past the last site
#pragma unroll
                for (int c = 0; c < 3; c++) pa[c * PITCH] = pb[c * PITCH] = make_float2(0.f, 0.f);
                continue;
            }
            const int i = ai[m], j = aj[m], k = bk[m], p = bp[m];
            const float2 *pu = phit + ((long long)i * V + x) * 3, *pw = phit + ((long long)k * V + x) * 3;
            const float2 u[3] = {__ldg(pu), __ldg(pu + 1), __ldg(pu + 2)};
            const float2 w[3] = {__ldg(pw), __ldg(pw + 1), __ldg(pw + 2)};
            const float2 ph = __ldg(phase + (long long)p * Vs + x);
            if (j >= 0) {
                const float2 *pv = phit + ((long long)j * V + x) * 3;
                const float2 v[3] = {__ldg(pv), __ldg(pv + 1), __ldg(pv + 2)};
#pragma unroll
                for (int c = 0; c < 3; c++) pa[c * PITCH] = cross_c(u, v, c);
            } else {
#pragma unroll
                for (int c = 0; c < 3; c++) pa[c * PITCH] = conjf2(u[c]);
            }
#pragma unroll
            for (int c = 0; c < 3; c++) pb[c * PITCH] = cmulf(ph, w[c]);
        }
    };

    const long long nchunks = (V + KS - 1) / KS;
    const int interval = (chunk_sites + DRAIN - 1) / DRAIN * DRAIN;
    int since = 0;
    bool first_drain = true;
    form(0, 0);
    __syncthreads();

    for (long long ch = 0; ch < nchunks; ch++) {
        const bool more = ch + 1 < nchunks;
        if (more) form(ch + 1, (int)(ch + 1) & 1);
        const float2 *As = sm + (int)(ch & 1) * 2 * KC * PITCH + r0, *Bs = As - r0 + KC * PITCH + c0;
        if (n0 == 0)
            mac<0>(acc, As, Bs);
        else if (n0 == 1)
            mac<1>(acc, As, Bs);
        __syncthreads();

        since += KS;
        if (since >= interval || !more) {
            // ---- FP64 reduction of this chunk's partial sums into the output
#pragma unroll
            for (int m = 0; m < 4; m++) {
                const int g = tile.row0 + r0 + (m & 1) + 16 * (m >> 1);
                if (g >= I.rows) continue;
                const bool meson = g < I.mes_rows;
                int pi = 0, pj = 0;
                long long q = 0;
                if (!meson) {
                    q = g - I.mes_rows;
                    pair_of(q, pi, pj);
                }
#pragma unroll
                for (int n = 0; n < 4; n++) {
                    const int col = tile.col0 + c0 + (n & 1) + 8 * (n >> 1);
                    if (col >= I.cols) continue;
                    const int k = col / P, p = col - k * P;
                    double2 *dst;
                    if (meson) {
                        dst = I.outM + (((long long)tile.t * P + p) * N + g) * N + k;
                    } else {
                        if (k <= pj) continue;
                        dst = I.outB + ((long long)tile.t * P + p) * I.n_trip + binom3(k) + q;
                    }
                    double2 d = make_double2((double)acc[m][n].x, (double)acc[m][n].y);
                    if (!first_drain) {
                        const double2 old = *dst;
                        d.x += old.x;
                        d.y += old.y;
                    }
                    *dst = d;
                }
            }
#pragma unroll
            for (int m = 0; m < 4; m++)
#pragma unroll
                for (int n = 0; n < 4; n++) acc[m][n] = make_float2(0.f, 0.f);
            since = 0;
            first_drain = false;
        }
    }
}

cudaError_t launch_simt(const InstDev *d_inst, const TileDev *d_tiles, long long n_tiles, const SimtConfig &cfg,
                        int *d_status, cudaStream_t s)
{
    (void)d_status;
    if (n_tiles <= 0) return cudaSuccess;
    const size_t smem = (size_t)4 * KC * PITCH * sizeof(float2);
    cudaError_t e = cudaFuncSetAttribute(simt_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    int chunk = cfg.chunk_sites > 0 ? cfg.chunk_sites : 1024;
    for (long long base = 0; base < n_tiles; base += 0x7fffffffLL) {
        const long long n = (n_tiles - base) < 0x7fffffffLL ? (n_tiles - base) : 0x7fffffffLL;
        simt_kernel<<<(unsigned)n, NTHREADS, smem, s>>>(d_inst, d_tiles + base, chunk);
        e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace laph
