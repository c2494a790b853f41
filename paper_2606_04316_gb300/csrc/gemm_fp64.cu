// gemm_fp64.cu -- the plain-form (all FP64) contractions.
//   first half  (Eq. firsthalf):  V[ab, (rs,i)] = sum_cd (ab|cd) Dq[cd, (rs,i)]
//       -> C = A B with a ragged K per 64-row tile (the screened ket prefix);
//   second half (Eq. secondhalf with the quaternion->two-spinor conversion of
//   the paper's Sec. 2.4.2 folded into real parts):
//       O[(pq,i), (rs,j)] = sum_ab Dq[ab, (pq,i)] V[ab, (rs,j)]
//       -> C = A^T B, symmetric, upper block tiles only, deterministic split-K.
#include "qdt_internal.cuh"

namespace qdt {

// The FP64 units bound both (about two multiply-adds per cycle and SM): a warp's DFMA
// holds its scheduler for tens of cycles, so one output per thread keeps the units as busy as
// sixteen would, and the loads, two shared values per multiply-add, hide behind it.
// What is left is the balance over the SMs, which small tiles give.  16 x 16 instead of
// 64 x 64: first half of a 7-centre chain (9.3 GFLOP) 16.9 -> 7.7 ms, 1.2 TFLOP/s; of an
// 8-function molecule (0.16 GFLOP) 0.86 -> 0.15 ms; their second halves 1.86 -> 0.37 and 0.12 -> 0.04.
// The sum of an output runs over k in order whatever the tile, so the tile decides no
// bit.  Row extents of the screened prefix stay per 64 rows.
constexpr int TM = 64;                   // rows of one prefix extent; the second half's upper tiles
constexpr int TS = 16, TK = 16;          // tile of a CTA; k per step (32: 7.80 ms instead of 7.74 below)
constexpr int kThreads = TS * TS;

int gemm_fp64_tile_m() { return TM; }

__global__ void __launch_bounds__(kThreads) dgemm_nn_ragged(const double *__restrict__ A, long long lda,
                                                            const double *__restrict__ B, long long ldb,
                                                            double *__restrict__ C, long long ldc,
                                                            long long M, long long N,
                                                            const long long *__restrict__ ktile, int accumulate) {
    __shared__ double As[TS][TK + 1];
    __shared__ double Bs[TK][TS];
    const unsigned nt = (unsigned)((N + TS - 1) / TS), mt = blockIdx.x / nt;
    const long long m0 = (long long)mt * TS, n0 = (long long)(blockIdx.x - mt * nt) * TS;
    const long long K = ktile[m0 / TM];
    const int tx = threadIdx.x % TS, ty = threadIdx.x / TS;
    const int ar = threadIdx.x / TK, ac = threadIdx.x % TK;
    double acc = 0.0;
    for (long long k0 = 0; k0 < K; k0 += TK) {
#pragma unroll
        for (int i = 0; i < TS; i += kThreads / TK) {
            const long long gr = m0 + ar + i, gc = k0 + ac;
            As[ar + i][ac] = (gr < M && gc < K) ? A[gr * lda + gc] : 0.0;
        }
#pragma unroll
        for (int i = 0; i < TK; i += kThreads / TS) {
            const long long gr = k0 + ty + i, gc = n0 + tx;
            Bs[ty + i][tx] = (gr < K && gc < N) ? B[gr * ldb + gc] : 0.0;
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < TK; ++k) acc = fma(As[ty][k], Bs[k][tx], acc);
        __syncthreads();
    }
    const long long r = m0 + ty, c = n0 + tx;
    if (r < M && c < N) C[r * ldc + c] = accumulate ? C[r * ldc + c] + acc : acc;
}

void gemm_fp64_nn_ragged(const double *A, long long lda, const double *B, long long ldb, double *C,
                         long long ldc, long long M, long long N, const long long *ktile, int tileM,
                         cudaStream_t s, bool accumulate) {
    if (M <= 0 || N <= 0) return;
    if (tileM != TM) throw Error{QDT_ERR_ARG, "ragged GEMM tile mismatch"};
    const long long tiles = ((N + TS - 1) / TS) * ((M + TS - 1) / TS);
    if (tiles > 0x7fffffffLL) throw Error{QDT_ERR_ARG, "FP64 GEMM: too many tiles"};
    dgemm_nn_ragged<<<(unsigned)tiles, kThreads, 0, s>>>(A, lda, B, ldb, C, ldc, M, N, ktile, accumulate ? 1 : 0);
    QDT_CHECK_LAUNCH();
}

// C (N x N) = A^T B over K rows; upper 64 x 64 tiles (bi <= bj; without `whole` only what
// the packer reads of the diagonal ones), TS x TS of them per CTA; split-K slices
// write partial[slice][N][N]; a second kernel sums slices in fixed order and
// mirrors nothing (only the upper tiles are consumed by the packer).
__global__ void __launch_bounds__(kThreads) dgemm_tn_upper(const double *__restrict__ A, long long lda,
                                                           const double *__restrict__ B, long long ldb,
                                                           double *__restrict__ P, long long N, long long K,
                                                           long long kchunk, int ntb, int whole) {
    constexpr int kSub = TM / TS;
    __shared__ double As[TK][TS];
    __shared__ double Bs[TK][TS];
    // decode the upper tile index
    const int sub = blockIdx.x % (kSub * kSub);
    int t = blockIdx.x / (kSub * kSub), bi = 0;
    while (t >= ntb - bi) { t -= ntb - bi; ++bi; }
    const int bj = bi + t;
    const long long m0 = (long long)bi * TM + sub / kSub * TS, n0 = (long long)bj * TM + sub % kSub * TS;
    if (m0 >= N || n0 >= N || (!whole && m0 > n0)) return;
    const long long kb = (long long)blockIdx.y * kchunk, ke = min(K, kb + kchunk);
    const int tx = threadIdx.x % TS, ty = threadIdx.x / TS;
    double acc = 0.0;
    for (long long k0 = kb; k0 < ke; k0 += TK) {
#pragma unroll
        for (int i = 0; i < TK; i += kThreads / TS) {
            const long long gk = k0 + ty + i;
            As[ty + i][tx] = (gk < ke && m0 + tx < N) ? A[gk * lda + m0 + tx] : 0.0;
            Bs[ty + i][tx] = (gk < ke && n0 + tx < N) ? B[gk * ldb + n0 + tx] : 0.0;
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < TK; ++k) acc = fma(As[k][ty], Bs[k][tx], acc);
        __syncthreads();
    }
    const long long r = m0 + ty, c = n0 + tx;
    if (r < N && c < N) P[(long long)blockIdx.y * N * N + r * N + c] = acc;
}

__global__ void reduce_slices(const double *P, int nslice, long long NN, double *C, int accumulate) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < NN;
         i += (long long)gridDim.x * blockDim.x) {
        double s = accumulate ? C[i] : 0.0;
        for (int k = 0; k < nslice; ++k) s += P[k * NN + i];
        C[i] = s;
    }
}

// C = A^T B (upper tiles valid).  `partial` must hold nslice * N * N doubles,
// nslice = partial_elems / (N*N) at most.
void gemm_fp64_tn_sym(const double *A, long long lda, const double *B, long long ldb, double *C,
                      long long N, long long K, double *partial, size_t partial_elems,
                      cudaStream_t s, bool whole) {
    if (N <= 0) return;
    int ntb = (int)((N + TM - 1) / TM);
    int ntiles = ntb * (ntb + 1) / 2;
    long long maxslice = (long long)(partial_elems / (size_t)(N * N));
    long long want = (2 * 152 + ntiles - 1) / ntiles;
    if (want < 1) want = 1;
    if (want > 64) want = 64;
    if (want > maxslice) want = maxslice;
    if (want < 1) throw Error{QDT_ERR_OOM, "no room for the second-half partial sums"};
    long long kchunk = (K + want - 1) / want;
    kchunk = ((kchunk + TK - 1) / TK) * TK;
    if (kchunk < TK) kchunk = TK;
    int nslice = (int)((K + kchunk - 1) / kchunk);
    if (nslice < 1) nslice = 1;
    dim3 grid(ntiles * (TM / TS) * (TM / TS), nslice);
    if (K > 0) {
        dgemm_tn_upper<<<grid, kThreads, 0, s>>>(A, lda, B, ldb, partial, N, K, kchunk, ntb, whole);
        QDT_CHECK_LAUNCH();
    } else {
        launch_zero(partial, N * N, s);
        nslice = 1;
    }
    long long NN = N * N;
    long long blocks = (NN + 255) / 256;
    if (blocks > 152 * 16) blocks = 152 * 16;
    reduce_slices<<<(unsigned)blocks, 256, 0, s>>>(partial, nslice, NN, C, 1);
    QDT_CHECK_LAUNCH();
}

}  // namespace qdt
