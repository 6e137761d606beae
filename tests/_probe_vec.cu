// The L-BFGS direction and the line search's scalar arithmetic by themselves (test
// helper, compiled by the test against the library).
#include "../paper_2412_14973_gb300/csrc/k_vec.cu"

namespace {

__global__ void k_scalar(const double* x, double* r, double* c, int n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    r[i] = tlr::recip(x[i]);
    c[i] = tlr::cube_root(x[i]);
}
__global__ void k_argmin(const double* c, double* a, int* ok, int n) {
    const int w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (w >= n) return;
    double v = 0.0;
    const bool f = tlr::quartic_argmin(c + 5 * w, lane, &v);
    if (lane == 0) {
        a[w] = v;
        ok[w] = f;
    }
}

}  // namespace

extern "C" {

int probe_scalar(const double* x, double* r, double* c, int n) {
    k_scalar<<<(n + 127) / 128, 128>>>(x, r, c, n);
    return cudaDeviceSynchronize();
}
int probe_argmin(const double* c, double* a, int* ok, int n) {
    k_argmin<<<(n + 3) / 4, 128>>>(c, a, ok, n);
    return cudaDeviceSynchronize();
}

// The direction with cnt pairs stored, the newest in slot newest of m + 1; all DEVICE.
// SY, YY: (m + 1)^2 by slot, kept by the caller from pair to pair; sums: the inner
// products' cluster sums summed up on the host, 5 (cnt) + 1 of them.
int probe_direction(long long n2, int m, int cnt, int newest, float* x, float* v, float* g, float* d, float* sh,
                    float* yh, double* SY, double* YY, double* sums) {
    using namespace tlr;
    char* buf = nullptr;
    const size_t doubles = 64 + (size_t)kLbPartDoubles + 16 + 3 * kRedBlocks;
    const size_t ints = CT_DIR + 1 + kLbClusters;
    cudaError_t e = cudaMalloc((void**)&buf, doubles * 8 + ints * 4);
    if (e == cudaSuccess) e = cudaMemset(buf, 0, doubles * 8 + ints * 4);
    if (e != cudaSuccess) return e;
    double* p = reinterpret_cast<double*>(buf);
    SolverDev S;
    memset(&S, 0, sizeof(S));
    S.n2 = n2, S.m = m, S.ring = m + 1;
    S.x = x, S.v = v, S.g = g, S.d = d, S.sh = sh, S.yh = yh;
    S.SYm = SY, S.YYm = YY;
    S.acoef = p;
    S.lbpart = p + 64;
    S.lbsum = S.lbpart + kLbSumOff;
    S.sc = S.lbpart + kLbPartDoubles;
    S.part3 = S.sc + 16;
    S.ints = reinterpret_cast<int*>(p + doubles);
    S.lbctr = reinterpret_cast<unsigned*>(S.ints + CT_DIR);
    int head[2] = {cnt, newest};
    static_assert(SI_CNT == 0 && SI_NEWEST == 1, "the first two counters");
    e = cudaMemcpy(S.ints, head, sizeof(head), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = sv_direction(S, 0);
    static double part[kLbGroups * kLbClusters * kLbRow];
    static unsigned ctr[1 + kLbClusters];
    if (e == cudaSuccess) e = cudaMemcpy(part, S.lbsum, sizeof(part), cudaMemcpyDeviceToHost);
    if (e == cudaSuccess) e = cudaMemcpy(ctr, S.lbctr, sizeof(ctr), cudaMemcpyDeviceToHost);
    cudaFree(buf);
    for (unsigned c : ctr)
        if (c != 0) return -1;   // the block counters are zero between launches
    for (int k = 0; k <= 5 * cnt; ++k) {
        const int grp = k == 5 * cnt ? 0 : k / (5 * kLbGroup), t = k == 5 * cnt ? kLbVals - 1 : k % (5 * kLbGroup);
        sums[k] = 0.0;
        for (int c = 0; c < kLbClusters; ++c) sums[k] += part[(grp * kLbClusters + c) * kLbRow + t];
    }
    return e;
}

}  // extern "C"
