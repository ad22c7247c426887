// Device check of the records of kept.cuh: the diagonal of each red node, which scales the
// residual handed to the children, is the FP32 sum of its four faces, bit for bit.
// Built and run by tests/test_gpu_kept_records.py.
#include "../paper_1907_12334_gb300/csrc/solver.cu"
#include <cstdio>
#include <random>
using namespace msg;

__global__ void k_records(SampleInfo S, const float* ax, const float* ay, float* got, float* want)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int2 at[kMidMax + 1];
    const MidItem<float> m = mid_item<float>((float*)smem_raw, at, kMidD + 1, kMidD + 1, kOpD + 1, kOpD + 1 + kKeepMid, kMidD, 2);
    const KeptTables t = kept_tables(m, kKeepMid, 2);
    __syncthreads();
    for (int x = 0; x < kKeepMid; ++x) kept_load(m, t, kOpD + 1 + x, S, ax, ay);
    __syncthreads();
    for (int x = 0; x < kKeepMid; ++x) {
        const int d = kOpD + 1 + x, k = x * blockDim.x + threadIdx.x;
        got[k] = want[k] = 0.f;
        if (!(t.last >> x & 1)) continue;
        const int p = mid_plo(d, m.qic) + (threadIdx.x >> (d + 1)), cell = (2 * threadIdx.x) & ((4 << d) - 1), W = (1 << p) + 1;
        const int j = cell >> p, i = (cell & ((1 << p) - 1)) + (j & 1);
        if (i == 0 || j == 0) continue;  // a boundary node
        const int o = grid_offset32(p, d + 2 - p, S.Q) + j * W + i;
        Pair<float> P;
        kept_pair(P, t, kept_row(t, x));
        got[k] = P.dR;
        want[k] = ax[o - 1] + ax[o] + ay[o - W] + ay[o];
    }
}

int main()
{
    const int P = kMidD + 1, n = (int)rect_nodes(P, P), nout = kKeepMid * kKeptThreads;
    std::mt19937 rng(3);
    std::uniform_real_distribution<float> u(0.5f, 100.f);
    std::vector<float> a(2 * n), r(2 * nout);
    for (float& v : a) v = u(rng);
    float *da, *dr;
    if (cudaMalloc(&da, sizeof(float) * a.size()) || cudaMalloc(&dr, sizeof(float) * r.size())) return 2;
    cudaMemcpy(da, a.data(), sizeof(float) * a.size(), cudaMemcpyHostToDevice);
    cudaFuncSetAttribute(k_records, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemMax - 1024);
    k_records<<<1, kKeptThreads, kept_mid_smem(2)>>>(SampleInfo{P, P, 0, 0, 0, 0}, da, da + n, dr, dr + nout);
    if (cudaMemcpy(r.data(), dr, sizeof(float) * r.size(), cudaMemcpyDeviceToHost) != cudaSuccess) return 2;
    int nodes = 0, bad = 0;
    for (int k = 0; k < nout; ++k) nodes += r[nout + k] != 0.f, bad += r[k] != r[nout + k];
    printf("%d red nodes, %d diagonals differ\n", nodes, bad);
    return bad || nodes != 367;  // red interior nodes: 103 of the five grids of diagonal 4, 264 of the six of diagonal 5
}
