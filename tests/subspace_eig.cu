// The subspace eigensolver of csrc/jacobi.cuh on given matrices, for
// test_gpu_subspace_signs.py.  G: m x m (leading dimension 64) whose leading
// m_prev block is decomposed first, from nothing; then the whole of it from that,
// in one of the ways below.
#include "jacobi.cuh"

using namespace shci;

// how 0: subspace_eig with signs, 1: jacobi_solve, 2: append_eig vector by vector (*did: how many it took)
__global__ void k_test(const double *G, int m, int m_prev, int how, double *eval, double *evec, int *did) {
    extern __shared__ double jsm[];
    constexpr int ld = SHCI_MAX_SUB;
    if (m_prev > 0) jacobi_solve(G, ld, m_prev, 0, eval, evec, jsm);
    __syncthreads();
    if (how == 0) {
        subspace_eig<true, true>(G, ld, m, m_prev, eval, evec, jsm);
    } else if (how == 1) {
        jacobi_solve(G, ld, m, m_prev, eval, evec, jsm);
    } else {
        int have = m_prev;
        while (have < m && append_eig(G, ld, have, eval, evec, jsm)) have++;
        if (threadIdx.x == 0) *did = have - m_prev;
    }
}

// host arrays: G [64][64], eval [64], evec [64][64]; a CUDA error code
extern "C" int subspace_eig_test(const double *G, int m, int m_prev, int how, double *eval, double *evec, int *did) {
    constexpr size_t MAT = sizeof(double) * SHCI_MAX_SUB * SHCI_MAX_SUB, VEC = sizeof(double) * SHCI_MAX_SUB;
    if (m < 1 || m > SHCI_MAX_SUB || m_prev < 0 || m_prev > m || (how == 2 && m_prev < 1)) return -1;
    char *p = nullptr;
    cudaError_t e = cudaMalloc((void **)&p, 2 * MAT + VEC + sizeof(int));
    if (e != cudaSuccess) return (int)e;
    double *dG = (double *)p, *dv = (double *)(p + MAT), *dl = (double *)(p + 2 * MAT);
    int *dn = (int *)(p + 2 * MAT + VEC);
    cudaMemset(p, 0, 2 * MAT + VEC + sizeof(int));
    cudaMemcpy(dG, G, MAT, cudaMemcpyHostToDevice);
    cudaFuncSetAttribute(k_test, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)JACOBI_SMEM_SIGNS);
    k_test<<<1, 256, JACOBI_SMEM_SIGNS>>>(dG, m, m_prev, how, dl, dv, dn);
    e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaMemcpy(eval, dl, VEC, cudaMemcpyDeviceToHost);
    if (e == cudaSuccess) e = cudaMemcpy(evec, dv, MAT, cudaMemcpyDeviceToHost);
    if (e == cudaSuccess) e = cudaMemcpy(did, dn, sizeof(int), cudaMemcpyDeviceToHost);
    cudaFree(p);
    return (int)e;
}
