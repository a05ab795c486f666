// One element through k_contract with coefficients of the caller's choice: the
// blocks before elimination, which no library call returns.
#include <vector>

#include "kernels.cuh"

using namespace hdg;

namespace {

std::vector<void*> g_bufs;

template <class T>
T* up(const std::vector<T>& v) {
    T* p = nullptr;
    if (cudaMalloc((void**)&p, sizeof(T) * v.size()) != cudaSuccess) return nullptr;
    g_bufs.push_back(p);
    if (cudaMemcpy(p, v.data(), sizeof(T) * v.size(), cudaMemcpyHostToDevice) != cudaSuccess) return nullptr;
    return p;
}

template <class T>
std::vector<T> as(const double* x, size_t n) {
    return std::vector<T>(x, x + n);
}

template <class T>
int down(const T* d, size_t n, double* out) {
    std::vector<T> v(n);
    if (cudaMemcpy(v.data(), d, sizeof(T) * n, cudaMemcpyDeviceToHost) != cudaSuccess) return 1;
    std::copy(v.begin(), v.end(), out);
    return 0;
}

template <int D, int P, class TA>
int run(const double* vcoef, const double* fcoef, const double* taup, const double* geo, double dt, double a_ii,
        double tau, double* a11, double* a12, double* a21, double* a22) {
    using C = Cfg<D, P>;
    using S = ContractShape<C, TA>;
    constexpr size_t NU = C::NU, NT = C::NT, MM = C::M * C::M;
    RefTables t;
    build_ref_tables(D, P, t);
    auto f32 = [](const std::vector<double>& v) { return std::vector<float>(v.begin(), v.end()); };
    BlkArgs<TA> A{};
    A.tab.dphi = up(t.dphi); A.tab.mu = up(t.mu); A.tab.wf = up(t.wf); A.tab.mf = up(t.mf); A.tab.mhat = up(t.mhat);
    A.tab.minv_c = up(t.minv_c); A.tab.minv_e = up(t.minv_e); A.tab.b1 = up(t.b1); A.tab.node_face = up(t.node_face);
    A.tab.fdphi = up(f32(t.dphi)); A.tab.fmu = up(f32(t.mu));
    A.vcoef = up(as<TA>(vcoef, MM * S::CV));
    A.fcoef = up(as<TA>(fcoef, MM * S::CF));
    A.geo = up(as<double>(geo, Geo<D>::N));
    A.taup = taup ? up(as<double>(taup, C::NF * C::NFQ)) : nullptr;
    A.dt = dt; A.a_ii = a_ii; A.tau = tau;
    auto& R = A.R;
    R.a11 = up(std::vector<double>(NU * NU)); R.a11_es = NU * NU; R.a11_rs = NU;
    R.a12 = up(std::vector<TA>(NU * NT)); R.a12_es = NU * NT; R.a12_rs = NT;
    R.a21 = up(std::vector<TA>(NT * NU)); R.a21_es = NT * NU; R.a21_rs = NU;
    R.a22 = up(std::vector<TA>(NT * NT)); R.a22_es = NT * NT; R.a22_rs = NT;
    int rc = 0;
    for (void* p : g_bufs) rc |= p == nullptr;
    if (g_bufs.size() != (taup ? 19u : 18u)) rc = 1;
    if (!rc) rc = cudaFuncSetAttribute(k_contract<C, TA, TA>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)S::smem_bytes) != cudaSuccess;
    if (!rc) {
        k_contract<C, TA, TA><<<S::NG, S::NTH, S::smem_bytes>>>(A);
        rc = cudaGetLastError() != cudaSuccess || cudaDeviceSynchronize() != cudaSuccess;
    }
    if (!rc) rc = down(R.a11, NU * NU, a11) | down(R.a12, NU * NT, a12) | down(R.a21, NT * NU, a21) | down(R.a22, NT * NT, a22);
    for (void* p : g_bufs) cudaFree(p);
    g_bufs.clear();
    return rc;
}

}  // namespace

extern "C" int contract_one(int d, int p, int fp32, const double* vcoef, const double* fcoef, const double* taup,
                            const double* geo, double dt, double a_ii, double tau, double* a11, double* a12,
                            double* a21, double* a22) {
#define CASE(D, P)                                                                                                \
    if (d == D && p == P)                                                                                         \
        return fp32 ? run<D, P, float>(vcoef, fcoef, taup, geo, dt, a_ii, tau, a11, a12, a21, a22)                 \
                    : run<D, P, double>(vcoef, fcoef, taup, geo, dt, a_ii, tau, a11, a12, a21, a22);
    CASE(2, 2)
    CASE(3, 2)
    return 2;
}
