// Launches of the strip kernel (sosfilt_strip.cuh), section counts 5, 6.
#include <cstring>

#include "sosfilt_strip.cuh"

namespace sosk {

namespace {
template <int K, bool NORM, bool TC>
KernelOnce g_once;

template <int K, bool NORM, bool TC>
cudaError_t launch_one(const StripParams<K, TC> &P, cudaStream_t s) {
    using Sd = StripDims<K, TC>;
    auto kern = sos_strip_kernel<K, NORM, TC>;
    cudaError_t e = raise_smem_once(g_once<K, NORM, TC>, kern, Sd::SMEM);
    if (e != cudaSuccess) return e;
    kern<<<static_cast<unsigned>(P.cut.n_strips), Sd::THREADS, Sd::SMEM, s>>>(P);
    return cudaGetLastError();
}

template <int K, bool TC>
cudaError_t launch_flavour(const LaneParams<K> &p, const StripCut &cut, long long grid, cudaStream_t s) {
    StripParams<K, TC> P;
    std::memset(static_cast<void *>(&P), 0, sizeof(P));
    P.p = p;
    P.cut = cut;
    P.in_place = p.x == p.y;
    P.x_aligned = reinterpret_cast<uintptr_t>(p.x) % 16 == 0;
    P.y_aligned = reinterpret_cast<uintptr_t>(p.y) % 16 == 0;
    P.host_tickets = static_cast<unsigned long long>(p.n_tiles + grid);
    if constexpr (!TC) std::memcpy(P.g, p.gresp, sizeof P.g);
    return p.norm ? launch_one<K, true, TC>(P, s) : launch_one<K, false, TC>(P, s);
}

template <int K>
bool launch_k(const LaneParams<K> &p, long long grid, cudaStream_t s, cudaError_t &err) {
    StripCut cut;
    if (!p.tail || !p.gimg || !strip_cut(p.n, p.warm_rows, cut)) return false;
    if constexpr (K <= 2) {
        if (cut.strip_rows + cut.warm_rows <= kStripFmaRows) {
            err = launch_flavour<K, false>(p, cut, grid, s);
            return true;
        }
    }
    err = launch_flavour<K, true>(p, cut, grid, s);
    return true;
}
}  // namespace

#define SOSK_STRIP_INST(k)                                                                                    \
    template <>                                                                                               \
    bool launch_strip<k>(const LaneParams<k> &p, long long grid, cudaStream_t s, cudaError_t &err) {          \
        return launch_k<k>(p, grid, s, err);                                                                  \
    }
SOSK_STRIP_INST(5)
SOSK_STRIP_INST(6)
#undef SOSK_STRIP_INST

}  // namespace sosk
