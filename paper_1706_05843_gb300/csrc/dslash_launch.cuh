// dslash_launch.cuh -- host-side dispatch of hop_kernel over (Ls, kind, tile
// variant) for one storage type.  Included by dslash_<prec>.cu (the four
// kinds of the inner CG: the Schur complement and its adjoint) and by
// dslash_<prec>_outer.cu (the FP64/FP32 outer-solver kinds), so the kernel
// instantiations compile as separate translation units.  The inner kinds
// exist in every tile variant the autotuner times (two CTA shapes, and for
// FP32 arithmetic each with and without a register cap); the others in
// the default variant only.
#pragma once

#include <atomic>
#include <mutex>

#include "dslash.cuh"

namespace eofa {

// devices a process may use the hop kernels on
constexpr int kHopMaxDevices = 64;

// The CTAs of one kernel that one SM holds, on the current device (the
// persistent grids are that many per SM).  Once per kernel and device, before
// its first launch there: the shared-memory limit, an attribute of the current
// device; not inside a stream capture (a context sets up its applications'
// kernels when it is created and a solve's before the first capture:
// prepare_solve).
struct HopResident {
    std::atomic<int> of[kHopMaxDevices] = {};
    std::mutex mu;
};
template <typename F>
static cudaError_t hop_resident(HopResident& r, F* kernel, int nt, size_t smem, cudaStream_t st, int* dev,
                                int* resident) {
    cudaError_t e = cudaGetDevice(dev);
    if (e != cudaSuccess) return e;
    if (*dev < 0 || *dev >= kHopMaxDevices) return cudaErrorInvalidDevice;
    *resident = r.of[*dev].load(std::memory_order_acquire);
    if (*resident) return cudaSuccess;
    std::lock_guard<std::mutex> lock(r.mu);
    *resident = r.of[*dev].load(std::memory_order_relaxed);
    if (*resident) return cudaSuccess;
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(st, &cs) != cudaSuccess || cs != cudaStreamCaptureStatusNone)
        return cudaErrorStreamCaptureUnsupported;
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(resident, kernel, nt, smem);
    if (e != cudaSuccess) return e;
    *resident = std::max(*resident, 1);
    r.of[*dev].store(*resident, std::memory_order_release);
    return cudaSuccess;
}

template <typename S, int LS, int K, int VAR>
static cudaError_t resident_one(cudaStream_t st, int* dev, int* resident) {
    static HopResident r;
    constexpr int NT = HopTile<S, LS, K, VAR>::NT;
    const size_t smem = hop_smem_bytes<S, LS, K, VAR>();
    static_assert(hop_smem_bytes<S, LS, K, VAR>() <= 232448, "tile exceeds the 227 KB of shared memory per CTA");
    if constexpr ((VAR & 2) != 0) return hop_resident(r, hop_kernel_rc<S, LS, K, VAR>, NT, smem, st, dev, resident);
    else return hop_resident(r, hop_kernel<S, LS, K, VAR>, NT, smem, st, dev, resident);
}

template <typename S, int LS, int K, int VAR>
static cudaError_t launch_one(const HopArgs& a, const SCoef<typename Traits<S>::R>& c,
                              cudaStream_t st) {
    constexpr int NS = HopTile<S, LS, K, VAR>::NS;
    constexpr int NT = HopTile<S, LS, K, VAR>::NT;
    const size_t smem = hop_smem_bytes<S, LS, K, VAR>();
    constexpr bool RCAP = (VAR & 2) != 0;
    int dev = 0, resident = 0;
    cudaError_t e = resident_one<S, LS, K, VAR>(st, &dev, &resident);
    if (e != cudaSuccess || a.prepare) return e;
    const long nblk = ((long)a.g.Vh + NS - 1) / NS;
    if (nblk == 0) return cudaSuccess;
    int sms = 0;
    e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    const int grid = (int)std::min<long>(nblk, (long)resident * sms);
    if constexpr (RCAP) hop_kernel_rc<S, LS, K, VAR><<<grid, NT, smem, st>>>(a, c);
    else hop_kernel<S, LS, K, VAR><<<grid, NT, smem, st>>>(a, c);
    return cudaGetLastError();
}

template <typename S, int LS, int K>
static cudaError_t resident_pair(cudaStream_t st, int* dev, int* resident) {
    static HopResident r;
    return hop_resident(r, hop_kernel_pair<S, LS, K>, HopTile<S, LS, K, 0>::NT, hop_smem_bytes<S, LS, K, 0>(), st, dev,
                        resident);
}

// An application's two hops (p.a[0], p.a[1]; FP64).  Up to 8 rounds of
// resident CTAs they share one grid (K at 4^4, Ls = 8: 21 us against 36 us for
// a grid each; 8^3x16, Ls = 8: 54 against 64 us; 16^4, Ls = 8, seven rounds: 325
// against 335 us); larger lattices fill the SMs with a grid each (12^3x24, Ls =
// 16, 8.5 rounds: 390 us in both; 16^4, Ls = 16, 13.5 rounds: K 613 us in one
// grid, 608 us in two, H 704 and 692 us).
template <typename S, int LS, int K>
static cudaError_t launch_pair(const HopPair& p, const SCoef<typename Traits<S>::R>& c, cudaStream_t st) {
    constexpr int NS = HopTile<S, LS, K, 0>::NS;
    constexpr int NT = HopTile<S, LS, K, 0>::NT;
    const size_t smem = hop_smem_bytes<S, LS, K, 0>();
    int dev = 0, resident = 0, sms = 0;
    cudaError_t e = resident_pair<S, LS, K>(st, &dev, &resident);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    const long nblk = ((long)p.a[0].g.Vh + NS - 1) / NS, full = (long)resident * sms;
    if (nblk > 8 * full) {
        e = launch_one<S, LS, K, 0>(p.a[0], c, st);
        return e != cudaSuccess ? e : launch_one<S, LS, K, 0>(p.a[1], c, st);
    }
    const dim3 grid((unsigned)std::min<long>(nblk, std::max<long>(1, full / 2)), 2);
    hop_kernel_pair<S, LS, K><<<grid, NT, smem, st>>>(p, c);
    return cudaGetLastError();
}

// the FP64 applications: kinds KIND_FULL, KIND_FULL_DAG, KIND_H
template <int LS>
static cudaError_t launch_pair_ls(int kind, const HopPair& p, const SCoef<double>& c, cudaStream_t st) {
    switch (kind) {
        case KIND_FULL: return launch_pair<double, LS, KIND_FULL>(p, c, st);
        case KIND_FULL_DAG: return launch_pair<double, LS, KIND_FULL_DAG>(p, c, st);
        case KIND_H: return launch_pair<double, LS, KIND_H>(p, c, st);
        default: return cudaErrorNotSupported;
    }
}

// both forms of every application's kernel
template <int LS>
static cudaError_t setup_apply_ls(cudaStream_t st) {
    int dev, n;
    cudaError_t e = cudaSuccess;
    auto one = [&](cudaError_t r) { if (e == cudaSuccess) e = r; };
    one(resident_pair<double, LS, KIND_FULL>(st, &dev, &n));
    one(resident_pair<double, LS, KIND_FULL_DAG>(st, &dev, &n));
    one(resident_pair<double, LS, KIND_H>(st, &dev, &n));
    one(resident_one<double, LS, KIND_FULL, 0>(st, &dev, &n));
    one(resident_one<double, LS, KIND_FULL_DAG, 0>(st, &dev, &n));
    one(resident_one<double, LS, KIND_H, 0>(st, &dev, &n));
    return e;
}

template <typename S, int LS, int K>
static cudaError_t launch_var(const HopArgs& a, const SCoef<typename Traits<S>::R>& c, cudaStream_t st) {
    if constexpr (kTileVariants<S> == 4) {
        switch (a.tile_var) {
            case 1: return launch_one<S, LS, K, 1>(a, c, st);
            case 2: return launch_one<S, LS, K, 2>(a, c, st);
            case 3: return launch_one<S, LS, K, 3>(a, c, st);
            default: return launch_one<S, LS, K, 0>(a, c, st);
        }
    } else {
        return (a.tile_var & 1) ? launch_one<S, LS, K, 1>(a, c, st) : launch_one<S, LS, K, 0>(a, c, st);
    }
}

template <typename S, int LS>
static cudaError_t launch_inner_ls(int kind, const HopArgs& a, const SCoef<typename Traits<S>::R>& c,
                                   cudaStream_t st) {
    switch (kind) {
        case KIND_R_EO: return launch_var<S, LS, KIND_R_EO>(a, c, st);
        case KIND_R_OE: return launch_var<S, LS, KIND_R_OE>(a, c, st);
        case KIND_R_EO_DAG: return launch_var<S, LS, KIND_R_EO_DAG>(a, c, st);
        case KIND_R_OE_DAG: return launch_var<S, LS, KIND_R_OE_DAG>(a, c, st);
        default: return cudaErrorNotSupported;
    }
}

// FP32: the adjoint halves serve the training solves; FP64: the operators
// of the outer solver and of the applications
template <typename S, int LS>
static cudaError_t launch_outer_ls(int kind, const HopArgs& a, const SCoef<typename Traits<S>::R>& c,
                                   cudaStream_t st) {
    if constexpr (sizeof(S) == 8) {
        switch (kind) {
            case KIND_RECON: return launch_one<S, LS, KIND_RECON, 0>(a, c, st);
            case KIND_SRC: return launch_one<S, LS, KIND_SRC, 0>(a, c, st);
            case KIND_FULL: return launch_one<S, LS, KIND_FULL, 0>(a, c, st);
            case KIND_FULL_DAG: return launch_one<S, LS, KIND_FULL_DAG, 0>(a, c, st);
            case KIND_LOC_DTMINV: return launch_one<S, LS, KIND_LOC_DTMINV, 0>(a, c, st);
            case KIND_LOC_DT: return launch_one<S, LS, KIND_LOC_DT, 0>(a, c, st);
            default: break;
        }
    } else {
        switch (kind) {
            case KIND_EO_MINV_DAG: return launch_one<S, LS, KIND_EO_MINV_DAG, 0>(a, c, st);
            case KIND_OE_SCHUR_DAG: return launch_one<S, LS, KIND_OE_SCHUR_DAG, 0>(a, c, st);
            default: break;
        }
    }
    switch (kind) {
        case KIND_EO_MINV: return launch_one<S, LS, KIND_EO_MINV, 0>(a, c, st);
        case KIND_OE_SCHUR: return launch_one<S, LS, KIND_OE_SCHUR, 0>(a, c, st);
        case KIND_LOC_DTINV: return launch_one<S, LS, KIND_LOC_DTINV, 0>(a, c, st);
        case KIND_R_BACK: return launch_one<S, LS, KIND_R_BACK, 0>(a, c, st);
        case KIND_D_EO: return launch_one<S, LS, KIND_D_EO, 0>(a, c, st);
        case KIND_D_OE: return launch_one<S, LS, KIND_D_OE, 0>(a, c, st);
        case KIND_D_EO_DAG: return launch_one<S, LS, KIND_D_EO_DAG, 0>(a, c, st);
        case KIND_D_OE_DAG: return launch_one<S, LS, KIND_D_OE_DAG, 0>(a, c, st);
        default: return cudaErrorNotSupported;
    }
}

// the halves of the inner operator (every storage type)
template <typename S>
static cudaError_t launch_inner_t(int kind, const HopArgs& a, const void* coef, cudaStream_t st) {
    typedef typename Traits<S>::R R;
    const SCoef<R>& c = *reinterpret_cast<const SCoef<R>*>(coef);
    switch (a.g.Ls) {
        case 4: return launch_inner_ls<S, 4>(kind, a, c, st);
        case 8: return launch_inner_ls<S, 8>(kind, a, c, st);
        case 12: return launch_inner_ls<S, 12>(kind, a, c, st);
        case 16: return launch_inner_ls<S, 16>(kind, a, c, st);
        default: return cudaErrorNotSupported;
    }
}

// every other kind (FP64 and FP32 storage)
template <typename S>
static cudaError_t launch_outer_t(int kind, const HopArgs& a, const void* coef, cudaStream_t st) {
    typedef typename Traits<S>::R R;
    const SCoef<R>& c = *reinterpret_cast<const SCoef<R>*>(coef);
    switch (a.g.Ls) {
        case 4: return launch_outer_ls<S, 4>(kind, a, c, st);
        case 8: return launch_outer_ls<S, 8>(kind, a, c, st);
        case 12: return launch_outer_ls<S, 12>(kind, a, c, st);
        case 16: return launch_outer_ls<S, 16>(kind, a, c, st);
        default: return cudaErrorNotSupported;
    }
}

}  // namespace eofa
