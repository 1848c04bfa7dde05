// One variant of the TMA-staged substep kernel: order RTPN_SN, CTA tile RTPN_STX x RTPN_STY x
// RTPN_STZ, RTPN_SNB stage buffers, RTPN_SEM sub-stages per column, both target classes, FP32 and
// BF16 storage; RTPN_SSC = 1: form SC, for cells with h_y != h_x.  kernels_stage.cu dispatches to it.
#include "stage_impl.cuh"

#if !defined(RTPN_SN) || !defined(RTPN_STX) || !defined(RTPN_STY) || !defined(RTPN_STZ) || !defined(RTPN_SNB) || \
    !defined(RTPN_SEM) || !defined(RTPN_SSC)
#error "compile with -DRTPN_SN=<order> -DRTPN_STX=.. -DRTPN_STY=.. -DRTPN_STZ=.. -DRTPN_SNB=.. -DRTPN_SEM=.. -DRTPN_SSC=0|1"
#endif

#define RTPN_SCAT2(a, b, c, d, e, f, g, h) a##_##b##_##c##_##d##_##e##_##f##_##g##_##h
#define RTPN_SCAT(a, b, c, d, e, f, g, h) RTPN_SCAT2(a, b, c, d, e, f, g, h)
#define RTPN_SVARIANT(name) RTPN_SCAT(name, RTPN_SN, RTPN_STX, RTPN_STY, RTPN_STZ, RTPN_SNB, RTPN_SEM, RTPN_SSC)

namespace rtpn {
namespace stg {

// Everything but the uniquely named entry points has internal linkage: every variant of this file
// defines a k_stage / launch_one of the same name, and the linker must not merge them.
namespace {

constexpr int kN = RTPN_SN, kTX = RTPN_STX, kTY = RTPN_STY, kTZ = RTPN_STZ, kNB = RTPN_SNB, kCH = RTPN_SEM;
constexpr bool kSC = RTPN_SSC != 0;
constexpr int kThreads = Layout<kN, 0, float, kTX, kTY, kTZ, kNB, kCH, kSC>::THREADS;
// Two CTAs per SM where two rings fit shared memory (228 KB, 1 KB of it reserved per CTA) and the
// registers that leaves a thread hold its window (six accumulators per slot) and 48 more; one
// otherwise.  A second CTA fills the issue slots while the first waits for a stage: P15, 96 x 96 x
// 128 cells, 64x2x2 tiles on a GB300: 0.351 ms a pass with two three-buffer CTAs per SM, 0.397 ms with
// one five-buffer CTA.
constexpr int kWarpsPerScheduler2 = (2 * (kThreads / 32) + 3) / 4;
constexpr int kRegs2 = 512 / kWarpsPerScheduler2 / 8 * 8;
template <typename S>
constexpr int min_blocks() {
    return 2 * (Layout<kN, 0, S, kTX, kTY, kTZ, kNB, kCH, kSC>::BYTES + 1024) <= 233472 && kRegs2 >= 6 * (kN / 2 + 1) + 48 ? 2 : 1;
}

// both forms of a variant run on the same storage types
static_assert(Layout<kN, 0, float, kTX, kTY, kTZ, kNB, kCH, true>::FITS == Layout<kN, 0, float, kTX, kTY, kTZ, kNB, kCH>::FITS &&
                  Layout<kN, 0, __nv_bfloat16, kTX, kTY, kTZ, kNB, kCH, true>::FITS ==
                      Layout<kN, 0, __nv_bfloat16, kTX, kTY, kTZ, kNB, kCH>::FITS,
              "form SC fits shared memory where the plain form does");

template <int A, typename S, int MODE>
__global__ void __launch_bounds__(kThreads, min_blocks<S>()) k_stage(Args a) {
    static_assert(Layout<kN, A, S, kTX, kTY, kTZ, kNB, kCH, kSC>::FITS, "stage ring exceeds shared memory");
    extern __shared__ __align__(128) unsigned char smem[];
    stage_kernel_body<kN, A, S, kTX, kTY, kTZ, kNB, kCH, MODE, kSC>(a, smem);
}

template <int A, typename S, int MODE>
int launch_one(const Args& a, int sms, cudaStream_t st) {
    using L = Layout<kN, A, S, kTX, kTY, kTZ, kNB, kCH, kSC>;
    if constexpr (!L::FITS) {
        return (int)cudaErrorNotSupported;  // this depth is compiled for the narrower storage only
    } else {
    static bool configured[64] = {};
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev < 0 || dev >= 64) return (int)cudaErrorInvalidDevice;
    if (!configured[dev]) {
        cudaError_t e = cudaFuncSetAttribute(k_stage<A, S, MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             L::BYTES);
        if (e != cudaSuccess) return (int)e;
        configured[dev] = true;
    }
    int per_sm = 0;
    cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_stage<A, S, MODE>, kThreads, L::BYTES);
    if (e != cudaSuccess) return (int)e;
    if (per_sm < 1) return (int)cudaErrorLaunchOutOfResources;
    long long grid = (long long)per_sm * sms;
    if (grid > a.tiles) grid = a.tiles;
    if (grid < 1) return 0;
    k_stage<A, S, MODE><<<(unsigned)grid, kThreads, L::BYTES, st>>>(a);
    return (int)cudaGetLastError();
    }
}

// dynamic shared memory of the variant, or 0 if it does not fit a CTA
template <int A, typename S>
constexpr int smem_of() {
    using L = Layout<kN, A, S, kTX, kTY, kTZ, kNB, kCH, kSC>;
    return L::FITS ? L::BYTES : 0;
}
// box geometry of the variant for a storage precision (the host builds its tensor maps with it):
// out = {maps per kind, CTAs per SM, x halo group width, x halo group rows}
template <typename S>
void geom_of(int* out) {
    using L = Layout<kN, 0, S, kTX, kTY, kTZ, kNB, kCH, kSC>;
    out[0] = L::NMAP;
    out[1] = min_blocks<S>();
    out[2] = L::XW;
    out[3] = L::RY;
}

}  // namespace

// mode FORWARD: FP32 or BF16 storage; mode ADJ_SOURCES: FP32 (the adjoint)
int RTPN_SVARIANT(stage_launch)(int cls, int precision, int mode, const Args& a, int sms, cudaStream_t st) {
    if (mode == ADJ_SOURCES) {
        if (precision != RTPN_FP32) return (int)cudaErrorNotSupported;
        return cls == 0 ? launch_one<0, float, ADJ_SOURCES>(a, sms, st) : launch_one<1, float, ADJ_SOURCES>(a, sms, st);
    }
    if (precision == RTPN_BF16)
        return cls == 0 ? launch_one<0, __nv_bfloat16, FORWARD>(a, sms, st)
                        : launch_one<1, __nv_bfloat16, FORWARD>(a, sms, st);
    return cls == 0 ? launch_one<0, float, FORWARD>(a, sms, st) : launch_one<1, float, FORWARD>(a, sms, st);
}

void RTPN_SVARIANT(stage_geom)(int precision, int* out) {
    if (precision == RTPN_BF16)
        geom_of<__nv_bfloat16>(out);
    else
        geom_of<float>(out);
}

int RTPN_SVARIANT(stage_smem)(int cls, int precision) {
    if (precision == RTPN_BF16) return cls == 0 ? smem_of<0, __nv_bfloat16>() : smem_of<1, __nv_bfloat16>();
    return cls == 0 ? smem_of<0, float>() : smem_of<1, float>();
}

}  // namespace stg
}  // namespace rtpn
