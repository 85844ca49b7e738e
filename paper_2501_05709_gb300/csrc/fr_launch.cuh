// Host launchers of the FR kernels for one (precision, dimension) pair; the
// including translation unit defines FR_REAL and FR_DIM.
#include "fr_kernels.cuh"

#include <algorithm>

namespace frl {

namespace {

// Opt every kernel in to the full 227 KB of dynamic shared memory on its first
// use (a launch with E == 0 does only this), so that later launches of any
// tile size, including those recorded into a CUDA graph, need no attribute call.
// `done` belongs to the caller's own kernel instantiation (kernels of
// different orders share a signature, so the flag cannot live here).
template <typename K>
cudaError_t prep(K kernel, size_t smem, unsigned long long& done) {
    if (smem > 227 * 1024) return cudaErrorInvalidValue;
    // the attribute belongs to the function on the current device: one bit
    // of `done` per device
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const unsigned long long bit = 1ull << (dev & 63);
    if (done & bit) return cudaSuccess;
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
    // and to the largest shared-memory carveout: left to itself the driver
    // configured too little shared memory for the blocks that the registers
    // admit (four blocks per SM at p = 4 in 3D where five or six fit)
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout,
                                 int(cudaSharedmemCarveoutMaxShared));
    if (e == cudaSuccess) done |= bit;
    return e;
}

// kernels that run beside the element kernels ask for the same carveout (an SM
// holds one split of its memory at a time), on their first use on a device (`done` as
// for prep)
template <typename K>
int side_prep(K kernel, unsigned long long& done) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    const unsigned long long bit = 1ull << (dev & 63);
    if (e != cudaSuccess || (done & bit)) return int(e);
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, int(cudaSharedmemCarveoutMaxShared));
    if (e == cudaSuccess) done |= bit;
    return int(e);
}

inline unsigned grid_of(int64_t E, int epb) { return unsigned((E + epb - 1) / epb); }

inline int sm_count() {
    int dev = 0, n = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return 1;
    return n;
}
template <typename K>
int blocks_per_sm(K kernel, int threads, size_t smem) {
    int n = 0;
    if (threads > 1024 || cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kernel, threads, smem) != cudaSuccess) n = 0;
    return n;
}

// Default elements per block of a kernel (T threads an element, smem(epb) bytes a
// block) on E elements: the tile that keeps most warps resident, found by the
// occupancy calculator, since these kernels wait on latency (FP32) and an SM holds
// 16 to 24 of their warps: at p = 3 k_residual runs 92 us on the 32^3 box with 20
// warps (2 or 4 elements a block) and 108 us with 16 (8 a block), on 100,000 curved
// elements 319 against 342 us.  With fewer than 20 elements per SM the last wave
// counts more than the number of warps, and blocks of one element level it in FP64
// (2,400 curved elements: 420 us against 440 to 510 us with 2 to 8); in FP32 blocks
// of two do (2,310 elements at p = 4: 20 us, with 1: 26, with 8: 20 to 21; at p <= 3
// all within 2%).  `tie`: taken
// instead if it keeps three quarters of those warps (2 for the persistent face
// kernel, whose elements of a block wait for each other at every tile: box of 32^3
// at p = 4 with 2 elements a block 88 us, with 3: 94; p = 3 39.2 against 39.8).
template <typename K, typename S>
int best_tile(K kernel, int T, S smem, int64_t E, int tie = 0) {
    int best = 1, most = blocks_per_sm(kernel, T, smem(1));
    if (E < 20 * int64_t(sm_count())) return sizeof(FR_REAL) == 8 ? 1 : 2;
    // FP64 is bound by its pipe, not by latency: whole warps a block count (4,096
    // affine elements at p = 3: 427 us a stage with 4, 432 with 2)
    if (sizeof(FR_REAL) == 8 && smem(4) <= 113 * 1024 && blocks_per_sm(kernel, 4 * T, smem(4)) > 0) return 4;
    for (int epb : {8, 6, 1, 4, 3, 2}) {   // of equal ones the last
        const int n = smem(epb) <= 227 * 1024 ? epb * blocks_per_sm(kernel, T * epb, smem(epb)) : 0;
        if (n >= most) {
            most = n;
            best = epb;
        }
    }
    if (tie && 4 * tie * blocks_per_sm(kernel, T * tie, smem(tie)) >= 3 * most) best = tie;
    return best;
}

// every launcher below: lc.epb < 0 asks for the default tile for E elements (a
// positive result; nothing is launched), E = 0 only sets the kernel up
template <int P>
int traces_p(const FR_REAL* u, FR_REAL* uf, int64_t E, const frk::Ops<FR_REAL>& op, frk::Launch lc,
             cudaStream_t s) {
    auto k = frk::k_traces<FR_DIM, P, FR_REAL>;
    const auto smem = [](int n) { return frk::smem_traces<FR_DIM, P, FR_REAL>(n); };
    const size_t sm = smem(std::max(lc.epb, 1));
    static unsigned long long done = 0;
    cudaError_t e = prep(k, sm, done);
    if (lc.epb < 0 && sizeof(FR_REAL) == 4) {
        // a copy with a few operations a value: in FP32 it wants large blocks (residual
        // of 64,000 elements in 2D at p = 2 45 us with 8 elements a block, 54 with 2)
        int epb = 8;
        while (epb > 1 && smem(epb) > 96 * 1024) epb /= 2;
        return epb;
    }
    if (lc.epb < 0) return e == cudaSuccess ? best_tile(k, frk::Grp<FR_DIM, P>::T, smem, E) : 1;
    if (e != cudaSuccess) return int(e);
    static std::atomic<int> most{0};
    const int epb = frk::fit_tile(k, frk::Grp<FR_DIM, P>::T, lc.epb, most);
    if (E == 0) return 0;
    k<<<grid_of(E, epb), frk::Grp<FR_DIM, P>::T * epb, smem(epb), s>>>(u, uf, E, op);
    return int(cudaGetLastError());
}

// metric path of the kernels: 0 per-point metrics, 1 affine, 2 affine with diagonal S
inline int metric_path(const frk::Geo<FR_REAL>& g) { return g.sS_sp != 0 ? 0 : g.diag ? 2 : 1; }

template <int P, int MP, bool BND>
int visc_p(const FR_REAL* u, const FR_REAL* uf, FR_REAL* fvn, int64_t E, const frk::Ops<FR_REAL>& op,
           const frk::Phys<FR_REAL>& ph, const frk::Geo<FR_REAL>& g, frk::Launch lc, cudaStream_t s) {
    if constexpr (MP == 0) {
        auto k = frk::k_visc_face<FR_DIM, P, FR_REAL>;
        const auto smem = [](int n) { return frk::smem_visc<FR_DIM, P, FR_REAL>(n, true); };
        const size_t sm = smem(std::max(lc.epb, 1));
        static unsigned long long done = 0;
        cudaError_t e = prep(k, sm, done);
        if (lc.epb < 0) return e == cudaSuccess ? best_tile(k, frk::Grp<FR_DIM, P>::T, smem, E) : 1;
        if (e != cudaSuccess) return int(e);
        static std::atomic<int> most{0};
        const int epb = frk::fit_tile(k, frk::Grp<FR_DIM, P>::T, lc.epb, most);
        if (E == 0) return 0;
        k<<<grid_of(E, epb), frk::Grp<FR_DIM, P>::T * epb, smem(epb), s>>>(u, uf, fvn, E, op, ph, g);
        return int(cudaGetLastError());
    } else {
        // affine meshes: the pipelined kernel on a persistent grid of as many
        // blocks as fit on every SM at once, at most one per tile of elements
        // (kept per tile: all devices are alike)
        auto k = frk::k_visc_face_aff<FR_DIM, P, FR_REAL, MP, BND>;
        const auto smem = [](int n) { return frk::smem_visc<FR_DIM, P, FR_REAL>(n, false); };
        const size_t sm = smem(std::max(lc.epb, 1));
        static unsigned long long done = 0;
        cudaError_t e = prep(k, sm, done);
        if (lc.epb < 0) return e == cudaSuccess ? best_tile(k, frk::Grp<FR_DIM, P>::T, smem, E, 2) : 1;
        if (e != cudaSuccess) return int(e);
        static std::atomic<int> most{0};
        const int epb = frk::fit_tile(k, frk::Grp<FR_DIM, P>::T, lc.epb, most);
        if (E == 0) return 0;
        const int threads = frk::Grp<FR_DIM, P>::T * epb;
        static std::atomic<int> resident[33];
        int cap = resident[epb & 31].load();
        if (cap == 0) {
            cap = std::max(1, blocks_per_sm(k, threads, smem(epb))) * sm_count();
            resident[epb & 31].store(cap);
        }
        k<<<std::min(grid_of(E, epb), unsigned(cap)), threads, smem(epb), s>>>(u, uf, fvn, E, op, ph, g);
        return int(cudaGetLastError());
    }
}

template <int P, int MP, bool VISC, bool BND>
int resid_p(const FR_REAL* u, const FR_REAL* uf, const FR_REAL* fvn, int64_t E,
            const frk::Ops<FR_REAL>& op, const frk::Phys<FR_REAL>& ph, const frk::Geo<FR_REAL>& g,
            const frk::Stage<FR_REAL>& st, frk::Launch lc, cudaStream_t s) {
    auto k = frk::k_residual<FR_DIM, P, FR_REAL, MP, VISC, BND>;
    const bool curved = g.sS_sp != 0;
    const auto smem = [curved](int n) { return frk::smem_resid<FR_DIM, P, FR_REAL>(n, curved); };
    const size_t sm = smem(std::max(lc.epb, 1));
    static unsigned long long done = 0;
    cudaError_t e = prep(k, sm, done);
    if (lc.epb < 0) return e == cudaSuccess ? best_tile(k, frk::Grp<FR_DIM, P>::T, smem, E) : 1;
    if (e != cudaSuccess) return int(e);
    static std::atomic<int> most{0};
    const int epb = frk::fit_tile(k, frk::Grp<FR_DIM, P>::T, lc.epb, most);
    if (E == 0) return 0;
    k<<<grid_of(E, epb), frk::Grp<FR_DIM, P>::T * epb, smem(epb), s>>>(u, uf, fvn, E, op, ph, g, st);
    return int(cudaGetLastError());
}

}  // namespace

#define FR_DISPATCH(CALL)                 \
    switch (P) {                          \
        case 1: return CALL(1);           \
        case 2: return CALL(2);           \
        case 3: return CALL(3);           \
        case 4: return CALL(4);           \
        default: return int(cudaErrorInvalidValue); \
    }

template <>
int traces<FR_REAL, FR_DIM>(int P, const FR_REAL* u, FR_REAL* uf, int64_t E, const frk::Ops<FR_REAL>& op,
                            frk::Launch lc, void* stream) {
    cudaStream_t s = static_cast<cudaStream_t>(stream);
#define C(PP) traces_p<PP>(u, uf, E, op, lc, s)
    FR_DISPATCH(C)
#undef C
}

template <>
int visc_face<FR_REAL, FR_DIM>(int P, const FR_REAL* u, const FR_REAL* uf, FR_REAL* fvn, int64_t E,
                               const frk::Ops<FR_REAL>& op, const frk::Phys<FR_REAL>& ph,
                               const frk::Geo<FR_REAL>& g, frk::Launch lc, void* stream) {
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const int mp = metric_path(g);
    // curved meshes always take the boundary-aware kernels
#define V(PP, M) (g.bnd ? visc_p<PP, M, true>(u, uf, fvn, E, op, ph, g, lc, s) \
                        : visc_p<PP, M, false>(u, uf, fvn, E, op, ph, g, lc, s))
#define C(PP) (mp == 0 ? visc_p<PP, 0, true>(u, uf, fvn, E, op, ph, g, lc, s) : mp == 1 ? V(PP, 1) : V(PP, 2))
    FR_DISPATCH(C)
#undef C
#undef V
}

template <>
int residual<FR_REAL, FR_DIM>(int P, const FR_REAL* u, const FR_REAL* uf, const FR_REAL* fvn, int64_t E,
                              const frk::Ops<FR_REAL>& op, const frk::Phys<FR_REAL>& ph,
                              const frk::Geo<FR_REAL>& g, const frk::Stage<FR_REAL>& st, frk::Launch lc,
                              void* stream) {
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const int mp = metric_path(g);
#define B(PP, M, V) (g.bnd ? resid_p<PP, M, V, true>(u, uf, fvn, E, op, ph, g, st, lc, s) \
                           : resid_p<PP, M, V, false>(u, uf, fvn, E, op, ph, g, st, lc, s))
#define R(PP, V) (mp == 0 ? resid_p<PP, 0, V, true>(u, uf, fvn, E, op, ph, g, st, lc, s) \
                  : mp == 1 ? B(PP, 1, V) : B(PP, 2, V))
#define C(PP) (ph.viscous ? R(PP, true) : R(PP, false))
    FR_DISPATCH(C)
#undef C
#undef R
#undef B
}

template <>
int threads_per_element<FR_REAL, FR_DIM>(int P) {
    switch (P) {
        case 1: return frk::Grp<FR_DIM, 1>::T;
        case 2: return frk::Grp<FR_DIM, 2>::T;
        case 3: return frk::Grp<FR_DIM, 3>::T;
        case 4: return frk::Grp<FR_DIM, 4>::T;
        default: return 32;
    }
}

template <>
size_t smem_bytes<FR_REAL, FR_DIM>(int P, int kernel, int epb, bool curved) {
#define C(PP) (kernel == 0 ? frk::smem_traces<FR_DIM, PP, FR_REAL>(epb)          \
               : kernel == 1 ? frk::smem_visc<FR_DIM, PP, FR_REAL>(epb, curved)  \
                             : frk::smem_resid<FR_DIM, PP, FR_REAL>(epb, curved))
    switch (P) {
        case 1: return C(1);
        case 2: return C(2);
        case 3: return C(3);
        case 4: return C(4);
        default: return 0;
    }
#undef C
}

template <>
int forces<FR_REAL, FR_DIM>(int P, const FR_REAL* uf, const FR_REAL* fvn, const int32_t* wall_ef,
                            const int64_t* wall_off, int ncand, const frk::Ops<FR_REAL>& op,
                            const frk::Geo<FR_REAL>& g, FR_REAL gm1, int viscous, double* part, double* fnow,
                            double* fsum, double* fcnt, void* stream) {
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (ncand <= 0) return 0;
    const dim3 grid(frk::FORCE_BLOCKS, unsigned(ncand));
#define C(PP) [] { static unsigned long long done = 0; return side_prep(frk::k_forces<FR_DIM, PP, FR_REAL>, done); }()
    [&]() -> int { FR_DISPATCH(C) }();
#undef C
#define C(PP) (frk::k_forces<FR_DIM, PP, FR_REAL><<<grid, 256, 0, s>>>(uf, fvn, wall_ef, wall_off, op, g, gm1, \
                                                                        viscous, part),                      \
               frk::k_forces_fin<<<ncand, 32, 0, s>>>(part, frk::FORCE_BLOCKS, fnow, fsum, fcnt),          \
               int(cudaGetLastError()))
    FR_DISPATCH(C)
#undef C
}

template <>
int sample<FR_REAL, FR_DIM>(int P, const FR_REAL* u, const frk::Surf<FR_REAL>* surf, int nsurf, int most,
                            const frk::Phys<FR_REAL>& ph, void* stream) {
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const dim3 grid(unsigned((int64_t(most) * 32 + 255) / 256), unsigned(nsurf));
#define C(PP) [] { static unsigned long long done = 0; return side_prep(frk::k_sample<FR_DIM, PP, FR_REAL>, done); }()
    [&]() -> int { FR_DISPATCH(C) }();
#undef C
#define C(PP) (frk::k_sample<FR_DIM, PP, FR_REAL><<<grid, 256, 0, s>>>(u, surf, ph),                            \
               frk::k_bump<FR_REAL><<<unsigned((nsurf + 31) / 32), 32, 0, s>>>(surf, nsurf), int(cudaGetLastError()))
    FR_DISPATCH(C)
#undef C
}

template <>
int integrals<FR_REAL, FR_DIM>(int P, const FR_REAL* u, int64_t e_first, int64_t ne,
                               const frk::Ops<FR_REAL>& op, const frk::Geo<FR_REAL>& g, double* partial,
                               int nblocks, void* stream) {
    cudaStream_t s = static_cast<cudaStream_t>(stream);
#define C(PP) (frk::k_integrals<FR_DIM, PP, FR_REAL><<<nblocks, 256, 0, s>>>(u, e_first, ne, op, g, partial), \
               int(cudaGetLastError()))
    FR_DISPATCH(C)
#undef C
}

template <>
int source_stage<FR_REAL, FR_DIM>(int P, const frk::Src<FR_REAL>& src, const frk::Stage<FR_REAL>& st,
                                  const frk::Ops<FR_REAL>& op, void* stream) {
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (src.nentry <= 0) return 0;
    const unsigned blocks = unsigned((src.nentry + 3) / 4);
#define C(PP) (frk::k_source_stage<FR_DIM, PP, FR_REAL><<<blocks, 128,                                    \
                   4 * frk::Sz<FR_DIM, PP>::NV * frk::Sz<FR_DIM, PP>::NSP * sizeof(FR_REAL), s>>>(src, st, op),                   \
               int(cudaGetLastError()))
    FR_DISPATCH(C)
#undef C
}

template <>
int sponge<FR_REAL, FR_DIM>(int P, const frk::Sponge<FR_REAL>& sp, FR_REAL* a, FR_REAL* b, FR_REAL* uf_out,
                            const frk::Ops<FR_REAL>& op, void* stream) {
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (sp.n <= 0) return 0;
    const unsigned blocks = unsigned((sp.n + 3) / 4);
#define C(PP) (frk::k_sponge<FR_DIM, PP, FR_REAL><<<blocks, 128,                                             \
                   8 * frk::Smem<FR_DIM, PP>::UA * sizeof(FR_REAL), s>>>(sp, a, b, \
                                                                                              uf_out, op), \
               int(cudaGetLastError()))
    FR_DISPATCH(C)
#undef C
}

template <>
int cfl<FR_REAL, FR_DIM>(int P, const FR_REAL* u, const FR_REAL* hlen, int64_t E, const int64_t* cand_off,
                         int ncand, const frk::Phys<FR_REAL>& ph, unsigned long long* lam, float* up, unsigned* low,
                         void* stream) {
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (E == 0) return 0;
    const unsigned blocks = unsigned((E + 7) / 8);
    // elements a warp looks at in k_cfl: one, or four where bounds leave most of them
    // out and the warps still fill every SM (125,000 elements at p = 2: 62 us with 4, 72
    // with 1; with 16 60, but 798 against 750 in a uniform flow, where all of them are
    // evaluated)
    const bool many = up && E >= 32 * int64_t(sm_count());
    const unsigned warps = unsigned(many ? (E + 3) / 4 : E);
#define C(PP) ((up ? (frk::k_cfl_bound<FR_DIM, PP, FR_REAL><<<blocks, 256, 0, s>>>(u, hlen, E, cand_off, ncand, ph, up, low), 0) : 0), \
               (many ? frk::k_cfl<FR_DIM, PP, FR_REAL, true> : frk::k_cfl<FR_DIM, PP, FR_REAL, false>)                        \
                   <<<(warps + 7) / 8, 256, 0, s>>>(u, hlen, E, cand_off, ncand, ph, up, low, lam),                           \
               int(cudaGetLastError()))
    FR_DISPATCH(C)
#undef C
}

#undef FR_DISPATCH

}  // namespace frl
