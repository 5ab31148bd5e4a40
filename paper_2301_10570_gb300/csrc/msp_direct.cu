// msp_direct.cu -- msp_direct, the comparison path: Eq. 8 by all-pairs
// evaluation over the tree's sorted copy (no cutoff, no expansion).  Points in
// frames (independent networks): a target takes only the sources of its own
// network, which are contiguous in Morton order (the key's top 3 L0 bits are
// the network's cell, fsh = 3 (21 - L0) bits below).
#include "msp_direct.cuh"

namespace msp {

void direct(msp_ctx& c, float* u_dev, cudaStream_t s) {
    if (!c.tree_built) throw Error(MSP_ERR_NOT_BUILT, "msp_build_tree must run first");
    const int64_t n = c.n;
    if (n == 0) return;
    const float k2 = (float)(1.4426950408889634 / (c.cfg.sigma * c.cfg.sigma));
    const bool framed = c.frame_level > 0;
    // the sorted keys of the build are still in keys0
    const uint64_t* keys = framed ? c.keys0.get<uint64_t>() : nullptr;
    const int fsh = framed ? 3 * (kMortonBits - c.frame_level) : 0;
    const DirPacked src{c.pts.get<float4>()};
    const int32_t* perm = c.perm.get<int32_t>();
    if (n <= kDirSmallN) {
        const unsigned g = (unsigned)((n + 31) / 32);
        if (framed)
            k_dir_small<true><<<g, kDirSmallWarps * 32, 0, s>>>(n, src, k2, keys, fsh, perm, u_dev);
        else
            k_dir_small<false><<<g, kDirSmallWarps * 32, 0, s>>>(n, src, k2, keys, fsh, perm, u_dev);
        MSP_LAUNCH("dir_small");
        return;
    }
    // the lists and the tiles' boxes sit in the scan scratch of the build
    // (at least n + 8 words each): nothing is allocated, so that a captured
    // step graph stays valid
    int32_t* list = c.cnt.ensure<int32_t>((size_t)n + 8);
    const DirScratch t(c.off.ensure<int32_t>((size_t)n + 8), n);
    if (framed)
        dir_launch_tiles<true>(n, src, nullptr, src.pts, list, t, k2, keys, fsh, perm, u_dev, s);
    else
        dir_launch_tiles<false>(n, src, nullptr, src.pts, list, t, k2, keys, fsh, perm, u_dev, s);
    g_kernel_launches.fetch_add(2, std::memory_order_relaxed);
    MSP_LAUNCH("dir_tiles");
}

}  // namespace msp
