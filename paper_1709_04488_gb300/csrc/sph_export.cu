// Exact FP64 neighbour lists (CSR, ids ascending) for one problem: a tree
// walk per leaf retrieves the candidates (Sec. 4.2); membership is
// r^2 = dx*dx + dy*dy + dz*dz < (R_K h_i)^2 (gather list) or < (R_K
// max(h_i,h_j))^2 (force list) on absolute FP64 positions with the periodic
// minimum image, formed without fused multiply-add, R_K the kernel's support
// in units of h (2 for M4, 3 for M6).
#include "sph_pairs.cuh"

namespace sph {

namespace {

constexpr int kExportCap = 1024;  // neighbours one particle may have in the export

template <bool F64>
__global__ void k_set_sorted_h(BatchView b, const double *h_in)
{
    chain_entry();
    long long s = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= b.ntot) return;
    int p = (int)(b.keys[0][s] >> kMortonTotal);
    long long i = (long long)b.perm[s] - b.prob[p].base;
    const double h = h_in ? h_in[i] : b.prob[p].h[i];
    b.sh[s] = h;
    b.hf[s] = __double2float_ru(F64 ? h * frame_of(b.prob[p].ph, b.dyn[p]).unit : h);
}

// the membership test's own arithmetic (i, j: sorted indices)
__device__ __forceinline__ bool export_member(const BatchView &b, const PhysParams &ph, long long i, long long j, int kind)
{
    const double dx = min_image(__dsub_rn(b.sx[i], b.sx[j]), ph.box_len[0], ph.periodic);
    const double dy = min_image(__dsub_rn(b.sy[i], b.sy[j]), ph.box_len[1], ph.periodic);
    const double dz = min_image(__dsub_rn(b.sz[i], b.sz[j]), ph.box_len[2], ph.periodic);
    const double r2 = __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
    const double hh = kind == 1 ? fmax(b.sh[i], b.sh[j]) : b.sh[i];
    const double Rk = __dmul_rn(ph.kr, hh);  // R_K h, rounded as the oracle's
    return r2 < __dmul_rn(Rk, Rk);
}

// One warp per leaf, as in the pair kernels: the leaf's candidates are staged
// in FP32 in its frame, and each lane tests them for its particle.  A pair
// within the rounding of the staged coordinates of the boundary (stage_err;
// a few in 1e4) is decided in FP64 (export_member); the others by FP32.
// (One walk per particle with every candidate tested in FP64, the first form
// of this kernel, was bound by the FP64 pipe, 1/64 of the FP32 rate: 3.04 ms
// per pass for 103823 particles; this form: 94-114 us.)  The pairs found wait in
// a short list per lane, so that the lanes write them together.
// FILL false: counts into cnt[i]; true: ids, in any order, at offsets[i].
// F64: an FP64 problem, whose FP32 copies are in the walk's frame.  SCALED: a
// mixed one whose raw lengths have squares that leave the range of FP32; they
// are brought to the size of its coordinates as they are read.
// (Raw lengths up to 2^60 have finite squares, and from 2^-20 on the squares
// of their spacings are far above kTinySq.  Scaled throughout, the count
// and fill of 103823 particles took 3 % longer, as one kernel with both
// forms 22 %.)
struct ExportCfg {
    static constexpr int CH = 64, LC = 32, SB = 16, WPB = 4;
    static constexpr size_t scratch = (sizeof(StageScratch<float>) + 31) & ~(size_t)31;
    static constexpr size_t per_warp = CH * (sizeof(float4) + sizeof(int)) + (size_t)LC * 32 * sizeof(int) + scratch;
};
template <bool FILL, bool F64, bool SCALED>
__global__ void __launch_bounds__(ExportCfg::WPB * 32, 7) k_export(BatchView b, int kind, unsigned *cnt,
                                                                const long long *offsets, int *idx, long long cap)
{
    chain_entry();
    using C = ExportCfg;
    __shared__ __align__(32) unsigned char smem[C::WPB * C::per_warp];
    __shared__ int wrote[C::WPB][32];
    if (!F64 && !SCALED && !lists_in_range(coord_bound<false>(b.prob[0].ph, b.dyn[0]))) {
        if (!FILL)  // (empty lists; the caller comes back for the scaled form)
            for (long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x; k < b.ntot; k += (long long)gridDim.x * blockDim.x)
                cnt[k] = 0u;
        return;
    }
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    unsigned char *mine = smem + wib * C::per_warp;
    float4 *cand = reinterpret_cast<float4 *>(mine);  // staged (x, y, z, R_K h rounded up)
    StageScratch<float> &sc = *reinterpret_cast<StageScratch<float> *>(cand + C::CH);
    int *code = reinterpret_cast<int *>(mine + C::CH * sizeof(float4) + C::scratch);  // sorted index per candidate
    int *lst = code + C::CH;  // 2 x sorted index + (decided in FP64)
    const ProbStatic &ps = b.prob[0];
    const ProbDyn &d = b.dyn[0];
    const PhysParams &ph = ps.ph;
    const int lpp = ps.lpp, pp = lane / lpp, sub = lane % lpp;
    const float u = SCALED ? (float)fmin(frame_unit((double)coord_bound<F64>(ph, d)), 0x1p126) : 1.f;
    const double unit = F64 ? frame_of(ph, d).unit : (double)u;
    const float cmax = coord_bound<F64>(ph, d) * u;
    auto reach = [&](float h) { return __fmul_ru(ph.kr_f, SCALED ? __fmul_ru(h, u) : h); };
    auto staged = [&](long long k) {
        float4 q = b.pmf[k];
        if (SCALED) q.x *= u, q.y *= u, q.z *= u;
        return q;
    };
    const int nleaf = b.counters[0];
    const int w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, nw = (gridDim.x * blockDim.x) >> 5;
    for (int leaf = w; leaf < nleaf; leaf += nw) {
        const NodeBox boxA = b.nodes[0][leaf];
        const int st = b.leaf_start[leaf], nA = b.leaf_start[leaf + 1] - st;
        const bool active = pp < nA;
        const int s = st + (active ? pp : 0);
        float4 pi = staged(s);
        pi.w = reach(b.hf[s]);
        float4 flo, fhi;
        frame_box<float4, float>(pi, active, flo, fhi);
        const float pmax = box_abs(flo, fhi);
        float emax = 0.f;  // this lane's largest stage_err since the buffer was last emptied
        const float R = reach(boxA.plo.w) * 1.0001f;
        // the largest reach of a pair of this leaf, for the image handling
        float Rall = R, extmax;
        if (kind == 1) problem_top_max(b, d, Rall, extmax), Rall = reach(Rall) * 1.0001f;
        if (ph.periodic) load_box(sc, ph, flo, fhi, u);
        const bool wrap2 = ph.periodic && half_width(flo, fhi) + Rall >= half_box(ph) * u;
        set_query(sc.qb, boxA.plo, boxA.phi, R, ph, cmax);
        int nbuf = 0, n = 0;
        const long long i = (long long)b.perm[s] - ps.base;
        const long long at = FILL ? offsets[i] : 0;
        int total = 0;
        if (FILL) wrote[wib][lane] = 0;
        __syncwarp();
        auto drain = [&]() {
            for (int e = 0; e < n; ++e) {
                const int c = lst[e * 32 + lane], j = c >> 1;
                if ((c & 1) && !export_member(b, ph, s, j, kind)) continue;
                ++total;
                if (FILL) {
                    const long long k = at + atomicAdd(&wrote[wib][pp], 1);
                    if (k < cap) idx[k] = (int)((long long)b.perm[j] - ps.base);
                }
            }
            n = 0;
        };
        auto test = [&]() {
            __syncwarp();  // staged candidates visible to every lane
            const float err = warp_max(emax);
            emax = 0.f;
            for (int k0 = 0; k0 < nbuf; k0 += C::SB) {
                if (__any_sync(FULL, n > C::LC - C::SB)) drain();
                const int ke = min(k0 + C::SB, nbuf);
                for (int k = k0 + sub; k < ke; k += lpp) {
                    const float4 c = cand[k];
                    float rx = pi.x - c.x, ry = pi.y - c.y, rz = pi.z - c.z;
                    if (wrap2) wrap3s<float>(sc, rx, ry, rz);
                    const float r2 = rx * rx + ry * ry + rz * rz;
                    const float Rk = kind == 1 ? fmaxf(pi.w, c.w) : pi.w;
                    const float gap = r2 - Rk * Rk, tol = Rk * (8.f * err + 1e-5f * Rk) + err * err + kTinySq;
                    const int j = code[k];
                    if (active && gap < tol && !(kind == 1 && j == s))
                        lst[n++ * 32 + lane] = 2 * j + (gap > -tol);
                }
            }
            __syncwarp();
            nbuf = 0;
        };
        auto node = [&](const NodeBox &nb) {
            return up_within(sc.qb, nb, u) || (kind == 1 && up_overlap(sc.qb, nb, u));
        };
        int j = 0;
        float Rj = 0.f;
        Walk wk;
        wk.start(d);
        for (;;) {
            const int nd = wk.next(b, d, node);
            if (nd < 0) break;
            const int first = d.node_off[0] + nd * kBranch;
            const bool in = (leaf_lanes(d.node_cnt[0], nd) >> lane) & 1u;
            const unsigned mask = __ballot_sync(FULL, node(b.nodes[0][first + (in ? lane : 0)]) && in);
            if (mask)
                stage_group<float, C::CH, F64 || SCALED>(
                b, leaf, mask, first, ph, unit, nbuf, sc, [](bool, int, int, int, const float4 &) {},
                [&](int jj) {
                    float4 q = staged(jj);
                    q.w = __int_as_float(jj);
                    return q;
                },
                [&](float4 &q, int o) {
                    j = __float_as_int(q.w);
                    Rj = reach(b.hf[j]);
                    const float aq = abs3(q);
                    if (ph.periodic) wrap_near<float>(sc, q, sc.C[0], sc.C[1], sc.C[2]);
                    // (scaled: the raw copies may be below the smallest normal number)
                    const float e = stage_err(abs3(sc.leaf[o]), aq, abs3(q), pmax) + (SCALED ? 1e-44f * u : 0.f);
                    const float Rt = (kind == 1 ? fmaxf(R, Rj) : R) * 1.0001f + 2.f * e;
                    if (!(box_dist2<float>(q, flo, fhi) < Rt * Rt + kTinySq)) return false;
                    emax = fmaxf(emax, e);
                    return true;
                },
                [&](int slot, const float4 &q, int, int) {
                    cand[slot] = make_float4(q.x, q.y, q.z, Rj);
                    code[slot] = j;
                },
                test);
        }
        test();
        drain();
        if (!FILL) {
            for (int x = 1; x < lpp; x <<= 1) total += __shfl_xor_sync(FULL, total, x);
            if (active && sub == 0) cnt[i] = (unsigned)total;
        }
        __syncwarp();
    }
}
// Sorts each particle's ids (one warp per particle; ids are distinct, so an
// id's place is the number of smaller ones).  A particle whose list crosses
// cap is left to k_export_cut.
__global__ void __launch_bounds__(128) k_export_sort(BatchView b, const long long *offsets, int *idx, long long cap)
{
    chain_entry();
    __shared__ int buf[4][kExportCap];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const int w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, nw = (gridDim.x * blockDim.x) >> 5;
    for (long long i = w; i < b.ntot; i += nw) {
        const long long o = offsets[i], end = offsets[i + 1];
        const int n = (int)(end - o);
        if (n > kExportCap) {
            if (lane == 0) atomicOr(&b.prob[0].diag->status, ST_OVERFLOW);
            continue;
        }
        if (end > cap) continue;
        for (int e = lane; e < n; e += 32) buf[wib][e] = idx[o + e];
        __syncwarp();
        for (int e = lane; e < n; e += 32) {
            const int v = buf[wib][e];
            int r = 0;
#pragma unroll 4
            for (int f = 0; f < n; ++f) r += buf[wib][f] < v;
            idx[o + r] = v;
        }
        __syncwarp();
    }
}

// The particle whose list crosses cap, if there is one (one block): its ids
// are gathered again from all particles and those below cap written in order.
// (As the call's last kernel it also has a force pass that follows walk the
// tree: the leaf pass cleared the mark that the groups recorded by the last
// density walk do not cover its h.)
__global__ void __launch_bounds__(1024) k_export_cut(BatchView b, int kind, const long long *offsets, int *idx, long long cap)
{
    chain_entry();
    __shared__ int buf[kExportCap];
    __shared__ int s_pos, s_n;
    if (threadIdx.x == 0) {
        b.dyn[0].lists_stale = 1;
        b.scratch64[1] = lists_in_range(coord_bound<false>(b.prob[0].ph, b.dyn[0]));
    }
    if (offsets[b.ntot] <= cap) return;
    const ProbStatic &ps = b.prob[0];
    long long lo = 0, hi = b.ntot - 1;  // the last particle that starts below cap
    while (lo < hi) {
        const long long mid = (lo + hi + 1) >> 1;
        if (offsets[mid] < cap) lo = mid;
        else hi = mid - 1;
    }
    const long long i = lo, o = offsets[i];
    const long long n = offsets[i + 1] - o;
    if (!(o < cap && cap < o + n) || n > kExportCap) return;
    if (threadIdx.x == 0) s_n = 0;
    for (long long t = threadIdx.x; t < b.ntot; t += blockDim.x)
        if ((long long)b.perm[t] - ps.base == i) s_pos = (int)t;
    __syncthreads();
    const long long s = s_pos;
    for (long long t = threadIdx.x; t < b.ntot; t += blockDim.x)
        if (!(kind == 1 && t == s) && export_member(b, ps.ph, s, t, kind)) {
            const int k = atomicAdd(&s_n, 1);
            if (k < kExportCap) buf[k] = (int)((long long)b.perm[t] - ps.base);
        }
    __syncthreads();
    for (int e = threadIdx.x; e < n; e += blockDim.x) {
        const int v = buf[e];
        int r = 0;
        for (int f = 0; f < n; ++f) r += buf[f] < v;
        if (o + r < cap) idx[o + r] = v;
    }
}

// Exclusive scan of n counts into int64 offsets: the sum of each block's
// share, then each block's scan of its share from the sums before it.
constexpr int kScanThreads = 1024, kScanBlocks = 1024;
__device__ __forceinline__ long long scan_share(long long n)
{
    const long long per = (n + kScanBlocks - 1) / kScanBlocks;
    return (per + kScanThreads - 1) / kScanThreads * kScanThreads;
}
__device__ __forceinline__ long long block_sum(long long v, long long *red)
{
    v = warp_sum(v);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    long long t = 0;
    for (int k = 0; k < kScanThreads / 32; ++k) t += red[k];
    return t;
}
__global__ void __launch_bounds__(kScanThreads) k_count_sums(const unsigned *cnt, long long n, long long *part)
{
    chain_entry();
    __shared__ long long red[kScanThreads / 32];
    const long long per = scan_share(n), lo = blockIdx.x * per, hi = lo + per < n ? lo + per : n;
    long long s = 0;
    for (long long k = lo + threadIdx.x; k < hi; k += kScanThreads) s += cnt[k];
    s = block_sum(s, red);
    if (threadIdx.x == 0) part[blockIdx.x] = s;
}
__global__ void __launch_bounds__(kScanThreads) k_offsets(const unsigned *cnt, long long n, const long long *part,
                                                          long long *offsets, long long *total)
{
    chain_entry();
    __shared__ long long red[kScanThreads / 32];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const long long per = scan_share(n), lo = blockIdx.x * per, hi = lo + per < n ? lo + per : n;
    long long run = block_sum(threadIdx.x < blockIdx.x ? part[threadIdx.x] : 0, red);
    for (long long k0 = lo; k0 < hi; k0 += kScanThreads) {
        const long long k = k0 + threadIdx.x;
        const int c = k < hi ? (int)cnt[k] : 0, incl = warp_incl_scan<int>(c);
        __syncthreads();
        if (lane == 31) red[wib] = incl;
        __syncthreads();
        long long before = run, all = 0;
        for (int v = 0; v < kScanThreads / 32; ++v) {
            if (v < wib) before += red[v];
            all += red[v];
        }
        if (k < hi) offsets[k] = before + incl - c;
        run += all;
    }
    if (hi == n && lo < n && threadIdx.x == 0) {
        offsets[n] = run;
        *total = run;
    }
}

}  // namespace

cudaError_t launch_set_sorted_h(const BatchView &b, int precision, const double *h_in, cudaStream_t st)
{
    if (b.ntot == 0) return cudaSuccess;
    const auto kern = precision == SPH_PREC_FP64 ? k_set_sorted_h<true> : k_set_sorted_h<false>;
    launch_chain(SPH_DEP(b), kern, (unsigned)((b.ntot + 255) / 256), 256, 0, st, b, h_in);
    return cudaGetLastError();
}

// The number of entries goes to scratch64[0]; scratch64[1]: 0 if the scaled form
// has to be launched (mixed precision; an isolated problem's coordinates are
// known on the device only).
cudaError_t launch_neighbour_export(const BatchView &b, int precision, bool scaled, int kind, long long *offsets, int *idx,
                                    long long cap, cudaStream_t st)
{
    if (b.ntot == 0) {
        cudaMemsetAsync(offsets, 0, sizeof(long long), st);
        cudaMemsetAsync(b.scratch64, 0, sizeof(long long), st);
        return cudaGetLastError();
    }
    // the sort's second buffers (the leaf of each particle, b.flag, serves the
    // slow density path of the steps that keep these leaves)
    unsigned *cnt = b.vals[0];
    long long *part = (long long *)b.keys[1];
    const int sms = dev_info().sm_count, grid = sms * 8;
    const long long n = b.ntot, share = (n + kScanBlocks - 1) / kScanBlocks;
    const int nb = (int)((n + (share + kScanThreads - 1) / kScanThreads * kScanThreads - 1) /
                         ((share + kScanThreads - 1) / kScanThreads * kScanThreads));
    const bool f64 = precision == SPH_PREC_FP64;
    auto launch = [&](auto kern) {
        launch_chain(SPH_DEP(b), kern, grid, ExportCfg::WPB * 32, 0, st, b, kind, cnt, (const long long *)offsets, idx, cap);
    };
    launch(f64 ? k_export<false, true, false> : scaled ? k_export<false, false, true> : k_export<false, false, false>);
    launch_chain(SPH_DEP(b), k_count_sums, nb, kScanThreads, 0, st, cnt, n, part);
    launch_chain(SPH_DEP(b), k_offsets, nb, kScanThreads, 0, st, cnt, n, part, offsets, b.scratch64);
    launch(f64 ? k_export<true, true, false> : scaled ? k_export<true, false, true> : k_export<true, false, false>);
    launch_chain(SPH_DEP(b), k_export_sort, grid, 128, 0, st, b, offsets, idx, cap);
    launch_chain(SPH_DEP(b), k_export_cut, 1, 1024, 0, st, b, kind, offsets, idx, cap);
    return cudaGetLastError();
}

}  // namespace sph
