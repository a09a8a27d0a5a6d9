// Meson two-point functions for arbitrary spin matrices G, from the 12
// columns of a point-source propagator in the host layout (the correlation
// functions Sec. 3.3 leaves to the user of the propagator):
//
//   C_G(t) = - sum_xvec tr[ (G x 1) S(x) (Gbar x 1) g5 S(x)^dag g5 ],
//   Gbar = g_t G^dag g_t,  x = (xvec, src_t + t mod T).
//
// Writing S_{ad} for the 3x3 colour block of sink spin a and source spin d,
// the trace is a sum over spin indices of coefficients times colour inner
// products:
//   C_G = sum_{a,b,c,d} k_abcd <S_ad, S_bc>,  k_abcd = - G_ab Gbar_cd g5_d g5_a,
//   <A, B> = sum_ij conj(A_ij) B_ij.
// The colour inner products enter linearly, so they are summed over the sites
// of a slice first and meet the k afterwards: a slice needs each distinct
// <S_p, S_q> (p <= q, the other order is the conjugate) once, whatever the
// number of matrices G.  That is at most 136 sums; the sixteen Clifford
// elements together need 40, sixteen of them the real norms <S_p, S_p>.
#include <algorithm>
#include <cstring>
#include <vector>

#include "lqcd_impl.h"

namespace lqcd {

struct MesonTerm {
    int pair, conj;  // index of the pair; 1: its conjugate
    double re, im;   // k_abcd
};

// chiral basis (spin index 0-3): g_t = [[0, -1], [-1, 0]] in 2x2 blocks, g5 = diag(1, 1, -1, -1)
static double gt_host(int a, int b) { return (a == b + 2 || b == a + 2) ? -1.0 : 0.0; }
static double g5_host(int a) { return a < 2 ? 1.0 : -1.0; }

// A tile is 32 consecutive sites of a slice, all 144 complex numbers of each,
// staged in shared memory by cp.async while the tile before it is worked on.
// A warp's lanes are the sites; its pairs run one after the other.  The sites
// of a column lie 208 bytes apart (13 16-byte words for 12), so the lanes'
// 16-byte reads meet no bank twice.
constexpr int kTileSites32 = 32, kMesonWarps = 8, kSiteWords = 13;
constexpr int kTileWords = 12 * kTileSites32 * kSiteWords;  // double2
constexpr int kMesonSmem = 2 * kTileWords * 16;

__device__ __forceinline__ void meson_stage(double2 *tile, const double2 *prop, long V, long x0, int nsites)
{
    for (int w = threadIdx.x; w < 12 * kTileSites32 * 12; w += kMesonWarps * 32) {
        const int j = w / (kTileSites32 * 12), r = w - j * (kTileSites32 * 12);
        const int site = r / 12, i = r - site * 12;
        const bool in = site < nsites;  // sites past the end of the slice are filled with zeros
        const double2 *src = prop + ((long)j * V + x0 + (in ? site : 0)) * 12 + i;
        const unsigned dst =
            unsigned(__cvta_generic_to_shared(tile + (j * kTileSites32 + site) * kSiteWords + i));
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(dst), "l"(src), "r"(in ? 16 : 0)
                     : "memory");
    }
    asm volatile("cp.async.commit_group;\n" ::: "memory");
}

// Sums of the pairs over the tiles [c per, (c + 1) per) of slice t (block (c,
// t)); partial[(t npairs + k) nchunk + c].  Bound by the FP64 pipe: 36
// instructions per site for a pair and 18 for a norm, 1152 for the sixteen
// Clifford elements against 2304 bytes read once: 4.66 ms on 32^3 x 64.  One
// thread per site that walked every matrix's terms took 9200 instructions and
// read the columns twice over: 62.5 ms.
template <int KP>
__global__ void __launch_bounds__(kMesonWarps * 32) meson_kernel(long V, long v3, int per, int npairs,
                                                                 const double2 *prop, const int2 *pairs,
                                                                 double2 *partial)
{
    extern __shared__ double2 tiles[];
    const int t = blockIdx.y, c = blockIdx.x, nchunk = gridDim.x;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int ntile = int((v3 + kTileSites32 - 1) / kTileSites32);
    const int k0 = c * per, k1 = min(ntile, k0 + per);
    double ar[KP], ai[KP];
    int op[KP], oq[KP];  // the pair's blocks as offsets into the lane's site
#pragma unroll
    for (int k = 0; k < KP; ++k) {
        ar[k] = ai[k] = 0.0;
        const int2 pq = pairs[min(warp + k * kMesonWarps, npairs - 1)];
        op[k] = ((pq.x & 3) * 3 * kTileSites32 + lane) * kSiteWords + 3 * (pq.x >> 2);
        oq[k] = ((pq.y & 3) * 3 * kTileSites32 + lane) * kSiteWords + 3 * (pq.y >> 2);
    }
    const long x0 = (long)t * v3;
    auto stage = [&](int k) {
        meson_stage(tiles + (k & 1) * kTileWords, prop, V, x0 + (long)k * kTileSites32,
                    int(min((long)kTileSites32, v3 - (long)k * kTileSites32)));
    };
    if (k0 < k1) stage(k0);
    for (int n = k0; n < k1; ++n) {
        if (n + 1 < k1) {
            stage(n + 1);
            asm volatile("cp.async.wait_group 1;\n" ::: "memory");
        } else {
            asm volatile("cp.async.wait_group 0;\n" ::: "memory");
        }
        __syncthreads();
        const double2 *s = tiles + (n & 1) * kTileWords;
#pragma unroll
        for (int k = 0; k < KP; ++k) {
            if (warp + k * kMesonWarps >= npairs) break;
            // S[3a+u][3d+v] = column 3d+v, component 3a+u
            if (op[k] == oq[k]) {
#pragma unroll
                for (int v = 0; v < 3; ++v)
#pragma unroll
                    for (int u = 0; u < 3; ++u) {
                        const double2 A = s[op[k] + v * kTileSites32 * kSiteWords + u];
                        ar[k] = fma(A.x, A.x, ar[k]);
                        ar[k] = fma(A.y, A.y, ar[k]);
                    }
            } else {
#pragma unroll
                for (int v = 0; v < 3; ++v)
#pragma unroll
                    for (int u = 0; u < 3; ++u) {
                        const double2 A = s[op[k] + v * kTileSites32 * kSiteWords + u];
                        const double2 B = s[oq[k] + v * kTileSites32 * kSiteWords + u];
                        ar[k] = fma(A.x, B.x, ar[k]);
                        ai[k] = fma(A.x, B.y, ai[k]);
                        ar[k] = fma(A.y, B.y, ar[k]);
                        ai[k] = fma(-A.y, B.x, ai[k]);
                    }
            }
        }
        __syncthreads();  // the tile's buffer is filled again in the next round
    }
#pragma unroll
    for (int k = 0; k < KP; ++k) {
        const int pair = warp + k * kMesonWarps;
        if (pair >= npairs) break;
        const double re = warp_sum(ar[k]), im = warp_sum(ai[k]);
        if (lane == 0) partial[((long)t * npairs + pair) * nchunk + c] = make_double2(re, im);
    }
}

// corr[g T + (t - src_t) mod T] = sum_terms k <S_p, S_q>; one block per slice:
// the chunks of each pair in a fixed order, then the terms of each matrix
__global__ void __launch_bounds__(256) meson_finish_kernel(int T, int ng, int npairs, int nchunk, int src_t,
                                                           const int2 *pairs, const MesonTerm *terms, const int *off,
                                                           const double2 *partial, double2 *corr)
{
    __shared__ double2 sum[136];
    const int t = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int k = warp; k < npairs; k += 8) {
        double sr = 0.0, si = 0.0;
        for (int n = lane; n < nchunk; n += 32) {
            const double2 v = partial[((long)t * npairs + k) * nchunk + n];
            sr += v.x;
            si += v.y;
        }
        sr = warp_sum(sr);
        si = warp_sum(si);
        // a norm is real (0 x its value keeps infinities and NaN out of the imaginary part's zero)
        if (pairs[k].x == pairs[k].y) si = 0.0 * sr;
        if (lane == 0) sum[k] = make_double2(sr, si);
    }
    __syncthreads();
    for (int g = threadIdx.x; g < ng; g += blockDim.x) {
        double ar = 0.0, ai = 0.0;
        for (int k = off[g]; k < off[g + 1]; ++k) {
            const MesonTerm m = terms[k];
            const double sr = sum[m.pair].x, si = m.conj ? -sum[m.pair].y : sum[m.pair].y;
            ar = fma(m.re, sr, fma(-m.im, si, ar));
            ai = fma(m.re, si, fma(m.im, sr, ai));
        }
        corr[(long)g * T + ((t - src_t) % T + T) % T] = make_double2(ar, ai);
    }
}

template <int KP>
static void meson_go(dim3 grid, long V, long v3, int per, int npairs, const double2 *prop, const int2 *pairs,
                     double2 *partial, cudaStream_t st)
{
    LQCD_CUDA(cudaFuncSetAttribute(meson_kernel<KP>, cudaFuncAttributeMaxDynamicSharedMemorySize, kMesonSmem));
    meson_kernel<KP><<<grid, kMesonWarps * 32, kMesonSmem, st>>>(V, v3, per, npairs, prop, pairs, partial);
    LQCD_CHECK_LAUNCH();
}

void meson_contract(lqcd_lattice_s *lat, const double *prop_dev, int src_t, const double *gammas, int ng,
                    double *corr_dev, cudaStream_t st)
{
    // host: term lists, and the pairs they need: index[p][q] for p <= q
    std::vector<MesonTerm> terms;
    std::vector<int2> pairs;
    int index[16][16];
    std::fill(&index[0][0], &index[0][0] + 256, -1);
    std::vector<int> off(1, 0);
    for (int g = 0; g < ng; ++g) {
        double G[4][4][2], Gb[4][4][2];
        for (int a = 0; a < 4; ++a)
            for (int b = 0; b < 4; ++b) {
                G[a][b][0] = gammas[2 * (16 * g + 4 * a + b)];
                G[a][b][1] = gammas[2 * (16 * g + 4 * a + b) + 1];
            }
        // Gbar = g_t G^dag g_t: (g_t)_{aa'} conj(G_{b'a'}) (g_t)_{b'b}
        for (int a = 0; a < 4; ++a)
            for (int b = 0; b < 4; ++b) {
                double re = 0.0, im = 0.0;
                for (int a2 = 0; a2 < 4; ++a2)
                    for (int b2 = 0; b2 < 4; ++b2) {
                        const double w = gt_host(a, a2) * gt_host(b2, b);
                        re += w * G[b2][a2][0];
                        im -= w * G[b2][a2][1];
                    }
                Gb[a][b][0] = re;
                Gb[a][b][1] = im;
            }
        for (int a = 0; a < 4; ++a)
            for (int b = 0; b < 4; ++b)
                for (int c = 0; c < 4; ++c)
                    for (int d = 0; d < 4; ++d) {
                        // k = - G_ab Gbar_cd g5_d g5_a
                        const double s = -g5_host(d) * g5_host(a);
                        const double re = s * (G[a][b][0] * Gb[c][d][0] - G[a][b][1] * Gb[c][d][1]);
                        const double im = s * (G[a][b][0] * Gb[c][d][1] + G[a][b][1] * Gb[c][d][0]);
                        if (re == 0.0 && im == 0.0) continue;
                        const int p = 4 * a + d, q = 4 * b + c;
                        int &k = index[std::min(p, q)][std::max(p, q)];
                        if (k < 0) {
                            k = int(pairs.size());
                            pairs.push_back(make_int2(std::min(p, q), std::max(p, q)));
                        }
                        terms.push_back(MesonTerm{k, p > q, re, im});
                    }
        off.push_back(int(terms.size()));
    }
    if (pairs.empty()) pairs.push_back(make_int2(0, 0));  // every matrix zero: the sums are not used
    // the norms (half the work) last, so that the warps' shares differ by one norm at most
    std::vector<int> place(pairs.size());
    std::vector<int2> sorted;
    for (int norm = 0; norm < 2; ++norm)
        for (size_t k = 0; k < pairs.size(); ++k)
            if ((pairs[k].x == pairs[k].y) == (norm == 1)) {
                place[k] = int(sorted.size());
                sorted.push_back(pairs[k]);
            }
    for (MesonTerm &m : terms) m.pair = place[m.pair];
    const int npairs = int(sorted.size());
    const int T = lat->dims[3];
    const long v3 = lat->V / T;
    const int ntile = int((v3 + kTileSites32 - 1) / kTileSites32);
    // chunks per slice: one block per SM at a time (its tiles fill the shared
    // memory), so the rounds of blocks times the tiles of a block are the time
    const int sms = 152;
    int nchunk = 1;
    long best = 0;
    for (int n = 1; n <= std::min(ntile, 64); ++n) {
        const long cost = ((long)T * n + sms - 1) / sms * ((ntile + n - 1) / n);
        if (n == 1 || cost < best) {
            best = cost;
            nchunk = n;
        }
    }
    const int per = (ntile + nchunk - 1) / nchunk;
    auto up16 = [](size_t n) { return (n + 15) / 16 * 16; };
    const size_t tbytes = up16(sizeof(MesonTerm) * terms.size()), pairbytes = up16(sizeof(int2) * npairs);
    const size_t obytes = up16(sizeof(int) * off.size());
    // one upload for the three tables (the lattice's buffers: calls on a lattice are serialised and end synchronised)
    std::vector<char> host(tbytes + pairbytes + obytes);
    if (!terms.empty()) std::memcpy(host.data(), terms.data(), sizeof(MesonTerm) * terms.size());
    std::memcpy(host.data() + tbytes, sorted.data(), sizeof(int2) * npairs);
    std::memcpy(host.data() + tbytes + pairbytes, off.data(), sizeof(int) * off.size());
    lat->tables.ensure(host.size());
    lat->red_partial.ensure(sizeof(double2) * (size_t)T * npairs * nchunk);
    char *b = lat->tables.as<char>();
    const MesonTerm *dterms = reinterpret_cast<const MesonTerm *>(b);
    const int2 *dpairs = reinterpret_cast<const int2 *>(b + tbytes);
    const int *doff = reinterpret_cast<const int *>(b + tbytes + pairbytes);
    double2 *dpart = lat->red_partial.as<double2>();
    const double2 *prop = reinterpret_cast<const double2 *>(prop_dev);
    LQCD_CUDA(cudaMemcpyAsync(b, host.data(), host.size(), cudaMemcpyHostToDevice, st));
    {
        // algorithmic bytes: the 12 columns once
        ProfScope prof("meson_contract", double(lat->V) * 12 * 192.0, st);
        const dim3 grid{unsigned(nchunk), unsigned(T)};
        const int kp = (npairs + kMesonWarps - 1) / kMesonWarps;
        if (kp <= 2) meson_go<2>(grid, lat->V, v3, per, npairs, prop, dpairs, dpart, st);
        else if (kp <= 5) meson_go<5>(grid, lat->V, v3, per, npairs, prop, dpairs, dpart, st);
        else if (kp <= 9) meson_go<9>(grid, lat->V, v3, per, npairs, prop, dpairs, dpart, st);
        else meson_go<17>(grid, lat->V, v3, per, npairs, prop, dpairs, dpart, st);
    }
    meson_finish_kernel<<<unsigned(T), 256, 0, st>>>(T, ng, npairs, nchunk, src_t, dpairs, dterms, doff, dpart,
                                                     reinterpret_cast<double2 *>(corr_dev));
    LQCD_CHECK_LAUNCH();
}

}  // namespace lqcd
