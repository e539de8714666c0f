// dm_potc.cu -- the power-of-d-choices experiment behind DualMap's choice of
// two candidates (App. A.8, "Optimal Candidate Set Size"): m balls into n
// bins, each ball to the least loaded of d uniformly random bins (ties to
// the earlier choice), the maximum bin load of each trial.
//
// Ball t's choice k in trial s uses counter c = (s * m + t) * d + k: the
// (c+1)-th output of SplitMix64 (Steele, Lea & Flood 2014) seeded with
// `seed`, scaled to a bin as floor(x * n / 2^64).
//
// A trial is one dependent chain (every ball reads loads that the balls
// before it wrote), but its choices are not part of the chain, and they are
// most of the arithmetic (about 22 integer instructions each).  So a CTA has
// one warp that places balls, a trial per lane, and eight warps that
// generate the choices of the next tile of balls into shared memory, as the
// byte offsets of the bins' loads.  The placing warp takes four balls at a
// time: all their loads are read together, and each ball's are corrected by
// the balls of the group before it, so one shared-memory round trip serves
// four balls.  A lane's loads are a column (bin b of lane j at word 32 b +
// j): distinct banks whatever the bins.
//
// Bound: integer issue of the generating warps.  10,000 trials of 32,000
// balls over 32 bins, d = 2, on GB300: 6.01 ms with a thread per trial doing
// both, 1.34 ms so.
#include "dm_internal.cuh"

namespace dm {

constexpr int kPotcGen = 256;           // generating threads
constexpr uint32_t kPotcRows = 128;     // rows of a tile: two choices per row and lane

// SplitMix64's output function of state z (after its increment), scaled to
// [0, n): the high word of the product decides unless the low words could
// carry into it (n / 2^32 of all cases).
__device__ __forceinline__ uint32_t potc_bin(uint64_t z, uint32_t n) {
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    const uint32_t zh = (uint32_t)(z >> 32), xh = zh ^ (zh >> 31);
    const uint64_t p = uint64_t(xh) * n;
    if ((uint32_t)p >= 0u - n) return (uint32_t)__umul64hi(z ^ (z >> 31), n);
    return (uint32_t)(p >> 32);
}

// kD > 0: d = kD choices, four balls at a time; 0: any d.  T <= 32 trials
// per CTA, tile balls per tile (a multiple of 4, tile * d <= 2 kPotcRows).
template <uint32_t kD>
__global__ void __launch_bounds__(32 + kPotcGen) k_potc(uint32_t n, uint64_t m, uint32_t d, uint32_t trials,
                                                        uint64_t seed, uint32_t *max_load, uint32_t T,
                                                        uint32_t tile) {
    extern __shared__ uint32_t s_load[];   // n x 32 loads
    __shared__ uint32_t s_off[2][kPotcRows][32];
    const uint32_t tid = threadIdx.x, s0 = blockIdx.x * T, here = min(T, trials - s0);   // trials of this CTA
    for (uint32_t i = tid; i < n * 32; i += blockDim.x) s_load[i] = 0;
    const uint64_t tiles = (m + tile - 1) / tile;
    constexpr uint64_t kPhi = 0x9E3779B97F4A7C15ull;
    // generating thread: trial j of the CTA, rows g, g + G, ...
    const uint32_t pt = tid - 32, j = pt % T, g = pt / T, G = kPotcGen / T;
    auto generate = [&](uint64_t i) {
        if (g >= G || j >= here) return;
        const uint32_t rows = ((uint32_t)min((uint64_t)tile, m - i * tile) * d + 1) / 2;   // of its balls
        // state after the increment of choice 0 of row g
        uint64_t z = seed + ((uint64_t(s0 + j) * m + i * tile) * d + 2 * g + 1) * kPhi;
        const uint64_t step = kPhi * (2 * G);
        uint32_t(*const out)[32] = s_off[i & 1];
        for (uint32_t r = g; r < rows; r += G, z += step) {
            const uint32_t a = potc_bin(z, n), b = potc_bin(z + kPhi, n);
            out[r][j] = (a * 128 + j * 4) | (b * 128 + j * 4) << 16;
        }
    };
    auto load_at = [&](uint32_t off) -> volatile uint32_t & {
        return *reinterpret_cast<volatile uint32_t *>(reinterpret_cast<unsigned char *>(s_load) + off);
    };
    auto place = [&](uint64_t i) {   // the CTA's first warp
        if (tid >= here) return;
        const uint32_t balls = (uint32_t)min((uint64_t)tile, m - i * tile);
        const uint32_t(*const in)[32] = s_off[i & 1];
        uint32_t t = 0;
        if constexpr (kD > 0) {
            for (; t + 4 <= balls; t += 4) {
                uint32_t off[4][kD], l[4][kD], best[4], val[4];
#pragma unroll
                for (uint32_t w = 0; w < 2 * kD; ++w) {
                    const uint32_t x = in[t * kD / 2 + w][tid];
                    off[2 * w / kD][2 * w % kD] = x & 0xFFFFu;
                    off[(2 * w + 1) / kD][(2 * w + 1) % kD] = x >> 16;
                }
#pragma unroll
                for (uint32_t q = 0; q < 4; ++q)
#pragma unroll
                    for (uint32_t k = 0; k < kD; ++k) l[q][k] = load_at(off[q][k]);
#pragma unroll
                for (uint32_t q = 0; q < 4; ++q) {
#pragma unroll
                    for (uint32_t p = 0; p < q; ++p)
#pragma unroll
                        for (uint32_t k = 0; k < kD; ++k) l[q][k] += off[q][k] == best[p];
                    best[q] = off[q][0];
                    val[q] = l[q][0];
#pragma unroll
                    for (uint32_t k = 1; k < kD; ++k)
                        if (l[q][k] < val[q]) {
                            best[q] = off[q][k];
                            val[q] = l[q][k];
                        }
                    ++val[q];
                }
#pragma unroll
                for (uint32_t q = 0; q < 4; ++q) load_at(best[q]) = val[q];   // in order: the last of a bin stays
            }
        }
        for (; t < balls; ++t) {
            uint32_t best = 0, bl = 0;
            for (uint32_t k = 0; k < d; ++k) {
                const uint32_t c = t * d + k, x = in[c / 2][tid], off = c & 1 ? x >> 16 : x & 0xFFFFu;
                const uint32_t l = load_at(off);
                if (k == 0 || l < bl) {
                    best = off;
                    bl = l;
                }
            }
            load_at(best) = bl + 1;
        }
    };
    __syncthreads();
    if (tid >= 32 && tiles) generate(0);
    __syncthreads();
    for (uint64_t i = 0; i < tiles; ++i) {
        if (tid < 32) place(i);
        else if (i + 1 < tiles) generate(i + 1);
        __syncthreads();
    }
    if (tid < here) {
        uint32_t mx = 0;
        for (uint32_t b = 0; b < n; ++b) mx = max(mx, s_load[b * 32 + tid]);
        max_load[s0 + tid] = mx;
    }
}

}  // namespace dm

extern "C" dm_status dm_potc_max_loads(uint32_t n_bins, uint64_t m_balls, uint32_t d, uint32_t trials,
                                       uint64_t seed, uint32_t *max_load_dev, void *stream) {
    if (n_bins < 1 || n_bins > 256 || d < 1 || d > 64 || m_balls > 0xFFFFFFFFull || !max_load_dev)
        return DM_ERR_INVALID_ARG;
    if (trials == 0) return DM_OK;
    const dm::PotcShape shape = dm::potc_shape(trials, (uint64_t)dm::sm_count());
    const uint32_t tile = 2 * dm::kPotcRows / d & ~3u;   // d <= 64: at least 4 balls
    const size_t smem = size_t(n_bins) * 32 * 4;         // at most 32 KB
    const auto st = static_cast<cudaStream_t>(stream);
    const auto k = d == 1 ? dm::k_potc<1> : d == 2 ? dm::k_potc<2> : d == 3 ? dm::k_potc<3> : d == 4 ? dm::k_potc<4>
                                                                                                     : dm::k_potc<0>;
    static dm::SmemOptIn opt[5];   // past 48 KB with the tiles
    cudaError_t e = dm::opt_in_smem(opt[d <= 4 ? d : 0], smem, k);
    if (e == cudaSuccess) {
        k<<<shape.grid, 32 + dm::kPotcGen, smem, st>>>(n_bins, m_balls, d, trials, seed, max_load_dev, shape.per_cta,
                                                       tile);
        e = cudaGetLastError();
    }
    return e == cudaSuccess ? DM_OK : DM_ERR_CUDA;
}
