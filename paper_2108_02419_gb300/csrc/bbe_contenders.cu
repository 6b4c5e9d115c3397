// bbe_contenders.cu -- which competitors of a race the rollout kernel (bbe_win.cuh) advances: those that can
// matter to the first finish, or the first K.  One warp a race, before the rollouts of a pass.
//
// The search is a chain of H dependent steps over the race (H: the steps that a rollout may take), about as
// long as one to four rollouts, and its code is as large as the rollout kernel's loop.  Run by every work item in the
// rollout kernel, it took up to a third of calls where hardly anybody is left out, 64 rollouts an item being
// too few to pay for it, and drove the loop out of the instruction cache.  Once a race, us per call (in every item,
// without it, once a race): 2285 races of 24 to the first place, 266 rollouts each, 1018, 880, 890; 105 of 28
// to the fourth, 2098 each, 749, 556, 568; 97 of 28 to the first, 14846 each, 2480, 2245, 1980; 4096 of 20,
// 10^4 each, 32100, 50000, 24400.
#include <cuda_runtime.h>

#include <climits>
#include <cmath>
#include <cstdint>

#include "bbe_internal.h"
#include "bbe_rng.cuh"

namespace bbe {

namespace {

constexpr unsigned kAll = 0xffffffffu;
constexpr int kWarps = 4;  // races a block

__device__ __forceinline__ float warp_max(float v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(kAll, v, o));
    return v;
}

// The contenders of a race.  The first K finishers are decided among the competitors near the front, and
// Eq. 1 passes influence from front to back only, so a competitor that is certain to stay short of the
// line until a rollout ends cannot change its first K places, nor when they are filled.
// contender_mask returns the competitors that are not ruled out so: in every rollout that ends within
// H steps (H is set here), a rollout of these alone, each on its own stream, has the same first K
// finishers and the same number of steps.
//
// The bound, for any draws.  E_i(t) bounds the position after t steps of every competitor that starts at or
// behind rank i (ranks by start position) and of everyone that one of them has affected (the affected
// were behind it, so the bound holds for them from there on).  A free step is at most F = max R P (mu +
// z_max sigma), the largest over the competitors (the generator's |z| is bounded: u1 >= 2^-24 gives a
// radius of at most 5.7681; sqrt(3) and 1 for the other two distributions) and at least the previous
// steps given.  A blocked step is R min(own previous step, that of the competitor in front), so with lambda
// the largest R where it happens,
//   S_c(t) > lambda^k F  =>  S(t-1) > lambda^(k-1) F for c and for the one in front of it, within theta,
// and the foremost of those who have S(t-i) > lambda^(k-i) F has one in front that is not among them:
// k levels take k members whose R can exceed 1, each within n theta of another at some of the last k
// steps.  A member that was there i steps ago has fallen back since by at most i steps' difference
// between the largest step and F, by less than M in all.  So if j is the rearmost member, c is at most M
// ahead of E_j, the others rank above j and started behind E_j + M + n theta, and those are counted
// (k_j, lambda_j):
//   V_j = F lambda_j^k_j,   E_i(t+1) = max over j <= i of min(E_j(t) + M, E_i(t)) + V_j.
// M for step t follows from the levels of the step before, which a step exceeds by one at most.  Rounding is
// covered by the factors and the margins.  A competitor is ruled out when its E stays short of the
// line for H steps.  (With one bound for everybody's advance, the closest groups anywhere on the
// track count against all: 10 contenders of 20 at the mean in the uniform batch, 4.8 with this one.)
//
// H is an estimate of the K-th finish with a margin of three standard deviations (two and four: within 2 % for
// 4096 spread races of 20, 10^4 uneven ones and places); the few rollouts that are still running after
// H steps are run again with everybody.
// x: 3 n floats of scratch; most: contenders, at most, that leave room for more segments (else everybody is
// returned, as soon as that is certain: a bound grows by its own advance of this step at least in every
// later one, as its members and their R only grow).  Called by the whole warp; lane c < n holds competitor c.
template <int DIST, int LAW>
__device__ __forceinline__ unsigned contender_mask(float *x, int n, int lane, float d, float mu, float sigma, float P,
                                                   float kr, float prev, float theta, float L, float invL, float t0,
                                                   float invT, int K, int most, int &H)
{
    const bool on = lane < n;
    const unsigned everybody = kAll >> (32 - n);
    constexpr float zmax = DIST == BBE_DIST_NORMAL ? 5.769f : (DIST == BBE_DIST_UNIFORM ? 1.7321f : 1.0f);
    // expected finish at the R of the middle of the way, and the horizon: the K-th least with its margin
    float T = (L - d) / (mu * P);
    T /= 1.0f + (LAW == BBE_LAW_TIME ? kr * (fminf((t0 + 0.5f * T) * invT, 1.0f) - 0.5f) : 0.5f * kr * d * invL);
    const float h = on ? T + 3.0f * sigma * sqrtf(T) / mu + 1.0f : INFINITY;
    int rank = 0, hrank = 0;  // by (start position, index) and by (horizon, index)
    for (int i = 0; i < n; ++i) {
        const float di = __shfl_sync(kAll, d, i), hi = __shfl_sync(kAll, h, i);
        rank += di < d || (di == d && i < lane) ? 1 : 0;
        hrank += hi < h || (hi == h && i < lane) ? 1 : 0;
    }
    const float hk = warp_max(on && hrank < K ? h : 0.0f);
    const float margin = float(n) * warp_max(on ? theta : 0.0f);
    if (!(hk < 1e6f) || !(margin < L)) return everybody;
    H = int(hk) + 1;
    // R is linear in the position or the time: largest at an end of its range
    const float lo = LAW == BBE_LAW_TIME ? fminf(t0 * invT, 1.0f) : d * invL;
    const float end = LAW == BBE_LAW_TIME ? fminf((t0 + float(H)) * invT, 1.0f) : (L + margin) * invL;
    const float Rlo = 1.0f + kr * (lo - 0.5f);
    const float R = 1.00001f * fmaxf(Rlo, 1.0f + kr * (end - 0.5f));
    const float F = 1.0001f * fmaxf(warp_max(on ? fmaxf(prev, R * P * (mu + zmax * sigma)) : 0.0f), kStepFloor);
    const float goal = 0.9999f * L;
    // too many get there even at the free pace
    if (__popc(__ballot_sync(kAll, on && !(goal - float(H) * F > d))) > most) return everybody;
    const float lambda = 1.00001f * fmaxf(warp_max(on ? R : 0.0f), 1.0f);  // anywhere
    // from here on lane i holds rank i
    if (on) {
        x[rank] = d;
        x[n + rank] = kr;
        x[2 * n + rank] = Rlo;
    }
    __syncwarp();
    float E = on ? x[lane] : INFINITY, M = margin;
    float rise = 0.0f, Rmax = 1.0f;  // of the ranks lane .. next - 1: the largest kr, and R at the range's start
    int next = lane, early = 0, late = 0;  // those whose R exceeds 1 there, and those later on only
    for (int t = 0; t < H;) {
        while (next < n && x[next] <= E + M + margin) {
            const float k1 = x[n + next], r1 = x[2 * n + next];
            Rmax = fmaxf(Rmax, r1);
            if (r1 > 0.9999f) ++early;
            else if (k1 > 0.0f) ++late;
            rise = fmaxf(rise, k1);
            ++next;
        }
        const float now = LAW == BBE_LAW_TIME ? fminf((t0 + float(t)) * invT, 1.0f) : fminf((E + M + margin) * invL, end);
        const int k = early + (now > 0.4999f ? late : 0);
        const float lam = 1.00001f * fmaxf(Rmax, 1.0f + rise * (now - 0.5f));
        const float V = on ? 1.0001f * F * powf(lam, float(k)) : 0.0f;
        float En = E + V;
        for (int j = 0; j + 1 < n; ++j) {
            const float Ej = __shfl_sync(kAll, E, j), Vj = __shfl_sync(kAll, V, j);
            if (j < lane) En = fmaxf(En, fminf(Ej + M, E) + Vj);
        }
        E = En;
        if (__popc(__ballot_sync(kAll, on && !(goal - float(H - t - 1) * V > E))) > most) {
            __syncwarp();
            return everybody;
        }
        const int km = __reduce_max_sync(kAll, on ? k : 0);
        M = fmaxf(M, margin + float(km) * F * (1.0002f * powf(lambda, float(km)) - 1.0f));
        ++t;
    }
    const float bound = __shfl_sync(kAll, E, rank & 31);
    const bool out = on && !(bound >= goal);
    __syncwarp();
    return everybody & ~__ballot_sync(kAll, out);
}

template <int DIST, int LAW>
__global__ void __launch_bounds__(32 * kWarps) contender_kernel(ContenderLaunch l)
{
    __shared__ float scratch[kWarps][3 * BBE_MAX_COMPETITORS];
    const DevBatch &b = l.b;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int r = blockIdx.x * kWarps + warp;
    if (r >= b.n_races) return;
    const int off = b.race_off[r];
    const int n = BBE_INDEX(b.race_off[r + 1] - off - 1, BBE_MAX_COMPETITORS, l.status) + 1;  // 1..32
    (void)BBE_INDEX(off + n - 1, b.n_total, l.status);
    const int K = min(l.places, n);
    const int slots = 32 * int(l.slots_by_n[n]);
    const unsigned everybody = kAll >> (32 - n);
    Contenders found{everybody, INT_MAX};
    // Only for races with eight rollouts a segment at least: of 200 batches of 1500 to 12000 races with 10 to
    // 400 rollouts none was then slower than with a kernel that knew no contenders; from four on the worst took
    // 28 % longer, from two on 48 %.
    const int seg_all = slots / n;
    bool worth = b.R[r] >= 8 * int64_t(seg_all);
#if defined(BBE_CHECKED) && BBE_CHECKED
    worth = worth || l.always;
#endif
    if (worth && K < n && slots > 0) {
        float d = INFINITY, mu = 1.0f, sigma = 0.0f, P = 1.0f, theta = 0.0f, kr = 0.0f, prev = 0.0f;
        if (lane < n) {
            const int ci = off + lane;
            mu = b.mu[ci];
            P = b.P[ci];
            sigma = b.sigma[ci];
            theta = b.theta[ci];
            d = b.d0[ci];
            kr = __fmul_rn(kKappa, __fsub_rn(__fmul_rn(2.0f, b.rho[ci]), 1.0f));
            prev = b.prev0 ? b.prev0[ci] : __fmul_rn(mu, P);
        }
        const float L = b.L[r];
        const float t0 = LAW == BBE_LAW_TIME ? b.t0[r] : 0.0f, invT = LAW == BBE_LAW_TIME ? b.invT[r] : 0.0f;
        int H = 0;
        const unsigned front = contender_mask<DIST, LAW>(scratch[warp], n, lane, d, mu, sigma, P, kr, prev, theta, L,
                                                         __fdiv_rn(1.0f, L), t0, invT, K, slots / (seg_all + 1), H);
        const int nf = __popc(front);
        const int cap = l.seg_cap > 0 ? l.seg_cap : slots;
        if (nf >= K && min(slots / nf, cap) > min(seg_all, cap)) found = Contenders{front, H};
    }
    if (lane == 0) l.found[r] = found;
}

template <int LAW>
void launch_law(const ContenderLaunch &l, cudaStream_t stream)
{
    const unsigned grid = unsigned((l.b.n_races + kWarps - 1) / kWarps);
    switch (l.b.dist) {
    case BBE_DIST_NORMAL: contender_kernel<BBE_DIST_NORMAL, LAW><<<grid, 32 * kWarps, 0, stream>>>(l); break;
    case BBE_DIST_UNIFORM: contender_kernel<BBE_DIST_UNIFORM, LAW><<<grid, 32 * kWarps, 0, stream>>>(l); break;
    default: contender_kernel<BBE_DIST_TWO_POINT, LAW><<<grid, 32 * kWarps, 0, stream>>>(l); break;
    }
}

}  // namespace

cudaError_t launch_contenders(const ContenderLaunch &l, cudaStream_t stream)
{
    if (l.b.law == BBE_LAW_TIME) launch_law<BBE_LAW_TIME>(l, stream);
    else launch_law<BBE_LAW_POSITION>(l, stream);
    return cudaGetLastError();
}

}  // namespace bbe
