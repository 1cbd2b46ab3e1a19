// Sample-resident step loop: every step of one update window of one sample
// in one CTA (grid = samples), for networks small enough to live on one SM.
//
// Within an update window the samples of a batch do not interact (weights
// change only at window ends), so a small network needs neither a launch per
// kernel and step nor a barrier over the grid: neuron state stays in
// registers, the delivery ring and the step's spike list in shared memory,
// and the steps are separated by block barriers only.  What bounds it is the
// chain of one step (neuron update -> spike list -> rows of the spiking
// neurons -> ring), not bandwidth.  Roles of the warps:
//   workers  (the rest)  neuron updates (NPT neurons per thread), then the
//            rows of the step's spiking neurons added to the ring;
//   inputs   (if there are input channels)  the rows of the input spikes, one
//            step ahead of the neurons and pipelined over three steps (ids;
//            row bounds; records), so their L2 latency is off the chain;
//   readout  (one warp per 32 readouts)  readout, error signal and loss of
//            the previous step, beside the current one.
// Measured (one GB300, whole calls, per-step launches or the cooperative step
// loop before -> this loop): 100 LIF, 1000 steps 10.4 -> 3.0 ms (the loop
// itself 1.40 ms, 1.4 us per step); batch of 64, 200 ALIF, 350 steps with 13
// input events each 7.7 -> 2.9 ms (loop 0.98 ms; with 4 instead of 16 input
// warps 2.24 ms, bound by the input rows); batch of 32, 100 ALIF, 2200 steps
// 43.1 -> 8.6 ms (loop 2.08 ms).
// One barrier of the workers (spike list complete) and one of the block per
// step.  The ring holds two 32-bit words per entry: an arrival's low word is
// added by a shared-memory atomic whose returned value gives the carry into
// the high word, so the 64-bit sums are exact in any order and equal those of
// the per-step kernels; the neuron update and the error signal are the same
// device functions (neuron_core.cuh): results are bit-identical to them.
#include "eprop_internal.cuh"
#include "eprop_launch.h"
#include "neuron_core.cuh"

namespace eprop {

constexpr int kSmpInCap = 256;         // input events per step in the pipelined buffers
constexpr int kSmpMaxOut = 128;        // readouts: at most 4 readout warps
constexpr int kSmpMaxRec = 1024;
constexpr int kSmpMaxIn = 32768;
constexpr long long kSmpMaxNnz = 1LL << 21;
constexpr int kSmpPart = 128;          // records of a row per delivery item: 4 per lane in flight

struct SampleShape {
    int R;          // ring slots (power of two >= D + 2)
    int NP;         // neurons padded to 32
    int threads;    // 512 or 1024
    int KR, KI;     // readout and input warps
    int in_words;   // words of one input bitset
};

__host__ __device__ inline SampleShape sample_shape(int n_in, int n_rec, int n_out, int D) {
    SampleShape s;
    s.R = 4;
    while (s.R < D + 2) s.R <<= 1;
    s.NP = (n_rec + 31) & ~31;
    s.KR = (n_out + 31) / 32;
    // many channels bring many input rows per step: half the warps of a block
    // of 1024 when one thread per neuron still fits beside them
    const bool wide = n_in >= 256 && s.NP / 32 <= 32 - 16 - s.KR;
    s.threads = wide ? 1024 : 512;
    s.KI = n_in == 0 ? 0 : wide ? 16 : 4;
    s.in_words = (n_in + 31) / 32;
    return s;
}

static size_t sample_smem(const SampleShape &s) {
    size_t b = ((size_t)s.R * s.NP + 32) * 8;                 // ring words and a spare one per lane
    b += (size_t)3 * s.NP * sizeof(int4);                     // spike lists of three steps
    if (s.KI) {
        b += (size_t)2 * kSmpInCap * (sizeof(int4) + sizeof(int));   // input rows and ids of two steps
        b += (size_t)2 * s.in_words * 4;                             // input bitsets
    }
    return b;
}

__device__ __forceinline__ void bar_sync(int id, int threads) {
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

// Adds up to 32 M records of a row to the ring (one warp).  No branch per
// record: absent ones add zero to the warp's spare words, so the conversions
// and the atomics of the batch overlap.
template <int M>
__device__ __forceinline__ void add_records(const Net &n, int start, int cnt, int i, int smask, int NP, int spare,
                                            uint32_t *ring_lo, uint32_t *ring_hi) {
    const int lane = threadIdx.x & 31;
    uint32_t td[M];
    float wv[M];
#pragma unroll
    for (int u = 0; u < M; ++u) {
        const int k = lane + 32 * u;
        td[u] = k < cnt ? __ldg(n.tgt_d + start + k) : 0u;
        wv[u] = k < cnt ? __ldg(n.w + start + k) : 0.f;
    }
    long long fx[M];
    to_fixed(wv, fx);
    int o[M];
    uint32_t old[M];
#pragma unroll
    for (int u = 0; u < M; ++u)
        o[u] = td[u] ? ((i + (int)(td[u] >> 24)) & smask) * NP + (int)(td[u] & 0xFFFFFFu) : spare;
#pragma unroll
    for (int u = 0; u < M; ++u) old[u] = atomicAdd(ring_lo + o[u], (uint32_t)fx[u]);
#pragma unroll
    for (int u = 0; u < M; ++u)
        atomicAdd(ring_hi + o[u],
                  (uint32_t)((unsigned long long)fx[u] >> 32) + (old[u] + (uint32_t)fx[u] < old[u] ? 1u : 0u));
}

template <bool VAR, int NPT, int BT>
__global__ void __launch_bounds__(BT, 1) sample_steps_kernel(Net n, int i0, int i1, int lists) {
    extern __shared__ __align__(16) unsigned char dsm[];
    __shared__ uint32_t thr_s[64];
    __shared__ int cnt_s[3];                     // spikes of a step (slot step mod 3)
    __shared__ int bcnt_s[4][kBkt];              // spike-list buckets of a step (slot step mod 4)
    __shared__ int xn_s[4];                      // input events of a step (slot step mod 4)
    __shared__ long long xq_s[4];
    __shared__ float red_s[4];
    const SampleShape sh = sample_shape(n.n_in, n.n_rec, n.n_out, n.D);
    uint32_t *ring_lo = reinterpret_cast<uint32_t *>(dsm);
    uint32_t *ring_hi = ring_lo + sh.R * sh.NP + 32;
    int4 *slist = reinterpret_cast<int4 *>(ring_hi + sh.R * sh.NP + 32);
    int4 *xrow = slist + 3 * sh.NP;
    int *xid = reinterpret_cast<int *>(xrow + 2 * kSmpInCap);
    uint32_t *xbit = reinterpret_cast<uint32_t *>(xid + 2 * kSmpInCap);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int b = blockIdx.x, N = n.n_rec, K = n.n_out, D = n.D, U = n.U, T = n.T;
    const int NW = BT / 32 - sh.KR - sh.KI;    // worker warps
    const Clock ck = *n.clock;
    const int len = n.lengths[b];
    const int i_last = min(i1, len);
    const int rmask = n.RW * 32 - 1;
    const long long nb0 = (long long)b * N;
    const int D1 = D + 1, smask = sh.R - 1, spare = sh.R * sh.NP + lane;
    long long *ring_g = n.ring + (long long)b * D1 * N;

    if (i0 <= i_last) {
        // ---- state of the sample
        for (int m = tid; m < n.n_thr; m += BT) thr_s[m] = n.drive_thr[m];
        if (tid < 3) cnt_s[tid] = 0;
        if (tid < 4 * kBkt) bcnt_s[tid >> 5][tid & 31] = 0;
        for (int q = tid; q < 2 * (sh.R * sh.NP + 32); q += BT) ring_lo[q] = 0;
        if (sh.KI)
            for (int q = tid; q < 2 * sh.in_words; q += BT) xbit[q] = 0;
        __syncthreads();
        for (int d = 0; d < D; ++d) {            // arrivals pending at steps i0 .. i0 + D - 1
            const long long *src = ring_g + (long long)((ck.ring0 + i0 + d) % D1) * N;
            const int so = ((i0 + d) & smask) * sh.NP;
            for (int j = tid; j < N; j += BT) {
                const unsigned long long v = (unsigned long long)src[j];
                ring_lo[so + j] = (uint32_t)v;
                ring_hi[so + j] = (uint32_t)(v >> 32);
            }
        }
        __syncthreads();
        unsigned long long ev = 0;

        // one delivery item (one warp): records [start, start + cnt), cnt <= kSmpPart
        auto deliver = [&](int start, int cnt, int i) {
            if (cnt <= kSmpPart / 2)
                add_records<kSmpPart / 64>(n, start, cnt, i, smask, sh.NP, spare, ring_lo, ring_hi);
            else
                add_records<kSmpPart / 32>(n, start, cnt, i, smask, sh.NP, spare, ring_lo, ring_hi);
        };

        if (warp < NW) {
            // ------------------------------------------------ workers
            NeuronRegs st[NPT];
            uint32_t *words[NPT];
            uint32_t word[NPT], rword[NPT];
            int rstart[NPT], rlen[NPT];
            float *psi_p[NPT];
#pragma unroll
            for (int q = 0; q < NPT; ++q) {
                const int j = tid + q * NW * 32;
                const bool in = j < N;
                const long long nb = nb0 + (in ? j : 0);
                st[q] = NeuronRegs{n.v[nb], n.v_lo[nb], n.a[nb], n.a_lo[nb], n.ref[nb], (float)n.z_prev[nb], 0.f};
                if (VAR && n.R_win) st[q].rate = n.rate[nb];
                words[q] = n.bits + ((long long)b * n.n_src + n.n_in + (in ? j : 0)) * n.RW;
                word[q] = rword[q] = 0u;
                const long long rb = n.row_ptr[n.n_in + (in ? j : 0)];
                rstart[q] = (int)rb;
                rlen[q] = (int)(n.row_ptr[n.n_in + (in ? j : 0) + 1] - rb);
                psi_p[q] = n.psi_hist + ((long long)b * (U + 1) + 1) * N + (in ? j : 0);
            }
            const int W32 = (T + 31) / 32;
            const int nch = (n.segs * kSeg + kSmpPart - 1) / kSmpPart;     // items per row
            __syncthreads();                     // inputs of step i0 delivered
            for (int i = i0; i <= i_last; ++i) {
                const int r = ck.r_base + i;
                const int so = (i & smask) * sh.NP;
                int4 *lst = slist + (i % 3) * sh.NP;
#pragma unroll
                for (int q = 0; q < NPT; ++q) {
                    const int j = tid + q * NW * 32;
                    int z = 0;
                    if (j < N) {
                        const long long acc = (long long)(((unsigned long long)ring_hi[so + j] << 32) | ring_lo[so + j]);
                        ring_lo[so + j] = 0u;
                        ring_hi[so + j] = 0u;
                        const int fz = n.forced ? (n.forced[((long long)b * T + (i - 1)) * N + j] ? 1 : 0) : -1;
                        float psi;
                        neuron_core<VAR>(n, j, ck.t_abs_base + i, drive_count(n, b, j, ck.t_abs_base + i, thr_s), acc, fz,
                                         st[q], psi, z);
                        *psi_p[q] = psi;
                        psi_p[q] += N;
                        if (VAR && n.R_win) n.R_win[((long long)b * U + (i - i0)) * N + j] = rate_signal(n, st[q].rate);
                        if (n.record_psi) n.rec_psi[((long long)b * T + (i - 1)) * N + j] = psi;
                    }
                    const unsigned m = __ballot_sync(0xffffffffu, z);
                    if (m) {
                        int base = 0;
                        if (lane == 0) base = atomicAdd(&cnt_s[i % 3], __popc(m));
                        base = __shfl_sync(0xffffffffu, base, 0);
                        if (z) {
                            lst[base + __popc(m & ((1u << lane) - 1u))] = make_int4(j, rstart[q], rlen[q], 0);
                            word[q] |= 1u << (r & 31);
                            rword[q] |= 1u << ((i - 1) & 31);
                            ev += (unsigned long long)rlen[q];
                            if (lists) {
                                const int src = n.n_in + j, bk = (src >> 8) & (kBkt - 1);
                                const int pos = atomicAdd(&bcnt_s[i & 3][bk], 1);
                                n.list_ids[(list_index(n, b, r % n.RS) + bk) * n.list_cap + pos] = src;
                            }
                        }
                    }
                    // spike bits leave the register at word ends
                    if ((r & 31) == 31 || i == i_last) {
                        if (word[q]) atomicOr(words[q] + ((r & rmask) >> 5), word[q]);
                        word[q] = 0u;
                    }
                    if (n.record_raster && (((i - 1) & 31) == 31 || i == i_last)) {
                        if (rword[q]) atomicOr(&n.rec_raster[((long long)b * W32 + ((i - 1) >> 5)) * N + j], rword[q]);
                        rword[q] = 0u;
                    }
                }
                bar_sync(1, NW * 32);            // the step's spike list is complete
                const int items = cnt_s[i % 3] * nch;
                for (int it = warp; it < items; it += NW) {
                    const int4 e = lst[nch == 1 ? it : it / nch];
                    const int c0 = nch == 1 ? 0 : (it % nch) * kSmpPart;
                    if (c0 < e.z) deliver(e.y + c0, min(kSmpPart, e.z - c0), i);
                }
                __syncthreads();
            }
            // ---- state back to memory
#pragma unroll
            for (int q = 0; q < NPT; ++q) {
                const int j = tid + q * NW * 32;
                if (j >= N) continue;
                const long long nb = nb0 + j;
                n.v[nb] = st[q].v_hi;
                n.v_lo[nb] = st[q].v_lo;
                n.a[nb] = st[q].a_hi;
                n.a_lo[nb] = st[q].a_lo;
                n.ref[nb] = st[q].ref;
                n.z_prev[nb] = (uint8_t)(st[q].zp != 0.f);
                if (VAR && n.R_win) n.rate[nb] = st[q].rate;
                ring_g[(long long)((ck.ring0 + i_last) % D1) * N + j] = 0;
                for (int d = 1; d <= D; ++d) {
                    const int so = ((i_last + d) & smask) * sh.NP;
                    ring_g[(long long)((ck.ring0 + i_last + d) % D1) * N + j] =
                        (long long)(((unsigned long long)ring_hi[so + j] << 32) | ring_lo[so + j]);
                }
            }
        } else if (warp < NW + sh.KI) {
            // ------------------------------------------------ inputs
            const int xt = tid - NW * 32, xw = warp - NW;
            const int XT = sh.KI * 32;
            const long long *xp = n.x_ptr + (long long)b * T;
            // an input spike of step t: bit, list entry, row; false if the
            // channel was already seen in this step
            auto take = [&](int t, int id) -> bool {
                const uint32_t m = 1u << (id & 31);
                if (atomicOr(&xbit[(t & 1) * sh.in_words + (id >> 5)], m) & m) return false;
                const int r = ck.r_base + t;
                atomicOr(n.bits + ((long long)b * n.n_src + id) * n.RW + ((r & rmask) >> 5), 1u << (r & 31));
                if (lists) {
                    const int bk = (id >> 8) & (kBkt - 1);
                    const int pos = atomicAdd(&bcnt_s[t & 3][bk], 1);
                    n.list_ids[(list_index(n, b, r % n.RS) + bk) * n.list_cap + pos] = id;
                }
                return true;
            };
            auto stage_ids = [&](int t) {
                if (t < i0 || t > i_last) return;
                const long long q0 = __ldg(xp + t - 1), q1 = __ldg(xp + t);
                const int m = (int)(q1 - q0);
                if (xt == 0) {
                    xn_s[t & 3] = m;
                    xq_s[t & 3] = q0;
                }
                for (int e = xt; e < min(m, kSmpInCap); e += XT) xid[(t & 1) * kSmpInCap + e] = __ldg(n.x_ids + q0 + e);
            };
            auto stage_rows = [&](int t) {
                if (t < i0 || t > i_last) return;
                const int m = min(xn_s[t & 3], kSmpInCap);
                for (int e = xt; e < m; e += XT) {
                    const int id = xid[(t & 1) * kSmpInCap + e];
                    const long long rb = __ldg(n.row_ptr + id), re = __ldg(n.row_ptr + id + 1);
                    const bool ok = take(t, id);
                    if (ok) ev += (unsigned long long)(re - rb);
                    xrow[(t & 1) * kSmpInCap + e] = make_int4(id, (int)rb, ok ? (int)(re - rb) : 0, 0);
                }
            };
            const int nch = (n.segs * kSeg + kSmpPart - 1) / kSmpPart;
            auto stage_deliver = [&](int t) {
                if (t < i0 || t > i_last) return;
                const int m = xn_s[t & 3], mc = min(m, kSmpInCap);
                for (int it = xw; it < mc * nch; it += sh.KI) {
                    const int4 e = xrow[(t & 1) * kSmpInCap + it / nch];
                    const int c0 = (it % nch) * kSmpPart;
                    if (c0 < e.z) deliver(e.y + c0, min(kSmpPart, e.z - c0), t);
                }
                // events beyond the buffers, one warp each
                for (int e = kSmpInCap + xw; e < m; e += sh.KI) {
                    const int id = n.x_ids[xq_s[t & 3] + e];
                    int ok = 0;
                    if (lane == 0) ok = take(t, id) ? 1 : 0;
                    if (!__shfl_sync(0xffffffffu, ok, 0)) continue;
                    const int rb = (int)n.row_ptr[id], re = (int)n.row_ptr[id + 1];
                    if (lane == 0) ev += (unsigned long long)(re - rb);
                    for (int c = rb; c < re; c += kSmpPart) deliver(c, min(kSmpPart, re - c), t);
                }
                if (m > kSmpInCap) bar_sync(2, XT);     // every event of the step is marked
                for (int e = xt; e < m; e += XT) {
                    const int id = e < mc ? xrow[(t & 1) * kSmpInCap + e].x : n.x_ids[xq_s[t & 3] + e];
                    xbit[(t & 1) * sh.in_words + (id >> 5)] = 0u;
                }
            };
            for (int i = i0 - 3; i < i0; ++i) {          // fill the pipeline
                stage_ids(i + 3);
                stage_rows(i + 2);
                stage_deliver(i + 1);
                bar_sync(2, XT);
            }
            __syncthreads();
            for (int i = i0; i <= i_last; ++i) {
                stage_ids(i + 3);
                stage_rows(i + 2);
                stage_deliver(i + 1);
                __syncthreads();
            }
        } else {
            // ------------------------------------------------ readout
            const int k = tid - (NW + sh.KI) * 32, rw = warp - NW - sh.KI;
            const int RT = sh.KR * 32;
            const bool has_k = k < K;
            const long long bk = (long long)b * K + (has_k ? k : 0);
            float y = has_k ? n.y[bk] : 0.f;
            float loss = k == 0 ? n.loss_acc[b] : 0.f;
            // lanes at and past K hold the neutral element: with few readouts
            // the wider exchanges change nothing (the first lanes have the result)
            int width = 16;
            while (sh.KR == 1 && width >= K && width > 1) width >>= 1;
            auto reduce = [&](float x, bool mx) -> float {
                for (int o = width; o > 0; o >>= 1) {
                    const float v = __shfl_xor_sync(0xffffffffu, x, o);
                    x = mx ? fmaxf(x, v) : x + v;
                }
                if (sh.KR == 1) return x;
                bar_sync(3, RT);
                if (lane == 0) red_s[rw] = x;
                bar_sync(3, RT);
                float t = mx ? -INFINITY : 0.0f;
                for (int q = 0; q < sh.KR; ++q) t = mx ? fmaxf(t, red_s[q]) : t + red_s[q];
                return t;
            };
            auto load_tgt = [&](int i) {
                return (has_k && i <= i_last) ? n.targets[((long long)b * T + (i - 1)) * K + k] : 0.f;
            };
            auto load_win = [&](int i) -> int {  // (converted where it is used, a step later)
                return i <= i_last ? n.window[(long long)b * T + (i - 1)] : 0;
            };
            float tgt = load_tgt(i0);
            int win = load_win(i0);
            auto finish = [&](int i) {           // readout of step i (its spike list is complete)
                const float tgt_n = load_tgt(i + 1);
                const int win_n = load_win(i + 1);
                const int c = cnt_s[i % 3];
                const int4 *lst = slist + (i % 3) * sh.NP;
                long long acc = 0;
                if (has_k) {
                    constexpr int kC = 4;
                    for (int e = 0; e < c; e += kC) {
                        float wv[kC];
                        long long fx[kC];
#pragma unroll
                        for (int u = 0; u < kC; ++u)
                            wv[u] = e + u < c ? __ldg(n.w_out + (long long)lst[e + u].x * K + k) : 0.f;
                        to_fixed(wv, fx);
#pragma unroll
                        for (int u = 0; u < kC; ++u) acc += fx[u];
                    }
                }
                if (has_k) {
                    y = readout_step(n, y, acc);
                    n.y_rec[((long long)b * T + (i - 1)) * K + k] = y;
                }
                float E;
                const float l = error_signal(n, y, tgt, (float)win, has_k, E, [&](float x) { return reduce(x, true); },
                                             [&](float x) { return reduce(x, false); });
                if (has_k) n.E_win[((long long)b * U + (i - i0)) * K + k] = E;
                const float tot = reduce(l, false);
                if (k == 0) loss += tot;
                if (lists && rw == 0) {          // the step's list is complete as well
                    n.list_cnt[list_index(n, b, (ck.r_base + i) % n.RS) + lane] = bcnt_s[i & 3][lane];
                    bcnt_s[i & 3][lane] = 0;
                }
                tgt = tgt_n;
                win = win_n;
            };
            __syncthreads();
            for (int i = i0; i <= i_last; ++i) {
                if (k == 0) cnt_s[(i + 1) % 3] = 0;
                if (i > i0) finish(i - 1);
                __syncthreads();
            }
            finish(i_last);
            if (has_k) n.y[bk] = y;
            if (k == 0) n.loss_acc[b] = loss;
        }
        for (int o = 16; o > 0; o >>= 1) ev += __shfl_xor_sync(0xffffffffu, ev, o);
        if (lane == 0 && ev) atomicAdd(n.events, ev);
    }
    // ---- steps after the sample's end: frozen, silent, no error
    for (int i = max(i0, len + 1); i <= i1; ++i) {
        float *psi_row = n.psi_hist + ((long long)b * (U + 1) + (i - i0 + 1)) * N;
        for (int j = tid; j < N; j += BT) {
            psi_row[j] = 0.f;
            if (VAR && n.R_win) n.R_win[((long long)b * U + (i - i0)) * N + j] = 0.f;
            if (n.record_psi) n.rec_psi[((long long)b * T + (i - 1)) * N + j] = 0.f;
        }
        for (int k = tid; k < K; k += BT) {
            n.E_win[((long long)b * U + (i - i0)) * K + k] = 0.f;
            n.y_rec[((long long)b * T + (i - 1)) * K + k] = 0.f;
        }
        if (lists && tid < kBkt) n.list_cnt[list_index(n, b, (ck.r_base + i) % n.RS) + tid] = 0;
    }
    if (lists && tid < kBkt) n.list_cnt[list_index(n, b, (ck.r_base + i1 + 1) % n.RS) + tid] = 0;
}

// One thread per neuron (at most four), synapses that fit one SM's L1/L2
// share and whose per-step events one SM adds faster than a step's launches
// take.
bool sample_net_small(const Net &n) {
    return n.n_rec <= kSmpMaxRec && n.n_in <= kSmpMaxIn && n.n_out <= kSmpMaxOut && n.nnz <= kSmpMaxNnz;
}
bool sample_steps_fit(const Net &n) {
    return sample_net_small(n) && n.pred_mode == 0 && n.d_out == 0 && !n.band && !(n.has_state && !n.dense);
}

#define EPROP_SMP_EACH(X) \
    X(true, 1, 512) X(true, 2, 512) X(true, 4, 512) X(true, 1, 1024) \
    X(false, 1, 512) X(false, 2, 512) X(false, 4, 512) X(false, 1, 1024)

void launch_sample_steps(const Net &n, int i0, int i1, cudaStream_t st) {
    const SampleShape s = sample_shape(n.n_in, n.n_rec, n.n_out, n.D);
    const size_t sm = sample_smem(s);
    const int nt = s.threads - (s.KR + s.KI) * 32;
    const int npt = n.n_rec <= nt ? 1 : n.n_rec <= 2 * nt ? 2 : 4;
    const bool var = n.surrogate || n.reset_mode || n.if_period || n.R_win;
    const int lists = n.B == 1 && n.RS > n.U;   // forms whose window kernels walk the spike lists
#define EPROP_SMP(V, P, BT)                            \
    if (var == V && npt == P && s.threads == BT) {     \
        sample_steps_kernel<V, P, BT><<<n.B, BT, sm, st>>>(n, i0, i1, lists); \
        return;                                        \
    }
    EPROP_SMP_EACH(EPROP_SMP)
#undef EPROP_SMP
}

void prepare_sample_attributes() {
#define EPROP_SMP(V, P, BT) \
    cudaFuncSetAttribute(sample_steps_kernel<V, P, BT>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
    EPROP_SMP_EACH(EPROP_SMP)
#undef EPROP_SMP
}

}  // namespace eprop
