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
//            rows of the step's spiking neurons added to the ring, and in the
//            same batch their readout weights to the step's readout input;
//   inputs   (if there are input channels)  the rows of the input spikes: each
//            event passes six stages, one per step of the loop, so that no
//            load is waited for in the step it was issued in;
//   readout  (one warp per 32 readouts)  readout, error signal and loss of
//            the previous step, beside the current one; outside the learning
//            window the softmax is skipped (its result is multiplied by zero).
// Measured (one GB300, whole calls, per-step launches or the cooperative step
// loop before -> this loop and the window-end kernels of today): 100 LIF, 1000
// steps 10.4 -> 1.21 ms (0.92 us per step); batch of 64, 200 ALIF, 350
// steps with 13 input events each 8.2 -> 1.10 ms (2.0 us per step, bound by the
// instructions of the input rows); batch of 32, 100 ALIF, 2200 steps 43.1 ->
// 2.04 ms (0.62 us per step).  With the inputs one step ahead and the readout
// summing the spikes itself: 1.34, 1.24 and 2.63 ms.
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

constexpr int kSmpMaxOut = 128;        // readouts: at most 4 readout warps
constexpr int kSmpMaxRec = 1024;
constexpr int kSmpMaxIn = 32768;
constexpr long long kSmpMaxNnz = 1LL << 21;      // all synapses
constexpr long long kSmpMaxNnzRec = 1LL << 19;   // recurrent synapses
constexpr int kSmpPart = 128;          // records of a row per delivery item: 4 per lane in flight

struct SampleShape {
    int R;          // ring slots (power of two >= D + 4: inputs run three steps ahead)
    int NP;         // neurons padded to 32
    int threads;    // 512, 768 or 1024
    int KR, KI;     // readout and input warps
    int in_words;   // words of one input bitset
};

__host__ __device__ inline SampleShape sample_shape(int n_in, int n_rec, int n_out, int D) {
    SampleShape s;
    s.R = 4;
    while (s.R < D + 4) s.R <<= 1;
    s.NP = (n_rec + 31) & ~31;
    s.KR = (n_out + 31) / 32;
    // many channels bring many input rows per step: 16 warps for them and the
    // readout, beside one thread per neuron (8 or 16 worker warps)
    const bool wide = n_in >= 256 && s.NP / 32 <= 16;
    s.threads = !wide ? 512 : s.NP / 32 <= 8 ? 768 : 1024;
    s.KI = n_in == 0 ? 0 : wide ? 16 - s.KR : 4;
    s.in_words = (n_in + 31) / 32;
    return s;
}

static size_t sample_smem(const SampleShape &s) {
    // ring words, a spare one per lane, the readout inputs of two steps
    size_t b = ((size_t)s.R * s.NP + 32 + 2 * s.KR * 32) * 8;
    b += (size_t)3 * s.NP * sizeof(int4);                     // spike lists of three steps
    if (s.KI) {
        b += (size_t)4 * s.KI * 32 * sizeof(int4);                   // input rows of four steps, one per thread
        b += (size_t)2 * s.in_words * 4;                             // input bitsets
    }
    return b;
}

__device__ __forceinline__ void bar_sync(int id, int threads) {
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

// Up to 32 M records of a row (one warp): loads, then adds to the ring.  No
// branch per record: absent ones add zero to the warp's spare words, so the
// conversions and the atomics of the batch overlap.
template <int M>
__device__ __forceinline__ void load_records(const Net &n, int start, int cnt, uint32_t (&td)[M], float (&wv)[M]) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int u = 0; u < M; ++u) {
        const int k = lane + 32 * u;
        td[u] = k < cnt ? __ldg(n.tgt_d + start + k) : 0u;
        wv[u] = k < cnt ? __ldg(n.w + start + k) : 0.f;
    }
}
__device__ __forceinline__ int ring_offset(uint32_t td, int i, int smask, int NP, int spare) {
    return td ? ((i + (int)(td >> 24)) & smask) * NP + (int)(td & 0xFFFFFFu) : spare;
}
// adds weight u at ring offset o[u]
template <int M>
__device__ __forceinline__ void add_words(const float (&wv)[M], const int (&o)[M], uint32_t *ring_lo,
                                          uint32_t *ring_hi) {
    long long fx[M];
    to_fixed(wv, fx);
    uint32_t old[M];
#pragma unroll
    for (int u = 0; u < M; ++u) old[u] = atomicAdd(ring_lo + o[u], (uint32_t)fx[u]);
#pragma unroll
    for (int u = 0; u < M; ++u)
        atomicAdd(ring_hi + o[u],
                  (uint32_t)((unsigned long long)fx[u] >> 32) + (old[u] + (uint32_t)fx[u] < old[u] ? 1u : 0u));
}
template <int M>
__device__ __forceinline__ void add_records(const uint32_t (&td)[M], const float (&wv)[M], int i, int smask, int NP,
                                            int spare, uint32_t *ring_lo, uint32_t *ring_hi) {
    int o[M];
#pragma unroll
    for (int u = 0; u < M; ++u) o[u] = ring_offset(td[u], i, smask, NP, spare);
    add_words(wv, o, ring_lo, ring_hi);
}

template <bool VAR, int NPT, int BT>
__global__ void __launch_bounds__(BT, 1) sample_steps_kernel(Net n, int i0, int i1, int lists) {
    extern __shared__ __align__(16) unsigned char dsm[];
    __shared__ uint32_t thr_s[64];
    __shared__ int cnt_s[3];                     // spikes of a step (slot step mod 3)
    __shared__ int bcnt_s[8][kBkt];              // spike-list buckets of a step (slot step mod 8)
    __shared__ int xn_s[8];                      // input events of a step (slot step mod 8)
    __shared__ long long xq_s[8];
    __shared__ float red_s[4];
    const SampleShape sh = sample_shape(n.n_in, n.n_rec, n.n_out, n.D);
    uint32_t *ring_lo = reinterpret_cast<uint32_t *>(dsm);
    const int ring_n = sh.R * sh.NP + 32 + 2 * sh.KR * 32;
    uint32_t *ring_hi = ring_lo + ring_n;
    int4 *slist = reinterpret_cast<int4 *>(ring_hi + ring_n);
    int4 *xrow = slist + 3 * sh.NP;
    uint32_t *xbit = reinterpret_cast<uint32_t *>(xrow + 4 * sh.KI * 32);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int b = blockIdx.x, N = n.n_rec, K = n.n_out, D = n.D, U = n.U, T = n.T;
    const int NW = BT / 32 - sh.KR - sh.KI;    // worker warps
    const Clock ck = *n.clock;
    const int len = n.lengths[b];
    const int i_last = min(i1, len);
    const int rmask = n.RW * 32 - 1;
    const long long nb0 = (long long)b * N;
    const int D1 = D + 1, smask = sh.R - 1, spare = sh.R * sh.NP + lane;
    const int y0 = sh.R * sh.NP + 32;            // readout input of even steps; odd steps KR * 32 words on
    long long *ring_g = n.ring + (long long)b * D1 * N;

    if (i0 <= i_last) {
        // ---- state of the sample
        for (int m = tid; m < n.n_thr; m += BT) thr_s[m] = n.drive_thr[m];
        if (tid < 3) cnt_s[tid] = 0;
        if (tid < 8 * kBkt) bcnt_s[tid >> 5][tid & 31] = 0;
        for (int q = tid; q < 2 * ring_n; q += BT) ring_lo[q] = 0;
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
            uint32_t td[kSmpPart / 32];
            float wv[kSmpPart / 32];
            load_records(n, start, cnt, td, wv);
            add_records(td, wv, i, smask, sh.NP, spare, ring_lo, ring_hi);
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
            int s3 = i0 % 3;                     // step mod 3
            for (int i = i0; i <= i_last; ++i, s3 = s3 == 2 ? 0 : s3 + 1) {
                const int r = ck.r_base + i;
                const int so = (i & smask) * sh.NP;
                int4 *lst = slist + s3 * sh.NP;
#pragma unroll
                for (int q = 0; q < NPT; ++q) {
                    const int j = tid + q * NW * 32;
                    int z = 0;
                    if (j < N) {
                        const long long acc = (long long)(((unsigned long long)ring_hi[so + j] << 32) | ring_lo[so + j]);
                        ring_lo[so + j] = 0u;
                        ring_hi[so + j] = 0u;
                        const int fz = (VAR && n.forced) ? (n.forced[((long long)b * T + (i - 1)) * N + j] ? 1 : 0) : -1;
                        float psi;
                        const int drive = VAR ? drive_count(n, b, j, ck.t_abs_base + i, thr_s) : 0;
                        neuron_core<VAR, VAR>(n, j, ck.t_abs_base + i, drive, acc, fz, st[q], psi, z);
                        *psi_p[q] = psi;
                        psi_p[q] += N;
                        if (VAR && n.R_win) n.R_win[((long long)b * U + (i - i0)) * N + j] = rate_signal(n, st[q].rate);
                        if (VAR && n.record_psi) n.rec_psi[((long long)b * T + (i - 1)) * N + j] = psi;
                    }
                    if (z) {
                        lst[atomicAdd(&cnt_s[s3], 1)] = make_int4(j, rstart[q], rlen[q], 0);
                        word[q] |= 1u << (r & 31);
                        if (VAR) rword[q] |= 1u << ((i - 1) & 31);
                        ev += (unsigned long long)rlen[q];
                        if (lists) {
                            const int src = n.n_in + j, bk = (src >> 8) & (kBkt - 1);
                            const int pos = atomicAdd(&bcnt_s[i & 7][bk], 1);
                            n.list_ids[(list_index(n, b, r % n.RS) + bk) * n.list_cap + pos] = src;
                        }
                    }
                    // spike bits leave the register at word ends
                    if ((r & 31) == 31 || i == i_last) {
                        if (word[q]) atomicOr(words[q] + ((r & rmask) >> 5), word[q]);
                        word[q] = 0u;
                    }
                    if (VAR && n.record_raster && (((i - 1) & 31) == 31 || i == i_last)) {
                        if (rword[q]) atomicOr(&n.rec_raster[((long long)b * W32 + ((i - 1) >> 5)) * N + j], rword[q]);
                        rword[q] = 0u;
                    }
                }
                bar_sync(1, NW * 32);            // the step's spike list is complete
                const int items = cnt_s[s3] * nch;
                const int yo = y0 + (i & 1) * sh.KR * 32;
                for (int it = warp; it < items; it += NW) {
                    const int4 e = lst[nch == 1 ? it : it / nch];
                    const int c0 = nch == 1 ? 0 : (it % nch) * kSmpPart;
                    if (c0 > 0) {
                        if (c0 < e.z) deliver(e.y + c0, min(kSmpPart, e.z - c0), i);
                        continue;
                    }
                    // the row's first part, and in the same batch the neuron's
                    // readout weights sum_j W_out[j][k] z_j^t
                    constexpr int M = kSmpPart / 32;
                    const float *wo = n.w_out + (long long)e.x * K;
                    uint32_t td[M];
                    float wv[M], wb[M + 1];
                    int o[M + 1];
                    load_records(n, e.y, min(kSmpPart, e.z), td, wv);
                    wb[M] = lane < K ? __ldg(wo + lane) : 0.f;
#pragma unroll
                    for (int u = 0; u < M; ++u) {
                        wb[u] = wv[u];
                        o[u] = ring_offset(td[u], i, smask, sh.NP, spare);
                    }
                    o[M] = lane < K ? yo + lane : spare;
                    add_words(wb, o, ring_lo, ring_hi);
                    for (int k = lane + 32; k < sh.KR * 32; k += 32) {
                        float w1[1] = {k < K ? __ldg(wo + k) : 0.f};
                        int o1[1] = {yo + k};
                        add_words(w1, o1, ring_lo, ring_hi);
                    }
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
            // A step's events pass six stages, one per step of the loop, so
            // every load is consumed a step after its issue: list bounds
            // (step i + 6), channel (i + 5), row bounds (i + 4), bits and row
            // list (i + 3), records (i + 2), ring (i + 1).  Thread e has event
            // e; events beyond the threads are delivered in the fourth stage.
            const int xt = tid - NW * 32, xw = warp - NW;
            const int XT = sh.KI * 32;
            constexpr int kPI = 2, kPM = kSmpPart / 32;          // items and records per lane held in registers
            const long long *xp = n.x_ptr + (long long)b * T;
            const int nch = (n.segs * kSeg + kSmpPart - 1) / kSmpPart;
            // an input spike of step t: bit and list entry; false if the
            // channel was already seen in this step
            auto take = [&](int t, int id) -> bool {
                const uint32_t m = 1u << (id & 31);
                if (atomicOr(&xbit[(t & 1) * sh.in_words + (id >> 5)], m) & m) return false;
                const int r = ck.r_base + t;
                atomicOr(n.bits + ((long long)b * n.n_src + id) * n.RW + ((r & rmask) >> 5), 1u << (r & 31));
                if (lists) {
                    const int bk = (id >> 8) & (kBkt - 1);
                    const int pos = atomicAdd(&bcnt_s[t & 7][bk], 1);
                    n.list_ids[(list_index(n, b, r % n.RS) + bk) * n.list_cap + pos] = id;
                }
                return true;
            };
            auto in_range = [&](int t) { return t >= i0 && t <= i_last; };
            long long q0 = 0, q1 = 0;                            // list bounds (stage 1)
            int id4 = -1, id3 = -1, id2 = -1;                    // channels of the later stages
            long long rb = 0, re = 0;                            // row bounds of id3
            int cnt1[kPI] = {0, 0};                              // records held (stage 5)
            uint32_t td[kPI][kPM];
            float wv[kPI][kPM];
            auto pipeline = [&](int i) {
                // step i + 1: ring
                if (in_range(i + 1)) {
                    const int t = i + 1, m = min(xn_s[t & 7], XT);
#pragma unroll
                    for (int p = 0; p < kPI; ++p)
                        if (cnt1[p] > 0) add_records(td[p], wv[p], t, smask, sh.NP, spare, ring_lo, ring_hi);
                    // what the registers do not hold
                    for (int ev_i = xw; ev_i < m; ev_i += sh.KI) {
                        const int4 e = xrow[(t & 3) * XT + ev_i];
                        const int held = nch == 1 ? (ev_i < kPI * sh.KI ? 1 : 0) : (ev_i < sh.KI ? kPI : 0);
                        for (int c0 = held * kSmpPart; c0 < e.z; c0 += kSmpPart)
                            deliver(e.y + c0, min(kSmpPart, e.z - c0), t);
                    }
                }
                // step i + 2: records: on short rows (one part) two events per
                // warp, else two parts of one; the step's bits of the channel set
#pragma unroll
                for (int p = 0; p < kPI; ++p) cnt1[p] = 0;
                if (in_range(i + 2)) {
                    const int t = i + 2, m = xn_s[t & 7], mc = min(m, XT);
#pragma unroll
                    for (int p = 0; p < kPI; ++p) {
                        const int ev_i = nch == 1 ? xw + p * sh.KI : xw;
                        if (ev_i >= mc) continue;
                        const int4 e = xrow[(t & 3) * XT + ev_i];
                        const int c0 = nch == 1 ? 0 : p * kSmpPart;
                        cnt1[p] = min(kSmpPart, e.z - c0);
                        if (cnt1[p] > 0) load_records(n, e.y + c0, cnt1[p], td[p], wv[p]);
                    }
                    if (id2 >= 0) xbit[(t & 1) * sh.in_words + (id2 >> 5)] = 0u;
                    for (int e = XT + xt; e < m; e += XT)
                        xbit[(t & 1) * sh.in_words + (n.x_ids[xq_s[t & 7] + e] >> 5)] = 0u;
                }
                // step i + 3: bits, spike list, row list (warps without events of
                // their own skip these stages: a step has few)
                if (in_range(i + 3)) {
                    const int t = i + 3, m = xn_s[t & 7];
                    if (id3 >= 0) {
                        const int len_r = take(t, id3) ? (int)(re - rb) : 0;
                        ev += (unsigned long long)len_r;
                        xrow[(t & 3) * XT + xt] = make_int4(id3, (int)rb, len_r, 0);
                    }
                    for (int e = XT + xw; e < m; e += sh.KI) {
                        const int id = n.x_ids[xq_s[t & 7] + e];
                        int ok = 0;
                        if (lane == 0) ok = take(t, id) ? 1 : 0;
                        if (!__shfl_sync(0xffffffffu, ok, 0)) continue;
                        const int b0 = (int)n.row_ptr[id], b1 = (int)n.row_ptr[id + 1];
                        if (lane == 0) ev += (unsigned long long)(b1 - b0);
                        for (int c = b0; c < b1; c += kSmpPart) deliver(c, min(kSmpPart, b1 - c), t);
                    }
                }
                id2 = id3;
                // step i + 4: row bounds
                id3 = id4;
                if (id3 >= 0) {
                    rb = __ldg(n.row_ptr + id3);
                    re = __ldg(n.row_ptr + id3 + 1);
                }
                // step i + 5: channel
                id4 = -1;
                if (in_range(i + 5)) {
                    const int t = i + 5, m = (int)(q1 - q0);
                    if (xt == 0) {
                        xn_s[t & 7] = m;
                        xq_s[t & 7] = q0;
                    }
                    if (xt < m) id4 = __ldg(n.x_ids + q0 + xt);
                }
                // step i + 6: list bounds
                if (in_range(i + 6)) {
                    q0 = __ldg(xp + i + 5);
                    q1 = __ldg(xp + i + 6);
                }
            };
            for (int i = i0 - 6; i < i0; ++i) {          // fill the pipeline
                pipeline(i);
                bar_sync(2, XT);
            }
            __syncthreads();
            for (int i = i0; i <= i_last; ++i) {
                pipeline(i);
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
            auto finish = [&](int i) {           // readout of step i (its input is complete)
                const float tgt_n = load_tgt(i + 1);
                const int win_n = load_win(i + 1);
                long long acc = 0;
                if (has_k) {
                    const int o = y0 + (i & 1) * sh.KR * 32 + k;
                    acc = (long long)(((unsigned long long)ring_hi[o] << 32) | ring_lo[o]);
                    ring_lo[o] = 0u;
                    ring_hi[o] = 0u;
                }
                if (has_k) {
                    y = readout_step(n, y, acc);
                    n.y_rec[((long long)b * T + (i - 1)) * K + k] = y;
                }
                // outside the learning window E and the loss are zero times
                // values that are finite while y, the target and their
                // differences are (a target of NaN where the window is closed
                // gives NaN, as in the per-step kernels)
                float E = 0.f;
                constexpr float kBig = 8.5e37f;      // below 2^126
                bool zero = win == 0 && fabsf(y) < kBig && fabsf(tgt) < kBig;
                zero = __all_sync(0xffffffffu, zero);
                if (sh.KR > 1) {
                    bar_sync(3, RT);
                    if (lane == 0) red_s[rw] = zero ? 0.f : 1.f;
                    bar_sync(3, RT);
                    for (int q = 0; q < sh.KR; ++q) zero = zero && red_s[q] == 0.f;
                }
                if (!zero) {
                    const float l = error_signal(n, y, tgt, (float)win, has_k, E, [&](float x) { return reduce(x, true); },
                                                 [&](float x) { return reduce(x, false); });
                    const float tot = reduce(l, false);
                    if (k == 0) loss += tot;
                }
                if (has_k) n.E_win[((long long)b * U + (i - i0)) * K + k] = E;
                if (lists && rw == 0) {          // the step's list is complete as well
                    n.list_cnt[list_index(n, b, (ck.r_base + i) % n.RS) + lane] = bcnt_s[i & 7][lane];
                    bcnt_s[i & 7][lane] = 0;
                }
                tgt = tgt_n;
                win = win_n;
            };
            __syncthreads();
            int next = (i0 + 1) % 3;             // list slot of step i + 1
            for (int i = i0; i <= i_last; ++i) {
                if (k == 0) cnt_s[next] = 0;
                if (i > i0) finish(i - 1);
                next = next == 2 ? 0 : next + 1;
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

// One thread per neuron (at most four), row starts in 32 bits, and events that
// one SM adds faster than a step's launches take.  The last is a matter of the
// recurrent synapses (a step of a strongly active network touches some percent
// of them); measured per call, this loop against the per-step kernels, all-to-
// all networks at 9e2 / 4e3 / 1e4 / 3.4e4 events per step: 100 neurons x 300 steps
// 0.35 / 3.8 ms, 400 1.2 / 4.1, 700 (4.9e5 synapses) 2.1 / 4.5, 1024 (1.05e6) 5.8 /
// 4.7.  With 10 % recurrent and 2312 inputs (100 steps): 600 neurons 0.77 / 1.5 (one
// sample), 850 neurons (2e6 synapses) x 64 samples 1.2 / 2.5.  The batch does not
// matter: one block per SM takes samples in waves, and 65 to 2047 samples of 40 to
// 1000 neurons are 4.6 to 12 times faster than in per-step launches (100 neurons, 288
// inputs, 100 steps, 512 samples 0.92 / 8.5).  Nor does the window: of one step
// (200 steps) 17.9 / 18.7 at 1000 neurons, 13.0 / 14.0 at 64.
bool sample_net_small(const Net &n) {
    return n.n_rec <= kSmpMaxRec && n.n_in <= kSmpMaxIn && n.n_out <= kSmpMaxOut && n.nnz <= kSmpMaxNnz &&
           n.nnz - n.nnz_in <= kSmpMaxNnzRec;
}
bool sample_steps_fit(const Net &n) {
    return sample_net_small(n) && n.pred_mode == 0 && n.d_out == 0 && !n.band && !(n.has_state && !n.dense);
}

#define EPROP_SMP_EACH(X) \
    X(true, 1, 512) X(true, 2, 512) X(true, 4, 512) X(true, 1, 768) X(true, 1, 1024) \
    X(false, 1, 512) X(false, 2, 512) X(false, 4, 512) X(false, 1, 768) X(false, 1, 1024)

cudaError_t launch_sample_steps(const Net &n, int i0, int i1, cudaStream_t st) {
    const SampleShape s = sample_shape(n.n_in, n.n_rec, n.n_out, n.D);
    const size_t sm = sample_smem(s);
    const int nt = s.threads - (s.KR + s.KI) * 32;
    const int npt = n.n_rec <= nt ? 1 : n.n_rec <= 2 * nt ? 2 : 4;
    // the plain instance has none of the variants, the drive, teacher forcing
    // or the recordings in its loop
    const bool var = n.surrogate || n.reset_mode || n.if_period || n.R_win || n.n_thr || n.forced || n.record_psi ||
                     n.record_raster;
    const int lists = n.B == 1 && n.RS > n.U;   // forms whose window kernels walk the spike lists
#define EPROP_SMP(V, P, BT)                            \
    if (var == V && npt == P && s.threads == BT) {     \
        sample_steps_kernel<V, P, BT><<<n.B, BT, sm, st>>>(n, i0, i1, lists); \
        return cudaSuccess;                            \
    }
    EPROP_SMP_EACH(EPROP_SMP)
#undef EPROP_SMP
    return cudaErrorInvalidConfiguration;        // a shape without an instance
}

void prepare_sample_attributes() {
#define EPROP_SMP(V, P, BT) \
    cudaFuncSetAttribute(sample_steps_kernel<V, P, BT>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
    EPROP_SMP_EACH(EPROP_SMP)
#undef EPROP_SMP
}

}  // namespace eprop
