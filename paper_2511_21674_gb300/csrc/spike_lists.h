// Length of the per-step spike-list ring.  Plain integer function, shared with
// host code.
#pragma once

namespace eprop {

// Steps the ring holds.  Window kernels that walk the lists need those of the
// window and of the delays before it (walked).  The batched single-window
// gradient reads the spike bits: two slots do, and d_out + 2 where the readout
// reads the list of d_out steps back.  But a ring longer than the window also
// lets the readout run beside the delivery and the next neuron updates; one
// sample with a readout delay, which runs step by step at any size, has that as
// long as the ring stays below 1 GB (300 steps of 200 neurons and 800 inputs 3.74
// ms without, 2.19 with).
inline int spike_list_slots(int window, int max_delay, int d_out, bool walked, int batch, long long slot_bytes) {
    const bool trailing = batch == 1 && d_out > 0 && (window + max_delay + 1LL) * slot_bytes <= (1LL << 30);
    const int slots = walked || trailing ? window + max_delay + 1 : 2;
    return slots > d_out + 2 ? slots : d_out + 2;
}

}  // namespace eprop
