// What a captured host-free step depends on: everything that a caller can change and that the launches of
// enqueue_host_free_layers carry in their arguments or geometry. A replay is right only where all of it is the same.
#pragma once

namespace spm {

struct HostFreeKey {
    int slot, nb;                        // trace mailboxes, sequences
    const float* h_out;
    bool predict;
    int grid, batched_path;              // CTAs of the GEMV, spm_set_batched_path
    unsigned long long wait_limit_ns;    // spm_set_device_wait_limit_us: an argument of every expert kernel
    bool operator==(const HostFreeKey& o) const {
        return slot == o.slot && nb == o.nb && h_out == o.h_out && predict == o.predict && grid == o.grid &&
               batched_path == o.batched_path && wait_limit_ns == o.wait_limit_ns;
    }
};

}  // namespace spm
