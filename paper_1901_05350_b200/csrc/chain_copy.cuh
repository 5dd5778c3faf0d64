// The order in which the copying warp of chain_cluster.cu fetches filters and takes part in the cluster's barriers.  No
// CUDA in here: the kernel runs it with barriers and bulk copies, a test runs it on the host with a model of both.
#pragma once

#ifdef __CUDACC__
#define TFJSB_CHAIN_FN __device__ __forceinline__
#else
#define TFJSB_CHAIN_FN inline
#endif

namespace tfjsb {

// The barriers of a block's filters: a chunk of the pointwise filter is in one of two buffers, the depthwise filter in one.
enum ChainBar { CHAIN_FULL0, CHAIN_FULL1, CHAIN_EMPTY0, CHAIN_EMPTY1, CHAIN_F_FULL, CHAIN_F_EMPTY, CHAIN_BARS };

template <class Op>
TFJSB_CHAIN_FN int chain_chunks(const Op& o, int group) {
    const int left = o.Co - group * o.group_cols;
    int cols = left < o.group_cols ? left : o.group_cols, n = 0;
    for (; cols > 0; cols -= o.tile_cols) ++n;
    return n * o.n_chunks;
}

// The cluster's barriers up to the one that ends layer `upto` - 1.
template <class Port>
TFJSB_CHAIN_FN void chain_meet(Port& port, int cs, int& met, int upto) {
    if (cs == 1 || met >= upto) return;
    port.converge();
    for (; met < upto; ++met) port.meet();
}

// Every chunk this block will need, in order, two ahead.  The warp takes part in the cluster's barriers, but no later than
// its next wait needs: a chunk of the next layer is on its way before the barrier.
//   port.wants(op)            whether this block has a unit of the operation
//   port.group(op, u)         the column group of unit u
//   port.wait(bar, parity)    false when the wait gave up
//   port.copy_filter(op), port.copy_chunk(op, first float of its filter, buffer)    arm the barrier and copy
//   port.converge()           the warp's threads together again, after a wait or a copy
//   port.meet()               one cluster barrier, by a converged warp
// After a wait that gave up nothing more is copied: the buffer was not handed back, and its barrier may be armed already.
// What is in flight is waited for, once more bounded, and the barriers that the cluster counts on are still taken part in.
template <class Op, class Port>
TFJSB_CHAIN_FN void chain_copy_filters(const Op* ops, int n_ops, int rank, int cs, int images, Port& port) {
    int chunk = 0, met = 0, before = 0, last = 0;  // chunks so far, barriers taken part in, layers of the two chunks before
    int filters = 0, f_before = 0;                 // depthwise filters so far, layer of the last
    bool going = true;
    for (int img = 0; going && img < images; ++img)
        for (int i = 0; going && i < n_ops; ++i) {
            const Op& o = ops[i];
            if (!port.wants(o)) continue;
            if (filters) {
                chain_meet(port, cs, met, f_before);
                if (!(going = port.wait(CHAIN_F_EMPTY, (filters - 1) & 1))) break;
            }
            f_before = img * n_ops + i;
            ++filters;
            port.copy_filter(o);
            for (int u = rank; going && u < o.units; u += cs) {
                const int group = port.group(o, u), chunks = chain_chunks(o, group);
                long long from = (long long)group * o.group_tiles * o.n_chunks * o.chunk_floats;
                for (int k = 0; k < chunks; ++k, ++chunk, from += o.chunk_floats) {
                    const int buf = chunk & 1;
                    if (chunk >= 2) {
                        // the buffer's last chunk is of layer `before`: its readers need the barriers up to that layer
                        chain_meet(port, cs, met, before);
                        if (!(going = port.wait(CHAIN_EMPTY0 + buf, ((chunk >> 1) - 1) & 1))) break;
                    }
                    before = last;
                    last = img * n_ops + i;
                    port.copy_chunk(o, from, buf);
                }
            }
        }
    // none of the copies is in flight when the block ends
    for (int c = chunk > 2 ? chunk - 2 : 0; c < chunk; ++c) port.wait(CHAIN_FULL0 + (c & 1), (c >> 1) & 1);
    if (filters) port.wait(CHAIN_F_FULL, (filters - 1) & 1);
    chain_meet(port, cs, met, images * n_ops);
}

}  // namespace tfjsb
