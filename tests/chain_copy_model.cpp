// A model of the barriers that csrc/chain_copy.cuh works with: which copies are in flight, what has been handed back, and a
// wait that gives up.  Reads "images cs rank fail_at, n_ops, then kind units groups group_cols tile_cols co n_chunks" from
// the command line and prints "ok <copies> <waits>", or what went wrong.
#include <cstdio>
#include <cstdlib>
#include <string>
#include <vector>

#include "chain_copy.cuh"

using namespace tfjsb;

struct Op {
    int block, units, groups, group_cols, tile_cols, Co, n_chunks, group_tiles, chunk_floats;
};

static void wrong(const std::string& what) {
    std::printf("%s\n", what.c_str());
    std::exit(0);
}

struct Port {
    int rank, fail_at;
    int waits = 0, meets = 0, copies = 0, gave_up = 0;
    int armed[CHAIN_BARS] = {};     // phases of a "full" barrier that were armed
    int drained[CHAIN_BARS] = {};   // and waited for by the copying warp itself
    int back[CHAIN_BARS] = {};      // phases of an "empty" barrier that a wait has seen complete
    std::vector<long long> chunks;  // first float of every chunk, in order

    bool converged = true;  // a wait and a copy by one thread leave the warp's threads apart

    bool wants(const Op& o) const { return o.block && rank < o.units; }
    int group(const Op& o, int u) const { return u % o.groups; }
    bool wait(int bar, unsigned parity) {
        converged = false;
        if (waits++ == fail_at) {
            gave_up = 1;
            return false;
        }
        const bool full = bar == CHAIN_FULL0 || bar == CHAIN_FULL1 || bar == CHAIN_F_FULL;
        int& seen = full ? drained[bar] : back[bar];
        if (full) seen = armed[bar];  // copies land in order of phases: the last one's parity says all have
        else ++seen;
        if (seen == 0 || (unsigned)((seen - 1) & 1) != parity) wrong("a wait for the wrong phase");
        return true;
    }
    void arm(int full, int empty) {
        if (gave_up) wrong("a copy after a wait that gave up");
        // one phase at a time: before phase n is armed, phase n - 1 has been handed back
        if (armed[full] != back[empty]) wrong("a buffer that was not handed back");
        converged = false;
        ++armed[full];
        ++copies;
    }
    void copy_filter(const Op&) { arm(CHAIN_F_FULL, CHAIN_F_EMPTY); }
    void copy_chunk(const Op&, long long from, int buf) {
        arm(CHAIN_FULL0 + buf, CHAIN_EMPTY0 + buf);
        chunks.push_back(from);
    }
    void converge() { converged = true; }
    void meet() {
        if (!converged) wrong("a cluster barrier by a warp that has not converged");
        ++meets;
    }
};

int main(int argc, char** argv) {
    std::vector<int> v;
    for (int i = 1; i < argc; ++i) v.push_back(std::atoi(argv[i]));
    const int images = v[0], cs = v[1], rank = v[2], fail_at = v[3], n_ops = v[4];
    std::vector<Op> ops;
    for (int i = 0; i < n_ops; ++i) {
        const int* p = &v[5 + 7 * i];
        ops.push_back({p[0], p[1], p[2], p[3], p[4], p[5], p[6], p[3] / p[4], 64});
    }
    Port port{rank, fail_at};
    chain_copy_filters(ops.data(), n_ops, rank, cs, images, port);
    if (port.meets != (cs > 1 ? images * n_ops : 0)) wrong("cluster barriers left out");
    const int fulls[] = {CHAIN_FULL0, CHAIN_FULL1, CHAIN_F_FULL};
    for (int bar : fulls)  // the wait that gives up may be one of the last, for a copy that does not land
        if (port.drained[bar] != port.armed[bar] && port.waits - 1 - port.fail_at > 2) wrong("a copy in flight at the end");
    if (fail_at < 0) {
        std::vector<long long> want;
        for (int img = 0; img < images; ++img)
            for (const Op& o : ops)
                for (int u = rank; o.block && u < o.units; u += cs) {
                    const int group = u % o.groups;
                    int tiles = 0;
                    for (int c = group * o.group_cols; c < o.Co && c < (group + 1) * o.group_cols; c += o.tile_cols) ++tiles;
                    for (int k = 0; k < tiles * o.n_chunks; ++k)
                        want.push_back(((long long)group * o.group_tiles * o.n_chunks + k) * o.chunk_floats);
                }
        if (want != port.chunks) wrong("other chunks than the computing warps read");
    }
    std::printf("ok %d %d\n", port.copies, port.waits);
}
