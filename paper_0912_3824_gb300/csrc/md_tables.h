// md_tables.h -- host-side chunk tables of the run kernel.
//
// Plain C++ over CUDA's int4 (x = first particle, y = end, z = replica,
// w = chunk index): no device code, so the tables can be checked on the CPU
// (tests/tables_unit.cpp).
#ifndef MD_GB300_TABLES_H
#define MD_GB300_TABLES_H

#include <vector_types.h>

#include <cstdint>
#include <vector>

namespace mdt {

inline int4 mk4(int x, int y, int z, int w)
{
    int4 v;
    v.x = x;
    v.y = y;
    v.z = z;
    v.w = w;
    return v;
}

// Order of the run kernel's chunks over its groups of threads, where there is a
// group for every chunk.  Group p works on SM p mod nsm (block p mod nsm of one
// block per SM), so groups p, p + nsm, p + 2 nsm, ... share an SM; giving them
// consecutive chunks (neighbouring cells along the cell curve) lets one SM's groups
// share the neighbour positions they gather in its L1.  With more chunks than
// `resident` groups the chunk order is kept (step_table then shares them out).
// Row p carries its chunk index in w, where its partial sums go with several
// replicas, so the per-replica sums keep their order.
inline std::vector<int4> sm_block_order(const std::vector<int4> &chunks, int nsm, int resident)
{
    const int nb = (int)chunks.size();
    std::vector<int4> out(chunks);
    for (int c = 0; c < nb; ++c)
        out[c].w = c;
    if (nsm <= 1 || nb <= nsm || nb > resident)
        return out;
    int c = 0;
    for (int s = 0; s < nsm; ++s)
        for (int p = s; p < nb; p += nsm, ++c) {
            out[p] = chunks[c];
            out[p].w = c;
        }
    return out;
}

// Rows of the run kernel's table (KArgs::blk_r), cpb per group.  With a group for
// every chunk (`sweep` false) they are the rows of sm_block_order.  With more chunks
// than groups (nsm * per_sm) the groups that share an SM (s, s + nsm, s + 2 nsm,
// ...) get one run of consecutive chunks along the cell curve and take neighbouring
// chunks of it side by side (group s + k nsm: chunks base_s + k, base_s + k +
// per_sm, ...), so that at any time they work on one compact region and share
// the neighbour positions they gather in the SM's L1.  Each row carries its chunk
// index in w; a group's rows end in padding (w = -1).  Returns the rows; nblk_s is
// the number of groups with chunks.
inline std::vector<int4> step_table(const std::vector<int4> &order, const std::vector<int4> &chunks, bool sweep,
                                    int nsm, int per_sm, int &nblk_s, int &cpb)
{
    const int nb = (int)chunks.size();
    if (!sweep || nsm < 1 || per_sm < 1) {
        nblk_s = nb;
        cpb = 1;
        return order;
    }
    if ((int64_t)nsm * per_sm > nb) {           // fewer chunks than groups: at most nb groups
        if (nb < nsm) {
            nsm = nb;
            per_sm = 1;
        } else {
            per_sm = nb / nsm;
        }
    }
    const int resident = nsm * per_sm;           // <= nb, so the rows (< nb + resident) fit 2 nb
    nblk_s = resident;
    cpb = (nb + resident - 1) / resident;
    std::vector<int4> rows((size_t)resident * cpb, mk4(0, 0, 0, -1));
    int base = 0;
    for (int s = 0; s < nsm; ++s) {
        const int ns = nb / nsm + (s < nb % nsm ? 1 : 0);   // chunks of SM s
        for (int k = 0; k < per_sm; ++k) {
            const int b = s + k * nsm;
            for (int q = 0; q < cpb; ++q) {
                const int c = q * per_sm + k;
                if (c >= ns)
                    break;
                rows[(size_t)b * cpb + q] = chunks[base + c];
                rows[(size_t)b * cpb + q].w = base + c;
            }
        }
        base += ns;
    }
    return rows;
}

}  // namespace mdt

#endif  // MD_GB300_TABLES_H
