// Commands that each block of the interaction-matrix rows (k_adjoint.cu) writes.  Plain C++, so that the
// arithmetic can be checked on the host.
#pragma once

#ifdef __CUDACC__
#define MCAO_HD __host__ __device__ __forceinline__
#else
#define MCAO_HD inline
#endif

namespace mcao {

struct CmdRange {
    int lo, hi;   // commands [lo, hi)
};

// part z of n_parts of the commands
MCAO_HD CmdRange command_part(int n_cmd, int n_parts, int z) {
    const int len = (n_cmd + n_parts - 1) / n_parts, lo = z * len < n_cmd ? z * len : n_cmd;
    return {lo, lo + len < n_cmd ? lo + len : n_cmd};
}

// A part's share of one DM's band rows, commands [c0, c1).  Both ends stay within the part: a DM that lies
// wholly before or behind it gets an empty range at the part's own end, so that no run of zeros below
// reaches commands that another block writes.
MCAO_HD CmdRange band_in_part(CmdRange part, int c0, int c1) {
    const int lo = c0 < part.lo ? part.lo : c0 > part.hi ? part.hi : c0;
    return {lo, c1 < lo ? lo : c1 > part.hi ? part.hi : c1};
}

// zeros between the bands of two DMs, before the first (no DM before) and after the last (none behind)
MCAO_HD CmdRange zeros_between(CmdRange part, const CmdRange* before, const CmdRange* behind) {
    return {before ? before->hi : part.lo, behind ? behind->lo : part.hi};
}

}  // namespace mcao
