// Host symbolic analysis of the bus graph, shared by every scenario of a network.
#pragma once

#include <string>
#include <vector>

struct Symbolic {
    int n = 0;                         // buses
    std::vector<int> perm, iperm;      // new -> old, old -> new
    std::vector<int> Lcolptr, Lrow, Lcol;
    std::vector<int> Lrowptr, Lrowcol, Lrowblk;
    int nlevels = 0;
    std::vector<int> lev_ptr, lev_col;
    std::vector<int> tgt_ptr, tgt;
    std::vector<int> upd_ptr, upd_a, upd_b;
    std::vector<int> blk_br_ptr, blk_br;
    std::vector<int> adj_ptr, adj_col, adj_blk;   // per row: its blocks that hold a branch
    // the update lists of each level dealt out to groups of threads (see level_shares)
    std::vector<int> rn_ptr, rn_first, rn_end, sh_a, sh_b, off_ptr, off;
    long long block_updates = 0;       // sum over targets of update pairs
};

// Minimum-degree elimination of the graph (n nodes, undirected edges f[k]-t[k],
// parallel edges allowed, self loops rejected) with node `last` (the reference
// bus, -1 for none) held back to the end, symbolic block factorisation,
// elimination-tree levels and left-looking update lists.  Returns an empty
// string on success, an error message otherwise.
std::string symbolic_analysis(int n, const std::vector<int>& f, const std::vector<int>& t, int last,
                              Symbolic& S);

// Deals the block updates of each level out to `groups` groups of threads in equal shares: the
// update lists of the level's targets, one after another, cut into as many contiguous shares.  A
// level with one column gives its diagonal target to groups 0 and 1 (half of its list each) and
// the others to the rest, cutting a target's list where a share ends; a level with several columns
// cuts between targets only.  Group q of level h takes the runs rn_ptr[h * groups + q] ..
// rn_ptr[h * groups + q + 1] - 1; run i sums the updates rn_first[i] .. rn_first[i + 1] - 1
// (blocks sh_a, sh_b) of one target, and rn_end[i] says what becomes of the sum: a target id, which
// takes it, or -1 - slot: the target's list is cut between groups, the sum goes to that slot (at
// most 2 * groups per level).  The off-diagonal blocks of level h, off_ptr[h] .. off_ptr[h + 1] - 1,
// have four entries each in off: the block, its column, the first slot and the number of slots
// (0: its list is not cut).
void level_shares(int groups, Symbolic& S);
