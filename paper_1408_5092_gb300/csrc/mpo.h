// Matrix product operators (Eq. 4) built from second-quantised term lists.
#pragma once
#include <array>
#include <atomic>
#include <map>
#include <memory>
#include <mutex>
#include <utility>
#include <vector>

#include "core.h"

namespace mpspt {

struct FOp {      // elementary fermion operator on spin-orbital j = 2p + s
    int j;
    bool dag;
};

struct Term {     // c * op[0] op[1] ... op[n-1] (product order)
    double c;
    int n;
    FOp op[4];
};

using Mat4 = std::array<double, 16>;   // row-major <n|o|n'> on |0>,|a>,|b>,|ab>

struct MpoEntry {
    int a, b;     // state at cut p, state at cut p+1
    int op;       // index into MPO::ops
    double coef;
};

struct MPO {
    int nsite = 0;
    std::vector<int> dim;                    // states per cut, cut = 0..nsite
    std::vector<std::vector<QN>> dq;         // QN change carried by each state
    std::vector<std::vector<MpoEntry>> W;    // per site, sorted by (a, b)
    std::vector<Mat4> ops;                   // local operator table
    // Entry indices of each site by source state (W[p][out_ptr[p][a] ..
    // out_ptr[p][a+1]]) and by target state (in_idx[p][in_ptr[p][b] ..
    // in_ptr[p][b+1]], in increasing a); filled by index().
    std::vector<std::vector<int>> out_ptr, in_ptr, in_idx;
    // The non-zero local elements v = coef <s|o|t> of each site, listed for
    // (state, s) in the entries' order: in_el of the entries into b, row
    // in_at[p][4 b + s] (x = a), and out_el of the entries out of a, row
    // out_at[p][4 a + s] (x = b).  The planners walk these instead of the
    // entries and their operator tables.  A site's lists are made when they are
    // first asked for (by any thread): 16 bytes an element and direction, 107 MB
    // and 130 ms for the full Hamiltonian of 8e/8o + 24, of which E3 reads one
    // direction and a local operator some sites.
    struct El {
        int x, t;
        double v;
    };
    class Lists {
      public:
        struct Site {                    // where the entries and their index are
            const MpoEntry* entry;
            const int *ptr, *idx;        // idx null: ptr numbers the entries themselves
            const Mat4* ops;
            int states;
        };
        explicit Lists(std::vector<Site> s) : src(std::move(s)), made(new Made[src.size()]) {}
        const std::vector<El>& el(int p) const { return get(p).el; }
        const std::vector<int>& at(int p) const { return get(p).at; }
        bool has(int p) const { return made[p].done.load(); }

      private:
        struct Made {
            std::once_flag once;
            std::atomic<bool> done{false};
            std::vector<El> el;
            std::vector<int> at;
        };
        const Made& get(int p) const;
        std::vector<Site> src;
        std::unique_ptr<Made[]> made;
    };
    struct ElTable {
        std::shared_ptr<const Lists> l;
        const std::vector<El>& operator[](int p) const { return l->el(p); }
    };
    struct AtTable {
        std::shared_ptr<const Lists> l;
        const std::vector<int>& operator[](int p) const { return l->at(p); }
    };
    ElTable in_el, out_el;
    AtTable in_at, out_at;
    // (the lists point into the entries and their index, which a move keeps in
    // place and a copy would not)
    MPO() = default;
    MPO(MPO&&) = default;
    MPO& operator=(MPO&&) = default;
    void index();
};

// Builds the MPO of sum(terms) on nsite sites.  Sites >= k_split are the
// "virtual" region (the centre rule differs there, see mpo.cpp).
MPO build_mpo(const std::vector<Term>& terms, int nsite, int k_split);

// Transfer of MPO states across a run of sites [s0, s1) on which bra and ket
// are both empty (identity sites, local state |0>): only the <0|o|0>
// element of each site operator acts, so the run is a sparse linear map of
// the MPO states at cut s0 to those at cut s1 (a state that needs a creator
// or annihilator on the run dies; the rest pass with their coefficients).
// CSR over the target states: sources of b are col[ptr[b] .. ptr[b+1]).
struct RunMap {
    std::vector<int> ptr, col;
    std::vector<double> val;
};

// Run maps of one MPO, computed on first use and shared by threads.
class RunMaps {
  public:
    explicit RunMaps(const MPO& W);
    const RunMap& get(int s0, int s1);

  private:
    const MPO& W;
    std::vector<std::vector<std::vector<std::pair<int, double>>>> out;   // site, a -> (b, coef <0|o|0>)
    std::mutex mu;
    std::map<std::pair<int, int>, std::unique_ptr<RunMap>> maps;
};

// Term generators (orbital index = site index).
void add_one_body(std::vector<Term>& out, const std::vector<double>& t, int k,
                  int p0, int p1, int q0, int q1);
// 1/2 sum (pq|rs) c+_ps c+_rt c_st c_qs over p in [p0,p1), q in [q0,q1),
// r in [p0,p1), s in [q0,q1), optionally keeping only quadruples with
// p >= vmin or r >= vmin.
void add_two_body(std::vector<Term>& out, const std::vector<double>& eri, int k,
                  int p0, int p1, int q0, int q1, int vmin);
void add_number(std::vector<Term>& out, const std::vector<double>& eps, int a0, int a1);

}  // namespace mpspt
