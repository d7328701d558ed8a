// kn_tables.cu -- a network's host-side set-up and its device tables:
// validation, the sorted and bank-aware reaction order, the reactant table,
// and the sliced gather list with its bank-aware term order and self-check.
#include <algorithm>
#include <array>
#include <cmath>
#include <cstring>
#include <functional>

#include "kn_host.h"

namespace kn {
namespace {
// Bank-aware order of one slice's terms.  Step k of a slice loads
// V[idx(k, l)] for the warp's 32 lanes l; the load takes one shared-memory
// wavefront when the words lie in distinct banks -- the index mod 32 for
// 4-byte values; 8-byte values take a bank pair (index mod 16), two lanes per
// pair in one step -- or are the same word.  A lane may sum its piece in any
// order, so each step is a maximum matching of lanes to banks (augmenting
// paths, Kuhn's method): lanes that must take a term now to end within the
// slice length come first, then the others by remaining terms; a lane that
// must take a term and is not matched takes one anyway (a conflict), an
// unmatched optional lane reads the zero entry (all such reads are one word).
// Returns the slice length (grows only when a lane could not keep up).
static int schedule_slice(const std::vector<std::vector<uint16_t>>& in, int len, int nbank, int cap, uint16_t zero,
                          std::vector<std::vector<uint16_t>>& out) {
    const int NL = (int)in.size();
    std::vector<std::vector<uint16_t>> rem = in;
    out.assign(NL, {});
    const int zb = zero % nbank;
    for (int k = 0;; ++k) {
        int mx = 0, busy = 0;
        for (auto& r : rem) {
            mx = std::max(mx, (int)r.size());
            busy += !r.empty();
        }
        if (mx == 0) return k;
        const int target = std::max(len, k + mx);
        std::vector<int> order;
        for (int l = 0; l < NL; ++l)
            if (!rem[l].empty()) order.push_back(l);
        std::stable_sort(order.begin(), order.end(), [&](int x, int y) {
            const bool mx_ = (int)rem[x].size() >= target - k, my_ = (int)rem[y].size() >= target - k;
            if (mx_ != my_) return mx_;
            return rem[x].size() > rem[y].size();
        });
        // bank slots: cap each; one slot of the zero bank is kept for padding
        // lanes whenever some lane will pad
        std::vector<int> cap_left(nbank, cap);
        if (busy < NL && cap_left[zb] > 0) cap_left[zb] -= 1;
        std::vector<std::vector<int>> holder(nbank);  // lanes matched to each bank
        std::vector<int> match(NL, -1);
        std::function<bool(int, std::vector<char>&)> augment = [&](int l, std::vector<char>& seen) -> bool {
            for (uint16_t v : rem[l]) {
                const int b = v % nbank;
                if (seen[b]) continue;
                seen[b] = 1;
                if ((int)holder[b].size() < cap_left[b]) {
                    holder[b].push_back(l);
                    match[l] = b;
                    return true;
                }
                for (size_t h = 0; h < holder[b].size(); ++h) {
                    const int o = holder[b][h];
                    if (augment(o, seen)) {  // o moved to another bank
                        holder[b][h] = l;
                        match[l] = b;
                        return true;
                    }
                }
            }
            return false;
        };
        for (int l : order) {
            std::vector<char> seen(nbank, 0);
            augment(l, seen);
        }
        for (int l = 0; l < NL; ++l) {
            uint16_t v = zero;
            if (!rem[l].empty()) {
                int pick = -1;
                if (match[l] >= 0) {
                    for (size_t t = 0; t < rem[l].size(); ++t)
                        if (rem[l][t] % nbank == match[l]) {
                            pick = (int)t;
                            break;
                        }
                } else if ((int)rem[l].size() >= target - k) {
                    pick = 0;  // must keep up: a conflict
                }
                if (pick >= 0) {
                    v = rem[l][pick];
                    rem[l].erase(rem[l].begin() + pick);
                }
            }
            out[l].push_back(v);
        }
    }
}

// The tables of one network for (precision, threads per zone group Q), built
// and checked on the host; `blob` is what goes to the device.
}  // namespace

kn_status build_tables_host(const kn_network* n, int prec, int Q, std::vector<unsigned char>& blob,
                                   Tables& T) {
    const int N = n->N, R = n->R;
    const int zero_idx = R + n->S_r;
    // sorted order: position jn holds caller reaction perm[jn]; reactant slots
    // are numbered in sorted order too
    // reactant-slot partials in planes: partial q of reaction jn at
    // plane_base(q) + jn, plane q holding the reactions with more than q
    // reactants (V = [fluxes R | plane 0: R | plane 1: R - R1 | plane 2: R - R12 | 0])
    const int R1 = n->R1, R12 = n->R12;
    const int plane_base[3] = {R, 2 * R - R1, 3 * R - R1 - R12};
    // rows 0..N-1: F+_i (value index jn, once per product slot naming i);
    // rows N..2N-1: k_i (value index R + reactant slot id naming i)
    std::vector<std::vector<uint16_t>> rows(2 * N);
    for (int jn = 0; jn < R; ++jn) {
        const int j = n->perm[jn];
        for (int q = 0; q < 3; ++q) {
            const int p = n->prod[j * 3 + q];
            if (p >= 0) rows[p].push_back((uint16_t)jn);
        }
        for (int q = 0; q < n->nr[j]; ++q) rows[N + n->reac[j * 3 + q]].push_back((uint16_t)(plane_base[q] + jn));
    }
    for (int r = 0; r < 2 * N; ++r)
        if (rows[r].empty()) rows[r].push_back((uint16_t)zero_idx);  // row written as 0
    const int real_bytes = prec == kPrecFP64 ? 8 : 4;
    const int fspan = fk_span(N, real_bytes);
    const int G = Q, W = G / 32;
    const int spare = fspan;  // padding lanes store here
    // Fk holds (F+_i, k_i) pairs: row r < N (F+) at slot 2r, row N + i (k) at 2i + 1
    auto slot_of = [N](int r) { return r < N ? 2 * r : 2 * (r - N) + 1; };
    auto row_of = [N](int slot) { return slot % 2 ? N + slot / 2 : slot / 2; };
    if ((spare + 1) * real_bytes > 0xffff) return fail(KN_ERR_INVALID_ARG, "network too large for the gather tables");
    size_t maxlen = 0;
    for (auto& r : rows) maxlen = std::max(maxlen, r.size());
    // One layout for a piece cap L.  A row of more than L terms is cut into
    // k = ceil(len / L) pieces placed in k consecutive lanes of one slice
    // (k <= 32), whose sums a segmented warp reduction combines.  Units
    // (rows) in order of piece length fill slices: a slice opens with the
    // longest remaining unit and takes every later unit that still fits its
    // lanes.  Slices go longest-first to the least-loaded warp; the cost is
    // the longest warp's load, a term counting 1 and the segmented reduction
    // of a slice with split rows kSegCost (its five shuffle rounds take about
    // as many instructions as that many terms).
    struct Piece {
        int row, start, len, dst;
    };
    struct Unit {
        int row, k, plen;
    };
    struct Layout {
        std::vector<std::vector<Piece>> slices;  // 32 pieces each
        std::vector<char> seg;                   // the slice holds a split row
        std::vector<std::vector<int>> warp_slices;
        std::vector<int> slice_len;
        int cost = 1 << 30, warp_len = 0, n_split = 0;
    };
    auto layout_for = [&](int L, Layout& out) -> bool {
        Layout lo;
        std::vector<Unit> units;
        for (int r = 0; r < 2 * N; ++r) {
            const int len = (int)rows[r].size();
            const int k = (len + L - 1) / L;
            if (k > 32) return false;
            units.push_back({r, k, (len + k - 1) / k});
            lo.n_split += k > 1;
        }
        std::stable_sort(units.begin(), units.end(), [](const Unit& x, const Unit& y) { return x.plen > y.plen; });
        std::vector<char> taken(units.size(), 0);
        size_t first = 0;
        for (;;) {
            while (first < units.size() && taken[first]) ++first;
            if (first == units.size()) break;
            std::vector<Piece> sl;
            char seg = 0;
            for (size_t u = first; u < units.size() && sl.size() < 32; ++u) {
                if (taken[u] || (int)sl.size() + units[u].k > 32) continue;
                taken[u] = 1;
                const int r = units[u].row, len = (int)rows[r].size(), k = units[u].k;
                seg |= k > 1;
                for (int q = 0, st = 0; q < k; ++q) {
                    const int pl = len / k + (q < len % k ? 1 : 0);
                    sl.push_back({r, st, pl, slot_of(r) * real_bytes});
                    st += pl;
                }
            }
            while (sl.size() < 32) sl.push_back({-1, 0, 0, spare * real_bytes});
            int sl_len = 0;
            for (auto& pc : sl) sl_len = std::max(sl_len, pc.len);
            lo.slice_len.push_back(sl_len);
            lo.seg.push_back(seg);
            lo.slices.push_back(std::move(sl));
        }
        constexpr int kSegCost = 6;
        const int ns = (int)lo.slices.size();
        std::vector<int> order(ns), cost(ns);
        for (int s = 0; s < ns; ++s) {
            order[s] = s;
            cost[s] = lo.slice_len[s] + (lo.seg[s] ? kSegCost : 0);
        }
        std::stable_sort(order.begin(), order.end(), [&](int x, int y) { return cost[x] > cost[y]; });
        lo.warp_slices.assign(W, {});
        std::vector<int> load(W, 0), terms(W, 0);
        for (int s : order) {
            const int w = (int)(std::min_element(load.begin(), load.end()) - load.begin());
            lo.warp_slices[w].push_back(s);
            load[w] += cost[s];
            terms[w] += lo.slice_len[s];
        }
        lo.warp_len = *std::max_element(terms.begin(), terms.end());
        lo.cost = *std::max_element(load.begin(), load.end());
        out = std::move(lo);
        return true;
    };
    Layout best;
    int L_best = 0;
    for (int L = 1; L <= (int)maxlen; ++L) {
        Layout lo;
        if (!layout_for(L, lo)) continue;
        if (lo.cost < best.cost || (lo.cost == best.cost && lo.n_split < best.n_split)) {
            best = std::move(lo);
            L_best = L;
        }
    }
    if (!L_best) return fail(KN_ERR_INVALID_ARG, "no gather layout fits %d threads per zone", G);
    // flatten: slices in warp order; header (base into sidx, length | split flag << 31)
    std::vector<uint16_t> wsl(W + 1, 0), sdst, sidx;
    // the terms as byte offsets into V when they fit 16 bits (the loads then
    // need no scaling), else as indices
    const bool byte_off = (zero_idx + 1) * real_bytes <= 0x10000;
    const int vscale = byte_off ? real_bytes : 1;
    std::vector<uint32_t> shdr;
    int n_slices = 0;
    T.order.slices.clear();
    for (int w = 0; w < W; ++w) {
        wsl[w] = (uint16_t)n_slices;
        for (int s : best.warp_slices[w]) {
            std::vector<std::vector<uint16_t>> lanes(32), ordered;
            for (int l = 0; l < 32; ++l) {
                const Piece& pc = best.slices[s][l];
                sdst.push_back((uint16_t)pc.dst);
                for (int k = 0; k < pc.len; ++k) lanes[l].push_back(rows[pc.row][pc.start + k]);
            }
            const int len = schedule_slice(lanes, best.slice_len[s], real_bytes == 4 ? 32 : 16,
                                           real_bytes == 4 ? 1 : 2, (uint16_t)zero_idx, ordered);
            shdr.push_back((uint32_t)sidx.size());
            shdr.push_back((uint32_t)len | (best.seg[s] ? 0x80000000u : 0u));
            const size_t base = sidx.size();
            sidx.resize(base + 32 * (size_t)len, (uint16_t)(zero_idx * vscale));
            for (int l = 0; l < 32; ++l)
                for (int k = 0; k < len; ++k) sidx[base + 32 * (size_t)k + l] = (uint16_t)(ordered[l][k] * vscale);
            if (prec == kPrecMixed) {
                GatherOrder::Slice os;
                os.len = len;
                for (int l = 0; l < 32; ++l) os.row.push_back(best.slices[s][l].row);
                for (int k = 0; k < len; ++k)
                    for (int l = 0; l < 32; ++l) os.terms.push_back(ordered[l][k]);
                T.order.slices.push_back(std::move(os));
            }
            ++n_slices;
        }
    }
    wsl[W] = (uint16_t)n_slices;
    // Host check of the tables before they reach a device: every index in
    // range, a split row's pieces in consecutive lanes of a flagged slice, and
    // the gather, run on the host with V[v] = v + 1, giving every row's sum
    // exactly once (integer sums, exact in FP64).
    {
        std::vector<double> got(2 * N, -1.0);
        for (int w = 0; w < W; ++w)
            for (int sl = wsl[w]; sl < wsl[w + 1]; ++sl) {
                const uint32_t base = shdr[2 * sl], len = shdr[2 * sl + 1] & 0x7fffffffu;
                const bool seg = (shdr[2 * sl + 1] >> 31) != 0;
                if (base + 32 * (size_t)len > sidx.size()) return fail(KN_ERR_INTERNAL, "gather table: slice out of range");
                double acc[32];
                for (int l = 0; l < 32; ++l) {
                    acc[l] = 0.0;
                    for (uint32_t k = 0; k < len; ++k) {
                        const int raw = sidx[base + 32 * k + l];
                        if (raw % vscale) return fail(KN_ERR_INTERNAL, "gather table: misaligned value offset");
                        const int v = raw / vscale;
                        if (v > zero_idx) return fail(KN_ERR_INTERNAL, "gather table: value index out of range");
                        acc[l] += v == zero_idx ? 0.0 : (double)v + 1.0;
                    }
                }
                for (int l = 0; l < 32;) {
                    const uint16_t d = sdst[32 * sl + l];
                    int e = l + 1;
                    double sum = acc[l];
                    while (e < 32 && sdst[32 * sl + e] == d) sum += acc[e++];
                    if (d % real_bytes || d / real_bytes > spare) return fail(KN_ERR_INTERNAL, "gather table: bad destination");
                    const int r = d / real_bytes < 2 * N ? row_of(d / real_bytes) : 2 * N;
                    if (r < 2 * N) {
                        if (e - l > 1 && !seg) return fail(KN_ERR_INTERNAL, "gather table: split row in an unflagged slice");
                        if (got[r] >= 0.0) return fail(KN_ERR_INTERNAL, "gather table: row %d stored twice", r);
                        got[r] = sum;
                    }
                    l = e;
                }
            }
        for (int r = 0; r < 2 * N; ++r) {
            double want = 0.0;
            for (uint16_t v : rows[r]) want += v == zero_idx ? 0.0 : (double)v + 1.0;
            if (got[r] != want) return fail(KN_ERR_INTERNAL, "gather table: row %d sums to %g, not %g", r, got[r], want);
        }
    }
    const int real = prec == kPrecFP64 ? 8 : 4;
    const int a_bytes = prec == kPrecMixed ? 4 : 8;  // A is read by the update: FP64 where the update is
    TableLayout tl{};
    int off = 0;
    tl.off_A = off;
    off = pad16(off + a_bytes * N);
    tl.off_rspec = off;
    off = pad16(off + 4 * R);
    tl.off_cexp = off;
    off = pad16(off + real * R);
    tl.off_wsl = off;
    off = pad16(off + 2 * (W + 1));
    tl.off_shdr = off;
    off = pad16(off + 4 * (int)shdr.size());
    tl.off_sdst = off;
    off = pad16(off + 2 * (int)sdst.size());
    tl.off_sidx = off;
    off = pad16(off + 2 * (int)sidx.size());
    // the slices dealt to a wide group's warps, longest first: to the scheduler (w mod 4)
    // with the least to do, and there to the warp with the least
    std::vector<uint16_t> deal;
    tl.bytes = tl.off_deal = off;
    if (prec == kPrecFP64) {
        const int D = wide_group(G) / 32;
        std::vector<int> by(n_slices), load(D, 0), sched(4, 0);
        auto cost_of = [&](int s) { return (int)(shdr[2 * s + 1] & 0x7fffffffu) + (shdr[2 * s + 1] >> 31 ? 6 : 0); };
        for (int s = 0; s < n_slices; ++s) by[s] = s;
        std::stable_sort(by.begin(), by.end(), [&](int x, int y) { return cost_of(x) > cost_of(y); });
        std::vector<std::vector<uint16_t>> mine(D);
        for (int s : by) {
            int w = (int)(std::min_element(sched.begin(), sched.end()) - sched.begin());
            for (int v = w; v < D; v += 4)
                if (load[v] < load[w]) w = v;
            mine[w].push_back((uint16_t)s);
            load[w] += cost_of(s);
            sched[w % 4] += cost_of(s);
        }
        deal.push_back(0);
        for (int w = 0; w < D; ++w) deal.push_back((uint16_t)(deal.back() + mine[w].size()));
        for (auto& m : mine) deal.insert(deal.end(), m.begin(), m.end());
        off = pad16(off + 2 * (int)deal.size());
    }
    tl.wide_bytes = off;
    blob.assign(off, 0);
    for (int i = 0; i < N; ++i) {
        if (a_bytes == 8) {
            memcpy(blob.data() + tl.off_A + 8 * i, &n->A[i], 8);
        } else {
            const float af = (float)n->A[i];
            memcpy(blob.data() + tl.off_A + 4 * i, &af, 4);
        }
    }
    for (int jn = 0; jn < R; ++jn) {
        const int j = n->perm[jn];
        const uint32_t ra = (uint32_t)n->reac[j * 3];
        const uint32_t rb = (uint32_t)(n->nr[j] >= 2 ? n->reac[j * 3 + 1] : N);
        const uint32_t rc = (uint32_t)(n->nr[j] >= 3 ? n->reac[j * 3 + 2] : N);
        const uint32_t rs = ra | rb << 10 | rc << 20;
        memcpy(blob.data() + tl.off_rspec + 4 * jn, &rs, 4);
        const double c = n->tn[j] + 3.0 * (n->nr[j] - 1);
        if (prec == kPrecFP64) {
            memcpy(blob.data() + tl.off_cexp + 8 * jn, &c, 8);
        } else {
            const float cf = (float)c;
            memcpy(blob.data() + tl.off_cexp + 4 * jn, &cf, 4);
        }
    }
    memcpy(blob.data() + tl.off_wsl, wsl.data(), 2 * wsl.size());
    memcpy(blob.data() + tl.off_shdr, shdr.data(), 4 * shdr.size());
    memcpy(blob.data() + tl.off_sdst, sdst.data(), 2 * sdst.size());
    memcpy(blob.data() + tl.off_sidx, sidx.data(), 2 * sidx.size());
    if (!deal.empty()) memcpy(blob.data() + tl.off_deal, deal.data(), 2 * deal.size());
    tl.sidx_bytes = byte_off ? 1 : 0;
    T.tl = tl;
    T.L = L_best;
    T.n_slices = n_slices;
    T.warp_len = best.warp_len;
    return KN_OK;
}


SlotLayout slot_layout(const kn_network* n, const SlotTables& st, int T, int NZ, bool qss) {
    const int W = T / 32, Tw = T > 32 ? T - 32 : 32;
    SlotLayout l{};
    int off = 0;
    l.off_V = off;
    off += 128 * NZ * st.vrows;
    l.off_Y = off;
    off += 128 * NZ * ((n->N + 32) / 32);
    l.off_K = off;
    off += 4 * NZ * Tw * st.slots;
    l.off_Fk = off;
    off = pad16(off + 8 * NZ * n->N);
    l.off_Fk2 = off;
    if (qss) off = pad16(off + 8 * NZ * n->N);
    l.off_red = off;
    off += 16 * W * NZ;
    l.off_ctl = off;
    off += kSlotCtlBytes;
    l.bytes = (off + 127) & ~127;  // the next group's interleaved arrays start at bank 0
    return l;
}

namespace {
// Banks for V's values.  A value is stored by one warp instruction (a block's 32
// lanes, one plane) and loaded by one to three (a gather step); each takes one
// wavefront when its distinct words lie in distinct banks.  Simulated annealing
// (Kirkpatrick, Gelatt & Vecchi, Science 220 (1983)) from a greedy start, the
// energy the pairs of values of one instruction in one bank, 400 trials a value: 20
// ms for 150/1604, whose 159 gather loads (and 17 of padding) go from 277 wavefronts,
// values in reaction order, to 217 (3000 trials: about 200).  Without it 1216 zones
// to 3e-11 s take 11.3 ms instead of 10.8, 1000 zones of 365/4400 35.8 instead of
// 33.9 ms.  zero: the instruction also reads the constant 0, which lies in bank 0.
// `rows`: the values that a bank holds at most.
static std::vector<int> place_banks(int nv, const std::vector<std::vector<int>>& groups, const std::vector<char>& zero,
                                    int rows) {
    std::vector<int> off(nv + 1, 0), of;
    for (const auto& g : groups)
        for (int v : g) ++off[v + 1];
    for (int v = 0; v < nv; ++v) off[v + 1] += off[v];
    of.resize(off[nv]);
    {
        std::vector<int> at(off.begin(), off.end() - 1);
        for (int g = 0; g < (int)groups.size(); ++g)
            for (int v : groups[g]) of[at[v]++] = g;
    }
    std::vector<std::array<uint8_t, 32>> cnt(groups.size());
    for (size_t g = 0; g < groups.size(); ++g) {
        cnt[g].fill(0);
        cnt[g][0] = (uint8_t)zero[g];
    }
    std::vector<int> bank(nv, -1), fill(32, 0);
    uint32_t rng = 12345;
    auto rnd = [&]() { return (rng = rng * 1664525u + 1013904223u) >> 8; };
    auto put = [&](int v, int b, int d) {
        fill[b] += d;
        for (int i = off[v]; i < off[v + 1]; ++i) cnt[of[i]][b] = (uint8_t)(cnt[of[i]][b] + d);
    };
    auto pick = [&](int v) {  // the bank with the fewest values of v's instructions
        int best = -1, cost = 1 << 30;
        const int start = (int)(rnd() >> 19);
        for (int k = 0; k < 32; ++k) {
            const int b = (start + k) & 31;
            if (fill[b] >= rows) continue;
            int c = 0;
            for (int i = off[v]; i < off[v + 1]; ++i) c += cnt[of[i]][b];
            if (c < cost) {
                cost = c;
                best = b;
            }
        }
        return best;
    };
    for (int v = 0; v < nv; ++v) {
        bank[v] = pick(v);
        put(v, bank[v], 1);
    }
    const int trials = 400 * nv, rounds = 64;
    for (int r = 0; r < rounds; ++r) {
        const double T = 0.3 * std::pow(0.05 / 0.3, (r + 0.5) / rounds);
        uint32_t lim[4];  // a rise of 1, 2, 3, 4 pairs is accepted below these 24-bit numbers
        for (int d = 0; d < 4; ++d) lim[d] = (uint32_t)(16777216.0 * std::exp(-(d + 1) / T));
        for (int i = 0; i < trials / rounds; ++i) {
            const uint32_t x = rnd();
            const int v = (int)((uint64_t)rnd() * (uint32_t)nv >> 24), b = (int)(x >> 19), o = bank[v];
            if (b == o || fill[b] >= rows) continue;
            int d = 0;
            for (int k = off[v]; k < off[v + 1]; ++k) d += cnt[of[k]][b] - (cnt[of[k]][o] - 1);
            if (d > 4 || (d > 0 && rnd() >= lim[d - 1])) continue;
            put(v, o, -1);
            bank[v] = b;
            put(v, b, 1);
        }
    }
    return bank;
}

// V's rows of 32 words, with room for the banks' search; the last holds the constant 0
static int slot_rows(const kn_network* n) {
    return (n->R + n->S_r + 31) / 32 + 1 + ((n->R + 31) / 32 > 4 ? 8 : 0);
}

// Banks for V's values, from the instructions that store and load them: the blocks of
// 32 reactions and the gather's steps, whichever thread has them, so one search serves
// every group size, number of zones and capacity of a summation order.
static std::vector<int> slot_banks(const kn_network* n, const Tables& tb) {
    const int R = n->R, blocks = (R + 31) / 32, zero_idx = R + n->S_r;
    const int plane[3] = {R, 2 * R - n->R1, 3 * R - n->R1 - n->R12};
    std::vector<std::vector<int>> groups;
    std::vector<char> zero;
    for (int b = 0; b < blocks; ++b)
        for (int q = 0; q < 4; ++q) {
            std::vector<int> g;
            for (int j = 32 * b; j < std::min(R, 32 * b + 32); ++j) {
                const int nr = n->nr[n->perm[j]];
                if (q == 0) g.push_back(j);
                else if (q <= nr && nr > 1) g.push_back(plane[q - 1] + j);  // (1-body partials: only at a refresh)
            }
            if (g.empty()) continue;
            groups.push_back(std::move(g));
            zero.push_back(0);
        }
    for (const auto& sl : tb.order.slices)
        for (int k = 0; k < sl.len; ++k) {
            std::vector<int> g;
            char z = 0;
            for (int l = 0; l < 32; ++l) {
                const int v = sl.terms[32 * (size_t)k + l];
                z |= v == zero_idx;
                if (v != zero_idx && std::find(g.begin(), g.end(), v) == g.end()) g.push_back(v);
            }
            groups.push_back(std::move(g));
            zero.push_back(z);
        }
    return place_banks(zero_idx, groups, zero, slot_rows(n) - 1);
}
}  // namespace

kn_status build_slots_host(const kn_network* n, Tables& tb, int T, int NZ, int cap, std::vector<unsigned char>& blob,
                           SlotTables& st, bool& fits) {
    fits = false;
    st = SlotTables{};
    const SlotCaps C = kSlotCaps[cap];
    const int N = n->N, R = n->R, W = T / 32, Ww = W > 1 ? W - 1 : 1, Tw = 32 * Ww, blocks = (R + 31) / 32,
              zero_idx = R + n->S_r;
    auto word = [NZ](int v) { return v / 32 * 32 * NZ + v % 32; };
    if (word(N) > 0xffff || 8 * NZ * N > 0xffff) return KN_OK;
    // ---- gather slices to workers: at most two each, the longest first to the
    // least loaded (costs in terms: set-up 6, a reduction round 2) ----
    const int ns = (int)tb.order.slices.size();
    std::vector<int> rounds(ns, 0), cost(ns), ord(ns);
    for (int s = 0; s < ns; ++s) {
        const auto& sl = tb.order.slices[s];
        int most = 1;
        for (int l = 0; l < 32;) {
            int e = l + 1;
            while (e < 32 && sl.row[l] >= 0 && sl.row[e] == sl.row[l]) ++e;
            most = std::max(most, e - l);
            l = e;
        }
        while ((1 << rounds[s]) < most) ++rounds[s];
        cost[s] = 6 + sl.len + 2 * rounds[s];
        ord[s] = s;
    }
    std::stable_sort(ord.begin(), ord.end(), [&](int x, int y) { return cost[x] > cost[y]; });
    if (ns > 2 * Ww) return KN_OK;
    std::vector<std::vector<int>> mine(Ww);
    std::vector<int> load(Ww, 0);
    for (int s : ord) {
        int w = -1;
        for (int i = 0; i < Ww; ++i)
            if (mine[i].size() < 2 && (w < 0 || load[i] < load[w])) w = i;
        // the first slice of a warp is its longest; the second has the smaller capacity
        if ((tb.order.slices[s].len + 3) / 4 * 2 > (mine[w].empty() ? C.ga : C.gb)) return KN_OK;
        mine[w].push_back(s);
        load[w] += cost[s];
    }
    // ---- blocks of reactions to workers: whole 1- and 2-body blocks to their own
    // slots, the others (and what overflows) to the slots for any block ----
    struct Bl {
        int b, cls, cost;
    };
    std::vector<Bl> bl;
    for (int b = 0; b < blocks; ++b) {
        const int j0 = 32 * b, j1 = j0 + 31;
        int cls = 3;
        if (j1 < n->R1) cls = 1;
        else if (j0 >= n->R1 && j1 < n->R12) cls = 2;
        bl.push_back({b, cls, cls == 1 ? 8 : (cls == 2 ? 19 : 30)});
    }
    std::stable_sort(bl.begin(), bl.end(), [](const Bl& x, const Bl& y) { return x.cost > y.cost; });
    std::vector<std::vector<int>> k1(Ww), k2(Ww), ka(Ww);
    std::vector<int> fl(Ww, 0);
    for (const Bl& x : bl) {
        int w = -1, to = 0;
        for (int pass = 0; pass < 2 && w < 0; ++pass)  // its own sort of slot, then any
            for (int i = 0; i < Ww; ++i) {
                const int t = pass == 0 ? x.cls : 3;
                const bool room = t == 1 ? (int)k1[i].size() < C.f1 : (t == 2 ? (int)k2[i].size() < C.f2 : (int)ka[i].size() < C.fa);
                if (room && (w < 0 || fl[i] < fl[w])) {
                    w = i;
                    to = t;
                }
            }
        if (w < 0) return KN_OK;
        (to == 1 ? k1 : (to == 2 ? k2 : ka))[w].push_back(x.b);
        fl[w] += to == 3 ? 30 : x.cost;
    }
    // ---- V: the values' places, by their banks (slot_banks) ----
    const int plane[3] = {R, 2 * R - n->R1, 3 * R - n->R1 - n->R12};
    st.vrows = slot_rows(n);
    if (32 * NZ * st.vrows > 0x10000) return KN_OK;
    if (tb.banks.empty()) tb.banks = slot_banks(n, tb);
    const std::vector<int>& bank = tb.banks;
    std::vector<int> at(zero_idx + 1), next(32, 0);
    for (int v = 0; v < zero_idx; ++v) at[v] = 32 * NZ * next[bank[v]]++ + bank[v];
    at[zero_idx] = 32 * NZ * (st.vrows - 1);
    st.zero = at[zero_idx];
    // ---- the words ----
    st.slots = C.f1 + C.f2 + C.fa;
    const int nwords = C.f1 + 3 * C.f2 + 4 * C.fa + C.ga + C.gb + 3;
    std::vector<uint32_t> wd((size_t)nwords * Tw, 0), p0((size_t)C.f1 * Tw, 0);
    std::vector<uint16_t> sj((size_t)st.slots * Tw, 0xffff);
    std::vector<float> ce((size_t)st.slots * Tw, 0.f);
    for (int w = 0; w < Ww; ++w)
        for (int l = 0; l < 32; ++l) {
            const int t = 32 * w + l;
            auto set = [&](int i, uint32_t lo, uint32_t hi) { wd[(size_t)i * Tw + t] = lo | hi << 16; };
            auto fill = [&](int slot, int jn, uint32_t (&a)[8]) {  // a, b, c; V, P0, P1, P2; reactants
                for (int q = 0; q < 8; ++q) a[q] = q < 3 ? (uint32_t)word(N) : 0;
                if (jn >= R) return;
                const int j = n->perm[jn];
                for (int q = 0; q < n->nr[j]; ++q) a[q] = (uint32_t)word(n->reac[j * 3 + q]);
                a[3] = (uint32_t)at[jn];
                for (int q = 0; q < n->nr[j]; ++q) a[4 + q] = (uint32_t)at[plane[q] + jn];
                a[7] = (uint32_t)n->nr[j];
                sj[(size_t)slot * Tw + t] = (uint16_t)jn;
                ce[(size_t)slot * Tw + t] = (float)(n->tn[j] + 3.0 * (n->nr[j] - 1));
            };
            uint32_t a[8];
            int i = 0;
            for (int k = 0; k < C.f1; ++k, ++i)
                if (k < (int)k1[w].size()) {
                    fill(k, 32 * k1[w][k] + l, a);
                    set(i, a[0], a[3]);
                    p0[(size_t)k * Tw + t] = a[4];
                }
            for (int k = 0; k < C.f2; ++k, i += 3)
                if (k < (int)k2[w].size()) {
                    fill(C.f1 + k, 32 * k2[w][k] + l, a);
                    set(i, a[0], a[1]);
                    set(i + 1, a[3], a[4]);
                    set(i + 2, a[5], 0);
                }
            for (int k = 0; k < C.fa; ++k, i += 4)
                if (k < (int)ka[w].size()) {
                    fill(C.f1 + C.f2 + k, 32 * ka[w][k] + l, a);
                    set(i, a[0], a[1]);
                    set(i + 1, a[2], a[3]);
                    set(i + 2, a[4], a[5]);
                    set(i + 3, a[6], a[7]);
                }
            uint32_t cnt = (uint32_t)k1[w].size() | (uint32_t)k2[w].size() << 4 | (uint32_t)ka[w].size() << 8;
            uint32_t dst[2] = {0, 0};
            for (int h = 0; h < 2; ++h) {
                const int room = h ? C.gb : C.ga;
                const bool has = h < (int)mine[w].size();
                if (has) {
                    const auto& sl = tb.order.slices[mine[w][h]];
                    // lengths rounded up to four by the constant 0 (adding +0 changes no
                    // sum of non-negative terms)
                    for (int k = 0; k < room; ++k) {
                        auto term = [&](int q) { return (uint32_t)at[q < sl.len ? sl.terms[32 * (size_t)q + l] : zero_idx]; };
                        set(i + k, term(2 * k), term(2 * k + 1));
                    }
                    const int rd = rounds[mine[w][h]], r = sl.row[l];
                    if (r >= 0) {
                        uint32_t d = (uint32_t)(8 * NZ * (r % N) + (r >= N ? 4 * NZ : 0));
                        if (l == 0 || sl.row[l - 1] != r) d |= 1u << 16;
                        for (int q = 0; q < rd; ++q)
                            if (l + (1 << q) < 32 && sl.row[l + (1 << q)] == r) d |= 1u << (17 + q);
                        dst[h] = d;
                    }
                    cnt |= (uint32_t)((sl.len + 3) / 4 * 2) << (h ? 18 : 12) | (uint32_t)rd << (h ? 28 : 24);
                }
                i += room;
            }
            wd[(size_t)i * Tw + t] = dst[0];
            wd[(size_t)(i + 1) * Tw + t] = dst[1];
            wd[(size_t)(i + 2) * Tw + t] = cnt;
        }
    // ---- host check, through the words: every reaction in one thread's block with
    // its reactants and its places in V, and the gather with V[v] = v + 1 giving
    // every row once ----
    {
        std::vector<double> V((size_t)32 * NZ * st.vrows, -1.0);
        std::vector<char> seen(R, 0);
        const int gaw = C.f1 + 3 * C.f2 + 4 * C.fa;
        for (int t = 0; t < Tw; ++t) {
            const uint32_t cnt = wd[(size_t)(nwords - 1) * Tw + t];
            auto wrd = [&](int i) { return wd[(size_t)i * Tw + t]; };
            for (int sl = 0; sl < st.slots; ++sl) {
                const int jn = sj[(size_t)sl * Tw + t];
                if (jn == 0xffff) continue;
                if (jn >= R || seen[jn]++) return fail(KN_ERR_INTERNAL, "slot tables: reaction %d dealt twice", jn);
                const int j = n->perm[jn], nr = n->nr[j];
                uint32_t y[3] = {(uint32_t)word(N), (uint32_t)word(N), (uint32_t)word(N)}, p[4] = {0, 0, 0, 0};
                int used;
                if (sl < C.f1) {
                    used = 1;
                    y[0] = wrd(sl) & 0xffff;
                    p[0] = wrd(sl) >> 16;
                    p[1] = p0[(size_t)sl * Tw + t];
                    if (sl >= (int)(cnt & 15)) return fail(KN_ERR_INTERNAL, "slot tables: block count");
                } else if (sl < C.f1 + C.f2) {
                    used = 2;
                    const int i = C.f1 + 3 * (sl - C.f1);
                    y[0] = wrd(i) & 0xffff;
                    y[1] = wrd(i) >> 16;
                    p[0] = wrd(i + 1) & 0xffff;
                    p[1] = wrd(i + 1) >> 16;
                    p[2] = wrd(i + 2);
                    if (sl - C.f1 >= (int)(cnt >> 4 & 15)) return fail(KN_ERR_INTERNAL, "slot tables: block count");
                } else {
                    const int i = C.f1 + 3 * C.f2 + 4 * (sl - C.f1 - C.f2);
                    y[0] = wrd(i) & 0xffff;
                    y[1] = wrd(i) >> 16;
                    y[2] = wrd(i + 1) & 0xffff;
                    p[0] = wrd(i + 1) >> 16;
                    p[1] = wrd(i + 2) & 0xffff;
                    p[2] = wrd(i + 2) >> 16;
                    p[3] = wrd(i + 3) & 0xffff;
                    used = (int)(wrd(i + 3) >> 16);
                    if (sl - C.f1 - C.f2 >= (int)(cnt >> 8 & 15)) return fail(KN_ERR_INTERNAL, "slot tables: block count");
                }
                if (used != nr) return fail(KN_ERR_INTERNAL, "slot tables: reactants of reaction %d", jn);
                for (int q = 0; q < 3; ++q)
                    if ((int)y[q] != word(q < nr ? n->reac[j * 3 + q] : N)) return fail(KN_ERR_INTERNAL, "slot tables: reactant");
                for (int q = 0; q <= nr; ++q) {
                    if (p[q] >= V.size() || p[q] % (32 * NZ) >= 32 || V[p[q]] >= 0.0)
                        return fail(KN_ERR_INTERNAL, "slot tables: a value's place");
                    V[p[q]] = (q == 0 ? jn : plane[q - 1] + jn) + 1.0;
                }
            }
        }
        for (int j = 0; j < R; ++j)
            if (!seen[j]) return fail(KN_ERR_INTERNAL, "slot tables: reaction %d not dealt", j);
        if (V[st.zero] >= 0.0) return fail(KN_ERR_INTERNAL, "slot tables: the constant 0's place");
        V[st.zero] = 0.0;
        std::vector<double> got(2 * (size_t)N, -1.0), want(2 * (size_t)N, 0.0);
        for (const auto& sl : tb.order.slices)
            for (int k = 0; k < sl.len; ++k)
                for (int l = 0; l < 32; ++l)
                    if (sl.row[l] >= 0 && sl.terms[32 * (size_t)k + l] != zero_idx)
                        want[sl.row[l]] += sl.terms[32 * (size_t)k + l] + 1.0;
        for (int w = 0; w < Ww; ++w)
            for (int h = 0; h < 2; ++h) {
                double acc[32];
                uint32_t d[32];
                int rd = 0;
                for (int l = 0; l < 32; ++l) {
                    const int t = 32 * w + l;
                    const uint32_t cnt = wd[(size_t)(nwords - 1) * Tw + t];
                    const int words = (int)(cnt >> (h ? 18 : 12) & 63);
                    rd = (int)(h ? cnt >> 28 : cnt >> 24 & 7);
                    d[l] = words ? wd[(size_t)(nwords - 3 + h) * Tw + t] : 0;
                    acc[l] = 0.0;
                    for (int k = 0; k < words; ++k) {
                        const uint32_t x = wd[(size_t)(gaw + (h ? C.ga : 0) + k) * Tw + t];
                        for (uint32_t v : {x & 0xffffu, x >> 16}) {
                            if (v >= V.size() || V[v] < 0.0) return fail(KN_ERR_INTERNAL, "slot tables: term out of range");
                            acc[l] += V[v];
                        }
                    }
                }
                for (int r = 0; r < rd; ++r)
                    for (int l = 0; l < 32; ++l)  // ascending: the lane up still holds the last round's sum
                        if (d[l] >> (17 + r) & 1) acc[l] += acc[l + (1 << r)];
                for (int l = 0; l < 32; ++l) {
                    if (!(d[l] >> 16 & 1)) continue;
                    const int o = (int)(d[l] & 0xffffu), i = o / (8 * NZ), q = o % (8 * NZ);
                    if (i >= N || (q != 0 && q != 4 * NZ)) return fail(KN_ERR_INTERNAL, "slot tables: bad destination");
                    double& x = got[(q ? N : 0) + i];
                    if (x >= 0.0) return fail(KN_ERR_INTERNAL, "slot tables: row stored twice");
                    x = acc[l];
                }
            }
        for (int r = 0; r < 2 * N; ++r)
            if (got[r] != want[r]) return fail(KN_ERR_INTERNAL, "slot tables: row %d sums to %g, not %g", r, got[r], want[r]);
    }
    int off = 4 * (int)ce.size();
    st.off_p0 = off;
    off += 4 * (int)p0.size();
    st.bytes = off = (off + 127) & ~127;
    st.off_words = off;
    off += 4 * (int)wd.size();
    st.off_sj = off;
    off += 2 * (int)sj.size();
    blob.assign(off, 0);
    memcpy(blob.data(), ce.data(), 4 * ce.size());
    memcpy(blob.data() + st.off_p0, p0.data(), 4 * p0.size());
    memcpy(blob.data() + st.off_words, wd.data(), 4 * wd.size());
    memcpy(blob.data() + st.off_sj, sj.data(), 2 * sj.size());
    fits = true;
    return KN_OK;
}

// Validation, the sorted reaction order and the host-side network data; no
// device work.
kn_status network_host_setup(const kn_network_desc* d, std::unique_ptr<kn_network>& n,
                                    std::vector<double>& r0) {
    const int N = d->n_species, R = d->n_reactions;
    if (N < 1 || N > kMaxSpecies) return fail(KN_ERR_INVALID_ARG, "n_species %d outside [1, %d]", N, kMaxSpecies);
    if (R < 1 || R > 16383) return fail(KN_ERR_INVALID_ARG, "n_reactions %d outside [1, 16383]", R);
    if (!d->A || !d->reac || !d->prod || !d->ln_k0 || !d->t9_exp)
        return fail(KN_ERR_INVALID_ARG, "kn_network_desc has a NULL array");
    n.reset(new kn_network());
    n->N = N;
    n->R = R;
    n->A.assign(d->A, d->A + N);
    for (int i = 0; i < N; ++i)
        if (!(std::isfinite(n->A[i]) && n->A[i] > 0)) return fail(KN_ERR_INVALID_ARG, "A[%d] must be finite and > 0", i);
    n->reac.assign(d->reac, d->reac + 3 * R);
    n->prod.assign(d->prod, d->prod + 3 * R);
    n->lnk0.assign(d->ln_k0, d->ln_k0 + R);
    n->tn.assign(d->t9_exp, d->t9_exp + R);
    n->nr.resize(R);
    n->slot0.resize(R);
    int slots = 0, pslots = 0;
    double nsum = 0, rsum = 0;
    for (int j = 0; j < R; ++j) {
        if (!std::isfinite(n->lnk0[j]) || !std::isfinite(n->tn[j]))
            return fail(KN_ERR_INVALID_ARG, "reaction %d: non-finite rate parameter", j);
        int c = 0, end = 0;
        for (int q = 0; q < 3; ++q) {
            const int s = n->reac[j * 3 + q];
            if (s < 0) {
                end = 1;
                continue;
            }
            if (end || s >= N) return fail(KN_ERR_INVALID_ARG, "reaction %d: bad reactant list", j);
            ++c;
        }
        if (c == 0) return fail(KN_ERR_INVALID_ARG, "reaction %d has no reactant", j);
        int pc = 0;
        for (int q = 0; q < 3; ++q) {
            const int s = n->prod[j * 3 + q];
            if (s >= N) return fail(KN_ERR_INVALID_ARG, "reaction %d: product id out of range", j);
            if (s >= 0) ++pc;
        }
        if (pc == 0) return fail(KN_ERR_INVALID_ARG, "reaction %d has no product", j);
        n->nr[j] = c;
        n->slot0[j] = slots;
        slots += c;
        pslots += pc;
        nsum += n->tn[j];
        rsum += c - 1;
    }
    n->S_r = slots;
    n->S_p = pslots;
    // sort reactions by reactant count (stable): 1-body, then 2-body, then 3-body
    n->perm.resize(R);
    for (int j = 0; j < R; ++j) n->perm[j] = j;
    std::stable_sort(n->perm.begin(), n->perm.end(), [&](int a, int b) { return n->nr[a] < n->nr[b]; });
    n->R1 = n->R12 = 0;
    for (int j = 0; j < R; ++j) {
        n->R1 += n->nr[j] == 1;
        n->R12 += n->nr[j] <= 2;
    }
    // Within each class, a warp of the flux pass handles an aligned block of
    // 32 consecutive sorted reactions and loads reactant q's abundance for
    // each; the loads are one wavefront when the species lie in distinct
    // banks (species mod 32) or coincide.  Greedy order: each position of a
    // block takes the remaining reaction of its class that adds the fewest
    // bank conflicts with what the block already reads, per operand.
    {
        const int bounds[4] = {0, n->R1, n->R12, R};
        std::vector<int> sorted(n->perm);
        for (int cls = 0; cls < 3; ++cls) {
            std::vector<int> pool(sorted.begin() + bounds[cls], sorted.begin() + bounds[cls + 1]);
            std::vector<char> used(pool.size(), 0);
            int block = -1;
            // distinct species the block reads per (operand, bank)
            std::vector<std::vector<std::vector<int>>> words(3, std::vector<std::vector<int>>(32));
            for (int pos = bounds[cls]; pos < bounds[cls + 1]; ++pos) {
                if (pos / 32 != block) {
                    block = pos / 32;
                    for (auto& wq : words)
                        for (auto& wb : wq) wb.clear();
                }
                int best = -1, best_cost = 1 << 30;
                for (size_t c = 0; c < pool.size() && best_cost > 0; ++c) {
                    if (used[c]) continue;
                    const int j = pool[c];
                    int cost = 0;
                    for (int q = 0; q < n->nr[j]; ++q) {
                        const int sp = n->reac[j * 3 + q];
                        const auto& wb = words[q][sp % 32];
                        cost += !wb.empty() && std::find(wb.begin(), wb.end(), sp) == wb.end();
                    }
                    if (cost < best_cost) {
                        best_cost = cost;
                        best = (int)c;
                    }
                }
                used[best] = 1;
                const int j = pool[best];
                n->perm[pos] = j;
                for (int q = 0; q < n->nr[j]; ++q) {
                    const int sp = n->reac[j * 3 + q];
                    auto& wb = words[q][sp % 32];
                    if (std::find(wb.begin(), wb.end(), sp) == wb.end()) wb.push_back(sp);
                }
            }
        }
    }
    r0.assign(2 * (size_t)R, 0.0);
    for (int jn = 0; jn < R; ++jn) {
        const int j = n->perm[jn];
        r0[2 * jn] = n->lnk0[j];
        r0[2 * jn + 1] = n->tn[j];
        n->cmax = std::max(n->cmax, std::fabs(n->tn[j] + 3.0 * (n->nr[j] - 1)));
    }
    if (R + slots + 1 > 0xffff) return fail(KN_ERR_INVALID_ARG, "network too large for 16-bit gather indices");
    n->nbar = nsum / R;
    n->rbar = rsum / R;
    return KN_OK;
}

}  // namespace kn
