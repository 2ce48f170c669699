// Walks through every interleaving of a data gradient's copying thread, its two issuing threads and its epilogue (x3_ring.cuh), with
// copies that land and products that end at any time, and reports the first state in which a slot is overwritten while products still
// read it, products read what has not landed, a thread is more than one phase away from the barrier it waits for, or nobody can go on.
#include <array>
#include <cstdio>
#include <cstdlib>
#include <string>
#include <unordered_set>
#include <vector>
#include "x3_gemm.cuh"
#include "x3_ring.cuh"

namespace {

enum Kind { WAIT, LOAD, MULTIPLY, COMMIT, ARRIVE };
struct Op { Kind kind; int bar, phase, a, b; };         // phase waited for; loads: a; products: loads a and b
enum { A_FULL = 0, A_EMPTY = 8, B_FULL = 16, B_EMPTY = 32, D_FULL = 48, D_EMPTY = 50, BARS = 52 };
enum { COPY, ISSUE0, ISSUE1, EPILOGUE, ACTORS };     // its eight warps as one

struct Load { int bar, slot; bool is_a; std::vector<std::pair<int, int>> readers; };    // (thread, its products up to and with this one)
std::vector<Op> ops[ACTORS];
std::vector<Load> loads;
int products[2];                                        // of each issuing thread, in total

struct Waits {                                          // the phase behind each parity: every wait is for the same one or the next
    int actor, phase[BARS];
    explicit Waits(int who) : actor(who) { for (int& ph : phase) ph = -2; }
    bool wait(int bar, unsigned parity)
    {
        int& ph = phase[bar];
        if (ph == -2) ph = parity ? -1 : 0;
        else if ((unsigned)(ph & 1) != parity) ++ph;
        ops[actor].push_back({WAIT, bar, ph, 0, 0});
        return true;
    }
};
struct CopyIo {
    Waits* w;
    bool wait_a_empty(int ea, unsigned par) { return w->wait(A_EMPTY + ea, par); }
    bool wait_b_empty(int sb, unsigned par) { return w->wait(B_EMPTY + sb, par); }
    void load(int bar, int slot, bool is_a)
    {
        ops[COPY].push_back({LOAD, bar, 0, (int)loads.size(), 0});
        loads.push_back({bar, slot, is_a, {}});
    }
    void load_a(int ea, int, int, int) { load(A_FULL + ea, ea, true); }
    void load_b(int sb, int, int, int) { load(B_FULL + sb, sb, false); }
};
struct IssueIo {
    Waits* w;
    int e, *done;
    void push(Kind k, int bar) { ops[ISSUE0 + e].push_back({k, bar, 0, 0, 0}); }
    bool wait_a_full(int ea, unsigned par) { return w->wait(A_FULL + ea, par); }
    bool wait_b_full(int sb, unsigned par) { return w->wait(B_FULL + sb, par); }
    bool wait_d_empty(unsigned par) { return w->wait(D_EMPTY + e, par); }
    // The copy that the products are meant for: the one of the phase last waited for.
    int copy_of(int bar)
    {
        int nth = w->phase[bar];
        for (size_t i = 0; i < loads.size(); ++i)
            if (loads[i].bar == bar && nth-- == 0) return (int)i;
        printf("products of a slot that is never filled\n");
        exit(1);
    }
    void multiply(int ea, int sb, int, bool)
    {
        const int a = copy_of(A_FULL + ea), b = copy_of(B_FULL + sb);
        ++*done;
        loads[a].readers.push_back({e, *done});
        loads[b].readers.push_back({e, *done});
        ops[ISSUE0 + e].push_back({MULTIPLY, 0, 0, a, b});
    }
    void commit_a_empty(int ea) { push(COMMIT, A_EMPTY + ea); }
    void commit_b_empty(int sb) { push(COMMIT, B_EMPTY + sb); }
    void commit_d_full() { push(COMMIT, D_FULL + e); }
    void arrive_a_empty(int ea) { push(ARRIVE, A_EMPTY + ea); }
    void arrive_b_empty(int sb) { push(ARRIVE, B_EMPTY + sb); }
};

struct State {
    uint16_t pc[ACTORS], done[2];
    unsigned __int128 landed;
};

// Arrivals on a barrier: of each actor's first `pc` operations, commits counted once the products before them have ended.
std::vector<std::vector<std::array<uint8_t, BARS>>> arrived[2];     // [issuing thread][pc][done]
std::vector<std::array<uint8_t, BARS>> epilogue_arrived;

int phases(const State& s, int bar)                     // completed ones
{
    int n = 0;
    if ((bar >= A_FULL && bar < A_EMPTY) || (bar >= B_FULL && bar < B_EMPTY)) {
        for (size_t i = 0; i < loads.size(); ++i) n += loads[i].bar == bar && (s.landed >> i & 1);
        return n;
    }
    for (int e = 0; e < 2; ++e) n += arrived[e][s.pc[ISSUE0 + e]][s.done[e]][bar];
    n += epilogue_arrived[s.pc[EPILOGUE]][bar];
    return bar >= D_FULL ? n : n / 2;
}

std::string wrong(const State& s, int who, const Op& op)
{
    char text[160];
    if (op.kind == WAIT) {
        const int n = phases(s, op.bar);
        if (n > op.phase + 1 || n < op.phase) {
            snprintf(text, sizeof text, "actor %d waits for phase %d of barrier %d, which has completed %d", who, op.phase, op.bar, n);
            return text;
        }
    }
    if (op.kind == LOAD) {
        const Load& l = loads[op.a];
        for (int i = 0; i < op.a; ++i)
            if (loads[i].bar == l.bar)
                for (auto [e, k] : loads[i].readers)
                    if (s.done[e] < k) {
                        snprintf(text, sizeof text, "copy %d overwrites %s slot %d, which thread %d's products still read", op.a, l.is_a ? "A" : "B", l.slot, e);
                        return text;
                    }
    }
    if (op.kind == MULTIPLY)
        for (int i : {op.a, op.b})
            if (!(s.landed >> i & 1)) {
                snprintf(text, sizeof text, "thread %d multiplies copy %d, which has not landed", who - ISSUE0, i);
                return text;
            }
    return "";
}

int walk(const hts::X3Ring& r)
{
    for (auto& o : ops) o.clear();
    loads.clear();
    products[0] = products[1] = 0;
    Waits wc(COPY), w0(ISSUE0), w1(ISSUE1), we(EPILOGUE);
    hts::x3_ring_copy(r, CopyIo{&wc});
    hts::x3_ring_issue(r, 0, IssueIo{&w0, 0, &products[0]});
    hts::x3_ring_issue(r, 1, IssueIo{&w1, 1, &products[1]});
    int tiles = 0;
    for (int t = r.first; t < r.m_tiles * r.n_tiles; t += r.blocks) ++tiles;
    const int parts = (r.chunks * r.taps + hts::kX3Part - 1) / hts::kX3Part;
    for (int it = 0; it < tiles * parts; ++it) {
        we.wait(D_FULL + (it & 1), it >> 1 & 1);
        ops[EPILOGUE].push_back({ARRIVE, D_EMPTY + (it & 1), 0, 0, 0});
    }
    if (loads.size() > 128) { printf("more copies than a state holds\n"); return 1; }
    for (int e = 0; e < 2; ++e) {
        auto& t = arrived[e];
        t.assign(ops[ISSUE0 + e].size() + 1, {});
        for (size_t pc = 0; pc < t.size(); ++pc) {
            t[pc].assign(products[e] + 1, {});
            for (int done = 0; done <= products[e]; ++done) {
                int before = 0;
                for (size_t i = 0; i < pc; ++i) {
                    const Op& op = ops[ISSUE0 + e][i];
                    before += op.kind == MULTIPLY;
                    if (op.kind == ARRIVE || (op.kind == COMMIT && before <= done)) ++t[pc][done][op.bar];
                }
            }
        }
    }
    epilogue_arrived.assign(ops[EPILOGUE].size() + 1, {});
    for (size_t i = 0; i < ops[EPILOGUE].size(); ++i) {
        epilogue_arrived[i + 1] = epilogue_arrived[i];
        if (ops[EPILOGUE][i].kind == ARRIVE) ++epilogue_arrived[i + 1][ops[EPILOGUE][i].bar];
    }
    std::unordered_set<std::string> seen;
    std::vector<State> todo;
    auto push = [&](const State& s) {
        std::string key((const char*)s.pc, sizeof s.pc);
        key.append((const char*)s.done, sizeof s.done);
        key.append((const char*)&s.landed, sizeof s.landed);
        if (seen.insert(std::move(key)).second) todo.push_back(s);
    };
    push(State{});
    while (!todo.empty()) {
        const State s = todo.back();
        todo.pop_back();
        bool moved = false, over = true;
        for (int a = 0; a < ACTORS; ++a) {
            if (s.pc[a] == ops[a].size()) continue;
            over = false;
            const Op& op = ops[a][s.pc[a]];
            const std::string why = wrong(s, a, op);
            if (!why.empty()) { printf("%s\n", why.c_str()); return 1; }
            if (op.kind == WAIT && phases(s, op.bar) <= op.phase) continue;
            State n = s;
            ++n.pc[a];
            push(n);
            moved = true;
        }
        for (int i = 0, seen_loads = 0; i < s.pc[COPY]; ++i)
            if (ops[COPY][i].kind == LOAD) {
                if (!(s.landed >> seen_loads & 1)) {
                    State n = s;
                    n.landed |= (unsigned __int128)1 << seen_loads;
                    push(n);
                    moved = true;
                }
                ++seen_loads;
            }
        for (int e = 0; e < 2; ++e) {
            int at = 0;
            for (int i = 0; i < s.pc[ISSUE0 + e]; ++i) at += ops[ISSUE0 + e][i].kind == MULTIPLY;
            if (s.done[e] < at) {
                State n = s;
                ++n.done[e];
                push(n);
                moved = true;
            }
        }
        if (!moved && !over) { printf("nobody can go on\n"); return 1; }
    }
    printf("%zu states\n", seen.size());
    return 0;
}

}  // namespace

// chunks taps grid-width m_tiles n_tiles first blocks
int main(int argc, char** argv)
{
    if (argc != 8) return 2;
    int v[7];
    for (int i = 0; i < 7; ++i) v[i] = atoi(argv[i + 1]);
    const int side = v[1] == 9 ? 3 : v[1] == 4 ? 2 : 1;
    int shift[9];
    for (int i = 0; i < v[1]; ++i) shift[i] = -(i / side * v[2] + i % side);
    hts::X3TapParams p{};
    if (!hts::x3_taps_plan(&p, v[0], v[1], shift)) { printf("no plan\n"); return 1; }
    printf("taps per entry %d, entries %d, stages %d: ", p.tpe, p.entries, p.b_stages);
    return walk({v[3], v[4], p.chunks, p.taps, p.tpe, p.entries, p.b_stages, v[5], v[6]});
}
