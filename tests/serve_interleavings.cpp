// Enumerates the interleavings of serve_publish / serve_take (serve_take.cuh):
// every warp publishes its launch's tail and then takes queries until it has
// its share or finds none. Reads "tail share" of each warp from the arguments
// and prints the finished executions' worst outcome.
//
// A warp's state is the list of results that its operations on the counts have
// returned so far: the functions are run again from the start for each step,
// and the first operation without a result is the warp's next one.
#include <cstdio>
#include <cstdlib>
#include <set>
#include <string>
#include <unordered_set>
#include <vector>

#include "serve_take.cuh"

using u64 = unsigned long long;

struct Memory {
    u64 v[ann::kServeCounts] = {};
};

struct Op {
    int kind = 0;   // 0 load, 1 add, 2 max
    uint32_t at = 0;
    u64 x = 0;
};

struct Next {
    Op op;
};

struct Counts {
    static constexpr uint32_t kLooks = 2;
    const std::vector<u64> &results;
    size_t used = 0;
    bool tired = false;
    u64 step(int kind, uint32_t at, u64 x)
    {
        if (used < results.size()) return results[used++];
        throw Next{Op{kind, at, x}};
    }
    u64 load(uint32_t at) { return step(0, at, 0); }
    u64 add(uint32_t at, u64 x) { return step(1, at, x); }
    u64 max(uint32_t at, u64 x) { return step(2, at, x); }
    void fence() {}
    void gave_up() { tired = true; }
};

struct Warp {
    u64 tail = 0;
    uint32_t share = 0;
    std::vector<u64> results, got;
    bool tired = false;
};

// Runs the warp up to its next operation; false if it has left.
static bool next(Warp &w, Op &op)
{
    Counts c{w.results};
    w.got.clear();
    try {
        ann::serve_publish(c, w.tail);
        for (uint32_t served = 0; served < w.share; ++served) {
            u64 h = 0;
            if (!ann::serve_take(c, &h)) break;
            w.got.push_back(h);
        }
    } catch (const Next &n) {
        op = n.op;
        return true;
    }
    w.tired = c.tired;
    return false;
}

static std::unordered_set<std::string> seen;
static u64 executions = 0, orphans = 0, repeats = 0, tired = 0;

static void explore(const Memory &m, const std::vector<Warp> &warps, u64 all)
{
    std::string key(reinterpret_cast<const char *>(m.v), sizeof(m.v));
    for (const Warp &w : warps) {
        key += '|';
        key.append(reinterpret_cast<const char *>(w.results.data()), w.results.size() * sizeof(u64));
    }
    if (!seen.insert(key).second) return;
    bool running = false;
    for (size_t i = 0; i < warps.size(); ++i) {
        std::vector<Warp> now = warps;
        Op op;
        if (!next(now[i], op)) continue;
        running = true;
        Memory after = m;
        u64 &x = after.v[op.at];
        now[i].results.push_back(x);
        if (op.kind == 1) x += op.x;
        if (op.kind == 2 && op.x > x) x = op.x;
        next(now[i], op);
        if (now[i].tired) ++tired;   // its looks ran out while the others stood still: reported, not lost
        else explore(after, now, all);
    }
    if (running) return;
    ++executions;
    std::multiset<u64> taken;
    for (Warp w : warps) {
        Op op;
        next(w, op);
        taken.insert(w.got.begin(), w.got.end());
    }
    for (u64 h : taken) repeats += taken.count(h) > 1 || h >= all;
    orphans += taken.size() < all;
}

int main(int argc, char **argv)
{
    std::vector<Warp> warps;
    u64 all = 0;
    for (int i = 1; i + 1 < argc; i += 2) {
        Warp w;
        w.tail = strtoull(argv[i], nullptr, 10);
        w.share = (uint32_t)atoi(argv[i + 1]);
        all = w.tail > all ? w.tail : all;
        warps.push_back(w);
    }
    explore(Memory{}, warps, all);
    printf("%llu executions, %llu left a query, %llu took one twice, %llu gave up\n", executions, orphans, repeats, tired);
    return orphans || repeats || !executions ? 1 : 0;
}
