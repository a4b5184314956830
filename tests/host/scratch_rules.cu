// The scratch cache (mcg_scratch.h) on a fake memory of limited size: growth,
// optional buffers and their share, and a required request that finds the memory
// taken by them.  Prints one line per case and exits non-zero on a failure.
#include <cstdio>
#include <cstdlib>
#include <map>

#include "mcg_scratch.h"

static int failures = 0;
static void check(bool ok, const char* name) {
    std::printf("%s %s\n", name, ok ? "ok" : "FAIL");
    if (!ok) ++failures;
}

struct Fake {
    static size_t total, used;
    static int syncs, unsynced;  // frees without a sync since the last allocation
    static std::map<void*, size_t> live;
    static bool synced;
    static int alloc(void** p, size_t n) {
        if (used + n > total) return 2;
        *p = std::malloc(1);
        live[*p] = n;
        used += n;
        synced = false;
        return 0;
    }
    static void free(void* p) {
        if (!synced) ++unsynced;
        used -= live.at(p);
        live.erase(p);
        std::free(p);
    }
    static void sync() {
        ++syncs;
        synced = true;
    }
    static size_t available() { return total - used; }
};
size_t Fake::total = 100000, Fake::used = 0;
int Fake::syncs = 0, Fake::unsynced = 0;
std::map<void*, size_t> Fake::live;
bool Fake::synced = false;

int main() {
    mcg::ScratchCache<Fake> c;
    int err = 0;
    void* a = c.get("a", 1000, &err);
    check(a && !err && Fake::used == 1000, "first");
    check(c.get("a", 900, &err) == a && !err && Fake::used == 1000, "kept");
    check(c.get("a", 2000, &err) && !err && Fake::used == 2000 && Fake::syncs == 1, "grown");
    check(c.get("e", 0, &err) && !err && Fake::used == 2256, "empty");
    // a quarter of the free memory
    check(!c.get_optional("o", 24437) && Fake::used == 2256, "above_share");
    void* o = c.get_optional("o", 24436);
    check(o && Fake::used == 2256 + 24436, "share");
    check(c.get_optional("o", 20000) == o && c.optional_room("o") == 24436, "optional_kept");
    check(!c.get_optional("o", 60000) && c.get_optional("o", 24436) == o, "optional_not_grown");
    check(c.get_optional("p", 15000) && c.optional_room("q") == (100000 - 2256 - 24436 - 15000) / 4, "second_optional");
    // a required buffer that only fits without the optional ones
    const int s = Fake::syncs;
    check(c.get("b", 90000, &err) && !err && Fake::used == 92256 && Fake::syncs == s + 2, "optional_gives_way");
    // one that does not fit at all: an error, and the cache is as before
    check(!c.get("d", 90000, &err) && err == 2 && Fake::used == 92256, "no_memory");
    err = 0;
    check(c.get("d", 5000, &err) && !err && Fake::used == 97256, "after_the_error");
    check(c.get_optional("o", 600) && Fake::used == 97856, "optional_again");
    // an optional buffer that a call requires is not given up for another one
    check(c.get("o", 500, &err) && !err && !c.get("f", 2500, &err) && err == 2 && Fake::used == 97856, "required_by_now");
    // growing a required buffer beyond the memory loses it, with an error
    err = 0;
    check(!c.get("b", 99000, &err) && err == 2 && Fake::used == 7856, "growth_fails");
    c.clear();
    check(Fake::used == 0 && Fake::live.empty(), "cleared");
    check(Fake::unsynced == 0, "waits_before_each_free");
    return failures != 0;
}
