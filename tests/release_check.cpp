// Order of the runtime calls of csrc/release.h, on a stand-in for the runtime.
#include <cstdio>
#include <string>

#include "release.h"

struct World {
    int current = 0, devices = 2;
    bool can_wait = true;
    std::string log;
} w;

struct Obj {
    int dev;
    const char *name;
};

struct FakeRt {
    bool device(int *d) { return *d = w.current, true; }
    bool set_device(int d) {
        if (d >= w.devices) return false;
        w.current = d;
        w.log += "set" + std::to_string(d) + " ";
        return true;
    }
    bool wait() {
        w.log += (w.can_wait ? "wait" : "nowait") + std::to_string(w.current) + " ";
        return w.can_wait;
    }
    void give_back(Obj *o) {
        w.log += std::string(o->name) + (o->dev == w.current ? " " : "@WRONG ");
    }
};

static int bad = 0;

static void expect(const char *what, const std::string &want) {
    if (w.log != want || w.current != 0) {
        std::printf("%s: got '%s' (current %d), want '%s'\n", what, w.log.c_str(), w.current, want.c_str());
        ++bad;
    }
    w.log.clear();
}

int main() {
    packsell::Retired<Obj, FakeRt> r;
    Obj a{0, "a"}, b{1, "b"}, c{0, "c"}, d{1, "d"}, e{0, "e"}, f{7, "f"};
    r.retire(0, &a, FakeRt{});
    expect("current device", "wait0 a ");
    r.retire(1, &b, FakeRt{});
    expect("another device: its own wait, then back", "set1 wait1 b set0 ");
    w.can_wait = false;
    r.retire(0, &c, FakeRt{});
    expect("cannot wait: nothing is given back", "nowait0 ");
    r.retire(1, &d, FakeRt{});
    expect("cannot wait on another device", "set1 nowait1 set0 ");
    w.can_wait = true;
    r.retire(0, &e, FakeRt{});
    expect("the next one takes the kept one along, its device's only", "wait0 c e ");
    r.flush(1, FakeRt{});
    expect("flush of the other device", "set1 wait1 d set0 ");
    r.retire(7, &f, FakeRt{});
    expect("a device that cannot be selected", "");
    r.flush(0, FakeRt{});
    r.flush(1, FakeRt{});
    expect("nothing left", "");
    std::printf(bad ? "%d failed\n" : "ok\n", bad);
    return bad != 0;
}
