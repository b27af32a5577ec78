// The order of a step's launches (step_order.h) with launches, capture and graph
// launches replaced by fakes that fail as told.  Prints a line per case: its
// name, the status, and how often plain, build and launch were called, with the
// steps that a state would have advanced.
#include <cstdio>

#include "../../paper_2509_04673_gb300/csrc/step_order.h"

struct Fake {
    bool have = false, build_ok = true, plain_ok = true;
    int plain = 0, build = 0, launch = 0, steps = 0;
    cgl_status step(bool capturable) {
        return cgl::one_step(
            have, capturable,
            [&] {
                ++plain;
                if (plain_ok) ++steps;
                return plain_ok ? CGL_OK : CGL_ECUDA;
            },
            [&] {
                ++build;
                have = build_ok;
                return build_ok ? CGL_OK : CGL_ECUDA;
            },
            [&] {
                ++launch;
                ++steps;
                return CGL_OK;
            });
    }
};

static void show(const char* name, const Fake& f, cgl_status rc) {
    std::printf("%s %d %d %d %d %d\n", name, (int)rc, f.plain, f.build, f.launch, f.steps);
}

int main() {
    Fake a;  // an ordinary state: plain once, then the graph
    a.step(true);
    a.step(true);
    show("ordinary", a, a.step(true));
    Fake b;  // the graph can never be built
    b.build_ok = false;
    b.step(true);
    show("no_graph", b, b.step(true));
    b.build_ok = true;  // and then it can
    b.step(true);
    show("graph_later", b, b.step(true));
    Fake c;  // a stream that cannot be captured
    c.build_ok = false;
    show("not_capturable", c, c.step(false));
    Fake d;  // a launch fails
    d.plain_ok = false;
    show("launch_fails", d, d.step(true));
    return 0;
}
