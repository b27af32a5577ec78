// step_order.h — the order of a step's launches on the host.
#pragma once

#include "../../include/cgl.h"

namespace cgl {

// One step: by the step graph (launch) where there is one.  Else, where the
// stream can be captured, by plain launches (plain), behind which the graph is
// built while they run: building costs about as much as a step of 256^2 elements.
// A graph that cannot be built is then no failure of the step, which has run;
// the next step goes the same way.  Where the stream cannot be captured the
// graph comes first, and its failure leaves the state as it was.
template <class Plain, class Build, class Launch>
cgl_status one_step(bool have_graph, bool capturable, const Plain& plain, const Build& build, const Launch& launch) {
    if (!have_graph && capturable) {
        const cgl_status rc = plain();
        if (rc == CGL_OK) (void)build();
        return rc;
    }
    if (!have_graph)
        if (const cgl_status rc = build()) return rc;
    return launch();
}

}  // namespace cgl
