// Prints the status and the number of lines a unit of ccf_ramp_plan for a mask of 2,000 lines, and the
// error text.
#include <cmath>
#include <cstdio>
#include <vector>

#include "soap_internal.cuh"

int main() {
    soap_ctx c{};
    c.n_px = 8192;
    c.lam_s = 5000.0;
    c.delta = 2.9e-6;
    std::vector<double> mask(2000);
    for (size_t l = 0; l < mask.size(); l++) mask[l] = c.lam_s * std::exp((60.0 + 4.0 * (double)l) * c.delta);
    soap::CcfState st;
    soap::CcfPlan p;
    p.n_spec = 8;
    p.n_lines = (int)mask.size();
    p.n_v = 177;
    p.v_lo = -22.0;
    p.v_step = 0.25;
    p.h = 0.45;
    const soap_status s = soap::ccf_ramp_plan(&c, st, mask.data(), p, 152);
    printf("%d %d %s\n", (int)s, p.ramp_L, soap_last_error());
    return 0;
}
