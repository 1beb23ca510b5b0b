// The form that a DNA solve takes on a device of `sms` multiprocessors, from the runtime's own
// estimate. Input lines: sms n m l d q single; output lines: middle letters, counter planes and
// warps per block of the sieve, or 0 0 0 for the tree.
#include "../../paper_2403_00306_gb300/csrc/pms_runtime.cu"

#include <cstdio>

int main()
{
    int sms, n, m, l, d, q, single;
    while (std::scanf("%d %d %d %d %d %d %d", &sms, &n, &m, &l, &d, &q, &single) == 7) {
        pms_ctx h;
        h.num_sms = sms;
        const SieveForm f = estimate_form(&h, n, m, l, d, q, single != 0);
        std::printf("%d %d %d\n", f.mid, f.planes, f.mid ? f.share : 0);
    }
    return 0;
}
