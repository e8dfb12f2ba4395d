// Test harness: the lines of the library's launch choice (latency_limit and pair_line in qldpc_host.cpp) for 465 rows
// of one degree of 6 to 9 with one single-shot block an SM, one "precision single pair" line per precision.
#define main layout_main
#include "host_layout_probe.cpp"
#undef main

int main()
{
    qldpc::KernelChoice kc{};
    kc.dc = 8;
    kc.uniform = true;
    for (int p : {QLDPC_FP32, QLDPC_INT16, QLDPC_INT8})
        std::printf("%lld %lld\n", static_cast<long long>(qldpc::detail::latency_limit(kc, p, 1)),
                    static_cast<long long>(qldpc::detail::pair_line(kc, p, 465)));
    return 0;
}
