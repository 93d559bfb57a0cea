// gq::delta_lower on every fp16 value, for tests/test_delta_lower.py: for each exponent on the command line 65536 words
// "result | ok << 16" to standard output.
#include <cstdio>
#include <cstdlib>

#include "../paper_2505_07004_b200/csrc/gq_gram_dot.cuh"

int main(int argc, char **argv)
{
    for (int a = 1; a < argc; ++a)
        for (unsigned h = 0; h < 65536u; ++h) {
            uint4 v = make_uint4(0u, 0u, 0u, 0u);
            (h & 1u ? v.z : v.x) = h << (h & 2u ? 16 : 0);
            const bool ok = gq::delta_lower(v, static_cast<unsigned>(std::atoi(argv[a])));
            const unsigned w = h & 1u ? v.z : v.x, out = ((w >> (h & 2u ? 16 : 0)) & 0xffffu) | (ok ? 1u << 16 : 0u);
            std::fwrite(&out, sizeof out, 1, stdout);
        }
    return 0;
}
