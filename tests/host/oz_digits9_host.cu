// Host driver for the nine-bit digits of the split kernels (paper_2509_23018_gb300/csrc/oz_digits.cuh):
// lines "<x bits> <column max bits> <s>" in, the s digits as BF16 bit patterns (d_0 first) out.
#include <cstdio>
#include "../../paper_2509_23018_gb300/csrc/oz_digits.cuh"

int main()
{
    unsigned long long xb, cb;
    int s;
    while (std::scanf("%llx %llx %d", &xb, &cb, &s) == 3) {
        const int E = gw::oz_expo_pos(gw::oz_bits_d(cb), -400);
        uint16_t d[8];
        gw::oz_store_digits<gw::kOzBeta>(gw::oz_round_scaled(gw::oz_bits_d(xb), gw::oz_frac_bits(s) - E), s,
                                         gw::oz_digit_bias<gw::kOzBeta>(s), d, 1);
        for (int i = 0; i < s; ++i) std::printf("%04x ", d[i]);
        std::printf("\n");
    }
    return 0;
}
