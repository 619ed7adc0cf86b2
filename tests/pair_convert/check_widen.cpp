// widen of the given floats (bit patterns in hexadecimal): one double's bits a line.
#include <cinttypes>
#include <cstdio>
#include <cstdlib>

#include "../../paper_2108_07031_gb300/csrc/pair_convert.cuh"

int main(int argc, char** argv) {
    for (int i = 1; i < argc; ++i)
        std::printf("%016" PRIx64 "\n", lskum::dword(lskum::widen(lskum::bitsf(uint32_t(std::strtoul(argv[i], nullptr, 16))))));
    return 0;
}
