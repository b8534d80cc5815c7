// The arguments of the launches that the tests look at, as JSON lines.
#include <cstdint>
#include <cstdio>
#include <string>

#include "mmod_internal.h"

static unsigned long long num(const void *p) { return (unsigned long long)(uintptr_t)p; }

std::string describe_launch(const std::string &name, void *const *args) {
    char line[512] = "";
    if (name.find("step_tma_kernel") != std::string::npos || name.find("step_tma_claim_kernel") != std::string::npos) {
        const mmod::StepArgs &a = *(const mmod::StepArgs *)args[0];
        snprintf(line, sizeof(line),
                 "{\"op\": \"step\", \"pdl\": %d, \"n\": %d, \"ucur\": %llu, \"uprev\": %llu, \"uout\": %llu, "
                 "\"gout\": %llu, \"c\": %llu, \"image\": %d}",
                 a.pdl, a.n, num(a.ucur), num(a.uprev), num(a.uout), num(a.gout), num(a.c), a.image);
    } else if (name.find("compress") != std::string::npos) {   // a checkpoint pair: volumes, then stored forms
        void *const *p = (void *const *)args[0];
        snprintf(line, sizeof(line), "{\"op\": \"ckpt\", \"restore\": %d, \"u\": [%llu, %llu], \"q\": [%llu, %llu]}",
                 name.find("decompress") != std::string::npos, num(p[0]), num(p[1]), num(p[2]), num(p[3]));
    }
    return line;
}
