// chimera_index_attach_rabitq with a CUDA runtime of which one call fails, each in turn (host only: fake_cudart.cpp).  After every failure the index has to be as it was, apart from
// copies that are an option, and nothing may be left allocated that the index does not hold.
#include <stdio.h>

#include <set>

#include "common.cuh"

// fake_cudart.cpp
extern std::set<void *> fake_live;               // allocations
extern int fake_calls, fake_fail_at;             // calls that can fail, and the one that does (from 1; 0 = none)
extern int fake_last_error;

int main()
{
    int bad = 0;
    auto check = [&](bool ok, const char *what, int n, bool again) {
        if (!ok) { printf("call %d fails, %s: %s\n", n, again ? "codes attached before" : "first codes", what); ++bad; }
    };
    int32_t tok[1];
    uint8_t bits[2][16];
    float inv[2][4], rotation[1];
    for (int again = 0; again < 2; ++again) {
        for (int n = 1;; ++n) {
            chimera::Index ix;
            ix.T = 1000; ix.D = 64; ix.CB = 16; ix.sm_count = 1; ix.tok_id = tok;
            chimera_index *h = reinterpret_cast<chimera_index *>(&ix);
            fake_fail_at = fake_last_error = 0;
            if (again && chimera_index_attach_rabitq(h, rotation, bits[0], inv[0], nullptr)) return 2;
            const chimera::Index before = ix;
            fake_calls = 0;
            fake_fail_at = n;
            const int rc = chimera_index_attach_rabitq(h, rotation, bits[1], inv[1], nullptr);
            const bool injected = fake_calls >= n;
            check((ix.list_bits == nullptr) == (ix.list_inv == nullptr), "one copy without the other", n, again);
            if (rc) {
                check(ix.rq_bits == before.rq_bits && ix.rq_inv == before.rq_inv && ix.rot_t == before.rot_t,
                      "codes and rotation of two attachments", n, again);
                check(ix.list_bits == nullptr, "a copy of other codes", n, again);
            } else {
                check(ix.rq_bits == bits[1] && ix.rq_inv == inv[1] && ix.rot_t != nullptr, "not attached", n, again);
            }
            check(fake_live.size() == (size_t)(ix.rot_t != nullptr) + ix.rq_mem.own, "memory is lost", n, again);
            while (!fake_live.empty()) cudaFree(*fake_live.begin());
            if (!injected) {
                check(rc == 0 && ix.list_bits != nullptr, "no failure, yet no copies", n, again);
                break;
            }
        }
    }
    printf("%d faults\n", bad);
    return bad ? 1 : 0;
}
