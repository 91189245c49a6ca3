// Host check of nat_word (csrc/team_fft.cuh) for all five tiles: distinct words inside the
// exchange buffer, contiguous rows, and 32 distinct banks for the lanes of every warp that
// writes or reads one element index in the pass-3 layout.
#include <cstdio>
#include <set>

#include "team_fft.cuh"

using namespace ptylm;

template <class G>
int check(const char* name) {
    int bad = 0;
    std::set<int> words;
    for (int ky = 0; ky < G::S; ++ky)
        for (int kx = 0; kx < G::S; ++kx) {
            const int w = nat_word<G>(ky, kx);
            bad += !words.insert(w).second || w < 0 || w >= 2 * G::EXW;
            bad += kx > 0 && w != nat_word<G>(ky, kx - 1) + 1;
        }
    for (int t0 = 0; t0 < G::T; t0 += 32)
        for (int e = 0; e < G::E; ++e) {
            std::set<int> banks;
            for (int l = 0; l < 32; ++l) banks.insert(nat_word<G>(freq_ky<G>(t0 + l), freq_kx<G>(t0 + l, e)) % 32);
            bad += banks.size() != 32;
        }
    printf("%s: %d failed checks\n", name, bad);
    return bad;
}

int main() {
    return check<Geo<5, 5>>("32/32") + check<Geo<5, 4>>("32/16") + check<Geo<6, 5>>("64/32") + check<Geo<6, 4>>("64/16") +
           check<Geo<7, 5>>("128/32");
}
