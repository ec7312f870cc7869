// How a CTA of the one-token 4-bit kernels goes through its tiles (pure C++, no CUDA).
//
// A ring of `stages` tiles is asked for ahead; the CTA then takes its tiles in rounds of up to kQ4Super between two barriers. The stages of
// a round are filled again behind the barrier that follows phase 1 of the round after it, the first point at which every warp is known to
// be done with them. A round can so only hold tiles that were asked for before the round ahead of it gave its stages back: two neighbouring
// rounds fit the ring together.
#pragma once

#ifdef __CUDACC__
#define SPM_HD __host__ __device__ __forceinline__
#else
#define SPM_HD inline
#endif

namespace spm {

constexpr int kQ4Super = 4;            // tiles of a round at most

struct Q4Rounds {
    int both;                          // tiles of two neighbouring rounds at most (0: all tiles are in the ring)
    int left;                          // rounds to come
    // All tiles in the ring: nothing is filled again. Else as many rounds as halves of the ring, rounded up and down in turn, take.
    SPM_HD Q4Rounds(int tiles, int stages) {
        both = tiles <= stages ? 0 : stages;
        if (both == 0) {
            left = tiles > kQ4Super ? 2 : tiles > 0 ? 1 : 0;
        } else {
            const int pairs = tiles / both, rest = tiles - pairs * both;
            left = 2 * pairs + (rest > (both + 1) / 2 ? 2 : rest > 0 ? 1 : 0);
        }
    }
    // Tiles of the next round, of `tiles` to come. In a ring that is filled again the last round takes half of it, rounded up, the one
    // ahead of it half rounded down, and so on, and the first what is left, which gives stages back early. Whole steps of one sequence, us
    // a layer, a tile at a time : half rounded down : the first round the largest : this; Qwen3 shape with 896 rows an expert (three
    // stages, four tiles) 20.8 : 21.6 : 21.1 : 20.1, with 1600 (six tiles) 25.6 : 27.4 : 26.2 : 25.5, 1536 x 1517 (five stages, six
    // tiles) 22.2 : 23.0 : 22.3 : 21.4.
    SPM_HD int next(int tiles) {
        --left;
        if (both == 0) return (tiles + left) >> left;
        return tiles - (left / 2 * both + (left & 1) * ((both + 1) / 2));
    }
};

}  // namespace spm
