// Host-only check of the gridding tables of the kernels that take cell pairs (x, y), (x, y + 1) (no GPU): builds them
// with the library's own builders from a cell-major mapping read from a text file, then walks them as the kernels do.
// The grid of 64 x 64 cells has the slot tables of the tensor-core form at N_p = 128; 128 x 128 cells the runs of the
// half-image kernels (one round of all rows, 16 warps); 256 x 256 cells those of the two-pass form (rounds of 16 rows, 8
// warps).  Checks that
//   every index stays inside the tables and every antenna inside the array, a run's steps are a multiple of the steps
//   read ahead, and the last step of every lane's pair is the same one for the warp's 32 lanes;
//   every cell pair is stored exactly once, at an in-range place;
//   the weights walked for a cell are its mapping entries, each exactly once (lanes past their list and padding steps
//   have zero weights), so its sum is that of the mapping within FP32 rounding.
// Exit status 0 when every check holds.
#include "../../paper_1510_08318_gb300/csrc/moff_dftgemm.cu"
#include "../../paper_1510_08318_gb300/csrc/moff_half256.cu"
#include <cstdio>
#include <fstream>
#include <map>

int main(int argc, char** argv) {
    if (argc < 2) return 2;
    std::ifstream f(argv[1]);
    int ncell = 0, nnz = 0;
    f >> ncell >> nnz;
    const int NG = ncell == 64 * 64 ? 64 : ncell == 128 * 128 ? 128 : ncell == 256 * 256 ? 256 : 0;
    if (NG == 0) return 2;
    std::vector<int> cptr(ncell + 1), ant(nnz);
    std::vector<float> wr(nnz), wi(nnz);
    for (auto& v : cptr) f >> v;
    for (auto& v : ant) f >> v;
    for (auto& v : wr) f >> v;
    for (auto& v : wi) f >> v;
    std::vector<int2> cent(nnz);
    int A = 1;
    for (int i = 0; i < nnz; ++i) {
        int b;
        std::memcpy(&b, &wr[i], 4);
        cent[i] = int2{b, ant[i]};
        A = std::max(A, ant[i] + 1);
    }
    int bad = 0;
    // what the walk gave a cell: antenna -> weight, and how often the cell was stored
    std::vector<std::map<int, std::pair<float, float>>> got(ncell);
    std::vector<int> stored(ncell, 0);
    auto take = [&](int cell, int a, float w, float v) {
        if (w == 0.f && v == 0.f) return;
        if (a >= A || !got[cell].emplace(a, std::make_pair(w, v)).second) ++bad;
    };
    struct Step { int ant; float2 w, wi; };
    if (NG == 64) {
        std::vector<uint32_t> lane;
        std::vector<int2> slot;
        std::vector<float2> w, wim;
        std::vector<uint16_t> an;
        if (!epic::dftgemm_pair_tables(cptr, cent, wi, lane, slot, w, wim, an)) return 1;
        using namespace epic::dg;
        if ((int)slot.size() != NPOS || (int)lane.size() != 32 * NPOS || w.size() != an.size() || wim.size() != an.size()) return 1;
        std::map<int, int> cell_of;                       // E^T table offset -> cell
        for (int y = 0; y < NG; ++y)
            for (int x = 0; x < NG; ++x) cell_of[epic::tc::koff(x, y, NG)] = y * NG + x;
        for (int s = 0; s < NPOS; ++s) {
            if (slot[s].y < 0) continue;
            unsigned banks = 0;
            for (int l = 0; l < 32; ++l) {
                const int off = lane[32 * s + l] & 0xffff, sum = lane[32 * s + l] >> 16;
                if (!cell_of.count(off) || cell_of[off] / NG % 2) { ++bad; continue; }
                const int c = cell_of[off];
                if (c / NG + c % NG != sum || epic::tc::koff(c % NG, c / NG + 1, NG) != off + 1) ++bad;
                banks |= 1u << ((off / 2) % 32);
                ++stored[c];
                ++stored[c + NG];
                for (int k = 0; k < slot[s].y; ++k) {
                    const long e = (long)slot[s].x + 32 * k + l;
                    if (e < 0 || e >= (long)an.size() || an[e] >= A) { ++bad; continue; }
                    take(c, an[e], w[e].x, wim[e].x);
                    take(c + NG, an[e], w[e].y, wim[e].y);
                }
            }
            if (banks != 0xffffffffu) ++bad;
        }
    } else {
        const int rows = NG == 128 ? 128 : 16, warps = NG == 128 ? 16 : 8, stride = NG == 128 ? epic::half256::RBS : 256;
        std::vector<int4> run;
        std::vector<float2> w, wim;
        std::vector<uint32_t> key;
        std::vector<uint16_t> empty;
        if (NG == 128) epic::half256_tables(cptr, cent, wi, run, w, wim, key, empty);
        else epic::pair_run_tables(NG, rows, stride, warps, 8, cptr, cent, wi, run, w, wim, key, empty);
        if ((int)run.size() != NG / rows * warps || w.size() != key.size() || wim.size() != key.size()) return 1;
        auto place = [&](int round, int off) -> int {     // cell of a place (in two rows' storage), -1 if there is none
            const int y = 2 * (off / (2 * stride)), x = off % (2 * stride);
            return y < rows && x < NG ? (round * rows + y) * NG + x : -1;
        };
        for (size_t r = 0; r < run.size(); ++r) {
            const int round = (int)r / warps;
            const int4 m = run[r];
            if (m.y % epic::kGridAhead || m.x < 0 || (size_t)m.x + 32 * (size_t)m.y > key.size() ||
                (size_t)m.z + 32 * (size_t)m.w > empty.size()) { ++bad; continue; }
            for (int z = 0; z < 32 * m.w; ++z) {
                const int c = place(round, empty[m.z + z]);
                if (c < 0) { ++bad; continue; }
                ++stored[c];
                ++stored[c + NG];
            }
            for (int l = 0; l < 32; ++l) {
                std::vector<Step> held;                   // since the last store
                for (int k = 0; k < m.y; ++k) {
                    const size_t e = (size_t)m.x + 32 * (size_t)k + l;
                    const bool last = (key[e] & epic::kGridLast) != 0;
                    if (last != ((key[e - l] & epic::kGridLast) != 0) || (int)(key[e] & 0xffff) >= A) ++bad;
                    held.push_back({(int)(key[e] & 0xffff), w[e], wim[e]});
                    if (!last) continue;
                    const int c = place(round, (key[e] >> 16) & 0x7fff);
                    if (c < 0) { ++bad; held.clear(); continue; }
                    ++stored[c];
                    ++stored[c + NG];
                    for (const Step& t : held) {
                        take(c, t.ant, t.w.x, t.wi.x);
                        take(c + NG, t.ant, t.w.y, t.wi.y);
                    }
                    held.clear();
                }
                for (const Step& t : held)                // padding at the run's end
                    if (t.w.x != 0.f || t.w.y != 0.f || t.wi.x != 0.f || t.wi.y != 0.f) ++bad;
            }
        }
    }
    int miss = 0, wrong = 0;
    for (int c = 0; c < ncell; ++c) {
        if (stored[c] != 1) ++miss;
        size_t n = 0;
        for (int i = cptr[c]; i < cptr[c + 1]; ++i) {
            if (wr[i] == 0.f && wi[i] == 0.f) continue;
            ++n;
            const auto it = got[c].find(ant[i]);
            if (it == got[c].end() || it->second.first != wr[i] || it->second.second != wi[i]) ++wrong;
        }
        if (n != got[c].size()) ++wrong;
    }
    std::printf("bad %d not stored once %d wrong entries %d\n", bad, miss, wrong);
    return (bad || miss || wrong) ? 1 : 0;
}
