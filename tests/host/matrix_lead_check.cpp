// Host-side check (compiled by tests/test_matrix_lead.py with g++): a launch
// that peels the matrix-ranked problems of a batch takes the launch shape of
// one of them, whatever else is in the batch.
#include <cstdio>
#include <utility>
#include <vector>

#include "../../paper_2503_20286_gb300/csrc/emo_internal.cuh"

using namespace emo;

static int lead(const std::vector<std::pair<int, long long>>& shapes)
{
    std::vector<ProbIn> ins;
    for (const auto& s : shapes) {
        ProbIn in{};
        in.m = s.first;
        in.n2 = s.second;
        in.mode = MODE_SELECT;
        ins.push_back(in);
    }
    return matrix_lead(ins.data(), (int)ins.size());
}

int main()
{
    const bool ok = lead({{3, 40000}, {6, 1000}}) == 1 && lead({{2, 9000}, {5, 9000}}) == -1 && lead({{6, 10}}) == 0 &&
                    lead({{5, 40000}, {6, 900}, {7, 1200}, {9, 1200}, {16, 30}}) == 2 && lead({{kTreeMaxM, 5}}) == -1 &&
                    lead({{kTreeMaxM + 1, 5}, {2, 6}}) == 0;
    std::printf(ok ? "lead ok\n" : "FAIL\n");
    return !ok;
}
