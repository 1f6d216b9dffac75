// Host-side check of the allocation-free selection's scratch (compiled by
// tests/test_noalloc_sizes.py with g++; no GPU involved): the largest
// selections of its first range, one per objective count and group size, still
// fit.
#include <cstdio>

#include "../../paper_2503_20286_gb300/csrc/emo_internal.cuh"

using namespace emo;

int main()
{
    // CTAs, objectives, points, references
    const long long cases[][4] = {
        {152, 2, 909, 158816},  {152, 3, 1000, 137280}, {152, 4, 1000, 121408}, {152, 5, 1000, 109862},
        {152, 6, 233, 100874},  {152, 7, 9162, 8576},   {152, 7, 7950, 20000},  {152, 8, 9175, 10416},
        {152, 8, 8264, 8264},   {152, 9, 1, 80135},     {152, 10, 259, 74252},  {152, 11, 3018, 59694},
        {152, 12, 9162, 5226},  {152, 13, 103, 61991},  {152, 14, 870, 57732},  {152, 15, 1734, 51268},
        {152, 16, 9215, 392},   {152, 16, 7479, 7479},  {304, 2, 961, 155808},  {304, 3, 961, 134890},
        {304, 4, 1000, 119232}, {304, 5, 961, 107968},  {304, 6, 63, 99466},    {304, 7, 9110, 6921},
        {304, 8, 9175, 8888},   {304, 9, 1, 78741},     {304, 10, 870, 72070},  {304, 11, 2992, 58513},
        {304, 12, 9032, 4197},  {304, 13, 1, 61006},    {304, 14, 961, 56585},  {304, 15, 1825, 50193},
        {304, 16, 8720, 4}};
    const long long plan_bytes = (long long)((sizeof(Plan) + 255) / 256 * 256);
    for (const auto& c : cases) {
        ProbIn in{};
        in.m = (int32_t)c[1];
        in.n2 = c[2];
        in.n_r = (int32_t)c[3];
        in.mode = MODE_SELECT;
        const long long need = plan_bytes + layout_problem(in, (int)c[0], nullptr, nullptr);
        if (need > (long long)kNoallocBytes) {
            std::printf("FAIL %lld CTAs, m = %lld, %lld points, %lld references: %lld bytes\n", c[0], c[1], c[2], c[3],
                        need);
            return 1;
        }
    }
    std::printf("noalloc ok\n");
    return 0;
}
