// tune_file.h -- the file of timed y-pass forms (ISOFFT_TUNE_FILE): JSON with a
// digest of the pass code that was timed and the entries
// [dtype, My, Kx, Ny, Nz, sm, forward, inverse].
#pragma once
#include <stdio.h>

#include <algorithm>
#include <map>
#include <utility>
#include <vector>

namespace isofft {

struct TuneKey {
    int v[6];
    bool operator<(const TuneKey &o) const { return std::lexicographical_compare(v, v + 6, o.v, o.v + 6); }
};
typedef std::map<TuneKey, std::pair<int, int>> TuneMap;

// Adds the entries of `path` to `map`.  Only those of a file that names this
// `code`: a form that was the fastest of other kernels, or on another workspace
// layout, may be far from it here.
inline void tune_file_read(const char *path, long code, int forms, TuneMap &map)
{
    FILE *f = fopen(path, "r");
    if (!f) return;
    // the integers of the file in order: the digest, then eight per entry
    std::vector<long> nums;
    long cur = 0;
    bool in = false, neg = false;
    for (int ch; (ch = fgetc(f)) != EOF;) {
        if (ch >= '0' && ch <= '9') {
            cur = cur * 10 + (ch - '0');
            in = true;
        } else {
            if (in) nums.push_back(neg ? -cur : cur);
            neg = ch == '-';
            cur = 0;
            in = false;
        }
    }
    if (in) nums.push_back(neg ? -cur : cur);
    fclose(f);
    if (nums.size() % 8 != 1 || nums[0] != code) return;
    for (size_t i = 1; i + 8 <= nums.size(); i += 8) {
        TuneKey k;
        for (int j = 0; j < 6; ++j) k.v[j] = (int)nums[i + j];
        const int a = (int)nums[i + 6], b = (int)nums[i + 7];
        if (a >= 0 && a < forms && b >= 0 && b < forms) map[k] = {a, b};
    }
}

inline void tune_file_write(const char *path, long code, const TuneMap &map)
{
    FILE *f = fopen(path, "w");
    if (!f) return;
    fprintf(f, "{\"code\": %ld,\n\"y_pass_forms\": [\n", code);
    size_t i = 0;
    for (const auto &kv : map) {
        const int *v = kv.first.v;
        fprintf(f, "  [%d, %d, %d, %d, %d, %d, %d, %d]%s\n", v[0], v[1], v[2], v[3], v[4], v[5], kv.second.first,
                kv.second.second, ++i < map.size() ? "," : "");
    }
    fprintf(f, "]}\n");
    fclose(f);
}

}  // namespace isofft
