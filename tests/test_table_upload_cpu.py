"""The small device tables of a plan are collected from host vectors and copied later in one go; a large one, which is not
staged, must not depend on what becomes of the vector it was added from.  Compiled with g++, malloc for the device."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

HARNESS = r"""
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include "table_upload.hpp"
struct Rec { int32_t v[84]; };   // 336 bytes, the size of a band's record and radix plan
static std::vector<Rec> records(int n, int seed) {
    std::vector<Rec> r(n);
    for (int i = 0; i < n; ++i) for (int j = 0; j < 84; ++j) r[i].v[j] = seed + 84 * i + j;
    return r;
}
static int check(const Rec *p, int n, int seed) {
    if (!p) return n == 0 ? 0 : 1;
    for (int i = 0; i < n; ++i) for (int j = 0; j < 84; ++j) if (p[i].v[j] != seed + 84 * i + j) return 1;
    return 0;
}
int main() {
    // tables below the limit for large ones, just above it, far above it
    const int counts[] = {0, 3, 3120, 3121, 40000};
    Rec *local[5], *lvalue[5];
    int calls = 0, bad = 0;
    cqt::TableUpload up([&](const void *src, size_t n, void *&dev) {
        ++calls;
        dev = std::malloc(n);
        std::memcpy(dev, src, n);
        return true;
    });
    std::vector<Rec> reused;
    for (int i = 0; i < 5; ++i) {
        {
            std::vector<Rec> items = records(counts[i], 1000 * i);   // gone before finish()
            up.add(local[i], items);
        }
        reused = records(counts[i], 500000 + i);                     // overwritten before finish()
        up.add(lvalue[i], reused);
    }
    reused.assign(50000, Rec{});
    std::vector<std::vector<Rec>> churn;
    for (int n : counts) churn.push_back(records(n, -1));
    const bool ok = up.finish();
    for (int i = 0; i < 5; ++i) bad += check(local[i], counts[i], 1000 * i) + check(lvalue[i], counts[i], 500000 + i);
    // a failing copy ends the upload: nothing is set after it
    int n_fail = 0;
    cqt::TableUpload fails([&](const void *, size_t, void *&dev) { dev = std::malloc(1); return ++n_fail < 2; });
    Rec *p = nullptr, *q = nullptr, *r = nullptr;
    fails.add(p, records(10, 0));
    fails.add(q, records(4000, 0));
    fails.add(r, records(4000, 0));
    const bool failed = !fails.finish() && q && !r && !p && n_fail == 2;
    std::printf("%d %d %d %d\n", (int)ok, bad, calls, (int)failed);
    return 0;
}
"""


def test_large_tables_survive_the_vector_they_were_added_from(tmp_path):
    src, exe = tmp_path / "check.cpp", tmp_path / "check"
    src.write_text(HARNESS)
    subprocess.run(["g++", "-O1", "-g", "-std=c++17", "-fsanitize=address,undefined", "-static-libasan", "-fno-sanitize-recover=all",
                    "-I", os.path.join(ROOT, "paper_2609_29119_b200", "csrc"), str(src), "-o", str(exe)], check=True)
    res = subprocess.run([str(exe)], capture_output=True, text=True, env={**os.environ, "ASAN_OPTIONS": "detect_leaks=0"})
    assert res.returncode == 0, res.stderr
    # the small tables in one copy, four large ones in one each
    assert res.stdout.split() == ["1", "0", "5", "1"], res.stdout
