"""Walking a row's slots U at a time with 32-bit numbers (gr_slots.cuh): every
slot once and in order, also in rows that end at 2^32 - 2, the last slot of a
graph of 2^31 - 1 edges, where `j += U` and `j + u < e` wrap; and plain steps
where slots_step_fits allows them."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
DRIVER = r"""
#include <cstdio>
#include <initializer_list>
#include "gr_slots.cuh"
int main() {
    long bad = 0;
    for (unsigned U = 1; U <= 8; ++U)
        for (unsigned e : {0u, 40u, 0x7fffffffu, 0xfffffffdu, 0xfffffffeu})
            for (unsigned len = 0; len <= 40 && len <= e; ++len) {
                unsigned want = e - len, rounds = 0;
                for (gr::SlotRun r(e - len, e); r.left && rounds <= len; r.next(U), ++rounds)
                    for (unsigned u = 0; u < U; ++u)
                        if (r.has(u)) bad += r.at + u != want++;
                bad += want != e || rounds != (len + U - 1) / U;
                // plain steps, where the rule allows them
                if (!gr::slots_step_fits(e, U)) continue;
                want = e - len, rounds = 0;
                for (unsigned j = e - len; j < e && rounds <= len; j += U, ++rounds)
                    for (unsigned u = 0; u < U; ++u)
                        if (j + u < e) bad += j + u != want++;
                bad += want != e || rounds != (len + U - 1) / U;
            }
    bad += !gr::slots_step_fits(0xfffffffeull, 2) || gr::slots_step_fits(0xfffffffeull, 4);
    printf("%ld\n", bad);
    return 0;
}
"""


def test_rows_at_the_end_of_the_slot_range(tmp_path):
    src, exe = tmp_path / "slots.cpp", tmp_path / "slots"
    src.write_text(DRIVER)
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", os.path.join(ROOT, "paper_1812_08942_gb300", "csrc"), "-o",
                    str(exe), str(src)], check=True)
    assert subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.strip() == "0"
