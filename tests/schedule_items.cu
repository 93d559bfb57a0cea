// The distribution of work units over CTA pairs, printed for tests/test_schedule.py.  Input: lines "units ksteps pairs
// balanced"; output per line: "plan full_waves tail_units tail_pairs", then "pair unit ks0 ks1" for every work item, "end".
// Where nothing is cut, both functions that give an item have to agree.
#include <cstdio>

#include "../paper_2505_07004_b200/csrc/gq_pipeline.cuh"

int main()
{
    int units, ksteps, pairs, balanced;
    while (std::scanf("%d %d %d %d", &units, &ksteps, &pairs, &balanced) == 4) {
        const gq::Schedule s = gq::plan_schedule(units, ksteps, pairs, balanced != 0);
        std::printf("plan %d %d %d\n", s.full_waves, s.tail_units, s.tail_pairs);
        for (int p = 0; p < pairs; ++p)
            for (int it = 0;; ++it) {
                gq::WorkItem w, v;
                const bool more = gq::work_item(s, p, it, w);
                if (!balanced && (gq::whole_unit(s, p, it, v) != more || (more && (v.unit != w.unit || v.ks0 != w.ks0 || v.ks1 != w.ks1)))) return 1;
                if (!more) break;
                std::printf("%d %d %d %d\n", p, w.unit, w.ks0, w.ks1);
            }
        std::printf("end\n");
    }
    return 0;
}
