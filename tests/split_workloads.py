"""Steps whose last round of items is split by key range on 76 CTA pairs, so
that parts are written and merged: the workload, and per cache type (E4M3 or
not) the numbers of parts that items are split into.  test_host_create checks
these without a GPU, test_gpu_split runs them."""
import workloads


def _w(name, heads, dim, reqs):
    return workloads.Workload(f"split_{name}_d{dim}", heads, dim, tuple(workloads.Request(*r) for r in reqs), 41)


def cases(dim):
    return [
        (_w("eight", 2, dim, [(5, 7, 230, 8300)]), [8], [8]),
        (_w("six", 12, dim, [(5, 7, 230, 6000)]), [6], [6]),
        # parts of two counts in one launch, tasks of 43, 54 and 256 rows
        (_w("uneven", 3, dim, [(0, 10, 300, 2000), (0, 3, 40, 5000)]), [3, 7], [4, 8]),
        # three tasks a head, the last of 18 rows
        (_w("short_tail", 5, dim, [(0, 30, 500, 3000)]), [4], [4]),
        # more items than the merge's first form takes
        (_w("many", 44, dim, [(0, 7, 100, 9000)]), [3], [3]),
    ]


NAMES = ["eight", "six", "uneven", "short_tail", "many"]
