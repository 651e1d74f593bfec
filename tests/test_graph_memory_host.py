"""Host memory of a graph's neighbourhood tables, in a process with a limit on its address space (no GPU
needed: gna_ball_sizes_host builds the same tables as gna_graph_create)."""
import subprocess
import sys
import textwrap

import pytest

from paper_2011_12453_gb300 import build as B


def _run(n_sites, edges, layers, limit_mb):
    code = f"""
    import resource
    import numpy as np
    from paper_2011_12453_gb300 import gna
    gna.lib()
    e = np.array({edges}, dtype=np.int32)
    used = int(open("/proc/self/statm").read().split()[0]) * resource.getpagesize()
    resource.setrlimit(resource.RLIMIT_AS, (used + ({limit_mb} << 20),) * 2)
    try:
        print("balls", int(gna.ball_sizes_host({n_sites}, e, {layers})[:, -1].max()))
    except gna.GnaError as x:
        print("status", x.status)
    """
    r = subprocess.run([sys.executable, "-c", textwrap.dedent(code)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return r.stdout.strip()


@pytest.fixture(scope="module", autouse=True)
def built():
    B.build()


def test_first_bond_of_a_hub_does_not_set_the_reservation():
    # a star of 500 leaves, then a ring of 3500 sites: 500 balls of 501 rows and 3500 of 4; every bond as
    # large as the first one would take some 80 MB, the tables themselves 10
    assert _run(4001, "[(0, v) for v in range(1, 501)] + [(501 + i, 501 + (i + 1) % 3500) for i in range(3500)]", 1,
                60) == "balls 501"


def test_tables_beyond_the_memory_are_refused():
    # 300 sites, all joined: 44850 bonds of 300 rows with 299 neighbours each
    assert _run(300, "[(i, j) for i in range(300) for j in range(i)]", 1, 500) == "status -6"
