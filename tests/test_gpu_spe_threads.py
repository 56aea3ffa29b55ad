"""spe_table from several threads at once: graphs of different sizes ask the same kernels for different amounts
of shared memory, and one call must not change what another's launches may ask for."""
import threading

import numpy as np
import pytest

from paper_2410_05911_gb300 import aecct as A
from paper_2410_05911_gb300 import inputs as I

pytest.importorskip("torch")


@pytest.mark.gpu
def test_tables_of_small_and_large_graphs_on_two_threads():
    graphs = [I.make_code("hamming7_4").H, I.ldpc_regular_code(600, 300, 3, 6, seed=4).H]
    params = [I.spe_params(H, 8, seed=2) for H in graphs]
    refs = [A.spe_table(H, p) for H, p in zip(graphs, params)]
    stop, faults = threading.Event(), []

    def small():
        while not stop.is_set():
            try:
                if not np.array_equal(A.spe_table(graphs[0], params[0]), refs[0]):
                    faults.append("small graph: another table")
            except Exception as e:  # noqa: BLE001
                faults.append(f"small graph: {e}")

    threads = [threading.Thread(target=small) for _ in range(3)]
    for t in threads:
        t.start()
    try:
        for _ in range(40):
            assert np.array_equal(A.spe_table(graphs[1], params[1]), refs[1])
    finally:
        stop.set()
        for t in threads:
            t.join()
    assert not faults, faults[0]
