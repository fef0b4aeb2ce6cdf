"""An export only reads: exports of one table from several host threads at once
all give what one alone gives, words and slots, whatever parts the words are
converted in."""
import threading

import numpy as np
import pytest

from paper_1605_05236_gb300 import ck, inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bins,B,ghost", [(2, 4, False), (100_003, 8, False), (1 << 15, 4, True), ((1 << 22) + 5, 4, False)])
def test_exports_side_by_side(bins, B, ghost):
    n = inputs.load_target(bins * B, 0.75 if bins == 2 else 0.93)
    keys, _ = inputs.distinct_keys(n, 13)
    t = ck.CuckooTable(bins, B, 2, ck.QUEUE | (ck.GHOST if ghost else 0), seed=4)
    t.insert(ck.as_u32_tensor(keys), ck.as_u32_tensor(inputs.values_for(keys)))
    slots, meta = t.export()
    bad = []

    def reader():
        for _ in range(12 if bins < 1 << 20 else 2):
            s, m = t.export()
            if not (np.array_equal(s, slots) and np.array_equal(m, meta)):
                bad.append(int((m != meta).sum()))

    threads = [threading.Thread(target=reader) for _ in range(4)]
    for x in threads:
        x.start()
    for x in threads:
        x.join()
    assert bad == []
    assert np.array_equal(t.export()[1], meta)
    t.close()
