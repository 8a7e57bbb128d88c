"""A batched workspace whose memory was used for something else in between: the next batch at the
same address, with the same problems and pointers, must copy its tables again after it was
prepared (donof_prepare_B_batched), grouped and as a graph replay."""
import numpy as np
import pytest

import synth
from test_gpu_batch import KEYS, _instances, _run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("graph", [False, True])
def test_tables_are_copied_again_after_prepare(graph):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2004_06142_gb300.build as b
    b.build()
    import paper_2004_06142_gb300 as dn
    cprobs, tens, _ = _instances(synth.batch_problems(4), 1)
    batch = dn.Batch(cprobs, tens)
    flags = dn.BATCH_BACKWARD | (dn.BATCH_GRAPH if graph else 0)
    batch.prepare()
    want = _run(batch, tens, flags)
    batch.ws.zero_()  # the memory given back and taken by others (all tables gone)
    batch.prepare()
    got = _run(batch, tens, flags)
    assert batch.status() == 0
    for w, g in zip(want, got):
        for k in KEYS:
            np.testing.assert_array_equal(w[k], g[k], err_msg=k)
