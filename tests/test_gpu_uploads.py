"""What an upload reports of a matrix with several faults."""

import numpy as np
import pytest

from synth import Bsr

pytestmark = pytest.mark.gpu


def test_an_unsymmetric_pattern_is_reported_before_its_values():
    from paper_2009_03551_gb300 import build as b
    b.build()
    from paper_2009_03551_gb300 import rdm
    va = np.tile(np.eye(4), (3, 1, 1))
    va[0, 1, 1] = np.nan
    m = Bsr(2, 4, 8, np.array([0, 2, 3], dtype=np.int32), np.array([0, 1, 1], dtype=np.int32), va)
    sol = rdm.Solver(0)
    with pytest.raises(rdm.RdmError, match="pattern is not symmetric") as e:
        rdm.rdm_upload_h0(sol.h, 0, m, 2)
    assert e.value.code == rdm.RDM_EBADBSR
    sol.close()
