"""FP64 sigmas of spaces with more strings than an SM's shared memory takes
(nstr + npair > 28,160) are refused with OOM before any work: no launch, no
workspace."""
import pytest
import torch

import paper_2307_10675_gb300 as ifci
from paper_2307_10675_gb300 import _capi

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda", 0)


def test_refused_before_any_work():
    n, m = 31, 4   # 31,465 strings
    npair = n * (n + 1) // 2
    h1 = torch.zeros((n, n), dtype=torch.float64, device=DEV)
    eri = torch.zeros((npair, npair), dtype=torch.float64, device=DEV)
    with ifci.Handle(0, 0) as h:
        t = ifci.ifci_build_strings(h, n, m)
        c = torch.empty(t.nstr * t.nstr, dtype=torch.float64, device=DEV)
        launches, held = h.launches(), h.workspace_bytes()
        with pytest.raises(ifci.IfciError) as err:
            ifci.ifci_sigma(h, t, h1, eri, c)
        assert err.value.code == _capi.IFCI_ERR_OOM
        assert (h.launches(), h.workspace_bytes()) == (launches, held)
