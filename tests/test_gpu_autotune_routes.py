"""What the autotuner varies is what its table's users run: tile settings where Householder tiles
run (by themselves or behind the workspace-free entry), none where only the exact pass does."""
import ctypes
import json

import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,n,tiles", [(1 << 16, 2, True), (1 << 17, 8, True), (1 << 16, 40, False), (1 << 15, 17, False)])
def test_settings_are_those_of_the_tiles(tmp_path, m, n, tiles):
    import torch

    import paper_2603_20889_gb300 as q

    L = q.load_library()
    nb = L.ql_autotune_workspace_bytes(m, n, q.QL_F64)
    ws = torch.empty(nb, dtype=torch.uint8, device="cuda")
    meth, ms = ctypes.c_int32(-1), ctypes.c_double(0.0)
    assert L.ql_autotune(m, n, q.QL_F64, 1e9, ws.data_ptr(), nb, q._stream_ptr(), ctypes.byref(meth),
                         ctypes.byref(ms)) == q.QL_OK
    assert meth.value == q.QL_TSQR and ms.value > 0.0
    out = tmp_path / "table.json"
    assert L.ql_autotune_save(str(out).encode()) == q.QL_OK
    e = [t for t in json.loads(out.read_text())["entries"]
         if (t["dtype"], t["n"], 1 << t["mlog2"], t["kbucket"]) == (0, n, m, 1)]
    assert len(e) == 1
    if tiles:
        assert e[0]["ctas"] in (1, 2, 4)
    else:
        assert (e[0]["ctas"], e[0]["variant"], e[0]["arity"]) == (0, 0, 0)
