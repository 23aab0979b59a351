"""The memory kept of freed join tables goes back to the device on request, for
other allocators of the process, while contexts live and work goes on."""
import pytest

from paper_2601_19911_gb300 import olap

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_trim_frees_kept_tables():
    keys = torch.randint(-(1 << 62), 1 << 62, (1 << 21,), device="cuda")
    with olap.Context(0) as ctx:
        olap.device_trim(0)
        before = torch.cuda.mem_get_info()[0]
        t = ctx.join_build(keys)
        table = t.info()["n_buckets"] * 32
        t.free()
        assert before - torch.cuda.mem_get_info()[0] >= table
        assert olap.device_trim(0) >= table
        assert before - torch.cuda.mem_get_info()[0] < (8 << 20)
        assert olap.device_trim(0) == 0
        t = ctx.join_build(keys)                 # live tables are not touched
        assert olap.device_trim(0) == 0
        out = torch.empty((1 << 21, 2), dtype=torch.int32, device="cuda")
        assert ctx.join_probe(t, keys, out=out).shape[0] == 1 << 21
        t.free()
    with pytest.raises(olap.OlapError):
        olap.device_trim(1000)
