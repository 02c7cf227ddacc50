"""What a profile says of its next scan (configuration, table memory,
footprint) against the launch that a scan makes and the device memory that
its tables take."""
import ctypes

import numpy as np
import pytest

from paper_1707_09683_gb300 import synth

pytestmark = pytest.mark.gpu

USED_MEM_CURRENT = 7     # attribute of a memory pool


class Pool:
    """Bytes in use of the device's stream-ordered pool, from which tables come."""

    def __init__(self):
        self.cu = ctypes.CDLL("libcuda.so.1")
        self.pool = ctypes.c_void_p()
        assert self.cu.cuDeviceGetDefaultMemPool(ctypes.byref(self.pool), 0) == 0

    def used(self):
        import torch

        torch.cuda.synchronize()
        v = ctypes.c_uint64()
        assert self.cu.cuMemPoolGetAttribute(self.pool, USED_MEM_CURRENT, ctypes.byref(v)) == 0
        return v.value

    def granularity(self):
        before, p = self.used(), ctypes.c_uint64()
        assert self.cu.cuMemAllocAsync(ctypes.byref(p), ctypes.c_size_t(1), None) == 0
        g = self.used() - before
        assert self.cu.cuMemFreeAsync(p, None) == 0
        return g


@pytest.mark.parametrize("f16", [False, True])
@pytest.mark.parametrize("M,config,shared", [
    (48, None, False), (100, None, False), (300, (4, 38), False), (400, None, False), (448, None, False),
    (449, None, False), (640, None, True), (640, (16, 20), False), (1000, None, False), (1280, None, False),
    (1281, None, False), (2405, None, False)])
def test_configuration_and_footprint_of_the_next_scan(M, config, shared, f16):
    import torch

    from paper_1707_09683_gb300 import mpf

    rng = np.random.default_rng(M)
    rec, dbh = synth.make_profile(M, rng), synth.make_database(200, 100, 10, 400, rng)
    ctx = mpf.Context(0)
    db = mpf.Database(ctx, dbh.residues, dbh.offsets, dbh.lengths)
    out = [torch.zeros(db.n_seqs, dtype=t, device="cuda") for t in (torch.uint8, torch.uint8, torch.float32)]
    pool = Pool()
    for filt, scan in ((mpf.MSV, mpf.msv_scan), (mpf.SSV, mpf.ssv_scan)):
        p = mpf.Profile(ctx, rec)
        if config:
            p.set_config(filt, *config)
        if shared:
            p.set_table_memory(filt, mpf.TABLE_SHARED)
        if f16:
            p.set_arith(filt, mpf.ARITH_F16)
        ctx.sync()
        g, before = pool.granularity(), pool.used()
        scan(ctx, p, db, *out)
        ctx.sync()
        smem, tables = p.footprint(filt)
        held = pool.used() - before
        assert tables <= held < tables + 3 * g, (filt, held, tables)   # at most three tables, each rounded up
        plan = mpf.Plan(ctx, filt, [p], db, *out)
        (group,) = plan.groups()
        assert p.get_config(filt) == (group["lanes"], group["words"])
        assert p.get_table_memory(filt) == group["table"]
        if group["table"] == mpf.TABLE_TENSOR:
            assert smem > 100 << 10                                     # one block per SM
        plan.close()
        p.close()
    db.close()
