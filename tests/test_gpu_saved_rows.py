"""Operand rows in a saved index: their own columns, whatever pitch they have on the
device.  Each array stands in the file as a record (id, 0, bytes, contents); 20 and 21
are the users' hi and lo operands, 24 and 25 the items'."""
import struct

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

rkr = pytest.importorskip("paper_2504_13446_gb300")


def _records(path, n, d):
    raw = open(path, "rb").read()
    at = raw.index(struct.pack("<IIQ", 1, 0, n * d * 4))    # the users' rows come first
    out = {}
    while at < len(raw) - 8:                                # a checksum ends the file
        key, _, size = struct.unpack_from("<IIQ", raw, at)
        out[key] = np.frombuffer(raw, np.uint8, size, at + 16)
        at += 16 + size
    assert at == len(raw) - 8
    return out


@pytest.mark.parametrize("d", [9, 30, 40, 70, 140, 200])
def test_operand_records_hold_no_padding(tmp_path, d):
    rng = np.random.default_rng(d)
    n, m, kp = 300, 200, (d + 15) // 16 * 16
    U = rng.standard_normal((n, d)).astype(np.float32)
    P = rng.standard_normal((m, d)).astype(np.float32)
    path = str(tmp_path / "index")
    with rkr.Index(U, P, tau=20, omega=3, s=10, exact_table=False) as idx:
        idx.save(path)
        order = idx.export("perm")
    rec = _records(path, n, d)
    for rows, hi, lo in ((U, 20, 21), (P[order], 24, 25)):
        bits = rows.view(np.uint32).astype(np.uint64)
        top = ((bits + 0x7fff + ((bits >> 16) & 1)) >> 16).astype(np.uint16)   # to nearest even
        rest = rows - (top.astype(np.uint32) << 16).view(np.float32)
        bits = rest.view(np.uint32).astype(np.uint64)
        low = ((bits + 0x7fff + ((bits >> 16) & 1)) >> 16).astype(np.uint16)
        for key, want in ((hi, top), (lo, low)):
            assert len(rec[key]) == len(rows) * kp * 2, key
            got = rec[key].view(np.uint16).reshape(len(rows), kp)
            assert np.array_equal(got[:, :d], want) and not got[:, d:].any(), key
