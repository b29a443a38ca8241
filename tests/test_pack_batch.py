"""Context.pack_batch: the batch layout of mixed inputs (dtypes, orders,
strides, sequences, empty matrices and batches) against a plain loop."""
import numpy as np
import pytest


def _plain(items):
    mats, offs, rows, cols, mults, roff, coff, at = [], [], [], [], [], [], [], 0
    for a, M, N in items:
        a = np.asarray(a, np.complex128)
        offs.append(at)
        at += a.size
        rows.append(a.shape[0])
        cols.append(a.shape[1])
        mats += list(a.reshape(-1))
        roff.append(len(mults))
        mults += [int(x) for x in np.asarray(M).reshape(a.shape[0])]
        coff.append(len(mults))
        mults += [int(x) for x in np.asarray(N).reshape(a.shape[1])]
    return (np.asarray(mats or [0], np.complex128), np.asarray(offs, np.int64), np.asarray(rows, np.int32),
            np.asarray(cols, np.int32), np.asarray(mults or [0], np.int32), np.asarray(roff, np.int64),
            np.asarray(coff, np.int64))


def test_pack_batch_layout(bslib):
    g = np.random.default_rng(5)
    z = g.standard_normal((4, 6)) + 1j * g.standard_normal((4, 6))
    items = [(z, [1, 2, 2, 1], np.ones(6, np.int64)), (np.asfortranarray(z), np.array([1, 2, 2, 1]), [1] * 6),
             (z[::-1, ::2], (1, 1, 1, 0), [1, 1, 1]), (z.astype(np.complex64), np.array([[6], [0], [0], [0]]), np.ones(6)),
             (z.real, [3, 1, 1, 1], [1] * 6), (z.astype(">c16"), [3, 1, 1, 1], [1] * 6), ([[1, 2j], [3, 4]], [1, 1], [1, 1]),
             (np.zeros((0, 0)), [], []), (z[:1, :1], [1], [1])]
    for batch in (items, items[::-1], items[2:3], []):
        got, ref = bslib.Context.pack_batch(batch), _plain(batch)
        for x, y in zip(got, ref):
            assert x.dtype == y.dtype and x.flags.c_contiguous and np.array_equal(x, y)
    for bad in [(z[0], [1], [1]), (z, [1, 1, 1], [1] * 6), (z, [1, 1, 1, 1], [1] * 5)]:
        with pytest.raises(ValueError):
            bslib.Context.pack_batch([bad])
