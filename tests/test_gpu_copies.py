"""Copies between the caller's arrays and the arrays of a batch or a server."""
import numpy as np
import pytest

import abilu_inputs as gen

pytestmark = pytest.mark.gpu

OPTS = dict(rtol=1e-6, build_sweeps=3, apply_sweeps_lower=3, apply_sweeps_upper=3, mode="sync")


def _systems(count):
    return [gen.small_system(3 + k % 5, 4 + k, seed=k, cfl=10.0 * (k + 1)) for k in range(count)]


def _place(v, where):
    """v's values in device memory, device memory 8 bytes off a 16-byte boundary,
    or pinned host memory."""
    import torch
    t = torch.from_numpy(np.ascontiguousarray(v))
    if where == "device":
        return t.cuda()
    if where == "pinned":
        return t.pin_memory()
    buf = torch.empty(t.numel() + 1, dtype=torch.float64, device="cuda")
    buf[1:] = t.flatten()
    out = buf[1:].view(t.shape)
    assert out.data_ptr() % 16 == 8
    return out


def _server(systems):
    import torch
    import paper_1912_00539_gb300.abilu as ab
    srv = ab.NativeServer(64 * len(systems) + sum(s.n for s in systems), sum(s.nnzb + 128 for s in systems),
                          len(systems), "f32")
    return srv, [srv.add(torch.from_numpy(s.rowptr).cuda(), torch.from_numpy(s.colind).cuda()) for s in systems]


def _alone(systems):
    import torch
    out = []
    for s in systems:
        srv, ids = _server([s])
        x = torch.zeros((s.n, 4), dtype=torch.float64, device="cuda")
        srv.step(ids, [_place(s.vals, "device")], [_place(s.b, "device")], [x], **OPTS)
        out.append(x.cpu().numpy())
    return out


@pytest.mark.parametrize("count", [1, 12, 13, 15])
def test_server_step_from_every_kind_of_memory(count):
    """Two arrays a system: below, at and above the copy kernel's 24 arrays, a
    second launch half full; the same values as each system alone, whatever
    memory the arrays lie in."""
    kinds = ("device", "off", "pinned")
    systems = _systems(count)
    want = _alone(systems)
    for shift in range(4):   # 3: device memory throughout
        place = lambda k: kinds[(k + shift) % 3] if shift < 3 else "device"
        srv, ids = _server(systems)
        A = [_place(s.vals, place(k)) for k, s in enumerate(systems)]
        b = [_place(s.b, place(k + 1)) for k, s in enumerate(systems)]
        x = [_place(np.zeros((s.n, 4)), place(k + 2)) for k, s in enumerate(systems)]
        srv.step(ids, A, b, x, **OPTS)
        for k in range(count):
            np.testing.assert_array_equal(x[k].cpu().numpy(), want[k])


def test_server_step_overlapping_results_in_the_order_given():
    """Results written over one another: the later system's values remain, both
    through the kernel (equal addresses) and through a copy of its own (8 bytes
    further)."""
    import torch
    s = gen.small_system(9, 7, seed=3)
    systems = [s, gen.small_system(9, 7, seed=4)]
    want = _alone(systems)
    nv = 4 * s.n
    for off in (0, 1, 2):
        for swap in (False, True):
            buf = torch.zeros(nv + 2, dtype=torch.float64, device="cuda")
            x = [buf[:nv].view(s.n, 4), buf[off:off + nv].view(s.n, 4)]
            if swap:
                x.reverse()
            srv, ids = _server(systems)
            srv.step(ids, [_place(t.vals, "device") for t in systems], [_place(t.b, "device") for t in systems],
                     x, **OPTS)
            first, last = (off, 0) if swap else (0, off)
            exp = np.zeros(nv + 2)
            exp[first:first + nv] = want[0].ravel()
            exp[last:last + nv] = want[1].ravel()
            np.testing.assert_array_equal(buf.cpu().numpy(), exp)


@pytest.mark.parametrize("where", ["device", "off"])
def test_batch_set_and_get(where):
    import torch
    import paper_1912_00539_gb300.abilu as ab
    systems = _systems(3)
    want = _alone(systems)
    ba = ab.Batch([(torch.from_numpy(s.rowptr).cuda(), torch.from_numpy(s.colind).cuda()) for s in systems], "f32")
    for k, s in enumerate(systems):
        ba.set_system(k, _place(s.vals, where), _place(s.b, where))
    ba.solve(**OPTS)
    for k, s in enumerate(systems):
        x = _place(np.full((s.n, 4), np.nan), where)
        ba.solution(k, x)
        np.testing.assert_array_equal(x.cpu().numpy(), want[k])
