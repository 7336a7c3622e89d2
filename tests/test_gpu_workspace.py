"""Workspaces through the C ABI: a call takes the bytes that its query asks for,
wherever they start, writes nothing beside them, and gives the result it gives
in a workspace of its own."""
import ctypes

import numpy as np
import pytest

import meshgen as M

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

O3 = (-0.5, -0.5, -0.5)
RES = 70


@pytest.fixture(scope="module")
def ldni():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1009_0794_gb300 as pkg
    pkg._lib.load()
    return pkg


class Call:
    """One entry point with its inputs; run(ws, bytes) fills new outputs and
    returns them."""

    def __init__(self, ldni, kind):
        from paper_1009_0794_gb300 import _lib
        self.ldni, self.lib, self.kind, self._lib = ldni, _lib.load(), kind, _lib
        self.grid = ldni.Grid.cube(O3, 1.0, RES)
        v, t = M.icosphere(7, r=0.33, noise=0.04, seed=3)
        self.v, self.t = torch.from_numpy(v).cuda(), torch.from_numpy(t).cuda()
        self.images = ldni.sample(self.v, self.t, self.grid, "all")
        self.n = [L.n for L in self.images]
        self.inside = ldni.classify_nodes(self.images)
        other = ldni.sample(*M.torus(0.25, 0.1, 24, 12), self.grid, "all")
        self.parts = [[A, B] for A, B in zip(self.images, other)]
        self.nn = (ctypes.c_int64 * 3)(*self.n)
        self.r = 1.4 / RES

    def _c(self, Ls):
        return (self._lib.Layers * len(Ls))(*[L.c() for L in Ls])

    def _items(self, outs):
        it = (self._lib.BatchItem * 1)()
        it[0].verts, it[0].tris, it[0].nv, it[0].nt = self.v.data_ptr(), self.t.data_ptr(), len(self.v), len(self.t)
        it[0].grid = self.grid.c()
        for a in range(3):
            it[0].out[a] = outs[a].c()
        return it

    def outs(self):
        room = [4 * n + 64 for n in self.n]
        return [self.ldni.empty_layers(self.grid, a, room[a]) for a in range(3)]

    def bytes(self):
        sz, k, lib = ctypes.c_size_t(0), self.kind, self.lib
        nv, nt = len(self.v), len(self.t)
        rc = {"sample": lambda: lib.ldni_sample_workspace_size(nv, nt, RES, 3, ctypes.byref(sz)),
              "binned": lambda: lib.ldni_sample_binned_workspace_size(nv, nt, RES, 3, ctypes.byref(sz)),
              "learned": lambda: lib.ldni_sample_learned_workspace_size(nv, nt, RES, 3, 20000, ctypes.byref(sz)),
              "batch": lambda: lib.ldni_sample_batch_workspace_size(ctypes.byref(self._items(self.outs())), 1, ctypes.byref(sz)),
              "chain": lambda: lib.ldni_union_chain_workspace_size(RES, 3, ctypes.byref(sz)),
              "nodes": lambda: lib.ldni_classify_nodes_workspace_size(RES, ctypes.byref(sz)),
              "contour": lambda: lib.ldni_contour_workspace_size(RES, 60000, ctypes.byref(sz)),
              "offset": lambda: lib.ldni_offset_workspace_size(self.nn, RES, self.r, 1.0, ctypes.byref(sz))}[k]()
        assert rc == 0
        return sz.value

    def run(self, ws, nbytes):
        k, lib, g = self.kind, self.lib, self.grid.c()
        outs, info = self.outs(), self.ldni.new_info()
        oc = self._c(outs)
        mesh = (self.v.data_ptr(), len(self.v), self.t.data_ptr(), len(self.t), ctypes.byref(g), 3)
        tail = (info.data_ptr(), ws, nbytes, None)
        torch.cuda.synchronize()
        if k in ("sample", "binned"):
            rc = lib.ldni_sample(*mesh, {"sample": 0, "binned": 2}[k], oc, *tail)
        elif k == "learned":
            rc = lib.ldni_sample_learned(*mesh, None, 2, 1, 20000, oc, info.data_ptr(), None, ws, nbytes, None)
        elif k == "batch":
            it = self._items(outs)
            dev = torch.frombuffer(bytearray(bytes(memoryview(it))), dtype=torch.uint8).cuda()
            torch.cuda.synchronize()
            rc = lib.ldni_sample_batch(dev.data_ptr(), ctypes.byref(it), 1, *tail)
            torch.cuda.synchronize()
        elif k == "chain":
            host = self._c([p for ps in self.parts for p in ps])
            dev = torch.frombuffer(bytearray(bytes(memoryview(host))), dtype=torch.uint8).cuda()
            torch.cuda.synchronize()
            rc = lib.ldni_union_chain(dev.data_ptr(), host, 2, 3, ctypes.byref(g), 0.0, oc, *tail)
            torch.cuda.synchronize()
        elif k == "nodes":
            words = torch.zeros_like(self.inside)
            rc = lib.ldni_classify_nodes(self._c(self.images), ctypes.byref(g), words.data_ptr(), *tail)
        elif k == "contour":
            cells = torch.zeros(60000, self.ldni.CELL_DTYPE.itemsize, dtype=torch.uint8, device="cuda")
            rc = lib.ldni_contour_cells(self._c(self.images), ctypes.byref(g), self.inside.data_ptr(), 60000,
                                        cells.data_ptr(), 60000, *tail)
        else:
            rc = lib.ldni_offset(self._c(self.images), self.nn, ctypes.byref(g), self.r, 0, 0.0, oc, *tail)
        torch.cuda.synchronize()
        assert rc == 0
        h = info.tolist()
        assert h[3] & 0xFFFFFFFF == 0
        if k == "nodes":
            return [words]
        if k == "contour":
            return [cells, info]
        for a in range(3):
            outs[a].n = h[a]
        return [x for L in outs for x in (L.offsets, L.depth[:L.n], L.nx[:L.n], L.ny[:L.n], L.nz[:L.n], L.tri[:L.n])]


@pytest.mark.parametrize("kind", ["sample", "binned", "learned", "batch", "chain", "nodes", "contour", "offset"])
def test_workspace_at_any_address(ldni, kind):
    call = Call(ldni, kind)
    need = call.bytes()
    own = torch.empty(need, dtype=torch.uint8, device="cuda")
    want = call.run(own.data_ptr(), need)
    for shift in (1, 4, 8, 24, 255):
        buf = torch.full((need + 512,), 0xA5, dtype=torch.uint8, device="cuda")
        got = call.run(buf.data_ptr() + shift, need)
        assert all(torch.equal(x.view(torch.uint8) if x.dtype != torch.uint8 else x,
                               y.view(torch.uint8) if y.dtype != torch.uint8 else y) for x, y in zip(got, want)), shift
        assert bool((buf[:shift] == 0xA5).all()) and bool((buf[shift + need:] == 0xA5).all()), shift
