"""Host threads with decoders of different codes on the kernels that take a code's
tile in shared memory (plain BP, training forward and backward): no thread's size
limits another's launch, and the results are those of one thread."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2512_07057_gb300 import binding as B  # noqa: E402
from paper_2512_07057_gb300 import decoder as D  # noqa: E402
from paper_2512_07057_gb300 import unrolled as U  # noqa: E402
from paper_2512_07057_gb300 import workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))
SHOTS, T = 9, 2


class Job(C.Structure):
    _fields_ = [("llr_dec", C.c_void_p), ("dec", C.c_void_p), ("synd", C.c_void_p), ("errs", C.c_void_p),
                ("B", C.c_int64), ("T", C.c_int32), ("ckpt", C.c_int32), ("w", C.c_void_p), ("grad_loss", C.c_void_p), ("llr", C.c_void_p),
                ("loss", C.c_void_p), ("grad", C.c_void_p), ("work", C.c_void_p), ("work_bytes", C.c_int64),
                ("stream", C.c_void_p)]


def test_threads_with_tiles_of_different_sizes(tmp_path):
    so = str(tmp_path / "tile_threads.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-pthread", "-I", os.path.join(HERE, "..", "include"),
                    "-o", so, os.path.join(HERE, "tile_threads_host.cpp")], check=True)
    lib = B.load()
    api = (C.c_void_p * 3)(*[C.cast(getattr(lib, f), C.c_void_p) for f in
                             ("bsd_bp_llr", "bsd_unrolled_forward", "bsd_unrolled_backward")])
    jobs, keep, want = (Job * 2)(), [], []
    for k, prob in enumerate([W.bb_phenomenological(12, 6, 12, 0.03, 0.03), W.bb_phenomenological(6, 6, 3, 0.03, 0.03)]):
        dec = D.BeamSearchDecoder(prob, D.make_params(max_rounds=0, group_warps=1))   # plain BP on tiles at any batch
        tr = U.UnrolledTrainer(prob, SHOTS, T, 1)
        synd, errs, _ = U.batch_tensors(prob, SHOTS, f"threads_{k}")
        w = torch.full((T, prob.n_edges), 0.625, device="cuda")
        gl = torch.tensor([1.0] + [0.0] * T, device="cuda")
        outs = [dec.bp_llr(synd, T)[0], tr.forward(w, synd, errs), tr.backward(w, gl)]
        want.append([x.cpu().numpy().copy() for x in outs])
        for x in outs:
            x.zero_()
        stream = torch.cuda.Stream()
        jobs[k] = Job(dec.h, tr.dec.h, synd.data_ptr(), errs.data_ptr(), SHOTS, T, 1, w.data_ptr(), gl.data_ptr(),
                      outs[0].data_ptr(), outs[1].data_ptr(), outs[2].data_ptr(), tr.work.data_ptr(), tr.work.numel(),
                      stream.cuda_stream)
        keep.append((dec, tr, synd, errs, w, gl, outs, stream))
    torch.cuda.synchronize()
    run = C.CDLL(so).tile_threads
    run.argtypes = [C.c_void_p, C.POINTER(Job), C.c_int]
    failed = run(C.addressof(api), jobs, 9_000)
    torch.cuda.synchronize()
    for (dec, tr, *_, outs, _stream), ref in zip(keep, want):
        assert failed or all(np.array_equal(a.cpu().numpy(), b) for a, b in zip(outs, ref))
        dec.close()
        tr.close()
    assert failed == 0
