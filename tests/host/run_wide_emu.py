"""Run the finder's kernels for wide windows under host warp emulation on one
synthetic batch and save the outputs (a separate process: a warp divergence ends it)."""
import ctypes as C
import json
import sys

import numpy as np


def main(so, root, out_path, cfg):
    sys.path.insert(0, root)
    from paper_1811_04141_gb300 import _native as NN
    from synth import make_batch
    b = make_batch(cfg["config"], cfg["events"], n_tracks=cfg["tracks"], n_noise=cfg["noise"], material=0.02, eloss=0.04)
    lay = b.layers
    arr = (NN.MkfLayer * len(lay))()
    for i, d in enumerate(lay):
        n_phi, n_zr = cfg["grid"] or (d["n_phi"], d["n_zr"])
        arr[i] = NN.MkfLayer(int(d["kind"]), float(d["r_or_z"]), float(d["lo"]), float(d["hi"]), float(d["sigma_u"]),
                             float(d["sigma_v"]), int(n_phi), int(n_zr))
    n, mo = b.n_seeds, len(lay) + 3
    X, Y, Z = [np.ascontiguousarray(b.xyz[i], dtype=np.float32) for i in range(3)]
    i32 = lambda a: np.ascontiguousarray(a, dtype=np.int32)
    keep = [i32(b.layer), i32(b.event_offsets), i32(b.seed_hits), i32(b.seed_event)]
    p = lambda a: a.ctypes.data_as(C.c_void_p)
    res, lib = {}, C.CDLL(so)
    for k, line in enumerate(cfg["lines"]):
        out = dict(par=np.zeros((6, n), np.float32), cov=np.zeros((21, n), np.float32), chi2=np.zeros(n, np.float32),
                   n_hits=np.zeros(n, np.int32), hits=np.full((mo, n), -7, np.int32), status=np.zeros(n, np.uint32),
                   counters=np.zeros((3, n), np.int32), fault=np.zeros(2, np.int32), left=np.zeros(1, np.int32))
        rc = lib.emu_wide(arr, len(lay), C.c_float(b.bz), C.c_float(0.02), C.c_float(0.04), p(X), p(Y), p(Z), p(keep[0]),
                          b.n_hits, p(keep[1]), len(b.event_offsets) - 1, p(keep[2]), p(keep[3]), n, cfg["n_best"],
                          C.c_float(30.0), mo, C.c_float(line), p(out["par"]), p(out["cov"]), p(out["chi2"]),
                          p(out["n_hits"]), p(out["hits"]), p(out["status"]), p(out["counters"]), p(out["fault"]),
                          p(out["left"]))
        if rc != 0:
            raise SystemExit(f"emu_wide failed: {rc}")
        res.update({f"{name}_{k}": v for name, v in out.items()})
    np.savez(out_path, n_seeds=n, **res)


if __name__ == "__main__":
    main(sys.argv[1], sys.argv[2], sys.argv[3], json.loads(sys.argv[4]))
