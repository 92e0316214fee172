"""The kernels of N' = 8192 (paired column passes, paired row passes), and dense
tiles of bright and faint samples, through the bounds-checking debug library, as
debug_bounds_run.py does for the smaller planes."""

import debug_bounds_run as R
import numpy as np
from debug_bounds_run import P, dev, random_points, solve, torch, values


def cases():
    rng = np.random.default_rng(8)
    lam, z, pitch = 633e-9, 0.05, 4e-6
    for n in (2048, 4096):
        p = P.make_params(n, pitch, lam, z)
        x, y = random_points(rng, 20001, n, pitch)
        for type_ in (1, 2):
            yield f"type {type_} N {n}", lambda p=p, t=type_, x=x, y=y: solve(p, x, y, t, "f32", rng)

        def type3(p=p, x=x, y=y, n=n):
            xd, yd = random_points(rng, 3001, n, pitch)
            a, b = P.nuasm_plan(p, dev(x), dev(y)), P.nuasm_plan(p, dev(xd), dev(yd))
            try:
                out = torch.zeros(len(xd), dtype=torch.complex64, device=R.DEV)
                P.nuasm3_execute(a, b, values(rng, len(x), "f32"), out)
                torch.cuda.synchronize()
            finally:
                a.destroy()
                b.destroy()
        yield f"type 3 N {n}", type3
    for tile, chunk in ((16, -1), (16, 64), (32, 0), (64, 0)):
        def bright(tile=tile, chunk=chunk):
            x, y = (rng.uniform(-75e-6, 75e-6, 9000) for _ in range(2))
            c = 1e-3 * values(rng, 9000, "f32")
            c[4000] = 1
            plan = P.nuasm_plan(P.make_params(64, 10e-6, lam, 0.01, tile=tile, spread_chunk=chunk), dev(x), dev(y))
            try:
                P.nuasm1_execute(plan, c, torch.zeros(64 * 64, dtype=torch.complex64, device=R.DEV))
                torch.cuda.synchronize()
            finally:
                plan.destroy()
        yield f"bright sample, tile {tile} chunk {chunk}", bright


R.cases = cases

if __name__ == "__main__":
    R.main()
