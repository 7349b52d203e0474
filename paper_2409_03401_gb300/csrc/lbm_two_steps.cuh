// Two steps without flow in one pass over memory (no-flow D2Q5, D2Q9 and D3Q7 lattices).
// Reads the populations of an even time level t of the in-place layout (slot k of node x
// holds the incoming population k) from ``src`` and writes time level t + 2, in the same
// layout, to ``dst``: the first collision's results travel one node through registers,
// shuffles and (3D, along y) shared memory instead of through HBM. The arithmetic of a node
// is collide_at_rest in both steps, so the result equals two calls of step_kernel bit for bit.
//
// A single step is bound by HBM (168 B a node on D3Q7, at 0.97 of the copy bandwidth); two steps
// a pass halve that traffic. Measured a step: 4096^2 D2Q9 543 -> 323 us, 256^3 D3Q7 423 -> 297 us.
// What the results move along x goes through shuffles before it is stored, so that every warp
// writes whole rows at its own x: stores shifted by a node leave partial sectors in a buffer
// that is not the one just read, and a copy in that pattern runs at 4.9 instead of 6.3 TB/s.
#pragma once

namespace lbm {

__device__ __forceinline__ float from_left(float v) { return __shfl_up_sync(0xffffffffu, v, 1); }
__device__ __forceinline__ float from_right(float v) { return __shfl_down_sync(0xffffffffu, v, 1); }

template <class T, int LAT>
__device__ __forceinline__ Node<T, LAT, false> load_node(const StateView& src, int node, const DevParams& P) {
    Addr<AA_EVEN> ad;
    ad.self = node;
    Node<T, LAT, false> nd;
    nd.gather_scalars(src, ad, P);
    return nd;
}

// First collision of a node.
template <class T, int LAT>
__device__ __forceinline__ void collide_first(Node<T, LAT, false> nd, const DevParams& P,
                                              typename RealOf<T>::type (&out)[3][Scalar<LAT>::Q]) {
    using R = typename RealOf<T>::type;
    nd.moments(P);
    collide_at_rest<T, LAT>(nd, P, [&](int set, int k, R r) {
        out[set - SET_G][k] = r;
        return r;
    });
}

// Second collision of every lane's node, incoming populations in[set][k], and the store of
// what comes in at each inner lane's node next: populations moving along x come from the lane
// beside, or, behind a wall (lo: x = -1, hi: x = nx), from the node itself (bounce-back), so that
// a warp stores whole rows at its own x. ``to(k)`` is the slot for population k of this x.
template <class T, int LAT, class To>
__device__ __forceinline__ void collide_second(const typename RealOf<T>::type (&in)[3][Scalar<LAT>::Q],
                                               const StateView& dst, int self, bool inner, bool lo, bool hi,
                                               const DevParams& P, To to) {
    using R = typename RealOf<T>::type;
    using L = Scalar<LAT>;
    Node<T, LAT, false> nd;
#pragma unroll
    for (int k = 0; k < L::Q; ++k) {
        nd.g[k] = in[0][k];
        nd.hA[k] = in[1][k];
        nd.hB[k] = in[2][k];
    }
    nd.moments(P);
    T held[3];
    collide_at_rest<T, LAT>(nd, P, [&](int set, int k, R r) {
        if (k == 0) {
            if (inner) store_rest_at<T, LAT>(dst, set, self, r, P);
            return r;
        }
        if (k & 1) {
            held[set - SET_G] = r;                                     // stored with its opposite
        } else {
            T a = held[set - SET_G], b = r;                            // moving along e_{k-1} and back
            if (L::ex(k - 1) != 0) {
                const bool fwd = L::ex(k - 1) > 0;
                const T ma = fwd ? from_left(a) : from_right(a), mb = fwd ? from_right(b) : from_left(b);
                const T oa = a;
                a = (fwd ? lo : hi) ? b : ma;
                b = (fwd ? hi : lo) ? oa : mb;
            }
            if (inner) {
                store_at<T, LAT>(dst, set, k - 1, to(k - 1), a);
                store_at<T, LAT>(dst, set, k, to(k), b);
            }
        }
        return r;
    });
}

__device__ __forceinline__ int wrapped(int q, int n) { return ((q % n) + n) % n; }

// A barrier of the block in shared memory, and a wait of a bounded number of tries for its phase.
__device__ __forceinline__ void block_barrier_init(unsigned b, int count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(b), "r"(count) : "memory");
}
__device__ __forceinline__ void block_barrier_arrive(unsigned b) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(b) : "memory");
}
__device__ __forceinline__ bool block_barrier_wait(unsigned b, unsigned parity) {
    for (int i = 0; i < (1 << 20); ++i) {
        unsigned done;
        asm volatile("{\n\t.reg .pred p;\n\t"
                     "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
                     "selp.u32 %0, 1, 0, p;\n\t}" : "=r"(done) : "r"(b), "r"(parity) : "memory");
        if (done) return true;
    }
    return false;
}

// 3D: a block of 32 x 16 threads marches along z; its 28 x 14 inner threads own nodes, the
// outer ring computes the first collision of the tile's neighbours again (two_steps_pay_3d: where
// that is worth it).
template <class T>
__global__ void __launch_bounds__(T2X * T2Y, kTwoStepsBlocks)
two_steps_3d_kernel(const DevParams P, const StateView src, const StateView dst, unsigned* fault, int zchunk) {
    begin_after_previous();
    using R = typename RealOf<T>::type;
    constexpr int Q = 7;
    // populations moving along y, of four planes, and a barrier for each that all warps reach when
    // theirs are written (256^3: 297 us a step; 321 with one __syncthreads a plane). A plane's are read a plane later, so that a warp seldom waits; a warp
    // that has seen a barrier knows that all have read what it overwrites two planes on.
    extern __shared__ __align__(16) unsigned char t2_smem[];
    R (*ys)[6][T2Y][T2X] = reinterpret_cast<R (*)[6][T2Y][T2X]>(t2_smem);
    const unsigned bars = unsigned(__cvta_generic_to_shared(t2_smem)) + 4 * 6 * T2Y * T2X * sizeof(R);
    const int tx = threadIdx.x, ty = threadIdx.y;
    const int x = int(blockIdx.x) * T2IX + tx - 2, y = int(blockIdx.y) * T2IY + ty - 1;
    const int zs = blockIdx.z * zchunk, ze = min(zs + zchunk, P.nz);
    // this thread's column, wrapped: lanes past the row's end read nodes whose values nobody takes
    const int gx = wrapped(x, P.nx), gy = wrapped(y, P.ny);
    const int nxy = P.nx * P.ny;
    const int col = gy * P.nx + gx;
    const bool row_in = ty >= 1 && ty <= T2IY && y < P.ny;             // whole warps
    const bool inner = tx >= 2 && tx < T2IX + 2 && x < P.nx;
    const bool wall_lo = P.wall_x && x == 0, wall_hi = P.wall_x && x == P.nx - 1;
    // columns of the neighbours along y
    const int cyp = (gy + 1 == P.ny ? 0 : gy + 1) * P.nx + gx, cym = (gy == 0 ? P.ny - 1 : gy - 1) * P.nx + gx;

    if (tx == 0 && ty == 0)
        for (int i = 0; i < 4; ++i) block_barrier_init(bars + 8 * i, T2Y);
    __syncthreads();
    bool ok = true;  // no wait ran out

    R in[3][Q];      // incoming populations of plane z (second step); +z from z - 1 in slot 5
    R up[3];         // moving +z out of plane z
    R o[3][Q];
    // first collision of plane zz; leaves what comes in along x in o[.][1], o[.][2] and its -z
    // movers in o[.][6]
    auto first = [&](int zz, int slot) {
        const int zr = zz < 0 ? zz + P.nz : (zz >= P.nz ? zz - P.nz : zz);
        collide_first<T, LAT_D3Q7>(load_node<T, LAT_D3Q7>(src, zr * nxy + col, P), P, o);
#pragma unroll
        for (int s = 0; s < 3; ++s) {
            ys[slot][2 * s][ty][tx] = o[s][3];
            ys[slot][2 * s + 1][ty][tx] = o[s][4];
            const R a = from_left(o[s][1]), b = from_right(o[s][2]), own = o[s][1];
            o[s][1] = wall_lo ? o[s][2] : a;
            o[s][2] = wall_hi ? own : b;
        }
        __syncwarp();
        if (tx == 0 && zz >= zs) block_barrier_arrive(bars + 8 * slot);   // nobody reads plane zs - 1
    };
    int slot = 0;
    if (zs > 0 || !P.wall_z) {
        first(zs - 1, 3);
#pragma unroll
        for (int s = 0; s < 3; ++s) in[s][5] = o[s][5];
        first(zs, slot);
    } else {
        first(zs, slot);
#pragma unroll
        for (int s = 0; s < 3; ++s) in[s][5] = o[s][6];                // bounced at the wall
    }
#pragma unroll
    for (int s = 0; s < 3; ++s) {
        in[s][0] = o[s][0]; in[s][1] = o[s][1]; in[s][2] = o[s][2];
        up[s] = o[s][5];
    }
    for (int z = zs; z < ze; ++z) {
        const int next = (slot + 1) & 3;
        const bool top = P.wall_z && z == P.nz - 1, low = P.wall_z && z == 0;
        if (!top) first(z + 1, next);
        if (ok) ok = block_barrier_wait(bars + 8 * slot, unsigned(z - zs) / 4 & 1);
        if (row_in) {
#pragma unroll
            for (int s = 0; s < 3; ++s) {
                in[s][3] = ys[slot][2 * s][ty - 1][tx];
                in[s][4] = ys[slot][2 * s + 1][ty + 1][tx];
                in[s][6] = top ? up[s] : o[s][6];
            }
            if (!ok) in[1][0] = __int_as_float(0x7fc00000);            // the wait ran out: the state shows it
            const int zp = z + 1 == P.nz ? 0 : z + 1, zm = z == 0 ? P.nz - 1 : z - 1;
            const int self = z * nxy + col;
            collide_second<T, LAT_D3Q7>(in, dst, self, inner, wall_lo, wall_hi, P, [&](int k) -> Slot {
                switch (k) {
                    case 3: return {z * nxy + cyp, 3};
                    case 4: return {z * nxy + cym, 4};
                    case 5: return top ? Slot{self, 6} : Slot{zp * nxy + col, 5};
                    case 6: return low ? Slot{self, 5} : Slot{zm * nxy + col, 6};
                    default: return {self, k};
                }
            });
        }
#pragma unroll
        for (int s = 0; s < 3; ++s) {
            in[s][0] = o[s][0]; in[s][1] = o[s][1]; in[s][2] = o[s][2];
            in[s][5] = up[s];
            up[s] = o[s][5];
        }
        slot = next;
    }
    if (!ok) *fault = kWaitFault;
}

// 2D: a warp marches along y on its own; its 28 inner lanes own nodes, the two outer ones on each
// side compute the neighbours' collisions again. No shared memory and no barrier; the next
// row's populations are loaded into registers before this row's collisions (4 blocks of 4 warps
// an SM at 124 registers: 323 us a step at 4096^2, against 361 without and 344 at 3 blocks).
// Four windows of a row to a block; FOLD: windows of a row and then of the next chunk of rows, for
// rows in which many warps would have no window.
template <class T, int LAT, bool FOLD>
__global__ void __launch_bounds__(32 * T2Warps, kTwoSteps2DBlocks)
two_steps_2d_kernel(const DevParams P, const StateView src, const StateView dst, int ychunk) {
    begin_after_previous();
    using R = typename RealOf<T>::type;
    using L = Scalar<LAT>;
    constexpr int Q = L::Q;
    const int lane = threadIdx.x & 31;
    const int item = blockIdx.x * T2Warps + (threadIdx.x >> 5);
    const int wins = FOLD ? (P.nx + T2IX - 1) / T2IX : 1, win = FOLD ? item % wins : item;
    const int chunk = FOLD ? item / wins : blockIdx.y;
    if (FOLD ? chunk * ychunk >= P.ny : win * T2IX >= P.nx) return;    // whole warps
    const int x = win * T2IX + lane - 2;
    const int ys = chunk * ychunk, ye = min(ys + ychunk, P.ny);
    const int gx = wrapped(x, P.nx);
    const bool inner = lane >= 2 && lane < T2IX + 2 && x < P.nx;
    const bool wall_lo = P.wall_x && x == 0, wall_hi = P.wall_x && x == P.nx - 1;

    R in[3][Q];      // incoming populations of row y: the rows y - 1 and y filled in, y + 1 to come
    R up[3][Q];      // of row y + 1: what row y sends up
    R o[3][Q];
    auto row = [&](int yy) {
        return load_node<T, LAT>(src, (yy < 0 ? yy + P.ny : (yy >= P.ny ? yy - P.ny : yy)) * P.nx + gx, P);
    };
    Node<T, LAT, false> next = row(ys - 1);
    auto first = [&](int yy) {
        const Node<T, LAT, false> nd = next;
        next = row(yy < ye ? yy + 1 : yy);
        collide_first<T, LAT>(nd, P, o);
#pragma unroll
        for (int s = 0; s < 3; ++s) {
            const R p1 = o[s][1], m1 = o[s][2];                        // +x and -x, for walls
#pragma unroll
            for (int k = 1; k < Q; ++k) {
                if (L::ex(k) > 0) o[s][k] = from_left(o[s][k]);
                if (L::ex(k) < 0) o[s][k] = from_right(o[s][k]);
            }
            if constexpr (LAT == LAT_D2Q5) {
                if (wall_lo) o[s][1] = m1;
                if (wall_hi) o[s][2] = p1;
            }
        }
    };
    // hand the outputs of a row on: its own level and downward movers are consumed by now
    auto rotate = [&]() {
#pragma unroll
        for (int s = 0; s < 3; ++s)
#pragma unroll
            for (int k = 0; k < Q; ++k) {
                if (L::ey(k) == 0) in[s][k] = o[s][k];
                if (L::ey(k) > 0) { in[s][k] = up[s][k]; up[s][k] = o[s][k]; }
            }
    };
    first(ys - 1);
    rotate();
    first(ys);
    rotate();
    for (int y = ys; y < ye; ++y) {
        first(y + 1);
#pragma unroll
        for (int s = 0; s < 3; ++s)
#pragma unroll
            for (int k = 0; k < Q; ++k)
                if (L::ey(k) < 0) in[s][k] = o[s][k];
        const int yp = y + 1 == P.ny ? 0 : y + 1, ym = y == 0 ? P.ny - 1 : y - 1;
        collide_second<T, LAT>(in, dst, y * P.nx + gx, inner, wall_lo, wall_hi, P, [&](int k) -> Slot {
            return {(L::ey(k) > 0 ? yp : (L::ey(k) < 0 ? ym : y)) * P.nx + gx, k};
        });
        rotate();
    }
}

template <class T, int LAT>
void launch_two_steps_at(const DevParams& P, const StateView& src, const StateView& dst, unsigned* fault, cudaStream_t s) {
    if constexpr (LAT == LAT_D3Q7) {
        const dim3 tiles((P.nx + T2IX - 1) / T2IX, (P.ny + T2IY - 1) / T2IY);
        const int zc = march_chunk((long long)tiles.x * tiles.y, P.nz, 152 * kTwoStepsBlocks, 2.0);
        constexpr int smem = 4 * 6 * T2Y * T2X * int(sizeof(float)) + 64;
        cudaFuncSetAttribute(two_steps_3d_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        launch_after_previous<float>(two_steps_3d_kernel<T>, dim3(tiles.x, tiles.y, (P.nz + zc - 1) / zc), dim3(T2X, T2Y),
                                     size_t(smem), s, P, src, dst, fault, zc);
    } else {
        const TwoSteps2D p(P.nx, P.ny);
        launch_after_previous<float>(p.fold ? two_steps_2d_kernel<T, LAT, true> : two_steps_2d_kernel<T, LAT, false>,
                                     dim3(p.bx, p.by), dim3(32 * T2Warps), 0, s, P, src, dst, p.rows);
    }
}

}  // namespace lbm
