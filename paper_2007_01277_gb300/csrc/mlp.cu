// mlp.cu -- the learned cost model's kernels: a 24 -> 64 -> ReLU -> 64 ->
// ReLU -> 1 perceptron in FP32 on the CUDA cores (it is far too small for
// the tensor cores to pay off).
//
// Parameters are one flat FP32 array, row-major:
//   W1[64][24] @0, b1[64] @1536, W2[64][64] @1600, b2[64] @5696,
//   w3[64] @5760, b3 @5824                                  (5825 values)
//
// k_mlp_forward scores samples grid-wide, in tiles of 32 samples; see its
// comment.
//
// k_mlp_train runs a whole training run in one launch of one cluster of eight
// blocks; see its comment.  k_mlp_train_block does it with one block.
#include <cmath>

#include "kernels.cuh"

namespace hf {
hf_status set_last_error(hf_status s, const char *msg);   // runtime.cu
}

namespace {

constexpr int IN = 24, HD = 64, NP = 5825;
constexpr int OW1 = 0, OB1 = 1536, OW2 = 1600, OB2 = 5696, OW3 = 5760, OB3 = 5824;
constexpr int kMaxBatch = 64;

// ------------------------------------------------------------------ forward
__device__ __forceinline__ float4 at4(const float *p) { return *reinterpret_cast<const float4 *>(p); }
__device__ __forceinline__ float part(const float4 &v, int i) { return i == 0 ? v.x : i == 1 ? v.y : i == 2 ? v.z : v.w; }

// A tile is 32 samples and belongs to two warps: lane = four samples (q) and
// eight units ug, ug + 8, ..., ug + 56, so that twelve 128-bit shared loads
// (four of activations, eight of weights) feed 128 multiply-adds.  The
// weights are staged once per block and the activations stay transposed
// ([unit][sample]); rows of 68, 28 and 36 values keep the loads free of
// bank conflicts.  A block has kSlots tiles in work; tiles go to blocks
// first and slots second, so few samples spread over the SMs.
//
// The bound is the shared-load pipe (an LDS.128 takes it four cycles
// whatever it broadcasts): about 2100 cycles a tile against 1400 of
// multiply-adds on four schedulers.  One warp per sample, with two 32-bit
// weight loads and a shuffle per two multiply-adds and a transpose of W2
// with 32-way bank conflicts in every block, took 32.8 us for 16086 samples
// and 7.4 for 100; this takes 7.1 and 4.6 us (most of the latter is the
// weights' way into shared memory: 7.3 us before all of a thread's loads
// were in flight at once).  Both sum in the same order: the same bits.
constexpr int kSlots = 2, kTile = 32, FS = 36;   // FS: row stride of a tile's rows
struct ForwardSmem {
    float W2[HD][68];
    float W1[HD][28];
    float A[kSlots][HD][FS];   // the batch (24 rows), then H1 in its place
    float b1[HD], b2[HD], w3[HD];
};
static_assert(sizeof(ForwardSmem) <= 48 * 1024, "static shared memory");

__device__ __forceinline__ void slot_sync(int slot)
{
    asm volatile("bar.sync %0, 64;" ::"r"(slot + 1) : "memory");
}

// acc[v][0..3] += sum over k (ascending) of W[ug + 8v][k] * A[k][4q .. 4q + 3]
template <int K, int WS>
__device__ __forceinline__ void units8(const float *w, const float *A, float (&acc)[8][4])
{
#pragma unroll 2
    for (int k = 0; k < K; k += 4) {
        float4 a[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) a[j] = at4(A + (k + j) * FS);
#pragma unroll
        for (int v = 0; v < 8; ++v) {
            const float4 w4 = at4(w + 8 * v * WS + k);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const float wk = part(w4, j);
                acc[v][0] = __fmaf_rn(wk, a[j].x, acc[v][0]);
                acc[v][1] = __fmaf_rn(wk, a[j].y, acc[v][1]);
                acc[v][2] = __fmaf_rn(wk, a[j].z, acc[v][2]);
                acc[v][3] = __fmaf_rn(wk, a[j].w, acc[v][3]);
            }
        }
    }
}

__global__ void __launch_bounds__(64 * kSlots) k_mlp_forward(const float *__restrict__ P, const float *__restrict__ X,
                                                            int n, float *__restrict__ y)
{
    __shared__ __align__(16) ForwardSmem T;
    const int tid = threadIdx.x;
    float w1[HD * IN / (64 * kSlots)], w2[HD * HD / (64 * kSlots)];   // every load in flight at once
#pragma unroll
    for (int i = 0; i < HD * IN / (64 * kSlots); ++i) w1[i] = __ldg(P + OW1 + tid + i * 64 * kSlots);
#pragma unroll
    for (int i = 0; i < HD * HD / (64 * kSlots); ++i) w2[i] = __ldg(P + OW2 + tid + i * 64 * kSlots);
#pragma unroll
    for (int i = 0; i < HD * IN / (64 * kSlots); ++i) {
        const int e = tid + i * 64 * kSlots;
        T.W1[e / IN][e % IN] = w1[i];
    }
#pragma unroll
    for (int i = 0; i < HD * HD / (64 * kSlots); ++i) {
        const int e = tid + i * 64 * kSlots;
        T.W2[e / HD][e % HD] = w2[i];
    }
    for (int e = tid; e < HD; e += 64 * kSlots) T.b1[e] = P[OB1 + e], T.b2[e] = P[OB2 + e], T.w3[e] = P[OW3 + e];
    const float b3 = P[OB3];
    __syncthreads();
    const int slot = tid >> 6, t64 = tid & 63, lane = tid & 31;
    const int ug = lane >> 2, q = 4 * (t64 >> 5) + (lane & 3);
    float(*A)[FS] = T.A[slot];
    const int tiles = n / kTile + (n % kTile != 0);
    for (int64_t tile = (int64_t)slot * gridDim.x + blockIdx.x; tile < tiles; tile += (int64_t)kSlots * gridDim.x) {
        const int64_t s0 = tile * kTile;
        const int m = (int)min((int64_t)kTile, n - s0);   // samples past the end count as zeros
#pragma unroll
        for (int e = t64; e < kTile * IN; e += 64) {
            const int s = e / IN;
            A[e - s * IN][s] = s < m ? __ldg(X + s0 * IN + e) : 0.f;
        }
        slot_sync(slot);
        float acc[8][4];
#pragma unroll
        for (int v = 0; v < 8; ++v)
#pragma unroll
            for (int i = 0; i < 4; ++i) acc[v][i] = T.b1[ug + 8 * v];
        units8<IN, 28>(T.W1[ug], &A[0][4 * q], acc);
        slot_sync(slot);
#pragma unroll
        for (int v = 0; v < 8; ++v) {
            *reinterpret_cast<float4 *>(&A[ug + 8 * v][4 * q]) =
                make_float4(fmaxf(acc[v][0], 0.f), fmaxf(acc[v][1], 0.f), fmaxf(acc[v][2], 0.f), fmaxf(acc[v][3], 0.f));
#pragma unroll
            for (int i = 0; i < 4; ++i) acc[v][i] = T.b2[ug + 8 * v];
        }
        slot_sync(slot);
        units8<HD, 68>(T.W2[ug], &A[0][4 * q], acc);
        // the output's sum as a butterfly over units: j with j + 32, then
        // distances 16 and 8 in the lane, 4, 2 and 1 across lanes
        float o[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            float h[4];
#pragma unroll
            for (int v = 0; v < 4; ++v)
                h[v] = __fmaf_rn(T.w3[ug + 8 * v], fmaxf(acc[v][i], 0.f), T.w3[ug + 8 * v + 32] * fmaxf(acc[v + 4][i], 0.f));
            o[i] = (h[0] + h[2]) + (h[1] + h[3]);
#pragma unroll
            for (int d = 16; d >= 4; d >>= 1) o[i] += __shfl_xor_sync(0xffffffffu, o[i], d);
        }
        if (ug == 0)
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if (4 * q + i < m) y[s0 + 4 * q + i] = o[i] + b3;
        slot_sync(slot);   // the tile is read before the next one is stored
    }
}

// ------------------------------------------------------------------ training
// One cluster of kCl blocks runs every step: gather, forward, backward (mean
// squared error) and Adam (Kingma & Ba).  Block r owns hidden units
// 8r .. 8r+7 of both layers: their rows of W1 and W2, the same columns of W2
// (a copy for the backward pass), their biases, their w3, and the moments of
// all of them, which stay in the registers of the threads that update them.
// Activations are kept transposed ([unit][sample]) so that every product is
// an outer-product tile of 128-bit shared loads:
//   columns<K>  out[u][s..s+3] += W[u][k] * A[k][s..s+3], lanes = 8 units x 4
//               groups of four samples: 5 loads per 16 multiply-adds
//               (forward layers, and the backward pass through W2)
//   gradient    g[u][i] += D[u][s] * A[i][s], lanes = 8 units x 4 inputs
// Blocks exchange the two activation layers through distributed shared
// memory: each writes its units' rows into all blocks, two cluster barriers a
// step; updated columns of W2 and w3 travel with the next step's first one.
// What a slower block may still read (H1, the W2 columns, w3) is double
// buffered: a block past a step's barriers knows that every other one has
// finished the step before.  Two warps gather the next step's batch meanwhile.
//
// The bound is latency: a step is a chain of five products of 24 to 64
// dependent multiply-adds, five block barriers and two exchanges of 16 KB
// over distributed shared memory, about 3500 of its 17000 cycles each (bulk
// copies and asynchronous stores with mbarriers took as long).  A single block with
// one output per thread and both operands from shared memory (10 block
// barriers, its load pipe 65 % busy) took 37.3 us a step at batch 64;
// this takes 8.2 us, with the same bits.  Every sum keeps one fixed order (inputs or samples
// ascending), so a run is deterministic; samples past the batch count as zero.
constexpr int kCl = 8, kU = HD / kCl;    // blocks of the cluster, units per block
constexpr int kWarps = 11, kTrainThreads = 32 * kWarps;
constexpr int S = 68;                    // row stride of sample rows: 8 rows hit distinct banks
constexpr int S1 = 28;                   // of W1's rows
struct TrainSmem {
    float Xt[2][IN][S];      // batch, transposed, of this and the next step
    float H1[2][HD][S];      // all units, written by their owners
    float H2[HD][S];
    float D2[HD][S];         // error at layer 2, all units
    float D1[kU][S];         // error at layer 1, own units
    float W2[kU][S];         // own rows (own units over all inputs)
    float W2c[2][kU][S];     // own columns: W2c[i][j] = W2[j][8r + i]
    float W1[kU][S1];
    float w3[2][HD];
    float Y[2][HD], dY[HD], e2[HD], ones[HD];
    float b1[kU], b2[kU], b3[2];
    float c[2][2];           // Adam's bias corrections of this and the next step
};
static_assert(HD == 64 && kMaxBatch == 64 && kU == 8, "lane layout of the training kernel");

__device__ __forceinline__ unsigned cluster_rank()
{
    unsigned r;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
// Every thread of the cluster arrives and waits (a hardware barrier over
// co-scheduled blocks); shared-memory writes before it, remote ones too, are
// visible after it.
__device__ __forceinline__ void cluster_sync()
{
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// address of `p`'s counterpart in block `rank` of the cluster
__device__ __forceinline__ unsigned remote(const void *p, int rank)
{
    unsigned a;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"((unsigned)__cvta_generic_to_shared(p)), "r"(rank));
    return a;
}
__device__ __forceinline__ void put(unsigned addr, float v)
{
    asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(addr), "f"(v) : "memory");
}
__device__ __forceinline__ void put4(unsigned addr, float4 v)
{
    asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w)
                 : "memory");
}

// ReLU of samples s .. s + 3; those past the batch are zero, so that the sums
// over samples add nothing for them, whatever the parameters (an infinite
// activation times an error of zero would be NaN).
__device__ __forceinline__ float4 relu4(const float4 &a, int s, int B)
{
    float4 h = make_float4(fmaxf(a.x, 0.f), fmaxf(a.y, 0.f), fmaxf(a.z, 0.f), fmaxf(a.w, 0.f));
    if (s + 4 > B) {
        if (s + 1 > B) h.x = 0.f;
        if (s + 2 > B) h.y = 0.f;
        if (s + 3 > B) h.z = 0.f;
        h.w = 0.f;
    }
    return h;
}

// acc[0..3] += sum over k (ascending) of w[k] * A[k][0..3]; A's rows S apart
template <int K>
__device__ __forceinline__ void columns(const float *w, const float *A, float4 &acc)
{
#pragma unroll 4
    for (int k = 0; k < K; k += 4) {
        const float4 w4 = at4(w + k);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float4 a = at4(A + (k + j) * S);
            const float wk = part(w4, j);
            acc.x = __fmaf_rn(wk, a.x, acc.x);
            acc.y = __fmaf_rn(wk, a.y, acc.y);
            acc.z = __fmaf_rn(wk, a.z, acc.z);
            acc.w = __fmaf_rn(wk, a.w, acc.w);
        }
    }
}
// g[v] += sum over s < n (ascending, n a multiple of 4) of d[s] * A_v[s],
// the rows A_v 4 * S apart
template <int N>
__device__ __forceinline__ void gradient(const float *d, const float *A, int n, float (&g)[N])
{
#pragma unroll 4
    for (int s = 0; s < n; s += 4) {
        const float4 d4 = at4(d + s);
#pragma unroll
        for (int v = 0; v < N; ++v) {
            const float4 a = at4(A + 4 * v * S + s);
            g[v] = __fmaf_rn(d4.x, a.x, g[v]);
            g[v] = __fmaf_rn(d4.y, a.y, g[v]);
            g[v] = __fmaf_rn(d4.z, a.z, g[v]);
            g[v] = __fmaf_rn(d4.w, a.w, g[v]);
        }
    }
}

// The moments' sums are one fused multiply-add each, spelled out so that
// every use rounds alike.
struct Adam {
    float lr, beta1, beta2, eps;
    __device__ __forceinline__ float step(float p, float &M, float &V, float g, const float *c) const
    {
        const float m = __fmaf_rn(1.f - beta1, g, beta1 * M);
        const float v = __fmaf_rn((1.f - beta2) * g, g, beta2 * V);
        M = m;
        V = v;
        return p - lr * (m / c[0]) / (sqrtf(v / c[1]) + eps);
    }
};

__global__ void __cluster_dims__(kCl, 1, 1) __launch_bounds__(kTrainThreads) k_mlp_train(
    float *__restrict__ Pg, float *__restrict__ Mg, float *__restrict__ Vg, const float *__restrict__ X,
    const float *__restrict__ Y, const int *__restrict__ idx, int steps, int B, float lr, float beta1, float beta2,
    float eps, int t0, float *__restrict__ loss_out, float *__restrict__ grad_out)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    TrainSmem &T = *reinterpret_cast<TrainSmem *>(smem_raw);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int r = (int)cluster_rank(), j0 = kU * r;
    const int n = (B + 3) / 4 * 4;            // samples of the padded batch
    const float invB = 1.0f / (float)B;
    const Adam adam{lr, beta1, beta2, eps};

    // parameters of this block's units (rows past n of the sample buffers are
    // never read)
    for (int e = tid; e < kU * IN; e += kTrainThreads) T.W1[e / IN][e % IN] = Pg[OW1 + j0 * IN + e];
    for (int e = tid; e < kU * HD; e += kTrainThreads) {
        T.W2[e / HD][e % HD] = Pg[OW2 + j0 * HD + e];
        T.W2c[0][e % kU][e / kU] = Pg[OW2 + e / kU * HD + j0 + e % kU];
    }
    for (int e = tid; e < HD; e += kTrainThreads) {
        T.w3[0][e] = Pg[OW3 + e];
        T.ones[e] = 1.f;
        if (e < kU) T.b1[e] = Pg[OB1 + j0 + e], T.b2[e] = Pg[OB2 + j0 + e];
        if (e == 0) T.b3[0] = Pg[OB3];
    }
    // Who updates what: warps 0-3 four elements of W2 each thread; tid < 192
    // one of W1; warp 8 the vectors (lanes 0-7 w3, 8-15 b2, 16 b3; then
    // lanes 0-7 b1).
    const int u = lane >> 2, q = lane & 3;
    const int p_w2 = OW2 + (j0 + u) * HD + 16 * warp + q;   // + 4 * v
    const int p_w1 = OW1 + j0 * IN + tid;
    const int p_vec = lane < 8 ? OW3 + j0 + lane : lane < 16 ? OB2 + j0 + lane - 8 : OB3;
    const int p_b1 = OB1 + j0 + (lane & 7);
    float m2[4], v2[4], m1 = 0.f, v1 = 0.f, mv = 0.f, vv = 0.f;
    if (warp < 4)
#pragma unroll
        for (int v = 0; v < 4; ++v) m2[v] = Mg[p_w2 + 4 * v], v2[v] = Vg[p_w2 + 4 * v];
    if (tid < kU * IN) m1 = Mg[p_w1], v1 = Vg[p_w1];
    if (warp == 8) {
        mv = Mg[p_vec], vv = Vg[p_vec];
        m1 = Mg[p_b1], v1 = Vg[p_b1];
    }
    // Warps 9 and 10, a lane per sample: the batch of step t is loaded into
    // registers a step ahead and stored into buffer t & 1 when its loads
    // have had two layers' time; its row number is loaded a step earlier still.
    const int sample = 32 * (warp - 9) + lane;
    float x[IN], y = 0.f;
    int row = 0;
    auto fetch_row = [&](int t) { row = sample < B && t < steps ? idx[(int64_t)t * B + sample] : 0; };
    auto fetch = [&]() {
#pragma unroll
        for (int k = 0; k < IN; ++k) x[k] = sample < B ? __ldg(X + (int64_t)row * IN + k) : 0.f;
        y = sample < B ? __ldg(Y + row) : 0.f;
    };
    auto stash = [&](int t) {
        if (sample < n) {
#pragma unroll
            for (int k = 0; k < IN; ++k) T.Xt[t & 1][k][sample] = x[k];
            T.Y[t & 1][sample] = y;
        }
        if (sample == 0) {
            const float tf = (float)(t0 + t + 1);
            T.c[t & 1][0] = 1.f - powf(beta1, tf);
            T.c[t & 1][1] = 1.f - powf(beta2, tf);
        }
    };
    if (warp >= 9) {
        fetch_row(0);
        fetch();
        stash(0);
        fetch_row(1);
    }
    cluster_sync();   // every block has started; its buffers are ready

    const int s4 = 16 * (warp & 3) + 4 * q;   // first sample of this lane's four
    for (int t = 0; t < steps; ++t) {
        const int cur = t & 1, nxt = cur ^ 1;
        const float *c = T.c[cur];
        if (warp >= 9 && t + 1 < steps) {
            fetch();
            fetch_row(t + 2);
        }
        // H1 = relu(X W1^T + b1), own units, into every block
        if (warp < 4 && s4 < n) {
            const float b = T.b1[u];
            float4 a = make_float4(b, b, b, b);
            columns<IN>(T.W1[u], &T.Xt[cur][0][s4], a);
            a = relu4(a, s4, B);
#pragma unroll
            for (int k = 0; k < kCl; ++k) put4(remote(&T.H1[cur][j0 + u][s4], k), a);
        }
        cluster_sync();
        // H2 = relu(H1 W2^T + b2), own units, into every block
        if (warp < 4 && s4 < n) {
            const float b = T.b2[u];
            float4 a = make_float4(b, b, b, b);
            columns<HD>(T.W2[u], &T.H1[cur][0][s4], a);
            a = relu4(a, s4, B);
#pragma unroll
            for (int k = 0; k < kCl; ++k) put4(remote(&T.H2[j0 + u][s4], k), a);
        }
        cluster_sync();
        // output, error and dL/dy of every sample, in every block
        if (tid < n) {
            float a = T.b3[0];
#pragma unroll 4
            for (int j = 0; j < HD; j += 4) {
                const float4 w = at4(T.w3[cur] + j);
                a = __fmaf_rn(w.x, T.H2[j][tid], a);
                a = __fmaf_rn(w.y, T.H2[j + 1][tid], a);
                a = __fmaf_rn(w.z, T.H2[j + 2][tid], a);
                a = __fmaf_rn(w.w, T.H2[j + 3][tid], a);
            }
            const float e = tid < B ? a - T.Y[cur][tid] : 0.f;
            T.dY[tid] = 2.f * e * invB;
            T.e2[tid] = e * e;
        }
        __syncthreads();
        // D2 = dY w3^T masked by the ReLU, all units
        for (int e = tid; e < HD * (n / 4); e += kTrainThreads) {
            const int j = e / (n / 4), s = 4 * (e - j * (n / 4));
            const float w = T.w3[cur][j];
            const float4 h = at4(&T.H2[j][s]), d = at4(T.dY + s);
            *reinterpret_cast<float4 *>(&T.D2[j][s]) =
                make_float4(h.x > 0.f ? d.x * w : 0.f, h.y > 0.f ? d.y * w : 0.f, h.z > 0.f ? d.z * w : 0.f,
                            h.w > 0.f ? d.w * w : 0.f);
        }
        __syncthreads();
        if (warp < 4) {
            // W2's own rows: gW2[j][i] = sum_s D2[s][j] H1[s][i]
            float g[4] = {0.f, 0.f, 0.f, 0.f};
            const int i0 = 16 * warp + q;
            gradient<4>(T.D2[j0 + u], T.H1[cur][i0], n, g);
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                const int i = i0 + 4 * v;
                if (grad_out && t == 0) grad_out[p_w2 + 4 * v] = g[v];
                const float w = adam.step(T.W2[u][i], m2[v], v2[v], g[v], c);
                T.W2[u][i] = w;
                put(remote(&T.W2c[nxt][i & 7][j0 + u], i >> 3), w);   // unit i's block
            }
        } else if (warp < 8) {
            // D1[s][i] = (sum_j D2[s][j] W2[j][i]) masked by the ReLU, own units
            if (s4 < n) {
                float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
                columns<HD>(T.W2c[cur][u], &T.D2[0][s4], a);
                const float4 h = at4(&T.H1[cur][j0 + u][s4]);
                *reinterpret_cast<float4 *>(&T.D1[u][s4]) =
                    make_float4(h.x > 0.f ? a.x : 0.f, h.y > 0.f ? a.y : 0.f, h.z > 0.f ? a.z : 0.f,
                                h.w > 0.f ? a.w : 0.f);
            }
        } else if (warp == 8) {
            // sums over the samples: gw3 and gb2 of the own units, gb3, loss
            if (lane < 18) {
                const float *d = lane < 8 ? T.dY : T.ones;
                const float *a = lane < 8 ? T.H2[j0 + lane] : lane < 16 ? T.D2[j0 + lane - 8] : lane == 16 ? T.dY : T.e2;
                float g[1] = {0.f};
                gradient<1>(d, a, n, g);
                if (lane == 17) {
                    if (r == 0 && loss_out) loss_out[t] = g[0] * invB;
                } else {
                    if (grad_out && t == 0 && (lane < 16 || r == 0)) grad_out[p_vec] = g[0];
                    const float old = lane < 8 ? T.w3[cur][j0 + lane] : lane < 16 ? T.b2[lane - 8] : T.b3[0];
                    const float w = adam.step(old, mv, vv, g[0], c);
                    if (lane < 8) {
#pragma unroll
                        for (int k = 0; k < kCl; ++k) put(remote(&T.w3[nxt][j0 + lane], k), w);
                    } else if (lane < 16) {
                        T.b2[lane - 8] = w;
                    } else {
                        T.b3[0] = w;   // the same bits in every block
                    }
                }
            }
        } else if (t + 1 < steps) {
            stash(t + 1);
        }
        __syncthreads();
        // W1's own rows: gW1[j][k] = sum_s D1[s][j] X[s][k]
        if (tid < kU * IN) {
            const int j = tid / IN, k = tid - j * IN;
            float g[1] = {0.f};
            gradient<1>(T.D1[j], T.Xt[cur][k], n, g);
            if (grad_out && t == 0) grad_out[p_w1] = g[0];
            T.W1[j][k] = adam.step(T.W1[j][k], m1, v1, g[0], c);
        } else if (warp == 8 && lane < 8) {
            float g[1] = {0.f};
            gradient<1>(T.ones, T.D1[lane], n, g);
            if (grad_out && t == 0) grad_out[p_b1] = g[0];
            T.b1[lane] = adam.step(T.b1[lane], m1, v1, g[0], c);
        }
        __syncthreads();
    }
    cluster_sync();   // no block leaves while others may write to it
    if (warp < 4)
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            Pg[p_w2 + 4 * v] = T.W2[u][16 * warp + q + 4 * v];
            Mg[p_w2 + 4 * v] = m2[v];
            Vg[p_w2 + 4 * v] = v2[v];
        }
    if (tid < kU * IN) {
        Pg[p_w1] = T.W1[tid / IN][tid % IN];
        Mg[p_w1] = m1;
        Vg[p_w1] = v1;
    }
    if (warp == 8) {
        if (lane < 16 || (lane == 16 && r == 0)) {
            Pg[p_vec] = lane < 8 ? T.w3[steps & 1][j0 + lane] : lane < 16 ? T.b2[lane - 8] : T.b3[0];
            Mg[p_vec] = mv;
            Vg[p_vec] = vv;
        }
        if (lane < 8) {
            Pg[p_b1] = T.b1[lane];
            Mg[p_b1] = m1;
            Vg[p_b1] = v1;
        }
    }
}

// The same run on one block, for devices (or partitions of one) that cannot
// hold the cluster: every parameter and activation in shared memory, a thread
// per output, rows padded so that lanes that walk samples hit distinct banks.
// Its sums keep k_mlp_train's order: the same bits, at 37.3 us a step of 64.
constexpr int kBlockThreads = 512;
constexpr int SX = IN + 1, SH = HD + 1;   // padded row strides
struct BlockSmem {
    float P[NP], M[NP], V[NP], G[NP];
    float X[kMaxBatch * SX];
    float H1[kMaxBatch * SH];
    float H2[kMaxBatch * SH];   // becomes the error at layer 2 after the output's gradient
    float D1[kMaxBatch * SH];
    float Y[kMaxBatch], dY[kMaxBatch];
};

__global__ void __launch_bounds__(kBlockThreads) k_mlp_train_block(
    float *__restrict__ Pg, float *__restrict__ Mg, float *__restrict__ Vg, const float *__restrict__ X,
    const float *__restrict__ Y, const int *__restrict__ idx, int steps, int B, float lr, float beta1, float beta2,
    float eps, int t0, float *__restrict__ loss_out, float *__restrict__ grad_out)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    BlockSmem &S = *reinterpret_cast<BlockSmem *>(smem_raw);
    const int tid = threadIdx.x, T = kBlockThreads;
    for (int p = tid; p < NP; p += T) S.P[p] = Pg[p], S.M[p] = Mg[p], S.V[p] = Vg[p];
    __syncthreads();
    const float invB = 1.0f / (float)B;
    const Adam adam{lr, beta1, beta2, eps};
    for (int step = 0; step < steps; ++step) {
        const int *rows = idx + (int64_t)step * B;
        for (int e = tid; e < B * IN; e += T) S.X[e / IN * SX + e % IN] = X[(int64_t)rows[e / IN] * IN + e % IN];
        for (int s = tid; s < B; s += T) S.Y[s] = Y[rows[s]];
        __syncthreads();
        for (int o = tid; o < B * HD; o += T) {
            const int j = o / B, s = o % B;
            float a = S.P[OB1 + j];
            for (int k = 0; k < IN; ++k) a = __fmaf_rn(S.P[OW1 + j * IN + k], S.X[s * SX + k], a);
            S.H1[s * SH + j] = fmaxf(a, 0.f);
        }
        __syncthreads();
        for (int o = tid; o < B * HD; o += T) {
            const int j = o / B, s = o % B;
            float a = S.P[OB2 + j];
            for (int i = 0; i < HD; ++i) a = __fmaf_rn(S.P[OW2 + j * HD + i], S.H1[s * SH + i], a);
            S.H2[s * SH + j] = fmaxf(a, 0.f);
        }
        __syncthreads();
        for (int s = tid; s < B; s += T) {
            float a = S.P[OB3];
            for (int j = 0; j < HD; ++j) a = __fmaf_rn(S.P[OW3 + j], S.H2[s * SH + j], a);
            const float e = a - S.Y[s];
            S.dY[s] = 2.f * e * invB;
            S.D1[s] = e * e;   // for the loss
        }
        __syncthreads();
        for (int j = tid; j <= HD + 1; j += T) {   // w3's gradient, b3's, and the loss
            float g = 0.f;
            if (j < HD)
                for (int s = 0; s < B; ++s) g = __fmaf_rn(S.dY[s], S.H2[s * SH + j], g);
            else
                for (int s = 0; s < B; ++s) g += j == HD ? S.dY[s] : S.D1[s];
            if (j <= HD) S.G[j < HD ? OW3 + j : OB3] = g;
            else if (loss_out) loss_out[step] = g * invB;
        }
        __syncthreads();
        for (int o = tid; o < B * HD; o += T) {
            const int j = o / B, s = o % B;
            S.H2[s * SH + j] = S.H2[s * SH + j] > 0.f ? S.dY[s] * S.P[OW3 + j] : 0.f;
        }
        __syncthreads();
        for (int o = tid; o < HD * HD; o += T) {
            float g = 0.f;
            for (int s = 0; s < B; ++s) g = __fmaf_rn(S.H2[s * SH + o / HD], S.H1[s * SH + o % HD], g);
            S.G[OW2 + o] = g;
        }
        for (int j = tid; j < HD; j += T) {
            float g = 0.f;
            for (int s = 0; s < B; ++s) g += S.H2[s * SH + j];
            S.G[OB2 + j] = g;
        }
        for (int o = tid; o < B * HD; o += T) {
            const int i = o / B, s = o % B;
            float a = 0.f;
            for (int j = 0; j < HD; ++j) a = __fmaf_rn(S.H2[s * SH + j], S.P[OW2 + j * HD + i], a);
            S.D1[s * SH + i] = S.H1[s * SH + i] > 0.f ? a : 0.f;
        }
        __syncthreads();
        for (int o = tid; o < HD * IN; o += T) {
            float g = 0.f;
            for (int s = 0; s < B; ++s) g = __fmaf_rn(S.D1[s * SH + o / IN], S.X[s * SX + o % IN], g);
            S.G[OW1 + o] = g;
        }
        for (int j = tid; j < HD; j += T) {
            float g = 0.f;
            for (int s = 0; s < B; ++s) g += S.D1[s * SH + j];
            S.G[OB1 + j] = g;
        }
        __syncthreads();
        const float tf = (float)(t0 + step + 1);
        const float c[2] = {1.f - powf(beta1, tf), 1.f - powf(beta2, tf)};
        for (int p = tid; p < NP; p += T) {
            if (grad_out && step == 0) grad_out[p] = S.G[p];
            S.P[p] = adam.step(S.P[p], S.M[p], S.V[p], S.G[p], c);
        }
        __syncthreads();
    }
    for (int p = tid; p < NP; p += T) Pg[p] = S.P[p], Mg[p] = S.M[p], Vg[p] = S.V[p];
}

// Whether the current device and stream can hold k_mlp_train's cluster.
bool cluster_fits(size_t smem, cudaStream_t stream)
{
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = kCl;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(kCl);
    cfg.blockDim = dim3(kTrainThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, k_mlp_train, &cfg) == cudaSuccess) return n > 0;
    cudaGetLastError();
    return false;
}

hf_status train(bool one_block, float *params, float *adam_m, float *adam_v, const float *X, const float *Y,
                const int *idx, int steps, int batch, float lr, float beta1, float beta2, float eps, int t0,
                float *loss_out, float *grad_out, cudaStream_t stream)
{
    if (!params || !adam_m || !adam_v || !X || !Y || !idx || steps < 0 || batch < 1 ||
        batch > kMaxBatch || t0 < 0)
        return hf::set_last_error(HF_ERR_INVALID, "bad MLP training arguments (batch 1..64)");
    if (steps == 0) return HF_OK;
    cudaError_t e = cudaSuccess;
    if (!one_block) {
        e = cudaFuncSetAttribute(k_mlp_train, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(TrainSmem));
        if (e == cudaSuccess) one_block = !cluster_fits(sizeof(TrainSmem), stream);
    }
    if (one_block && e == cudaSuccess)
        e = cudaFuncSetAttribute(k_mlp_train_block, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(BlockSmem));
    if (e != cudaSuccess) return hf::set_last_error(HF_ERR_CUDA, cudaGetErrorString(e));
    if (one_block)
        k_mlp_train_block<<<1, kBlockThreads, sizeof(BlockSmem), stream>>>(
            params, adam_m, adam_v, X, Y, idx, steps, batch, lr, beta1, beta2, eps, t0, loss_out, grad_out);
    else
        k_mlp_train<<<kCl, kTrainThreads, sizeof(TrainSmem), stream>>>(
            params, adam_m, adam_v, X, Y, idx, steps, batch, lr, beta1, beta2, eps, t0, loss_out, grad_out);
    e = cudaGetLastError();
    return e == cudaSuccess ? HF_OK : hf::set_last_error(HF_ERR_CUDA, cudaGetErrorString(e));
}

} // namespace

extern "C" {

hf_status hf_mlp_forward(const float *params, const float *X, int n, float *y, void *stream)
{
    if (n < 0 || (n > 0 && (!params || !X || !y))) return hf::set_last_error(HF_ERR_INVALID, "bad MLP forward arguments");
    if (n == 0) return HF_OK;
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    // two blocks an SM share its shared-load pipe; fewer while tiles last
    const int blocks = std::min(n / kTile + (n % kTile != 0), 2 * sms);
    k_mlp_forward<<<blocks, 64 * kSlots, 0, static_cast<cudaStream_t>(stream)>>>(params, X, n, y);
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? HF_OK : hf::set_last_error(HF_ERR_CUDA, cudaGetErrorString(e));
}

hf_status hf_mlp_train(float *params, float *adam_m, float *adam_v, const float *X, const float *Y,
                       const int *idx, int steps, int batch, float lr, float beta1, float beta2,
                       float eps, int t0, float *loss_out, float *grad_out, void *stream)
{
    return train(false, params, adam_m, adam_v, X, Y, idx, steps, batch, lr, beta1, beta2, eps, t0, loss_out, grad_out,
                 static_cast<cudaStream_t>(stream));
}

hf_status hf_mlp_train_block(float *params, float *adam_m, float *adam_v, const float *X, const float *Y,
                             const int *idx, int steps, int batch, float lr, float beta1, float beta2,
                             float eps, int t0, float *loss_out, float *grad_out, void *stream)
{
    return train(true, params, adam_m, adam_v, X, Y, idx, steps, batch, lr, beta1, beta2, eps, t0, loss_out, grad_out,
                 static_cast<cudaStream_t>(stream));
}

int hf_mlp_nparams(void) { return NP; }

} // extern "C"
