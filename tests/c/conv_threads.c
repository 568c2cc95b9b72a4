// One host thread per width, each calling the channels-last layer functions
// `calls` times on its own stream and buffers.  Returns the calls refused.
#include <pthread.h>
#include <stddef.h>

typedef int (*forward_t)(const void*, const void*, const float*, float*, void*, int, int, int, int, int, int, void*);
typedef int (*data_t)(const void*, const float*, const void*, void*, float*, int, int, int, int, int, void*, size_t, void*);
typedef int (*weight_t)(const void*, const void*, float*, int, int, int, int, int, void*, size_t, void*);

typedef struct {
    forward_t forward;
    data_t data;
    weight_t weight;
    const void* a;
    const float* w;
    void** p;  // x, act, g, dw, db, workspace, stream
    size_t bytes;
    int ch, H, W, calls, refused;
} job_t;

static void* run(void* arg) {
    job_t* j = arg;
    void** p = j->p;
    for (int k = 0; k < j->calls; ++k) {
        j->refused += j->forward(p[0], j->a, NULL, NULL, p[1], 1, j->ch, j->ch, j->H, j->W, 1, p[6]) != 0;
        j->refused += j->data(p[0], j->w, p[1], p[2], p[4], 1, j->ch, j->ch, j->H, j->W, p[5], j->bytes, p[6]) != 0;
        j->refused += j->weight(p[0], p[0], p[3], 1, j->ch, j->ch, j->H, j->W, p[5], j->bytes, p[6]) != 0;
    }
    return NULL;
}

int conv_threads(void* forward, void* data, void* weight, const void* a, const float* w, int ch, int H, int n,
                 const int* widths, void** ptrs, const size_t* bytes, int calls) {
    enum { MOST = 8 };
    pthread_t th[MOST];
    job_t job[MOST];
    if (n > MOST) return -1;
    for (int i = 0; i < n; ++i) {
        job_t j = {(forward_t)forward, (data_t)data, (weight_t)weight, a, w, ptrs + 7 * i, bytes[i], ch, H, widths[i],
                   calls, 0};
        job[i] = j;
        if (pthread_create(&th[i], NULL, run, &job[i])) return -1;
    }
    int refused = 0;
    for (int i = 0; i < n; ++i) {
        pthread_join(th[i], NULL);
        refused += job[i].refused;
    }
    return refused;
}
